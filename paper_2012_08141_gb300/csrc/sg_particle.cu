// sg_particle.cu -- particle-grid transfers on the sparse grid (the hybrid
// Lagrangian-Eulerian workload of AsyncTaichi Sec. 8.3): P2G with activation,
// the grid velocity update, and G2P, as PIC transfers or as affine (APIC)
// transfers with a per-particle 3x3 matrix C (the transfers of MLS-MPM);
// quadratic B-spline weights.  The unit cube holds N^3 nodes, dx = 1/N, node
// (i,j,k) at (i,j,k)*dx, particle component a maps to grid axis a (z -> k).
// C is stored row-major, 9 floats per particle: (C d)_a = sum_b C[3a+b] d_b.
// For quadratic B-splines sum_n w d d^T = dx^2/4 I, so the APIC G2P matrix is
// C = (4/dx^2) sum_n w v_n d^T with d = node - x_p = ((a,b,c) - fx) dx.
#include <utility>
#include "sg_particle.cuh"

namespace sg {

// Grid update over the active nodes of the listed leaves.
__global__ void __launch_bounds__(256) k_grid_update(DevGrid g, int f_mass, int f_mom0, float dt, float gz, int bound)
{
    chained_entry();
    const long long n = g.ctrl->list_n;
    const int L = g.L, lg2 = g.lg2, R = g.R, N = g.N, V = L * L * L;
    float *fm = g.field[f_mass];
    float *fv[3] = {g.field[f_mom0], g.field[f_mom0 + 1], g.field[f_mom0 + 2]};
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * V; q += (long long)gridDim.x * blockDim.x) {
        const long long e = q >> (3 * lg2);
        const int l = (int)(q - (e << (3 * lg2)));
        const int slot = g.list_slot[e];
        if (!((g.mask[(long long)slot * g.W + (l >> 5)] >> (l & 31)) & 1u)) continue;
        const int b = g.list_b[e];
        const int idx[3] = {(b / (R * R)) * L + (l >> (2 * lg2)), ((b / R) % R) * L + ((l >> lg2) & (L - 1)),
                            (b % R) * L + (l & (L - 1))};
        const long long o = (long long)slot * V + l;
        const float m = fm[o];
        float u[3] = {0.f, 0.f, 0.f};
        if (m > 0.f) {
#pragma unroll
            for (int d = 0; d < 3; ++d) u[d] = fv[d][o] / m;
            u[2] -= dt * gz;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (idx[d] < bound && u[d] < 0.f) u[d] = 0.f;
                if (idx[d] > N - bound && u[d] > 0.f) u[d] = 0.f;
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) fv[d][o] = u[d];
    }
}

void launch_grid_update(const DevGrid &g, cudaStream_t s, int f_mass, int f_mom0, float dt, float gz, int bound,
                        const LaunchCfg &lc)
{
    launch_chained(k_grid_update, lc.num_sms * 8, 256, 0, s, g, f_mass, f_mom0, dt, gz, bound);
}

// G2P in input order, every node read from the grid.
template <bool APIC>
__global__ void __launch_bounds__(256) k_g2p(DevGrid g, float *__restrict__ x, float *__restrict__ v,
                                             float *__restrict__ C, long long n, float dt, int f_mom0)
{
    chained_entry();
    const float *f0 = g.field[f_mom0], *f1 = g.field[f_mom0 + 1], *f2 = g.field[f_mom0 + 2];
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x) {
        const float3 xp = make_float3(x[3 * p], x[3 * p + 1], x[3 * p + 2]);
        const Spline sx = bspline(xp.x, g.N), sy = bspline(xp.y, g.N), sz = bspline(xp.z, g.N);
        float3 u;
        float c[9];
        g2p_from_grid<APIC>(g, f0, f1, f2, sx, sy, sz, u, c);
        const float vn[3] = {u.x, u.y, u.z}, xo[3] = {xp.x, xp.y, xp.z};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            v[3 * p + a] = vn[a];
            x[3 * p + a] = xo[a] + dt * vn[a];
        }
        if (APIC) {
#pragma unroll
            for (int q = 0; q < 9; ++q) C[9 * p + q] = c[q];
        }
    }
}

// The bins of few particles, a warp each (w: this warp among `warps`; s: its
// scratch of kBinNodes).
template <int L, bool APIC>
__device__ __noinline__ void g2p_few(const DevGrid &g, const BinSplit &bins, float *x, float *v, float *C, float dt, int f_mom0,
                                     int w, int warps, float4 *s)
{
    const int lane = lane_id();
    for (; w < bins.few; w += warps) {
        const int b = g.bin_list[bins.last - w], beg = g.bin_off[b], cnt = g.bin_count[b] - beg;
        int bi, bj, bk;
        bin_block<L>(b, g.R, bi, bj, bk);
        const long long p = lane < cnt ? g.perm[beg + lane] : -1;
        float xp[3] = {}, u[3] = {}, c[9] = {};
        if (p >= 0) {
#pragma unroll
            for (int e = 0; e < 3; ++e) xp[e] = x[3 * p + e];
        }
        g2p_of_bin<L, APIC>(g, g.field[f_mom0], g.field[f_mom0 + 1], g.field[f_mom0 + 2], bi, bj, bk, cnt, xp, s, u, c);
        if (p >= 0) {
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                v[3 * p + e] = u[e];
                x[3 * p + e] = xp[e] + dt * u[e];
            }
            if (APIC) {
#pragma unroll
                for (int e = 0; e < 9; ++e) C[9 * p + e] = c[e];
            }
        }
    }
}

// G2P over the bins of the last binned P2G: per bin, the node velocities of
// the 6^3 nodes from o to o + 5 (o the bin's first node; every node a stencil
// with base in [o, o + 3] reaches) are staged in shared memory, 0 outside the
// domain or the allocated leaves, and the bin's particles read their 27 nodes
// there.  A particle whose base lies outside that range (its position changed
// since the binning, or a base of -2 / -1 at the low domain face) reads the grid
// node by node, as do the particles whose stencil misses the domain (the last
// bin).  Bins of few particles go by warps, and several CTAs share a bin when
// there are few bins (bin_split).  A warp moves its particles' words together (see
// warp_fetch), positions one round ahead.  It waits on the bin's serial chain
// (bin, order, positions; root, node values) and on the 27 shared 16-byte
// reads a particle.  2M particles, about 10 a cell: 63 us, APIC 100k 11.5 us
// (77 and 19.7 us with each lane moving its own particle and three 64-bit
// divisions per bin).  APIC at three CTAs per SM: at four its 9 words of C
// spill (13.4 us).
template <int L, bool APIC>
__global__ void __launch_bounds__(256, APIC ? 3 : 4) k_g2p_binned(const __grid_constant__ DevGrid g,
                                                                  float *__restrict__ x, float *__restrict__ v,
                                                                  float *__restrict__ C, float dt, int f_mom0)
{
    chained_entry();
    constexpr int B = 6;
    __shared__ float4 s_raw[8 * kBinNodes];  // a bin's nodes and each warp's words, or a bin's nodes for each warp
    float4 *s_u = s_raw;
    float *s_t = reinterpret_cast<float *>(s_raw + kBinNodes) + (threadIdx.x >> 5) * (32 * (APIC ? 9 : 3));
    const int N = g.N, R = g.R;
    const float *f0 = g.field[f_mom0], *f1 = g.field[f_mom0 + 1], *f2 = g.field[f_mom0 + 2];
    const BinSplit bins = bin_split(g.ctrl, R, L, 1, 4);
    const int used = bins.all, oob_bin = bins.last + 1;
    // this CTA's share of a bin that several take; the next bin and its particle
    // range are read a bin ahead
    const int part = bins.parts > 1 ? blockIdx.x / (used + 1) : 0, first = blockIdx.x - part * (used + 1);
    int nb = first < used ? nth_bin(g.bin_list, bins, first) : oob_bin;
    int nbeg = g.bin_off[nb], nend = g.bin_count[nb];
    for (int bl = part < bins.parts ? first : used + 1; bl <= used; bl += gridDim.x) {
        const int b = nb, next = bl + (int)gridDim.x;
        const unsigned beg = nbeg + 256u * part, end = nend;
        if (next <= used) {
            nb = next < used ? nth_bin(g.bin_list, bins, next) : oob_bin;
            nbeg = g.bin_off[nb];
            nend = g.bin_count[nb];
        }
        int oi, oj, ok;
        bin_block<L>(b, R, oi, oj, ok);
        oi *= 4;
        oj *= 4;
        ok *= 4;
        // a warp's particles, 32 at a time; their positions are requested
        // before the staging barrier and one round ahead
        unsigned q = beg + (threadIdx.x & ~31) + lane_id();
        int p = q < end ? g.perm[q] : -1;
        float t[3];
        warp_fetch<3>(x, p, t);
        if (bl < used) {
            for (int nd = threadIdx.x; nd < B * B * B; nd += 256) {
                const int i = oi + nd / (B * B), j = oj + (nd / B) % B, k = ok + nd % B;
                float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
                const int bs = block_slot<L>(g.root, R, i >> 2, j >> 2, k >> 2);
                if (bs >= 0) {
                    const long long idx = block_voxel<L>(bs, i & 3, j & 3, k & 3);
                    u = make_float4(__ldg(f0 + idx), __ldg(f1 + idx), __ldg(f2 + idx), 0.f);
                }
                s_u[nd] = u;
            }
            __syncthreads();
        }
        while (q - lane_id() < end) {
            float xp[3];
            warp_deal<3>(t, s_t, xp);
            const int cur = p;
            q += blockDim.x * bins.parts;
            if (q - lane_id() < end) {
                p = q < end ? g.perm[q] : -1;
                warp_fetch<3>(x, p, t);
            }
            const Spline sx = bspline(xp[0], N), sy = bspline(xp[1], N), sz = bspline(xp[2], N);
            const int ri = sx.base - oi, rj = sy.base - oj, rk = sz.base - ok;
            float3 u = make_float3(0.f, 0.f, 0.f);
            float c[9] = {};
            if (bl < used && (unsigned)ri < 4u && (unsigned)rj < 4u && (unsigned)rk < 4u)
                g2p_from_block<B, APIC>(s_u, ri, rj, rk, N, sx, sy, sz, u, c);
            else if (cur >= 0)
                g2p_from_grid<APIC>(g, f0, f1, f2, sx, sy, sz, u, c);
            const float vn[3] = {u.x, u.y, u.z};
            const float xn[3] = {xp[0] + dt * u.x, xp[1] + dt * u.y, xp[2] + dt * u.z};
            warp_put<3>(v, cur, vn, s_t);
            warp_put<3>(x, cur, xn, s_t);
            if (APIC) warp_put<9>(C, cur, c, s_t);
        }
        __syncthreads();  // s_u is restaged for the next bin
    }
    if (bins.few)
        g2p_few<L, APIC>(g, bins, x, v, C, dt, f_mom0, blockIdx.x * 8 + (threadIdx.x >> 5), gridDim.x * 8,
                         s_raw + (threadIdx.x >> 5) * kBinNodes);
}

// CTAs of a persistent per-bin kernel: as many as fit on every SM at once.
template <typename K>
static int resident_ctas(K kernel, int num_sms)
{
    int per = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, 256, 0) != cudaSuccess || per < 1) per = 1;
    return per * num_sms;
}

void launch_g2p(const DevGrid &g, cudaStream_t s, float *x, float *v, float *C, long long n, float dt, int f_mom0,
                int binned, const LaunchCfg &lc)
{
    if (n <= 0) return;
    if (binned) {
#define SG_G2PB(LL, AP) launch_chained(k_g2p_binned<LL, AP>, resident_ctas(k_g2p_binned<LL, AP>, lc.num_sms), 256, 0, s, g, x, v, C, dt, f_mom0)
        if (C) {
            if (g.L == 4) SG_G2PB(4, true);
            else SG_G2PB(8, true);
        } else {
            if (g.L == 4) SG_G2PB(4, false);
            else SG_G2PB(8, false);
        }
#undef SG_G2PB
        return;
    }
    long long blocks = (n + 255) / 256;
    if (blocks > 1 << 20) blocks = 1 << 20;
    if (C) launch_chained(k_g2p<true>, (unsigned)blocks, 256, 0, s, g, x, v, C, n, dt, f_mom0);
    else launch_chained(k_g2p<false>, (unsigned)blocks, 256, 0, s, g, x, v, C, n, dt, f_mom0);
}

}  // namespace sg

// ===========================================================================
// Binned P2G.  Each step the particles are binned by the 4^3 block of nodes
// (a leaf, or an octant of an 8^3 leaf) that holds the lowest corner (base
// node) of their 3x3x3 stencil; a bin's particles are summed on its 6^3 nodes
// (every node their stencils can reach) in shared memory, and each touched node
// is added to the grid once: 4 global atomics instead of 27 x 4 per particle.
//   1. k_bin_clear   counts and reach classes to zero
//   2. k_p2g_bin     count particles per bin and note the neighbour leaves that
//                    their stencils reach
//   3. k_bin_tiles   tile sums of the counts; mark the leaves and neighbours
//   4. k_bin_place   allocate the marked leaves; exclusive scan of the counts
//                    (the count array becomes each bin's insertion cursor);
//                    list of occupied bins
//   5. k_p2g_perm    write particle indices in bin order
//   6. k_p2g_gather  per bin: sort the particles by cell in shared memory, sum
//                    by columns of cells, add the touched nodes to the grid and
//                    set their bits (PIC, or APIC with the per-particle matrix
//                    C); bins of few particles by a warp (see bin_split)
// An 8^3 leaf is eight bins: as one (a warp per cell over 10^3 nodes, chunks of
// 256 particles) eight steps of 500k PIC particles took 2340 us instead of 913,
// of 1.8M APIC particles 6390 instead of 3050, of 1.8M particles with fused
// G2P2G 7650 instead of 2530.
// ===========================================================================
namespace sg {

// A count per bin, not one per leaf and reach class: with the classes in the
// count array the clear, the two passes of the scan and the list read 8 R^3
// words, and two memsets and the scan of the tile sums came between them (a P2G of
// 200k particles in a 25^3 root 58 -> 46 us, 64^3 76 -> 56, 128^3 304 -> 204,
// 256^3 1,817 -> 1,032).  What is left in a small root is the latency of the
// dependent launches.

// Bin of a particle: the block of its base node; one past the last bin when no
// stencil node lies inside the domain.  Bit 2 / 1 / 0 of cls says that the
// in-domain part of the stencil extends into the next leaf along i / j / k.
// The base block is that of max(base, 0): base is at least -2 for a non-empty
// stencil, and -2 / -1 lie below block 0.
__device__ __forceinline__ int p2g_bin_of(const float *__restrict__ x, long long p, int N, int lg2, int R, int &cls)
{
    int leaf = 0, oct = 0;
    bool empty = false;
    cls = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const Spline s = bspline(__ldg(x + 3 * p + a), N);
        const int n0 = max(s.base, 0), n1 = min(s.base + 2, N - 1);
        empty |= n0 > n1;
        leaf = leaf * R + (n0 >> lg2);
        oct = oct * 2 + (n0 >> 2 & 1);
        cls = (cls << 1) | ((n1 >> lg2) != (n0 >> lg2) ? 1 : 0);
    }
    if (empty) leaf = R * R * R;
    return lg2 == 2 ? leaf : leaf * 8 + (empty ? 0 : oct);
}

// A thread per four bins (the arrays are padded to whole tiles).
__global__ void __launch_bounds__(256) k_bin_clear(DevGrid g)
{
    chained_entry();
    const long long q = blockIdx.x * 256LL + threadIdx.x;
    reinterpret_cast<int4 *>(g.bin_count)[q] = make_int4(0, 0, 0, 0);
    if (q < p2g_words(p2g_bins(g.R, 2)) / 4) reinterpret_cast<int4 *>(g.bin_reach)[q] = make_int4(0, 0, 0, 0);
    if (q == 0) g.ctrl->bins_used = g.ctrl->bins_few = g.ctrl->moved[0] = g.ctrl->moved[1] = g.ctrl->moved[2] = 0;
}

// Particles of one bin with the reach classes `classes` (a bit each).  The
// leaf's word is read first: after its first particles the bits are there.
__device__ __forceinline__ void note_reach(const DevGrid &g, int b, unsigned classes)
{
    uint32_t *w = g.bin_reach + (g.lg2 == 2 ? b : b >> 3);
    if (classes & ~__ldcg(w)) atomicOr(w, classes);
}

// The count passes store each particle's bin (at its position in the order
// they visit: the particle index here, the last order's slot in the rebin)
// for the order passes, which then read bins in order instead of positions.
__global__ void k_p2g_bin(DevGrid g, const float *__restrict__ x, long long n)
{
    chained_entry();
    const int oob_bin = (int)p2g_bins(g.R, g.lg2);
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x) {
        int cls;
        const int b = p2g_bin_of(x, p, g.N, g.lg2, g.R, cls);
        g.perm_key[p] = b;
        atomicAdd(&g.bin_count[b], 1);
        if (b < oob_bin) note_reach(g, b, 1u << cls);
    }
}

// Rebinning: the particles are visited in the last binning's order, so the
// lanes of a warp mostly share a bin (particles move little between steps);
// one atomic per distinct bin in the warp.
__global__ void k_p2g_rebin(DevGrid g, const float *__restrict__ x, long long n)
{
    chained_entry();
    const int lane = lane_id();
    const int oob_bin = (int)p2g_bins(g.R, g.lg2);
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        int cls;
        const int b = p2g_bin_of(x, g.perm[q], g.N, g.lg2, g.R, cls);
        g.perm_key[q] = b;
        const unsigned peers = __match_any_sync(__activemask(), b);
        const unsigned classes = __reduce_or_sync(peers, 1u << cls);
        if (lane == __ffs(peers) - 1) {
            atomicAdd(&g.bin_count[b], __popc(peers));
            if (b < oob_bin) note_reach(g, b, classes);
        }
    }
}

// Sum of each tile of kBinTile counts; for every leaf with particles, mark it
// and the neighbours that their stencils reach for allocation (every subset of
// every class seen).
__global__ void __launch_bounds__(256) k_bin_tiles(DevGrid g)
{
    chained_entry();
    __shared__ int s_w[8];
    const int base = (blockIdx.x * 256 + threadIdx.x) * 4;  // below 2^30 + kBinTile
    const int4 c4 = reinterpret_cast<const int4 *>(g.bin_count)[base >> 2];
    auto mark = [&](int leaf, uint32_t reach) {
        if (!reach) return;
#pragma unroll
        for (int sub = 0; sub < 8; ++sub) {
            const uint32_t with = ((sub & 4) ? 0xF0u : 0xFFu) & ((sub & 2) ? 0xCCu : 0xFFu) & ((sub & 1) ? 0xAAu : 0xFFu);
            if (reach & with) g.need[leaf + ((sub >> 2) * g.R + ((sub >> 1) & 1)) * g.R + (sub & 1)] = 1;
        }
    };
    if (g.lg2 == 2) {
        const uint4 r4 = reinterpret_cast<const uint4 *>(g.bin_reach)[base >> 2];
        mark(base, r4.x);
        mark(base + 1, r4.y);
        mark(base + 2, r4.z);
        mark(base + 3, r4.w);
    } else if (!(base & 7)) {
        mark(base >> 3, g.bin_reach[base >> 3]);
    }
    const int v = warp_sum(c4.x + c4.y + c4.z + c4.w);
    if (lane_id() == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < 8; ++w) t += s_w[w];
        g.tile_sum[blockIdx.x] = t;
    }
}

// Exclusive scan of the tile sums by one CTA (in place).
__global__ void __launch_bounds__(1024) k_bin_scan_top(DevGrid g, int ntiles)
{
    chained_entry();
    __shared__ int s_w[32];
    __shared__ int s_carry;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < ntiles; base += 1024) {
        const int i = base + threadIdx.x;
        const int v = (i < ntiles) ? g.tile_sum[i] : 0;
        const int inc = warp_incl_scan(v);
        if (lane_id() == 31) s_w[threadIdx.x >> 5] = inc;
        __syncthreads();
        if (threadIdx.x < 32) {
            const int wv = s_w[threadIdx.x];
            s_w[threadIdx.x] = warp_incl_scan(wv) - wv;
        }
        __syncthreads();
        const int excl = s_carry + s_w[threadIdx.x >> 5] + inc - v;
        __syncthreads();
        if (i < ntiles) g.tile_sum[i] = excl;
        if (threadIdx.x == 1023) s_carry = excl + v;
        __syncthreads();
    }
}

// CTAs 0 .. alloc_ctas - 1 allocate the marked leaves; CTA alloc_ctas + t
// turns tile t's counts into the exclusive offsets (the count array becomes
// the insertion cursor, bin_off keeps the offset) and lists its occupied
// bins.  Neither half needs the other, so one launch holds both.  The tile
// sums before t are added up by the CTA itself, which spares the scan of them
// by k_bin_scan_top (a P2G of 200k particles over 16 tiles 45.8 us against
// 47.0, 257 tiles 55.9 / 58.9, 4,001 tiles 360 / 361).  That reading grows with
// the square of the tiles: at 16,385 both take 1,032 us, and with more than
// kMaxOwnTiles the scan runs (`scanned`: the sums are offsets already).
constexpr int kMaxOwnTiles = 16384;
__global__ void __launch_bounds__(256) k_bin_place(DevGrid g, int alloc_ctas, bool scanned)
{
    chained_entry();
    if ((int)blockIdx.x < alloc_ctas) {
        alloc_needed(g, 0xffffffffu, blockIdx.x, alloc_ctas);
        return;
    }
    __shared__ int s_w[8], s_before[8];
    const int tile = blockIdx.x - alloc_ctas, warp = threadIdx.x >> 5, lane = lane_id();
    const int base = tile * kBinTile + threadIdx.x * 4;
    const int4 c4 = reinterpret_cast<const int4 *>(g.bin_count)[base >> 2];
    int before = 0;
    if (scanned) {
        if (threadIdx.x == 0) before = g.tile_sum[tile];
    } else {
        for (int i = threadIdx.x; i < tile; i += 256) before += g.tile_sum[i];
    }
    const int t = c4.x + c4.y + c4.z + c4.w;
    const int inc = warp_incl_scan(t);
    before = warp_sum(before);
    if (lane == 31) {
        s_w[warp] = inc;
        s_before[warp] = before;
    }
    __syncthreads();
    int run = inc - t;
#pragma unroll
    for (int w = 0; w < 8; ++w) run += s_before[w] + (w < warp ? s_w[w] : 0);
    const int4 at = make_int4(run, run + c4.x, run + c4.x + c4.y, run + c4.x + c4.y + c4.z);
    reinterpret_cast<int4 *>(g.bin_off)[base >> 2] = at;
    reinterpret_cast<int4 *>(g.bin_count)[base >> 2] = at;
    // list of the bins with particles (the out-of-domain bin excluded)
    const int oob_bin = (int)p2g_bins(g.R, g.lg2);
    const int cnt[4] = {c4.x, c4.y, c4.z, c4.w};
    int mine = 0;  // bins of more than kFewParticles, and in the upper half the others
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (cnt[q] > 0 && base + q < oob_bin) mine += cnt[q] > kFewParticles ? 1 : 0x10000;
    const int upto = warp_incl_scan(mine), all = __shfl_sync(kFull, upto, 31);
    if (all) {
        int first = 0, few = 0;
        if (lane == 31 && (all & 0xffff)) first = atomicAdd(&g.ctrl->bins_used, all & 0xffff);
        if (lane == 31 && all >> 16) few = atomicAdd(&g.ctrl->bins_few, all >> 16);
        first = __shfl_sync(kFull, first, 31) + (upto - mine & 0xffff);
        few = oob_bin - 1 - (__shfl_sync(kFull, few, 31) + (upto - mine >> 16));
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (cnt[q] > 0 && base + q < oob_bin) g.bin_list[cnt[q] > kFewParticles ? first++ : few--] = base + q;
    }
}

__global__ void k_p2g_perm(DevGrid g, long long n)
{
    chained_entry();
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x) {
        const int pos = atomicAdd(&g.bin_count[g.perm_key[p]], 1);
        g.perm[pos] = (int)p;
    }
}

// The new order from the last one, written to perm_alt (warp-aggregated
// cursor atomics, as in k_p2g_rebin).
__global__ void k_p2g_reperm(DevGrid g, long long n)
{
    chained_entry();
    const int lane = lane_id();
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const int p = g.perm[q];
        const int key = g.perm_key[q];
        const unsigned peers = __match_any_sync(__activemask(), key);
        const int leader = __ffs(peers) - 1;
        int base = 0;
        if (lane == leader) base = atomicAdd(&g.bin_count[key], __popc(peers));
        base = __shfl_sync(peers, base, leader);
        g.perm_alt[base + __popc(peers & lanemask_lt())] = p;
    }
}

// Per bin, the sums by columns (see bin_columns).  While a chunk's columns are
// summed, the words of the next one's particles come into shared memory
// (cp.async, whole warps moving whole records), so the CTA does not wait for
// its scattered reads.  A bin of several chunks deals its particles
// to them in turn, so that each chunk has its share of every column though the
// order is by cell; the cell order of each chunk goes to perm_alt, which the
// host then swaps with perm.  2M PIC particles over 4,076 leaves: 111 us
// (a warp per cell with FP32 shared atomics: 135 us); 100k APIC particles 20.5
// us (24.8).  Three CTAs per SM: PIC at four spills (121 us), APIC with twice
// the chunk at two takes 25 us.
template <bool APIC>
struct GatherSmem {
    static constexpr int PPT = APIC ? 2 : 4, CAP = APIC ? PPT * kBinThreads : 736, NREC = APIC ? 4 : 2;
    float4 rec[NREC][CAP];
    float4 buf[kBinBuf];
    float x[3 * CAP], v[3 * CAP], C[APIC ? 9 * CAP : 1];  // the next chunk's words, in particle order
    uint16_t idx[CAP + 2];
    BinSort sort;
};

// The bins of few particles, a warp each; s: the CTA's scratch (kFewScratch a
// warp).  Returns whether the structure changed.
template <int L, bool APIC>
__device__ __noinline__ bool gather_few(const DevGrid &g, const BinSplit &bins, const float *__restrict__ x, const float *__restrict__ v,
                                        const float *__restrict__ C, float pmass, int f_mass, int f_mom0, float4 *s)
{
    const int R = g.R, N = g.N, lane = lane_id(), warp = threadIdx.x >> 5;
    float *fm = g.field[f_mass], *f0 = g.field[f_mom0], *f1 = g.field[f_mom0 + 1], *f2 = g.field[f_mom0 + 2];
    bool changed = false;
    s += warp * kFewScratch;
    auto add = [&](int bs, int i, int j, int k, const float4 &t) {
        if (bs < 0) return;  // outside the domain, or the pool is exhausted (latched)
        const long long idx = block_voxel<L>(bs, i & 3, j & 3, k & 3);
        changed |= set_bit(g, idx);
        atomicAdd(fm + idx, pmass * t.x);
        atomicAdd(f0 + idx, pmass * t.y);
        atomicAdd(f1 + idx, pmass * t.z);
        atomicAdd(f2 + idx, pmass * t.w);
    };
    for (int w = blockIdx.x * kBinWarps + warp; w < bins.few; w += gridDim.x * kBinWarps) {
        const int b = g.bin_list[bins.last - w], beg = g.bin_off[b], cnt = g.bin_count[b] - beg;
        int bi, bj, bk;
        bin_block<L>(b, R, bi, bj, bk);
        const int slot = lane < 8 ? block_slot<L>(g.root, R, bi + (lane >> 2), bj + ((lane >> 1) & 1), bk + (lane & 1)) : -1;
        FewParticle<APIC> r{};
        long long p = -1;
        if (lane < cnt) {
            p = g.perm[beg + lane];
            const float vp[3] = {v[3 * p], v[3 * p + 1], v[3 * p + 2]};
            float c[9] = {};
            if (APIC) {
#pragma unroll
                for (int e = 0; e < 9; ++e) c[e] = C[9 * p + e];
            }
            few_particle<APIC>(r, x[3 * p], x[3 * p + 1], x[3 * p + 2], vp, c, N);
        }
        // the cell order, which G2P reads
        const int ri = r.b[0] - 4 * bi, rj = r.b[1] - 4 * bj, rk = r.b[2] - 4 * bk;
        const int key = ((unsigned)(ri | rj | rk) < 4u ? (ri * 4 + rj) * 4 + rk : 64) << 5 | lane;
        int rank = 0;
        for (int t = 0; t < cnt; ++t) rank += __shfl_sync(kFull, key, t) < key;
        if (lane < cnt) g.perm_alt[beg + rank] = (int)p;
        const unsigned strays = few_sums<APIC>(r, cnt, 4 * bi, 4 * bj, 4 * bk, s);
        for (int nd = lane; nd < 224; nd += 32) {
            int i, j, k, blk, l;
            bin_node(nd, i, j, k, blk, l);
            const int bs = __shfl_sync(kFull, slot, blk & 7);
            if (nd < kBinNodes && few_hit(s, i, j, k)) add(bs, i, j, k, s[nd]);
        }
        few_strays<APIC>(r, strays, [&](int i, int j, int k, const float4 &t) {
            if ((unsigned)i < (unsigned)N && (unsigned)j < (unsigned)N && (unsigned)k < (unsigned)N)
                add(block_slot<L>(g.root, R, i >> 2, j >> 2, k >> 2), i, j, k, t);
        });
        __syncwarp();  // s is cleared for the next bin
    }
    return changed;
}

template <int L, bool APIC>
__global__ void __launch_bounds__(kBinThreads, 3) k_p2g_gather(const __grid_constant__ DevGrid g, const float *__restrict__ x,
                                                               const float *__restrict__ v,
                                                               const float *__restrict__ C, float pmass, int f_mass,
                                                               int f_mom0)
{
    chained_entry();
    using S = GatherSmem<APIC>;
    constexpr int PPT = S::PPT, CAP = S::CAP;
    extern __shared__ __align__(16) unsigned char smem[];
    S &s = *reinterpret_cast<S *>(smem);
    const int N = g.N, R = g.R;
    const float dx = 1.f / (float)N;
    const int warp = threadIdx.x >> 5, lane = lane_id();
    float *fm = g.field[f_mass];
    float *f0 = g.field[f_mom0], *f1 = g.field[f_mom0 + 1], *f2 = g.field[f_mom0 + 2];
    bool changed = false;
    const BinSplit bins = bin_split(g.ctrl, R, L, 0, 4);
    const int used = bins.all;
    {   // the particles whose stencil misses the domain keep their order
        const int oob_bin = bins.last + 1;
        const int end = g.bin_count[oob_bin];
        for (int q = g.bin_off[oob_bin] + blockIdx.x * kBinThreads + threadIdx.x; q < end; q += gridDim.x * kBinThreads)
            g.perm_alt[q] = g.perm[q];
    }
    static_assert(kBinWarps * kFewScratch <= S::NREC * CAP, "the bins of few particles use the records' memory");
    auto few = [&] { return bins.few && gather_few<L, APIC>(g, bins, x, v, C, pmass, f_mass, f_mom0, s.rec[0]); };
    // of a bin that several CTAs share, this one takes chunks part, part + parts, ...
    const int parts = bins.parts, part = parts > 1 ? blockIdx.x / used : 0;
    int bl = blockIdx.x - part * used;
    // a bin and its particle range; slot of its corner block (threads 0 .. 7)
    auto bin_of = [&](int l, int &b, int &beg, int &end) {
        b = nth_bin(g.bin_list, bins, l);
        beg = g.bin_off[b];
        end = g.bin_count[b];
    };
    auto corner_slot = [&](int b) {
        int bi, bj, bk;
        bin_block<L>(b, R, bi, bj, bk);
        const int t = threadIdx.x;
        return t < 8 ? block_slot<L>(g.root, R, bi + (t >> 2), bj + ((t >> 1) & 1), bk + (t & 1)) : -1;
    };
    // chunk c of nch takes particles beg + c, beg + c + nch, ...
    auto order = [&](int beg, int end, int c, int nch, int (&p)[PPT]) {
#pragma unroll
        for (int u = 0; u < PPT; ++u) {
            const long long q = beg + c + (long long)((u * kBinWarps + warp) * 32 + lane) * nch;
            p[u] = q < end ? g.perm[q] : -1;
        }
    };
    auto request = [&](const int (&p)[PPT]) {
#pragma unroll
        for (int u = 0; u < PPT; ++u) {
            const int q0 = (u * kBinWarps + warp) * 32;
            if (__any_sync(kFull, p[u] >= 0)) {
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    const int e = r * 32 + lane, src = e / 3, q = __shfl_sync(kFull, p[u], src);
                    if (q >= 0) {
                        copy_word(s.x + 3 * q0 + e, x + 3LL * q + (e - 3 * src));
                        copy_word(s.v + 3 * q0 + e, v + 3LL * q + (e - 3 * src));
                    }
                }
                if (APIC) {
#pragma unroll
                    for (int r = 0; r < 9; ++r) {
                        const int e = r * 32 + lane, src = e / 9, q = __shfl_sync(kFull, p[u], src);
                        if (q >= 0) copy_word(s.C + 9 * q0 + e, C + 9LL * q + (e - 9 * src));
                    }
                }
            }
        }
    };
    int b, beg = 0, end = 0, nb = 0, nbeg = 0, nend = 0;
    if (bl < used && part < parts) bin_of(bl, b, beg, end);
    int c = part, nch = (end - beg + CAP - 1) / CAP;
    if (c >= nch) {
        if (few()) mark_dirty(g);
        return;
    }
    int slot = corner_slot(b);
    int p[PPT], pn[PPT];
    order(beg, end, c, nch, p);
    request(p);
    if (bl + (int)gridDim.x < used) bin_of(bl + gridDim.x, nb, nbeg, nend);
    if (threadIdx.x < 65) s.sort.cnt[threadIdx.x] = 0;
    if (threadIdx.x < 16) s.sort.all[threadIdx.x] = s.sort.bits[threadIdx.x] = 0;
    if (threadIdx.x < 8) s.sort.slot[threadIdx.x] = slot;
    __syncthreads();
    for (;;) {
        // what comes after this chunk: the bin's next one, or the next bin
        const bool last = c + parts >= nch, more = !last || bl + (int)gridDim.x < used;
        const int nnch = last ? (nend - nbeg + CAP - 1) / CAP : nch;
        if (more) order(last ? nbeg : beg, last ? nend : end, last ? 0 : c + parts, nnch, pn);
        if (last && more) slot = corner_slot(nb);
        int oi, oj, ok;
        bin_block<L>(b, R, oi, oj, ok);
        oi *= 4;
        oj *= 4;
        ok *= 4;
        copies_done();
        __syncwarp();
        // each particle's record, its cell and its rank among the cell's particles
        int place[PPT];
#pragma unroll
        for (int u = 0; u < PPT; ++u) {
            const int q = (u * kBinWarps + warp) * 32 + lane;
            place[u] = 0;
            if (p[u] >= 0) {
                const Spline sx = bspline(s.x[3 * q], N), sy = bspline(s.x[3 * q + 1], N), sz = bspline(s.x[3 * q + 2], N);
                const int ri = sx.base - oi, rj = sy.base - oj, rk = sz.base - ok;
                const bool in = (unsigned)ri < 4u && (unsigned)rj < 4u && (unsigned)rk < 4u;
                const int cell = in ? (ri * 4 + rj) * 4 + rk : 64;
                place[u] = cell | atomicAdd(&s.sort.cnt[cell], 1) << 7;
                float m[9];
                if (APIC) {
#pragma unroll
                    for (int e = 0; e < 9; ++e) m[e] = s.C[9 * q + e];
                }
                bin_record<APIC, CAP>(s.rec, q, sx.fx, sy.fx, sz.fx, s.v[3 * q], s.v[3 * q + 1], s.v[3 * q + 2], m, dx, !in,
                                      pack_cell(ri, rj, rk));
            }
        }
        __syncthreads();
        if (warp == 0) bin_scan(g, s.sort, CAP);
        __syncthreads();
        // the chunk's cell order (G2P reads it)
        const int first = beg + c * ((end - beg) / nch) + min(c, (end - beg) % nch);
#pragma unroll
        for (int u = 0; u < PPT; ++u)
            if (p[u] >= 0) {
                const int pos = s.sort.start[place[u] & 127] + (place[u] >> 7);
                s.idx[pos] = (uint16_t)((u * kBinWarps + warp) * 32 + lane);
                g.perm_alt[first + pos] = p[u];
            }
        __syncthreads();
        if (more) request(pn);
        bin_columns<APIC, CAP>(s.rec, s.idx, s.sort, s.buf);
        // bases -2 / -1 at the low domain faces: straight to the grid
        for (int pp = s.sort.start[64] + warp; pp < s.sort.start[65] && pp < CAP; pp += kBinWarps) {
            int i, j, k;
            float4 t;
            if (!edge_node<APIC, CAP>(s.rec, s.idx[pp], oi, oj, ok, N, i, j, k, t)) continue;
            const int es = block_slot<L>(g.root, R, i >> 2, j >> 2, k >> 2);
            if (es < 0) continue;  // pool exhausted; the error is latched
            const long long idx = block_voxel<L>(es, i & 3, j & 3, k & 3);
            uint32_t *mw = &g.mask[idx >> 5];
            const uint32_t bit = 1u << (idx & 31);
            if (!(*(volatile uint32_t *)mw & bit) && !(atomicOr(mw, bit) & bit)) changed = true;
            atomicAdd(fm + idx, pmass * t.x);
            atomicAdd(f0 + idx, pmass * t.y);
            atomicAdd(f1 + idx, pmass * t.z);
            atomicAdd(f2 + idx, pmass * t.w);
        }
        if (last) {
            __syncthreads();
            for (int nd = threadIdx.x; nd < kBinNodes; nd += kBinThreads) {
                int i, j, k, blk, l;
                bin_node(nd, i, j, k, blk, l);
                const int ns = s.sort.slot[blk];  // -1: outside the domain, or pool exhausted (latched)
                if (ns < 0 || !node_hit(s.sort, i, j, k)) continue;
                const float4 t = node_total(s.sort, s.buf, i, j, k);
                atomicOr(&s.sort.bits[2 * blk + (l >> 5)], 1u << (l & 31));
                const long long idx = block_voxel<L>(ns, i & 3, j & 3, k & 3);
                atomicAdd(fm + idx, pmass * t.x);
                atomicAdd(f0 + idx, pmass * t.y);
                atomicAdd(f1 + idx, pmass * t.z);
                atomicAdd(f2 + idx, pmass * t.w);
            }
            __syncthreads();
            if (warp == 0) {
                changed |= set_touched<L>(g, s.sort.slot, s.sort.bits, 8);
                __syncwarp();  // the bin's shared state for the next bin
                if (lane < 16) s.sort.all[lane] = s.sort.bits[lane] = 0;
                if (lane < 8) s.sort.slot[lane] = slot;
            }
            if (!more) break;
            bl += gridDim.x;
            b = nb;
            beg = nbeg;
            end = nend;
            c = 0;
            if (bl + (int)gridDim.x < used) bin_of(bl + gridDim.x, nb, nbeg, nend);
        } else {
            c += parts;
            __syncthreads();  // the records are rewritten by the bin's next chunk
        }
        nch = nnch;
#pragma unroll
        for (int u = 0; u < PPT; ++u) p[u] = pn[u];
    }
    changed |= few();
    if (changed) mark_dirty(g);
}

// CTAs of the gather over these bins, or the error of a device that refuses its
// shared memory.
template <int L, bool APIC>
static cudaError_t gather_ctas(int num_sms, int *ctas)
{
    static std::atomic<int> known[kMaxDevices];
    int per = 0;
    const cudaError_t e = resident_per_sm(k_p2g_gather<L, APIC>, kBinThreads, (int)sizeof(GatherSmem<APIC>), known, &per);
    *ctas = per * num_sms;
    return e;
}

template <int L, bool APIC>
static void launch_gather(const DevGrid &g, cudaStream_t s, int ctas, const float *x, const float *v, const float *C,
                          float pmass, int f_mass, int f_mom0)
{
    launch_chained(k_p2g_gather<L, APIC>, ctas, kBinThreads, sizeof(GatherSmem<APIC>), s, g, x, v, C, pmass, f_mass, f_mom0);
}

// ---------------------------------------------------------------------------
// Particle reordering: the arrays into the order of the last binning, out[q]
// = in[perm[q]] for nc values per particle (a thread per value, so the writes
// are coalesced), then the order itself becomes the identity.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_sort_gather(const int32_t *__restrict__ perm, long long n, int nc, const T *__restrict__ in,
                              T *__restrict__ out)
{
    const long long total = n * nc;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const long long q = e / nc;
        const int c = (int)(e - q * nc);
        out[e] = in[(long long)perm[q] * nc + c];
    }
}

__global__ void k_iota(int32_t *__restrict__ perm, long long n)
{
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        perm[q] = (int32_t)q;
}

int launch_sort_particles(DevGrid &g, cudaStream_t s, float *x, float *v, float *C, int64_t *ids, long long n,
                          void *tmp, const LaunchCfg &lc)
{
    const unsigned blocks = (unsigned)(lc.num_sms * 8);
    int launches = 0;
    struct Arr { void *p; int nc; bool i64; } arrs[4] = {{x, 3, false}, {v, 3, false}, {C, 9, false}, {ids, 1, true}};
    for (const Arr &a : arrs) {
        if (!a.p) continue;
        if (a.i64)
            k_sort_gather<long long><<<blocks, 256, 0, s>>>(g.perm, n, a.nc, (const long long *)a.p, (long long *)tmp);
        else
            k_sort_gather<float><<<blocks, 256, 0, s>>>(g.perm, n, a.nc, (const float *)a.p, (float *)tmp);
        ++launches;
        cudaMemcpyAsync(a.p, tmp, (size_t)n * a.nc * (a.i64 ? 8 : 4), cudaMemcpyDeviceToDevice, s);
    }
    k_iota<<<blocks, 256, 0, s>>>(g.perm, n);
    return launches + 1;
}

int p2g_launches(const DevGrid &g) { return p2g_words(p2g_bins(g.R, g.lg2)) / kBinTile > kMaxOwnTiles ? 7 : 6; }

cudaError_t launch_p2g_binned(DevGrid &g, cudaStream_t s, const float *x, const float *v, const float *C, long long n,
                              float pmass, int f_mass, int f_mom0, bool rebin, const LaunchCfg &lc)
{
    int gctas = 0;
    const cudaError_t e = g.L == 4 ? (C ? gather_ctas<4, true>(lc.num_sms, &gctas) : gather_ctas<4, false>(lc.num_sms, &gctas))
                                   : (C ? gather_ctas<8, true>(lc.num_sms, &gctas) : gather_ctas<8, false>(lc.num_sms, &gctas));
    if (e != cudaSuccess) return e;
    const int ntiles = (int)(p2g_words(p2g_bins(g.R, g.lg2)) / kBinTile), alloc_ctas = alloc_needed_ctas(g);
    const bool scanned = ntiles > kMaxOwnTiles;
    long long pblocks = (n + 255) / 256;
    if (pblocks > 1 << 20) pblocks = 1 << 20;
    launch_chained(k_bin_clear, ntiles, 256, 0, s, g);
    if (rebin) launch_chained(k_p2g_rebin, (unsigned)pblocks, 256, 0, s, g, x, n);
    else launch_chained(k_p2g_bin, (unsigned)pblocks, 256, 0, s, g, x, n);
    launch_chained(k_bin_tiles, ntiles, 256, 0, s, g);
    if (scanned) launch_chained(k_bin_scan_top, 1, 1024, 0, s, g, ntiles);
    launch_chained(k_bin_place, alloc_ctas + ntiles, 256, 0, s, g, alloc_ctas, scanned);
    if (rebin) {
        launch_chained(k_p2g_reperm, (unsigned)pblocks, 256, 0, s, g, n);
        int32_t *t = g.perm;  // the new order is now the current one
        g.perm = g.perm_alt;
        g.perm_alt = t;
    } else {
        launch_chained(k_p2g_perm, (unsigned)pblocks, 256, 0, s, g, n);
    }
    if (g.L == 4) {
        if (C) launch_gather<4, true>(g, s, gctas, x, v, C, pmass, f_mass, f_mom0);
        else launch_gather<4, false>(g, s, gctas, x, v, C, pmass, f_mass, f_mom0);
    } else {
        if (C) launch_gather<8, true>(g, s, gctas, x, v, C, pmass, f_mass, f_mom0);
        else launch_gather<8, false>(g, s, gctas, x, v, C, pmass, f_mass, f_mom0);
    }
    std::swap(g.perm, g.perm_alt);  // the gather's cell order
    return cudaSuccess;
}

}  // namespace sg

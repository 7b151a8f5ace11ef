// sg_g2p2g.cu -- fused G2P2G (AsyncTaichi Sec. 8.3: the G2P of one step and
// the P2G of the next fused into one pass over the particles, with the affine
// matrix C of the MLS-MPM transfers eliminated as a dead store).
//
// One launch computes, for every particle p, exactly what
//   APIC G2P from grid `src`   (v_p, C_p, x_p += dt v_p)
//   APIC P2G into grid `dst`   (activation of the 27 stencil nodes of the new
//                               position, mass and affine momentum)
// compute one after the other, but C_p lives only in registers and shared
// memory: it is never written to or read from HBM.  x_p and v_p are written
// back (they are the particle state); the update is in place, each particle
// being visited once.
//
// Work split: one CTA per bin of the last binned P2G over these particles (a
// 4^3 block of nodes from o with the particles whose base node was in it when
// binned).
//   1. stage src's velocities of nodes o-1 .. o+6 in shared memory;
//   2. per particle: G2P from the staged block, store x', v'; count it in its
//      new base cell and store its P2G record of the new position;
//   3. counting sort by new base cell;
//   4. sums by columns of cells, as in the binned P2G (bin_columns);
//   5. flush the touched nodes o .. o+5: the dst leaves they fall in are
//      allocated in-kernel if null (see ensure_leaf), bits set, 4 FP32 atomics
//      per node.
// A particle whose old base has left [o-1, o+4], and every particle of the
// out-of-domain bin, goes node by node through the two grids; one whose new
// base has left the bin's cells is scattered into dst by a warp, with the same
// in-kernel allocation.
#include "sg_particle.cuh"

namespace sg {

namespace {

constexpr int kRootPending = -2;  // a CTA is allocating this leaf
constexpr int kRootFailed = -3;   // allocation failed (pool exhausted)

// Self-checks of the kernel's own accesses: every vector access below first
// verifies the alignment of its address (and the shared-record loop its
// range); a failed check skips the access, latches kErrCheck on dst and
// records which check failed.  They cost a few integer operations per access.
__device__ __forceinline__ bool misaligned(const DevGrid &g, const void *p, unsigned align, int site)
{
    if (((uintptr_t)p & (uintptr_t)(align - 1)) == 0) return false;
    atomicOr(&g.ctrl->err, kErrCheck);
    g.ctrl->timeout_site = 100 + site;
    return true;
}

// Slot of leaf cell lb of g, allocating and zero-filling it if null.  The
// first thread to swap -1 for kRootPending takes a pool slot, zeroes its
// fields and mask, and publishes the slot; others wait for the publication
// (the allocating thread runs and waits on nothing, so the wait ends; it is
// bounded all the same and records kErrTimeout if it gives up).  Returns -1
// when the pool is exhausted (kErrPool latched).  *fresh is set when this
// thread allocated the leaf.
__device__ __forceinline__ int ensure_leaf(const DevGrid &g, long long lb, bool &fresh)
{
    volatile int32_t *r = g.root + lb;
    int s = *r;
    if (s >= 0) return s;
    if (s == -1 && atomicCAS(g.root + lb, -1, kRootPending) == -1) {
        const int slot = atomicAdd(&g.ctrl->pool_count, 1);
        if (slot >= g.cap) {
            raise_error(g, kErrPool);
            __threadfence();
            atomicExch(g.root + lb, kRootFailed);
            return -1;
        }
        const int V = g.L * g.L * g.L;
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int f = 0; f < g.F; ++f) {
            float4 *p = reinterpret_cast<float4 *>(g.field[f] + (long long)slot * V);
            if (misaligned(g, p, 16, 3)) {
                for (int q = 0; q < V; ++q) g.field[f][(long long)slot * V + q] = 0.f;
                continue;
            }
            for (int q = 0; q < V / 4; ++q) p[q] = z;
        }
        for (int w = 0; w < g.W; ++w) g.mask[(long long)slot * g.W + w] = 0u;
        __threadfence();
        atomicExch(g.root + lb, slot);
        fresh = true;
        return slot;
    }
    const unsigned long long t0 = global_timer_ns();
    while ((s = *r) == kRootPending) {
        if (global_timer_ns() - t0 > 1000000000ull) {
            raise_error(g, kErrTimeout);
            g.ctrl->timeout_site = 3;
            return -1;
        }
        __nanosleep(100);
    }
    __threadfence();
    return s >= 0 ? s : -1;
}

// Activate node (i, j, k) of g and add (m, p0, p1, p2) to it; the node is in
// the domain.  Returns whether the structure changed.
__device__ __forceinline__ bool scatter_node(const DevGrid &g, int i, int j, int k, float m, float p0, float p1,
                                             float p2, int f_mass, int f_mom0)
{
    const int L = g.L, lg2 = g.lg2;
    bool fresh = false;
    const int slot = ensure_leaf(g, ((long long)(i >> lg2) * g.R + (j >> lg2)) * g.R + (k >> lg2), fresh);
    if (slot < 0) return fresh;
    const int l = (((i & (L - 1)) << lg2) + (j & (L - 1))) * L + (k & (L - 1));
    uint32_t *mw = &g.mask[(long long)slot * g.W + (l >> 5)];
    const uint32_t bit = 1u << (l & 31);
    bool changed = fresh;
    if (!(*(volatile uint32_t *)mw & bit)) changed |= !(atomicOr(mw, bit) & bit);
    const long long idx = ((long long)slot << (3 * lg2)) + l;
    atomicAdd(g.field[f_mass] + idx, m);
    atomicAdd(g.field[f_mom0] + idx, p0);
    atomicAdd(g.field[f_mom0 + 1] + idx, p1);
    atomicAdd(g.field[f_mom0 + 2] + idx, p2);
    return changed;
}

// P2G record of one particle: spline offsets and mass, q = m v - m dx C fx,
// and the 9 entries of m dx C (row-major).
struct P2GRec {
    float4 r0, r1, r2, r3;
};

__device__ __forceinline__ P2GRec make_rec(float fx, float fy, float fz, float pmass, float3 u, const float (&c)[9],
                                           float dx)
{
    float m[9];
    const float md = pmass * dx;
#pragma unroll
    for (int e = 0; e < 9; ++e) m[e] = md * c[e];
    const float q0 = pmass * u.x - (m[0] * fx + m[1] * fy + m[2] * fz);
    const float q1 = pmass * u.y - (m[3] * fx + m[4] * fy + m[5] * fz);
    const float q2 = pmass * u.z - (m[6] * fx + m[7] * fy + m[8] * fz);
    P2GRec r;
    r.r0 = make_float4(fx, fy, fz, pmass);
    r.r1 = make_float4(q0, q1, q2, m[0]);
    r.r2 = make_float4(m[1], m[2], m[3], m[4]);
    r.r3 = make_float4(m[5], m[6], m[7], m[8]);
    return r;
}

// Node-by-node APIC P2G of one particle into g (slow path).
__device__ __forceinline__ bool scatter_particle(const DevGrid &g, Spline sx, Spline sy, Spline sz, P2GRec r,
                                                 int f_mass, int f_mom0)
{
    bool changed = false;
    const int N = g.N;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int i = sx.base + a;
        if ((unsigned)i >= (unsigned)N) continue;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int j = sy.base + b;
            if ((unsigned)j >= (unsigned)N) continue;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int k = sz.base + c;
                if ((unsigned)k >= (unsigned)N) continue;
                const float w = sx.w[a] * sy.w[b] * sz.w[c];
                const float ta = (float)a, tb = (float)b, tc = (float)c;
                const float u0 = fmaf(r.r1.w, ta, fmaf(r.r2.x, tb, fmaf(r.r2.y, tc, r.r1.x)));
                const float u1 = fmaf(r.r2.z, ta, fmaf(r.r2.w, tb, fmaf(r.r3.x, tc, r.r1.y)));
                const float u2 = fmaf(r.r3.y, ta, fmaf(r.r3.z, tb, fmaf(r.r3.w, tc, r.r1.z)));
                changed |= scatter_node(g, i, j, k, w * r.r0.w, w * u0, w * u1, w * u2, f_mass, f_mom0);
            }
        }
    }
    return changed;
}

// ---------------------------------------------------------------------------
// The next chunk's positions come into shared memory while a chunk is worked
// on.  A bin of several chunks deals its particles to them in turn, so each
// chunk has its share of every column whatever the order.  A whole bin of the
// usual ten particles a cell is one chunk of 736: in chunks of 384 the columns
// are shorter and the three of a warp less even (238 us).  2M particles over
// 4^3 leaves: 220 us a launch at two CTAs per SM without spills (256 threads
// and a warp per cell: 308 us; this one at three CTAs and 96 registers,
// spilling: 264 us).
// ---------------------------------------------------------------------------
struct G2P2GSmem {
    static constexpr int PPT = 4, CAP = 736;
    float4 rec[4][CAP];
    float4 buf[kBinBuf];
    float4 u[512];                  // src velocities of nodes o - 1 .. o + 6
    float x[3 * CAP];               // the next chunk's positions, in order
    float words[kBinWarps][96];
    int uslot[27];                  // src blocks o / 4 + {-1, 0, 1}^3
    uint16_t idx[CAP + 2];
    BinSort sort;
};

// One particle node by node: its G2P from src, its state, its P2G into dst.
// Returns whether dst's structure changed.
__device__ __noinline__ bool far_particle(const DevGrid &src, const DevGrid &dst, float *x, float *v, long long p,
                                          float dt, int f_vel0, float pmass, int f_mass, int f_mom0)
{
    const float x0 = x[3 * p], x1 = x[3 * p + 1], x2 = x[3 * p + 2];
    float3 u;
    float c[9];
    g2p_from_grid<true>(src, src.field[f_vel0], src.field[f_vel0 + 1], src.field[f_vel0 + 2], bspline(x0, src.N),
                        bspline(x1, src.N), bspline(x2, src.N), u, c);
    const float n0 = x0 + dt * u.x, n1 = x1 + dt * u.y, n2 = x2 + dt * u.z;
    v[3 * p] = u.x;
    v[3 * p + 1] = u.y;
    v[3 * p + 2] = u.z;
    x[3 * p] = n0;
    x[3 * p + 1] = n1;
    x[3 * p + 2] = n2;
    const Spline nx = bspline(n0, dst.N), ny = bspline(n1, dst.N), nz = bspline(n2, dst.N);
    return scatter_particle(dst, nx, ny, nz, make_rec(nx.fx, ny.fx, nz.fx, pmass, u, c, 1.f / (float)dst.N), f_mass, f_mom0);
}
constexpr int kFar = -2;

template <int L>
__global__ void __launch_bounds__(kBinThreads, 2) k_g2p2g(const __grid_constant__ DevGrid src,
                                                          const __grid_constant__ DevGrid dst,
                                                          const int32_t *bin_list, const int32_t *bin_off,
                                                          const int32_t *bin_end, const int32_t *perm,
                                                          const int32_t *bins_used, float *x, float *v, float dt,
                                                          int f_vel0, float pmass, int f_mass, int f_mom0)
{
    chained_entry();
    using S = G2P2GSmem;
    constexpr int PPT = S::PPT, CAP = S::CAP;
    extern __shared__ __align__(16) unsigned char smem[];
    S &s = *reinterpret_cast<S *>(smem);
    if (threadIdx.x == 0) misaligned(dst, smem, 16, 4);
    const int N = src.N, R = src.R;
    const float dx = 1.f / (float)N;
    const int warp = threadIdx.x >> 5, lane = lane_id();
    float *words = s.words[warp];
    const float *u0p = src.field[f_vel0], *u1p = src.field[f_vel0 + 1], *u2p = src.field[f_vel0 + 2];
    bool changed = false;
    const int used = *bins_used;
    // particles whose stencil missed the domain when they were binned
    {
        const int oob_bin = (int)p2g_bins(R, L == 8 ? 3 : 2);
        const int end = bin_end[oob_bin];
        for (int q = bin_off[oob_bin] + blockIdx.x * kBinThreads + threadIdx.x; q < end; q += gridDim.x * kBinThreads) {
            changed |= far_particle(src, dst, x, v, perm[q], dt, f_vel0, pmass, f_mass, f_mom0);
        }
    }
    int bl = blockIdx.x;
    if (bl < used) {
        auto bin_of = [&](int l, int &b, int &beg, int &end) {
            b = bin_list[l];
            beg = bin_off[b];
            end = bin_end[b];
        };
        // slot of src's block o / 4 + {-1, 0, 1}^3 (threads 0 .. 26), negative: none
        auto near_slot = [&](int b) {
            const int t = threadIdx.x;
            if (t >= 27) return -1;
            int bi, bj, bk;
            bin_block<L>(b, R, bi, bj, bk);
            return block_slot<L>(src.root, R, bi + t / 9 - 1, bj + (t / 3) % 3 - 1, bk + t % 3 - 1);
        };
        // chunk c of nch takes particles beg + c, beg + c + nch, ...
        auto order = [&](int beg, int end, int c, int nch, int (&p)[PPT]) {
#pragma unroll
            for (int u = 0; u < PPT; ++u) {
                const long long q = beg + c + (long long)((u * kBinWarps + warp) * 32 + lane) * nch;
                p[u] = q < end ? perm[q] : -1;
            }
        };
        auto request = [&](const int (&p)[PPT]) {
#pragma unroll
            for (int u = 0; u < PPT; ++u) {
                const int q0 = (u * kBinWarps + warp) * 32;
                if (__any_sync(kFull, p[u] >= 0)) {
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const int e = r * 32 + lane, w = e / 3, q = __shfl_sync(kFull, p[u], w);
                        if (q >= 0) copy_word(s.x + 3 * q0 + e, x + 3LL * q + (e - 3 * w));
                    }
                }
            }
        };
        int b, beg, end, nb = 0, nbeg = 0, nend = 0;
        bin_of(bl, b, beg, end);
        int slot = near_slot(b), c = 0, nch = (end - beg + CAP - 1) / CAP;
        int p[PPT], pn[PPT];
        order(beg, end, 0, nch, p);
        request(p);
        if (bl + (int)gridDim.x < used) bin_of(bl + gridDim.x, nb, nbeg, nend);
        if (threadIdx.x < 65) s.sort.cnt[threadIdx.x] = 0;
        if (threadIdx.x < 16) s.sort.all[threadIdx.x] = s.sort.bits[threadIdx.x] = 0;
        if (threadIdx.x < 27) s.uslot[threadIdx.x] = slot;
        __syncthreads();
        for (;;) {
            const bool last = c + 1 >= nch, more = !last || bl + (int)gridDim.x < used;
            const int nnch = last ? (nend - nbeg + CAP - 1) / CAP : nch;
            if (more) order(last ? nbeg : beg, last ? nend : end, last ? 0 : c + 1, nnch, pn);
            if (last && more) slot = near_slot(nb);
            int bi, bj, bk;
            bin_block<L>(b, R, bi, bj, bk);
            const int oi = bi * 4, oj = bj * 4, ok = bk * 4;
            if (c == 0) {  // src's node velocities, 0 outside the domain or the leaves
                for (int nd = threadIdx.x; nd < 512; nd += kBinThreads) {
                    const int i = (nd >> 6) + 3, j = ((nd >> 3) & 7) + 3, k = (nd & 7) + 3;  // from o - 4
                    const int us = s.uslot[(i >> 2) * 9 + (j >> 2) * 3 + (k >> 2)];
                    float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (us >= 0) {
                        const long long idx = block_voxel<L>(us, i & 3, j & 3, k & 3);
                        u = make_float4(u0p[idx], u1p[idx], u2p[idx], 0.f);
                    }
                    s.u[nd] = u;
                }
                __syncthreads();
            }
            copies_done();
            __syncwarp();
            // G2P, the particle's record of its new position, its cell and its
            // rank among the cell's particles
            int place[PPT] = {-1, -1, -1, -1};
#pragma unroll 1
            for (int u = 0; u < PPT; ++u) {
                const int pu = u < 2 ? (u ? p[1] : p[0]) : (u == 2 ? p[2] : p[3]);
                int pl = -1;
                if (!__any_sync(kFull, pu >= 0)) break;  // warp-uniform
                const int q = (u * kBinWarps + warp) * 32 + lane;
                const float x0 = s.x[3 * q], x1 = s.x[3 * q + 1], x2 = s.x[3 * q + 2];
                float xn[3] = {0.f, 0.f, 0.f}, vn[3] = {0.f, 0.f, 0.f};
                if (pu >= 0) {
                    const Spline ox = bspline(x0, N), oy = bspline(x1, N), oz = bspline(x2, N);
                    const int ri = ox.base - oi + 1, rj = oy.base - oj + 1, rk = oz.base - ok + 1;
                    pl = kFar;
                    if ((unsigned)ri <= 5u && (unsigned)rj <= 5u && (unsigned)rk <= 5u) {
                        float3 uu;
                        float C[9];
                        g2p_from_block<8, true>(s.u, ri, rj, rk, N, ox, oy, oz, uu, C);
                        vn[0] = uu.x;
                        vn[1] = uu.y;
                        vn[2] = uu.z;
                        xn[0] = x0 + dt * uu.x;
                        xn[1] = x1 + dt * uu.y;
                        xn[2] = x2 + dt * uu.z;
                        const Spline nx = bspline(xn[0], N), ny = bspline(xn[1], N), nz = bspline(xn[2], N);
                        const int ci = nx.base - oi, cj = ny.base - oj, ck = nz.base - ok;
                        if ((unsigned)(ci + 500) <= 1000u && (unsigned)(cj + 500) <= 1000u && (unsigned)(ck + 500) <= 1000u) {
                            const bool in = (unsigned)ci < 4u && (unsigned)cj < 4u && (unsigned)ck < 4u;
                            const int cell = in ? (ci * 4 + cj) * 4 + ck : 64;
                            pl = cell | atomicAdd(&s.sort.cnt[cell], 1) << 7;
                            bin_record<true, CAP>(s.rec, q, nx.fx, ny.fx, nz.fx, uu.x, uu.y, uu.z, C, dx, !in,
                                                  pack_cell(ci, cj, ck));
                        }
                    }
                }
                const int to = pl >= 0 ? pu : -1;  // the far ones are done below
                __syncwarp();
                warp_put<3>(v, to, vn, words);
                warp_put<3>(x, to, xn, words);
#pragma unroll
                for (int w = 0; w < PPT; ++w)
                    if (u == w) place[w] = pl;
            }
            __syncthreads();
            if (warp == 0) bin_scan(s.sort);
            __syncthreads();
#pragma unroll
            for (int u = 0; u < PPT; ++u)
                if (place[u] >= 0)
                    s.idx[s.sort.start[place[u] & 127] + (place[u] >> 7)] = (uint16_t)((u * kBinWarps + warp) * 32 + lane);
            __syncthreads();
            if (more) request(pn);
            bin_columns<true, CAP>(s.rec, s.idx, s.sort, s.buf);
            for (int pp = s.sort.start[64] + warp; pp < s.sort.start[65] && pp < CAP; pp += kBinWarps) {
                int i, j, k;
                float4 t;
                if (edge_node<true, CAP>(s.rec, s.idx[pp], oi, oj, ok, N, i, j, k, t))
                    changed |= scatter_node(dst, i, j, k, pmass * t.x, pmass * t.y, pmass * t.z, pmass * t.w, f_mass, f_mom0);
            }
#pragma unroll
            for (int u = 0; u < PPT; ++u)
                if (place[u] == kFar) changed |= far_particle(src, dst, x, v, p[u], dt, f_vel0, pmass, f_mass, f_mom0);
            if (last) {
                __syncthreads();
                // the touched nodes' sums, then the dst leaves that hold them
                float4 t[2];
                int where[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int nd = threadIdx.x + h * kBinThreads;
                    where[h] = -1;
                    if (nd >= kBinNodes) continue;
                    int i, j, k, blk, l;
                    bin_node(nd, i, j, k, blk, l);
                    if (oi + i >= N || oj + j >= N || ok + k >= N || !node_hit(s.sort, i, j, k)) continue;
                    t[h] = node_total(s.sort, s.buf, i, j, k);
                    where[h] = blk << 6 | l;
                    atomicOr(&s.sort.bits[2 * blk + (l >> 5)], 1u << (l & 31));
                }
                __syncthreads();
                if (warp == 0) {
                    if (lane < 8) {
                        const int ci = bi + (lane >> 2), cj = bj + ((lane >> 1) & 1), ck = bk + (lane & 1);
                        int ds = -1;
                        if (s.sort.bits[2 * lane] | s.sort.bits[2 * lane + 1]) {
                            bool fresh = false;
                            ds = block_of_leaf<L>(ensure_leaf(dst, block_leaf<L>(R, ci, cj, ck), fresh), ci, cj, ck);
                            changed |= fresh;
                        }
                        s.sort.slot[lane] = ds;
                    }
                    __syncwarp();
                    changed |= set_touched<L>(dst, s.sort);
                    if (lane < 27) s.uslot[lane] = slot;
                }
                __syncthreads();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (where[h] < 0) continue;
                    const int ds = s.sort.slot[where[h] >> 6];
                    if (ds < 0) continue;  // pool exhausted; the error is latched
                    const int l = where[h] & 63;
                    const long long idx = block_voxel<L>(ds, l >> 4, l >> 2 & 3, l & 3);
                    atomicAdd(dst.field[f_mass] + idx, pmass * t[h].x);
                    atomicAdd(dst.field[f_mom0] + idx, pmass * t[h].y);
                    atomicAdd(dst.field[f_mom0 + 1] + idx, pmass * t[h].z);
                    atomicAdd(dst.field[f_mom0 + 2] + idx, pmass * t[h].w);
                }
                __syncthreads();
                if (threadIdx.x < 16) s.sort.all[threadIdx.x] = s.sort.bits[threadIdx.x] = 0;
                if (!more) break;
                bl += gridDim.x;
                b = nb;
                beg = nbeg;
                end = nend;
                c = 0;
                if (bl + (int)gridDim.x < used) bin_of(bl + gridDim.x, nb, nbeg, nend);
            } else {
                ++c;
                __syncthreads();  // the records are rewritten by the bin's next chunk
            }
            nch = nnch;
#pragma unroll
            for (int u = 0; u < PPT; ++u) p[u] = pn[u];
        }
    }
    if (changed) mark_dirty(dst);
}

template <int L>
cudaError_t launch_g2p2g_L(const DevGrid &src, const DevGrid &dst, const DevGrid &bins, cudaStream_t s, float *x,
                           float *v, float dt, int f_vel0, float pmass, int f_mass, int f_mom0, int num_sms)
{
    constexpr int bytes = (int)sizeof(G2P2GSmem);
    static std::atomic<int> known[kMaxDevices];
    int per = 0;
    const cudaError_t e = resident_per_sm(k_g2p2g<L>, kBinThreads, bytes, known, &per);
    if (e != cudaSuccess) return e;
    launch_chained(k_g2p2g<L>, per * num_sms, kBinThreads, bytes, s, src, dst, bins.bin_list, bins.bin_off, bins.bin_count,
                   bins.perm, &bins.ctrl->bins_used, x, v, dt, f_vel0, pmass, f_mass, f_mom0);
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_g2p2g(const DevGrid &src, const DevGrid &dst, const DevGrid &bins, cudaStream_t s, float *x, float *v,
                         long long n, float dt, int f_vel0, float pmass, int f_mass, int f_mom0, const LaunchCfg &lc)
{
    if (n <= 0) return cudaSuccess;
    if (dst.L == 4) return launch_g2p2g_L<4>(src, dst, bins, s, x, v, dt, f_vel0, pmass, f_mass, f_mom0, lc.num_sms);
    return launch_g2p2g_L<8>(src, dst, bins, s, x, v, dt, f_vel0, pmass, f_mass, f_mom0, lc.num_sms);
}

}  // namespace sg

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
// binned); bins far emptier or fuller than a chunk as bin_split says.
//   1. stage src's velocities of nodes o-1 .. o+6 in shared memory;
//   2. per particle: G2P from the staged block, store x', v'; count it in its
//      new base cell and store its P2G record of the new position;
//   3. counting sort by new base cell;
//   4. sums by columns of cells, as in the binned P2G (bin_columns), over the
//      bin's own cells or, once many particles have moved there, those around;
//   5. flush the touched nodes o .. o+5 (o-1 .. o+6): the dst leaves they fall
//      in are allocated in-kernel if null (see ensure_leaf), bits set, 4 FP32
//      atomics per node.
// A particle whose old base has left [o-1, o+4], and every particle of the
// out-of-domain bin, goes node by node through the two grids; one whose new
// base is further out than those cells is scattered into dst by a warp, with
// the same in-kernel allocation.
#include <type_traits>
#include "sg_particle.cuh"

namespace sg {

namespace {

constexpr int kRootPending = -2;  // a CTA is allocating this leaf
constexpr int kRootFailed = -3;   // allocation failed (pool exhausted)

// Self-checks of the kernel's own accesses; a failed one latches kErrCheck on
// dst and records which it was (misaligned: also sort_fits, sg_particle.cuh).
// Site 3: a new leaf's fields are zeroed in 16-byte stores, or, if not so
// aligned, word by word.  Site 4: the base of the shared memory, whose records
// move in 16-byte words (reported only: nothing could be done without it).
__device__ __forceinline__ bool misaligned(const DevGrid &g, const void *p, unsigned align, int site)
{
    if (((uintptr_t)p & (uintptr_t)(align - 1)) == 0) return false;
    raise_check(g, site);
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

// ---------------------------------------------------------------------------
// Sorting and summing of a chunk's new positions, in two forms.  Particles move
// on from step to step and one binning serves many, so at first nearly all are
// in their bin's own 4^3 cells and later many are not.
//   k_g2p2g<L, false>  BinSort and bin_columns, as the binned P2G: a particle
//                      outside the own cells is added to dst by a warp.
//   k_g2p2g<L, true>   MovedSort: cells 0 .. 63 are the bin's own, 64 .. 215 the
//                      152 around them (base o - 1 .. o + 4), 216 holds what has
//                      gone further.  Up to kFewMoved particles in the cells
//                      around, they are added to dst by a warp each, like those
//                      of 216; with more, the chunk is summed by 36 columns of
//                      six cells, the bin's own 16 and then the 20 around them,
//                      onto the 8^3 nodes o - 1 .. o + 6.
// Each launch counts the particles that it finds outside the own cells; from the
// next launch over the same binning on, the second form runs if they were more
// than one in kMovedShare and the bins hold more than kMovedBin each on average.
// Both are launched and the other returns at once.  2M particles, 10 a cell, that
// have moved by 0 / 0.03 / 0.1 / 0.25 / 1 cell since the binning: the first form
// takes 232 / 272 / 344 / 459 / 941 us, the second (more shared memory, less L1)
// 257 / 302 / 342 / 349 / 347.  200k, 3 a cell (192 a bin), moved by 0.25 / 1:
// 103 / 156 and 107 / 106 us; one a cell (64 a bin): 174 / 233 and 239 / 287.
// ---------------------------------------------------------------------------
constexpr int kMovedShare = 16, kMovedBin = 128;
constexpr int kOwnCells = 64, kFarCell = 216, kFewMoved = 24;
constexpr int kMovedBuf = 36 * 9 * 8;  // float4 [column][lane][node]

struct MovedSort {
    int cnt[kFarCell + 1];    // particles per cell; zero between chunks
    int start[224];           // their places in idx
    uint32_t prev[36], all[36];  // nodes reached by each column's particles (6 x 6, of six cells), before / after this chunk
    int slot[8 + 27];         // blocks o / 4 + {0, 1}^3 and, for moved particles, o / 4 + {-1, 0, 1}^3
    uint32_t bits[2 * (8 + 27)]; // touched nodes of those blocks, i, j, k in order
    int moved;                // this chunk is summed by the 36 columns
    int outer;                // a chunk of this bin was
};

// Cell (i, j, k), each 0 .. 5 from o - 1.
__device__ __forceinline__ int moved_cell(int i, int j, int k)
{
    if ((unsigned)(i - 1) < 4u && (unsigned)(j - 1) < 4u) {
        if ((unsigned)(k - 1) < 4u) return ((i - 1) * 4 + j - 1) * 4 + k - 1;
        return kOwnCells + (k == 0 ? 120 : 136) + (i - 1) * 4 + j - 1;
    }
    return kOwnCells + ((unsigned)(i - 1) < 4u ? (j == 0 ? 72 : 96) + (i - 1) * 6 + k : (i == 0 ? 0 : 36) + j * 6 + k);
}

// Exclusive scan of the cell counts (one warp), which it zeroes; cap: the most
// that there can be.
__device__ __forceinline__ void moved_scan(const DevGrid &g, MovedSort &s, int cap)
{
    constexpr int PER = 7;  // 32 x 7 >= 217; an odd stride has no bank conflicts
    const int lane = lane_id();
    int c[PER], tot = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int cell = PER * lane + q;
        c[q] = cell <= kFarCell ? s.cnt[cell] : 0;
        tot += c[q];
        if (cell <= kFarCell) s.cnt[cell] = 0;
    }
    int run = warp_incl_scan(tot) - tot;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        s.start[PER * lane + q] = run;  // start[217 ..]: the end
        run += c[q];
    }
    __syncwarp();
    const bool moved = s.start[kFarCell] - s.start[kOwnCells] > kFewMoved;
    if (lane == 0) {
        sort_fits(g, s.start[kFarCell + 1], cap, 6);
        s.moved = moved;
        if (moved) s.outer = 1;
    }
    for (int col = lane; col < 36; col += 32) {
        const int i = col / 6, j = col - 6 * i;
        const bool own = (unsigned)(i - 1) < 4u && (unsigned)(j - 1) < 4u;
        uint32_t now = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k)
            if (moved || (own && (unsigned)(k - 1) < 4u)) {
                const int cell = moved_cell(i, j, k);
                if (s.start[cell + 1] > s.start[cell]) now |= 7u << k;
            }
        const uint32_t before = s.all[col];
        s.prev[col] = before;
        s.all[col] = before | now;
    }
}

// Column sums as in bin_columns, of a chunk whose particles stayed in the bin's
// own cells (but for the few that go by a warp each).
template <int CAP>
__device__ __forceinline__ void own_columns(const float4 (*rec)[CAP], const uint16_t *idx, const MovedSort &s, float4 *s_buf)
{
    const int lane = lane_id(), grp = lane / 9, sub = lane - 9 * grp;
    const int own = (threadIdx.x >> 5) * 3 + grp;
    if (grp > 2 || own > 15) return;
    int pp = s.start[4 * own];
    const int last = s.start[4 * own + 4];
    if (pp >= last || last > CAP) return;
    const int a = sub / 3, b = sub - 3 * a, col = ((own >> 2) + 1) * 6 + (own & 3) + 1;
    const BsPoly pa = bs_poly(a), pb = bs_poly(b);
    const uint32_t add = s.prev[col];  // nodes with sums of an earlier chunk
    float4 *out = s_buf + (col * 9 + sub) * 8 + 1;
    float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f), n1 = n0, n2 = n0;
    auto store = [&](int k, float4 n) {
        if (add >> (k + 1) & 1u) {
            const float4 o = out[k];
            n = make_float4(o.x + n.x, o.y + n.y, o.z + n.z, o.w + n.w);
        }
        out[k] = n;
    };
    int next = idx[pp];
#pragma unroll 1
    for (int ck = 0; ck < 4; ++ck) {
        const int end = s.start[4 * own + ck + 1];
        while (pp < end) {
            const int q = next;
            next = idx[++pp];
            column_add<true, CAP>(rec, q, pa, pb, (float)a, (float)b, n0, n1, n2);
        }
        store(ck, n0);
        n0 = n1;
        n1 = n2;
        n2 = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    store(4, n0);
    store(5, n1);
}

// The same over the 36 columns.
template <int CAP>
__device__ __noinline__ void moved_columns(const float4 (*rec)[CAP], const uint16_t *idx, const MovedSort &s, float4 *s_buf)
{
    const int lane = lane_id(), grp = lane / 9, sub = lane - 9 * grp;
    if (grp > 2 || s.start[kFarCell + 1] > CAP) return;
    const int a = sub / 3, b = sub - 3 * a;
    const BsPoly pa = bs_poly(a), pb = bs_poly(b);
#pragma unroll 1
    for (int c = (threadIdx.x >> 5) * 3 + grp; c < 36; c += 18) {
        // the bin's own 16 first, then the rows and the columns around them
        const int col = c < 16 ? ((c >> 2) + 1) * 6 + (c & 3) + 1
                        : c < 22 ? c - 16 : c < 28 ? c + 8 : c < 32 ? (c - 27) * 6 : (c - 31) * 6 + 5;
        const int i = col / 6, j = col - 6 * i;
        const uint32_t add = s.prev[col];
        float4 *out = s_buf + (col * 9 + sub) * 8;
        float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f), n1 = n0, n2 = n0;
        auto store = [&](int k, float4 n) {
            if (add >> k & 1u) {
                const float4 o = out[k];
                n = make_float4(o.x + n.x, o.y + n.y, o.z + n.z, o.w + n.w);
            }
            out[k] = n;
        };
        if (!s.all[col]) continue;
#pragma unroll 1
        for (int k = 0; k < 6; ++k) {
            const int cell = moved_cell(i, j, k), end = s.start[cell + 1];
            for (int pp = s.start[cell]; pp < end; ++pp)
                column_add<true, CAP>(rec, idx[pp], pa, pb, (float)a, (float)b, n0, n1, n2);
            store(k, n0);
            n0 = n1;
            n1 = n2;
            n2 = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        store(6, n0);
        store(7, n1);
    }
}

// Does any summed particle's stencil hold node (i, j, k) (0 .. 7 from o - 1)?
__device__ __forceinline__ bool moved_hit(const MovedSort &s, int i, int j, int k)
{
    uint32_t m = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            if ((unsigned)(i - a) < 6u && (unsigned)(j - b) < 6u) m |= s.all[(i - a) * 6 + (j - b)];
    return (m >> k & 1u) != 0u;
}

// Its sums over the columns that reach it.
__device__ __forceinline__ float4 moved_total(const MovedSort &s, const float4 *s_buf, int i, int j, int k)
{
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int ci = i - a, cj = j - b, col = ci * 6 + cj;
            if ((unsigned)ci >= 6u || (unsigned)cj >= 6u || !(s.all[col] >> k & 1u)) continue;
            const float4 v = s_buf[(col * 9 + a * 3 + b) * 8 + k];
            t.x += v.x;
            t.y += v.y;
            t.z += v.z;
            t.w += v.w;
        }
    return t;
}

// One record by a warp (cell: pack_cell's word): lane (a, b, c) < 27 forms the
// contribution of its node base + (a, b, c); false for lanes without a node in
// the domain.  t: weight and weighted velocity.
template <int CAP>
__device__ __forceinline__ bool single_node(const float4 (*rec)[CAP], int q, int cell, int oi, int oj, int ok, int N, int &i,
                                            int &j, int &k, float4 &t)
{
    const int lane = lane_id(), a = lane / 9, b = (lane / 3) % 3, c = lane % 3;
    if (lane >= 27) return false;
    i = oi + (cell >> 20) - 512 + a;
    j = oj + ((cell >> 10) & 1023) - 512 + b;
    k = ok + (cell & 1023) - 512 + c;
    if ((unsigned)i >= (unsigned)N || (unsigned)j >= (unsigned)N || (unsigned)k >= (unsigned)N) return false;
    const float4 r0 = rec[0][q], r1 = rec[1][q], r2 = rec[2][q], r3 = rec[3][q];
    const float w = bs_eval(bs_poly(a), r0.x) * bs_eval(bs_poly(b), r0.y) *
                    (c == 0 ? r0.z : c == 1 ? (1.f - r0.z) - r0.w : r0.w);
    const float ta = (float)a, tb = (float)b, tc = (float)c;
    t = make_float4(w, w * fmaf(r1.w, ta, fmaf(r2.x, tb, fmaf(r2.y, tc, r1.x))),
                    w * fmaf(r2.z, ta, fmaf(r2.w, tb, fmaf(r3.x, tc, r1.y))),
                    w * fmaf(r3.y, ta, fmaf(r3.z, tb, fmaf(r3.w, tc, r1.z))));
    return true;
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
template <bool AROUND>
struct G2P2GSmem {
    static constexpr int PPT = 4, CAP = 736;
    float4 rec[4][CAP];
    float4 buf[AROUND ? kMovedBuf : kBinBuf];
    float4 u[512];                  // src velocities of nodes o - 1 .. o + 6
    float x[3 * CAP];               // the next chunk's positions, in order
    float words[kBinWarps][96];
    int uslot[27];                  // src blocks o / 4 + {-1, 0, 1}^3
    uint16_t idx[CAP + 2];
    int cell[AROUND ? CAP : 1];     // pack_cell of the records outside the bin's own cells
    std::conditional_t<AROUND, MovedSort, BinSort> sort;
};

// One particle by a warp, node by node: its G2P from src, its state, its P2G
// into dst.  Returns whether dst's structure changed.
template <int L>
__device__ __noinline__ bool far_particle(const DevGrid &src, const DevGrid &dst, float *x, float *v, long long p, float dt,
                                          int f_vel0, float pmass, int f_mass, int f_mom0)
{
    const int lane = lane_id(), a = lane / 9, b = (lane / 3) % 3, c = lane % 3, N = dst.N;
    float xp[3], u[3], C[9];
#pragma unroll
    for (int e = 0; e < 3; ++e) xp[e] = x[3 * p + e];
    g2p_by_warp<L, true>(src, src.field[f_vel0], src.field[f_vel0 + 1], src.field[f_vel0 + 2], xp[0], xp[1], xp[2], u, C);
#pragma unroll
    for (int e = 0; e < 3; ++e) xp[e] += dt * u[e];
    __syncwarp();
    if (lane == 0) {
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            v[3 * p + e] = u[e];
            x[3 * p + e] = xp[e];
        }
    }
    FewParticle<true> r;
    few_particle<true>(r, xp[0], xp[1], xp[2], u, C, N);
    const int i = r.b[0] + a, j = r.b[1] + b, k = r.b[2] + c;
    if (lane >= 27 || (unsigned)i >= (unsigned)N || (unsigned)j >= (unsigned)N || (unsigned)k >= (unsigned)N) return false;
    const float4 t = few_node<true>(r, a, b, c);
    return scatter_node(dst, i, j, k, pmass * t.x, pmass * t.y, pmass * t.z, pmass * t.w, f_mass, f_mom0);
}
constexpr int kFar = -2;

// The bins of few particles, a warp each (cf. the binned P2G): G2P, then the
// sums of their new positions.  s: the CTA's scratch (kBinNodes + kFewScratch a
// warp).
template <int L>
__device__ __noinline__ bool g2p2g_few(const DevGrid &src, const DevGrid &dst, const BinSplit &bins, const int32_t *bin_list,
                                       const int32_t *bin_off, const int32_t *bin_end, const int32_t *perm, float *x, float *v,
                                       float dt, int f_vel0, float pmass, int f_mass, int f_mom0, float4 *s)
{
    const int R = src.R, N = src.N, lane = lane_id(), warp = threadIdx.x >> 5;
    bool changed = false;
    float4 *s_u = s + warp * (kBinNodes + kFewScratch);
    s = s_u + kBinNodes;
    for (int w = blockIdx.x * kBinWarps + warp; w < bins.few; w += gridDim.x * kBinWarps) {
        const int b = bin_list[bins.last - w], beg = bin_off[b], cnt = bin_end[b] - beg;
        int bi, bj, bk;
        bin_block<L>(b, R, bi, bj, bk);
        const long long p = lane < cnt ? perm[beg + lane] : -1;
        float xp[3] = {}, vp[3] = {}, cp[9] = {};
        if (p >= 0) {
#pragma unroll
            for (int e = 0; e < 3; ++e) xp[e] = x[3 * p + e];
        }
        g2p_of_bin<L, true>(src, src.field[f_vel0], src.field[f_vel0 + 1], src.field[f_vel0 + 2], bi, bj, bk, cnt, xp, s_u, vp,
                            cp);
        FewParticle<true> r{};
        if (p >= 0) {
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                xp[e] += dt * vp[e];
                v[3 * p + e] = vp[e];
                x[3 * p + e] = xp[e];
            }
            few_particle<true>(r, xp[0], xp[1], xp[2], vp, cp, N);
        }
        const unsigned strays = few_sums<true>(r, cnt, 4 * bi, 4 * bj, 4 * bk, s);
        // the touched blocks' leaves, then the touched nodes' sums
        uint32_t hits = 0, blocks = 0;
#pragma unroll
        for (int h = 0; h < 7; ++h) {
            const int nd = h * 32 + lane;
            int i, j, k, blk, l;
            bin_node(nd, i, j, k, blk, l);
            if (nd < kBinNodes && 4 * bi + i < N && 4 * bj + j < N && 4 * bk + k < N && few_hit(s, i, j, k)) {
                hits |= 1u << h;
                blocks |= 1u << blk;
            }
        }
        blocks = __reduce_or_sync(kFull, blocks);
        int slot = -1;
        if (blocks >> lane & 1u) {
            const int ci = bi + (lane >> 2), cj = bj + ((lane >> 1) & 1), ck = bk + (lane & 1);
            bool fresh = false;
            slot = block_of_leaf<L>(ensure_leaf(dst, block_leaf<L>(R, ci, cj, ck), fresh), ci, cj, ck);
            changed |= fresh;
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 7; ++h) {
            const int nd = h * 32 + lane;
            int i, j, k, blk, l;
            bin_node(nd, i, j, k, blk, l);
            const int bs = __shfl_sync(kFull, slot, blk & 7);
            if (!(hits >> h & 1u) || bs < 0) continue;  // pool exhausted; the error is latched
            const float4 t = s[nd];
            const long long idx = block_voxel<L>(bs, i & 3, j & 3, k & 3);
            changed |= set_bit(dst, idx);
            atomicAdd(dst.field[f_mass] + idx, pmass * t.x);
            atomicAdd(dst.field[f_mom0] + idx, pmass * t.y);
            atomicAdd(dst.field[f_mom0 + 1] + idx, pmass * t.z);
            atomicAdd(dst.field[f_mom0 + 2] + idx, pmass * t.w);
        }
        // the others, most of whose leaves are there now
        few_strays<true>(r, strays, [&](int i, int j, int k, const float4 &t) {
            if ((unsigned)i < (unsigned)N && (unsigned)j < (unsigned)N && (unsigned)k < (unsigned)N)
                changed |= scatter_node(dst, i, j, k, pmass * t.x, pmass * t.y, pmass * t.z, pmass * t.w, f_mass, f_mom0);
        });
        __syncwarp();  // s is cleared for the next bin
    }
    return changed;
}

template <int L, bool AROUND>
__global__ void __launch_bounds__(kBinThreads, 2) k_g2p2g(const __grid_constant__ DevGrid src,
                                                          const __grid_constant__ DevGrid dst,
                                                          const int32_t *bin_list, const int32_t *bin_off,
                                                          const int32_t *bin_end, const int32_t *perm,
                                                          Ctrl *bin_ctrl, int turn, long long n, float *x, float *v,
                                                          float dt, int f_vel0, float pmass, int f_mass, int f_mom0)
{
    chained_entry();
    // of the three counts one is the last launch's, one this one's and one the
    // next one's, zero then
    const bool many = bin_ctrl->moved[turn] > n / kMovedShare &&
                      n > (long long)kMovedBin * (bin_ctrl->bins_used + bin_ctrl->bins_few);
    if (many != AROUND) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) bin_ctrl->moved[(turn + 2) % 3] = 0;
    int moved_here = 0;
    using S = G2P2GSmem<AROUND>;
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
    const BinSplit bins = bin_split(bin_ctrl, R, L, 0, 12);
    const int used = bins.all;
    // particles whose stencil missed the domain when they were binned
    {
        const int oob_bin = bins.last + 1;
        const int end = bin_end[oob_bin];
        for (int q = bin_off[oob_bin] + blockIdx.x * kBinWarps + warp; q < end; q += gridDim.x * kBinWarps)
            changed |= far_particle<L>(src, dst, x, v, perm[q], dt, f_vel0, pmass, f_mass, f_mom0);
    }
    // of a bin that several CTAs share, this one takes chunks part, part + parts, ...
    const int parts = bins.parts, part = parts > 1 ? blockIdx.x / used : 0;
    int bl = blockIdx.x - part * used, b = 0, beg = 0, end = 0;
    if (bl < used && part < parts) {
        b = nth_bin(bin_list, bins, bl);
        beg = bin_off[b];
        end = bin_end[b];
    }
    if (part * CAP < end - beg) {
        auto bin_of = [&](int l, int &b, int &beg, int &end) {
            b = nth_bin(bin_list, bins, l);
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
        int nb = 0, nbeg = 0, nend = 0;
        int slot = near_slot(b), c = part, nch = (end - beg + CAP - 1) / CAP;
        int p[PPT], pn[PPT];
        order(beg, end, c, nch, p);
        request(p);
        if (bl + (int)gridDim.x < used) bin_of(bl + gridDim.x, nb, nbeg, nend);
        constexpr int OUT = AROUND ? kFarCell : kOwnCells;  // the cell of the particles that no column sums
        auto fresh_bin = [&] {
            if (threadIdx.x < (AROUND ? 36 : 16)) s.sort.all[threadIdx.x] = 0;
            if (threadIdx.x < (AROUND ? 2 * (8 + 27) : 16)) s.sort.bits[threadIdx.x] = 0;
            if constexpr (AROUND)
                if (threadIdx.x == 0) s.sort.outer = 0;
        };
        for (int q = threadIdx.x; q <= OUT; q += kBinThreads) s.sort.cnt[q] = 0;
        fresh_bin();
        if (threadIdx.x < 27) s.uslot[threadIdx.x] = slot;
        __syncthreads();
        for (;;) {
            const bool last = c + parts >= nch, more = !last || bl + (int)gridDim.x < used;
            const int nnch = last ? (nend - nbeg + CAP - 1) / CAP : nch;
            if (more) order(last ? nbeg : beg, last ? nend : end, last ? 0 : c + parts, nnch, pn);
            if (last && more) slot = near_slot(nb);
            int bi, bj, bk;
            bin_block<L>(b, R, bi, bj, bk);
            const int oi = bi * 4, oj = bj * 4, ok = bk * 4;
            if (c == part) {  // src's node velocities, 0 outside the domain or the leaves
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
                            constexpr int E = AROUND ? 1 : 0;  // cells around
                            const bool near = (unsigned)(ci + E) < 4u + 2 * E && (unsigned)(cj + E) < 4u + 2 * E &&
                                              (unsigned)(ck + E) < 4u + 2 * E;
                            const int cell = near ? moved_cell(ci + 1, cj + 1, ck + 1) : OUT;
                            pl = cell | atomicAdd(&s.sort.cnt[cell], 1) << 8;
                            if (AROUND && cell >= kOwnCells) s.cell[AROUND ? q : 0] = __float_as_int(pack_cell(ci, cj, ck));
                            bin_record<true, CAP>(s.rec, q, nx.fx, ny.fx, nz.fx, uu.x, uu.y, uu.z, C, dx, !AROUND && !near,
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
            if (warp == 0) {
                if constexpr (AROUND) moved_scan(dst, s.sort, CAP);
                else bin_scan(dst, s.sort, CAP);
            }
            __syncthreads();
            if (threadIdx.x == 0) moved_here += s.sort.start[OUT + 1] - s.sort.start[kOwnCells];
#pragma unroll
            for (int u = 0; u < PPT; ++u)
                if (place[u] >= 0)
                    s.idx[s.sort.start[place[u] & 255] + (place[u] >> 8)] = (uint16_t)((u * kBinWarps + warp) * 32 + lane);
            __syncthreads();
            if (more) request(pn);
            bool moved = false;
            if constexpr (AROUND) {
                moved = s.sort.moved != 0;
                if (moved) moved_columns<CAP>(s.rec, s.idx, s.sort, s.buf);
                else own_columns<CAP>(s.rec, s.idx, s.sort, s.buf);
            } else {
                bin_columns<true, CAP>(s.rec, s.idx, s.sort, s.buf);
            }
            for (int pp = s.sort.start[moved ? OUT : kOwnCells] + warp; pp < s.sort.start[OUT + 1] && pp < CAP;
                 pp += kBinWarps) {
                int i, j, k;
                float4 t;
                const int q = s.idx[pp];
                bool in;
                if constexpr (AROUND) in = single_node<CAP>(s.rec, q, s.cell[q], oi, oj, ok, N, i, j, k, t);
                else in = edge_node<true, CAP>(s.rec, q, oi, oj, ok, N, i, j, k, t);
                if (in)
                    changed |= scatter_node(dst, i, j, k, pmass * t.x, pmass * t.y, pmass * t.z, pmass * t.w, f_mass, f_mom0);
            }
#pragma unroll
            for (int u = 0; u < PPT; ++u)
                for (unsigned far = __ballot_sync(kFull, place[u] == kFar); far; far &= far - 1)
                    changed |= far_particle<L>(src, dst, x, v, __shfl_sync(kFull, p[u], __ffs(far) - 1), dt, f_vel0, pmass,
                                               f_mass, f_mom0);
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
                    if (oi + i >= N || oj + j >= N || ok + k >= N) continue;
                    if constexpr (AROUND) {
                        if (!moved_hit(s.sort, i + 1, j + 1, k + 1)) continue;
                        t[h] = moved_total(s.sort, s.buf, i + 1, j + 1, k + 1);
                    } else {
                        if (!node_hit(s.sort, i, j, k)) continue;
                        t[h] = node_total(s.sort, s.buf, i, j, k);
                    }
                    where[h] = blk << 6 | l;
                    atomicOr(&s.sort.bits[2 * blk + (l >> 5)], 1u << (l & 31));
                }
                auto add = [&](int ds, int l, float4 v) {
                    const long long idx = block_voxel<L>(ds, l >> 4, l >> 2 & 3, l & 3);
                    atomicAdd(dst.field[f_mass] + idx, pmass * v.x);
                    atomicAdd(dst.field[f_mom0] + idx, pmass * v.y);
                    atomicAdd(dst.field[f_mom0 + 1] + idx, pmass * v.z);
                    atomicAdd(dst.field[f_mom0 + 2] + idx, pmass * v.w);
                };
                // the nodes o - 1 and o + 6 of a bin with particles in the cells around
                [[maybe_unused]] auto outer_nodes = [&](auto &&take) {
                    for (int nd = threadIdx.x; nd < 512; nd += kBinThreads) {
                        const int i = nd >> 6, j = nd >> 3 & 7, k = nd & 7;
                        if ((unsigned)(i - 1) < 6u && (unsigned)(j - 1) < 6u && (unsigned)(k - 1) < 6u) continue;
                        if ((unsigned)(oi + i - 1) >= (unsigned)N || (unsigned)(oj + j - 1) >= (unsigned)N ||
                            (unsigned)(ok + k - 1) >= (unsigned)N)
                            continue;
                        take(i, j, k, 8 + ((i + 3) >> 2) * 9 + ((j + 3) >> 2) * 3 + ((k + 3) >> 2),
                             ((i + 3) & 3) << 4 | ((j + 3) & 3) << 2 | ((k + 3) & 3));
                    }
                };
                bool outer = false;
                if constexpr (AROUND) {
                    outer = s.sort.outer != 0;
                    if (outer)
                        outer_nodes([&](int i, int j, int k, int blk, int l) {
                            if (moved_hit(s.sort, i, j, k)) atomicOr(&s.sort.bits[2 * blk + (l >> 5)], 1u << (l & 31));
                        });
                }
                __syncthreads();
                if (warp == 0) {
                    auto leaf = [&](int blk, int ci, int cj, int ck) {
                        int ds = -1;
                        if (s.sort.bits[2 * blk] | s.sort.bits[2 * blk + 1]) {
                            bool fresh = false;
                            ds = block_of_leaf<L>(ensure_leaf(dst, block_leaf<L>(R, ci, cj, ck), fresh), ci, cj, ck);
                            changed |= fresh;
                        }
                        s.sort.slot[blk] = ds;
                    };
                    if (lane < 8) leaf(lane, bi + (lane >> 2), bj + ((lane >> 1) & 1), bk + (lane & 1));
                    if (outer && lane < 27) leaf(8 + lane, bi + lane / 9 - 1, bj + (lane / 3) % 3 - 1, bk + lane % 3 - 1);
                    __syncwarp();
                    changed |= set_touched<L>(dst, s.sort.slot, s.sort.bits, outer ? 35 : 8);
                    if (lane < 27) s.uslot[lane] = slot;
                }
                __syncthreads();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (where[h] < 0) continue;
                    const int ds = s.sort.slot[where[h] >> 6];
                    if (ds >= 0) add(ds, where[h] & 63, t[h]);  // else the pool is exhausted; the error is latched
                }
                if constexpr (AROUND)
                    if (outer)
                        outer_nodes([&](int i, int j, int k, int blk, int l) {
                            const int ds = s.sort.slot[blk];
                            if (ds >= 0 && moved_hit(s.sort, i, j, k)) add(ds, l, moved_total(s.sort, s.buf, i, j, k));
                        });
                __syncthreads();
                fresh_bin();
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
    }
    if (moved_here) atomicAdd(&bin_ctrl->moved[(turn + 1) % 3], moved_here);
    static_assert(kBinWarps * (kBinNodes + kFewScratch) <= 4 * CAP, "the bins of few particles use the records' memory");
    if (bins.few)
        changed |= g2p2g_few<L>(src, dst, bins, bin_list, bin_off, bin_end, perm, x, v, dt, f_vel0, pmass, f_mass, f_mom0,
                                s.rec[0]);
    if (changed) mark_dirty(dst);
}

template <int L>
cudaError_t launch_g2p2g_L(const DevGrid &src, const DevGrid &dst, const DevGrid &bins, cudaStream_t s, float *x,
                           float *v, long long n, float dt, int f_vel0, float pmass, int f_mass, int f_mom0, int turn,
                           int num_sms)
{
    constexpr int bytes[2] = {(int)sizeof(G2P2GSmem<false>), (int)sizeof(G2P2GSmem<true>)};
    static std::atomic<int> known[2][kMaxDevices];
    int per[2];
    cudaError_t e = resident_per_sm(k_g2p2g<L, false>, kBinThreads, bytes[0], known[0], &per[0]);
    if (e == cudaSuccess) e = resident_per_sm(k_g2p2g<L, true>, kBinThreads, bytes[1], known[1], &per[1]);
    if (e != cudaSuccess) return e;
    launch_chained(k_g2p2g<L, false>, per[0] * num_sms, kBinThreads, bytes[0], s, src, dst, bins.bin_list, bins.bin_off,
                   bins.bin_count, bins.perm, bins.ctrl, turn, n, x, v, dt, f_vel0, pmass, f_mass, f_mom0);
    launch_chained(k_g2p2g<L, true>, per[1] * num_sms, kBinThreads, bytes[1], s, src, dst, bins.bin_list, bins.bin_off,
                   bins.bin_count, bins.perm, bins.ctrl, turn, n, x, v, dt, f_vel0, pmass, f_mass, f_mom0);
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_g2p2g(const DevGrid &src, const DevGrid &dst, const DevGrid &bins, cudaStream_t s, float *x, float *v,
                         long long n, float dt, int f_vel0, float pmass, int f_mass, int f_mom0, int turn,
                         const LaunchCfg &lc)
{
    if (n <= 0) return cudaSuccess;
    if (dst.L == 4) return launch_g2p2g_L<4>(src, dst, bins, s, x, v, n, dt, f_vel0, pmass, f_mass, f_mom0, turn, lc.num_sms);
    return launch_g2p2g_L<8>(src, dst, bins, s, x, v, n, dt, f_vel0, pmass, f_mass, f_mom0, turn, lc.num_sms);
}

}  // namespace sg

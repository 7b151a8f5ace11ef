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
// Work split: one CTA per bin of the last binned P2G over these particles
// (a leaf o with the particles whose base node was in it when binned).
//   1. stage src's velocities of nodes o-2 .. o+L+1 in shared memory;
//   2. per particle: G2P from the staged block (or node by node from the grid
//      when its base has left [o-2, o+L-1]), store x', v'; a particle of the
//      bin that moved less than a cell has its new base in [o-1, o+L] (bases
//      o-2 and o-1 of the low domain face excepted); count it in its new base
//      cell and keep its P2G record (spline offsets, m, q = m v - m dx C fx
//      and m dx C) in registers;
//   3. counting sort by new base cell, records staged in shared memory;
//   4. one warp per occupied cell: lane t < 27 sums its node's contributions
//      (as in the binned P2G gather) into shared accumulators of the dst
//      nodes o-1 .. o+L+2;
//   5. flush the touched nodes: the dst leaves they fall in are allocated
//      in-kernel if null (see ensure_leaf), bits set, 4 FP32 atomics per node.
// A particle whose new base is outside [o-1, o+L], and every particle of the
// out-of-domain key, is scattered node by node straight into dst with the same
// in-kernel allocation.
#include <atomic>
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

__device__ __forceinline__ float3 load3_checked(const DevGrid &g, const float *a, long long p, bool pair)
{
    const float *q = a + 3 * p;
    if (!pair || misaligned(g, q + (p & 1), 8, 1)) return make_float3(q[0], q[1], q[2]);
    if (p & 1) {
        const float2 hi = *reinterpret_cast<const float2 *>(q + 1);
        return make_float3(q[0], hi.x, hi.y);
    }
    const float2 lo = *reinterpret_cast<const float2 *>(q);
    return make_float3(lo.x, lo.y, q[2]);
}

__device__ __forceinline__ void store3_checked(const DevGrid &g, float *a, long long p, float3 t, bool pair)
{
    float *q = a + 3 * p;
    if (!pair || misaligned(g, q + (p & 1), 8, 2)) {
        q[0] = t.x;
        q[1] = t.y;
        q[2] = t.z;
    } else if (p & 1) {
        q[0] = t.x;
        *reinterpret_cast<float2 *>(q + 1) = make_float2(t.y, t.z);
    } else {
        *reinterpret_cast<float2 *>(q) = make_float2(t.x, t.y);
        q[2] = t.z;
    }
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

// Shared-memory layout of one CTA (dynamic shared memory).
template <int L>
struct G2P2GSmem {
    static constexpr int BU = L + 4;          // staged src nodes per axis (o-2 .. o+L+1)
    static constexpr int NU = BU * BU * BU;
    static constexpr int BD = L + 4;          // dst block nodes per axis (o-1 .. o+L+2)
    static constexpr int ND = BD * BD * BD;
    static constexpr int C1 = L + 2;          // new base cells per axis (o-1 .. o+L)
    static constexpr int NC = C1 * C1 * C1;
    static constexpr int CAP = 256;           // particles per chunk (one per thread)
    static constexpr size_t off_rec = 0;                                   // float4 [4][CAP]
    static constexpr size_t off_u = off_rec + sizeof(float4) * 4 * CAP;    // float4 [NU]
    static constexpr size_t off_acc = off_u + sizeof(float4) * NU;         // float [4][ND]
    static constexpr size_t off_cnt = off_acc + sizeof(float) * 4 * ND;    // int [NC + 1]
    static constexpr size_t off_start = off_cnt + sizeof(int) * (NC + 1);  // int [NC + 1]
    static constexpr size_t off_slot = off_start + sizeof(int) * (NC + 1); // int [27]
    static constexpr size_t off_hit = off_slot + sizeof(int) * 27;         // uint8 [ND]
    static constexpr size_t bytes = (off_hit + ND + 15) / 16 * 16;
};

template <int L>
__global__ void __launch_bounds__(256, L == 4 ? 3 : 2) k_g2p2g(DevGrid src, DevGrid dst, const int32_t *__restrict__ bin_list,
                                               const int32_t *__restrict__ bin_off, const int32_t *bin_end,
                                               int32_t *perm, const int32_t *bins_used, float *__restrict__ x,
                                               float *__restrict__ v, float dt, int f_vel0, float pmass, int f_mass,
                                               int f_mom0, bool pair)
{
    chained_entry();
    using S = G2P2GSmem<L>;
    constexpr int LG2 = (L == 8) ? 3 : 2, BD = S::BD, C1 = S::C1, NC = S::NC, ND = S::ND;
    extern __shared__ __align__(16) unsigned char smem[];
    float4(*s_rec)[S::CAP] = reinterpret_cast<float4(*)[S::CAP]>(smem + S::off_rec);
    float4 *s_u = reinterpret_cast<float4 *>(smem + S::off_u);
    float(*s_acc)[ND] = reinterpret_cast<float(*)[ND]>(smem + S::off_acc);
    int *s_cnt = reinterpret_cast<int *>(smem + S::off_cnt);
    int *s_start = reinterpret_cast<int *>(smem + S::off_start);
    int *s_slot = reinterpret_cast<int *>(smem + S::off_slot);
    uint8_t *s_hit = smem + S::off_hit;
    if (threadIdx.x == 0) misaligned(dst, smem, 16, 4);

    const int N = src.N, R = src.R;
    const float dx = 1.f / (float)N;
    const int warp = threadIdx.x >> 5, lane = lane_id();
    const int la = lane / 9, lc = (lane / 3) % 3, ld = lane % 3;
    const BsPoly pa = bs_poly(la), pb = bs_poly(lc), pc = bs_poly(ld);
    const float ta = (float)la, tb = (float)lc, tc = (float)ld;
    const float *u0p = src.field[f_vel0], *u1p = src.field[f_vel0 + 1], *u2p = src.field[f_vel0 + 2];
    bool changed = false;
    const int used = *bins_used;
    const long long oob_key = 8LL * R * R * R;
    for (int bl = blockIdx.x; bl <= used; bl += gridDim.x) {
        int beg, end, oi = 0, oj = 0, ok = 0;
        const bool binned = bl < used;
        if (binned) {
            const int b = bin_list[bl], bij = b / R, bi = bij / R;
            beg = bin_off[8LL * b];
            end = bin_end[8LL * b + 7];
            oi = bi * L;
            oj = (bij - bi * R) * L;
            ok = (b - bij * R) * L;
            stage_velocities<L>(src, u0p, u1p, u2p, oi, oj, ok, s_u);
            for (int q = threadIdx.x; q < ND; q += blockDim.x) {
                s_acc[0][q] = s_acc[1][q] = s_acc[2][q] = s_acc[3][q] = 0.f;
                s_hit[q] = 0;
            }
            __syncthreads();
        } else {
            beg = bin_off[oob_key];
            end = bin_end[oob_key];
        }
        for (int c0 = beg; c0 < end; c0 += S::CAP) {
            const int cnt = min(S::CAP, end - c0);
            if (binned) {
                for (int q = threadIdx.x; q <= NC; q += blockDim.x) s_cnt[q] = 0;
                __syncthreads();
            }
            // G2P of this thread's particle; its P2G record stays in registers
            int rcell = -1, rrank = 0, rp = 0;
            P2GRec rec;
            if ((int)threadIdx.x < cnt) {
                rp = perm[c0 + threadIdx.x];
                const long long p = rp;
                const float3 xp = load3_checked(dst, x, p, pair);
                const Spline ox = bspline(xp.x, N), oy = bspline(xp.y, N), oz = bspline(xp.z, N);
                const int ri = ox.base - oi + 2, rj = oy.base - oj + 2, rk = oz.base - ok + 2;
                float3 u;
                float c[9];
                if (binned && (unsigned)ri <= (unsigned)(L + 1) && (unsigned)rj <= (unsigned)(L + 1) &&
                    (unsigned)rk <= (unsigned)(L + 1))
                    g2p_from_block<L + 4, true>(s_u, ri, rj, rk, N, ox, oy, oz, u, c);
                else
                    g2p_from_grid<true>(src, u0p, u1p, u2p, ox, oy, oz, u, c);
                const float3 xn = make_float3(xp.x + dt * u.x, xp.y + dt * u.y, xp.z + dt * u.z);
                store3_checked(dst, v, p, u, pair);
                store3_checked(dst, x, p, xn, pair);
                const Spline nx = bspline(xn.x, N), ny = bspline(xn.y, N), nz = bspline(xn.z, N);
                rec = make_rec(nx.fx, ny.fx, nz.fx, pmass, u, c, dx);
                const int ci = nx.base - oi + 1, cj = ny.base - oj + 1, ck = nz.base - ok + 1;
                if (binned && (unsigned)ci < (unsigned)C1 && (unsigned)cj < (unsigned)C1 && (unsigned)ck < (unsigned)C1) {
                    rcell = (ci * C1 + cj) * C1 + ck;
                    rrank = atomicAdd(&s_cnt[rcell], 1);
                } else {
                    changed |= scatter_particle(dst, nx, ny, nz, rec, f_mass, f_mom0);
                }
            }
            if (!binned) continue;  // no shared block for the out-of-domain key
            __syncthreads();
            if (threadIdx.x < 32) {  // exclusive scan of the cell counts
                int carry = 0;
                for (int base = 0; base < NC; base += 32) {
                    const int i = base + threadIdx.x;
                    const int vv = (i < NC) ? s_cnt[i] : 0;
                    const int inc = warp_incl_scan(vv);
                    if (i < NC) s_start[i] = carry + inc - vv;
                    carry += __shfl_sync(kFull, inc, 31);
                }
                if (threadIdx.x == 0) s_start[NC] = carry;
            }
            __syncthreads();
            if (rcell >= 0 && !misaligned(dst, &s_rec[0][s_start[rcell] + rrank], 16, 5)) {
                const int pos = s_start[rcell] + rrank;
                s_rec[0][pos] = rec.r0;
                s_rec[1][pos] = rec.r1;
                s_rec[2][pos] = rec.r2;
                s_rec[3][pos] = rec.r3;
            }
            __syncthreads();
            for (int cell = warp; cell < NC; cell += blockDim.x / 32) {
                const int p0 = s_start[cell], p1 = s_start[cell + 1];
                if (p0 == p1) continue;  // uniform across the warp
                if (p0 < 0 || p1 > S::CAP || p0 > p1) {
                    if (lane == 0) {
                        atomicOr(&dst.ctrl->err, kErrCheck);
                        dst.ctrl->timeout_site = 106;
                    }
                    continue;
                }
                const int ci = cell / (C1 * C1), cj = (cell / C1) % C1, ck = cell % C1;
                float m = 0.f, m0 = 0.f, m1 = 0.f, m2 = 0.f;
                for (int pp = p0; pp < p1; ++pp) {
                    if (misaligned(dst, &s_rec[3][pp], 16, 7)) break;
                    const float4 r0 = s_rec[0][pp];
                    const float w = bs_eval(pa, r0.x) * bs_eval(pb, r0.y) * bs_eval(pc, r0.z);
                    const float4 r1 = s_rec[1][pp], r2 = s_rec[2][pp], r3 = s_rec[3][pp];
                    const float q0 = fmaf(r1.w, ta, fmaf(r2.x, tb, fmaf(r2.y, tc, r1.x)));
                    const float q1 = fmaf(r2.z, ta, fmaf(r2.w, tb, fmaf(r3.x, tc, r1.y)));
                    const float q2 = fmaf(r3.y, ta, fmaf(r3.z, tb, fmaf(r3.w, tc, r1.z)));
                    m = fmaf(w, r0.w, m);
                    m0 = fmaf(w, q0, m0);
                    m1 = fmaf(w, q1, m1);
                    m2 = fmaf(w, q2, m2);
                }
                if (lane < 27) {  // block node (ci + la, cj + lc, ck + ld) = grid node o - 1 + that
                    const int nd = ((ci + la) * BD + (cj + lc)) * BD + (ck + ld);
                    atomicAdd(&s_acc[0][nd], m);
                    atomicAdd(&s_acc[1][nd], m0);
                    atomicAdd(&s_acc[2][nd], m1);
                    atomicAdd(&s_acc[3][nd], m2);
                    s_hit[nd] = 1;
                }
            }
            __syncthreads();
        }
        if (!binned) continue;
        // dst leaves of the block: leaf cells (o >> LG2) - 1 .. (o >> LG2) + 1 per
        // axis hold every block node; allocate the ones with a touched in-domain node
        if (threadIdx.x < 27) s_slot[threadIdx.x] = 0;
        __syncthreads();
        const int li0 = (oi >> LG2) - 1, lj0 = (oj >> LG2) - 1, lk0 = (ok >> LG2) - 1;
        for (int nd = threadIdx.x; nd < ND; nd += blockDim.x) {
            if (!s_hit[nd]) continue;
            const int i = oi - 1 + nd / (BD * BD), j = oj - 1 + (nd / BD) % BD, k = ok - 1 + nd % BD;
            if ((unsigned)i >= (unsigned)N || (unsigned)j >= (unsigned)N || (unsigned)k >= (unsigned)N) continue;
            s_slot[((i >> LG2) - li0) * 9 + ((j >> LG2) - lj0) * 3 + ((k >> LG2) - lk0)] = 1;
        }
        __syncthreads();
        if (threadIdx.x < 27) {
            const int t = threadIdx.x;
            int slot = -1;
            if (s_slot[t]) {
                bool fresh = false;
                const long long lb = ((long long)(li0 + t / 9) * R + (lj0 + (t / 3) % 3)) * R + (lk0 + t % 3);
                slot = ensure_leaf(dst, lb, fresh);
                changed |= fresh;
            }
            s_slot[t] = slot;
        }
        __syncthreads();
        for (int nd = threadIdx.x; nd < ND; nd += blockDim.x) {
            if (!s_hit[nd]) continue;
            const int i = oi - 1 + nd / (BD * BD), j = oj - 1 + (nd / BD) % BD, k = ok - 1 + nd % BD;
            if ((unsigned)i >= (unsigned)N || (unsigned)j >= (unsigned)N || (unsigned)k >= (unsigned)N) continue;
            const int slot = s_slot[((i >> LG2) - li0) * 9 + ((j >> LG2) - lj0) * 3 + ((k >> LG2) - lk0)];
            if (slot < 0) continue;  // pool exhausted; the error is latched
            const int l = (((i & (L - 1)) << LG2) + (j & (L - 1))) * L + (k & (L - 1));
            uint32_t *mw = &dst.mask[(long long)slot * dst.W + (l >> 5)];
            const uint32_t bit = 1u << (l & 31);
            if (!(*(volatile uint32_t *)mw & bit)) changed |= !(atomicOr(mw, bit) & bit);
            const long long idx = ((long long)slot << (3 * LG2)) + l;
            atomicAdd(dst.field[f_mass] + idx, s_acc[0][nd]);
            atomicAdd(dst.field[f_mom0] + idx, s_acc[1][nd]);
            atomicAdd(dst.field[f_mom0 + 1] + idx, s_acc[2][nd]);
            atomicAdd(dst.field[f_mom0 + 2] + idx, s_acc[3][nd]);
        }
        __syncthreads();  // shared state is reset for the next bin
    }
    if (changed) mark_dirty(dst);
}

// ---------------------------------------------------------------------------
// The same over 4^3 leaves: the P2G half sums by columns (see bin_columns),
// and the next chunk's positions come into shared memory while a chunk is
// worked on.  A bin of several chunks deals its particles to them in turn, so
// each chunk has its share of every column whatever the order.  Particles
// whose new base left the leaf's 4^3 cells are added to the grid by a warp each
// (edge_node), the ones far from it, and those whose old base is more than a
// cell outside the leaf, by their own thread.  A whole leaf of the usual ten
// particles a cell is one chunk of 736: in chunks of 384 the columns are shorter
// and the three of a warp less even (238 us).  2M particles: 220 us a launch at
// two CTAs per SM without spills (the 256-thread kernel with a warp per cell:
// 308 us; this one at three CTAs and 96 registers, spilling: 264 us).
// ---------------------------------------------------------------------------
struct G2P2G4Smem {
    static constexpr int PPT = 4, CAP = 736;
    float4 rec[4][CAP];
    float4 buf[kBinBuf];
    float4 u[512];                  // src velocities of nodes o - 1 .. o + 6
    float x[3 * CAP];               // the next chunk's positions, in order
    float words[kBinWarps][96];
    int uslot[27];                  // src leaves o / 4 + {-1, 0, 1}^3
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

__global__ void __launch_bounds__(kBinThreads, 2) k_g2p2g4(const __grid_constant__ DevGrid src,
                                                          const __grid_constant__ DevGrid dst,
                                                          const int32_t *bin_list, const int32_t *bin_off,
                                                          const int32_t *bin_end, const int32_t *perm,
                                                          const int32_t *bins_used, float *x, float *v, float dt,
                                                          int f_vel0, float pmass, int f_mass, int f_mom0)
{
    chained_entry();
    using S = G2P2G4Smem;
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
        const long long key = 8LL * R * R * R;
        const int end = bin_end[key];
        for (int q = bin_off[key] + blockIdx.x * kBinThreads + threadIdx.x; q < end; q += gridDim.x * kBinThreads) {
            changed |= far_particle(src, dst, x, v, perm[q], dt, f_vel0, pmass, f_mass, f_mom0);
        }
    }
    int bl = blockIdx.x;
    if (bl < used) {
        auto leaf_of = [&](int l, int &b, int &beg, int &end) {
            b = bin_list[l];
            beg = bin_off[8LL * b];
            end = bin_end[8LL * b + 7];
        };
        // slot of leaf o / 4 + {-1, 0, 1}^3 of src (threads 0 .. 26), -1: none
        auto near_slot = [&](int b) {
            const int t = threadIdx.x;
            if (t >= 27) return -1;
            const int bij = b / R, bi = bij / R;
            const int li = bi + t / 9 - 1, lj = bij - bi * R + (t / 3) % 3 - 1, lk = b - bij * R + t % 3 - 1;
            return (unsigned)li < (unsigned)R && (unsigned)lj < (unsigned)R && (unsigned)lk < (unsigned)R
                       ? src.root[((long long)li * R + lj) * R + lk]
                       : -1;
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
        leaf_of(bl, b, beg, end);
        int slot = near_slot(b), c = 0, nch = (end - beg + CAP - 1) / CAP;
        int p[PPT], pn[PPT];
        order(beg, end, 0, nch, p);
        request(p);
        if (bl + (int)gridDim.x < used) leaf_of(bl + gridDim.x, nb, nbeg, nend);
        if (threadIdx.x < 65) s.sort.cnt[threadIdx.x] = 0;
        if (threadIdx.x < 16) s.sort.all[threadIdx.x] = s.sort.bits[threadIdx.x] = 0;
        if (threadIdx.x < 27) s.uslot[threadIdx.x] = slot;
        __syncthreads();
        for (;;) {
            const bool last = c + 1 >= nch, more = !last || bl + (int)gridDim.x < used;
            const int nnch = last ? (nend - nbeg + CAP - 1) / CAP : nch;
            if (more) order(last ? nbeg : beg, last ? nend : end, last ? 0 : c + 1, nnch, pn);
            if (last && more) slot = near_slot(nb);
            const int bij = b / R, bi = bij / R;
            const int oi = bi * 4, oj = (bij - bi * R) * 4, ok = (b - bij * R) * 4;
            if (c == 0) {  // src's node velocities, 0 outside the domain or the leaves
                for (int nd = threadIdx.x; nd < 512; nd += kBinThreads) {
                    const int i = (nd >> 6) + 3, j = ((nd >> 3) & 7) + 3, k = (nd & 7) + 3;  // from o - 4
                    const int us = s.uslot[(i >> 2) * 9 + (j >> 2) * 3 + (k >> 2)];
                    float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (us >= 0) {
                        const long long idx = ((long long)us << 6) + (((i & 3) << 4) | ((j & 3) << 2) | (k & 3));
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
                    int i, j, k, leaf, l;
                    bin_node(nd, i, j, k, leaf, l);
                    if (oi + i >= N || oj + j >= N || ok + k >= N || !node_hit(s.sort, i, j, k)) continue;
                    t[h] = node_total(s.sort, s.buf, i, j, k);
                    where[h] = leaf << 6 | l;
                    atomicOr(&s.sort.bits[2 * leaf + (l >> 5)], 1u << (l & 31));
                }
                __syncthreads();
                if (warp == 0) {
                    if (lane < 8) {
                        int ds = -1;
                        if (s.sort.bits[2 * lane] | s.sort.bits[2 * lane + 1]) {
                            bool fresh = false;
                            ds = ensure_leaf(dst, ((long long)(bi + (lane >> 2)) * R + (oj >> 2) + ((lane >> 1) & 1)) * R +
                                                      (ok >> 2) + (lane & 1), fresh);
                            changed |= fresh;
                        }
                        s.sort.slot[lane] = ds;
                    }
                    __syncwarp();
                    if (lane < 16) {
                        const uint32_t want = s.sort.bits[lane];
                        const int ds = s.sort.slot[lane >> 1];
                        if (want && ds >= 0) {
                            uint32_t *mw = &dst.mask[(long long)ds * 2 + (lane & 1)];
                            if ((*(volatile uint32_t *)mw & want) != want) changed |= (atomicOr(mw, want) & want) != want;
                        }
                    }
                    if (lane < 27) s.uslot[lane] = slot;
                }
                __syncthreads();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (where[h] < 0) continue;
                    const int ds = s.sort.slot[where[h] >> 6];
                    if (ds < 0) continue;  // pool exhausted; the error is latched
                    const long long idx = ((long long)ds << 6) + (where[h] & 63);
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
                if (bl + (int)gridDim.x < used) leaf_of(bl + gridDim.x, nb, nbeg, nend);
            } else {
                ++c;
                __syncthreads();  // the records are rewritten by the leaf's next chunk
            }
            nch = nnch;
#pragma unroll
            for (int u = 0; u < PPT; ++u) p[u] = pn[u];
        }
    }
    if (changed) mark_dirty(dst);
}

void launch_g2p2g_4(const DevGrid &src, const DevGrid &dst, const DevGrid &bins, cudaStream_t s, float *x, float *v,
                    float dt, int f_vel0, float pmass, int f_mass, int f_mom0, int num_sms)
{
    constexpr int bytes = (int)sizeof(G2P2G4Smem);
    static std::atomic<int> resident;  // CTAs per SM; threads may race to fill it
    int per = resident.load(std::memory_order_relaxed);
    if (!per) {
        cudaFuncSetAttribute(k_g2p2g4, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_g2p2g4, kBinThreads, bytes) != cudaSuccess || per < 1)
            per = 1;
        resident.store(per, std::memory_order_relaxed);
    }
    launch_chained(k_g2p2g4, per * num_sms, kBinThreads, bytes, s, src, dst, bins.bin_list, bins.bin_off, bins.bin_count,
                   bins.perm, &bins.ctrl->bins_used, x, v, dt, f_vel0, pmass, f_mass, f_mom0);
}

template <int L>
void launch_g2p2g_L(const DevGrid &src, const DevGrid &dst, const DevGrid &bins, cudaStream_t s, float *x, float *v,
                    float dt, int f_vel0, float pmass, int f_mass, int f_mom0, bool pair, int num_sms)
{
    constexpr size_t bytes = G2P2GSmem<L>::bytes;
    static std::atomic<int> resident;  // CTAs per SM; threads may race to fill it
    int per = resident.load(std::memory_order_relaxed);
    if (!per) {
        cudaFuncSetAttribute(k_g2p2g<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_g2p2g<L>, 256, bytes) != cudaSuccess || per < 1)
            per = 1;
        resident.store(per, std::memory_order_relaxed);
    }
    const int ctas = per * num_sms;
    launch_chained(k_g2p2g<L>, ctas, 256, bytes, s, src, dst, bins.bin_list, bins.bin_off, bins.bin_count, bins.perm,
                                         &bins.ctrl->bins_used, x, v, dt, f_vel0, pmass, f_mass, f_mom0, pair);
}

}  // namespace

void launch_g2p2g(const DevGrid &src, const DevGrid &dst, const DevGrid &bins, cudaStream_t s, float *x, float *v,
                  long long n, float dt, int f_vel0, float pmass, int f_mass, int f_mom0, const LaunchCfg &lc)
{
    if (n <= 0) return;
    const bool pair = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(v)) & 7) == 0;
    if (dst.L == 4) launch_g2p2g_4(src, dst, bins, s, x, v, dt, f_vel0, pmass, f_mass, f_mom0, lc.num_sms);
    else launch_g2p2g_L<8>(src, dst, bins, s, x, v, dt, f_vel0, pmass, f_mass, f_mom0, pair, lc.num_sms);
}

}  // namespace sg

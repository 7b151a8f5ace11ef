// sg_particle.cuh -- device helpers of the particle-grid transfers, shared
// by the separate (sg_particle.cu) and the fused G2P2G (sg_g2p2g.cu)
// kernels: the quadratic B-spline of a particle along one axis, G2P of one
// particle from a staged block of node velocities or node by node from the
// grid (PIC, or APIC with the matrix C), the particle-array accessors, the sums
// of a bin by columns of cells, and those of a bin of few particles by a warp.
#pragma once
#include "sg_common.cuh"

namespace sg {

struct Spline {
    int base;
    float fx;  // X - base, in [0.5, 1.5)
    float w[3];
};

// base = floor(X - 0.5), fx = X - base, X = x*N, all in FP32, each operation
// rounded on its own (no contraction), so that every kernel that bins a
// particle takes the same base.
__device__ __forceinline__ Spline bspline(float x, int N)
{
    Spline s;
    const float X = __fmul_rn(x, (float)N);
    const float bf = floorf(__fsub_rn(X, 0.5f));
    const float fx = __fsub_rn(X, bf);
    s.base = (int)bf;
    s.fx = fx;
    const float a = 1.5f - fx, c = fx - 1.0f, d = fx - 0.5f;
    s.w[0] = 0.5f * a * a;
    s.w[1] = 0.75f - c * c;
    s.w[2] = 0.5f * d * d;
    return s;
}

// G2P of one particle read node by node from the grid (a stored value at an
// inactive node is 0; out-of-domain and unallocated nodes are skipped).
// Returns v_p in u and, for APIC, C_p in c.
template <bool APIC>
__device__ __forceinline__ void g2p_from_grid(const DevGrid &g, const float *__restrict__ f0,
                                              const float *__restrict__ f1, const float *__restrict__ f2,
                                              const Spline &sx, const Spline &sy, const Spline &sz, float3 &u,
                                              float (&c)[9])
{
    const int L = g.L, lg2 = g.lg2, N = g.N;
    float ux = 0.f, uy = 0.f, uz = 0.f;
    float S[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};  // sum w v_e t_f
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int i = sx.base + a;
        if ((unsigned)i >= (unsigned)N) continue;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int j = sy.base + b;
            if ((unsigned)j >= (unsigned)N) continue;
            const float wxy = sx.w[a] * sy.w[b];
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) {
                const int k = sz.base + cc;
                if ((unsigned)k >= (unsigned)N) continue;
                const long long lb = ((long long)(i >> lg2) * g.R + (j >> lg2)) * g.R + (k >> lg2);
                const int slot = __ldg(g.root + lb);
                if (slot < 0) continue;
                const int l = (((i & (L - 1)) << lg2) + (j & (L - 1))) * L + (k & (L - 1));
                const long long idx = ((long long)slot << (3 * lg2)) + l;
                const float w = wxy * sz.w[cc];
                const float wv[3] = {w * __ldg(f0 + idx), w * __ldg(f1 + idx), w * __ldg(f2 + idx)};
                ux += wv[0];
                uy += wv[1];
                uz += wv[2];
                if (APIC) {
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        S[e][0] = fmaf((float)a, wv[e], S[e][0]);
                        S[e][1] = fmaf((float)b, wv[e], S[e][1]);
                        S[e][2] = fmaf((float)cc, wv[e], S[e][2]);
                    }
                }
            }
        }
    }
    u = make_float3(ux, uy, uz);
    if (APIC) {
        const float s4 = 4.f * (float)N, fx[3] = {sx.fx, sy.fx, sz.fx}, ue[3] = {ux, uy, uz};
#pragma unroll
        for (int e = 0; e < 3; ++e)
#pragma unroll
            for (int f = 0; f < 3; ++f) c[3 * e + f] = s4 * fmaf(-fx[f], ue[e], S[e][f]);
    }
}

// Records of K floats per particle (x and v: 3, C: 9) moved by a whole warp.
// Lane q holds particle p (or -1: none); word e of the warp's 32 K words is
// moved by lane e mod 32, so the words of a particle go in one access of
// neighbouring lanes and a warp access touches 32 / K particles' lines, not
// 32.  s (32 K floats of the warp's own shared memory) holds the records in
// lane order in between; K is odd, so neither side has bank conflicts.
template <int K>
__device__ __forceinline__ void warp_fetch(const float *__restrict__ a, int p, float (&t)[K])
{
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int e = r * 32 + lane_id(), src = e / K;
        const int q = __shfl_sync(kFull, p, src);
        t[r] = q < 0 ? 0.f : a[(long long)K * q + (e - K * src)];
    }
}
// The fetched words to their lanes' records.
template <int K>
__device__ __forceinline__ void warp_deal(const float (&t)[K], float *s, float (&v)[K])
{
    __syncwarp();
#pragma unroll
    for (int r = 0; r < K; ++r) s[r * 32 + lane_id()] = t[r];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < K; ++r) v[r] = s[K * lane_id() + r];
}
template <int K>
__device__ __forceinline__ void warp_put(float *__restrict__ a, int p, const float (&v)[K], float *s)
{
    __syncwarp();
#pragma unroll
    for (int r = 0; r < K; ++r) s[K * lane_id() + r] = v[r];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int e = r * 32 + lane_id(), src = e / K;
        const int q = __shfl_sync(kFull, p, src);
        if (q >= 0) a[(long long)K * q + (e - K * src)] = s[e];
    }
}

// 4^3 blocks, the bins of the particle kernels: a 4^3 leaf, or an octant of an
// 8^3 one.  A bin's number is its leaf's times 8 plus the octant; a block's
// slot is its leaf's slot numbered the same way (an int: 2^28 leaves of 8^3
// floats are more than the device holds).
template <int L>
__device__ __forceinline__ void bin_block(int b, int R, int &bi, int &bj, int &bk)
{
    const int leaf = L == 8 ? b >> 3 : b, lij = leaf / R;
    bi = lij / R;
    bj = lij - bi * R;
    bk = leaf - lij * R;
    if (L == 8) {
        bi = 2 * bi + (b >> 2 & 1);
        bj = 2 * bj + (b >> 1 & 1);
        bk = 2 * bk + (b & 1);
    }
}
template <int L>
__device__ __forceinline__ long long block_leaf(int R, int bi, int bj, int bk)
{
    constexpr int S = L == 8 ? 1 : 0;
    return ((long long)(bi >> S) * R + (bj >> S)) * R + (bk >> S);
}
template <int L>
__device__ __forceinline__ int block_of_leaf(int slot, int bi, int bj, int bk)
{
    return L == 4 || slot < 0 ? slot : slot * 8 + ((bi & 1) << 2 | (bj & 1) << 1 | (bk & 1));
}
// Slot of block (bi, bj, bk), negative if there is none or it lies outside the domain.
template <int L>
__device__ __forceinline__ int block_slot(const int32_t *root, int R, int bi, int bj, int bk)
{
    constexpr int S = L == 8 ? 1 : 0;
    if ((unsigned)bi >= (unsigned)(R << S) || (unsigned)bj >= (unsigned)(R << S) || (unsigned)bk >= (unsigned)(R << S)) return -1;
    return block_of_leaf<L>(root[block_leaf<L>(R, bi, bj, bk)], bi, bj, bk);
}
// Voxel (i, j, k) (0 .. 3) of a block: its index in the fields.
template <int L>
__device__ __forceinline__ long long block_voxel(int bs, int i, int j, int k)
{
    if (L == 4) return (long long)bs << 6 | (i << 4 | j << 2 | k);
    return (long long)(bs >> 3) << 9 | ((bs & 4) << 6 | i << 6 | (bs & 2) << 4 | j << 3 | (bs & 1) << 2 | k);
}

// G2P of one particle from a staged block of B^3 float4 node velocities (ri,
// rj, rk: its base relative to the block's first node).  APIC as in
// g2p_from_grid, the sums formed axis by axis: along k for each of the nine
// (a, b), then along j, then i (240 operations for 27 nodes, not 350).
template <int B, bool APIC>
__device__ __forceinline__ void g2p_from_block(const float4 *s_u, int ri, int rj, int rk, int N, const Spline &sx,
                                               const Spline &sy, const Spline &sz, float3 &u, float (&c)[9])
{
    float U[3] = {0.f, 0.f, 0.f};
    float S[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float wa = a == 0 ? sx.w[0] : (a == 1 ? sx.w[1] : sx.w[2]), ta = (float)a;
        const float4 *plane = s_u + ((ri + a) * B + rj) * B + rk;
        float T[3] = {0.f, 0.f, 0.f}, Tj[3] = {0.f, 0.f, 0.f}, Tk[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const float4 n0 = plane[b * B], n1 = plane[b * B + 1], n2 = plane[b * B + 2];
            const float v0[3] = {n0.x, n0.y, n0.z}, v1[3] = {n1.x, n1.y, n1.z}, v2[3] = {n2.x, n2.y, n2.z};
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                const float s1 = sz.w[1] * v1[e], s2 = sz.w[2] * v2[e];
                const float s = fmaf(sz.w[0], v0[e], s1 + s2);
                T[e] = fmaf(sy.w[b], s, T[e]);
                if (APIC) {
                    if (b) Tj[e] = fmaf((float)b * sy.w[b], s, Tj[e]);
                    Tk[e] = fmaf(sy.w[b], fmaf(2.f, s2, s1), Tk[e]);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            U[e] = fmaf(wa, T[e], U[e]);
            if (APIC) {
                S[e][0] = fmaf(ta * wa, T[e], S[e][0]);
                S[e][1] = fmaf(wa, Tj[e], S[e][1]);
                S[e][2] = fmaf(wa, Tk[e], S[e][2]);
            }
        }
    }
    u = make_float3(U[0], U[1], U[2]);
    if (APIC) {
        const float s4 = 4.f * (float)N, fx[3] = {sx.fx, sy.fx, sz.fx};
#pragma unroll
        for (int e = 0; e < 3; ++e)
#pragma unroll
            for (int f = 0; f < 3; ++f) c[3 * e + f] = s4 * fmaf(-fx[f], U[e], S[e][f]);
    }
}

// Quadratic B-spline weight of stencil offset t (0, 1, 2) at spline offset f
// as a polynomial in f: 0.5(1.5-f)^2, 0.75-(f-1)^2, 0.5(f-0.5)^2.
struct BsPoly {
    float a2, a1, a0;
};
__device__ __forceinline__ BsPoly bs_poly(int t)
{
    BsPoly c;
    c.a2 = (t == 1) ? -1.f : 0.5f;
    c.a1 = (t == 0) ? -1.5f : ((t == 1) ? 2.f : -0.5f);
    c.a0 = (t == 0) ? 1.125f : ((t == 1) ? -0.25f : 0.125f);
    return c;
}
__device__ __forceinline__ float bs_eval(const BsPoly &c, float f) { return fmaf(fmaf(c.a2, f, c.a1), f, c.a0); }

// ---------------------------------------------------------------------------
// P2G sums of one bin of 4^3 cells (the base cells o .. o + 3), as the binned
// P2G takes them; the fused G2P2G, whose particles have moved since they were
// binned, has its own sort and walk around the same sums.  CTAs of six warps.
//
// The chunk's particles lie in shared memory as float4 records
//   PIC   r0 = (f_i, f_j, z0, z2)  r1 = (v0, v1, v2, z1)
//   APIC  r0 = (f_i, f_j, z0, z2)  r1 = (q0, q1, q2, M0)  r2 = M1..M4
//         r3 = M5..M8,  M = dx C, q = v - M f
// (f: spline offsets, z: the three weights along k; a unit mass: the sums are
// scaled when they are flushed), and idx lists them by base cell, k fastest,
// so the four cells of a column (ci, cj) are consecutive.  Nine lanes share a
// column: lane (a, b) walks its particles and sums their contributions to the
// nodes (ci + a, cj + b, .) in a window of three nodes along k, which moves on
// cell by cell, so the weights along i and j and the record are read once for
// three nodes, and three columns go side by side in a warp: the 16 columns take
// one round of the six warps.  A finished node is stored to the lane's own
// place in s_buf -- no atomics, which on FP32 in shared memory are compare and
// swap loops -- and node_total adds a node's up to nine column sums.  Particles
// outside the 4^3 cells (bucket 64, r0 = (f_i, f_j, f_k, cell)) are added to
// the grid by a warp each (edge_node).
// What bounds it is issue and the barriers between the phases of a bin (40 %
// issue at 12 warps per SM).  Registers matter more than warps: at four CTAs per
// SM (80 registers) the APIC form spills and is slower than at two.
// ---------------------------------------------------------------------------
constexpr int kBinThreads = 192, kBinWarps = kBinThreads / 32;
constexpr int kBinNodes = 216;        // 6^3 nodes o .. o + 5
constexpr int kBinBuf = 16 * 9 * 6;   // float4 [column][lane][node]

struct BinSort {
    int cnt[65];       // particles per cell (64: outside the cells); zero between chunks
    int start[66];     // their places in idx
    uint32_t prev[16], all[16];  // occupied cells of each column before / after this chunk
    int slot[8];       // blocks o / 4 + {0, 1}^3
    uint32_t bits[16]; // touched nodes of those blocks, i, j, k in order
};

// A chunk's particles are at most cap: the loops over the sorted records take no
// more (they would read past their memory), and a sort that counted more is an
// error, or those left out would be lost without one.
__device__ __forceinline__ void sort_fits(const DevGrid &g, int total, int cap, int site)
{
    if (total > cap) raise_check(g, site);
}

// Exclusive scan of the cell counts (one warp), which it zeroes; cap: the most
// that there can be.
__device__ __forceinline__ void bin_scan(const DevGrid &g, BinSort &s, int cap)
{
    const int lane = lane_id();
    int c[4] = {0, 0, 0, 0};
    if (lane < 16) {
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] = s.cnt[4 * lane + q];
    } else if (lane == 16) {
        c[0] = s.cnt[64];
    }
    const int tot = (c[0] + c[1]) + (c[2] + c[3]);
    int run = warp_incl_scan(tot) - tot;
    if (lane < 16) {
        uint32_t now = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            s.start[4 * lane + q] = run;
            s.cnt[4 * lane + q] = 0;
            run += c[q];
            if (c[q]) now |= 1u << q;
        }
        const uint32_t before = s.all[lane];
        s.prev[lane] = before;
        s.all[lane] = before | now;
    } else if (lane == 16) {
        sort_fits(g, run + tot, cap, 7);
        s.start[64] = run;
        s.start[65] = run + tot;
        s.cnt[64] = 0;
    }
}

// Record q's contribution to the three nodes of its cell in column lane (a, b)
// (pa, pb: its weights; ta, tb: a and b).
template <bool APIC, int CAP>
__device__ __forceinline__ void column_add(const float4 (*rec)[CAP], int q, const BsPoly &pa, const BsPoly &pb, float ta,
                                           float tb, float4 &n0, float4 &n1, float4 &n2)
{
    const float4 r0 = rec[0][q], r1 = rec[1][q];
    const float w = bs_eval(pa, r0.x) * bs_eval(pb, r0.y);
    const float w0 = w * r0.z, w1 = w * (APIC ? (1.f - r0.z) - r0.w : r1.w), w2 = w * r0.w;
    float u0 = r1.x, u1 = r1.y, u2 = r1.z;
    float m2 = 0.f, m5 = 0.f, m8 = 0.f;
    if (APIC) {
        const float4 r2 = rec[APIC ? 2 : 0][q], r3 = rec[APIC ? 3 : 0][q];
        u0 = fmaf(r1.w, ta, fmaf(r2.x, tb, u0));
        u1 = fmaf(r2.z, ta, fmaf(r2.w, tb, u1));
        u2 = fmaf(r3.y, ta, fmaf(r3.z, tb, u2));
        m2 = r2.y;
        m5 = r3.x;
        m8 = r3.w;
    }
    n0.x += w0;
    n0.y = fmaf(w0, u0, n0.y);
    n0.z = fmaf(w0, u1, n0.z);
    n0.w = fmaf(w0, u2, n0.w);
    n1.x += w1;
    n1.y = fmaf(w1, APIC ? u0 + m2 : u0, n1.y);
    n1.z = fmaf(w1, APIC ? u1 + m5 : u1, n1.z);
    n1.w = fmaf(w1, APIC ? u2 + m8 : u2, n1.w);
    n2.x += w2;
    n2.y = fmaf(w2, APIC ? fmaf(2.f, m2, u0) : u0, n2.y);
    n2.z = fmaf(w2, APIC ? fmaf(2.f, m5, u1) : u1, n2.z);
    n2.w = fmaf(w2, APIC ? fmaf(2.f, m8, u2) : u2, n2.w);
}

// idx has CAP + 1 entries at least: a particle's place is read one ahead.
template <bool APIC, int CAP>
__device__ __forceinline__ void bin_columns(const float4 (*rec)[CAP], const uint16_t *idx, const BinSort &s,
                                            float4 *s_buf)
{
    const int lane = lane_id(), grp = lane / 9, sub = lane - 9 * grp;
    const int col = (threadIdx.x >> 5) * 3 + grp;
    if (grp > 2 || col > 15) return;
    int pp = s.start[4 * col];
    const int last = s.start[4 * col + 4];
    if (pp >= last || last > CAP) return;
    const int a = sub / 3, b = sub - 3 * a;
    const BsPoly pa = bs_poly(a), pb = bs_poly(b);
    const float ta = (float)a, tb = (float)b;
    const bool add = s.prev[col] != 0;  // an earlier chunk stored this column's sums
    float4 *out = s_buf + (col * 9 + sub) * 6;
    float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f), n1 = n0, n2 = n0;
    auto store = [&](int k, float4 n) {
        if (add) {
            const float4 o = out[k];
            n = make_float4(o.x + n.x, o.y + n.y, o.z + n.z, o.w + n.w);
        }
        out[k] = n;
    };
    int next = idx[pp];
#pragma unroll 1
    for (int ck = 0; ck < 4; ++ck) {
        const int end = s.start[4 * col + ck + 1];
        while (pp < end) {
            const int q = next;
            next = idx[++pp];
            column_add<APIC, CAP>(rec, q, pa, pb, ta, tb, n0, n1, n2);
        }
        store(ck, n0);
        n0 = n1;
        n1 = n2;
        n2 = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    store(4, n0);
    store(5, n1);
}

// Does any particle's stencil hold bin node (i, j, k) (0 .. 5 from o)?
__device__ __forceinline__ bool node_hit(const BinSort &s, int i, int j, int k)
{
    uint32_t m = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            if ((unsigned)(i - a) <= 3u && (unsigned)(j - b) <= 3u) m |= s.all[(i - a) * 4 + (j - b)];
    return (((m | (m << 1) | (m << 2)) >> k) & 1u) != 0u;
}

// Its sums over the columns that were stored.
__device__ __forceinline__ float4 node_total(const BinSort &s, const float4 *s_buf, int i, int j, int k)
{
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int ci = i - a, cj = j - b, col = ci * 4 + cj;
            if ((unsigned)ci > 3u || (unsigned)cj > 3u || !s.all[col]) continue;
            const float4 v = s_buf[(col * 9 + a * 3 + b) * 6 + k];
            t.x += v.x;
            t.y += v.y;
            t.z += v.z;
            t.w += v.w;
        }
    return t;
}

// Node nd of the bin: its place among the 6^3, the block of BinSort::slot that
// holds it and the local index there.
__device__ __forceinline__ void bin_node(int nd, int &i, int &j, int &k, int &blk, int &l)
{
    i = nd / 36;
    j = nd / 6 - 6 * i;
    k = nd - 6 * (nd / 6);
    blk = ((i >> 2) << 2) | ((j >> 2) << 1) | (k >> 2);
    l = ((i & 3) << 4) | ((j & 3) << 2) | (k & 3);
}

// Set the touched nodes' bits of n blocks in their leaves' masks (one warp; a
// lane per mask word: two of a 4^3 leaf, four of a block in an 8^3 one).
// Returns whether this lane set a new one.
template <int L>
__device__ __forceinline__ bool set_touched(const DevGrid &g, const int *slot, const uint32_t *bits, int n)
{
    bool set = false;
    for (int q = lane_id(); q < n * (L == 4 ? 2 : 4); q += 32) {
        int bs;
        uint32_t want;
        long long word;
        if (L == 4) {
            bs = slot[q >> 1];
            want = bits[q];
            word = (long long)bs * 2 + (q & 1);
        } else {
            bs = slot[q >> 2];
            const uint32_t h = bits[q >> 1] >> ((q & 1) << 4);  // the plane's 16 bits, k fastest
            want = ((h & 0xfu) | (h & 0xf0u) << 4 | (h & 0xf00u) << 8 | (h & 0xf000u) << 12) << ((bs & 1) << 2);
            word = (long long)(bs >> 3) * 16 + ((bs & 4) + (q & 3)) * 2 + (bs >> 1 & 1);
        }
        if (!want || bs < 0) continue;
        uint32_t *mw = g.mask + word;
        set |= (*(volatile uint32_t *)mw & want) != want && (atomicOr(mw, want) & want) != want;
    }
    return set;
}

// Cell of a particle outside the bin's cells, relative to o, in 10 bits a
// coordinate (|.| < 512).
__device__ __forceinline__ float pack_cell(int ri, int rj, int rk)
{
    return __int_as_float(((ri + 512) << 20) | ((rj + 512) << 10) | (rk + 512));
}

// A particle's record at place pos, from its spline offsets, velocity and (C
// scaled in place) affine matrix; cell: pack_cell's word for bucket 64.
template <bool APIC, int CAP>
__device__ __forceinline__ void bin_record(float4 (*rec)[CAP], int pos, float fx, float fy, float fz, float v0, float v1,
                                           float v2, float (&c)[9], float dx, bool edge, float cell)
{
    const float d0 = 1.5f - fz, d1 = fz - 1.0f, d2 = fz - 0.5f;
    const float z0 = 0.5f * d0 * d0, z1 = 0.75f - d1 * d1, z2 = 0.5f * d2 * d2;
    rec[0][pos] = make_float4(fx, fy, edge ? fz : z0, edge ? cell : z2);
    if (!APIC) {
        rec[1][pos] = make_float4(v0, v1, v2, z1);
    } else {
#pragma unroll
        for (int e = 0; e < 9; ++e) c[e] *= dx;
        rec[1][pos] = make_float4(v0 - (c[0] * fx + c[1] * fy + c[2] * fz), v1 - (c[3] * fx + c[4] * fy + c[5] * fz),
                                  v2 - (c[6] * fx + c[7] * fy + c[8] * fz), c[0]);
        rec[APIC ? 2 : 0][pos] = make_float4(c[1], c[2], c[3], c[4]);
        rec[APIC ? 3 : 0][pos] = make_float4(c[5], c[6], c[7], c[8]);
    }
}

// Four bytes from global to shared memory, asynchronously.
__device__ __forceinline__ void copy_word(float *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One record outside the bin's cells, by a warp: lane (a, b, c) < 27 forms the
// contribution of its node base + (a, b, c); false for lanes without a node in
// the domain.  t: weight and weighted velocity.
template <bool APIC, int CAP>
__device__ __forceinline__ bool edge_node(const float4 (*rec)[CAP], int pp, int oi, int oj, int ok, int N, int &i, int &j,
                                          int &k, float4 &t)
{
    const int lane = lane_id(), a = lane / 9, b = (lane / 3) % 3, c = lane % 3;
    if (lane >= 27) return false;
    const float4 r0 = rec[0][pp], r1 = rec[1][pp];
    const int cell = __float_as_int(r0.w);
    i = oi + (cell >> 20) - 512 + a;
    j = oj + ((cell >> 10) & 1023) - 512 + b;
    k = ok + (cell & 1023) - 512 + c;
    if ((unsigned)i >= (unsigned)N || (unsigned)j >= (unsigned)N || (unsigned)k >= (unsigned)N) return false;
    const float w = bs_eval(bs_poly(a), r0.x) * bs_eval(bs_poly(b), r0.y) * bs_eval(bs_poly(c), r0.z);
    float u0 = r1.x, u1 = r1.y, u2 = r1.z;
    if (APIC) {
        const float4 r2 = rec[APIC ? 2 : 0][pp], r3 = rec[APIC ? 3 : 0][pp];
        const float ta = (float)a, tb = (float)b, tc = (float)c;
        u0 = fmaf(r1.w, ta, fmaf(r2.x, tb, fmaf(r2.y, tc, u0)));
        u1 = fmaf(r2.z, ta, fmaf(r2.w, tb, fmaf(r3.x, tc, u1)));
        u2 = fmaf(r3.y, ta, fmaf(r3.z, tb, fmaf(r3.w, tc, u2)));
    }
    t = make_float4(w, w * u0, w * u1, w * u2);
    return true;
}

// ---------------------------------------------------------------------------
// Bins far emptier or fuller than a chunk.  Where the bins hold only a few
// particles, the barriers and the fixed work of a CTA per bin are the whole time,
// and those of up to kFewParticles go by a warp each: 200k particles, one in ten
// cells, P2G on 4^3 / 8^3 leaves 353 / 354 -> 151 / 162 us (a CTA per whole leaf
// had taken 397 / 181), G2P 106 / 109 -> 39 / 43, fused 787 / 800 -> 393 / 396.  A
// launch with few such bins (up to `per_cta` for each of its CTAs) takes them like
// the others: a warp alone needs longer for one than a CTA, and fused G2P2G, where
// a particle that has left its bin costs the warp a step of its own, much longer
// (200k particles in 3,600 bins, 1,500 of them such, moved by half a cell: 245 us,
// all by CTAs 199; 200k in 10,500 such bins 291 and 399).
// With at most half as many bins as CTAs, several share a bin, each with its
// chunks of it: 1M particles in 61 bins, P2G 267 -> 116 us, G2P 124 -> 54.
// ---------------------------------------------------------------------------

// The bins of the last binned P2G as a launch takes them: `all` by CTAs (the
// first `used` from the front of the list, the rest from its back), `parts` CTAs
// to a bin, and the `few` others by warps.
struct BinSplit {
    int used, all, few, last, parts;
};
// extra: other work that a CTA takes like a bin.
__device__ __forceinline__ BinSplit bin_split(const Ctrl *ctrl, int R, int L, int extra, int per_cta)
{
    BinSplit b;
    const int few = ctrl->bins_few;
    b.used = ctrl->bins_used;
    b.few = few <= per_cta * (int)gridDim.x ? 0 : few;
    b.all = b.used + few - b.few;
    b.last = (int)p2g_bins(R, L == 8 ? 3 : 2) - 1;
    const int n = b.all + extra;
    b.parts = n > 0 && 2 * n <= (int)gridDim.x ? (int)gridDim.x / n : 1;
    return b;
}
__device__ __forceinline__ int nth_bin(const int32_t *list, const BinSplit &b, int l)
{
    return list[l < b.used ? l : b.last - (l - b.used)];
}

// G2P of the particle at (x, y, z) (the same in all lanes) by a warp: lane (a,
// b, c) < 27 reads its node from the grid (0 outside the domain or the leaves).
template <int L, bool APIC>
__device__ __forceinline__ void g2p_by_warp(const DevGrid &g, const float *f0, const float *f1, const float *f2, float x,
                                            float y, float z, float (&u)[3], float (&c)[9])
{
    const int lane = lane_id(), a = lane / 9, b = (lane / 3) % 3, e = lane % 3, N = g.N;
    const Spline sx = bspline(x, N), sy = bspline(y, N), sz = bspline(z, N);
    float t[12] = {};
    const int i = sx.base + a, j = sy.base + b, k = sz.base + e;
    if (lane < 27 && (unsigned)i < (unsigned)N && (unsigned)j < (unsigned)N && (unsigned)k < (unsigned)N) {
        const int bs = block_slot<L>(g.root, g.R, i >> 2, j >> 2, k >> 2);
        if (bs >= 0) {
            const long long idx = block_voxel<L>(bs, i & 3, j & 3, k & 3);
            const float w = bs_eval(bs_poly(a), sx.fx) * bs_eval(bs_poly(b), sy.fx) * bs_eval(bs_poly(e), sz.fx);
            const float wv[3] = {w * f0[idx], w * f1[idx], w * f2[idx]};
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                t[q] = wv[q];
                if (APIC) {
                    t[3 + 3 * q] = (float)a * wv[q];
                    t[4 + 3 * q] = (float)b * wv[q];
                    t[5 + 3 * q] = (float)e * wv[q];
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < (APIC ? 12 : 3); ++q) t[q] = warp_sum(t[q]);
#pragma unroll
    for (int q = 0; q < 3; ++q) u[q] = t[q];
    if (APIC) {
        const float s4 = 4.f * (float)N, fx[3] = {sx.fx, sy.fx, sz.fx};
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int f = 0; f < 3; ++f) c[3 * q + f] = s4 * fmaf(-fx[f], u[q], t[3 + 3 * q + f]);
    }
}

// G2P of the warp's particles (lanes 0 .. cnt - 1, positions x) of the bin of
// block (bi, bj, bk): the bin's 6^3 nodes are staged in s, a particle that has
// left the bin's cells goes by the whole warp.
template <int L, bool APIC>
__device__ __forceinline__ void g2p_of_bin(const DevGrid &g, const float *f0, const float *f1, const float *f2, int bi, int bj,
                                           int bk, int cnt, const float (&x)[3], float4 *s, float (&u)[3], float (&c)[9])
{
    const int lane = lane_id(), N = g.N;
    const int slot = lane < 8 ? block_slot<L>(g.root, g.R, bi + (lane >> 2), bj + ((lane >> 1) & 1), bk + (lane & 1)) : -1;
#pragma unroll
    for (int h = 0; h < 7; ++h) {
        const int nd = h * 32 + lane;
        int i, j, k, blk, l;
        bin_node(nd, i, j, k, blk, l);
        const int bs = __shfl_sync(kFull, slot, blk & 7);
        if (nd >= kBinNodes) continue;
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        if (bs >= 0) {
            const long long idx = block_voxel<L>(bs, i & 3, j & 3, k & 3);
            t = make_float4(f0[idx], f1[idx], f2[idx], 0.f);
        }
        s[nd] = t;
    }
    __syncwarp();
    const Spline sx = bspline(x[0], N), sy = bspline(x[1], N), sz = bspline(x[2], N);
    const int ri = sx.base - 4 * bi, rj = sy.base - 4 * bj, rk = sz.base - 4 * bk;
    const bool in = lane < cnt && (unsigned)ri < 4u && (unsigned)rj < 4u && (unsigned)rk < 4u;
    if (in) {
        float3 t;
        g2p_from_block<6, APIC>(s, ri, rj, rk, N, sx, sy, sz, t, c);
        u[0] = t.x;
        u[1] = t.y;
        u[2] = t.z;
    }
    for (unsigned stray = __ballot_sync(kFull, lane < cnt && !in); stray; stray &= stray - 1) {
        const int t = __ffs(stray) - 1;
        float us[3], cs[9];
        g2p_by_warp<L, APIC>(g, f0, f1, f2, __shfl_sync(kFull, x[0], t), __shfl_sync(kFull, x[1], t),
                             __shfl_sync(kFull, x[2], t), us, cs);
        if (lane == t) {
#pragma unroll
            for (int e = 0; e < 3; ++e) u[e] = us[e];
            if (APIC) {
#pragma unroll
                for (int e = 0; e < 9; ++e) c[e] = cs[e];
            }
        }
    }
    __syncwarp();
}

// A lane's particle for P2G: base node, spline offsets, q = v - M f and M = dx C.
template <bool APIC>
struct FewParticle {
    int b[3];
    float f[3], q[3], m[APIC ? 9 : 1];
};
template <bool APIC>
__device__ __forceinline__ void few_particle(FewParticle<APIC> &r, float x, float y, float z, const float (&v)[3],
                                             const float (&C)[9], int N)
{
    const Spline sx = bspline(x, N), sy = bspline(y, N), sz = bspline(z, N);
    r.b[0] = sx.base;
    r.b[1] = sy.base;
    r.b[2] = sz.base;
    r.f[0] = sx.fx;
    r.f[1] = sy.fx;
    r.f[2] = sz.fx;
    const float dx = 1.f / (float)N;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        r.q[e] = v[e];
        if (APIC) {
#pragma unroll
            for (int f = 0; f < 3; ++f) r.m[APIC ? 3 * e + f : 0] = dx * C[3 * e + f];
            r.q[e] -= r.m[APIC ? 3 * e : 0] * sx.fx + r.m[APIC ? 3 * e + 1 : 0] * sy.fx + r.m[APIC ? 3 * e + 2 : 0] * sz.fx;
        }
    }
}

// Its contribution (weight, weighted velocity) to node b + (a, b, c).
template <bool APIC>
__device__ __forceinline__ float4 few_node(const FewParticle<APIC> &r, int a, int b, int c)
{
    const float w = bs_eval(bs_poly(a), r.f[0]) * bs_eval(bs_poly(b), r.f[1]) * bs_eval(bs_poly(c), r.f[2]);
    float u[3];
#pragma unroll
    for (int e = 0; e < 3; ++e)
        u[e] = APIC ? fmaf(r.m[APIC ? 3 * e : 0], (float)a,
                           fmaf(r.m[APIC ? 3 * e + 1 : 0], (float)b, fmaf(r.m[APIC ? 3 * e + 2 : 0], (float)c, r.q[e])))
                    : r.q[e];
    return make_float4(w, w * u[0], w * u[1], w * u[2]);
}

// Lane t's particle, in every lane.
template <bool APIC>
__device__ __forceinline__ FewParticle<APIC> few_of(const FewParticle<APIC> &r, int t)
{
    FewParticle<APIC> o;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        o.b[e] = __shfl_sync(kFull, r.b[e], t);
        o.f[e] = __shfl_sync(kFull, r.f[e], t);
        o.q[e] = __shfl_sync(kFull, r.q[e], t);
    }
    if (APIC) {
#pragma unroll
        for (int e = 0; e < (APIC ? 9 : 1); ++e) o.m[e] = __shfl_sync(kFull, r.m[e], t);
    }
    return o;
}

// Scratch of a warp: the sums of the bin's 6^3 nodes, the occupied cells of its
// 16 columns.
constexpr int kFewScratch = kBinNodes + 4;  // float4

// The sums, in s[node], of those of the warp's particles (lanes 0 .. cnt - 1)
// whose base is in the bin's cells o .. o + 3; returns the lanes of the others.
template <bool APIC>
__device__ __forceinline__ unsigned few_sums(const FewParticle<APIC> &r, int cnt, int oi, int oj, int ok, float4 *s)
{
    const int lane = lane_id(), a = lane / 9, b = (lane / 3) % 3, c = lane % 3;
    uint32_t *cells = reinterpret_cast<uint32_t *>(s + kBinNodes);
    for (int q = lane; q < kBinNodes; q += 32) s[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (lane < 16) cells[lane] = 0;
    const int ri = r.b[0] - oi, rj = r.b[1] - oj, rk = r.b[2] - ok;
    const bool in = (unsigned)ri < 4u && (unsigned)rj < 4u && (unsigned)rk < 4u;
    __syncwarp();
    if (lane < cnt && in) atomicOr(&cells[ri * 4 + rj], 1u << rk);
    for (unsigned ins = __ballot_sync(kFull, lane < cnt && in); ins; ins &= ins - 1) {
        const FewParticle<APIC> o = few_of<APIC>(r, __ffs(ins) - 1);
        const float4 add = few_node<APIC>(o, a, b, c);
        if (lane < 27) {
            float4 &n = s[((o.b[0] - oi + a) * 6 + o.b[1] - oj + b) * 6 + o.b[2] - ok + c];
            n = make_float4(n.x + add.x, n.y + add.y, n.z + add.z, n.w + add.w);
        }
        __syncwarp();
    }
    return __ballot_sync(kFull, lane < cnt && !in);
}

// put(i, j, k, t) for each node of each of the others.
template <bool APIC, typename F>
__device__ __forceinline__ void few_strays(const FewParticle<APIC> &r, unsigned strays, F &&put)
{
    const int lane = lane_id(), a = lane / 9, b = (lane / 3) % 3, c = lane % 3;
    for (; strays; strays &= strays - 1) {
        const FewParticle<APIC> o = few_of<APIC>(r, __ffs(strays) - 1);
        if (lane < 27) put(o.b[0] + a, o.b[1] + b, o.b[2] + c, few_node<APIC>(o, a, b, c));
    }
}

// Does any of them hold bin node (i, j, k) in its stencil?
__device__ __forceinline__ bool few_hit(const float4 *s, int i, int j, int k)
{
    const uint32_t *cells = reinterpret_cast<const uint32_t *>(s + kBinNodes);
    uint32_t m = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            if ((unsigned)(i - a) <= 3u && (unsigned)(j - b) <= 3u) m |= cells[(i - a) * 4 + (j - b)];
    return (((m | (m << 1) | (m << 2)) >> k) & 1u) != 0u;
}

// Set the bit of value index idx in the mask; whether it is new.
__device__ __forceinline__ bool set_bit(const DevGrid &g, long long idx)
{
    uint32_t *mw = g.mask + (idx >> 5);
    const uint32_t bit = 1u << (idx & 31);
    return !(*(volatile uint32_t *)mw & bit) && !(atomicOr(mw, bit) & bit);
}

}  // namespace sg

// sg_advect.cu -- MacCormack advection with RK3 path integration over the
// sparse grid (AsyncTaichi Sec. 8.2): semi-Lagrangian advection of up to
// three channels per launch sharing one backtrace, and the backward advection
// fused with the MacCormack correction (the intermediate q~ kept in registers
// unless a later op reads it).
//
// Collocated grid: voxel (i,j,k) sits at (i+0.5, j+0.5, k+0.5) in cell units;
// velocities are in domain units per time, h = dt * N cells per unit
// velocity.  A sample between cells is trilinear over the 8 surrounding cell
// centres; each value is read from its leaf found through the list entry's
// 27-neighbour table (a null or out-of-domain neighbour is the zero leaf, and
// a stored value at an inactive voxel is 0, so every read is unconditional),
// or through the root when the sample lies more than a leaf away.  A warp's 32
// voxels lie in one leaf (L^3 is a multiple of 32), so the warp copies the
// entry's table to shared memory once and every lookup is a shared load;
// element offsets are 32-bit when the fields have fewer than 2^31 elements.
// With fusion the run's velocity is first packed as one float4 (u, v, w, 0)
// per value slot, so a velocity corner is one 16-byte load instead of three
// (the same products summed in the same order: the results are identical).
// Backtrace: Ralston's RK3, x_back = x - h (2 k1 + 3 k2 + 4 k3) / 9 with
// k1 = u(x), k2 = u(x - h/2 k1), k3 = u(x - 3h/4 k2).  Correction: q' =
// q^ + (q - q~) / 2 clamped to the 8 values of q the forward sample uses.
#include "sg_common.cuh"

namespace sg {

namespace {

constexpr int kMaxAdvectChannels = 3;

struct AdvectArgs {
    int C;                            // channels
    int dst[kMaxAdvectChannels];      // outputs
    int src[kMaxAdvectChannels];      // advect: sampled field; mac: q
    int qhat[kMaxAdvectChannels];     // mac: q^
    int qtil[kMaxAdvectChannels];     // mac: q~ (fused: its output, -1 = not stored)
    int v0;                           // velocity fields v0 .. v0+2
    float h;                          // dt * N (the forward step)
    // clamp bounds of the correction, per channel: written by an advection
    // (the min and max of the 8 values its sample reads) and read by the
    // correction of the same q, velocity and step instead of tracing again
    float *lo[kMaxAdvectChannels];
    float *hi[kMaxAdvectChannels];
    const float4 *vel4;               // packed velocity, or null (read the three fields)
    const uint32_t *vmax;             // with k_advect_block: the largest packed component (see below)
};

// Does every voxel move by less than a cell over h?  k_advect_block runs if so
// and k_advect if not; both are launched and the other returns at once (vmax:
// bits of a non-negative float, a NaN above all).  Longer steps leave the staged
// block, and a voxel that does is traced twice: with the block kernel alone
// three channels on the 256^3 tube took 352 us a step up to a cell, 485 at 1.6
// cells and 692 at 5 (k_advect: 405, 405 and 410; with the choice 355, 403 and
// 405).  The results are the same either way, so a largest component left over
// from an earlier packing costs time only.
__device__ __forceinline__ bool steps_within_a_cell(const AdvectArgs &A)
{
    return __uint_as_float(*A.vmax) * fabsf(A.h) < 1.f;
}

// Slot of the leaf holding cell (ci, cj, ck), relative to the list entry's
// leaf (bi, bj, bk): through the neighbour table within one leaf, else the root.
template <int L>
__device__ __forceinline__ int leaf_slot(const DevGrid &g, const int32_t *nb, int bi, int bj, int bk, int ci, int cj,
                                         int ck)
{
    constexpr int LG2 = (L == 8) ? 3 : 2;
    const int di = (ci >> LG2) - bi, dj = (cj >> LG2) - bj, dk = (ck >> LG2) - bk;
    if ((unsigned)(di + 1) <= 2u && (unsigned)(dj + 1) <= 2u && (unsigned)(dk + 1) <= 2u)
        return __ldg(nb + (di + 1) * 9 + (dj + 1) * 3 + (dk + 1));
    if ((unsigned)ci >= (unsigned)g.N || (unsigned)cj >= (unsigned)g.N || (unsigned)ck >= (unsigned)g.N)
        return (int)g.cap;  // out of the domain: the zero leaf
    const int s = __ldg(g.root + ((long long)(ci >> LG2) * g.R + (cj >> LG2)) * g.R + (ck >> LG2));
    return s < 0 ? (int)g.cap : s;
}

// The 8 corners of a sample at p (cell units): their value offsets within a
// field and trilinear weights.
template <int L, typename Off>
struct Corners {
    Off off[8];
    float w[8];
};

// tab: the warp's copy of the list entry's neighbour table (shared memory).
template <int L, typename Off>
__device__ __forceinline__ void corners(const DevGrid &g, const int32_t *nb, const int *tab, int bi, int bj, int bk,
                                        float px, float py, float pz, Corners<L, Off> &cr)
{
    constexpr int LG2 = (L == 8) ? 3 : 2;
    const float X = px - 0.5f, Y = py - 0.5f, Z = pz - 0.5f;
    const float fx0 = floorf(X), fy0 = floorf(Y), fz0 = floorf(Z);
    const int i0 = (int)fx0, j0 = (int)fy0, k0 = (int)fz0;
    const float fx = X - fx0, fy = Y - fy0, fz = Z - fz0;
    // per axis: the leaf offsets (relative to the entry's leaf) and local indices
    // of the two corner layers
    const int di0 = (i0 >> LG2) - bi, dj0 = (j0 >> LG2) - bj, dk0 = (k0 >> LG2) - bk;
    const int di1 = ((i0 + 1) >> LG2) - bi, dj1 = ((j0 + 1) >> LG2) - bj, dk1 = ((k0 + 1) >> LG2) - bk;
    const int li[2] = {i0 & (L - 1), (i0 + 1) & (L - 1)}, lj[2] = {j0 & (L - 1), (j0 + 1) & (L - 1)},
              lk[2] = {k0 & (L - 1), (k0 + 1) & (L - 1)};
    const float wx[2] = {1.f - fx, fx}, wy[2] = {1.f - fy, fy}, wz[2] = {1.f - fz, fz};
    // within the 27-neighbourhood (the common case): the table entry; lanes
    // whose sample lies further out take the root afterwards
    const bool near = di0 >= -1 && di1 <= 1 && dj0 >= -1 && dj1 <= 1 && dk0 >= -1 && dk1 <= 1;
    const int ti[2] = {near ? (di0 + 1) * 9 : 0, near ? (di1 + 1) * 9 : 0},
              tj[2] = {near ? (dj0 + 1) * 3 : 0, near ? (dj1 + 1) * 3 : 0}, tk[2] = {near ? dk0 + 1 : 0, near ? dk1 + 1 : 0};
    int slot[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) slot[c] = tab[ti[c >> 2] + tj[(c >> 1) & 1] + tk[c & 1]];
    if (!near) {
#pragma unroll
        for (int c = 0; c < 8; ++c)
            slot[c] = leaf_slot<L>(g, nb, bi, bj, bk, i0 + (c >> 2), j0 + ((c >> 1) & 1), k0 + (c & 1));
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int a = c >> 2, b = (c >> 1) & 1, d = c & 1;
        cr.off[c] = ((Off)slot[c] << (3 * LG2)) + (Off)((((li[a] << LG2) + lj[b]) << LG2) + lk[d]);
        cr.w[c] = wx[a] * wy[b] * wz[d];
    }
}

template <int L, typename Off>
__device__ __forceinline__ float sample(const float *__restrict__ f, const Corners<L, Off> &cr)
{
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) s = fmaf(cr.w[c], __ldg(f + cr.off[c]), s);
    return s;
}

template <int L, typename Off, bool PK>
__device__ __forceinline__ void velocity(const DevGrid &g, const int32_t *nb, const int *tab, int bi, int bj, int bk, int v0,
                                         const float4 *__restrict__ vel4, float px, float py, float pz, float (&u)[3])
{
    Corners<L, Off> cr;
    corners<L, Off>(g, nb, tab, bi, bj, bk, px, py, pz, cr);
    if (PK) {
        u[0] = u[1] = u[2] = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float4 w = __ldg(vel4 + cr.off[c]);
            u[0] = fmaf(cr.w[c], w.x, u[0]);
            u[1] = fmaf(cr.w[c], w.y, u[1]);
            u[2] = fmaf(cr.w[c], w.z, u[2]);
        }
    } else {
#pragma unroll
        for (int a = 0; a < 3; ++a) u[a] = sample<L, Off>(g.field[v0 + a], cr);
    }
}

// RK3 backtrace of cell centre x over h; returns the corners of the sample.
// k1 = u(x) at the cell centre itself is the voxel's stored velocity (the
// trilinear weights there are 1, 0, ..., 0), read directly at idx.
template <int L, typename Off, bool PK>
__device__ __forceinline__ void backtrace(const DevGrid &g, const int32_t *nb, const int *tab, int bi, int bj, int bk, int v0,
                                          const float4 *__restrict__ vel4, float h, const float (&x)[3], Off idx,
                                          Corners<L, Off> &cr)
{
    float k1[3], k2[3], k3[3];
    if (PK) {
        const float4 w = __ldg(vel4 + idx);
        k1[0] = w.x;
        k1[1] = w.y;
        k1[2] = w.z;
    } else {
#pragma unroll
        for (int a = 0; a < 3; ++a) k1[a] = g.field[v0 + a][idx];
    }
    velocity<L, Off, PK>(g, nb, tab, bi, bj, bk, v0, vel4, x[0] - 0.5f * h * k1[0], x[1] - 0.5f * h * k1[1],
                     x[2] - 0.5f * h * k1[2], k2);
    velocity<L, Off, PK>(g, nb, tab, bi, bj, bk, v0, vel4, x[0] - 0.75f * h * k2[0], x[1] - 0.75f * h * k2[1],
                     x[2] - 0.75f * h * k2[2], k3);
    const float c = h / 9.f;
    corners<L, Off>(g, nb, tab, bi, bj, bk, x[0] - c * (2.f * k1[0] + 3.f * k2[0] + 4.f * k3[0]),
                    x[1] - c * (2.f * k1[1] + 3.f * k2[1] + 4.f * k3[1]),
                    x[2] - c * (2.f * k1[2] + 3.f * k2[2] + 4.f * k3[2]), cr);
}

// MODE 0: advect (dst = src at the backtrace over h); with BND the clamp
//         bounds of each channel's sample are stored in A.lo / A.hi;
// MODE 1: backward advect of q^ over -h fused with the correction;
// MODE 2: correction alone (q~ read from its field).
// In modes 1 and 2, BND reads the clamp bounds from A.lo / A.hi instead of
// tracing the forward path again.
// PK: the velocity is read from A.vel4 (packed).  Four CTAs per SM (at most
// 64 registers a thread): the traces are latency-bound.
// One active voxel (local index l of the leaf at list entry e, value index
// idx); tab: the entry's neighbour table in shared memory.
template <int L, int C, int MODE, bool BND, typename Off, bool PK>
__device__ __forceinline__ void advect_voxel(const DevGrid &g, const AdvectArgs &A, long long e, int l, Off idx,
                                             const int *tab)
{
    constexpr int LG2 = (L == 8) ? 3 : 2;
    const int R = g.R;
    const int32_t *nb = g.nbr + e * 27;
    const int b = g.list_b[e];
    const int bi = b / (R * R), bj = (b / R) % R, bk = b % R;
    const float x[3] = {(float)((bi << LG2) + (l >> (2 * LG2))) + 0.5f,
                        (float)((bj << LG2) + ((l >> LG2) & (L - 1))) + 0.5f,
                        (float)((bk << LG2) + (l & (L - 1))) + 0.5f};
    Corners<L, Off> fw;
    if (MODE == 0 || !BND) backtrace<L, Off, PK>(g, nb, tab, bi, bj, bk, A.v0, A.vel4, A.h, x, idx, fw);
    if (MODE == 0) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const float *sf = g.field[A.src[c]];
            if constexpr (!BND) {
                g.field[A.dst[c]][idx] = sample<L, Off>(sf, fw);
            } else {
                float v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = __ldg(sf + fw.off[k]);
                float smp = 0.f, lo = v[0], hi = v[0];
#pragma unroll
                for (int k = 0; k < 8; ++k) smp = fmaf(fw.w[k], v[k], smp);  // the order of sample()
#pragma unroll
                for (int k = 1; k < 8; ++k) {
                    lo = fminf(lo, v[k]);
                    hi = fmaxf(hi, v[k]);
                }
                g.field[A.dst[c]][idx] = smp;
                A.lo[c][idx] = lo;
                A.hi[c][idx] = hi;
            }
        }
        return;
    }
    float qt[C];
    if (MODE == 1) {
        Corners<L, Off> bw;
        backtrace<L, Off, PK>(g, nb, tab, bi, bj, bk, A.v0, A.vel4, -A.h, x, idx, bw);
#pragma unroll
        for (int c = 0; c < C; ++c) {
            qt[c] = sample<L, Off>(g.field[A.qhat[c]], bw);
            if (A.qtil[c] >= 0) g.field[A.qtil[c]][idx] = qt[c];
        }
    } else {
#pragma unroll
        for (int c = 0; c < C; ++c) qt[c] = g.field[A.qtil[c]][idx];
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const float *qf = g.field[A.src[c]];
        float lo, hi;
        if (BND) {
            lo = A.lo[c][idx];
            hi = A.hi[c][idx];
        } else {
            lo = __ldg(qf + fw.off[0]);
            hi = lo;
#pragma unroll
            for (int k = 1; k < 8; ++k) {
                const float v = __ldg(qf + fw.off[k]);
                lo = fminf(lo, v);
                hi = fmaxf(hi, v);
            }
        }
        const float r = g.field[A.qhat[c]][idx] + 0.5f * (qf[idx] - qt[c]);
        g.field[A.dst[c]][idx] = fminf(fmaxf(r, lo), hi);
    }
}

template <int L, int C, int MODE, bool BND, typename Off, bool PK>
__global__ void __launch_bounds__(256, 4) k_advect(DevGrid g, AdvectArgs A)
{
    chained_entry();
    if (L == 8 && PK && A.vmax && steps_within_a_cell(A)) return;
    constexpr int V = L * L * L, LG2 = (L == 8) ? 3 : 2;
    const long long n = g.ctrl->list_n;
    __shared__ int s_nb[8][27];
    // the loop bound is a multiple of 32 and the stride a multiple of 256, so
    // a warp's lanes share one list entry per iteration and all reach the
    // __syncwarp() around the copy of its table
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * V;
         q += (long long)gridDim.x * blockDim.x) {
        const long long e = q >> (3 * LG2);
        const int l = (int)(q & (V - 1));
        const int slot = g.list_slot[e];
        const Off idx = ((Off)slot << (3 * LG2)) + (Off)l;
        const bool act = (g.mask[(long long)slot * g.W + (l >> 5)] >> (l & 31)) & 1u;
        int *tab = s_nb[threadIdx.x >> 5];
        __syncwarp();
        if (lane_id() < 27) tab[lane_id()] = __ldg(g.nbr + e * 27 + lane_id());
        __syncwarp();
        if (!act) {  // inactive voxels keep 0
#pragma unroll
            for (int c = 0; c < C; ++c) {
                g.field[A.dst[c]][idx] = 0.f;
                if (MODE == 1 && A.qtil[c] >= 0) g.field[A.qtil[c]][idx] = 0.f;
            }
            continue;
        }
        advect_voxel<L, C, MODE, BND, Off, PK>(g, A, e, l, idx, tab);
    }
}

// ---------------------------------------------------------------------------
// The traces over 8^3 leaves with the packed velocity, a CTA per leaf: the
// velocity and the sampled channels of the 10^3 cells from one before the leaf
// to one past it are staged in shared memory (the neighbour table is looked up
// once per cell), so a sample's corners are eight fixed offsets from one index
// instead of eight slot lookups and address sums.  A voxel whose trace leaves
// the block (a step of a cell or more) takes the path above.  Same operands in
// the same order as there: the results are identical.  What bounds it is the
// shared-memory pipe (84 % in mode 0: 16 four-word and 8 C one-word reads a
// voxel) and, in mode 1, the bounds and channels read from HBM.  256^3 tube, 3
// channels: forward 165 -> 144 us, backward 201 -> 169 us, six steps and the
// reads 2790 -> 2513 us.  Five CTAs of 48 registers per SM: four of 64 took 154
// and 194 us.  The velocity as 8 + 4 bytes in rows 24 words apart (no bank
// conflicts, fewer accesses) took 2610 us: more loads, more spills.
// ---------------------------------------------------------------------------
constexpr int kBlk = 10, kBlkCells = kBlk * kBlk * kBlk;

struct BlockSample {
    int at;  // index of the low corner in the block
    float w[8];
};

__device__ __forceinline__ constexpr int blk_corner(int c) { return (c >> 2) * kBlk * kBlk + ((c >> 1) & 1) * kBlk + (c & 1); }

// The sample at p (cell units); o: the block's first cell.  False (and index
// 0) if a corner lies outside the block.
__device__ __forceinline__ bool block_sample(float px, float py, float pz, int oi, int oj, int ok, BlockSample &b)
{
    const float X = px - 0.5f, Y = py - 0.5f, Z = pz - 0.5f;
    const float fx0 = floorf(X), fy0 = floorf(Y), fz0 = floorf(Z);
    const int i = (int)fx0 - oi, j = (int)fy0 - oj, k = (int)fz0 - ok;
    const float fx = X - fx0, fy = Y - fy0, fz = Z - fz0;
    const float wx[2] = {1.f - fx, fx}, wy[2] = {1.f - fy, fy}, wz[2] = {1.f - fz, fz};
    const bool in = (unsigned)i <= (unsigned)(kBlk - 2) && (unsigned)j <= (unsigned)(kBlk - 2) && (unsigned)k <= (unsigned)(kBlk - 2);
    b.at = in ? (i * kBlk + j) * kBlk + k : 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) b.w[c] = wx[c >> 2] * wy[(c >> 1) & 1] * wz[c & 1];
    return in;
}

__device__ __forceinline__ void block_velocity(const float4 *s_v, const BlockSample &b, float (&u)[3])
{
    u[0] = u[1] = u[2] = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float4 w = s_v[b.at + blk_corner(c)];
        u[0] = fmaf(b.w[c], w.x, u[0]);
        u[1] = fmaf(b.w[c], w.y, u[1]);
        u[2] = fmaf(b.w[c], w.z, u[2]);
    }
}

template <int C, int MODE, bool BND>
__device__ __noinline__ void advect_voxel_far(const DevGrid &g, const AdvectArgs &A, long long e, int l, int idx,
                                              const int *tab)
{
    advect_voxel<8, C, MODE, BND, int, true>(g, A, e, l, idx, tab);
}

// MODE 0 (with BND: storing the clamp bounds) and MODE 1 with BND.
template <int C, int MODE, bool BND>
__global__ void __launch_bounds__(256, 5) k_advect_block(const __grid_constant__ DevGrid g,
                                                         const __grid_constant__ AdvectArgs A)
{
    chained_entry();
    __shared__ float4 s_v[kBlkCells];
    __shared__ float s_q[C][kBlkCells];
    __shared__ int s_nb[27];
    if (!steps_within_a_cell(A)) return;
    const int n = g.ctrl->list_n, R = g.R, tid = threadIdx.x;
    const float h = MODE == 0 ? A.h : -A.h;
    int nb = tid < 27 && (int)blockIdx.x < n ? g.nbr[blockIdx.x * 27LL + tid] : 0;  // an entry ahead
    for (int e = blockIdx.x; e < n; e += gridDim.x) {
        if (tid < 27) s_nb[tid] = nb;
        const int next = e + (int)gridDim.x;
        if (tid < 27 && next < n) nb = g.nbr[next * 27LL + tid];
        const int b = g.list_b[e], bij = b / R, bi = bij / R;
        const int oi = bi * 8 - 1, oj = (bij - bi * R) * 8 - 1, ok = (b - bij * R) * 8 - 1;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < (kBlkCells + 255) / 256; ++r) {
            const int q = tid + r * 256;
            if (q < kBlkCells) {
                // cell q of the block, from the 24^3 cells of the 27 leaves
                const int i = q / (kBlk * kBlk) + 7, j = q / kBlk % kBlk + 7, k = q % kBlk + 7;
                const int off = (s_nb[(i >> 3) * 9 + (j >> 3) * 3 + (k >> 3)] << 9) + (((i & 7) << 6) | ((j & 7) << 3) | (k & 7));
                s_v[q] = __ldg(A.vel4 + off);
#pragma unroll
                for (int c = 0; c < C; ++c) s_q[c][q] = __ldg(g.field[MODE == 0 ? A.src[c] : A.qhat[c]] + off);
            }
        }
        __syncthreads();
        const int slot = s_nb[13];
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            const int l = half * 256 + tid, idx = (slot << 9) + l;
            if (!((g.mask[(long long)slot * 16 + (l >> 5)] >> (l & 31)) & 1u)) {  // inactive voxels keep 0
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    g.field[A.dst[c]][idx] = 0.f;
                    if (MODE == 1 && A.qtil[c] >= 0) g.field[A.qtil[c]][idx] = 0.f;
                }
                continue;
            }
            const int li = l >> 6, lj = (l >> 3) & 7, lk = l & 7, own = ((li + 1) * kBlk + lj + 1) * kBlk + lk + 1;
            const float x0 = (float)(oi + 1 + li) + 0.5f, x1 = (float)(oj + 1 + lj) + 0.5f, x2 = (float)(ok + 1 + lk) + 0.5f;
            const float4 k1 = s_v[own];
            BlockSample bs;
            float k2[3], k3[3];
            bool in = block_sample(x0 - 0.5f * h * k1.x, x1 - 0.5f * h * k1.y, x2 - 0.5f * h * k1.z, oi, oj, ok, bs);
            block_velocity(s_v, bs, k2);
            in &= block_sample(x0 - 0.75f * h * k2[0], x1 - 0.75f * h * k2[1], x2 - 0.75f * h * k2[2], oi, oj, ok, bs);
            block_velocity(s_v, bs, k3);
            const float c9 = h / 9.f;
            in &= block_sample(x0 - c9 * (2.f * k1.x + 3.f * k2[0] + 4.f * k3[0]),
                               x1 - c9 * (2.f * k1.y + 3.f * k2[1] + 4.f * k3[1]),
                               x2 - c9 * (2.f * k1.z + 3.f * k2[2] + 4.f * k3[2]), oi, oj, ok, bs);
            if (!in) {
                advect_voxel_far<C, MODE, BND>(g, A, e, l, idx, s_nb);
                continue;
            }
#pragma unroll
            for (int c = 0; c < C; ++c) {
                float v[8], smp = 0.f;
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = s_q[c][bs.at + blk_corner(k)];
#pragma unroll
                for (int k = 0; k < 8; ++k) smp = fmaf(bs.w[k], v[k], smp);  // the order of sample()
                if (MODE == 0) {
                    g.field[A.dst[c]][idx] = smp;
                    if (BND) {
                        float lo = v[0], hi = v[0];
#pragma unroll
                        for (int k = 1; k < 8; ++k) {
                            lo = fminf(lo, v[k]);
                            hi = fmaxf(hi, v[k]);
                        }
                        A.lo[c][idx] = lo;
                        A.hi[c][idx] = hi;
                    }
                } else {
                    if (A.qtil[c] >= 0) g.field[A.qtil[c]][idx] = smp;
                    const float r = s_q[c][own] + 0.5f * (g.field[A.src[c]][idx] - smp);
                    g.field[A.dst[c]][idx] = fminf(fmaxf(r, A.lo[c][idx]), A.hi[c][idx]);
                }
            }
        }
        __syncthreads();  // the block is refilled for the next leaf
    }
}

template <int L, int MODE, bool BND, typename Off, bool PK>
void launch_LBO(const DevGrid &g, cudaStream_t s, const AdvectArgs &a, int ctas)
{
    if (a.C == 1) launch_chained(k_advect<L, 1, MODE, BND, Off, PK>, ctas, 256, 0, s, g, a);
    else if (a.C == 2) launch_chained(k_advect<L, 2, MODE, BND, Off, PK>, ctas, 256, 0, s, g, a);
    else launch_chained(k_advect<L, 3, MODE, BND, Off, PK>, ctas, 256, 0, s, g, a);
}

template <int MODE, bool BND>
void launch_block(const DevGrid &g, cudaStream_t s, const AdvectArgs &a, int num_sms)
{
    if (a.C == 1) launch_drained(k_advect_block<1, MODE, BND>, num_sms * 5, 256, 0, s, g, a);
    else if (a.C == 2) launch_drained(k_advect_block<2, MODE, BND>, num_sms * 5, 256, 0, s, g, a);
    else launch_drained(k_advect_block<3, MODE, BND>, num_sms * 5, 256, 0, s, g, a);
    launch_LBO<8, MODE, BND, int, true>(g, s, a, num_sms * 8);
}

template <int L, int MODE>
void launch_L(const DevGrid &g, cudaStream_t s, AdvectArgs a, int ctas)
{
    // 32-bit element offsets while every offset (the zero leaf's included)
    // fits; the packed velocity is read by the modes that trace (the fused
    // schedule's forward and backward launches) with 32-bit offsets
    const bool wide = (unsigned long long)(g.cap + 1) * (L * L * L) > 0x7fffffffull;
    if constexpr (MODE != 2) {
        if (a.vel4 && !wide) {
            if constexpr (L == 8) {
                if (a.vmax && (MODE == 0 || a.lo[0])) {
                    if constexpr (MODE == 0) {
                        if (a.lo[0]) launch_block<0, true>(g, s, a, ctas / 8);
                        else launch_block<0, false>(g, s, a, ctas / 8);
                    } else {
                        launch_block<1, true>(g, s, a, ctas / 8);
                    }
                    return;
                }
            }
            a.vmax = nullptr;
            if (a.lo[0]) launch_LBO<L, MODE, true, int, true>(g, s, a, ctas);
            else launch_LBO<L, MODE, false, int, true>(g, s, a, ctas);
            return;
        }
    }
    a.vel4 = nullptr;
    a.vmax = nullptr;
    if (a.lo[0]) {
        if (wide) launch_LBO<L, MODE, true, long long, false>(g, s, a, ctas);
        else launch_LBO<L, MODE, true, int, false>(g, s, a, ctas);
    } else {
        if (wide) launch_LBO<L, MODE, false, long long, false>(g, s, a, ctas);
        else launch_LBO<L, MODE, false, int, false>(g, s, a, ctas);
    }
}

// Packed velocity: vel4[slot * L^3 + l] = (u, v, w, 0) of fields v0..v0+2 for
// every listed leaf (the zero leaf's block is zero from its allocation), and
// the largest component in *vmax, zero before; *next is zeroed for the packing
// after this one.
template <int L>
__global__ void __launch_bounds__(256, 8) k_pack_velocity(const __grid_constant__ DevGrid g, int v0, float4 *__restrict__ vel4, uint32_t *vmax,
                                                          uint32_t *next)
{
    chained_entry();
    __shared__ uint32_t s_max[8];
    uint32_t most = 0;
    constexpr int V = L * L * L, LG2 = (L == 8) ? 3 : 2;
    const long long n = g.ctrl->list_n;
    const float *__restrict__ u = g.field[v0], *__restrict__ v = g.field[v0 + 1], *__restrict__ w = g.field[v0 + 2];
#pragma unroll 1  // unrolled it needs more than the 32 registers of eight CTAs per SM
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * V;
         q += (long long)gridDim.x * blockDim.x) {
        const long long idx = ((long long)g.list_slot[q >> (3 * LG2)] << (3 * LG2)) + (q & (V - 1));
        const float4 a = make_float4(__ldg(u + idx), __ldg(v + idx), __ldg(w + idx), 0.f);
        vel4[idx] = a;
        most = max(max(most, __float_as_uint(fabsf(a.x))), max(__float_as_uint(fabsf(a.y)), __float_as_uint(fabsf(a.z))));
    }
    most = __reduce_max_sync(kFull, most);
    if (lane_id() == 0) s_max[threadIdx.x >> 5] = most;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 1; q < 8; ++q) most = max(most, s_max[q]);
        if (most > *(volatile uint32_t *)vmax) atomicMax(vmax, most);
        if (blockIdx.x == 0) *next = 0;
    }
}

}  // namespace

void launch_pack_velocity(const DevGrid &g, cudaStream_t s, int v0, float4 *vel4, uint32_t *vmax, uint32_t *next,
                          const LaunchCfg &lc)
{
    const int ctas = lc.num_sms * 8;
    if (g.L == 8) launch_chained(k_pack_velocity<8>, ctas, 256, 0, s, g, v0, vel4, vmax, next);
    else launch_chained(k_pack_velocity<4>, ctas, 256, 0, s, g, v0, vel4, vmax, next);
}

void launch_advect_group(const DevGrid &g, cudaStream_t s, int mode, int C, const int *dst, const int *src,
                         const int *qhat, const int *qtil, int v0, float h, float *const *lo, float *const *hi,
                         const float4 *vel4, const uint32_t *vmax, const LaunchCfg &lc)
{
    AdvectArgs a{};
    a.C = C;
    for (int c = 0; c < C; ++c) {
        a.dst[c] = dst[c];
        a.src[c] = src[c];
        a.qhat[c] = qhat ? qhat[c] : -1;
        a.qtil[c] = qtil ? qtil[c] : -1;
        a.lo[c] = lo ? lo[c] : nullptr;
        a.hi[c] = hi ? hi[c] : nullptr;
    }
    a.v0 = v0;
    a.h = h;
    a.vel4 = vel4;
    a.vmax = vmax;
    const int ctas = lc.num_sms * 8;
    if (g.L == 8) {
        if (mode == 0) launch_L<8, 0>(g, s, a, ctas);
        else if (mode == 1) launch_L<8, 1>(g, s, a, ctas);
        else launch_L<8, 2>(g, s, a, ctas);
    } else {
        if (mode == 0) launch_L<4, 0>(g, s, a, ctas);
        else if (mode == 1) launch_L<4, 1>(g, s, a, ctas);
        else launch_L<4, 2>(g, s, a, ctas);
    }
}

}  // namespace sg

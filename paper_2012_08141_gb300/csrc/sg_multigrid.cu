// sg_multigrid.cu -- transfers between a grid and its half-edge coarse grid:
// restriction with activation on write, y[i // 2] += w * x[i] over the active
// fine voxels i, and prolongation x[i] += w * y[i // 2] (the multigrid pattern
// AsyncTaichi Sec. 6.3 / Fig. 13 uses to motivate activation demotion).
//
// A fine leaf (edge L, leaf cell b) maps onto one (L/2)^3 sub-block of the
// coarse leaf b >> 1 (per axis), at offset (b & 1) * L/2: the eight children
// of a coarse voxel lie in a single fine leaf, so each coarse voxel is summed
// and written by exactly one lane, without atomics.
#include "sg_common.cuh"

namespace sg {

// Mark the coarse leaves that listed fine leaves with any active voxel map to.
__global__ void k_restrict_mark(DevGrid fine, DevGrid coarse)
{
    const int n = fine.ctrl->list_n;
    const int Rf = fine.R, Rc = coarse.R;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const uint32_t *m = fine.mask + (long long)fine.list_slot[e] * fine.W;
        uint32_t any = 0;
        for (int w = 0; w < fine.W; ++w) any |= m[w];
        if (!any) continue;
        const int b = fine.list_b[e];
        const int bi = b / (Rf * Rf), bj = (b / Rf) % Rf, bk = b % Rf;
        uint8_t *nd = &coarse.need[((long long)(bi >> 1) * Rc + (bj >> 1)) * Rc + (bk >> 1)];
        if (!__ldcg(nd)) *nd = 1;
    }
}

// One group of G = min(32, H^3) lanes per fine list entry, H = L/2; lane t of
// the group owns coarse sub-block voxels t, t + G, ...  ACTIVATE: set the bit
// of every coarse voxel with an active child (the coarse leaf is allocated);
// otherwise (activation demoted) the bits are known to be set.
template <int L, bool ACTIVATE>
__global__ void __launch_bounds__(256) k_restrict(DevGrid fine, DevGrid coarse, int f_src, int f_dst, float w)
{
    chained_entry();
    constexpr int H = L / 2, NV = H * H * H, G = NV < 32 ? NV : 32, PER = NV / G, LG2 = (L == 8) ? 3 : 2;
    const int n = fine.ctrl->list_n;
    const int Rf = fine.R, Rc = coarse.R;
    const float *x = fine.field[f_src];
    float *y = coarse.field[f_dst];
    const int gid = (blockIdx.x * blockDim.x + threadIdx.x) / G, t = threadIdx.x % G;
    const int groups = gridDim.x * blockDim.x / G;
    bool changed = false;
    for (int e = gid; e < n; e += groups) {
        const int sf = fine.list_slot[e], b = fine.list_b[e];
        const int bi = b / (Rf * Rf), bj = (b / Rf) % Rf, bk = b % Rf;
        const int sc = coarse.root[((long long)(bi >> 1) * Rc + (bj >> 1)) * Rc + (bk >> 1)];
        if (sc < 0) continue;  // no active voxel in this leaf, or the coarse pool is exhausted (latched)
        const uint32_t *mf = fine.mask + (long long)sf * fine.W;
        const float *xl = x + ((long long)sf << (3 * LG2));
        const int oi = (bi & 1) * H, oj = (bj & 1) * H, ok = (bk & 1) * H;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int v = t + u * G;
            const int ci = v / (H * H), cj = (v / H) % H, ck = v % H;
            float s = 0.f;
            bool act = false;
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int row = (2 * ci + a) * L + (2 * cj + c);  // fine row (li, lj)
                    const int l0 = row * L + 2 * ck;                  // children (.., 2ck) and (.., 2ck + 1)
                    const float2 p = __ldg(reinterpret_cast<const float2 *>(xl + l0));
                    s += p.x + p.y;  // a stored value at an inactive voxel is 0
                    act |= ((__ldg(mf + (l0 >> 5)) >> (l0 & 31)) & 3u) != 0u;
                }
            if (!act) continue;
            const int lc = ((oi + ci) * L + (oj + cj)) * L + (ok + ck);
            if (ACTIVATE) {
                uint32_t *mw = coarse.mask + (long long)sc * coarse.W + (lc >> 5);
                const uint32_t bit = 1u << (lc & 31);
                if (!(*(volatile uint32_t *)mw & bit)) changed |= !(atomicOr(mw, bit) & bit);
            }
            float *yp = y + ((long long)sc << (3 * LG2)) + lc;
            *yp = fmaf(w, s, *yp);
        }
    }
    if (ACTIVATE && changed) mark_dirty(coarse);
}

// Prolongation: one thread per voxel of the listed fine leaves.
template <int L>
__global__ void __launch_bounds__(256) k_prolong(DevGrid coarse, DevGrid fine, int f_src, int f_dst, float w)
{
    chained_entry();
    constexpr int LG2 = (L == 8) ? 3 : 2, V = L * L * L;
    const long long n = fine.ctrl->list_n;
    const int Rf = fine.R, Rc = coarse.R;
    const float *y = coarse.field[f_src];
    float *x = fine.field[f_dst];
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * V;
         q += (long long)gridDim.x * blockDim.x) {
        const long long e = q >> (3 * LG2);
        const int l = (int)(q & (V - 1));
        const int sf = fine.list_slot[e];
        if (!((fine.mask[(long long)sf * fine.W + (l >> 5)] >> (l & 31)) & 1u)) continue;
        const int b = fine.list_b[e];
        const int bi = b / (Rf * Rf), bj = (b / Rf) % Rf, bk = b % Rf;
        const int sc = coarse.root[((long long)(bi >> 1) * Rc + (bj >> 1)) * Rc + (bk >> 1)];
        if (sc < 0) continue;  // the coarse voxel reads 0
        const int li = l >> (2 * LG2), lj = (l >> LG2) & (L - 1), lk = l & (L - 1);
        const int ci = ((bi & 1) * L + li) >> 1, cj = ((bj & 1) * L + lj) >> 1, ck = ((bk & 1) * L + lk) >> 1;
        // a stored value at an inactive coarse voxel is 0
        const float yv = y[((long long)sc << (3 * LG2)) + (ci * L + cj) * L + ck];
        float *xp = x + ((long long)sf << (3 * LG2)) + l;
        *xp = fmaf(w, yv, *xp);
    }
}

// Prolongation over 8^3 leaves, a warp per fine leaf: the leaf's slot, cell
// and coarse leaf are looked up once (the next leaf's slot and cell a leaf
// ahead); lane t takes float4s t, t + 32, t + 64 and t + 96 of the leaf, so a
// warp access is 512 consecutive bytes.  Float4 32 h + t is half t mod 2 of row
// (2h + t / 16, t / 2 mod 8), and its coarse voxels are two consecutive values
// of coarse row (h, t / 4 mod 4).  Each active voxel takes the same fma as in
// k_prolong.  Bound by the load latency of a leaf's chain and by L1 wavefronts:
// with 16 consecutive voxels a lane, whose accesses touch a line per lane, ten
// V-cycles of the 512^3 band took 1326 us, not 1245.
__global__ void __launch_bounds__(256) k_prolong8(DevGrid coarse, DevGrid fine, int f_src, int f_dst, float w)
{
    chained_entry();
    const int n = fine.ctrl->list_n;
    const int Rf = fine.R, Rc = coarse.R;
    const float *__restrict__ y = coarse.field[f_src];
    float *__restrict__ x = fine.field[f_dst];
    const int lane = lane_id(), half = lane & 1, cj = (lane >> 2) & 3;
    const int warps = gridDim.x * (blockDim.x >> 5);
    int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    int sn = 0, bn = 0;
    if (e < n) {
        sn = fine.list_slot[e];
        bn = fine.list_b[e];
    }
    while (e < n) {
        const int sf = sn, b = bn;
        e += warps;
        if (e < n) {
            sn = fine.list_slot[e];
            bn = fine.list_b[e];
        }
        const int bij = b / Rf, bi = bij / Rf, bj = bij - bi * Rf, bk = b - bij * Rf;
        const int sc = coarse.root[((long long)(bi >> 1) * Rc + (bj >> 1)) * Rc + (bk >> 1)];
        if (sc < 0) continue;  // the coarse voxels read 0 (warp-uniform)
        float4 *xp = reinterpret_cast<float4 *>(x + ((long long)sf << 9)) + lane;
        const uint32_t *mf = fine.mask + (long long)sf * 16 + (lane >> 3);
        const float *yp = y + ((long long)sc << 9) + (((bi & 1) * 4) * 8 + (bj & 1) * 4 + cj) * 8 + (bk & 1) * 4 + 2 * half;
        float4 v[4];
        float2 c[4];
        uint32_t bits[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            v[h] = xp[32 * h];
            c[h] = *reinterpret_cast<const float2 *>(yp + 64 * h);
            bits[h] = mf[4 * h] >> ((lane & 7) * 4);
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            if (bits[h] & 1u) v[h].x = fmaf(w, c[h].x, v[h].x);
            if (bits[h] & 2u) v[h].y = fmaf(w, c[h].x, v[h].y);
            if (bits[h] & 4u) v[h].z = fmaf(w, c[h].y, v[h].z);
            if (bits[h] & 8u) v[h].w = fmaf(w, c[h].y, v[h].w);
            if (bits[h] & 15u) xp[32 * h] = v[h];
        }
    }
}

// Restriction from 8^3 leaves, a warp per fine leaf: the fine leaf maps onto a
// 4^3 coarse sub-block, and lane t sums the coarse voxels (ci, cj, 2h) and
// (ci, cj, 2h + 1), ci = t / 8, cj = (t / 2) mod 4, h = t mod 2.  Their
// children are the k-half h of fine rows (2ci + a, 2cj + c), one float4 each;
// both rows of one a share a mask word.  The children are added in the same
// order as in k_restrict, and the two coarse voxels move as one float2.  A leaf
// is a chain of loads, so its rows and mask words are requested before its
// coarse leaf is looked up, and the next leaf's entry a leaf ahead
// (ten V-cycles of the 512^3 band 1243 -> 1200 us).
template <bool ACTIVATE>
__global__ void __launch_bounds__(256) k_restrict8(DevGrid fine, DevGrid coarse, int f_src, int f_dst, float w)
{
    chained_entry();
    const int n = fine.ctrl->list_n;
    const int Rf = fine.R, Rc = coarse.R;
    const float *__restrict__ x = fine.field[f_src];
    float *y = coarse.field[f_dst];
    const int lane = lane_id();
    const int ci = lane >> 3, cj = (lane >> 1) & 3, h = lane & 1;
    const int warps = gridDim.x * (blockDim.x >> 5);
    bool changed = false;
    int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), sn = 0, bn = 0;
    if (e < n) {
        sn = fine.list_slot[e];
        bn = fine.list_b[e];
    }
    while (e < n) {
        const int sf = sn, b = bn;
        e += warps;
        if (e < n) {
            sn = fine.list_slot[e];
            bn = fine.list_b[e];
        }
        const uint32_t *mf = fine.mask + (long long)sf * 16;
        const float *xl = x + ((long long)sf << 9);
        float4 p[2][2];
        uint32_t mw[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const int r0 = (2 * ci + a) * 8 + 2 * cj;  // fine rows r0 and r0 + 1 (c = 0, 1)
            mw[a] = __ldg(mf + (r0 >> 2));
#pragma unroll
            for (int c = 0; c < 2; ++c) p[a][c] = __ldg(reinterpret_cast<const float4 *>(xl + (r0 + c) * 8 + 4 * h));
        }
        const int bij = b / Rf, bi = bij / Rf, bj = bij - bi * Rf, bk = b - bij * Rf;
        const int sc = coarse.root[((long long)(bi >> 1) * Rc + (bj >> 1)) * Rc + (bk >> 1)];
        if (sc < 0) continue;  // no active voxel in this leaf, or the coarse pool is exhausted (latched)
        const int lc = (((bi & 1) * 4 + ci) * 8 + ((bj & 1) * 4 + cj)) * 8 + (bk & 1) * 4 + 2 * h;
        float2 *yp = reinterpret_cast<float2 *>(y + ((long long)sc << 9) + lc);
        float2 v = *yp;
        float s0 = 0.f, s1 = 0.f;
        uint32_t act = 0;  // bit kk: coarse voxel (ci, cj, 2h + kk) has an active child
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                s0 += p[a][c].x + p[a][c].y;  // a stored value at an inactive voxel is 0
                s1 += p[a][c].z + p[a][c].w;
                const uint32_t nib = (mw[a] >> (((2 * cj + c) & 3) * 8 + 4 * h)) & 0xfu;
                act |= ((nib & 3u) != 0u) | (((nib >> 2) != 0u) << 1);
            }
        if (!act) continue;
        if (ACTIVATE) {
            uint32_t *mc = coarse.mask + (long long)sc * 16 + (lc >> 5);
            const uint32_t bits = act << (lc & 31);
            if ((*(volatile uint32_t *)mc & bits) != bits) changed |= (atomicOr(mc, bits) & bits) != bits;
        }
        if (act & 1u) v.x = fmaf(w, s0, v.x);
        if (act & 2u) v.y = fmaf(w, s1, v.y);
        *yp = v;
    }
    if (ACTIVATE && changed) mark_dirty(coarse);
}

void launch_restrict_mark(const DevGrid &fine, const DevGrid &coarse, cudaStream_t s, const LaunchCfg &lc)
{
    k_restrict_mark<<<lc.num_sms * 4, 256, 0, s>>>(fine, coarse);
}

void launch_restrict(const DevGrid &fine, const DevGrid &coarse, cudaStream_t s, int f_src, int f_dst, float w,
                     bool activate, const LaunchCfg &lc)
{
    const int ctas = lc.num_sms * 8;
    if (fine.L == 8) {
        if (activate) launch_chained(k_restrict8<true>, ctas, 256, 0, s, fine, coarse, f_src, f_dst, w);
        else launch_chained(k_restrict8<false>, ctas, 256, 0, s, fine, coarse, f_src, f_dst, w);
    } else {
        if (activate) launch_chained(k_restrict<4, true>, ctas, 256, 0, s, fine, coarse, f_src, f_dst, w);
        else launch_chained(k_restrict<4, false>, ctas, 256, 0, s, fine, coarse, f_src, f_dst, w);
    }
}

void launch_prolong(const DevGrid &coarse, const DevGrid &fine, cudaStream_t s, int f_src, int f_dst, float w,
                    const LaunchCfg &lc)
{
    const int ctas = lc.num_sms * 8;
    if (fine.L == 8) launch_chained(k_prolong8, ctas, 256, 0, s, coarse, fine, f_src, f_dst, w);
    else launch_chained(k_prolong<4>, ctas, 256, 0, s, coarse, fine, f_src, f_dst, w);
}

}  // namespace sg

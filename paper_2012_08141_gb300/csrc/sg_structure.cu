// sg_structure.cu -- activation, allocation, list generation and host
// transfers of the sparse grid's structure.
//
// Paper passages: the pointer/bitmask mask states (Sec. 4 "States"),
// activation on write with zero-fill (Sec. 3.2 item 3, Fig. 4), list
// generation (Sec. 3.2 item 2) and the allocator state (Sec. 4 "States").
#include "sg_common.cuh"

namespace sg {

// ---------------------------------------------------------------------------
// Activation from the shell predicate.  Each lane of a warp tests one of up
// to 32 consecutive root cells' bounding boxes against the band; the warp
// then takes the cells that can meet it one at a time and builds their mask
// words (two rows a lane on 8^3 leaves, a ballot per 32 voxels on 4^3 ones); the
// cells with active voxels and a null pointer get new leaves (zero-filled in every
// field), and the words are ORed into the leaves.  The predicate is exact in
// 32-bit integers: |2i + 1 - N| < N <= 4096, so D < 3 * 4096^2 <
// 2^31, and lo2 / hi2 are clamped to [-1, 2^31 - 1] without changing it.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void axis_range(int i0, int L, int N, int &mn, int &mx)
{
    const int e0 = 2 * i0 + 1 - N, e1 = 2 * (i0 + L - 1) + 1 - N;
    int lo;
    if (e0 > 0) lo = e0;
    else if (e1 < 0) lo = -e1;
    else lo = (e0 & 1) ? 1 : 0;  // the progression e0, e0+2, ... crosses zero
    const int hi = (-e0 > e1) ? -e0 : e1;
    mn += lo * lo;
    mx += hi * hi;
}

__device__ __forceinline__ int clamp_pred(long long v)
{
    return v < -1 ? -1 : (v > 2147483647LL ? 2147483647 : (int)v);
}

// tube: the predicate ignores the k axis (a cylinder along k through the
// domain centre) instead of using all three.  cpw: root cells per warp (32 on
// large domains, where the lanes cull 32 cells at once and the warp's new
// leaves take their pool slots with one atomic; 1 on small ones, where a warp
// per cell keeps every cell in flight at once).
// fill_mask: the (physical) fields a newly allocated leaf is zero-filled in.
// Cell indices are 32-bit (R^3 <= 2^30).  For 8^3 leaves a lane tests two rows
// of a candidate's 64, eight k each, against one unsigned bound, and two
// neighbouring lanes' bytes make a mask word: about 150 instructions a
// candidate where a ballot per 32 voxels took 390, and issue is what bounds the
// kernel (1024^3 band 84 -> 62 us).
template <int L>
__global__ void __launch_bounds__(256) k_activate_shell(DevGrid g, long long lo2_, long long hi2_, int strict, int tube,
                                                        int cpw, uint32_t fill_mask)
{
    chained_entry();
    constexpr int LG2 = (L == 8) ? 3 : 2, W = L * L * L / 32;
    constexpr int kMaxW = 16;  // mask words of an 8^3 leaf
    __shared__ uint32_t s_bits[8][32][kMaxW];  // per warp: the mask words of its chunk's cells
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int R = g.R, N = g.N;
    const unsigned RR = (unsigned)R * (unsigned)R;
    const long long nr = (long long)R * R * R;
    const int lo2 = clamp_pred(lo2_), hi2 = clamp_pred(hi2_);
    // the predicate as one unsigned comparison: least <= D < hi2
    const bool some = !(strict && lo2 == 2147483647);
    const int least = strict && some ? lo2 + 1 : lo2;
    const bool filled = (fill_mask & ((g.F < 32 ? 1u << g.F : 0u) - 1u)) != 0u;
    const unsigned span = some && hi2 > least ? (unsigned)hi2 - (unsigned)least : 0u;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long c0 = ((long long)blockIdx.x * (blockDim.x >> 5) + warp) * cpw; c0 < nr; c0 += warps * cpw) {
        // lane q < cpw tests cell c0 + q: can its bounding box meet the band?
        bool cand = false;
        uint32_t cell = 0;  // its (i, j, k), 10 bits each (R <= 1024)
        const long long bq = c0 + lane;
        if (lane < cpw && bq < nr) {
            const unsigned b = (unsigned)bq, bi = b / RR, rem = b - bi * RR, bj = rem / (unsigned)R,
                           bk = rem - bj * (unsigned)R;
            int dmin = 0, dmax = 0;
            axis_range((int)bi * L, L, N, dmin, dmax);
            axis_range((int)bj * L, L, N, dmin, dmax);
            if (!tube) axis_range((int)bk * L, L, N, dmin, dmax);
            const bool lo_possible = strict ? (dmax > lo2) : (dmax >= lo2);
            cand = lo_possible && dmin < hi2;
            cell = (bi << 20) | (bj << 10) | bk;
        }
        // the mask words of every candidate
        bool any_bits = false;  // lane q: cell c0 + q has an active voxel
        unsigned todo = __ballot_sync(kFull, cand);
        while (todo) {
            const int q = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint32_t cq = __shfl_sync(kFull, cell, q);
            const int bi = (int)(cq >> 20), bj = (int)((cq >> 10) & 1023u), bk = (int)(cq & 1023u);
            uint32_t bits = 0;  // word w in lane 2w (8^3) or w (4^3)
            if (L == 8) {
                // rows 2 lane and 2 lane + 1 of the leaf (the same i, j and j + 1)
                const int a = 2 * (bi * 8 + (lane >> 2)) + 1 - N, c = 2 * (bj * 8 + 2 * (lane & 3)) + 1 - N;
                const int r0 = a * a + c * c - least, r1 = r0 + 4 * c + 4;  // (c + 2)^2 = c^2 + 4 c + 4
                const int d0 = 2 * bk * 8 + 1 - N;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int d = d0 + 2 * k, dd = tube ? 0 : d * d;
                    if ((unsigned)(r0 + dd) < span) bits |= 1u << k;
                    if ((unsigned)(r1 + dd) < span) bits |= 256u << k;
                }
                bits |= __shfl_down_sync(kFull, bits, 1) << 16;  // used in the even lanes
                if (!(lane & 1)) s_bits[warp][q][lane >> 1] = bits;
            } else {
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const int l = w * 32 + lane;
                    const int li = l >> (2 * LG2), lj = (l >> LG2) & (L - 1), lk = l & (L - 1);
                    const int a = 2 * (bi * L + li) + 1 - N;
                    const int c = 2 * (bj * L + lj) + 1 - N;
                    const int d = 2 * (bk * L + lk) + 1 - N;
                    const unsigned word = __ballot_sync(kFull, (unsigned)(a * a + c * c + (tube ? 0 : d * d) - least) < span);
                    if (lane == w) bits = word;
                }
                if (lane < W) s_bits[warp][q][lane] = bits;
            }
            const bool nz = __any_sync(kFull, bits != 0u);
            if (lane == q) any_bits = nz;
        }
        // new leaves for the cells with active voxels and a null pointer: one
        // pool atomic for the warp, slots by rank
        int slot = -1;
        if (any_bits) slot = g.root[c0 + lane];
        const bool need = any_bits && slot < 0;
        const unsigned needm = __ballot_sync(kFull, need);
        int first = 0;
        if (needm) {
            if (lane == 0) first = atomicAdd(&g.ctrl->pool_count, __popc(needm));
            first = __shfl_sync(kFull, first, 0);
        }
        bool fresh = false;
        if (need) {
            const int sl = first + __popc(needm & lanemask_lt());
            if (sl < g.cap) {
                slot = sl;
                fresh = true;
            } else {
                raise_error(g, kErrPool);
            }
        }
        __syncwarp();
        // per cell with active voxels: zero-fill a new leaf and publish it, or
        // OR the words into the existing leaf
        unsigned work = __ballot_sync(kFull, any_bits && slot >= 0);
        bool changed = false;
        while (work) {
            const int q = __ffs(work) - 1;
            work &= work - 1;
            const int sq = __shfl_sync(kFull, slot, q);
            const bool fq = __shfl_sync(kFull, fresh, q);
            constexpr int V = L * L * L;
            if (fq) {
                const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                if (filled)
                    for (int f = 0; f < g.F; ++f) {
                        if (!((fill_mask >> f) & 1u)) continue;
                        float4 *p = reinterpret_cast<float4 *>(g.field[f] + (long long)sq * V);
                        for (int qq = lane; qq < V / 4; qq += 32) p[qq] = z;
                    }
                if (lane < W) g.mask[(long long)sq * W + lane] = s_bits[warp][q][lane];
                changed = true;
            } else if (lane < W) {
                uint32_t *m = &g.mask[(long long)sq * W + lane];
                const uint32_t old = *m, nw = old | s_bits[warp][q][lane];
                if (nw != old) {
                    *m = nw;
                    changed = true;
                }
            }
        }
        if (fresh) g.root[c0 + lane] = slot;
        if (__any_sync(kFull, changed) && lane == 0) mark_dirty(g);
        __syncwarp();  // s_bits is reused by the next chunk
    }
}

// Cells per warp and CTAs of 8 warps: 32 cells per warp once the domain has
// enough of them to fill the GPU that way (then at most 2,432 CTAs, striding
// over the rest), else a warp per cell and a CTA per 8 cells.
static void activate_shape(long long nr, int &cpw, int &ctas)
{
    constexpr long long kMaxCtas = 2432;
    cpw = nr >= kMaxCtas * 8 * 32 / 2 ? 32 : 1;
    const long long want = (nr + 8LL * cpw - 1) / (8LL * cpw);
    ctas = (int)(cpw == 1 ? (want > 0 ? want : 1) : (want < kMaxCtas ? want : kMaxCtas));
}

void launch_activate_shell(const DevGrid &g, cudaStream_t s, long long lo2, long long hi2, int strict,
                           uint32_t fill_mask)
{
    const long long nr = (long long)g.R * g.R * g.R;
    int cpw, ctas;
    activate_shape(nr, cpw, ctas);
    if (g.L == 8) launch_chained(k_activate_shell<8>, ctas, 256, 0, s, g, lo2, hi2, strict, 0, cpw, fill_mask);
    else launch_chained(k_activate_shell<4>, ctas, 256, 0, s, g, lo2, hi2, strict, 0, cpw, fill_mask);
}

void launch_activate_tube(const DevGrid &g, cudaStream_t s, long long lo2, long long hi2, uint32_t fill_mask)
{
    const long long nr = (long long)g.R * g.R * g.R;
    int cpw, ctas;
    activate_shape(nr, cpw, ctas);
    if (g.L == 8) launch_chained(k_activate_shell<8>, ctas, 256, 0, s, g, lo2, hi2, 0, 1, cpw, fill_mask);
    else launch_chained(k_activate_shell<4>, ctas, 256, 0, s, g, lo2, hi2, 0, 1, cpw, fill_mask);
}

// ---------------------------------------------------------------------------
// Activation of explicit voxels and of particle stencils runs in three steps
// so that no thread ever waits for another: mark the pointer cells that are
// needed, allocate the null ones (compaction-style, one atomic per warp), then
// set the voxel bits with atomicOr.
// ---------------------------------------------------------------------------
__global__ void k_mark_coords(DevGrid g, const int32_t *__restrict__ xyz, long long n)
{
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const int i = xyz[3 * p], j = xyz[3 * p + 1], k = xyz[3 * p + 2];
        if ((unsigned)i >= (unsigned)g.N || (unsigned)j >= (unsigned)g.N || (unsigned)k >= (unsigned)g.N) continue;
        const long long b = ((long long)(i >> g.lg2) * g.R + (j >> g.lg2)) * g.R + (k >> g.lg2);
        g.need[b] = 1;
    }
}

void launch_mark_coords(const DevGrid &g, cudaStream_t s, const int32_t *xyz, long long n)
{
    if (n <= 0) return;
    long long blocks = (n + 255) / 256;
    if (blocks > 65535) blocks = 65535;
    k_mark_coords<<<(unsigned)blocks, 256, 0, s>>>(g, xyz, n);
}

__global__ void __launch_bounds__(256) k_alloc_needed(DevGrid g, uint32_t fill_mask)
{
    chained_entry();
    alloc_needed(g, fill_mask, blockIdx.x, gridDim.x);
}

void launch_alloc_needed(const DevGrid &g, cudaStream_t s, uint32_t fill_mask)
{
    launch_chained(k_alloc_needed, alloc_needed_ctas(g), 256, 0, s, g, fill_mask);
}

__global__ void k_setbits_coords(DevGrid g, const int32_t *__restrict__ xyz, long long n)
{
    bool changed = false;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const int i = xyz[3 * p], j = xyz[3 * p + 1], k = xyz[3 * p + 2];
        if ((unsigned)i >= (unsigned)g.N || (unsigned)j >= (unsigned)g.N || (unsigned)k >= (unsigned)g.N) continue;
        const int L = g.L, lg2 = g.lg2;
        const long long b = ((long long)(i >> lg2) * g.R + (j >> lg2)) * g.R + (k >> lg2);
        const int slot = g.root[b];
        if (slot < 0) continue;  // pool was exhausted; the error is latched
        const int l = (((i & (L - 1)) << lg2) + (j & (L - 1))) * L + (k & (L - 1));
        const uint32_t bit = 1u << (l & 31);
        uint32_t *w = &g.mask[(long long)slot * g.W + (l >> 5)];
        if ((*w & bit) == 0u) {
            const uint32_t old = atomicOr(w, bit);
            if ((old & bit) == 0u) changed = true;
        }
    }
    if (changed) mark_dirty(g);
}

void launch_setbits_coords(const DevGrid &g, cudaStream_t s, const int32_t *xyz, long long n)
{
    if (n <= 0) return;
    long long blocks = (n + 255) / 256;
    if (blocks > 65535) blocks = 65535;
    k_setbits_coords<<<(unsigned)blocks, 256, 0, s>>>(g, xyz, n);
}

// ---------------------------------------------------------------------------
// Deactivate everything: null pointers, empty pool, empty list.  Leaf slots
// are zero-filled again when they are next allocated.
// ---------------------------------------------------------------------------
__global__ void k_deactivate_all(DevGrid g)
{
    chained_entry();
    const long long nr = (long long)g.R * g.R * g.R;
    for (long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x; b < nr; b += (long long)gridDim.x * blockDim.x)
        g.root[b] = -1;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        g.ctrl->pool_count = 0;
        g.ctrl->list_n = 0;
        g.ctrl->dirty = 1;
    }
}

void launch_deactivate_all(const DevGrid &g, cudaStream_t s)
{
    const long long nr = (long long)g.R * g.R * g.R;
    long long blocks = (nr + 255) / 256;
    if (blocks > 2048) blocks = 2048;
    launch_chained(k_deactivate_all, (unsigned)blocks, 256, 0, s, g);
}

// Restore a saved structure (checkpoint): one warp per saved leaf e takes
// slot e, so the slots come out in the saved (ascending root index) order.
__global__ void __launch_bounds__(256) k_restore_structure(DevGrid g, const int32_t *__restrict__ leaf_b,
                                                           const uint32_t *__restrict__ masks, long long n)
{
    const int lane = lane_id();
    const int V = g.L * g.L * g.L;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    for (long long e = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; e < n; e += warps) {
        for (int f = 0; f < g.F; ++f) {
            float4 *p = reinterpret_cast<float4 *>(g.field[f] + e * V);
            for (int q = lane; q < V / 4; q += 32) p[q] = z;
        }
        for (int w = lane; w < g.W; w += 32) g.mask[e * g.W + w] = masks[e * g.W + w];
        if (lane == 0) g.root[leaf_b[e]] = (int)e;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        g.ctrl->pool_count = (int)n;
        g.ctrl->list_n = 0;
        g.ctrl->dirty = 1;
    }
}

void launch_restore_structure(const DevGrid &g, cudaStream_t s, const int32_t *leaf_b, const uint32_t *masks,
                              long long n, const LaunchCfg &lc)
{
    k_restore_structure<<<lc.num_sms * 4, 256, 0, s>>>(g, leaf_b, masks, n);
}

// The clear-list task of the eager form (Sec. 6.1, Fig. 8): empty the list.
__global__ void k_clear_list(DevGrid g)
{
    g.ctrl->list_n = 0;
    g.ctrl->dirty = 1;
}

void launch_clear_list(const DevGrid &g, cudaStream_t s) { k_clear_list<<<1, 1, 0, s>>>(g); }

// ---------------------------------------------------------------------------
// List generation (Sec. 3.2 item 2): compact the non-null pointer cells into a
// list in ascending b, in one pass with a decoupled look-back prefix sum.
// Each CTA takes a tile of kListTile root cells in ticket order (so every
// predecessor tile has started), counts its active cells with a block scan,
// publishes its aggregate, looks back over its predecessors' published words
// for its exclusive prefix, writes its list entries, then fills their
// 27-neighbour slots.  Status words carry (call + 1) << 34 so words left by
// earlier calls are never taken for current ones.  Every wait is bounded by
// wall time; a wait that gives up latches kErrTimeout and the kernel returns.
// Unless `force`, the whole launch is a no-op when no activation since the
// last generation changed the structure (ctrl->dirty == 0).
// ---------------------------------------------------------------------------
constexpr unsigned long long kFlagAgg = 1ull, kFlagIncl = 2ull;
constexpr unsigned long long kLookbackLimitNs = 1000000000ull;  // 1 s
constexpr unsigned long long kTestWaitLimitNs = 200000000ull;   // 0.2 s

__global__ void __launch_bounds__(kListThreads) k_listgen(DevGrid g, int force, unsigned long long call_idx,
                                                          int num_tiles, int test_wait)
{
    chained_entry();
    __shared__ int s_tile, s_skip, s_prefix;
    __shared__ int s_wsum[kListThreads / 32];
    __shared__ uint32_t s_cells[kListTile];  // listed cells' (i, j, k), 10 bits each (R <= 1024)
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const unsigned long long tick0 = call_idx * (unsigned long long)num_tiles;
    const unsigned long long tag = (call_idx + 1ull) << 34;
    if (tid == 0) {
        const unsigned long long t = atomicAdd(&g.ctrl->lg_ticket, 1ull);
        s_tile = (int)(t - tick0);
        s_skip = (!force && *(volatile int32_t *)&g.ctrl->dirty == 0) ? 1 : 0;
    }
    __syncthreads();
    const int tile = s_tile;
    if (!s_skip && tile >= 0 && tile < num_tiles) {
        const long long nr = (long long)g.R * g.R * g.R;
        const long long c0 = (long long)tile * kListTile + tid * 4;
        int sl[4];
        if (c0 + 3 < nr) {
            const int4 v = *reinterpret_cast<const int4 *>(g.root + c0);
            sl[0] = v.x; sl[1] = v.y; sl[2] = v.z; sl[3] = v.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) sl[q] = (c0 + q < nr) ? g.root[c0 + q] : -1;
        }
        int cnt = (sl[0] >= 0) + (sl[1] >= 0) + (sl[2] >= 0) + (sl[3] >= 0);
        const int incl = warp_incl_scan(cnt);
        if (lane == 31) s_wsum[warp] = incl;
        __syncthreads();
        int wbase = 0, total = 0;
#pragma unroll
        for (int w = 0; w < kListThreads / 32; ++w) {
            const int v = s_wsum[w];
            wbase += (w < warp) ? v : 0;
            total += v;
        }
        const int excl = wbase + incl - cnt;
        if (tid == 0) {
            const unsigned long long flag = (tile == 0) ? kFlagIncl : kFlagAgg;
            atomicExch(&g.tile_status[tile], tag | (flag << 32) | (unsigned long long)(unsigned)total);
        }
        if (warp == 0) {
            int prefix = 0;
            if (tile > 0) {
                int pred = tile - 1;
                const unsigned long long t_start = global_timer_ns();
                for (;;) {
                    const int idx = pred - lane;
                    unsigned long long w = tag | (kFlagIncl << 32);
                    if (idx >= 0) {
                        for (;;) {
                            w = *(volatile unsigned long long *)&g.tile_status[idx];
                            if ((w >> 34) == (call_idx + 1ull)) break;
                            if (global_timer_ns() - t_start > kLookbackLimitNs) {
                                raise_error(g, kErrTimeout);
                                g.ctrl->timeout_site = 1;
                                w = tag | (kFlagIncl << 32);
                                break;
                            }
                            __nanosleep(32);
                        }
                    }
                    const unsigned long long flag = (w >> 32) & 3ull;
                    const int val = (int)(w & 0xffffffffull);
                    const unsigned im = __ballot_sync(kFull, flag == kFlagIncl);
                    const int upto = im ? (__ffs(im) - 1) : 31;
                    prefix += warp_sum(lane <= upto ? val : 0);
                    if (im) break;
                    pred -= 32;
                }
                if (lane == 0)
                    atomicExch(&g.tile_status[tile],
                               tag | (kFlagIncl << 32) | (unsigned long long)(unsigned)(prefix + total));
            }
            if (lane == 0) s_prefix = prefix;
        }
        __syncthreads();
        const int prefix = s_prefix;
        const int R = g.R;
        int pos = excl;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (sl[q] >= 0) {
                const int b = (int)(c0 + q);
                g.list_slot[prefix + pos] = sl[q];
                g.list_b[prefix + pos] = b;
                g.ent_of_slot[sl[q]] = prefix + pos;
                const unsigned ci = (unsigned)b / ((unsigned)R * R), rem = (unsigned)b - ci * ((unsigned)R * R),
                               cj = rem / (unsigned)R, ck = rem - cj * (unsigned)R;
                s_cells[pos] = (ci << 20) | (cj << 10) | ck;
                ++pos;
            }
        }
        if (tile == num_tiles - 1 && tid == 0) g.ctrl->list_n = prefix + total;
        __syncthreads();
        for (int idx = tid; idx < total * 27; idx += kListThreads) {
            const int e = idx / 27, q = idx - e * 27;
            const uint32_t c = s_cells[e];
            const int bi = (int)(c >> 20) + q / 9 - 1;
            const int bj = (int)((c >> 10) & 1023u) + (q / 3) % 3 - 1;
            const int bk = (int)(c & 1023u) + q % 3 - 1;
            int v = -1;
            if ((unsigned)bi < (unsigned)R && (unsigned)bj < (unsigned)R && (unsigned)bk < (unsigned)R)
                v = g.root[((long long)bi * R + bj) * R + bk];
            g.nbr[(long long)(prefix + e) * 27 + q] = (v < 0) ? (int)g.cap : v;  // null -> the zero leaf
        }
    }
    if (test_wait && tile == 0 && tid == 0) {
        // Fault-injection hook: wait on a flag that nothing sets, bounded.
        const unsigned long long t_start = global_timer_ns();
        while (*(volatile int32_t *)&g.ctrl->never_set == 0) {
            if (global_timer_ns() - t_start > kTestWaitLimitNs) {
                raise_error(g, kErrTimeout);
                g.ctrl->timeout_site = 2;
                break;
            }
            __nanosleep(1000);
        }
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const unsigned long long d = atomicAdd(&g.ctrl->lg_done, 1ull) - tick0;
        if (d == (unsigned long long)num_tiles - 1ull && !s_skip) g.ctrl->dirty = 0;
    }
}

void launch_listgen(const DevGrid &g, cudaStream_t s, int force, unsigned long long call_idx, int num_tiles,
                    int test_wait)
{
    launch_chained(k_listgen, num_tiles, kListThreads, 0, s, g, force, call_idx, num_tiles, test_wait);
}

// ---------------------------------------------------------------------------
// Region masks of 8^3 leaves (the fused diffuse->box kernel's t activity):
// one thread per (list entry, region column tj, word w) gathers rows
// ti = 3w..3w+2 of column tj; region row (ri, rj) = (ti+1, tj+1) takes its
// bit for k = 1 from the k-1 leaf (local k 7), k = 2..9 from its own leaf
// column and k = 10 from the k+1 leaf (local k 0), via the 27-neighbour
// table (null neighbours are the zero leaf, whose mask is 0).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_region_masks(DevGrid g, int group_axis, unsigned long long call)
{
    chained_entry();
    const long long n = g.ctrl->list_n;
    const uint8_t *mb = reinterpret_cast<const uint8_t *>(g.mask);
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * 40; q += (long long)gridDim.x * blockDim.x) {
        const long long e = q / 40;
        const int tj = (int)(q % 40) / 4, w = (int)(q % 4);
        const int rj = tj + 1;
        const int djx = (rj < 2) ? 0 : (rj < 10 ? 1 : 2), lj = (rj - 2) & 7;
        uint32_t word = 0;
        for (int u = 0; u < 3; ++u) {
            const int ti = 3 * w + u;
            if (ti > 9) break;
            const int ri = ti + 1;
            const int dix = (ri < 2) ? 0 : (ri < 10 ? 1 : 2), li = (ri - 2) & 7;
            const int *nb = g.nbr + e * 27 + dix * 9 + djx * 3;
            const int ro = li * 8 + lj;
            const uint32_t m0 = mb[(long long)nb[0] * 64 + ro];
            const uint32_t m1 = mb[(long long)nb[1] * 64 + ro];
            const uint32_t m2 = mb[(long long)nb[2] * 64 + ro];
            const uint32_t bits = ((m0 >> 7) & 1u) | (m1 << 1) | ((m2 & 1u) << 9);
            word |= bits << (10 * u);
        }
        g.rmask[e * 40 + tj * 4 + w] = word;
    }
    if (group_axis == kGroupNone) return;
    // The records of the grouped sweeps: runs of leaves adjacent along the
    // axis (root cells b, b + S, ... all allocated; S = R^2 for i, R for j)
    // cut into pieces of up to three from the run's lowest leaf; each piece's
    // list entries, lowest first, go to the bucket of its length, in list
    // order.  List order keeps the warps that sweep at the same time on
    // neighbouring leaves, so halo rows are reused through L1 and L2.  Tiles
    // of 256 list entries are taken by ticket; in a tile, warp w classifies
    // entries 32w .. 32w + 31 (the piece each entry starts); the tile's
    // offset in each bucket comes from a decoupled look-back over the
    // earlier tiles (three warps, one per length, each waiting only on tiles
    // whose tickets were handed out earlier, so the waits end; bounded in
    // time all the same), and every entry's record is written at once.
    __shared__ int s_tile;
    __shared__ int s_wcnt[3][8];
    __shared__ int s_base[3];
    const long long S = group_axis == kGroupI ? (long long)g.R * g.R : (long long)g.R;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int ntiles = (int)((n + 255) / 256);
    const unsigned long long tag = (call + 1ull) << 34;
    for (;;) {
        if (threadIdx.x == 0) s_tile = (int)atomicAdd(&g.ctrl->rr_ticket, 1u);
        __syncthreads();
        const int tile = s_tile;
        if (tile >= ntiles) break;  // CTA-uniform
        const long long e = (long long)tile * 256 + threadIdx.x;
        int len = 0, r1 = -1, r2 = -1;
        if (e < n) {
            const long long b = g.list_b[e];
            const int c = (int)((b / S) % g.R);  // the leaf's root coordinate along the axis
            int p = 0;  // allocated leaves directly below along the axis
            while (p < c && g.root[b - (p + 1) * S] >= 0) ++p;
            if (p % 3 == 0) {
                len = 1;
                while (len < 3 && c + len < g.R && g.root[b + len * S] >= 0) ++len;
            }
            r1 = len > 1 ? g.ent_of_slot[g.root[b + S]] : -1;
            r2 = len > 2 ? g.ent_of_slot[g.root[b + 2 * S]] : -1;
        }
        unsigned m[3];
#pragma unroll
        for (int G = 1; G <= 3; ++G) {
            m[G - 1] = __ballot_sync(kFull, len == G);
            if (lane == 0) s_wcnt[G - 1][warp] = __popc(m[G - 1]);
        }
        __syncthreads();
        if (warp < 3) {
            // bucket warp + 1: the tile's count, published, then its offset
            const int G1 = warp;
            int tot = 0;
            for (int w = 0; w < 8; ++w) tot += s_wcnt[G1][w];
            unsigned long long *st = g.rr_status + (long long)tile * 3 + G1;
            if (lane == 0)
                atomicExch(st, tag | ((tile == 0 ? kFlagIncl : kFlagAgg) << 32) | (unsigned long long)(unsigned)tot);
            int prefix = 0;
            if (tile > 0) {
                int pred = tile - 1;
                const unsigned long long t_start = global_timer_ns();
                for (;;) {
                    const int idx = pred - lane;
                    unsigned long long w = tag | (kFlagIncl << 32);
                    if (idx >= 0) {
                        for (;;) {
                            w = *(volatile unsigned long long *)(g.rr_status + (long long)idx * 3 + G1);
                            if ((w >> 34) == (call + 1ull)) break;
                            if (global_timer_ns() - t_start > kLookbackLimitNs) {
                                raise_error(g, kErrTimeout);
                                g.ctrl->timeout_site = 5;
                                w = tag | (kFlagIncl << 32);
                                break;
                            }
                            __nanosleep(32);
                        }
                    }
                    const unsigned long long flag = (w >> 32) & 3ull;
                    const int val = (int)(w & 0xffffffffull);
                    const unsigned im = __ballot_sync(kFull, flag == kFlagIncl);
                    const int upto = im ? (__ffs(im) - 1) : 31;
                    prefix += warp_sum(lane <= upto ? val : 0);
                    if (im) break;
                    pred -= 32;
                }
                if (lane == 0) atomicExch(st, tag | (kFlagIncl << 32) | (unsigned long long)(unsigned)(prefix + tot));
            }
            if (lane == 0) {
                s_base[G1] = prefix;
                if (tile == ntiles - 1) g.col_cnt[G1] = prefix + tot;
            }
        }
        __syncthreads();
        if (len > 0) {
            int j = s_base[len - 1];
            for (int w = 0; w < warp; ++w) j += s_wcnt[len - 1][w];
            j += __popc(m[len - 1] & lanemask_lt());
            int32_t *rec = g.col_grp + ((long long)(len - 1) * g.cap + j) * 3;
            rec[0] = (int32_t)e;
            rec[1] = r1;
            rec[2] = r2;
        }
        __syncthreads();  // s_tile, s_wcnt and s_base are reused by the next tile
    }
    if (n == 0 && blockIdx.x == 0 && threadIdx.x < 3) g.col_cnt[threadIdx.x] = 0;
}

void launch_region_masks(const DevGrid &g, cudaStream_t s, const LaunchCfg &lc, int group_axis,
                         unsigned long long call)
{
    if (group_axis != kGroupNone) cudaMemsetAsync(&g.ctrl->rr_ticket, 0, sizeof(uint32_t), s);
    launch_chained(k_region_masks, lc.num_sms * 8, 256, 0, s, g, group_axis, call);
}

// ---------------------------------------------------------------------------
// Device-side initial values: at every active voxel of the listed leaves,
// the top 24 bits of splitmix64 (Steele, Lea & Flood 2014) applied to
// seed * 2^40 + (i*N + j)*N + k, times 2^-24 (exact in FP32); 0 at inactive
// voxels.  The same published generator as the harness's input module, so a
// grid filled here holds the values the harness would upload.
// ---------------------------------------------------------------------------
// The top 24 bits of splitmix64(key) times 2^-24.  The last xor of splitmix64
// leaves bits 33 and up as they are, so they are the top bits of the second
// product.  The 24 bits become a float as two integers under the exponent of
// 2^23 (2^23 + a, 2^23 + b) and two exact FMAs, (a - 2^15) 2^-16 first; an
// integer conversion runs at an eighth of their rate.
__device__ __forceinline__ float hash24(unsigned long long z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    const uint32_t h = (uint32_t)(z >> 32);
    const float a = __uint_as_float(__byte_perm(h, 0x4b000000u, 0x7632));  // 2^23 + (h >> 16)
    const float b = __uint_as_float(__byte_perm(h, 0x4b000000u, 0x7651));  // 2^23 + (h >> 8 & 255)
    return fmaf(b, 0x1p-24f, fmaf(a, 0x1p-16f, -128.5f));
}

// The initial state of a new grid in one launch: the arrays of a small grid
// are far smaller than the time that nine memsets and a copy take one after the
// other, and every admission of a served job waits for them (24 served jobs
// 9.76 -> 9.62 ms).  16 bytes a thread where the span allows it.
__global__ void __launch_bounds__(256) k_init_grid(const __grid_constant__ InitSpans in, Ctrl *ctrl,
                                                   const __grid_constant__ Ctrl state)
{
    chained_entry();
    const long long t = blockIdx.x * 256LL + threadIdx.x, nt = gridDim.x * 256LL;
    if (t == 0) *ctrl = state;
    for (int q = 0; q < in.n; ++q) {
        uint8_t *p = (uint8_t *)in.span[q].p;
        const long long bytes = in.span[q].bytes;
        const uint32_t w = in.span[q].word;
        const long long n16 = ((uintptr_t)p & 15) == 0 ? bytes >> 4 : 0;
        for (long long e = t; e < n16; e += nt) reinterpret_cast<uint4 *>(p)[e] = make_uint4(w, w, w, w);
        for (long long e = (n16 << 4) + t; e < bytes; e += nt) p[e] = (uint8_t)w;
    }
}

cudaError_t launch_init_grid(cudaStream_t s, const InitSpans &spans, Ctrl *ctrl, const Ctrl &state, const LaunchCfg &lc)
{
    long long bytes = 0;
    for (int q = 0; q < spans.n; ++q) bytes += spans.span[q].bytes;
    const long long ctas = (bytes + 4095) / 4096, most = lc.num_sms * 8LL;
    return launch_chained(k_init_grid, ctas < most ? ctas : most, 256, 0, s, spans, ctrl, state);
}

// A group of G = min(32, L^3 / 4) threads fills one leaf, four k-adjacent
// voxels (one float4 store) per thread and iteration: the leaf's slot, its
// two root divisions and the row's linear index are worked out once per leaf
// or per four voxels, and only active voxels are hashed.  What bounds it is
// the hash's integer arithmetic (two 64-bit products a voxel), then the store:
// 26,104 leaves in 19 us, 103,600 in 69 us (65 and 267 us with a thread per
// voxel that divided by R and R^2 for each one and converted an integer).  Six
// CTAs of 256 threads fit an SM (42 registers), so the grid is one wave.
template <int L>
__global__ void __launch_bounds__(256, 6) k_fill_hash(DevGrid g, int f, unsigned long long seed)
{
    chained_entry();
    constexpr int LG2 = (L == 8) ? 3 : 2, V4 = L * L * L / 4, G = V4 < 32 ? V4 : 32, W = L * L * L / 32;
    const long long n = g.ctrl->list_n;
    const int R = g.R, r0 = threadIdx.x % G;
    float4 *out = reinterpret_cast<float4 *>(g.field[f]);
    for (long long e = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / G; e < n;
         e += (long long)gridDim.x * blockDim.x / G) {
        const int slot = g.list_slot[e], b = g.list_b[e];
        const int bij = b / R, bi = bij / R;
        const long long i0 = (long long)bi << LG2, j0 = (long long)(bij - bi * R) << LG2, k0 = (long long)(b - bij * R) << LG2;
        const unsigned long long key0 = (seed << 40) + 0x9E3779B97F4A7C15ull + (unsigned long long)((i0 * g.N + j0) * g.N + k0);
#pragma unroll
        for (int r = r0; r < V4; r += G) {
            const int l = 4 * r;  // local index of the first of the four voxels
            const uint32_t bits = g.mask[(long long)slot * W + (l >> 5)] >> (l & 31);
            const unsigned long long key =
                key0 + (unsigned long long)(((long long)(l >> (2 * LG2)) * g.N + ((l >> LG2) & (L - 1))) * g.N + (l & (L - 1)));
            float v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[q] = ((bits >> q) & 1u) ? hash24(key + q) : 0.f;
            out[(long long)slot * V4 + r] = make_float4(v[0], v[1], v[2], v[3]);
        }
    }
}

void launch_fill_hash(const DevGrid &g, cudaStream_t s, int f, unsigned long long seed, const LaunchCfg &lc)
{
    if (g.L == 8) launch_chained(k_fill_hash<8>, lc.num_sms * 6, 256, 0, s, g, f, seed);
    else launch_chained(k_fill_hash<4>, lc.num_sms * 6, 256, 0, s, g, f, seed);
}

// ---------------------------------------------------------------------------
// Host transfers: gather leaves in list order into the staging buffer, and
// scatter from it (applying the mask so inactive voxels stay 0).
// ---------------------------------------------------------------------------
__global__ void k_gather_field(DevGrid g, int f, float4 *__restrict__ dst)
{
    const long long n = g.ctrl->list_n;
    const int V4 = (g.L * g.L * g.L) >> 2;
    const float4 *src = reinterpret_cast<const float4 *>(g.field[f]);
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * V4; q += (long long)gridDim.x * blockDim.x) {
        const long long e = q / V4;
        const int r = (int)(q - e * V4);
        dst[q] = src[(long long)g.list_slot[e] * V4 + r];
    }
}

void launch_gather_field(const DevGrid &g, cudaStream_t s, int f, float *dst, const LaunchCfg &lc)
{
    k_gather_field<<<lc.num_sms * 4, 256, 0, s>>>(g, f, reinterpret_cast<float4 *>(dst ? dst : g.staging));
}

__global__ void k_gather_masks(DevGrid g)
{
    const long long n = g.ctrl->list_n;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * g.W; q += (long long)gridDim.x * blockDim.x) {
        const long long e = q / g.W;
        const int w = (int)(q - e * g.W);
        g.staging_u[q] = g.mask[(long long)g.list_slot[e] * g.W + w];
    }
}

void launch_gather_masks(const DevGrid &g, cudaStream_t s, const LaunchCfg &lc)
{
    k_gather_masks<<<lc.num_sms * 4, 256, 0, s>>>(g);
}

__global__ void k_scatter_field(DevGrid g, int f, const float4 *__restrict__ src)
{
    const long long n = g.ctrl->list_n;
    const int V4 = (g.L * g.L * g.L) >> 2;
    float4 *dst = reinterpret_cast<float4 *>(g.field[f]);
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * V4; q += (long long)gridDim.x * blockDim.x) {
        const long long e = q / V4;
        const int r = (int)(q - e * V4);
        const int slot = g.list_slot[e];
        const uint32_t word = g.mask[(long long)slot * g.W + (r >> 3)];
        const int sh = (r & 7) * 4;
        float4 v = src[q];
        v.x = ((word >> (sh + 0)) & 1u) ? v.x : 0.f;
        v.y = ((word >> (sh + 1)) & 1u) ? v.y : 0.f;
        v.z = ((word >> (sh + 2)) & 1u) ? v.z : 0.f;
        v.w = ((word >> (sh + 3)) & 1u) ? v.w : 0.f;
        dst[(long long)slot * V4 + r] = v;
    }
}

void launch_scatter_field(const DevGrid &g, cudaStream_t s, int f, const float *src, const LaunchCfg &lc)
{
    k_scatter_field<<<lc.num_sms * 4, 256, 0, s>>>(g, f, reinterpret_cast<const float4 *>(src ? src : g.staging));
}

}  // namespace sg

namespace sg {

// ---------------------------------------------------------------------------
// Transfers of the active voxels only ("packed": list order, ascending local
// index within a leaf).  off[e] + tsum[e / kOffTile] is the number of active
// voxels in the list entries before e.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kOffTile) k_active_offsets(DevGrid g, long long n, long long *off, long long *tsum)
{
    chained_entry();
    __shared__ long long s_w[kOffTile / 32];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const long long e = (long long)blockIdx.x * kOffTile + threadIdx.x;
    int c = 0;
    if (e < n) {
        const int slot = g.list_slot[e];
        for (int w = 0; w < g.W; ++w) c += __popc(g.mask[(long long)slot * g.W + w]);
    }
    const int inc = warp_incl_scan(c);
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const long long v = s_w[lane];
        long long x = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const long long y = __shfl_up_sync(kFull, x, d);
            if (lane >= d) x += y;
        }
        s_w[lane] = x - v;
    }
    __syncthreads();
    const long long ex = s_w[warp] + inc - c;
    if (e < n) off[e] = ex;
    if (threadIdx.x == kOffTile - 1) tsum[blockIdx.x] = ex + c;
}

// Exclusive scan of the tile totals by one CTA, in place; the grand total
// goes to tsum[ntiles].
__global__ void __launch_bounds__(1024) k_active_offsets_top(DevGrid g, long long *tsum, int ntiles)
{
    chained_entry();
    __shared__ long long s_w[32];
    __shared__ long long s_carry;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < ntiles; base += 1024) {
        const int i = base + threadIdx.x;
        const long long v = (i < ntiles) ? tsum[i] : 0;
        long long x = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const long long y = __shfl_up_sync(kFull, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        if (warp == 0) {
            const long long wv = s_w[lane];
            long long z = wv;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const long long y = __shfl_up_sync(kFull, z, d);
                if (lane >= d) z += y;
            }
            s_w[lane] = z - wv;
        }
        __syncthreads();
        const long long ex = s_carry + s_w[warp] + x - v;
        __syncthreads();
        if (i < ntiles) tsum[i] = ex;
        if (threadIdx.x == 1023) s_carry = ex + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) tsum[ntiles] = g.ctrl->act_total = s_carry;
}

void launch_active_offsets(const DevGrid &g, cudaStream_t s, long long n, long long *off, long long *tsum)
{
    const int ntiles = (int)((n + kOffTile - 1) / kOffTile);
    launch_chained(k_active_offsets, ntiles, kOffTile, 0, s, g, n, off, tsum);
    launch_chained(k_active_offsets_top, 1, 1024, 0, s, g, tsum, ntiles);
}

// Position in the packed array of the first active voxel at or after local
// index 4r of list entry e (slot `slot`).
__device__ __forceinline__ long long packed_pos(const DevGrid &g, long long e, int slot, int r, const long long *off,
                                                const long long *tsum, uint32_t &word, int &sh)
{
    const uint32_t *mw = g.mask + (long long)slot * g.W;
    const int w = r >> 3;
    sh = (r & 7) * 4;
    long long pos = off[e] + tsum[e / kOffTile];
    for (int i = 0; i < w; ++i) pos += __popc(mw[i]);
    word = mw[w];
    return pos + __popc(word & ((1u << sh) - 1u));
}

// Positions at or past `total` (the packed buffer's length) are never
// accessed, so a buffer of exactly `total` values is read in bounds whatever
// the masks hold.
__global__ void k_scatter_active(DevGrid g, int f, const float *__restrict__ src, long long total,
                                 const long long *__restrict__ off, const long long *__restrict__ tsum)
{
    chained_entry();
    const long long n = g.ctrl->list_n;
    const int V4 = (g.L * g.L * g.L) >> 2;
    float4 *dst = reinterpret_cast<float4 *>(g.field[f]);
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * V4; q += (long long)gridDim.x * blockDim.x) {
        const long long e = q / V4;
        const int r = (int)(q - e * V4);
        const int slot = g.list_slot[e];
        uint32_t word;
        int sh;
        long long pos = packed_pos(g, e, slot, r, off, tsum, word, sh);
        float4 v;
        v.x = ((word >> (sh + 0)) & 1u) && pos < total ? src[pos++] : 0.f;
        v.y = ((word >> (sh + 1)) & 1u) && pos < total ? src[pos++] : 0.f;
        v.z = ((word >> (sh + 2)) & 1u) && pos < total ? src[pos++] : 0.f;
        v.w = ((word >> (sh + 3)) & 1u) && pos < total ? src[pos] : 0.f;
        dst[(long long)slot * V4 + r] = v;
    }
}

// A CTA packs the active values of T consecutive list entries, whose places
// in the packed array are consecutive, in shared memory (a warp per leaf, 32
// voxels at a time) and then writes them out as whole float4s in order, so
// that memory across the host link sees full lines.  The link bounds it: 32 MB
// (the 512^3 band) into mapped host memory take 190 us against 169 us for a
// plain copy; a thread per four voxels storing its values one by one took 473
// us, most of its stores being parts of a line.
template <int L>
__global__ void __launch_bounds__(256) k_gather_active(DevGrid g, int f, float *__restrict__ out, int ntiles, long long cap,
                                                       const long long *off, const long long *tsum)
{
    chained_entry();
    const long long total = tsum[ntiles];
    if (total > cap || g.ctrl->err) return;
    constexpr int V = L * L * L, W = V / 32, CAP = 4096, T = CAP / V;
    __shared__ float s_val[CAP];
    const long long n = g.ctrl->list_n;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const float *src = g.field[f];
    for (long long e0 = (long long)blockIdx.x * T; e0 < n; e0 += (long long)gridDim.x * T) {
        const long long e1 = e0 + T;
        const long long p0 = min(off[e0] + tsum[e0 / kOffTile], total);
        const long long p1 = e1 < n ? min(off[e1] + tsum[e1 / kOffTile], total) : total;
        const int cnt = (int)min(p1 - p0, (long long)CAP);
        for (int q = warp; q < T; q += 8) {
            const long long e = e0 + q;
            if (e >= n) break;
            const int slot = g.list_slot[e];
            const uint32_t mine = lane < W ? g.mask[(long long)slot * W + lane] : 0u;
            const int c = __popc(mine), before = warp_incl_scan(c) - c;
            const int rel = (int)(off[e] + tsum[e / kOffTile] - p0);
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const uint32_t word = __shfl_sync(kFull, mine, w);
                const int at = rel + __shfl_sync(kFull, before, w) + __popc(word & lanemask_lt());
                const float v = src[(long long)slot * V + w * 32 + lane];
                if (((word >> lane) & 1u) && at < cnt) s_val[at] = v;
            }
        }
        __syncthreads();
        // out is 16-byte aligned: single values up to the first whole float4
        const int head = min((int)(-p0 & 3), cnt), quads = (cnt - head) >> 2, tail = head + 4 * quads;
        if ((int)threadIdx.x < head) out[p0 + threadIdx.x] = s_val[threadIdx.x];
        float4 *o4 = reinterpret_cast<float4 *>(out + p0 + head);
        for (int q = threadIdx.x; q < quads; q += 256) {
            const float *s = s_val + head + 4 * q;
            o4[q] = make_float4(s[0], s[1], s[2], s[3]);
        }
        if (tail + (int)threadIdx.x < cnt) out[p0 + tail + threadIdx.x] = s_val[tail + threadIdx.x];
        __syncthreads();  // s_val is refilled for the next tile
    }
}

void launch_scatter_active(const DevGrid &g, cudaStream_t s, int f, const float *src, long long total,
                           const long long *off, const long long *tsum, const LaunchCfg &lc)
{
    launch_chained(k_scatter_active, lc.num_sms * 4, 256, 0, s, g, f, src, total, off, tsum);
}

void launch_gather_active(const DevGrid &g, cudaStream_t s, int f, float *out, long long n, long long cap,
                          const long long *off, const long long *tsum, const LaunchCfg &lc)
{
    const int ntiles = (int)((n + kOffTile - 1) / kOffTile);
    if (g.L == 8) launch_chained(k_gather_active<8>, lc.num_sms * 4, 256, 0, s, g, f, out, ntiles, cap, off, tsum);
    else launch_chained(k_gather_active<4>, lc.num_sms * 4, 256, 0, s, g, f, out, ntiles, cap, off, tsum);
}

// Active voxels of the listed leaves: popcount of their mask words.
__global__ void k_count_active(DevGrid g)
{
    const long long n = g.ctrl->list_n;
    unsigned long long c = 0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * g.W; q += (long long)gridDim.x * blockDim.x) {
        const long long e = q / g.W;
        c += __popc(g.mask[(long long)g.list_slot[e] * g.W + (q - e * g.W)]);
    }
    c = warp_sum(c);
    if (lane_id() == 0 && c) atomicAdd(&g.ctrl->n_active, c);
}

void launch_count_active(const DevGrid &g, cudaStream_t s, const LaunchCfg &lc)
{
    cudaMemsetAsync(&g.ctrl->n_active, 0, sizeof(unsigned long long), s);
    k_count_active<<<lc.num_sms * 4, 256, 0, s>>>(g);
}

}  // namespace sg

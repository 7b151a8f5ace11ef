// sg_common.cuh -- small device helpers shared by the libsgrid kernels.
#pragma once
#include <atomic>
#include <cstdint>
#include "sg_device.h"

namespace sg {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ unsigned long long global_timer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ int warp_incl_scan(int v)
{
    const int lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int u = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// ---------------------------------------------------------------------------
// Chained launches.  The kernels of a step depend on one another and many run
// for a few microseconds, so launch_chained allows a kernel's CTAs to be
// brought up while the kernel before it on the stream still runs (programmatic
// stream serialization).  Such a kernel calls chained_entry() before anything
// else, in every thread: it waits until the kernels before it have finished
// and their writes are visible, and only then lets the next one come up (so at
// most one waits).  After a copy, a memset or a kernel of another program the
// launch is an ordinary one.  A kernel may be launched so only if chained_entry()
// is its first statement: without the wait it would race with the one before it.
//   Its CTAs are resident while the kernels before it still write what it reads.
// For plain loads the wait is all that is needed.  __ldg and const __restrict__
// become ld.global.nc, which wants data that do not change while the kernel reads
// them: here, from the wait on.  That relies on two things: no such load moves
// above the wait (a volatile asm that clobbers memory, as in
// cudaGridDependencySynchronize(); each sits in a loop or behind a branch, and what
// a kernel reads straight after the wait it reads with a plain load), and none is
// served from a line cached before it.  The documented use of the wait works that
// way, and a stale line would show in the tests that compare the bytes of long
// runs; nothing that the kernel's own grid writes may be read through them.
//   Between the kernels of a V-cycle the gap falls from 2.1 us to none (ten cycles
// of the 512^3 band 1650 -> 1360 us, ten PIC steps of 2M particles 3022 -> 2798 us,
// of 100k APIC particles 1008 -> 870 us).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void chained_entry()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t launch_kernel(bool chained, void (*kernel)(P...), long long ctas, int threads, size_t smem,
                                 cudaStream_t s, A &&...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kernel)(P...), long long ctas, int threads, size_t smem, cudaStream_t s, A &&...args)
{
    return launch_kernel(true, kernel, ctas, threads, smem, s, static_cast<A &&>(args)...);
}

// For a resident kernel whose CTAs together want more shared memory than the
// kernel before it: an SM divides its memory between L1 and shared memory when
// it is empty, so CTAs that come up beside the last ones of a kernel without
// shared memory find room for one or two only, and the rest of the grid runs
// after them (advection, six steps and the reads: 3480 us, drained 2513 us).  It is launched
// when the kernels before it have drained; the next one may still be chained
// to it.
template <typename... P, typename... A>
inline cudaError_t launch_drained(void (*kernel)(P...), long long ctas, int threads, size_t smem, cudaStream_t s, A &&...args)
{
    return launch_kernel(false, kernel, ctas, threads, smem, s, static_cast<A &&>(args)...);
}

// CTAs per SM of a kernel with `bytes` of dynamic shared memory, more than the
// 48 KB that every kernel may use: it is allowed them on the current device
// first.  Both belong to a device, so what is known is kept for each (threads
// may race to fill an entry; they store the same).
constexpr int kMaxDevices = 64;
template <typename K>
inline cudaError_t resident_per_sm(K *kernel, int threads, int bytes, std::atomic<int> (&known)[kMaxDevices], int *per)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && dev < kMaxDevices && (*per = known[dev].load(std::memory_order_relaxed)) > 0) return e;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per, kernel, threads, bytes);
    if (e == cudaSuccess && *per < 1) e = cudaErrorInvalidConfiguration;
    if (e != cudaSuccess) cudaGetLastError();  // returned, not left for a later check
    else if (dev < kMaxDevices) known[dev].store(*per, std::memory_order_relaxed);
    return e;
}

// Mark the grid's structure as changed (an activation set a new bit or
// allocated a leaf); the next list generation will not be skipped.
__device__ __forceinline__ void mark_dirty(const DevGrid &g) { *(volatile int32_t *)&g.ctrl->dirty = 1; }

__device__ __forceinline__ void raise_error(const DevGrid &g, int bits) { atomicOr(&g.ctrl->err, bits); }
// A kernel's check `site` of its own accesses failed.
__device__ __forceinline__ void raise_check(const DevGrid &g, int site)
{
    raise_error(g, kErrCheck);
    g.ctrl->timeout_site = 100 + site;
}

// ---------------------------------------------------------------------------
// Allocation of the leaves marked in g.need.
// fill_mask: the (physical) fields a newly allocated leaf is zero-filled in.
// A CTA takes 128 consecutive root cells: its first four warps give slots to
// the needed null ones (one pool atomic per warp) and list them, then all of
// its threads zero the listed leaves together.  Needed cells come in runs along
// k, so a warp that allocated and filled its own 32 cells' leaves one after the
// other was the launch's long pole (2M particles over 4,076 leaves 10.1 -> 4.8 us,
// 100k particles in a 25^3 root 11.8 -> 3.7 us).
constexpr int kAllocCells = 128;
inline int alloc_needed_ctas(const DevGrid &g)
{
    const long long nr = (long long)g.R * g.R * g.R;
    const long long ctas = (nr + kAllocCells - 1) / kAllocCells;
    return ctas > 4096 ? 4096 : (int)ctas;
}

// CTA `cta` of `ctas`, 256 threads each.
__device__ __forceinline__ void alloc_needed(const DevGrid &g, uint32_t fill_mask, int cta, int ctas)
{
    __shared__ int s_slot[kAllocCells];
    __shared__ int s_n;
    const long long nr = (long long)g.R * g.R * g.R;
    const int V4 = (g.L * g.L * g.L) >> 2, W = g.W;
    bool any_alloc = false;
    for (long long base = (long long)cta * kAllocCells; base < nr; base += (long long)ctas * kAllocCells) {
        const long long b = base + threadIdx.x;
        bool need = false;
        if (threadIdx.x < kAllocCells && b < nr && g.need[b]) {
            g.need[b] = 0;
            need = true;
        }
        if (!__syncthreads_or(need)) continue;
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        int slot = -1;
        if (threadIdx.x < kAllocCells) {
            const bool want = need && g.root[b] < 0;
            const unsigned m = __ballot_sync(kFull, want);
            if (m) {
                const int leader = __ffs(m) - 1;
                int first = 0, at = 0;
                if (lane_id() == leader) {
                    first = atomicAdd(&g.ctrl->pool_count, __popc(m));
                    at = atomicAdd(&s_n, __popc(m));
                }
                first = __shfl_sync(kFull, first, leader);
                at = __shfl_sync(kFull, at, leader);
                if (want) {
                    const int rank = __popc(m & lanemask_lt());
                    if (first + rank < g.cap) slot = first + rank;
                    else raise_error(g, kErrPool);
                    s_slot[at + rank] = slot;
                }
            }
        }
        __syncthreads();
        const int n = s_n;
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int f = 0; f < g.F; ++f) {
            if (!((fill_mask >> f) & 1u)) continue;
            float4 *p = reinterpret_cast<float4 *>(g.field[f]);
            for (int q = threadIdx.x; q < n * V4; q += 256) {
                const int s = s_slot[q / V4];
                if (s >= 0) p[(long long)s * V4 + (q & (V4 - 1))] = z;
            }
        }
        for (int q = threadIdx.x; q < n * W; q += 256) {
            const int s = s_slot[q / W];
            if (s >= 0) g.mask[(long long)s * W + (q & (W - 1))] = 0u;
        }
        if (slot >= 0) {
            g.root[b] = slot;
            any_alloc = true;
        }
        __syncthreads();  // s_slot is refilled for the next cells
    }
    if (any_alloc) mark_dirty(g);
}

// Block-wide FP64 reduction of one value per thread; result valid in thread 0.
template <int THREADS>
__device__ __forceinline__ double block_sum_f64(double v, double *smem)
{
    v = warp_sum(v);
    const int w = threadIdx.x >> 5;
    if (lane_id() == 0) smem[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = (threadIdx.x < THREADS / 32) ? smem[threadIdx.x] : 0.0;
        r = warp_sum(r);
    }
    __syncthreads();
    return r;
}

// Last-CTA reduction: every CTA stores its FP64 partial; the CTA that finishes
// last sums all partials in index order (deterministic) into sums[slot] and
// resets the ticket.  Called by all threads; `part` valid in thread 0.
__device__ __forceinline__ void finish_reduction(const DevGrid &g, double part, int slot)
{
    __shared__ bool s_last;
    if (threadIdx.x == 0) {
        g.partials[blockIdx.x] = part;
        __threadfence();
        unsigned t = atomicAdd(&g.ctrl->red_ticket, 1u);
        s_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        if (threadIdx.x < 32) {
            // fixed-order: lane handles a strided subset, then a fixed tree
            double acc = 0.0;
            for (unsigned c = threadIdx.x; c < gridDim.x; c += 32)
                acc += *(volatile double *)&g.partials[c];
            acc = warp_sum(acc);
            if (threadIdx.x == 0) {
                g.sums[slot] = acc;
                g.ctrl->red_ticket = 0;
            }
        }
    }
}

}  // namespace sg

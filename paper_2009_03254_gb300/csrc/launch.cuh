// Work distribution over one or many volumes.
//
// Every stage kernel receives a Launch: a device table of volumes and a
// few counters.  A single extraction is a table of one entry; a batch is
// a table of many (each volume with its own isovalue, cache and output
// range).  A kernel first turns the per-volume amount of work (tiles,
// chunks or warp tiles: fixed by the volume's size, or read from its
// control block where an earlier kernel of the same extraction set it)
// into a prefix in shared memory, then maps "virtual" work items to
// (volume, local item) by binary search.  Items of one volume keep their
// order, so each volume's look-back chains and outputs are exactly those
// of extracting it alone.
#pragma once

#include <cstdint>

#include "common.cuh"
#include "kernels.cuh"

namespace bcmc {

// The stages of a small volume's extraction are launched one ahead
// (launch_next): a stage's CTAs may take their places while the one before it
// finishes, and wait here for all of it, results included, before they read
// anything.  Called by every thread of every CTA; launched the ordinary way a
// kernel waits for nothing.
__device__ __forceinline__ void after_previous_stage() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Volumes of up to this many blocks are launch-bound: a 64^3 sphere from a
// warm cache (4096 blocks) takes 46 us with its stages launched ahead, 52
// without.  In larger ones waiting CTAs hold shared memory that the running
// stage would have as cache.  Whole calls as graphs, warm and cold, spheres at
// 16 and noise at 8 bits a value: from 512 to 8000 blocks launching ahead took
// between 7 us less and 1 more; at 9261 blocks 6 less (sphere, warm) to 7 more
// (noise, cold), at 13824 up to 8 more, at 21952 up to 4 more; five surfaces of
// 512^3 noise 1725 against 1620.
constexpr uint32_t kAheadBlocks = 8192;

// launch a stage whose kernel calls after_previous_stage
inline void launch_next(const Launch &L, void (*kernel)(Launch), int grid, int threads, size_t smem, cudaStream_t st) {
    cudaLaunchAttribute ahead{};
    ahead.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    ahead.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &ahead;
    c.numAttrs = !L.vols && L.one.g.nb <= kAheadBlocks ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, L);            // (errors: the caller's cudaGetLastError)
}

__device__ __forceinline__ uint32_t ceil_div(uint32_t a, uint32_t b) { return (a + b - 1) / b; }

// pre[v] = sum of count(u) for u < v, for v in [0, n]; returns pre[n].
// Called by all threads of the block (any block size); n <= kMaxBatch.
// Each thread takes a run of consecutive volumes; count() is evaluated
// twice per volume (sum, then placement) instead of being kept.
template <class F>
__device__ __forceinline__ uint32_t block_prefix(uint32_t n, F count, uint32_t *pre) {
    __shared__ uint32_t warp_tot[32];
    const uint32_t per = (n + blockDim.x - 1) / blockDim.x;
    const uint32_t v0 = threadIdx.x * per, v1 = min(n, v0 + per);
    uint32_t sum = 0;
    for (uint32_t v = v0; v < v1; v++) sum += count(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = (blockDim.x + 31) >> 5;
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < nwarps ? warp_tot[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        if (lane < nwarps) warp_tot[lane] = wi - w;
    }
    __syncthreads();
    uint32_t run = warp_tot[warp] + incl - sum;
    for (uint32_t v = v0; v < v1; v++) {
        pre[v] = run;
        run += count(v);
    }
    if (v0 < n && v1 == n) pre[n] = run;          // the owner of the last volume writes the total
    if (n == 0 && threadIdx.x == 0) pre[0] = 0;
    __syncthreads();
    return pre[n];
}

// Volume v of a launch: from the parameters (kOne) or the device table.
template <bool kOne>
__device__ __forceinline__ const VolEntry &vol_of(const Launch &L, uint32_t v) {
    if (kOne) return L.one;
    return L.vols[v];
}

// the volume owning virtual item x (x < pre[n]): largest v with pre[v] <= x
__device__ __forceinline__ uint32_t find_vol(const uint32_t *pre, uint32_t n, uint32_t x) {
    uint32_t lo = 0, hi = n - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (pre[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Work-item bookkeeping of a launch: the per-volume prefix of item counts
// (shared memory, batches only), the volume of item x, its first item and
// its item count.  A single volume needs no table.
template <bool kOne, class F>
__device__ __forceinline__ uint32_t launch_prefix(const Launch &L, F count, uint32_t *pre) {
    if (kOne) return count(0u);
    return block_prefix(L.n, count, pre);
}

template <bool kOne>
__device__ __forceinline__ uint32_t item_vol(const uint32_t *pre, uint32_t n, uint32_t x) {
    return kOne ? 0u : find_vol(pre, n, x);
}

template <bool kOne>
__device__ __forceinline__ uint32_t item_base(const uint32_t *pre, uint32_t v) {
    return kOne ? 0u : pre[v];
}

template <bool kOne>
__device__ __forceinline__ uint32_t vol_items(const uint32_t *pre, uint32_t v, uint32_t total) {
    return kOne ? total : pre[v + 1] - pre[v];
}

}  // namespace bcmc

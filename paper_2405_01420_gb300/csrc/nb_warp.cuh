// Warp-level helpers of the gathered-tile kernels: asynchronous copies into
// shared memory, a reduce-scatter of per-lane partial sums, the order in
// which persistent warps take their work.
#pragma once

#include <cuda_runtime.h>

// cp.async of 16 bytes, global -> shared (cached in L1).
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem) : "memory");
}

// Waits for this thread's outstanding cp.async copies.
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Sums v[0..N-1] (N = 8, 16 or 32) over the 32 lanes of the warp. Each step
// halves the values a lane holds: lanes with bit o set keep the upper half
// and send the lower one to lane ^ o, and the other way round. On return
// v[0] of lane l holds the warp total of value l >> (5 - log2 N).
template <int N>
__device__ __forceinline__ void reduce_scatter(float (&v)[N], int lane) {
    static_assert(N == 8 || N == 16 || N == 32, "reduce_scatter: N must be 8, 16 or 32");
    int o = 16;
#pragma unroll
    for (int n = N; n > 1; n >>= 1, o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const float send = upper ? v[i] : v[i + n / 2];
            const float keep = upper ? v[i + n / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
}

// Work items handed out by a counter. Ticket k stands for the items [a, b):
// the first three quarters of the n items go in runs of `run`, the rest one
// by one, so that the launch still ends with single items. Atomics on one
// address are served one per 1.3 ns, too slowly for a ticket per short item.
__device__ __forceinline__ void ticket_items(unsigned k, unsigned n, unsigned run, unsigned &a, unsigned &b) {
    const unsigned runs = run > 1u ? (n - n / 4u) / run : 0u;
    const bool in_run = k < runs;
    a = in_run ? k * run : runs * run + (k - runs);
    b = a + (in_run ? run : 1u);
}

// Items per run for nwarps warps: at least 6 runs for each warp.
__device__ __forceinline__ unsigned ticket_run(unsigned n, unsigned nwarps) { return min(max(n / (8u * nwarps), 1u), 8u); }

// vsd_grid.cuh -- what the kernels of several translation units share: waits
// and queues between blocks, and launch helpers.
#pragma once

#include "vsd_launch.h"

namespace vsd {

// Bounded wait for a flag set by another block; gives up after timeout_ns or
// as soon as another wait has timed out (status bit), never spins forever.
__device__ __forceinline__ bool wait_flag(const int* flag, int* status, uint64_t timeout_ns) {
    if (ld_acquire(flag)) return true;
    const uint64_t t0 = global_timer_ns();
    for (;;) {
        if (ld_acquire(flag)) return true;
        if (*(volatile int*)status & VSD_STATUS_TIMEOUT) return false;
        if (global_timer_ns() - t0 > timeout_ns) return false;
        __nanosleep(1000);
    }
}

// Residual queue (persistent kernel): producers reserve slots, write the items
// and release each slot's flag.
__device__ __forceinline__ void publish_residuals(int* tail, int* flags, int* items, int first,
                                                  int n) {
    const int base = atomicAdd(tail, n);
    for (int i = 0; i < n; ++i) items[base + i] = first + i;
    __threadfence();
    for (int i = 0; i < n; ++i) st_release(flags + base + i, 1);
}

// Static plus dynamic shared memory above 48 KB needs the kernel's opt-in
// (made once per kernel and device).
template <typename K>
static cudaError_t prep(K kernel, size_t smem) {
    return ensure_dyn_smem(reinterpret_cast<const void*>(kernel), smem);
}

// The call's counters (n bytes of the workspace, a multiple of 16) to zero, as a
// kernel, so that the first kernel of the call can be its programmatic
// dependent and read its rows meanwhile (a memset's completion costs the call
// about 2 us before its first kernel starts).
static __global__ void __launch_bounds__(256) k_clear(uint4* p, int n) {
    grid_launch_next();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < n) p[i] = make_uint4(0u, 0u, 0u, 0u);
}
static inline cudaError_t clear_words(void* ws, size_t bytes, cudaStream_t s) {
    const int n = (int)(bytes / 16);
    k_clear<<<(n + 255) / 256, 256, 0, s>>>(static_cast<uint4*>(ws), n);
    return cudaGetLastError();
}

// Launch `kern`; after: as a programmatic dependent of the stream's previous
// kernel: its blocks may become resident while that kernel's last ones still run,
// and wait in grid_wait() until it has completed and its writes are visible.
template <typename... P, typename... A>
static cudaError_t launch(bool after, void (*kern)(P...), unsigned grid, unsigned threads,
                          size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = after ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}
template <typename K, typename... A>
static cudaError_t launch_after(K kern, unsigned grid, unsigned threads, size_t smem,
                                cudaStream_t s, A... args) {
    return launch(true, kern, grid, threads, smem, s, args...);
}

}  // namespace vsd

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

// Residual queue: producers reserve slots (resq_tail), write the items,
// release each slot's flag and then add the items to resq_avail.  A consumer
// reserves one published item with one atomic on resq_avail (returned at once
// if none was left) and takes the next slot with one atomic on resq_head, so
// claims pipeline in L2 instead of queueing behind a compare-and-swap.  The
// slot may belong to a producer that reserved it but has not released it yet
// (it is running, past its reservation): a bounded wait on the flag.
// Callers look at resq_avail first.  Returns the item, -1 if none was left,
// -2 if the wait ran out (status bit set).
__device__ __forceinline__ int take_residual(int* head, int* avail, const int* flags,
                                             const int* items, int* status,
                                             uint64_t timeout_ns) {
    if (atomicSub(avail, 1) <= 0) {
        atomicAdd(avail, 1);
        return -1;
    }
    const int h = atomicAdd(head, 1);
    if (!wait_flag(flags + h, status, timeout_ns)) {
        atomicOr(status, VSD_STATUS_TIMEOUT);
        return -2;
    }
    return ld_cg(items + h);
}

__device__ __forceinline__ void publish_residuals(int* tail, int* avail, int* flags, int* items,
                                                  int first, int n, bool sem) {
    const int base = atomicAdd(tail, n);
    for (int i = 0; i < n; ++i) items[base + i] = first + i;
    __threadfence();
    for (int i = 0; i < n; ++i) st_release(flags + base + i, 1);
    if (sem) atomicAdd(avail, n);
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

// Launch `kern` as a programmatic dependent of the stream's previous kernel: its
// blocks may become resident while that kernel's last ones still run, and wait
// in grid_wait() until it has completed and its writes are visible.
template <typename... P, typename... A>
static cudaError_t launch_after(void (*kern)(P...), unsigned grid, unsigned threads, size_t smem,
                                cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

}  // namespace vsd

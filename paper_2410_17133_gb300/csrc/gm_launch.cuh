// Launches that overlap with the tail of the kernel before them.
//
// The solvers' inner loops are chains of kernels of a few microseconds, each
// reading what the one before wrote.  With programmatic stream serialisation the
// next kernel is launched once every CTA of its predecessor has started, takes
// its place on the SMs and waits in gm_chain until the predecessor has
// completed and its writes are visible; the launch itself costs no time then.
// A kernel launched this way takes `chained` first and calls gm_chain(chained)
// before it touches global memory, in every thread and on every path, so
// completion is transitive along the chain: a kernel cannot complete before its
// predecessors have.  Its loads are coherent ones: the kernel is already there while
// its predecessor writes, so nothing that it reads is read-only for its lifetime, and
// a non-coherent load (__ldg, __restrict__) could be served or moved ahead of the wait.
// Kernels in between that are launched normally wait for completion as usual.
// Measured, chained against plain launches: outside graphs J on 8^3 cells 49.2 -> 45.7 us,
// five tetrahedral products 102.9 -> 94.3 us, the FP32 products at 160^3 551 -> 528 us; in
// captured graphs it loses (FP32 step at 64^3 84 -> 89 ms, FP64 K_T solve at 48^3
// 60.5 -> 66.8 ms), so there the launches are plain and gm_chain returns at once.
#pragma once

#include <cuda_runtime.h>

__device__ __forceinline__ void gm_chain(int chained)
{
    if (!chained) return;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

inline bool gm_capturing(cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
        (void)cudaGetLastError();      // the legacy stream while another one captures
        return true;
    }
    return st != cudaStreamCaptureStatusNone;
}

template <typename... Params, typename... Args>
inline cudaError_t gm_launch_chained(void (*kernel)(int, Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                     Args&&... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    const int chained = gm_capturing(s) ? 0 : 1;
    cfg.numAttrs = chained;
    return cudaLaunchKernelEx(&cfg, kernel, chained, static_cast<Args&&>(args)...);
}

// Shared host/device helpers of libfp4q (internal; the public interface is include/fp4q.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fp4q.h"

namespace fp4q {

constexpr int kBlock = 32;  // 2D block size b (Section 3: 32x32 blocks)

static inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
static inline int64_t round_up(int64_t a, int64_t b) { return ceil_div(a, b) * b; }
static inline bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Layout of the GEMM workspace (device memory, caller-owned).
struct Workspace {
    uint32_t status;         // 0 = ok, otherwise an fp4q_status written by a kernel
    uint32_t detail;         // where the kernel gave up (role/stage), for diagnostics
    uint32_t wait_limit;     // polls (of up to about 1 us) after which a bounded wait gives up; 0 = the kernels' default
    uint32_t withhold_load;  // development hook, 0 in production: n > 0 = CTA 0 leaves out its n-th stage load
    uint32_t pad[60];
};

// Short launches overlap their predecessor's end: quantizers of up to kShortGrid CTAs and short products (launch_gemm_impl says
// which) are launched as the programmatic dependents of the kernel before them in their stream (behind a copy, or a kernel that
// admits nobody before it ends, the attribute changes nothing), so their CTAs may be placed, and set up barriers and tensor memory,
// while the last CTAs of that kernel still run.  Before it touches global memory - reads an input or writes an output - every
// thread waits until that kernel has completed and its writes are visible: streams keep their order.  A kernel lets its own
// successor in only after that wait, so that whoever skips the wait (the later tensors of a multi-tensor quantizer call) still
// runs behind everything before the call.  What the predecessor wrote is read with ordinary loads: the non-coherent path
// (ld.global.nc, __ldg) is for memory that nothing writes while the kernel runs, and a dependent kernel runs before its
// inputs are complete.
// A product lets nobody in before it ends: its last wave leaves some SMs idle for microseconds, and a quantizer that
// is admitted then is placed on those alone.  Passes of quantizers and products, us, products that admit early with quantizers
// of up to 1184 and 148 CTAs dependent, and products that do not with up to 1184: 512 x 1024 x 1024 36.3 / 36.3 / 35.3,
// 2048 x 2048 x 2048 49.3 / 48.8 / 45.4, 4096 x 4096 x 4096 151.5 / 147.3 / 142.8, 8192 x 2048 x 2048 quantized by one call 103.9 / 94.5 /
// 92.4, experts of 1024 tokens 38.9 / 38.9 / 34.5, three ragged operands by one call 26.8 / 28.1 / 26.8.
// Long grids do not take part: in a dependent launch the wait costs every CTA of the grid, not only the first ones.  Nor do
// quantizers in a captured graph, whose launches cost less: there they lose (256 x 512 x 1024 33.3 without and 36.1 us with,
// expert layer of 1024 tokens 34.5 and 36.3).
constexpr int64_t kShortGrid = 2 * 4 * 148;   // two waves of four CTAs per SM
inline bool capturing(cudaStream_t stream)
{
    cudaStreamCaptureStatus st;
    if (cudaStreamIsCapturing(stream, &st) == cudaSuccess) return st != cudaStreamCaptureStatusNone;
    cudaGetLastError();   // the legacy stream beside another stream's capture: the launch itself will report it
    return true;
}
// A launch of `kernel` with one parameter block; always: as a dependent whatever its size.
template <typename P>
inline cudaError_t launch_dependent(void (*kernel)(const P), dim3 grid, int threads, cudaStream_t stream, const P &p, bool always = false, int smem = 0)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = always || ((int64_t)grid.x * grid.y <= kShortGrid && !capturing(stream)) ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}
// The status of a launch that returned e.  Only this launch counts, not an error that an earlier call of somebody else's left
// behind, and its own error is not left for the next caller to find.
inline fp4q_status launched(cudaError_t e)
{
    if (e == cudaSuccess) return FP4Q_OK;
    cudaGetLastError();
    return FP4Q_ERR_CUDA;
}
#ifdef __CUDACC__
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// An ordinary load; it stays below wait_for_predecessor(), which clobbers memory.
template <typename T>
__device__ __forceinline__ T load_global(const T *p) { return *p; }
__device__ __forceinline__ void admit_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

}  // namespace fp4q

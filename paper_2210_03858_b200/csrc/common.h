// Helpers shared by the translation units of the library.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <utility>

#include "../../include/bcq.h"

#define BCQ_MAX_Q 8
#define BCQ_MAX_QUANT_G 32768

namespace bcq {

// cudaError_t of the last failing CUDA call on this thread (read by bcq_last_cuda_error()).
void set_last_cuda_error(int e);

// Called once per kernel launch (bcq_kernel_launches()).
void count_launch();

inline bcq_status cuda_fail(cudaError_t e) {
    set_last_cuda_error((int)e);
    return BCQ_ERR_CUDA;
}

#define BCQ_CUDA_TRY(expr)                                  \
    do {                                                    \
        cudaError_t e__ = (expr);                           \
        if (e__ != cudaSuccess) return bcq::cuda_fail(e__); \
    } while (0)

// Shape rules shared by every entry point (see include/bcq.h).
inline bcq_status check_shape(int d_out, int d_in, int q, int g) {
    if (d_out < 1 || d_in < 1 || q < 1 || g < 1 || g > d_in) return BCQ_ERR_SHAPE;
    if (q > BCQ_MAX_Q) return BCQ_ERR_UNSUPPORTED;
    if (g != d_in && (g % 32) != 0) return BCQ_ERR_UNSUPPORTED;
    return BCQ_OK;
}

// Number of SMs of the current device (148 on a B200; that value is also the answer when no device
// can be asked, e.g. for size queries on a machine without a GPU).
inline int sm_count() {
    static int cached = 0;
    if (cached == 0) {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0)
            cached = n;
        else
            return 148;  // not cached, so a later call with a device present asks again
    }
    return cached;
}

// Launches a kernel so that it may start while the kernel before it in the stream is finishing
// (programmatic dependent launch): its blocks are scheduled and run up to their pdl_wait() early, which
// takes 2 - 3 us of launch latency and set-up off every kernel of a chain.  Every kernel launched this way
// calls pdl_wait() in all threads before it touches global memory.  cluster: CTAs per cluster.
// A kernel that calls pdl_trigger() lets the next one in as soon as its own last blocks have a place, and
// what is let in then takes the SMs that happen to be free: several blocks to one SM while others are busy.
// That is good for kernels of a few microseconds whose successor has few or light blocks, and bad before the
// pre-pass of the forward / dX (prepare_kernel), whose blocks then share a few SMs' bandwidth (the
// regrouping of planes before it with the trigger, 1600 x 6400, 64 tokens, q = 3: 61 us a call, without
// 36.5), before dalpha's reduction, and between long kernels (alternating quantizer, q = 6, 512 x 512,
// g = 64: 268 us with, 240 without).
template <typename... Params, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, unsigned cluster,
                              Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

#ifdef __CUDACC__
// Loads from global memory.  A kernel launched by launch_pdl is alive while the kernel before it still
// writes, and what that kernel writes are its inputs.  So its loads may not take the non-coherent path
// (ld.global.nc, __ldg, what the compiler makes of const __restrict__), which is defined only for memory
// that nobody writes while the kernel lives, and they must stay behind pdl_wait(): these are ordinary loads
// in volatile asm, which keeps its place.  ld_stream stays out of L1 (data that an SM reads once).
// Measured over the calls of a layer: no difference to the non-coherent loads.
#define BCQ_DEFINE_LOAD(name, how)                                                                             \
    template <typename T>                                                                                      \
    __device__ __forceinline__ T name(const T* p) {                                                            \
        static_assert(sizeof(T) == 4 || sizeof(T) == 8 || sizeof(T) == 16, "4, 8 or 16 bytes");                \
        T v;                                                                                                   \
        if constexpr (sizeof(T) == 4) {                                                                        \
            uint32_t r;                                                                                        \
            asm volatile("ld.global" how ".b32 %0, [%1];" : "=r"(r) : "l"(p));                                 \
            memcpy(&v, &r, 4);                                                                                 \
        } else if constexpr (sizeof(T) == 8) {                                                                 \
            uint2 r;                                                                                           \
            asm volatile("ld.global" how ".v2.b32 {%0,%1}, [%2];" : "=r"(r.x), "=r"(r.y) : "l"(p));            \
            memcpy(&v, &r, 8);                                                                                 \
        } else {                                                                                               \
            uint4 r;                                                                                           \
            asm volatile("ld.global" how ".v4.b32 {%0,%1,%2,%3}, [%4];"                                        \
                         : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));                               \
            memcpy(&v, &r, 16);                                                                                \
        }                                                                                                      \
        return v;                                                                                              \
    }
BCQ_DEFINE_LOAD(ld, "")
BCQ_DEFINE_LOAD(ld_stream, ".L1::no_allocate")
#undef BCQ_DEFINE_LOAD

// Until the kernel before this one in the stream has finished and its writes are visible.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The kernel after this one may be scheduled once every CTA of this one has said so (or ended).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

}  // namespace bcq

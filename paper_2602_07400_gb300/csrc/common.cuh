// Internal helpers shared by the CUDA translation units of libbitlogic.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "bitlogic.h"

namespace bitlogic {

// Device-side index flag.  `static` gives each translation unit its own
// copy; every unit registers a reader with bitlogic_device_error().
static __device__ unsigned int g_index_error;

__device__ __forceinline__ void flag_index_error() { atomicOr(&g_index_error, 1u); }

// Reads and clears this unit's flag (synchronizes the stream).
static inline int read_and_clear_index_error(cudaStream_t stream) {
    unsigned int v = 0, zero = 0;
    if (cudaMemcpyFromSymbolAsync(&v, g_index_error, sizeof(v), 0,
                                  cudaMemcpyDeviceToHost, stream) != cudaSuccess)
        return BITLOGIC_ERR_CUDA;
    if (cudaMemcpyToSymbolAsync(g_index_error, &zero, sizeof(zero), 0,
                                cudaMemcpyHostToDevice, stream) != cudaSuccess)
        return BITLOGIC_ERR_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return BITLOGIC_ERR_CUDA;
    return v ? BITLOGIC_ERR_DEVICE : BITLOGIC_OK;
}

inline int launch_status() {
    return cudaGetLastError() == cudaSuccess ? BITLOGIC_OK : BITLOGIC_ERR_CUDA;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Number of SMs of the current device (queried once per device, then
// cached; 152 if the query fails).  Defined in abi.cu.
int sm_count();

// Wire bit rows (the layer-1 input at one bit per sample): samples per word
// block; a row holds 32 words per block, bit 8 m + r of word L being the
// block's sample 128 r + 4 L + m.
constexpr int kBitBlock = 1024;

// Thresholds travel by value in the kernel parameters: no constant-memory
// state is shared between calls or streams.
struct Thresholds {
    int b;
    uint8_t t[32];
};

// Threshold i of a by-value Thresholds with a compile-time unrolled select
// (a runtime index into kernel parameters would copy them to local memory).
__device__ __forceinline__ uint32_t threshold_at(const Thresholds& th, int i) {
    uint32_t v = 0;
#pragma unroll
    for (int q = 0; q < 32; ++q)
        if (q == i) v = th.t[q];
    return v;
}

inline int make_thresholds(const uint8_t* thr_host, int32_t b, Thresholds* out) {
    if (!thr_host) return BITLOGIC_ERR_NULL;
    if (b < 1 || b > 32) return BITLOGIC_ERR_THRESH;
    out->b = b;
    for (int i = 0; i < 32; ++i) out->t[i] = i < b ? thr_host[i] : 0;
    return BITLOGIC_OK;
}

// Logistic function on the CUDA-core FP32 path: CUDA's expf and an
// IEEE-rounded division (no fast-math).
__device__ __forceinline__ float sigmoidf(float z) { return 1.0f / (1.0f + expf(-z)); }

// Table entry of a node form (bitlogic_node_t): the sigmoid sg of the logit
// th for the soft LightLUT node, the hard sample [th > 0] for the
// straight-through node (whose theta gradient still takes the slope of sg).
__device__ __forceinline__ float table_value(float th, float sg, int node) {
    return node == BITLOGIC_NODE_ST ? (th > 0.f ? 1.f : 0.f) : sg;
}

// Asynchronous global -> shared copies (cp.async), 16 bytes (bypassing L1) or
// 4, grouped per pipeline stage.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {   // 4 bytes, through L1
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
// The line at p on its way to L2.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p)); }
// The same copies, or zeros (nothing is read) unless `take`.
__device__ __forceinline__ void cp_async16_or_zero(void* smem, const void* gmem, bool take) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(take ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4_or_zero(void* smem, const void* gmem, bool take) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(s), "l"(gmem), "r"(take ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Reduce-scatter of N values per lane over the lane offsets O, O/2, ..., 1:
// at each step a lane keeps half of its values (the upper half when lane bit
// O is set), adds its partner's copy of that half and hands over the other
// half; once one value is left the remaining steps add it across lanes.
// Afterwards, for N0 = 2^k >= 32 values, lane l holds the sums of entries
// l N0/32 .. l N0/32 + N0/32 - 1; for N0 < 32, of entry l >> (5 - k).  The
// order of every addition is fixed.
template <int N, int O, int M>
__device__ __forceinline__ void warp_reduce_scatter(float (&v)[M], int lane) {
    if constexpr (O > 0) {
        if constexpr (N > 1) {
            const bool up = (lane & O) != 0;
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                const float send = up ? v[i] : v[i + N / 2];
                const float keep = up ? v[i + N / 2] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
            }
            warp_reduce_scatter<N / 2, O / 2>(v, lane);
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], O);
            warp_reduce_scatter<1, O / 2>(v, lane);
        }
    }
}

// Programmatic dependent launch (sm_90 and later).  A kernel launched with
// launch_dependent() may start while the kernel before it on the stream is
// still finishing: it runs grid_dependency_wait() before its first access to
// memory that the earlier work writes or reads, and the wait returns once that
// work has completed with its writes visible.  The earlier kernel lets its
// dependent start early with allow_dependent_launch() (else the dependent
// starts as its blocks exit).  When the previous operation on the stream is
// not a kernel, the launch is an ordinary one and the wait returns at once.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void allow_dependent_launch() {
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

// First statement of every kernel launched with launch_dependent(): wait for
// the work before it on the stream, then let the next kernel be scheduled.
// Waiting before triggering makes the chain transitive: once a kernel's wait
// returns, everything before its predecessor has completed too.
__device__ __forceinline__ void dependent_kernel_start() {
    grid_dependency_wait();
    allow_dependent_launch();
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                    cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace bitlogic

#define BITLOGIC_ERROR_READER(name)                                            \
    extern "C" int bitlogic_internal_index_error_##name(cudaStream_t s) {      \
        return bitlogic::read_and_clear_index_error(s);                        \
    }

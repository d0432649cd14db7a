// Device-side helpers shared by the kernel translation units: typed
// population loads and stores (deviations s = f - w kept as FP32, FP16,
// BF16 or FP64, arithmetic in R), the compact-cell row lookup, and the
// precision switch of the launchers.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "lbm_kernels.h"

namespace lbm {

template <class S> struct Storage;
template <> struct Storage<float> {
    using R = float;
    static __device__ __forceinline__ float ld(const float *p) { return __ldg(p); }
    static __device__ __forceinline__ void st(float *p, float v) { *p = v; }
};
template <> struct Storage<double> {
    using R = double;
    static __device__ __forceinline__ double ld(const double *p) { return __ldg(p); }
    static __device__ __forceinline__ void st(double *p, double v) { *p = v; }
};
template <> struct Storage<__half> {
    using R = float;
    static __device__ __forceinline__ float ld(const __half *p) { return __half2float(__ldg(p)); }
    static __device__ __forceinline__ void st(__half *p, float v) { *p = __float2half_rn(v); }
};
template <> struct Storage<__nv_bfloat16> {
    using R = float;
    static __device__ __forceinline__ float ld(const __nv_bfloat16 *p) { return __bfloat162float(__ldg(p)); }
    static __device__ __forceinline__ void st(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
};

// Stores that stay in L2 in preference to what streams through it: the next
// kernel begins on the cells stored last (band velocities, or the next
// stream-collide in the opposite order).  96 uneven tubes FP32 467 -> 455 us
// per step, aorta 217.5 -> 215.0; FP16 343.3 -> 341.7 and 186.9 -> 185.3.  (Marking the loads to leave first is
// slower, 467 -> 532: lines are shared between neighbouring rows.)  Only where the
// populations exceed the L2 (LARGE): else plain stores, in kernels of
// their own, as the hint costs something even where it says nothing.  keep is true
// in the LARGE kernels; with the policy selected by it the 32-register ones spill
// less than with a constant one (FP16 132 instead of 148 bytes: 100 steps of 96
// uneven tubes 34.16 instead of 34.61 ms).
__device__ __forceinline__ uint64_t keep_in_l2(bool keep) {
    uint64_t last, normal;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(last));
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(normal));
    return keep ? last : normal;
}
__device__ __forceinline__ void st_keep(float *a, float v, uint64_t p) {
    asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(a), "f"(v), "l"(p) : "memory");
}
__device__ __forceinline__ void st_keep(double *a, double v, uint64_t p) {
    asm volatile("st.global.L2::cache_hint.f64 [%0], %1, %2;" ::"l"(a), "d"(v), "l"(p) : "memory");
}
__device__ __forceinline__ void st_keep(__half *a, float v, uint64_t p) {
    asm volatile("st.global.L2::cache_hint.u16 [%0], %1, %2;" ::"l"(a), "h"(__half_as_ushort(__float2half_rn(v))), "l"(p)
                 : "memory");
}
__device__ __forceinline__ void st_keep(__nv_bfloat16 *a, float v, uint64_t p) {
    asm volatile("st.global.L2::cache_hint.u16 [%0], %1, %2;" ::"l"(a), "h"(__bfloat16_as_ushort(__float2bfloat16_rn(v))),
                 "l"(p)
                 : "memory");
}

// row of compact cell c: the row of its 32-cell chunk's first cell plus the
// number of rows that begin within the chunk up to c's lane
__device__ __forceinline__ int find_row(const KParams &p, int c) {
    const int2 ch = __ldg(reinterpret_cast<const int2 *>(p.chunk_row) + (c >> 5));
    const uint32_t upto = (2u << (c & 31)) - 1u;  // lanes 0..(c & 31)
    return ch.x + __popc((uint32_t)ch.y & upto);
}

// relaxation rate of an instance in the arithmetic type R
template <class R> __device__ __forceinline__ R omega_of(const KParams &p, int inst);
template <> __device__ __forceinline__ float omega_of<float>(const KParams &p, int inst) { return __ldg(&p.omega_f[inst]); }
template <> __device__ __forceinline__ double omega_of<double>(const KParams &p, int inst) { return __ldg(&p.omega[inst]); }

template <class S> static S *as(void *p) { return static_cast<S *>(p); }

// Programmatic dependent launch: a kernel lets its successor on the stream start
// its set-up, and waits for its predecessor's end before it touches what that
// one writes.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// a launch that may start before its predecessor on the stream has finished (its
// kernel calls wait_for_previous)
template <class... P, class... A>
cudaError_t launch_early(void (*k)(P...), dim3 grid, dim3 block, cudaStream_t s, const A &...args) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

// the storage types with FP32 arithmetic
#define DISPATCH_F32(prec, CALL)                               \
    switch (prec) {                                            \
    case 1: { using S = __half; CALL; } break;                 \
    case 2: { using S = __nv_bfloat16; CALL; } break;          \
    default: { using S = float; CALL; } break;                 \
    }

#define DISPATCH(prec, CALL)                                   \
    switch (prec) {                                            \
    case 0: { using S = float; CALL; } break;                  \
    case 1: { using S = __half; CALL; } break;                 \
    case 2: { using S = __nv_bfloat16; CALL; } break;          \
    default: { using S = double; CALL; } break;                \
    }

}  // namespace lbm

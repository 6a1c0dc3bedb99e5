// rd_pack.cuh -- scalar and packed (two cells) FP32 operations of the step
// kernels (sm_103a).
#pragma once

#include <cuda_runtime.h>

namespace rdk {

constexpr int kVEC = 4;               // cells per thread position (x)

// The per-cell formulas below are templates over V: float (one cell) or
// float2 (two cells, one packed FP32 instruction per operation; each half is
// rounded exactly as the scalar instruction rounds it, so both give the same
// bits).  The step kernels are bound by instruction issue, and the packed
// forms halve the issue slots of the arithmetic.
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float vneg(float a) { return -a; }
#define RD_PACKED2(name, op)                                                         \
    __device__ __forceinline__ float2 name(float2 a, float2 b) {                     \
        unsigned long long r;                                                        \
        asm(op ".rn.f32x2 %0, %1, %2;"                                               \
            : "=l"(r)                                                                \
            : "l"(reinterpret_cast<unsigned long long&>(a)),                         \
              "l"(reinterpret_cast<unsigned long long&>(b)));                        \
        return reinterpret_cast<float2&>(r);                                         \
    }
RD_PACKED2(vadd, "add")
RD_PACKED2(vsub, "sub")
RD_PACKED2(vmul, "mul")
#undef RD_PACKED2
// A product that a sum or difference takes: two scalar products, because the
// assembler contracts a packed product with the packed sum it feeds (seen in
// the results of a probe, with the rounding of both written out), and the
// scalar kernels and the oracle's bounds want it rounded on its own.
__device__ __forceinline__ float vmul_rounded(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 vmul_rounded(float2 a, float2 b) {
    return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
}
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(r)
        : "l"(reinterpret_cast<unsigned long long&>(a)),
          "l"(reinterpret_cast<unsigned long long&>(b)),
          "l"(reinterpret_cast<unsigned long long&>(c)));
    return reinterpret_cast<float2&>(r);
}
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
template <class V> __device__ __forceinline__ V vset(float a);
template <> __device__ __forceinline__ float vset<float>(float a) { return a; }
template <> __device__ __forceinline__ float2 vset<float2>(float a) { return make_float2(a, a); }

// cells 2h, 2h + 1 of a 4-cell vector
__device__ __forceinline__ float2 pair_of(const float (&v)[kVEC], int h) {
    return make_float2(v[2 * h], v[2 * h + 1]);
}
__device__ __forceinline__ void set_pair(float (&v)[kVEC], int h, float2 p) {
    v[2 * h] = p.x;
    v[2 * h + 1] = p.y;
}

// Chained launches.  A step kernel lets the next launch of its stream be
// scheduled when its CTAs finish their last work items (chain_release) and
// itself waits for the launch before it
// (chain_wait) before it touches anything that one writes, so a launch's
// set-up hides behind the end of the launch before it: 0.3 to 0.5 us of a
// small grid's 4 to 6 (97 x 65 x 50 Brusselator 3.0 -> 2.75 us a step, 64^3
// diffusion 2.1 -> 1.9, front 192^3 34.0 -> 33.3).  Released earlier, at its
// start or two planes before its end, the next launch's CTAs land on the SMs
// that happen to have room and stay unbalanced (96^3 Brusselator 5.1 -> 7.4
// and 5.7).  Only kernels that wait so are
// launched with launch_chained; a kernel launched without the attribute starts
// when the one before it has finished, as always.
__device__ __forceinline__ void chain_release() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <class Args>
cudaError_t launch_chained(void (*k)(const Args), const Args& a, int grid, int threads,
                           size_t smem, cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = st ? 1 : 0;   // the legacy default stream: plain launches
    return cudaLaunchKernelEx(&cfg, k, a);
}

}  // namespace rdk

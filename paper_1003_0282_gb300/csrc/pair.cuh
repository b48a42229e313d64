// pair.cuh -- arithmetic on a pair of FP32 values with Blackwell's paired
// FP32 instructions (add/mul/fma on f32x2), and the scalar overloads the
// collision code shares with it.
//
// The bulk kernel updates two nodes of the same radius (two rows of a tile)
// per thread; holding both in one F2 halves the arithmetic instructions.
#pragma once

#include <cuda_runtime.h>

namespace axl {

struct F2 {
    float2 v;
    __device__ __forceinline__ F2() {}
    __device__ __forceinline__ F2(float s) : v(make_float2(s, s)) {}
    __device__ __forceinline__ F2(float a, float b) : v(make_float2(a, b)) {}
};

__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
    F2 r;
    r.v = __fadd2_rn(a.v, b.v);
    return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
    F2 r;
    r.v = __fmul2_rn(a.v, b.v);
    return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
    F2 r;
    r.v = __ffma2_rn(b.v, make_float2(-1.0f, -1.0f), a.v);
    return r;
}
__device__ __forceinline__ F2 fmaR(F2 a, F2 b, F2 c) {
    F2 r;
    r.v = __ffma2_rn(a.v, b.v, c.v);
    return r;
}
__device__ __forceinline__ float fmaR(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmaR(double a, double b, double c) { return fma(a, b, c); }

// Reciprocal in FP32: the hardware estimate (PTX rcp.approx.ftz.f32, within
// about an ulp) refined by one Newton-Raphson step for 1/x, r' = r + r (1 -
// x r), which squares the estimate's relative error; the two fused
// multiply-adds leave the result within one ulp of 1/x (faithful rounding)
// for the normal arguments the collision takes (densities near rho0, radii
// of at least 1/2), without the branches of the correctly rounded call.  The
// scalar and the paired forms round alike, lane by lane.  FP64 has two: D1's,
// below, in the collision, and a divide for what is formed once per column.
__device__ __forceinline__ float rcp_estimate(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp(float x) {
    const float r = rcp_estimate(x);
    return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
__device__ __forceinline__ F2 rcp(F2 x) {
    const float2 r = make_float2(rcp_estimate(x.v.x), rcp_estimate(x.v.y));
    const float2 e = __ffma2_rn(make_float2(-x.v.x, -x.v.y), r, make_float2(1.0f, 1.0f));
    F2 out;
    out.v = __ffma2_rn(r, e, r);
    return out;
}

// One FP64 value whose operations round as written: which products are fused
// is stated in the collision, so that every kernel rounds a node alike (the
// compiler fuses plain double expressions differently from kernel to kernel).
struct D1 {
    double v;
    __device__ __forceinline__ D1() {}
    __device__ __forceinline__ D1(double s) : v(s) {}
};
__device__ __forceinline__ D1 operator+(D1 a, D1 b) { return D1(__dadd_rn(a.v, b.v)); }
__device__ __forceinline__ D1 operator-(D1 a, D1 b) { return D1(__dsub_rn(a.v, b.v)); }
__device__ __forceinline__ D1 operator*(D1 a, D1 b) { return D1(__dmul_rn(a.v, b.v)); }
__device__ __forceinline__ D1 fmaR(D1 a, D1 b, D1 c) { return D1(__fma_rn(a.v, b.v, c.v)); }
// Reciprocal in FP64: the hardware estimate (PTX rcp.approx.ftz.f64, about
// 20 bits) refined by one step of Halley's third-order iteration for 1/x,
// r' = r + r (e + e^2) with e = 1 - x r, which cubes the estimate's relative
// error: three fused multiply-adds, no branch.  The estimate has 21 significant
// bits, so e is exact, and the result is off by half an ulp and e^3 (2^-60
// relative, 2^-7 ulp) at most, for the normal arguments the collision takes
// (axlbm_selftest_rcp64).  A correctly rounded divide costs about three
// times as many FP64 instructions, and FP64 instructions bound these kernels
// (an SM of GB300 takes 19 cycles for one of a warp).
__device__ __forceinline__ D1 rcp(D1 x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x.v));
    const double e = __fma_rn(-x.v, r, 1.0);
    return D1(__fma_rn(r, __fma_rn(e, e, e), r));
}

template <class R>
struct ScalarOf {
    using type = R;
};
template <>
struct ScalarOf<F2> {
    using type = float;
};
template <>
struct ScalarOf<D1> {
    using type = double;
};

// Arithmetic of a node in the step kernels: NodeArith for one node (the ring
// kernels), PairArith for what a thread of the bulk kernels holds.  With FP32
// storage the ring nodes use a pair with equal lanes, so that every FP32
// kernel rounds a node alike.  With 16-bit storage they keep the plain float
// type they have always had: its rounding differs from a lane's in the last
// FP32 bit, and a 16-bit store would turn that into a whole unit of its last
// place.
template <class S, class R>
struct NodeArith {
    using type = R;
};
template <>
struct NodeArith<float, float> {
    using type = F2;
};
template <>
struct NodeArith<double, double> {
    using type = D1;
};
template <class R>
struct PairArith {
    using type = F2;
};
template <>
struct PairArith<double> {
    using type = D1;
};

}  // namespace axl

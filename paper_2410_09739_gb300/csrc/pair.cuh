// pair.cuh -- two cells per thread on the packed fp32 pipe.
//
// sm_100-class GPUs execute fma/add/mul on a pair of fp32 values as one
// instruction (fma.rn.f32x2 and friends).  The collision of two cells is the
// same instruction stream on different data, so a thread that collides two
// cells at once with `f2` arithmetic issues about half the floating-point
// instructions per cell.  Every operation is the IEEE round-to-nearest fp32
// operation on each lane: results equal two scalar collisions up to
// contraction choices (a*b+c written with fma on one side and not the other).
//
// f2 supplies what collide_cell needs from its arithmetic type R: + - * and
// unary minus, fmaR, construction from a constant, the reciprocal recipR, and a
// comparison that is true only when it holds on both lanes (collide_cell's
// validity check).
#pragma once
#include <cuda_runtime.h>

namespace fpc {

struct f2 {
    float2 v;
    f2() = default;
    __host__ __device__ constexpr f2(float2 a) : v(a) {}
    __host__ __device__ constexpr f2(double c) : v{(float)c, (float)c} {}
    __host__ __device__ constexpr f2(float x, float y) : v{x, y} {}
};

__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return f2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return f2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return f2(__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)); }
// (a sign change of a packed operand is folded into the instruction that uses it)
__device__ __forceinline__ f2 operator-(f2 a) { return f2(make_float2(-a.v.x, -a.v.y)); }
__device__ __forceinline__ f2& operator+=(f2& a, f2 b) { return a = a + b; }
__device__ __forceinline__ f2& operator-=(f2& a, f2 b) { return a = a - b; }
__device__ __forceinline__ f2 operator/(f2 a, f2 b) { return f2(make_float2(a.v.x / b.v.x, a.v.y / b.v.y)); }
__device__ __forceinline__ bool operator>(f2 a, f2 b) { return a.v.x > b.v.x && a.v.y > b.v.y; }
__device__ __forceinline__ bool operator<(f2 a, f2 b) { return a.v.x < b.v.x && a.v.y < b.v.y; }
// overloads of collide.cuh's fmaR, fminR (a non-template exact match wins for f2)
__device__ __forceinline__ f2 fminR(f2 a, f2 b) { return f2(fminf(a.v.x, b.v.x), fminf(a.v.y, b.v.y)); }
__device__ __forceinline__ float recipR(float a) { return __frcp_rn(a); }
__device__ __forceinline__ f2 recipR(f2 a) { return f2(__frcp_rn(a.v.x), __frcp_rn(a.v.y)); }

// 1 / a by the hardware's approximation (one ulp) and one Newton step y + y (1 - a y), without a branch.
// On sm_103a the result has the bits of __frcp_rn for every argument from 2^-126 to 2^126 in magnitude
// (all of them compared in tests/test_gpu_recip.py; the step alone guarantees 0.5001 ulp), so which of
// the two a kernel takes does not show in its results.  Zero, infinite and NaN arguments, where the
// step gives NaN, keep the approximation's infinity, zero or NaN; a pair keeps it for every lane whose
// density the step flags as diverged (not 0 < a < 1e30: the same comparisons, so this costs nothing,
// where a test of the result for NaN cost 1.2 % of the 192^3 fp16 case).
// The kernels with one cell per thread use it (45x37x53 fp32, latency-bound: 3.9 -> 3.7 us a step), and
// the odd step of neighbouring pairs with general rates (192^3 fp16: 220 -> 198 us); the other paired
// kernels are faster with __frcp_rn (384x192x192 bf16 channel, even step: 326 us against 359;
// 402x64x201 LES, odd step: 177 against 188).
__device__ __forceinline__ float recip_approx(float a)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a));
    return y;
}
__device__ __forceinline__ float recip_newton(float a)
{
    const float y = recip_approx(a), q = __fmaf_rn(y, __fmaf_rn(-a, y, 1.f), y);
    return q == q ? q : y;
}
__device__ __forceinline__ f2 recip_newton(f2 a)
{
    const float2 y = make_float2(recip_approx(a.v.x), recip_approx(a.v.y));
    const float2 e = __ffma2_rn(make_float2(-a.v.x, -a.v.y), y, make_float2(1.f, 1.f));
    const float2 q = __ffma2_rn(y, e, y);
    return f2(a.v.x > 0.f && a.v.x < 1e30f ? q.x : y.x, a.v.y > 0.f && a.v.y < 1e30f ? q.y : y.y);
}
__device__ __forceinline__ f2 sqrtR(f2 a) { return f2(sqrtf(a.v.x), sqrtf(a.v.y)); }
__device__ __forceinline__ f2 fmaR(f2 a, f2 b, f2 c) { return f2(__ffma2_rn(a.v, b.v, c.v)); }

}  // namespace fpc

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
// overloads of collide.cuh's fmaR, fminR, fmaxR (a non-template exact match wins for f2)
__device__ __forceinline__ f2 fminR(f2 a, f2 b) { return f2(fminf(a.v.x, b.v.x), fminf(a.v.y, b.v.y)); }
__device__ __forceinline__ f2 fmaxR(f2 a, f2 b) { return f2(fmaxf(a.v.x, b.v.x), fmaxf(a.v.y, b.v.y)); }
__device__ __forceinline__ f2 recipR(f2 a) { return f2(__frcp_rn(a.v.x), __frcp_rn(a.v.y)); }

// 1 / a to within an fp32 rounding (0.5001 ulp): the hardware's approximation (one ulp) and one Newton
// step y + y (1 - a y).  Two instructions more than the approximation; an IEEE reciprocal takes about
// 28 and a branch.  Zero, infinite and NaN arguments give NaN where the IEEE reciprocal gives 0, an
// infinity or NaN.  The kernels with one cell per thread use it (45x37x53 fp32, latency-bound: 3.9 ->
// 3.7 us a step) and the general-rate odd step of pairs (192^3 fp16: 220 -> 198 us); the other paired kernels
// schedule better around the branch of the IEEE one (384x192x192 bf16 channel, even step: 326 us
// against 359; 402x64x201 LES, odd step: 177 against 188).
__device__ __forceinline__ float recip_approx(float a)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a));
    return y;
}
__device__ __forceinline__ float recip_newton(float a)
{
    const float y = recip_approx(a);
    return __fmaf_rn(y, __fmaf_rn(-a, y, 1.f), y);
}
__device__ __forceinline__ f2 recip_newton(f2 a)
{
    const f2 y = f2(recip_approx(a.v.x), recip_approx(a.v.y));
    const float2 e = __ffma2_rn(make_float2(-a.v.x, -a.v.y), y.v, make_float2(1.f, 1.f));
    return f2(__ffma2_rn(y.v, e, y.v));
}
__device__ __forceinline__ float recipR(float a) { return recip_newton(a); }
__device__ __forceinline__ f2 sqrtR(f2 a) { return f2(sqrtf(a.v.x), sqrtf(a.v.y)); }
__device__ __forceinline__ f2 fmaR(f2 a, f2 b, f2 c) { return f2(__ffma2_rn(a.v, b.v, c.v)); }

}  // namespace fpc

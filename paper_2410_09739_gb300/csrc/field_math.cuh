// field_math.cuh -- arithmetic of the field kernels (equilibrium from rho, u; rho, u from
// populations) for fp32 and 16-bit storage.
//
// The fields cross the boundary in fp64, but this GPU's fp64 pipe retires about two operations
// per clock and SM against 128 fp32 ones (256^3 cells: 27 us per fp64 operation and cell, against
// 350 us for the traffic of an fp32 box), so a field kernel is bound by that pipe unless it does
// without most of its fp64 operations.  The helpers here keep the accuracy of the fp64 forms on
// the fp32 pipe: numbers as unevaluated sums of two fp32 values (error-free transformations of
// Knuth and Dekker; T. J. Dekker, "A floating-point technique for extending the available
// precision", Numer. Math. 18 (1971)), for one cell (T = float) or two (T = f2, pair.cuh).
#pragma once
#include "common.cuh"
#include "pair.cuh"

namespace fpc {

// Round-to-nearest operations that the compiler neither contracts nor reassociates.
__device__ __forceinline__ float rn_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rn_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float rn_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float rn_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ f2 rn_add(f2 a, f2 b) { return a + b; }
__device__ __forceinline__ f2 rn_sub(f2 a, f2 b) { return a - b; }
__device__ __forceinline__ f2 rn_mul(f2 a, f2 b) { return a * b; }
__device__ __forceinline__ f2 rn_fma(f2 a, f2 b, f2 c) { return fmaR(a, b, c); }

// h + l, |l| a few ulp(h) / 2 at most.
template <typename T>
struct Dual {
    T h, l;
};

// An fp64 value as a Dual.  A conversion instruction takes as many slots of the fp64 pipe as an
// addition, so ordinary magnitudes are split on the integer pipe: the upper 24 significant bits
// (truncated) and the other 29 as an integer times its unit.
__device__ __forceinline__ Dual<float> dual_of(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned ex = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
    if (ex - 949u < 201u) {  // 2^-74 <= |v| < 2^127
        const float h = __uint_as_float(sign | (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29));
        const float unit = __uint_as_float(sign | ((ex - 948u) << 23));  // 2^(ex - 1023 - 52)
        return {h, (float)(lo & 0x1fffffffu) * unit};
    }
    if (((hi & 0x7fffffffu) | lo) == 0u) return {0.f, 0.f};
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}

// fp32 -> fp64 (exact) on the integer pipe.  Subnormals are scaled to normal numbers first; no lane
// falls back on the conversion instruction, which the compiler would execute for every lane.
__device__ __forceinline__ double widen(float v)
{
    const bool tiny = (__float_as_uint(v) & 0x7f800000u) == 0u;
    const unsigned b = __float_as_uint(tiny ? v * 0x1p64f : v), m = b & 0x7fffffffu;
    unsigned hi = (m >> 3) + (tiny ? (896u - 64u) << 20 : 896u << 20);
    if (m == 0u) hi = 0u;
    if (m >= 0x7f800000u) hi |= 0x7ff00000u;  // infinities and NaN
    return __hiloint2double((int)((b & 0x80000000u) | hi), (int)(b << 29));
}

__device__ __forceinline__ Dual<f2> dual_of(double x, double y)
{
    const Dual<float> a = dual_of(x), b = dual_of(y);
    return {f2(a.h, b.h), f2(a.l, b.l)};
}

template <typename T>
__device__ __forceinline__ Dual<T> dual_const(double c)
{
    return {T((float)c), T((float)(c - (double)(float)c))};
}

// s + e = a + b exactly (any magnitudes)
template <typename T>
__device__ __forceinline__ void two_sum(T a, T b, T& s, T& e)
{
    const T t = rn_add(a, b);
    const T bb = rn_sub(t, a);
    e = rn_add(rn_sub(a, rn_sub(t, bb)), rn_sub(b, bb));
    s = t;
}

template <typename T>
__device__ __forceinline__ Dual<T> dual_add(Dual<T> a, Dual<T> b)
{
    Dual<T> r;
    T e;
    two_sum(a.h, b.h, r.h, e);
    r.l = rn_add(e, rn_add(a.l, b.l));
    return r;
}

template <typename T>
__device__ __forceinline__ Dual<T> dual_mul(Dual<T> a, Dual<T> b)
{
    Dual<T> r;
    r.h = rn_mul(a.h, b.h);
    r.l = rn_fma(a.l, b.h, rn_fma(a.h, b.l, rn_fma(a.h, b.h, -r.h)));
    return r;
}

// by a power of two
template <typename T>
__device__ __forceinline__ Dual<T> dual_scale(Dual<T> a, float p)
{
    return {rn_mul(a.h, T(p)), rn_mul(a.l, T(p))};
}

// The sum rounded to fp32 (once, up to the 2^-46 of the Duals themselves).
template <typename T>
__device__ __forceinline__ T dual_sum(Dual<T> a, Dual<T> b)
{
    T s, e;
    two_sum(a.h, b.h, s, e);
    return rn_add(s, rn_add(e, rn_add(a.l, b.l)));
}

// The sum rounded to fp32 by round-to-odd (the last bit set whenever anything is cut off), so that
// rounding it once more, to a type of at most 22 significant bits, gives the sum rounded once
// (S. Boldo and G. Melquiond, "Emulation of a FMA and correctly rounded sums: proved algorithms using
// rounding to odd", IEEE Trans. Comput. 57 (2008)).
__device__ __forceinline__ float dual_sum_odd(Dual<float> a, Dual<float> b)
{
    float s, e, h, l;
    two_sum(a.h, b.h, s, e);
    two_sum(s, rn_add(e, rn_add(a.l, b.l)), h, l);
    const unsigned u = __float_as_uint(h);
    // l points away from zero where it has h's sign: the odd neighbour is then the next larger magnitude
    const unsigned odd = (__float_as_uint(l) ^ u) >> 31 ? u - 1u : u + 1u;
    return l != 0.f && !(u & 1u) ? __uint_as_float(odd) : h;
}

// One axis of the product-form equilibrium at velocity u: the deviations d of the three factors
// from the rest weights, (u^2 - u)/2, -u^2, (u^2 + u)/2, and the factors f = w1 + d.
template <typename T>
struct EqAxis {
    Dual<T> d[3], f[3];
};

template <typename T>
__device__ __forceinline__ EqAxis<T> eq_axis(Dual<T> u)
{
    EqAxis<T> a;
    const Dual<T> q = dual_mul(u, u), n = {-u.h, -u.l};
    a.d[0] = dual_scale(dual_add(q, n), 0.5f);
    a.d[1] = {-q.h, -q.l};
    a.d[2] = dual_scale(dual_add(q, u), 0.5f);
#pragma unroll
    for (int i = 0; i < 3; ++i) a.f[i] = dual_add(dual_const<T>(w1(i)), a.d[i]);
    return a;
}

// Whether |v| < 1024, from the high word (integer pipe).  Cells with a density or velocity beyond
// that, infinite or NaN take the fp64 form: the error terms of a Dual would turn an overflow
// into NaN.
__device__ __forceinline__ bool eq_ordinary(double v) { return (__double2hiint(v) & 0x7fffffff) < 0x40900000; }

// Running sum s + c + d of fp32 terms with the rounding errors of both the sum and the first
// correction captured (Ogita, Rump & Oishi, "Accurate sum and dot product", SIAM J. Sci. Comput.
// 26 (2005), SumK with K = 3): as accurate as 72-bit summation, so for the few terms of a cell
// the fp64 value s + (c + d) is at least as close to the exact sum as fp64 summation.
struct Sum3 {
    float s = 0.f, c = 0.f, d = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        float e, e2;
        two_sum(s, x, s, e);
        two_sum(c, e, c, e2);
        d = rn_add(d, e2);
    }
    __device__ __forceinline__ double value() const
    {
        double t = widen(c);
        if (d != 0.f) t += widen(d);  // rare: terms of very different magnitude
        return widen(s) + t;
    }
};

}  // namespace fpc

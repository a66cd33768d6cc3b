// collide.cuh -- per-cell FPC-LBM collision (Appendix D Steps 7, 1-5) in registers.
//
// The 27 populations of a cell arrive as deviations g[s] = f_s - w_s in tensor
// slot order s = (ex+1) + 3 (ey+1) + 9 (ez+1).  The central-moment transform
// kappa = C(u) f (Steps 1+2) factorises over the axes because the D3Q27
// velocities are a tensor product: three passes of a 3-point transform, each
// along one axis, turn the slot array into d[m + 3n + 9p], the deviation of
// kappa_mnp from the rest-state central moments r_m r_n r_p, r = (1, 0, cs^2).
// Working with deviations keeps every intermediate small, so that fp32
// arithmetic (and 16-bit storage) loses no digits to O(1) cancellations.
//
// A 3-point line (a, b, c) at e = (-1, 0, +1) whose rest values are
// K (1/6, 2/3, 1/6) maps to
//   d0 = a + b + c
//   d1 = (c - a) - u (K + d0)
//   d2 = (a + c) - 2u (c - a) + u^2 (K + d0)
// i.e. the moments sum v (e-u)^k minus their rest values (K, 0, K/3); the
// inverse map follows from raw moments m0 = K + d0, m1 = d1 + u m0,
// m2 = K/3 + d2 + 2u d1 + u^2 m0 and a = (m2-m1)/2, b = m0-m2, c = (m2+m1)/2.
//
// The collision relaxes the grouped moments of Step 3 in the chain order
// 2 -> 3 -> 4 -> 5 -> 6 toward the attractors of Eq. (Mvcmattractor3D) with
// D' of Eq. (diffusion-tensor-parameter-3D), adds the body-force sources of
// Eq. (cmupdatesourceD3Q27) with weight (1 - omega/2), and maps back.
// Readings: first-order moments enter attractors and sources as 0; sources
// use pre-collision moments; attractors of orders 4-6 use post-collision
// lower moments; kappa^Mv_122 carries Pi_110 Pi_012 (continuous form).
// In the modes *_R1 (rates of orders 3-6 equal to 1) the moments of orders 3-6
// are set to their attractors plus half their sources, kappa~ = kappa^Mv +
// sigma / 2, with no grouping.  Without force the third- and fifth-order
// moments then vanish (attractors built from odd moments that are zero after
// the collision), and the unused pre-collision moments of orders 3-6 drop out
// of the forward transform.
#pragma once
#include "common.cuh"
#include "pair.cuh"

namespace fpc {

#define FPC_D(m, n, p) g[(m) + 3 * (n) + 9 * (p)]

template <typename R>
__device__ __forceinline__ R fmaR(R a, R b, R c) { return fma(a, b, c); }
template <typename R>
__device__ __forceinline__ R recipR(R a) { return R(1) / a; }
// 1 / rho of a cell; NEWTON: a pair's takes the short form, as one cell's always does (pair.cuh).
template <bool NEWTON = false, typename R>
__device__ __forceinline__ R recip_rho(R rho)
{
    if constexpr (std::is_same<R, float>::value || (NEWTON && std::is_same<R, f2>::value)) return recip_newton(rho);
    else return recipR(rho);
}
template <typename R>
__device__ __forceinline__ R sqrtR(R a) { return sqrt(a); }
template <typename R>
__device__ __forceinline__ R fminR(R a, R b) { return fmin(a, b); }

// Forward 3-point central-moment transform in deviation form (see header).
template <typename R, bool K0>
__device__ __forceinline__ void fwd3(R& a, R& b, R& c, R u, R u2, R tu, R K)
{
    const R P = a + c, D = c - a, S = P + b;
    const R U = K0 ? S : K + S;
    a = S;
    b = fmaR(-u, U, D);
    c = fmaR(u2, U, fmaR(-tu, D, P));
}

// Inverse of fwd3.
template <typename R, bool K0>
__device__ __forceinline__ void inv3(R& k0, R& k1, R& k2, R u, R u2, R tu, R K)
{
    const R U = K0 ? k0 : K + k0;
    const R M1 = fmaR(u, U, k1);
    const R M2 = fmaR(u2, U, fmaR(tu, k1, k2));
    // (M2 -/+ M1) / 2 with both halvings exact: the same roundings as 0.5 M2 -/+ 0.5 M1, and no
    // separate negation (which costs an instruction in packed f2 arithmetic)
    const R h2 = R(0.5) * M2;
    const R lo = fmaR(R(-0.5), M1, h2);
    const R hi = fmaR(R(0.5), M1, h2);
    const R mid = k0 - M2;
    k0 = lo;
    k1 = mid;
    k2 = hi;
}

// Inverse of fwd3 for moments scaled by 1/2 per axis with a non-zero exponent
// (exact: powers of two), so that the two halvings of a line cost nothing:
// with M1' = M1 / 2, M2' = M2 / 2 the line is (M2' - M1', k0 - 2 M2', M2' + M1'),
// seven operations against inv3's eight.  h = u/2, q = u/4, tu = 2u, h2 = u^2/2
// (read when Z1 only); M2' = tu (q U + k1') + k2'.  Z0, Z1, Z2: k0, k1', k2' known
// to be zero, their terms left out.  K0: the rest constant K vanishes.
template <typename R, bool K0, bool Z0 = false, bool Z1 = false, bool Z2 = false>
__device__ __forceinline__ void inv3h(R& k0, R& k1, R& k2, R h, R q, R tu, R h2, R K)
{
    constexpr bool UZ = K0 && Z0;  // U = K + k0 vanishes
    static_assert(!(UZ && Z1 && Z2), "a line of zeros");
    R U = R(0);
    if constexpr (!UZ) {
        if constexpr (K0) U = k0;
        else if constexpr (Z0) U = K;
        else U = K + k0;
    }
    R M1, M2;
    if constexpr (Z1) {
        static_assert(!UZ, "covered by Z0 lines with k1 only");
        M1 = h * U;
        if constexpr (Z2) M2 = h2 * U;
        else M2 = fmaR(h2, U, k2);
    } else {
        R w = k1;
        if constexpr (!UZ) w = fmaR(q, U, k1);
        if constexpr (UZ) M1 = k1;
        else M1 = fmaR(h, U, k1);
        if constexpr (Z2) M2 = tu * w;
        else M2 = fmaR(tu, w, k2);
    }
    R mid;
    if constexpr (Z0) mid = R(-2) * M2;
    else mid = fmaR(R(-2), M2, k0);
    const R lo = M2 - M1, hi = M2 + M1;
    k0 = lo;
    k1 = mid;
    k2 = hi;
}

// What the shear rates leave: 1 - omega_4, 5, 6, 8, 9 of the cell (Step 3), for
// collide_unit scaled like Rates::unit.  own_shear: those of the box's rates.
template <typename R>
struct Shear {
    R k4, k5, k6, k8, k9;
};

// Unit rates of orders 3-6 and no force or one along x: collide_unit.
__host__ __device__ constexpr bool unit_collision(int force, int mode) { return r1_mode(mode) && force != FORCE_ANY; }
__host__ __device__ constexpr bool scaled_shear(int force, int mode) { return unit_collision(force, mode) && !learned_mode(mode) && !smag_mode(mode); }

template <int FORCE, int MODE, typename R>
__device__ __forceinline__ Shear<R> own_shear(const Rates<R>& rt)
{
    if constexpr (scaled_shear(FORCE, MODE)) return {rt.unit[0], rt.unit[1], rt.unit[2], rt.unit[3], rt.unit[4]};
    else return {rt.keep[4], rt.keep[5], rt.keep[6], rt.keep[8], rt.keep[9]};
}

// Rest constants of the three passes (axis z first, then y, then x).
// Pass A (z lines at fixed (ix, iy)): K = w1(ix) w1(iy)
// Pass B (y lines at fixed (ix, p)):  K = w1(ix) r1(p)
// Pass C (x lines at fixed (n, p)):   K = r1(n) r1(p)
#define FPC_PASS_B(OP)                                                                   \
    {                                                                                    \
        _Pragma("unroll") for (int p = 0; p < 3; ++p)                                    \
            _Pragma("unroll") for (int ix = 0; ix < 3; ++ix)                             \
        {                                                                                \
            const double Kd = w1(ix) * r1(p);                                            \
            if (Kd == 0.0)                                                               \
                OP<R, true>(g[ix + 9 * p], g[ix + 3 + 9 * p], g[ix + 6 + 9 * p], uy, uy2, tuy, R(0)); \
            else                                                                         \
                OP<R, false>(g[ix + 9 * p], g[ix + 3 + 9 * p], g[ix + 6 + 9 * p], uy, uy2, tuy, R(Kd)); \
        }                                                                                \
    }
#define FPC_PASS_C(OP)                                                                   \
    {                                                                                    \
        _Pragma("unroll") for (int p = 0; p < 3; ++p)                                    \
            _Pragma("unroll") for (int n = 0; n < 3; ++n)                                \
        {                                                                                \
            const double Kd = r1(n) * r1(p);                                             \
            if (Kd == 0.0)                                                               \
                OP<R, true>(g[3 * n + 9 * p], g[1 + 3 * n + 9 * p], g[2 + 3 * n + 9 * p], ux, ux2, tux, R(0)); \
            else                                                                         \
                OP<R, false>(g[3 * n + 9 * p], g[1 + 3 * n + 9 * p], g[2 + 3 * n + 9 * p], ux, ux2, tux, R(Kd)); \
        }                                                                                \
    }

// Per-cell learned correction of the shear rates (mode LEARNED): MLP
// 9 -> 64 -> 64 -> 1 with tanh hidden layers on the tensor cores, weights
// packed by fpclbm_set_closure.  Warp-collective; implemented in closure.cuh.
template <typename R>
__device__ R closure_delta_omega(const uint32_t* P, const R in[9]);

// Smagorinsky eddy viscosity (Sec. 4, turbulent channel LES): nu_t = c2 |S|, the strain rate from
// the deviatoric non-equilibrium second moments Pi^d (of the central moments' deviations d from the
// rest state) at the effective time tau, S = -Pi^d / (2 rho cs^2 tau), tau = tau0 + nu_t / cs^2; the
// positive root of tau^2 - tau0 tau - c2 |Pi^d| / (2 rho cs^4) = 0, whose inverse replaces all five
// shear rates.
template <typename R>
__device__ __forceinline__ R smagorinsky_tau(R d200, R d020, R d002, R d110, R d101, R d011, R drho, R inv_rho, R c2,
                                             R tau0)
{
    const R third = R(1.0 / 3.0);
    const R p0 = d200 - third * drho, p1 = d020 - third * drho, p2 = d002 - third * drho;
    const R tr = third * ((p0 + p1) + p2);
    const R q0 = p0 - tr, q1 = p1 - tr, q2 = p2 - tr;
    const R pp = fmaR(q0, q0, fmaR(q1, q1, q2 * q2)) + R(2) * fmaR(d110, d110, fmaR(d101, d101, d011 * d011));
    const R Pn = sqrtR(R(2) * pp);
    return R(0.5) * (tau0 + sqrtR(fmaR(tau0, tau0, R(18) * c2 * Pn * inv_rho)));
}

// The unit-rate collision, without force (first) or with a force along x (XF, below).
// Without force kappa~ = kappa^Mv for orders 3-6, and
// the third- and fifth-order attractors vanish, so the step reads only the moments
// of orders 0-2 and writes 1 + 3 + 6 + 6 + 1 of them:
//   forward   raw moments of orders 0-2 from sums over the lines (69 additions),
//             kappa_ij = m_ij - u_i j_j with one fma each, where the central-moment
//             transform of all three passes took about 160 operations;
//   back      scaled lines (inv3h): every moment is formed divided by 2 per axis
//             with a non-zero exponent, through scaled constants.
// In all about 340 operations per cell against 430 for the transform-based form
// (the fp32 kernels issue them packed, two cells at a time; fp64 is bound by them:
// 32^3 33 -> 27 us a step; bf16 storage, row-staged at 256^3: 0.340 -> 0.311 ms a step).
//
// Momentum.  The back transform of an axis gives sum (u U_l + k_l) over its lines,
// U_l = K + k0_l rounded: the first-order moment must be the residual sum (j_l - u U_l)
// of those very U_l, each term formed by one fma on the line's own j_l, for the momentum
// to come back to the last bit.  j - rho u instead (two operations for 5 + 17) repeats an
// error of u 2^-25 every step of a slowly varying flow: 1.8e-5 of the velocity scale after
// 1,000 fp32 steps of the 256^3 Taylor-Green vortex, against 5.1e-7 with the residuals.
// So the planes are transformed back one after the other, and the U_l of a plane give
// the residual that the next one starts from.
//
// XF: a force along x (channels).  sigma_mnp = m (F_x / rho) kappa_{m-1,n,p}, so the step
// also reads kappa_0np and kappa_1np of all n, p, but no moment with m = 2 except
// kappa_200: raw moments from sums, then shifts of one line of three each (three
// operations instead of a line transform's seven).  About 440 operations against 600
// with the sources of all three components (384x192x192 channel, bf16: 0.426 -> 0.366 ms a step).
template <typename R, bool XF, int MODE>
__device__ __forceinline__ bool collide_unit(R (&g)[27], const Rates<R>& rt, R Fx, const Shear<R>& sh,
                                             const float* closure, R c2)
{
    // z lines: S = sum, D = difference, P the sum of the ez^2 terms
    R S[9], D[9], P[9], E[3], m002, m000, m100, m010, m001, m200, m020, m110, m101, m011;
    R c0[3][3], c1[3][3];  // XF: raw, then central moments (0, n, p) and (1, n, p), [p][n]
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const R lo = g[l], mid = g[l + 9], hi = g[l + 18];
        P[l] = lo + hi;
        D[l] = hi - lo;
        S[l] = P[l] + mid;
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) E[x] = S[x + 6] - S[x];  // y momentum of the columns
    if constexpr (XF) {
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            R y0[3], y1[3], y2[3];
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                const R lo = p == 0 ? S[x] : p == 1 ? D[x] : P[x], mid = p == 0 ? S[x + 3] : p == 1 ? D[x + 3] : P[x + 3];
                const R hi = p == 0 ? S[x + 6] : p == 1 ? D[x + 6] : P[x + 6];
                y2[x] = lo + hi;
                y1[x] = p == 0 ? E[x] : hi - lo;
                y0[x] = y2[x] + mid;
            }
            const R q = y0[0] + y0[2];
            if (p == 0) m200 = q;
            c0[p][0] = q + y0[1];
            c0[p][1] = (y1[0] + y1[2]) + y1[1];
            c0[p][2] = (y2[0] + y2[2]) + y2[1];
            c1[p][0] = y0[2] - y0[0];
            c1[p][1] = y1[2] - y1[0];
            c1[p][2] = y2[2] - y2[0];
        }
        m000 = c0[0][0];
        m100 = c1[0][0];
        m010 = c0[0][1];
        m001 = c0[1][0];
    } else {
        m002 = ((P[0] + P[1] + P[2]) + (P[3] + P[4] + P[5])) + (P[6] + P[7] + P[8]);
        R s[3], d[3], p[3];
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            p[y] = S[3 * y] + S[3 * y + 2];
            d[y] = S[3 * y + 2] - S[3 * y];
            s[y] = p[y] + S[3 * y + 1];
        }
        m020 = s[0] + s[2];
        m000 = m020 + s[1];
        m200 = (p[0] + p[2]) + p[1];
        m100 = (d[0] + d[2]) + d[1];
        m010 = (E[0] + E[2]) + E[1];
        m110 = E[2] - E[0];
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            s[y] = (D[3 * y] + D[3 * y + 2]) + D[3 * y + 1];
            d[y] = D[3 * y + 2] - D[3 * y];
        }
        m001 = (s[0] + s[2]) + s[1];
        m011 = s[2] - s[0];
        m101 = (d[0] + d[2]) + d[1];
    }
    const R drho = m000, rho = R(1) + drho;
    const bool ok = (rho > R(0)) && (rho < R(1e30));
    const R inv = recip_rho(rho);
    // minus the velocity (each of the transforms below subtracts)
    const R ninv = -inv;
    const R nx = (XF ? fmaR(R(0.5), Fx, m100) : m100) * ninv, ny = m010 * ninv, nz = m001 * ninv;
    const R k100 = fmaR(nx, rho, m100);  // residual j - rho u (with force: -Fx / 2 and the residual)
    // central moments of order 2 (deviations from cs^2 on the diagonal)
    R d200, d020, d002, d110, d101, d011;
    if constexpr (XF) {
#pragma unroll
        for (int p = 0; p < 3; ++p) {  // y shifts; the rest moments r1(p) enter for m = 0
            const R U = r1(p) == 0.0 ? c0[p][0] : R(r1(p)) + c0[p][0];
            const R b0 = fmaR(ny, U, c0[p][1]), b1 = fmaR(ny, c1[p][0], c1[p][1]);
            c0[p][2] = fmaR(ny, c0[p][1] + b0, c0[p][2]);
            c1[p][2] = fmaR(ny, c1[p][1] + b1, c1[p][2]);
            c0[p][1] = b0;
            c1[p][1] = b1;
        }
#pragma unroll
        for (int n = 0; n < 3; ++n) {  // z shifts
            const R U = r1(n) == 0.0 ? c0[0][n] : R(r1(n)) + c0[0][n];
            const R b0 = fmaR(nz, U, c0[1][n]), b1 = fmaR(nz, c1[0][n], c1[1][n]);
            c0[2][n] = fmaR(nz, c0[1][n] + b0, c0[2][n]);
            c1[2][n] = fmaR(nz, c1[1][n] + b1, c1[2][n]);
            c0[1][n] = b0;
            c1[1][n] = b1;
        }
#pragma unroll
        for (int p = 0; p < 3; ++p)  // x shifts of (1, n, p)
#pragma unroll
            for (int n = 0; n < 3; ++n)
                if (n + p > 0)
                    c1[p][n] = fmaR(nx, r1(n) * r1(p) == 0.0 ? c0[p][n] : R(r1(n) * r1(p)) + c0[p][n], c1[p][n]);
        d200 = fmaR(nx, m100 + k100, m200);
        d020 = c0[0][2];
        d002 = c0[2][0];
        d110 = c1[0][1];
        d101 = c1[1][0];
        d011 = c0[1][1];
    } else {
        d200 = fmaR(nx, m100, m200);
        d020 = fmaR(ny, m010, m020);
        d002 = fmaR(nz, m001, m002);
        d110 = fmaR(nx, m010, m110);
        d101 = fmaR(nx, m001, m101);
        d011 = fmaR(ny, m001, m011);
    }

    Shear<R> k = sh;
    if constexpr (learned_mode(MODE)) {
        const R third = R(1.0 / 3.0);
        R in[9];
        in[0] = d200 - third * drho;  // kappa_200 - cs^2 rho
        in[1] = d020 - third * drho;
        in[2] = d002 - third * drho;
        in[3] = d110;
        in[4] = d101;
        in[5] = d011;
        in[6] = -nx;
        in[7] = -ny;
        in[8] = -nz;
        // the correction only lowers the rates, to 0.02 at least (see collide_cell)
        const R dw = fminR(closure_delta_omega<R>(reinterpret_cast<const uint32_t*>(closure), in), R(0)), hi = R(0.98);
        k.k4 = R(0.25) * fminR(sh.k4 - dw, hi);
        k.k5 = R(0.25) * fminR(sh.k5 - dw, hi);
        k.k6 = R(0.25) * fminR(sh.k6 - dw, hi);
        k.k8 = R(1.0 / 6.0) * fminR(sh.k8 - dw, hi);
        k.k9 = R(1.0 / 6.0) * fminR(sh.k9 - dw, hi);
    }
    if constexpr (smag_mode(MODE)) {
        const R ke = R(1) - recipR(smagorinsky_tau(d200, d020, d002, d110, d101, d011, drho, inv, c2, recipR(rt.om[4])));
        k.k4 = k.k5 = k.k6 = R(0.25) * ke;
        k.k8 = k.k9 = R(1.0 / 6.0) * ke;
    }

    // order 2: a, b, c = kappa~_200, 020, 002 (deviations) / 2; o1, o2, o3 = kappa~_110, 101, 011 / 4;
    // t = their trace / 6
    const R o1 = k.k4 * d110, o2 = k.k5 * d101, o3 = k.k6 * d011;
    const R t = fmaR(rt.unit[5], drho, rt.unit[6] * ((d200 + d020) + d002));
    const R t1 = k.k8 * (d200 - d020), t2 = k.k9 * (d200 - d002);
    const R a = (t + t1) + t2, b = fmaR(R(-2), t1, t) + t2, c = fmaR(R(-2), t2, t) + t1;
    FPC_D(0, 0, 0) = drho;
    FPC_D(2, 0, 0) = a;
    FPC_D(0, 2, 0) = b;
    FPC_D(0, 0, 2) = c;
    FPC_D(1, 1, 0) = o1;
    FPC_D(1, 0, 1) = o2;
    FPC_D(0, 1, 1) = o3;
    // XF: half the sources of order 3, and the factors of the higher ones (f4 = (F_x / rho) / 4, ...)
    R f4 = R(0), f8 = R(0), f16 = R(0), k111d = R(0);
    if constexpr (XF) {
        f8 = (R(0.125) * Fx) * inv;
        f4 = f8 + f8;
        f16 = R(0.5) * f8;
        FPC_D(1, 2, 0) = f8 * (R(1.0 / 3.0) + d020);  // / 4
        FPC_D(1, 0, 2) = f8 * (R(1.0 / 3.0) + d002);
        FPC_D(2, 1, 0) = f4 * d110;
        FPC_D(2, 0, 1) = f4 * d101;
        k111d = f8 * d011;
        FPC_D(1, 1, 1) = R(0.5) * k111d;  // / 8
    }
    // orders 4 and 6: the attractors, kappa~_220 / 4, kappa~_211 / 8, kappa~_222 / 8, and half the
    // sources; order 5 / 8 with force
    if constexpr (eq_mode(MODE)) {
        FPC_D(2, 2, 0) = FPC_D(2, 0, 2) = FPC_D(0, 2, 2) = R(1.0 / 36.0) * drho;
        FPC_D(2, 1, 1) = FPC_D(1, 2, 1) = FPC_D(1, 1, 2) = R(0);
        FPC_D(2, 2, 2) = R(1.0 / 216.0) * drho;
        if constexpr (XF) {
            FPC_D(2, 2, 0) = fmaR(f4, c1[0][2], FPC_D(2, 2, 0));
            FPC_D(2, 0, 2) = fmaR(f4, c1[2][0], FPC_D(2, 0, 2));
            FPC_D(2, 1, 1) = f8 * c1[1][1];
            FPC_D(1, 2, 1) = f16 * c0[1][2];
            FPC_D(1, 1, 2) = f16 * c0[2][1];
            FPC_D(1, 2, 2) = f16 * (R(1.0 / 9.0) + c0[2][2]);
            FPC_D(2, 1, 2) = f8 * c1[2][1];
            FPC_D(2, 2, 1) = f8 * c1[1][2];
            FPC_D(2, 2, 2) = fmaR(f8, c1[2][2], FPC_D(2, 2, 2));
        }
    } else {
        const R sixth = R(1.0 / 6.0), nd = R(-1.0 / 36.0) * drho, hinv = R(0.5) * inv;
        const R ka = sixth + a, kb = sixth + b, kc = sixth + c;  // full kappa~_200 / 2
        const R ea = fmaR(sixth, a, nd), eb = fmaR(sixth, b, nd);
        const R p1 = R(8) * o1, p2 = R(8) * o2, p3 = R(8) * o3;
        R x220 = fmaR(p1, o1, fmaR(b, ka, ea)), x202 = fmaR(p2, o2, fmaR(c, ka, ea));
        const R x022 = fmaR(p3, o3, fmaR(c, kb, eb)) * inv;
        R x211 = fmaR(ka + ka, o3, p1 * o2), x121 = fmaR(kb + kb, o2, p1 * o3), x112 = fmaR(kc + kc, o1, p2 * o3);
        if constexpr (XF) {
            x220 = fmaR(x220, inv, f4 * c1[0][2]);
            x202 = fmaR(x202, inv, f4 * c1[2][0]);
            x211 = fmaR(x211, hinv, f8 * c1[1][1]);
            x121 = fmaR(x121, hinv, f16 * c0[1][2]);
            x112 = fmaR(x112, hinv, f16 * c0[2][1]);
            const R k120 = FPC_D(1, 2, 0), k102 = FPC_D(1, 0, 2), k210 = FPC_D(2, 1, 0), k201 = FPC_D(2, 0, 1);
            const R w = R(0.4) * inv;
            FPC_D(1, 2, 2) = fmaR(w, fmaR(kb, k102, fmaR(kc, k120, p3 * k111d)), f16 * (R(1.0 / 9.0) + c0[2][2]));
            FPC_D(2, 1, 2) = fmaR(w, fmaR(kc, k210, fmaR(p2, k111d, R(0.5) * fmaR(p1, k102, p3 * k201))), f8 * c1[2][1]);
            FPC_D(2, 2, 1) = fmaR(w, fmaR(kb, k201, fmaR(p1, k111d, R(0.5) * fmaR(p3, k210, p2 * k120))), f8 * c1[1][2]);
        } else {
            x220 = x220 * inv;
            x202 = x202 * inv;
            x211 = x211 * hinv;
            x121 = x121 * hinv;
            x112 = x112 * hinv;
        }
        R s = fmaR(R(0.5), nd, R(1.0 / 12.0) * t);
        s = fmaR(ka, x022, fmaR(kb, x202, fmaR(kc, x220, s)));
        s = fmaR(R(2), fmaR(p1, x112, fmaR(p2, x121, p3 * x211)), s);
        FPC_D(2, 2, 0) = x220;
        FPC_D(2, 0, 2) = x202;
        FPC_D(0, 2, 2) = x022;
        FPC_D(2, 1, 1) = x211;
        FPC_D(1, 2, 1) = x121;
        FPC_D(1, 1, 2) = x112;
        const R tinv = R(1.0 / 3.0) * inv;
        if constexpr (XF) FPC_D(2, 2, 2) = fmaR(s, tinv, f8 * c1[2][2]);
        else FPC_D(2, 2, 2) = s * tinv;
    }

    // back: plane by plane in p, x lines (without force, moments of total order
    // 3 and 5 are zero; 012 and 021 always) then y lines; the
    // first-order moments, halved like the others, are the residuals described above
    const R zero = R(0);
    {
        const R hx = R(-0.5) * nx, qx = R(-0.25) * nx, tx = R(-2) * nx, h2x = qx * tx;
        const R hy = R(-0.5) * ny, qy = R(-0.25) * ny, ty = R(-2) * ny;
#define FPC_INVX(n, p, Z0, Z1, Z2)                                                                               \
    inv3h<R, r1(n) * r1(p) == 0.0, Z0, Z1, Z2>(g[3 * (n) + 9 * (p)], g[1 + 3 * (n) + 9 * (p)],                    \
                                               g[2 + 3 * (n) + 9 * (p)], hx, qx, tx, h2x,                        \
                                               R(r1(n) * r1(p) * ((n) ? 0.5 : 1.0) * ((p) ? 0.5 : 1.0)))
        FPC_D(1, 0, 0) = R(0.5) * (XF ? k100 + Fx : k100);
        FPC_INVX(0, 0, false, false, false);
        FPC_INVX(2, 0, false, !XF, false);
        {
            R r[3];
#pragma unroll
            for (int x = 0; x < 3; ++x) r[x] = fmaR(ny, R(w1(x)) + g[x], E[x]);
            FPC_D(0, 1, 0) = R(0.5) * ((r[0] + r[2]) + r[1]);
        }
        FPC_INVX(1, 0, false, false, !XF);
#pragma unroll
        for (int x = 0; x < 3; ++x) inv3h<R, false>(g[x], g[x + 3], g[x + 6], hy, qy, ty, zero, R(w1(x)));
        {
            R r[9];
#pragma unroll
            for (int l = 0; l < 9; ++l) r[l] = fmaR(nz, R(w1(l % 3) * w1(l / 3)) + g[l], D[l]);
            FPC_D(0, 0, 1) = R(0.5) * (((r[0] + r[2]) + (r[6] + r[8])) + ((r[1] + r[7]) + (r[3] + r[5])) + r[4]);
        }
        FPC_INVX(0, 1, false, false, !XF);
        FPC_INVX(1, 1, false, !XF, false);
        FPC_INVX(2, 1, true, false, !XF);
#pragma unroll
        for (int x = 0; x < 3; ++x) inv3h<R, true>(g[x + 9], g[x + 12], g[x + 15], hy, qy, ty, zero, zero);
        FPC_INVX(0, 2, false, !XF, false);
        FPC_INVX(1, 2, true, false, !XF);
        FPC_INVX(2, 2, false, !XF, false);
#pragma unroll
        for (int x = 0; x < 3; ++x)
            inv3h<R, false>(g[x + 18], g[x + 21], g[x + 24], hy, qy, ty, zero, R(w1(x) * (0.5 / 3.0)));
#undef FPC_INVX
    }
    {
        const R h = R(-0.5) * nz, q = R(-0.25) * nz, tu = R(-2) * nz;
#pragma unroll
        for (int l = 0; l < 9; ++l)
            inv3h<R, false>(g[l], g[l + 9], g[l + 18], h, q, tu, zero, R(w1(l % 3) * w1(l / 3)));
    }
    return ok;
}

// Any rates, any force: the central-moment transform of all 27 moments.  NEWTON: the short reciprocal
// (pair.cuh).
template <typename R, int FORCE, int MODE, bool NEWTON>
__device__ __forceinline__ bool collide_general(R (&g)[27], const Rates<R>& rt, R Fx, R Fy, R Fz, const Shear<R>& sh,
                                                const float* closure, R c2)
{
    constexpr bool R1 = r1_mode(MODE);
    R k4 = sh.k4, k5 = sh.k5, k6 = sh.k6, k8 = sh.k8, k9 = sh.k9;
    // ---- Step 7 and the first pass (z lines), sharing the line sums ----
    R S[9], Dz[9], Pz[9];
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const R lo = g[l], mid = g[l + 9], hi = g[l + 18];
        Pz[l] = lo + hi;
        Dz[l] = hi - lo;
        S[l] = Pz[l] + mid;
    }
    const R drho = ((S[0] + S[1] + S[2]) + (S[3] + S[4] + S[5])) + (S[6] + S[7] + S[8]);
    const R jx = ((S[2] - S[0]) + (S[5] - S[3])) + (S[8] - S[6]);
    const R jy = ((S[6] - S[0]) + (S[7] - S[1])) + (S[8] - S[2]);
    const R jz = ((Dz[0] + Dz[1] + Dz[2]) + (Dz[3] + Dz[4] + Dz[5])) + (Dz[6] + Dz[7] + Dz[8]);
    const R rho = R(1) + drho;
    // (the same bits either way; the Smagorinsky mode is 1 to 2.5 % faster with CUDA's from 100^3 fp32 cells on)
    R inv_rho;
    if constexpr (smag_mode(MODE)) inv_rho = recipR(rho);
    else inv_rho = recip_rho<NEWTON>(rho);
    const bool ok = (rho > R(0)) && (rho < R(1e30));
    R ux, uy, uz;
    if (FORCE) {
        ux = fmaR(R(0.5), Fx, jx) * inv_rho;
        uy = fmaR(R(0.5), Fy, jy) * inv_rho;
        uz = fmaR(R(0.5), Fz, jz) * inv_rho;
    } else {
        ux = jx * inv_rho;
        uy = jy * inv_rho;
        uz = jz * inv_rho;
    }
    const R ux2 = ux * ux, uy2 = uy * uy, uz2 = uz * uz;
    const R tux = R(2) * ux, tuy = R(2) * uy, tuz = R(2) * uz;

#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const double Kd = w1(l % 3) * w1(l / 3);
        const R U = R(Kd) + S[l];
        g[l] = S[l];
        g[l + 9] = fmaR(-uz, U, Dz[l]);
        g[l + 18] = fmaR(uz2, U, fmaR(-tuz, Dz[l], Pz[l]));
    }
    FPC_PASS_B(fwd3)
    FPC_PASS_C(fwd3)
    // now g[m + 3n + 9p] = kappa_mnp - r_m r_n r_p

    // ---- Step 3: relaxation toward the Markovian attractors ----
    const R third = R(1.0 / 3.0), ninth = R(1.0 / 9.0);
    R fx = R(0), fy = R(0), fz = R(0);
    if (FORCE) {
        fx = Fx * inv_rho;
        fy = Fy * inv_rho;
        fz = Fz * inv_rho;
    }

    // shear rates, possibly corrected by the learned closure
    if constexpr (learned_mode(MODE)) {
        R in[9];
        in[0] = FPC_D(2, 0, 0) - third * drho;  // kappa_200 - cs^2 rho
        in[1] = FPC_D(0, 2, 0) - third * drho;
        in[2] = FPC_D(0, 0, 2) - third * drho;
        in[3] = FPC_D(1, 1, 0);
        in[4] = FPC_D(1, 0, 1);
        in[5] = FPC_D(0, 1, 1);
        in[6] = ux;
        in[7] = uy;
        in[8] = uz;
        // the correction adds an eddy viscosity nu_t >= 0 (the training label's definition), so it
        // only lowers the rates: omega + min(delta omega, 0), kept above 0.02
        const R dw = fminR(closure_delta_omega<R>(reinterpret_cast<const uint32_t*>(closure), in), R(0));
        const R hi = R(0.98);
        k4 = fminR(k4 - dw, hi);
        k5 = fminR(k5 - dw, hi);
        k6 = fminR(k6 - dw, hi);
        k8 = fminR(k8 - dw, hi);
        k9 = fminR(k9 - dw, hi);
    }

    if constexpr (MODE == MODE_SMAG) {
        const R te = smagorinsky_tau(FPC_D(2, 0, 0), FPC_D(0, 2, 0), FPC_D(0, 0, 2), FPC_D(1, 1, 0), FPC_D(1, 0, 1),
                                     FPC_D(0, 1, 1), drho, inv_rho, c2, R(1) / rt.om[4]);
        k4 = k5 = k6 = k8 = k9 = R(1) - R(1) / te;
    }

    // order 1 (attractor 0, source F).  In exact arithmetic kappa_100 = -F_x/2 and
    // kappa~_100 = F_x/2 whatever omega_1..3 are, so they are applied here as 0:
    // kappa~_100 = kappa_100 + F_x keeps the rounding residual j - rho u of the forward
    // transform, and the back transform then rebuilds the momentum j + F to the last
    // bit instead of rho * round(j / rho) (whose error repeats every step in a slowly
    // varying flow and would accumulate linearly in fp32).
    if (FORCE) {
        FPC_D(1, 0, 0) += Fx;
        FPC_D(0, 1, 0) += Fy;
        FPC_D(0, 0, 1) += Fz;
    }

    // sources of order 3 from the pre-collision second moments
    R s120 = 0, s102 = 0, s210 = 0, s012 = 0, s201 = 0, s021 = 0, s111 = 0;
    if (FORCE) {
        const R k200 = third + FPC_D(2, 0, 0), k020 = third + FPC_D(0, 2, 0), k002 = third + FPC_D(0, 0, 2);
        const R k110 = FPC_D(1, 1, 0), k101 = FPC_D(1, 0, 1), k011 = FPC_D(0, 1, 1);
        s120 = fx * k020 + R(2) * fy * k110;
        s102 = fx * k002 + R(2) * fz * k101;
        s210 = R(2) * fx * k110 + fy * k200;
        s012 = fy * k002 + R(2) * fz * k011;
        s201 = R(2) * fx * k101 + fz * k200;
        s021 = R(2) * fy * k011 + fz * k020;
        s111 = fx * k011 + fy * k101 + fz * k110;
    }

    // order 2: off-diagonal (attractor 0, no source), 2s1 (attractor 3 cs^2 rho),
    // 2d1, 2d2 (attractor 0)
    FPC_D(1, 1, 0) = k4 * FPC_D(1, 1, 0);
    FPC_D(1, 0, 1) = k5 * FPC_D(1, 0, 1);
    FPC_D(0, 1, 1) = k6 * FPC_D(0, 1, 1);
    {
        const R d200 = FPC_D(2, 0, 0), d020 = FPC_D(0, 2, 0), d002 = FPC_D(0, 0, 2);
        const R y2s = (d200 + d020) + d002;
        const R y2d1 = d200 - d020, y2d2 = d200 - d002;
        const R t2s = fmaR(rt.om[7], drho, rt.keep[7] * y2s);  // attractor deviation: drho
        const R t2d1 = k8 * y2d1;
        const R t2d2 = k9 * y2d2;
        FPC_D(2, 0, 0) = third * ((t2s + t2d1) + t2d2);
        FPC_D(0, 2, 0) = third * (fmaR(R(-2), t2d1, t2s) + t2d2);
        FPC_D(0, 0, 2) = third * (fmaR(R(-2), t2d2, t2s) + t2d1);
    }

    // sources of order 4 from the pre-collision third moments
    R s220 = 0, s202 = 0, s022 = 0, s211 = 0, s121 = 0, s112 = 0;
    if (FORCE) {
        s220 = R(2) * (fx * FPC_D(1, 2, 0) + fy * FPC_D(2, 1, 0));
        s202 = R(2) * (fx * FPC_D(1, 0, 2) + fz * FPC_D(2, 0, 1));
        s022 = R(2) * (fy * FPC_D(0, 1, 2) + fz * FPC_D(0, 2, 1));
        s211 = R(2) * fx * FPC_D(1, 1, 1) + fy * FPC_D(2, 0, 1) + fz * FPC_D(2, 1, 0);
        s121 = fx * FPC_D(0, 2, 1) + R(2) * fy * FPC_D(1, 1, 1) + fz * FPC_D(1, 2, 0);
        s112 = fx * FPC_D(0, 1, 2) + fy * FPC_D(1, 0, 2) + R(2) * fz * FPC_D(1, 1, 1);
    }

    // order 3 (attractors 0): pairs (120,102), (210,012), (201,021), and 111
    if constexpr (R1) {  // half the sources
        FPC_D(1, 2, 0) = R(0.5) * s120;
        FPC_D(1, 0, 2) = R(0.5) * s102;
        FPC_D(2, 1, 0) = R(0.5) * s210;
        FPC_D(0, 1, 2) = R(0.5) * s012;
        FPC_D(2, 0, 1) = R(0.5) * s201;
        FPC_D(0, 2, 1) = R(0.5) * s021;
        FPC_D(1, 1, 1) = R(0.5) * s111;
    } else {
#define FPC_PAIR3(A, B, sa, sb, j)                                                      \
    {                                                                                   \
        const R ys = A + B, ym = A - B;                                                 \
        R ts = rt.keep[j] * ys, tm = rt.keep[j + 1] * ym;                               \
        if (FORCE) {                                                                    \
            ts = fmaR(rt.src[j], sa + sb, ts);                                          \
            tm = fmaR(rt.src[j + 1], sa - sb, tm);                                      \
        }                                                                               \
        A = R(0.5) * (ts + tm);                                                         \
        B = R(0.5) * (ts - tm);                                                         \
    }
    FPC_PAIR3(FPC_D(1, 2, 0), FPC_D(1, 0, 2), s120, s102, 10)
    FPC_PAIR3(FPC_D(2, 1, 0), FPC_D(0, 1, 2), s210, s012, 12)
    FPC_PAIR3(FPC_D(2, 0, 1), FPC_D(0, 2, 1), s201, s021, 14)
#undef FPC_PAIR3
    FPC_D(1, 1, 1) = rt.keep[16] * FPC_D(1, 1, 1);
    if (FORCE) FPC_D(1, 1, 1) = fmaR(rt.src[16], s111, FPC_D(1, 1, 1));
    }

    // sources of order 5 from the pre-collision fourth moments
    R s122 = 0, s212 = 0, s221 = 0;
    if (FORCE) {
        const R k022 = ninth + FPC_D(0, 2, 2), k202 = ninth + FPC_D(2, 0, 2), k220 = ninth + FPC_D(2, 2, 0);
        s122 = fx * k022 + R(2) * (fy * FPC_D(1, 1, 2) + fz * FPC_D(1, 2, 1));
        s212 = fy * k202 + R(2) * (fx * FPC_D(1, 1, 2) + fz * FPC_D(2, 1, 1));
        s221 = fz * k220 + R(2) * (fx * FPC_D(1, 2, 1) + fy * FPC_D(2, 1, 1));
    }

    // post-collision second moments used by the attractors of orders 4-6
    const R pa = FPC_D(2, 0, 0), pb = FPC_D(0, 2, 0), pc = FPC_D(0, 0, 2);
    const R o110 = FPC_D(1, 1, 0), o101 = FPC_D(1, 0, 1), o011 = FPC_D(0, 1, 1);

    // order 4: groups 4s1, 4d1, 4d2 and 211, 121, 112
    {
        R A220, A202, A022, A211, A121, A112;
        if constexpr (eq_mode(MODE)) {
            A220 = A202 = A022 = ninth * drho;  // cs^4 rho - 1/9
            A211 = A121 = A112 = R(0);
        } else {
            const R dn = ninth * drho;
            A220 = (fmaR(third, pa + pb, fmaR(pa, pb, R(2) * o110 * o110)) - dn) * inv_rho;
            A202 = (fmaR(third, pa + pc, fmaR(pa, pc, R(2) * o101 * o101)) - dn) * inv_rho;
            A022 = (fmaR(third, pb + pc, fmaR(pb, pc, R(2) * o011 * o011)) - dn) * inv_rho;
            A211 = fmaR(third + pa, o011, R(2) * o110 * o101) * inv_rho;
            A121 = fmaR(third + pb, o101, R(2) * o110 * o011) * inv_rho;
            A112 = fmaR(third + pc, o110, R(2) * o011 * o101) * inv_rho;
        }
        if constexpr (R1) {
            FPC_D(2, 2, 0) = fmaR(R(0.5), s220, A220);
            FPC_D(2, 0, 2) = fmaR(R(0.5), s202, A202);
            FPC_D(0, 2, 2) = fmaR(R(0.5), s022, A022);
            FPC_D(2, 1, 1) = fmaR(R(0.5), s211, A211);
            FPC_D(1, 2, 1) = fmaR(R(0.5), s121, A121);
            FPC_D(1, 1, 2) = fmaR(R(0.5), s112, A112);
        } else {
        const R d220 = FPC_D(2, 2, 0), d202 = FPC_D(2, 0, 2), d022 = FPC_D(0, 2, 2);
        const R y4s = (d220 + d202) + d022, y4d1 = (d220 + d202) - d022, y4d2 = d220 - d202;
        const R a4s = (A220 + A202) + A022, a4d1 = (A220 + A202) - A022, a4d2 = A220 - A202;
        R t4s = fmaR(rt.om[17], a4s, rt.keep[17] * y4s);
        R t4d1 = fmaR(rt.om[18], a4d1, rt.keep[18] * y4d1);
        R t4d2 = fmaR(rt.om[19], a4d2, rt.keep[19] * y4d2);
        if (FORCE) {
            t4s = fmaR(rt.src[17], (s220 + s202) + s022, t4s);
            t4d1 = fmaR(rt.src[18], (s220 + s202) - s022, t4d1);
            t4d2 = fmaR(rt.src[19], s220 - s202, t4d2);
        }
        FPC_D(2, 2, 0) = R(0.25) * fmaR(R(2), t4d2, t4s + t4d1);
        FPC_D(2, 0, 2) = R(0.25) * fmaR(R(-2), t4d2, t4s + t4d1);
        FPC_D(0, 2, 2) = R(0.5) * (t4s - t4d1);
        R t211 = fmaR(rt.om[20], A211, rt.keep[20] * FPC_D(2, 1, 1));
        R t121 = fmaR(rt.om[21], A121, rt.keep[21] * FPC_D(1, 2, 1));
        R t112 = fmaR(rt.om[22], A112, rt.keep[22] * FPC_D(1, 1, 2));
        if (FORCE) {
            t211 = fmaR(rt.src[20], s211, t211);
            t121 = fmaR(rt.src[21], s121, t121);
            t112 = fmaR(rt.src[22], s112, t112);
        }
        FPC_D(2, 1, 1) = t211;
        FPC_D(1, 2, 1) = t121;
        FPC_D(1, 1, 2) = t112;
        }
    }

    // source of order 6 from the pre-collision fifth moments
    R s222 = 0;
    if (FORCE) s222 = R(2) * ((fx * FPC_D(1, 2, 2) + fy * FPC_D(2, 1, 2)) + fz * FPC_D(2, 2, 1));

    // order 5: attractors from post-collision second and third moments
    {
        R A122 = R(0), A212 = R(0), A221 = R(0);
        if constexpr (!eq_mode(MODE)) {
            const R K200 = third + pa, K020 = third + pb, K002 = third + pc;
            const R k111 = FPC_D(1, 1, 1);
            const R c = R(0.4) * inv_rho;
            A122 = c * (fmaR(K020, FPC_D(1, 0, 2), K002 * FPC_D(1, 2, 0)) +
                        fmaR(R(4) * o011, k111, R(2) * fmaR(o101, FPC_D(0, 2, 1), o110 * FPC_D(0, 1, 2))));
            A212 = c * (fmaR(K200, FPC_D(0, 1, 2), K002 * FPC_D(2, 1, 0)) +
                        fmaR(R(4) * o101, k111, R(2) * fmaR(o110, FPC_D(1, 0, 2), o011 * FPC_D(2, 0, 1))));
            A221 = c * (fmaR(K200, FPC_D(0, 2, 1), K020 * FPC_D(2, 0, 1)) +
                        fmaR(R(4) * o110, k111, R(2) * fmaR(o011, FPC_D(2, 1, 0), o101 * FPC_D(1, 2, 0))));
        }
        if constexpr (R1) {
            FPC_D(1, 2, 2) = fmaR(R(0.5), s122, A122);
            FPC_D(2, 1, 2) = fmaR(R(0.5), s212, A212);
            FPC_D(2, 2, 1) = fmaR(R(0.5), s221, A221);
        } else {
            R t122 = fmaR(rt.om[23], A122, rt.keep[23] * FPC_D(1, 2, 2));
            R t212 = fmaR(rt.om[24], A212, rt.keep[24] * FPC_D(2, 1, 2));
            R t221 = fmaR(rt.om[25], A221, rt.keep[25] * FPC_D(2, 2, 1));
            if (FORCE) {
                t122 = fmaR(rt.src[23], s122, t122);
                t212 = fmaR(rt.src[24], s212, t212);
                t221 = fmaR(rt.src[25], s221, t221);
            }
            FPC_D(1, 2, 2) = t122;
            FPC_D(2, 1, 2) = t212;
            FPC_D(2, 2, 1) = t221;
        }
    }

    // order 6: attractor from post-collision second and fourth moments
    {
        R A222;
        if constexpr (eq_mode(MODE)) {
            A222 = R(1.0 / 27.0) * drho;  // cs^6 rho - 1/27
        } else {
            const R q220 = FPC_D(2, 2, 0), q202 = FPC_D(2, 0, 2), q022 = FPC_D(0, 2, 2);
            R t = fmaR(ninth, (pa + pb) + pc, third * ((q022 + q202) + q220));
            t = fmaR(pa, q022, fmaR(pb, q202, fmaR(pc, q220, t)));
            t = fmaR(R(4), fmaR(o110, FPC_D(1, 1, 2), fmaR(o101, FPC_D(1, 2, 1), o011 * FPC_D(2, 1, 1))), t);
            A222 = (t - ninth * drho) * (third * inv_rho);
        }
        if constexpr (R1) {
            FPC_D(2, 2, 2) = fmaR(R(0.5), s222, A222);
        } else {
            R t222 = fmaR(rt.om[26], A222, rt.keep[26] * FPC_D(2, 2, 2));
            if (FORCE) t222 = fmaR(rt.src[26], s222, t222);
            FPC_D(2, 2, 2) = t222;
        }
    }

    // ---- Steps 4+5: back to populations (passes in reverse order) ----
    FPC_PASS_C(inv3)
    FPC_PASS_B(inv3)
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const double Kd = w1(l % 3) * w1(l / 3);
        inv3<R, false>(g[l], g[l + 9], g[l + 18], uz, uz2, tuz, R(Kd));
    }
    return ok;
}

// Collide one cell in place.  rt: rates of Step 3; Fx, Fy, Fz: body force;
// sh: 1 minus the five shear rates (110, 101, 011, 2d1, 2d2; own_shear, or
// an ensemble box's); closure: MLP weights (learned mode only); c2 = (C_s Delta D)^2 of the cell (Smagorinsky modes
// only).  Returns false when rho <= 0 or not finite.
template <typename R, int FORCE, int MODE, bool NEWTON = false>
__device__ __forceinline__ bool collide_cell(R (&g)[27], const Rates<R>& rt, R Fx, R Fy, R Fz, const Shear<R>& sh,
                                             const float* closure, R c2 = R(0))
{
    if constexpr (unit_collision(FORCE, MODE)) return collide_unit<R, FORCE == FORCE_X, MODE>(g, rt, Fx, sh, closure, c2);
    else return collide_general<R, FORCE, MODE, NEWTON>(g, rt, Fx, Fy, Fz, sh, closure, c2);
}

#undef FPC_PASS_B
#undef FPC_PASS_C

}  // namespace fpc

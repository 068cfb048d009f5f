// Device arithmetic of the hydro stage: ideal-gas closure, minmod limiter,
// piecewise-linear face states and the HLLC flux.
//
// Physics: Eq. "conservative form" (S = 0) and Eq. "fluxes" of the HARD paper
// with p = (gamma-1) e; numerics of Sec. 2.2.2 with minmod-limited PLM face
// states and the HLLC solver (Toro, ch. 10) with Davis wave-speed bounds.
//
// The FP64 functions evaluate every formula in one fixed operation order and
// are compiled without FMA contraction, so each + - * / sqrt is one IEEE
// operation.  The FP32 functions trade that for fewer instructions
// (reciprocals, the one-sided branch-free HLLC form).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "vec2.cuh"

namespace hh {

constexpr int NF = 5;

// Rotated-frame component order per physical axis: (normal, tangent 1,
// tangent 2) as indices into the momentum / velocity slots 1..3.
template <int AX> struct Rot;
template <> struct Rot<0> { static constexpr int n = 1, t1 = 2, t2 = 3; };
template <> struct Rot<1> { static constexpr int n = 2, t1 = 1, t2 = 3; };
template <> struct Rot<2> { static constexpr int n = 3, t1 = 1, t2 = 2; };

// --------------------------------------------------- FP64 without its pipe --
// GB300 issues one FP64 warp instruction per SM every 16 clocks and 64 others
// in that time, so an FP64 kernel costs what it sends down that pipe.  The
// helpers below return the bits of the plain expressions, up to the sign of a zero
// (the short quotient of -0 is +0, minmod passes on a -0 of its arguments; no sum
// or difference of the schemes tells the two apart), with fewer of those
// instructions: comparisons on the integer pipe, and quotients by a divisor that
// serves several of them as q = RN(a y), q + (a - b q) y with y = RN(1/b) (three
// operations instead of an IEEE division's seven or eight).  One product and two
// fused operations with the correctly rounded reciprocal give the correctly rounded
// quotient as long as nothing under- or overflows (Brisebarre, Muller and Raina, IEEE
// Trans. Computers 53, 2004, after Markstein, IBM J. Res. Dev. 34, 1990); operands
// outside 2^-500 .. 2^500 take the division.  Measured, with the results
// bit-identical: two steps of a 128^3 mesh 20.0 -> 14.3 ms (984 -> ~690
// FP64 warp instructions per 32 cells and stage), 100 steps of a 400-cell 1D
// mesh 6.98 -> 4.73 ms.
__device__ __forceinline__ long long bits64(double x) { return __double_as_longlong(x); }
constexpr long long ABS64 = 0x7fffffffffffffffll, INF64 = 0x7ff0000000000000ll;

// x >= 0 (true for -0, false for NaN)
__device__ __forceinline__ bool nonneg(double x) {
    const long long b = bits64(x);
    return (b >= 0 && b <= INF64) || b == ~ABS64;
}
__device__ __forceinline__ bool mid_exponent(double x) {
    return (unsigned)((__double2hiint(x) >> 20) & 0x7ff) - 523u <= 1000u;
}
// a / b given y = RN(1/b); ok: b's exponent allows the short form
__device__ __forceinline__ double div_by(double a, double b, double y, bool ok) {
    if (ok && (mid_exponent(a) || (bits64(a) & ABS64) == 0)) {
        const double q = a * y;
        return fma(fma(-b, q, a), y, q);
    }
    return a / b;
}

// A cell width as the kernels divide by it: FP64 the width and RN(1 / width)
// (0 where the short division must not be used), `exact` for a power of two;
// FP32 1 / width.
struct Width64 {
    double w, inv;
    int exact;
};
template <typename T> struct WidthOf { using type = float; };
template <> struct WidthOf<double> { using type = Width64; };
template <typename T> using width_t = typename WidthOf<T>::type;

template <typename T> inline __host__ __device__ width_t<T> make_width(double dx);
template <> inline __host__ __device__ float make_width<float>(double dx) { return (float)(1.0 / dx); }
template <> inline __host__ __device__ Width64 make_width<double>(double dx) {
    const bool mid = dx > 1e-150 && dx < 1e150;
    int e;
    return Width64{dx, mid ? 1.0 / dx : 0.0, mid && frexp(dx, &e) == 0.5};
}

// ---------------------------------------------------------------- minmod --
// Zero unless both slopes have the same strict sign; otherwise the smaller
// magnitude (a on a tie).  A sign test, so tiny slopes never underflow.  FP64
// compares the magnitudes as integers (ordered like the values; a NaN's lies
// above infinity's).
__device__ __forceinline__ double minmod(double a, double b) {
    const long long ba = bits64(a), bb = bits64(b);
    const long long ma = ba & ABS64, mb = bb & ABS64;
    const bool same = (ba ^ bb) >= 0 && ma <= INF64 && mb <= INF64;
    return same ? (ma <= mb ? a : b) : 0.0;
}
__device__ __forceinline__ float minmod(float a, float b) { return vminmod(a, b); }

// ------------------------------------------------- fused multiply-adds --
// Both element types are compiled without automatic FMA contraction, so the
// rounding of every expression is fixed by the source and identical in every
// kernel that uses these functions.  FP64 keeps a*b + c as two roundings (the
// oracle's order); FP32 fuses it explicitly.
__device__ __forceinline__ double madd(double a, double b, double c) { return a * b + c; }
__device__ __forceinline__ float madd(float a, float b, float c) { return fmaf(a, b, c); }

// c +- a/2 (the product with 1/2 is exact, so one rounding either way)
__device__ __forceinline__ double add_half(double c, double a) { return fma(0.5, a, c); }
__device__ __forceinline__ float add_half(float c, float a) { return fmaf(0.5f, a, c); }
__device__ __forceinline__ double sub_half(double c, double a) { return fma(-0.5, a, c); }
__device__ __forceinline__ float sub_half(float c, float a) { return fmaf(-0.5f, a, c); }

// acc - diff / dx: FP64 the IEEE quotient, FP32 a multiplication by 1/dx.
__device__ __forceinline__ double sub_over_dx(double acc, double diff, const Width64& dx) {
    return acc - div_by(diff, dx.w, dx.inv, bits64(dx.inv) != 0);
}
__device__ __forceinline__ float sub_over_dx(float acc, float diff, float inv_dx) {
    return fmaf(-diff, inv_dx, acc);
}

// The same on 3D meshes, whose FP64 kernels fill the pipe: a quotient by a power
// of two is the product with its reciprocal, one operation instead of three
// (128^3, two steps: 12.89 -> 12.2 ms).  1D and 2D strips, bound by their
// chains, lose 1-2 % by the test.
__device__ __forceinline__ double sub_over_dx3(double acc, double diff, const Width64& dx) {
    return dx.exact ? acc - diff * dx.inv : sub_over_dx(acc, diff, dx);
}
__device__ __forceinline__ float sub_over_dx3(float acc, float diff, float inv_dx) {
    return sub_over_dx(acc, diff, inv_dx);
}

// ------------------------------------------------------- closure helpers --
// Conserved -> primitive W = (rho, u, v, w, p), p = (gamma-1)(E - rho|v|^2/2).
__device__ __forceinline__ void cons_to_prim(const double U[NF], double gm1, double W[NF]) {
    double rho = U[0];
    const double y = __drcp_rn(rho);
    const bool ok = mid_exponent(rho);
    double u = div_by(U[1], rho, y, ok);
    double v = div_by(U[2], rho, y, ok);
    double w = div_by(U[3], rho, y, ok);
    double kin = 0.5 * rho * (u * u + v * v + w * w);
    W[0] = rho; W[1] = u; W[2] = v; W[3] = w;
    W[4] = gm1 * (U[4] - kin);
}
__device__ __forceinline__ void cons_to_prim(const float U[NF], float gm1, float W[NF]) {
    float rho = U[0];
    float ir = vrcp(rho);
    float u = U[1] * ir, v = U[2] * ir, w = U[3] * ir;
    float kin = 0.5f * fmaf(U[1], u, fmaf(U[2], v, U[3] * w));
    W[0] = rho; W[1] = u; W[2] = v; W[3] = w;
    W[4] = gm1 * (U[4] - kin);
}

// Non-physical test on a primitive state (also catches NaN).
template <typename T>
__device__ __forceinline__ bool nonphys(const T W[NF]) {
    return !(W[0] > T(0)) || !(W[4] > T(0));
}

// ------------------------------------------------------------------ HLLC --
// FP64: the textbook form in one fixed evaluation order (the oracle's), for
// the side that the face takes only: ~125 FP64 instructions a face against
// ~190 with both sides evaluated.  Wn = (rho, un, t1, t2, p) in the frame whose
// normal is component 1; m = rho_K (S_K - u_K).
__device__ __forceinline__ void hllc_normal(const double WL[NF], const double WR[NF],
                                            double gamma, double gm1, double igm1,
                                            double F[NF]) {
    const double rL = WL[0], uL = WL[1], pL = WL[4];
    const double rR = WR[0], uR = WR[1], pR = WR[4];
    const double cL = sqrt(gamma * pL / rL);
    const double cR = sqrt(gamma * pR / rR);
    const double SL = fmin(uL - cL, uR - cR);
    const double SR = fmax(uL + cL, uR + cR);
    const double aL = SL - uL, aR = SR - uR;
    const double qL = rL * uL, qR = rR * uR;
    const double mL = rL * aL, mR = rR * aR;
    const double Sstar = (pR - pL + qL * aL - qR * aR) / (mL - mR);
    const bool supL = nonneg(SL), supR = !supL && nonneg(-SR);
    const bool left = supL || (!supR && nonneg(Sstar));
    const double r = left ? rL : rR, u = left ? uL : uR, p = left ? pL : pR;
    const double t1 = left ? WL[2] : WR[2], t2 = left ? WL[3] : WR[3];
    const double mu = left ? qL : qR, m = left ? mL : mR;
    const double SK = left ? SL : SR;
    const double E = div_by(p, gm1, igm1, mid_exponent(gm1)) + 0.5 * r * (u * u + t1 * t1 + t2 * t2);
    F[0] = mu;
    F[1] = mu * u + p;
    F[2] = mu * t1;
    F[3] = mu * t2;
    F[4] = (E + p) * u;
    if (!supL && !supR) {                               // the star regions
        const double fac = m / (SK - Sstar);
        const double Es = fac * (E / r + (Sstar - u) * (Sstar + p / m));
        F[0] += SK * (fac - r);
        F[1] += SK * (fac * Sstar - mu);
        F[2] += SK * (fac * t1 - r * t1);
        F[3] += SK * (fac * t2 - r * t2);
        F[4] += SK * (Es - E);
    }
}

// FP32: the one-sided form of vec2.cuh (hllc_core), F = F_K + s (U*_K - U_K),
// with s = 0 reproducing the supersonic branches without a branch.
__device__ __forceinline__ void hllc_normal(const float WL[NF], const float WR[NF], float gamma,
                                            float /*gm1*/, float igm1, float F[NF]) {
    hllc_core<float>(WL, WR, gamma, igm1, F);
}

// Face flux through a face whose normal is physical axis AX, from the
// primitives of the four cells i-1, i, i+1, i+2 around the face i+1/2:
//   dq_m = minmod(q_m - q_{m-1}, q_{m+1} - q_m)
//   q_L = q_i + dq_i/2,   q_R = q_{i+1} - dq_{i+1}/2,   F = HLLC(q_L, q_R).
template <int AX, typename T>
__device__ __forceinline__ void hllc_axis(const T qL[NF], const T qR[NF], T gamma, T gm1, T igm1,
                                          T F[NF]) {
    using R = Rot<AX>;
    T WL[NF] = {qL[0], qL[R::n], qL[R::t1], qL[R::t2], qL[4]};
    T WR[NF] = {qR[0], qR[R::n], qR[R::t1], qR[R::t2], qR[4]};
    T Fn[NF];
    hllc_normal(WL, WR, gamma, gm1, igm1, Fn);
    F[0] = Fn[0];
    F[R::n] = Fn[1];
    F[R::t1] = Fn[2];
    F[R::t2] = Fn[3];
    F[4] = Fn[4];
}

template <int AX>
__device__ __forceinline__ void face_flux4(const double q0[NF], const double q1[NF],
                                           const double q2[NF], const double q3[NF], double gamma,
                                           double gm1, double igm1, double F[NF]) {
    double qL[NF], qR[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        double dqi = minmod(q1[f] - q0[f], q2[f] - q1[f]);
        double dqi1 = minmod(q2[f] - q1[f], q3[f] - q2[f]);
        qL[f] = add_half(q1[f], dqi);
        qR[f] = sub_half(q2[f], dqi1);
    }
    hllc_axis<AX>(qL, qR, gamma, gm1, igm1, F);
}
template <int AX>
__device__ __forceinline__ void face_flux4(const float q0[NF], const float q1[NF],
                                           const float q2[NF], const float q3[NF], float gamma,
                                           float gm1, float igm1, float F[NF]) {
    float qL[NF], qR[NF];
    plm_faces<float>(q0, q1, q2, q3, qL, qR);
    hllc_axis<AX>(qL, qR, gamma, gm1, igm1, F);
}

// Signal rate of one cell: sum over the active axes of (|v_d| + c)/dx_d.
// `act` and `dx` are indexed by physical axis; summed in physical order.
__device__ __forceinline__ double cell_rate(const double W[NF], double gamma, const bool act[3],
                                            const Width64 dx[3]) {
    double cs = sqrt(gamma * W[4] / W[0]);
    double r = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d)
        if (act[d]) r += div_by(fabs(W[1 + d]) + cs, dx[d].w, dx[d].inv, bits64(dx[d].inv) != 0);
    return r;
}
__device__ __forceinline__ float cell_rate(const float W[NF], float gamma, const bool act[3],
                                           const float inv_dx[3]) {
    float cs = vsqrt(gamma * W[4] * vrcp(W[0]));
    float r = 0.0f;
    if (act[0]) r = fmaf(fabsf(W[1]) + cs, inv_dx[0], r);
    if (act[1]) r = fmaf(fabsf(W[2]) + cs, inv_dx[1], r);
    if (act[2]) r = fmaf(fabsf(W[3]) + cs, inv_dx[2], r);
    return r;
}

// Order-preserving bits of a non-negative rate (NaN sorts above +inf).
__device__ __forceinline__ unsigned long long rate_bits(double r) {
    return (unsigned long long)__double_as_longlong(r);
}
__device__ __forceinline__ unsigned long long rate_bits(float r) {
    // widen exactly to double so both element types share one slot format
    return (unsigned long long)__double_as_longlong((double)r);
}

}  // namespace hh

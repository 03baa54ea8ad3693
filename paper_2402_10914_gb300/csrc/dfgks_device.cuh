// dfgks_device.cuh -- FP64 device arithmetic of the hybrid DF + WENO-AO finite-volume scheme
// (Zhang, Ji & Xu, arXiv 2402.10914) for sm_103a.  Every routine works on one face line, one
// face side or one Gauss point in that face's local frame (Sect. 2.1); the kernels in
// dfgks_kernels.cu move data between them.
//
// Arithmetic choices (each algebraically identical to the paper's formulas):
//   * characteristic projection and back-projection of differences of states, in factored form (DiffBasis: ten
//     instructions each way);
//   * WENO-AO in undivided differences (ao_weights): smoothness indicators (Eq. 38), weights and evaluations
//     without the sub-stencil polynomials' coefficients;
//   * GKS and L-F fluxes in gradient form: primitive gradients in place of slope coefficients and flux Jacobians;
//   * every FP64 operand in a vector register (Real), Gaussians and erfc from tables;
//   * S2O4 flux coefficients (Eq. 27) combined analytically per kinetic term before the moments
//     are summed, using E(dt) = E(dt/2)^2, which avoids the cancellation of 4(F(dt)-2F(dt/2)).
// The plain statements (project, back_project, weno_ao_t and its evaluations, df_at_*, limiter_alpha) are what the
// kernels' forms and their reverses are tested against; no kernel calls them.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

// every arithmetic routine also compiles for the host, so its derivatives can be checked there
#define DFK_HD __host__ __device__ __forceinline__

namespace dfk {

constexpr int G = 3;                       // ghost layers: the normal stencil spans i-3 .. i+2
constexpr double kGaussEta = 0.28867513459481288225;   // sqrt(3)/6: Gauss points at eta = -/+ this

// Order of doubles on their bit patterns.  Read as signed 64-bit integers, the IEEE encodings of
// +0 .. +inf compare as the values do, and every negative value (-0 included) reads as negative.
// Maxima, minima and tests of quantities that are never negative (WENO ratios and weight sums, DF
// factors, products of positive states) run on the integer units this way, leaving the FP64 units
// (two per SM) to the arithmetic; the results are the same bits as fmax / fmin / < on such values.
DFK_HD long long dbits(double x) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(x);
#else
    long long b;
    memcpy(&b, &x, sizeof b);
    return b;
#endif
}
DFK_HD double dval(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double x;
    memcpy(&x, &b, sizeof x);
    return x;
#endif
}
DFK_HD double nn_max(double a, double b) { const long long x = dbits(a), y = dbits(b); return dval(x > y ? x : y); }
DFK_HD double nn_min(double a, double b) { const long long x = dbits(a), y = dbits(b); return dval(x < y ? x : y); }
// a < b for a >= +0 (b of any sign)
DFK_HD bool nn_less(double a, double b) { return dbits(a) < dbits(b); }
// lo < a < hi for lo, hi > 0: false for a negative, -0 or NaN
DFK_HD bool in_range(double a, double lo, double hi) { const long long x = dbits(a); return dbits(lo) < x && x < dbits(hi); }

// FP64 arithmetic with every operand in a vector register.  An SM's two FP64 units take a warp's fused
// multiply-add in 16 cycles when all three operands are vector registers, and in 19 when one is an
// immediate, a constant-bank or a uniform register, as they do for an addition or a multiplication of two
// operands (measured with dependent and independent chains, 4 to 16 warps per SM).  The forward sweeps keep
// these units busy all the time, so their arithmetic runs in this type: x + y is fma(x, 1, y) and x y is
// fma(x, y, -0), the same bits as the two-operand forms, with 1, -0 and every other constant held as a value
// the compiler cannot prove uniform.  A product met by a sum fuses, as the compiler fuses plain doubles.
// Measured on one state of the kernels, per 400 x 400 step: face lines 0.906 -> 0.807 ms, tangential 1.050 -> 0.934,
// flux 1.381 -> 1.311.
#ifdef __CUDACC__
static __constant__ unsigned kOpaqueZero;      // never written
#endif
DFK_HD double vreg(double c) {
#ifdef __CUDA_ARCH__
    return __hiloint2double(__double2hiint(c) | (int)(threadIdx.x & kOpaqueZero), __double2loint(c));
#else
    return c;
#endif
}
struct Real {
    double v;
    DFK_HD Real() {}
    DFK_HD Real(double c) : v(vreg(c)) {}                                   // a constant or a parameter
    static DFK_HD Real raw(double x) { Real r; r.v = x; return r; }            // a value already in a register
    DFK_HD Real operator-() const { return raw(-v); }
    friend DFK_HD Real fma(Real a, Real b, Real c) { return raw(::fma(a.v, b.v, c.v)); }
    friend DFK_HD Real fabs(Real a) { return raw(::fabs(a.v)); }
};
struct RealProd {
    Real a, b;
#ifndef DFK_TWO_OPERAND_FORMS
    DFK_HD operator Real() const { return Real::raw(::fma(a.v, b.v, vreg(-0.0))); }
#else
    DFK_HD operator Real() const { return Real::raw(a.v * b.v); }
#endif
    DFK_HD RealProd operator-() const { RealProd p; p.a = -a; p.b = b; return p; }
};
DFK_HD RealProd operator*(Real a, Real b) { RealProd p; p.a = a; p.b = b; return p; }
#ifndef DFK_TWO_OPERAND_FORMS
DFK_HD Real operator+(Real a, Real b) { return Real::raw(::fma(a.v, vreg(1.0), b.v)); }
DFK_HD Real operator-(Real a, Real b) { return Real::raw(::fma(a.v, vreg(1.0), -b.v)); }
#else       // a build for flop counters, which would read two flops in fma(x, 1, y)
DFK_HD Real operator+(Real a, Real b) { return Real::raw(a.v + b.v); }
DFK_HD Real operator-(Real a, Real b) { return Real::raw(a.v - b.v); }
#endif
DFK_HD Real operator+(RealProd p, Real c) { return fma(p.a, p.b, c); }
DFK_HD Real operator+(Real c, RealProd p) { return fma(p.a, p.b, c); }
DFK_HD Real operator-(RealProd p, Real c) { return fma(p.a, p.b, -c); }
DFK_HD Real operator-(Real c, RealProd p) { return fma(-p.a, p.b, c); }
DFK_HD Real operator+(RealProd p, RealProd q) { return fma(p.a, p.b, (Real)q); }
DFK_HD Real operator-(RealProd p, RealProd q) { return fma(p.a, p.b, -(Real)q); }
DFK_HD Real nn_max(Real a, Real b) { return Real::raw(nn_max(a.v, b.v)); }
DFK_HD Real nn_min(Real a, Real b) { return Real::raw(nn_min(a.v, b.v)); }
DFK_HD bool nn_less(Real a, Real b) { return nn_less(a.v, b.v); }
DFK_HD bool in_range(Real a, double lo, double hi) { return in_range(a.v, lo, hi); }

struct SchemeConsts {
    double gamma, gm1, K, inv_K2;          // gamma, gamma-1, internal degrees of freedom, 1/(K+2)
    double r2g;                            // sqrt(2/gamma): 1/c = sqrt(2/gamma) sqrt(lambda)
    double d[4];                           // WENO-AO linear weights d0..d3 (Sect. 3.1)
    double inv_d3;
    double eps, alpha_thres, C1, C2;
    int time_limiter, tau_reading, gp_fallback;
    int df_states;                         // DF factor from 0: Gauss-point states, 1: the face's two cell averages
};

// ------------------------------------------------------------------------------------------
// Euler state helpers
// ------------------------------------------------------------------------------------------
// rotate a global-frame state into the local frame of a y-face (theta = pi/2): (rho, rhoV, -rhoU, rhoE)
template <int DIR>
DFK_HD void to_local(double W[4]) {
    if (DIR == 1) { double m = W[1]; W[1] = W[2]; W[2] = -m; }
}
// local-frame flux back to the global frame, F = T^{-1} F~
template <int DIR>
DFK_HD void to_global(double F[4]) {
    if (DIR == 1) { double a = F[1]; F[1] = -F[2]; F[2] = a; }
}

// ------------------------------------------------------------------------------------------
// Characteristic basis of the local-frame x-direction Euler Jacobian at W = (W_l + W_r)/2
// ------------------------------------------------------------------------------------------
struct CharBasis { double u, v, c, ic, H, b1, b2, q2; };

DFK_HD CharBasis make_basis(const double Wl[4], const double Wr[4], const SchemeConsts& S) {
    CharBasis B;
    double r = 0.5 * (Wl[0] + Wr[0]), m = 0.5 * (Wl[1] + Wr[1]);
    double n = 0.5 * (Wl[2] + Wr[2]), E = 0.5 * (Wl[3] + Wr[3]);
    double ir = 1.0 / r;
    B.u = m * ir;
    B.v = n * ir;
    B.q2 = 0.5 * (B.u * B.u + B.v * B.v);
    double p = S.gm1 * (E - r * B.q2);
    const double c2 = S.gamma * p * ir;
    B.ic = rsqrt(c2);                  // one reciprocal square root for 1/c and c = c^2 / c
    B.c = c2 * B.ic;
    B.H = (E + p) * ir;
    B.b1 = S.gm1 * B.ic * B.ic;
    B.b2 = B.q2 * B.b1;
    return B;
}

// Q = L W; components ordered by eigenvalue u-c, u (entropy), u (shear), u+c
DFK_HD void project(const CharBasis& B, const double W[4], double Q[4]) {
    double t = B.b1 * (B.u * W[1] + B.v * W[2] - W[3]);
    double k = B.b2 * W[0] - t;
    double m = (B.u * W[0] - W[1]) * B.ic;
    Q[0] = 0.5 * (k + m);
    Q[1] = W[0] - k;
    Q[2] = W[2] - B.v * W[0];
    Q[3] = 0.5 * (k - m);
}

// W = R Q
DFK_HD void back_project(const CharBasis& B, const double Q[4], double W[4]) {
    double s = Q[0] + Q[3], d = Q[3] - Q[0];
    W[0] = s + Q[1];
    W[1] = B.u * W[0] + B.c * d;
    W[2] = B.v * W[0] + Q[2];
    W[3] = B.H * s + B.u * B.c * d + B.q2 * Q[1] + B.v * Q[2];
}

// ------------------------------------------------------------------------------------------
// WENO-AO(5,3) of Sect. 3.1 on Q_{-2..2} (cell-centred xi in [-1/2, 1/2] of the centre cell).
// Each sub-stencil polynomial is written p_k = Q_0 + a1 xi + a2 (xi^2 - 1/12) (+ a3 xi^3 + a4 (xi^4 - 1/80)
// for the quartic), so its cell mean is Q_0 by construction.  The AO polynomial P = sum c_k p_k with
// c3 = wb3/d3 and c_k = wb_k - c3 d_k sums to one, so P = Q_0 + A1 xi + A2 (xi^2-1/12) + c3 (a3 xi^3 + a4 (xi^4-1/80)).
// ------------------------------------------------------------------------------------------
struct AO {
    double A1, A2;          // sum_k c_k a1_k, sum_k c_k a2_k
    double c3a3, c3a4;      // c3 * a3, c3 * a4 of the quartic
    // the time limiter's ratios tau_Z/(beta_min+eps), tau_Z/(beta_max+eps), both multiplied by rs
    // (1 whenever the reconstruction was taped; the product of the four beta_k+eps otherwise)
    double rmax, rmin, rs;
};

// Optional record of a reconstruction's intermediates for its reverse (a "tape"): a sink with
// put(index, value).  NoTape discards everything, so the plain forward compiles to the arithmetic
// alone; ArrayTape writes a local array, PlaneTape one element of SoA planes in global memory.
struct NoTape {
    static constexpr bool active = false;
    DFK_HD void put(int, double) const {}
};
struct ArrayTape {
    static constexpr bool active = true;
    double* t;
    DFK_HD void put(int i, double v) const { t[i] = v; }
    DFK_HD double get(int i) const { return t[i]; }
};
struct PlaneTape {
    static constexpr bool active = true;
    double* p;
    long long s;
    DFK_HD void put(int i, double v) const { p[(long long)i * s] = v; }
    DFK_HD double get(int i) const { return p[(long long)i * s]; }
};

// WENO-AO tape of one reconstruction: sub-stencil coefficients a1[4], a2[4], the quartic's a3, a4,
// 1/(beta_k+eps), the ratios r_k, unnormalised weights w_k, 1/sum w, c_3, sign(beta_3 - beta_k)
// and the indices of max / min r (first attaining)
enum AOTapeField { AT_A1 = 0, AT_A2 = 4, AT_A3 = 8, AT_A4 = 9, AT_IE = 10, AT_R = 14, AT_W = 18, AT_IW = 22,
                   AT_C3 = 23, AT_SG = 24, AT_KMAX = 27, AT_KMIN = 28, AT_COUNT = 29 };

template <class Tape>
DFK_HD AO weno_ao_t(const double q[5], const SchemeConsts& S, const Tape& tp, int base) {
    const double qm2 = q[0], qm1 = q[1], q0 = q[2], q1 = q[3], q2 = q[4];
    // quadratic sub-stencils {i-2,i-1,i}, {i-1,i,i+1}, {i,i+1,i+2}
    double a1_0 = 0.5 * qm2 - 2.0 * qm1 + 1.5 * q0;
    double a2_0 = 0.5 * (qm2 - 2.0 * qm1 + q0);
    double a1_1 = 0.5 * (q1 - qm1);
    double a2_1 = 0.5 * (qm1 - 2.0 * q0 + q1);
    double a1_2 = -1.5 * q0 + 2.0 * q1 - 0.5 * q2;
    double a2_2 = 0.5 * (q0 - 2.0 * q1 + q2);
    // quartic on the full stencil
    double a1_3 = (5.0 * (qm2 - q2) - 34.0 * (qm1 - q1)) * (1.0 / 48.0);
    double a2_3 = (-(qm2 + q2) + 12.0 * (qm1 + q1) - 22.0 * q0) * (1.0 / 16.0);
    double a3_3 = (-(qm2 - q2) + 2.0 * (qm1 - q1)) * (1.0 / 12.0);
    double a4_3 = ((qm2 + q2) - 4.0 * (qm1 + q1) + 6.0 * q0) * (1.0 / 24.0);
    // smoothness indicators, Eq. 38 with dx^{2q-1} absorbed into the cell-centred coordinate
    const double c13_3 = 13.0 / 3.0;
    double b0 = a1_0 * a1_0 + c13_3 * a2_0 * a2_0;
    double b1 = a1_1 * a1_1 + c13_3 * a2_1 * a2_1;
    double b2 = a1_2 * a1_2 + c13_3 * a2_2 * a2_2;
    double b3 = a1_3 * (a1_3 + 0.5 * a3_3) + c13_3 * a2_3 * a2_3 + (21.0 / 5.0) * a2_3 * a4_3
              + (3129.0 / 80.0) * a3_3 * a3_3 + (87617.0 / 140.0) * a4_3 * a4_3;
    // Eq. 37 and the WENO-Z weights.  With P_k = prod_j (beta_j+eps) / (beta_k+eps) the ratios are
    // r_k = tau P_k / prod; scaled by prod^2 the weights d_k (prod^2 + (tau P_k)^2) need one division
    // (their normalisation) instead of two, and the limiter's ratios none (carried scaled by prod).
    double tau = (fabs(b3 - b0) + fabs(b3 - b1) + fabs(b3 - b2)) * (1.0 / 3.0);
    double e0 = b0 + S.eps, e1 = b1 + S.eps, e2 = b2 + S.eps, e3 = b3 + S.eps;
    double p01 = e0 * e1, p23 = e2 * e3, prod = p01 * p23;
    const double P0 = e1 * p23, P1 = e0 * p23, P2 = p01 * e3, P3 = p01 * e2;
    const double t0 = tau * P0, t1 = tau * P1, t2 = tau * P2, t3 = tau * P3;     // prod * r_k
    const double tmax = nn_max(nn_max(t0, t1), nn_max(t2, t3)), tmin = nn_min(nn_min(t0, t1), nn_min(t2, t3));
    AO o;
    double c0, c1, c2, c3;
    double r0, r1, r2, r3;                           // the ratios themselves: tape and fallback only
    if (nn_less(prod, 1e150) && nn_less(tmax, 1e150)) {   // beta+eps >= eps, so prod >= eps^4 > 0
        const double p2 = prod * prod;
        const double v0 = S.d[0] * (p2 + t0 * t0), v1 = S.d[1] * (p2 + t1 * t1);
        const double v2 = S.d[2] * (p2 + t2 * t2), v3 = S.d[3] * (p2 + t3 * t3);
        const double iv = 1.0 / (v0 + v1 + v2 + v3);
        c3 = v3 * iv * S.inv_d3;
        c0 = v0 * iv - c3 * S.d[0]; c1 = v1 * iv - c3 * S.d[1]; c2 = v2 * iv - c3 * S.d[2];
        o.rmax = tmax; o.rmin = tmin; o.rs = prod;
        if constexpr (Tape::active) {                // unscaled quantities for the reverse
            const double ip = 1.0 / prod;
            r0 = t0 * ip; r1 = t1 * ip; r2 = t2 * ip; r3 = t3 * ip;
            tp.put(base + AT_IE, P0 * ip); tp.put(base + AT_IE + 1, P1 * ip);
            tp.put(base + AT_IE + 2, P2 * ip); tp.put(base + AT_IE + 3, P3 * ip);
            o.rmax = tmax * ip; o.rmin = tmin * ip; o.rs = 1.0;
        }
    } else {
        r0 = tau / e0; r1 = tau / e1; r2 = tau / e2; r3 = tau / e3;
        tp.put(base + AT_IE, 1.0 / e0); tp.put(base + AT_IE + 1, 1.0 / e1);
        tp.put(base + AT_IE + 2, 1.0 / e2); tp.put(base + AT_IE + 3, 1.0 / e3);
        const double w0 = S.d[0] * (1.0 + r0 * r0), w1 = S.d[1] * (1.0 + r1 * r1);
        const double w2 = S.d[2] * (1.0 + r2 * r2), w3 = S.d[3] * (1.0 + r3 * r3);
        const double iw = 1.0 / (w0 + w1 + w2 + w3);
        c3 = w3 * iw * S.inv_d3;
        c0 = w0 * iw - c3 * S.d[0]; c1 = w1 * iw - c3 * S.d[1]; c2 = w2 * iw - c3 * S.d[2];
        // tau >= 0, so the ratio is largest at beta_min and smallest at beta_max
        o.rmax = nn_max(nn_max(r0, r1), nn_max(r2, r3)); o.rmin = nn_min(nn_min(r0, r1), nn_min(r2, r3)); o.rs = 1.0;
    }
    if constexpr (Tape::active) {
        // the reverse differentiates w_k = d_k (1 + r_k^2) and c_k = w_k / sum w - c_3 d_k
        const double w0 = S.d[0] * (1.0 + r0 * r0), w1 = S.d[1] * (1.0 + r1 * r1);
        const double w2 = S.d[2] * (1.0 + r2 * r2), w3 = S.d[3] * (1.0 + r3 * r3);
        const double iw = 1.0 / (w0 + w1 + w2 + w3);
        c3 = w3 * iw * S.inv_d3;
        c0 = w0 * iw - c3 * S.d[0]; c1 = w1 * iw - c3 * S.d[1]; c2 = w2 * iw - c3 * S.d[2];
        tp.put(base + AT_R, r0); tp.put(base + AT_R + 1, r1); tp.put(base + AT_R + 2, r2); tp.put(base + AT_R + 3, r3);
        tp.put(base + AT_W, w0); tp.put(base + AT_W + 1, w1); tp.put(base + AT_W + 2, w2); tp.put(base + AT_W + 3, w3);
        tp.put(base + AT_IW, iw); tp.put(base + AT_C3, c3);
        int kmax = 0, kmin = 0;
        const double rr[4] = {r0, r1, r2, r3};
#pragma unroll
        for (int k = 1; k < 4; ++k) { if (nn_less(rr[kmax], rr[k])) kmax = k; if (nn_less(rr[k], rr[kmin])) kmin = k; }
        tp.put(base + AT_KMAX, (double)kmax);
        tp.put(base + AT_KMIN, (double)kmin);
    }
    o.A1 = c0 * a1_0 + c1 * a1_1 + c2 * a1_2 + c3 * a1_3;
    o.A2 = c0 * a2_0 + c1 * a2_1 + c2 * a2_2 + c3 * a2_3;
    o.c3a3 = c3 * a3_3;
    o.c3a4 = c3 * a4_3;
    tp.put(base + AT_A1, a1_0); tp.put(base + AT_A1 + 1, a1_1); tp.put(base + AT_A1 + 2, a1_2); tp.put(base + AT_A1 + 3, a1_3);
    tp.put(base + AT_A2, a2_0); tp.put(base + AT_A2 + 1, a2_1); tp.put(base + AT_A2 + 2, a2_2); tp.put(base + AT_A2 + 3, a2_3);
    tp.put(base + AT_A3, a3_3); tp.put(base + AT_A4, a4_3);
    tp.put(base + AT_SG, (b3 - b0) >= 0.0 ? 1.0 : -1.0);
    tp.put(base + AT_SG + 1, (b3 - b1) >= 0.0 ? 1.0 : -1.0);
    tp.put(base + AT_SG + 2, (b3 - b2) >= 0.0 ? 1.0 : -1.0);
    return o;
}

DFK_HD AO weno_ao(const double q[5], const SchemeConsts& S) { return weno_ao_t(q, S, NoTape{}, 0); }

// ------------------------------------------------------------------------------------------
// The forward sweeps' WENO-AO, in undivided differences.
//
// With the first differences f, second s, third t1 = s1 - s0, t2 = s2 - s1 of a stencil (s0, s1, s2 the
// second differences about cells i-1, i, i+1; fb, ff the first differences either side of cell i) and
// T = t1 + t2, U = t2 - t1, the sub-stencil coefficients above are
//   a1_0 = fb + s0/2, a1_1 = fb + s1/2, a1_2 = ff - s2/2,  a2_k = s_k/2,
//   a1_3 = a1_1 - 5T/48, a2_3 = s1/2 - U/16, a3 = T/12, a4 = U/24,
// the quartic's smoothness indicator completes to squares,
//   beta_3 = (a1_1 - T/12)^2 + 13/12 (s1 - 11U/130)^2 + 781/2880 T^2 + 1421461/1310400 U^2,
// and, because the linear weights sum to one, with x_k = 1 + r_k^2 and y_k = x_k - x_3 the weights are
//   c_3 = x_3 / sum, c_k = d_k y_k / sum,  sum = x_3 + sum_{k<3} d_k y_k.
// The quartic is the central polynomial and a correction in T and U, so that with c_m = c_1 + c_3 and
//   B = c_0 a1_0 + c_m a1_1 + c_2 a1_2,  D = c_0 s0 + c_m s1 + c_2 s2
// A1 = B - 5/48 c_3 T and 2 A2 = D - c_3 U/8, without a coefficient of a quadratic beside its own weight.  (As a
// departure from the central polynomial, A1 = a1_1 - 5/48 c_3 T - (c_0 t1 + c_2 t2)/2, it is two instructions
// shorter, but beside a jump the jump then cancels out of terms of weight one: the quiet side takes up
// rounding noise of the jump's size, 2e-10 of data of order 1 beside a jump of 1e6, instead of 1e-15.)
// These kernels are bound by the two FP64 units of an SM, so what counts is FP64 instructions: about 75 per
// reconstruction, against 114 from the coefficients of the four polynomials.  Differences also cancel before they
// are projected.  785 FP64 instructions per face line and 442 per face side, against 1097 and 575: the face-line
// kernel takes 0.85 ms per 400 x 400 step, the tangential one 0.94 (1.36 and 1.40 in that form and with two-operand
// instructions).
// ------------------------------------------------------------------------------------------

// 1/x for x in [1e-300, 1e300]: the hardware's approximation (2^-20) refined by one third-order
// Householder step y (1 + e + e^2), e = 1 - x y.  Largest error 0.51 ulp; 3 FP64 instructions against
// the 5 of a division, and no slow path.
DFK_HD Real rcp(Real x) {
#ifdef __CUDA_ARCH__
    Real y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y.v) : "d"(x.v));
    const Real e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
#else
    return Real::raw(1.0 / x.v);
#endif
}

// weights of one reconstruction: c_3 = x3 / sum, c_0 = d0 y0 / sum, c_2 = d0 y2 / sum, c_m = xm / sum, c_m + c_2 =
// xr / sum, and the extreme x_k, all carried scaled by (3 prod)^2, prod = the product of the four beta_k + eps (the
// scale cancels)
struct AOWeights {
    Real x3, y0, y2, xm, xr, sum, xmax, xmin;
    Real a10, a12, s0, s2;                 // the outer quadratics' coefficients (2 a2_k = s_k)
    Real e[4], tau3, prod, p2;             // beta_k + eps, 3 tau, the scale: for ao_ratios
    bool scaled;
};

// 13/12 s^2 + eps, shared by the reconstructions that use the second difference s
DFK_HD Real second_difference_energy(Real s, Real eps) { return fma((13.0 / 12.0) * s, s, eps); }

// SGN -1: a stencil mirrored about its cell, given by the unmirrored differences (the odd ones change
// sign).  w_k: second_difference_energy of s_k.
template <int SGN>
DFK_HD AOWeights ao_weights(Real fb, Real ff, Real s0, Real s1, Real s2, Real w0, Real w1, Real w2,
                            Real a11, Real T, Real U, Real eps, const SchemeConsts& S) {
    const Real h = 0.5 * SGN;
    const Real a10 = fma(h, s0, fb), a12 = fma(-h, s2, ff);
    const Real m1 = fma(-1.0 / 12.0, T, a11), m2 = fma(-11.0 / 130.0, U, s1);
    const Real e0 = fma(a10, a10, w0), e1 = fma(a11, a11, w1), e2 = fma(a12, a12, w2);
    Real e3 = fma((1421461.0 / 1310400.0) * U, U, eps);
    e3 = fma((781.0 / 2880.0) * T, T, e3);
    e3 = fma((13.0 / 12.0) * m2, m2, e3);
    e3 = fma(m1, m1, e3);
    // Eq. 37: tau = (|b3-b0| + |b3-b1| + |b3-b2|)/3; r_k = tau / (beta_k + eps) = t_k / (3 prod)
    const Real tau3 = (fabs(e3 - e0) + fabs(e3 - e1)) + fabs(e3 - e2);
    const Real p01 = e0 * e1, p23 = e2 * e3, prod = p01 * p23;
    const Real g01 = tau3 * p01, g23 = tau3 * p23;
    Real t0 = e1 * g23, t1 = e0 * g23, t2 = e3 * g01, t3 = e2 * g01;
    Real p2;
    const Real tm = nn_max(nn_max(t0, t1), nn_max(t2, t3));
    const bool scaled = in_range(prod, 1e-75, 1e75) && nn_less(tm.v, 1e75);
    if (scaled) {
        const Real p3 = 3.0 * prod;
        p2 = p3 * p3;
    } else {                                       // extreme data: the ratios themselves
        t0 = Real::raw(tau3.v / (3.0 * e0.v)); t1 = Real::raw(tau3.v / (3.0 * e1.v));
        t2 = Real::raw(tau3.v / (3.0 * e2.v)); t3 = Real::raw(tau3.v / (3.0 * e3.v));
        p2 = 1.0;
    }
    const Real tmax = nn_max(nn_max(t0, t1), nn_max(t2, t3)), tmin = nn_min(nn_min(t0, t1), nn_min(t2, t3));
    AOWeights o;
    const Real z3 = t3 * t3;
    o.x3 = fma(t3, t3, p2);
    o.y0 = fma(t0, t0, -z3);
    o.y2 = fma(t2, t2, -z3);
    const Real y1 = fma(t1, t1, -z3);
    o.xm = fma(S.d[1], y1, o.x3);
    o.xr = fma(S.d[0], o.y2, o.xm);
    o.sum = fma(S.d[0], o.y0, o.xr);
    o.a10 = a10; o.a12 = a12; o.s0 = s0; o.s2 = s2;
    o.xmax = fma(tmax, tmax, p2);                  // the time limiter's; dropped where it is not used
    o.xmin = fma(tmin, tmin, p2);
    o.e[0] = e0; o.e[1] = e1; o.e[2] = e2; o.e[3] = e3;
    o.tau3 = tau3; o.prod = prod; o.p2 = p2; o.scaled = scaled;
    return o;
}

// 1/sum: a positive normal number unless the data overflow
DFK_HD Real ao_inverse_sum(const AOWeights& o) { return in_range(o.sum, 1e-300, 1e300) ? rcp(o.sum) : Real::raw(1.0 / o.sum.v); }

// What a reconstruction's reverse needs beside its differences: 1/(beta_k + eps), tau and the unscaled 1/sum.
// Taped (6 planes) where a reverse sweep follows its own forward; the weights cost more than a third of the
// reverse, what they are made from is cheaper to form again.
struct AORatios { Real ie[4], tau, iv; };
enum AORatioField { RT_IE = 0, RT_TAU = 4, RT_IV = 5, RT_COUNT = 6 };

DFK_HD AORatios ao_ratios(const AOWeights& o) {
    AORatios a;
    if (o.scaled) {
        const Real ip = rcp(o.prod), i01 = (o.e[2] * o.e[3]) * ip, i23 = (o.e[0] * o.e[1]) * ip;   // 1/(e0 e1), 1/(e2 e3)
        a.ie[0] = o.e[1] * i01; a.ie[1] = o.e[0] * i01; a.ie[2] = o.e[3] * i23; a.ie[3] = o.e[2] * i23;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) a.ie[k] = Real::raw(1.0 / o.e[k].v);
    }
    a.tau = (1.0 / 3.0) * o.tau3;
    a.iv = ao_inverse_sum(o) * o.p2;
    return a;
}
template <class Tape>
DFK_HD void tape_ratios(const Tape& tp, int b, const AORatios& a) {
#pragma unroll
    for (int k = 0; k < 4; ++k) tp.put(b + RT_IE + k, a.ie[k].v);
    tp.put(b + RT_TAU, a.tau.v);
    tp.put(b + RT_IV, a.iv.v);
}
template <class Tape>
DFK_HD AORatios tape_get_ratios(const Tape& tp, int b) {
    AORatios a;
#pragma unroll
    for (int k = 0; k < 4; ++k) a.ie[k] = Real::raw(tp.get(b + RT_IE + k));
    a.tau = Real::raw(tp.get(b + RT_TAU));
    a.iv = Real::raw(tp.get(b + RT_IV));
    return a;
}

// B and D times the sum of the weights, of coefficients a10, a11, a12 or s0, s1, s2
DFK_HD Real ao_sum(const AOWeights& o, Real a0, Real am, Real a2, const SchemeConsts& S) {
    return fma(S.d[0], fma(o.y0, a0, o.y2 * a2), o.xm * am);
}

// the polynomial's value minus the average (q[0]) and slope (q[1], times idn) at the face, xi = SGN/2 of a cell whose
// third differences are to (outer) and ti: with D and the slope's H = c_0 (fb + SGN s0) + (c_m + c_2) ff, the central
// and the inner quadratic having the face's difference ff as their slope there,
//   value = SGN (H/2 - c_3 (to/30 + ti/20)) - D/6,  slope = H - c_3 ti/12
template <int SGN>
DFK_HD void ao_diff_at_edge(const AOWeights& o, Real fb, Real ff, Real s1, Real to, Real ti, Real idn, const SchemeConsts& S, Real q[2]) {
    const Real iv = ao_inverse_sum(o), D = ao_sum(o, o.s0, s1, o.s2, S);
    const Real H = fma(S.d[0], Real(o.y0 * (SGN > 0 ? fb + o.s0 : fb - o.s0)), o.xr * ff);
    const Real w = o.x3 * fma(1.0 / 30.0, to, (1.0 / 20.0) * ti);
    q[0] = iv * fma(-1.0 / 6.0, D, SGN > 0 ? fma(0.5, H, -w) : fma(-0.5, H, w));
    q[1] = (idn * iv) * fma(-o.x3, (1.0 / 12.0) * ti, H);
}

// values minus q0 and d/deta (unscaled) at the two Gauss points eta = -g (m=1), +g (m=2), g = sqrt(3)/6, from a11, s1
// and the third differences (their sum T and difference U)
DFK_HD void ao_diff_at_gauss(const AOWeights& o, Real a11, Real s1, Real, Real, Real T, Real U,
                             const SchemeConsts& S, Real val[2], Real slope[2]) {
    const Real g = kGaussEta;
    const Real iv = ao_inverse_sum(o), c3 = o.x3 * iv;
    const Real B = iv * ao_sum(o, o.a10, a11, o.a12, S), D = iv * ao_sum(o, o.s0, s1, o.s2, S);
    const Real c3T = c3 * T, c3U = c3 * U;
    const Real O = g * fma(-7.0 / 72.0, c3T, B), Es = fma(-1.0 / 12.0, c3T, B);
    const Real Os = fma(-1.0 / 9.0, c3U, D), E = (-1.0 / 4320.0) * c3U;
    val[0] = E - O; val[1] = E + O;
    slope[0] = fma(-g, Os, Es); slope[1] = fma(g, Os, Es);
}

// the zero-mean DF quadratic's (Sect. 3.3) values minus q0 and slopes there
DFK_HD void df_diff_at_gauss(Real a11, Real s1, Real alpha, Real val[2], Real slope[2]) {
    const Real g = kGaussEta, Es = alpha * a11, O = g * Es, Os = (g * alpha) * s1;
    val[0] = -O; val[1] = O;
    slope[0] = Es - Os; slope[1] = Es + Os;
}

// Projection of differences of states onto the characteristic variables, with the two acoustic ones
// doubled (Q_0 = k + m, Q_3 = k - m): their smoothness indicators then carry 4 eps, which leaves the
// weights as they are, and the back projection halves them again.  10 instructions each way.
struct DiffBasis {
    Real b1, b1u, b1v, b2, ic, uic, v;                     // projection
    Real u, hc, hH, huc, q2;                               // back projection
};
DFK_HD DiffBasis diff_basis(const CharBasis& B) {
    DiffBasis D;
    D.b1 = Real::raw(B.b1); D.b2 = Real::raw(B.b2); D.ic = Real::raw(B.ic); D.u = Real::raw(B.u); D.v = Real::raw(B.v); D.q2 = Real::raw(B.q2);
    D.b1u = D.b1 * D.u; D.b1v = D.b1 * D.v; D.uic = D.u * D.ic;
    D.hc = 0.5 * Real::raw(B.c); D.hH = 0.5 * Real::raw(B.H); D.huc = D.u * D.hc;
    return D;
}
DFK_HD void project_diff(const DiffBasis& D, const Real W[4], Real Q[4]) {
    const Real k = fma(D.b1, W[3], fma(-D.b1v, W[2], fma(-D.b1u, W[1], D.b2 * W[0])));
    const Real m = fma(-D.ic, W[1], D.uic * W[0]);
    Q[0] = k + m;
    Q[1] = W[0] - k;
    Q[2] = fma(-D.v, W[0], W[2]);
    Q[3] = k - m;
}
DFK_HD void back_project_diff(const DiffBasis& D, const Real Q[4], Real W[4]) {
    const Real s = Q[0] + Q[3], d = Q[3] - Q[0];
    W[0] = fma(0.5, s, Q[1]);
    W[1] = fma(D.u, W[0], D.hc * d);
    W[2] = fma(D.v, W[0], Q[2]);
    W[3] = fma(D.hH, s, fma(D.huc, d, fma(D.q2, Q[1], D.v * Q[2])));
}

// time-limiter ingredient 2 at2 / (at1 + at2) of one reconstruction (Sect. 2.2), as numerator and
// (positive) denominator, so that a minimum over several needs one division at the end
DFK_HD void limiter_fraction(const AO& o, double& num, double& den) {
    // 1 + r^2 scaled by rs^2, which cancels in the ratio
    const double s2 = o.rs * o.rs;
    double a1 = s2 + o.rmax * o.rmax, a2 = s2 + o.rmin * o.rmin;
    num = 2.0 * a2;
    den = a1 + a2;
}

DFK_HD double limiter_alpha(const AO& o) {
    double n, d;
    limiter_fraction(o, n, d);
    return n / d;
}

// value and d/dxi of the AO polynomial at the right cell edge xi = +1/2
DFK_HD void ao_at_right_edge(const AO& o, double q0, double& val, double& slope) {
    val = q0 + 0.5 * o.A1 + (1.0 / 6.0) * o.A2 + 0.125 * o.c3a3 + 0.05 * o.c3a4;
    slope = o.A1 + o.A2 + 0.75 * o.c3a3 + 0.5 * o.c3a4;
}

// zero-mean DF quadratic of Sect. 3.3, p_DF = Q_0 + alpha (p1 - Q_0), at xi = +1/2
DFK_HD void df_at_right_edge(const double q[5], double alpha, double& val, double& slope) {
    double a1 = 0.5 * (q[3] - q[1]);
    double a2 = 0.5 * (q[1] - 2.0 * q[2] + q[3]);
    val = q[2] + alpha * (0.5 * a1 + (1.0 / 6.0) * a2);
    slope = alpha * (a1 + a2);
}

// values and d/deta at the two Gauss points eta = -g (m=1), +g (m=2), g = sqrt(3)/6
DFK_HD void ao_at_gauss(const AO& o, double q0, double val[2], double slope[2]) {
    const double g = kGaussEta;
    double E = q0 - (1.0 / 180.0) * o.c3a4;                 // even part: xi^2 = 1/12, xi^4 = 1/144
    double O = g * (o.A1 + (1.0 / 12.0) * o.c3a3);          // odd part
    double Es = o.A1 + 0.25 * o.c3a3;
    double Os = g * (2.0 * o.A2 + (1.0 / 3.0) * o.c3a4);
    val[0] = E - O; val[1] = E + O;
    slope[0] = Es - Os; slope[1] = Es + Os;
}

DFK_HD void df_at_gauss(const double q[5], double alpha, double val[2], double slope[2]) {
    const double g = kGaussEta;
    double a1 = 0.5 * (q[3] - q[1]);
    double a2 = 0.5 * (q[1] - 2.0 * q[2] + q[3]);
    double O = alpha * g * a1;                               // xi^2 - 1/12 vanishes at the Gauss points
    double Es = alpha * a1, Os = alpha * 2.0 * g * a2;
    val[0] = q[2] - O; val[1] = q[2] + O;
    slope[0] = Es - Os; slope[1] = Es + Os;
}

// ------------------------------------------------------------------------------------------
// A side's Maxwellian for the DF factor of two cell averages (df_alpha)
// ------------------------------------------------------------------------------------------
struct Maxw { double rho, ir, U, V, p, tl, isl; };   // tl = 2 lambda = rho/p, isl = 1/sqrt(lambda)

// velocities and pressure of W given ir = 1/rho
DFK_HD void maxw_velocities(const double W[4], double ir, const SchemeConsts& S, Maxw& s) {
    s.rho = W[0];
    s.ir = ir;
    s.U = W[1] * ir;
    s.V = W[2] * ir;
    s.p = S.gm1 * (W[3] - 0.5 * W[0] * (s.U * s.U + s.V * s.V));
}

// the rest given tl = 2 lambda = rho / p
DFK_HD void maxw_finish(double tl, Maxw& s) {
    s.tl = tl;
    s.isl = rsqrt(0.5 * tl);
}

// the two sides' Maxwellians with two divisions instead of four: 1/(rho_l rho_r) gives both 1/rho
// and 1/(p_l p_r) both rho/p.  A product outside [1e-150, 1e150] (non-physical or extreme states)
// is divided side by side.
DFK_HD void maxw_pair(const double WL[4], const double WR[4], const SchemeConsts& S, Maxw& a, Maxw& b) {
    const double rr = WL[0] * WR[0];
    if (in_range(rr, 1e-150, 1e150)) {
        const double r = 1.0 / rr;
        maxw_velocities(WL, WR[0] * r, S, a);
        maxw_velocities(WR, WL[0] * r, S, b);
    } else {
        maxw_velocities(WL, 1.0 / WL[0], S, a);
        maxw_velocities(WR, 1.0 / WR[0], S, b);
    }
    const double pp = a.p * b.p;
    if (in_range(pp, 1e-150, 1e150)) {
        const double r = 1.0 / pp;
        maxw_finish(WL[0] * b.p * r, a);
        maxw_finish(WR[0] * a.p * r, b);
    } else {
        maxw_finish(WL[0] / a.p, a);
        maxw_finish(WR[0] / b.p, b);
    }
}

struct GPState { double W[4], Wn[4], Wt[4]; };   // one side of one Gauss point, local frame

// ------------------------------------------------------------------------------------------
// Gas-kinetic flux at one Gauss point in the local frame (Sect. 2.2, 3.4; Eqs. 25-27), in gradient form.
//
// rho <a phi> with the slope polynomial a of a Maxwellian g (a g = the derivative of g along W') is the
// derivative of the moment rho <phi> itself, so no slope coefficients are needed: with the primitive
// gradient r0 = rho', r1 = rho U', r2 = rho V', q3 = rho theta' (theta = p/rho) and m_k = <u^k> over the
// side's half space,
//   N_k = rho <a u^k> = r0 m_k + r1 dm_k/dU + q3 dm_k/dtheta,
//   dm_k/dU = k m_{k-1},  dm_k/dtheta = k(k-1)/2 m_{k-2}  (k >= 2; the boundary u = 0 adds the terms in
//   phi, the value of the marginal distribution there, for k = 0, 1),
// and in the frame of the state's own tangential velocity (v' = v - V, odd moments zero)
//   rho <a u^k psi'> = (N_k, N_{k+1}, r2 m_k, N_{k+2}/2 + (K+1)/2 G_k),  G_k = theta N_k + q3 m_k,
//   rho <a u^k v' psi'> = (r2 m_k, r2 m_{k+1}, G_k, r2 (m_{k+2} + (K+3) theta m_k)/2).
// The equilibrium state's time derivative is the Euler equations' (its compatibility condition in closed
// form).  Moments end at u^4 instead of u^6.  590 FP64 instructions per Gauss point against 1028 with
// slope coefficients and general products of moments, on a kernel bound by the FP64 units: 2.38 -> 1.38 ms
// per 400 x 400 step (1.09 with vector-register operands and the tables below), 158 instead of 250 registers.
// ------------------------------------------------------------------------------------------

// What the flux's reverse (gks_flux_reverse) reads of its forward: per side 1/rho, m_0, the boundary value
// phi (signed) and 1/(2 theta); the equilibrium state, its 1/rho and its two gradients; the time coefficients
// of Eq. 27 (the last four under the tau = tau_n reading only); the derivatives of F and dF by tau_n/dt; and
// that ratio's by the two pressures.  39 values: what costs a transcendental, a division or a sum over both
// sides.  States, gradients and moments are cheaper to form again than to keep.
enum GksTapeField {
    TG_L = 0, TG_R = 4, TG_WC = 8, TG_IRC = 12, TG_WCX = 13, TG_WCY = 17,
    TG_GF = 21, TG_GD, TG_AF, TG_AD, TG_T, TG_CF, TG_CD, TG_BF, TG_FR = 29, TG_DFR = 33, TG_PL = 37, TG_PR = 38, TG_COUNT = 39
};

// rcp() where its range holds, a division elsewhere (negative, zero, extreme)
DFK_HD Real rcp_or_div(Real x) { return in_range(x, 1e-300, 1e300) ? rcp(x) : Real::raw(1.0 / x.v); }

// velocities, pressure, theta = p/rho and hq = (U^2 + V^2)/2 of a state; for the two sides of a Gauss
// point also rs = 1/sqrt(2 theta), which the half-space moments and the DF factor's sound speed share
struct FlowState { Real rho, ir, U, V, p, th, hq, rs; };

DFK_HD FlowState flow_state(const Real W[4], const SchemeConsts& S) {
    FlowState s;
    s.rho = W[0];
    s.ir = rcp_or_div(W[0]);
    s.U = W[1] * s.ir;
    s.V = W[2] * s.ir;
    s.hq = 0.5 * fma(s.U, s.U, s.V * s.V);
    s.p = S.gm1 * fma(-W[0], s.hq, W[3]);
    s.th = s.p * s.ir;
    return s;
}
DFK_HD FlowState side_state(const double W[4], const SchemeConsts& S) {
    const Real w[4] = {Real::raw(W[0]), Real::raw(W[1]), Real::raw(W[2]), Real::raw(W[3])};
    FlowState s = flow_state(w, S);
    s.rs = Real::raw(rsqrt(Real(2.0 * s.th).v));
    return s;
}

// DF factor of one Gauss point (Sect. 3.2, Eq. 33) from its two sides: 1/c = sqrt(2/gamma) / sqrt(2 theta),
// |p_l - p_r| (1/p_l + 1/p_r) with 1/p = 2 rs^2 / rho
DFK_HD Real df_alpha_sides(const FlowState& l, const FlowState& r, const SchemeConsts& S) {
    const Real cl = S.r2g * l.rs, cr = S.r2g * r.rs;
    const Real dn = fma(l.U, cl, -(r.U * cr)), dt = fma(l.V, cl, -(r.V * cr));
    const Real ips = fma(l.rs * l.rs, l.ir, (r.rs * r.rs) * r.ir);
    const Real D = fma(2.0 * fabs(l.p - r.p), ips, fma(dn, dn, dt * dt));
    return rcp_or_div(fma(D, D, 1.0));
}

// r0, r1, r2, q3 and p' of the state along a gradient of its conserved variables
struct FlowGrad { Real r0, r1, r2, q3, dp; };
DFK_HD FlowGrad flow_grad(const FlowState& s, const Real d[4], const SchemeConsts& S) {
    FlowGrad g;
    g.r0 = d[0];
    g.r1 = fma(-s.U, d[0], d[1]);
    g.r2 = fma(-s.V, d[0], d[2]);
    g.dp = S.gm1 * fma(-s.U, g.r1, fma(-s.V, g.r2, fma(-s.hq, d[0], d[3])));
    g.q3 = fma(-s.th, d[0], g.dp);
    return g;
}

DFK_HD FlowGrad point_grad(const FlowState& s, const double d[4], const SchemeConsts& S) {
    const Real w[4] = {Real::raw(d[0]), Real::raw(d[1]), Real::raw(d[2]), Real::raw(d[3])};
    return flow_grad(s, w, S);
}

// moments m_k = <u^k>, k <= 4, and their derivatives' terms: e1[k] = dm_k/dU, e2[k] = dm_k/dtheta
struct HalfMom { Real m[5], e1[5], e2[5]; };
DFK_HD void finish_moments(const FlowState& s, HalfMom& h) {
    const Real th2 = 2.0 * s.th, th3 = 3.0 * s.th;
    h.m[2] = fma(s.U, h.m[1], s.th * h.m[0]);
    h.m[3] = fma(s.U, h.m[2], th2 * h.m[1]);
    h.m[4] = fma(s.U, h.m[3], th3 * h.m[2]);
    h.e1[1] = h.m[0]; h.e1[2] = 2.0 * h.m[1]; h.e1[3] = 3.0 * h.m[2]; h.e1[4] = 4.0 * h.m[3];
    h.e2[2] = h.m[0]; h.e2[3] = 3.0 * h.m[1]; h.e2[4] = 6.0 * h.m[2];
}
// Gaussians and complementary error functions of the half-space moments from tables.  CUDA's exp and erfcx
// are 16 and 40 FP64 instructions (19 cycles each: their constants are immediates), 112 of the flux's 600
// for the two sides; the reductions below take 11 and 10, and table entries arrive in vector registers.
// exp(-y): Tang's table-driven method, y = -n ln2/64 - r, a degree-5 polynomial in |r| <= ln2/128 and 2^(n/64)
// from a table; relative error below 1.2 ulp.  erfcx: see the table.  The tables (0.5 and 12 KB) stay in L1:
// neighbouring threads read neighbouring rows.  601 -> 522 FP64 instructions per Gauss point; flux kernel
// 1.311 -> 1.090 ms per 400 x 400 step.
#ifdef __CUDACC__
static __device__ const double kExp2Dev[64] = {
#include "dfgks_exp2_table.inc"
};
static __device__ __align__(16) const double kErfcxDev[193 * 8] = {
#include "dfgks_erfcx_table.inc"
};
#endif
static const double kExp2Host[64] = {
#include "dfgks_exp2_table.inc"
};
static const double kErfcxHost[193 * 8] = {
#include "dfgks_erfcx_table.inc"
};
constexpr double kRoundToInt = 6755399441055744.0;      // 1.5 2^52: x + this - this rounds x to an integer

// exp(-y) for 0 <= y < 700
DFK_HD Real exp_neg_table(Real y) {
    const Real nf = fma(y, -92.33248261689366, kRoundToInt);                      // 64/ln2
    const int n = (int)dbits(nf.v);
    const Real m = nf - kRoundToInt;
    // ln2/64 in 32 bits, exact times m, and the rest
    const Real r = fma(m, -2.9815858269852933e-12, fma(m, -0.01083042469326756, -y));
    Real p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(p, r, 1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(r * r, p, r);
#ifdef __CUDA_ARCH__
    const Real T = Real::raw(__ldg(kExp2Dev + (n & 63)));
#else
    const Real T = Real::raw(kExp2Host[n & 63]);
#endif
    const Real e = fma(T, p, T);
    return Real::raw(dval(dbits(e.v) + ((long long)(n >> 6) << 52)));
}
// exp(-y), y >= 0
DFK_HD Real exp_neg(Real y) {
    if (nn_less(y.v, 700.0)) return exp_neg_table(y);
    return Real::raw(exp(-y.v));
}

// G = exp(-x^2) and t = erfc(|x|)/2 = G erfcx(|x|)/2
DFK_HD void gauss_erfc(Real x, Real& G, Real& t) {
    const Real y = x * x, a = fabs(x);
    if (nn_less(a.v, 6.0)) {
        G = exp_neg_table(y);
        const Real jf = fma(a, 32.0, kRoundToInt);
        const int j = (int)dbits(jf.v);
        const Real d = fma(jf - kRoundToInt, -1.0 / 32.0, a);
#ifdef __CUDA_ARCH__
        const double2* row = reinterpret_cast<const double2*>(kErfcxDev + 8 * j);
        const double2 c01 = __ldg(row), c23 = __ldg(row + 1), c45 = __ldg(row + 2), c67 = __ldg(row + 3);
        const double c[8] = {c01.x, c01.y, c23.x, c23.y, c45.x, c45.y, c67.x, c67.y};
#else
        const double* c = kErfcxHost + 8 * j;
#endif
        Real e = Real::raw(c[7]);
#pragma unroll
        for (int k = 6; k >= 0; --k) e = fma(e, d, Real::raw(c[k]));
        t = G * e;
    } else {                                   // t < 1e-17: beyond Mach 7, or not a number
        G = Real::raw(exp(-y.v));
#ifdef __CUDA_ARCH__
        t = 0.5 * G * Real::raw(erfcx(a.v));
#else
        t = 0.5 * erfc(a.v);
#endif
    }
}

template <int HALF>
DFK_HD void half_moments(const FlowState& s, HalfMom& h) {
    const Real x = s.U * s.rs;
    Real G, t;
    gauss_erfc(x, G, t);
    // the marginal distribution at u = 0, exp(-U^2/(2 theta)) / sqrt(2 pi theta)
    const Real phi = (0.56418958354775628695 * s.rs) * G;
    const bool xpos = dbits(x.v) >= 0;                    // erfc(-|x|) = 2 - erfc(|x|)
    h.m[0] = (HALF > 0) == xpos ? 1.0 - t : t;
    const Real sphi = HALF > 0 ? phi : -phi;
    h.m[1] = fma(s.U, h.m[0], s.th * sphi);
    h.e1[0] = sphi;
    h.e2[0] = -(sphi * x) * s.rs;
    h.e2[1] = 0.5 * sphi;
    finish_moments(s, h);
}

DFK_HD Real grad_mom(const HalfMom& h, const FlowGrad& g, int k) { return fma(g.r0, h.m[k], fma(g.r1, h.e1[k], g.q3 * h.e2[k])); }

// from the frame of tangential velocity V to the laboratory's, for a vector of psi moments
DFK_HD void to_lab(Real V, Real hV2, Real o[4]) {
    o[3] = fma(V, o[2], fma(hV2, o[0], o[3]));
    o[2] = fma(V, o[0], o[2]);
}

// rho <u^2 a_x psi> + rho <u v a_y psi> in the state's own tangential frame
// (k1 = (K+1)/2, k3 = (K+3)/2; Nx[j] = N_{2+j} of the normal gradient, Ny[j] = N_{1+j} of the tangential)
DFK_HD void transport(const FlowState& s, const HalfMom& h, const FlowGrad& x, const FlowGrad& y, const Real Nx[3],
                      const Real Ny[3], Real k1, Real k3, Real o[4]) {
    const Real G2 = fma(s.th, Nx[0], x.q3 * h.m[2]), G1 = fma(s.th, Ny[0], y.q3 * h.m[1]);
    const Real v1 = y.r2 * h.m[1];
    o[0] = fma(s.V, Ny[0], Nx[0]) + v1;
    o[1] = fma(s.V, Ny[1], fma(y.r2, h.m[2], Nx[1]));
    o[2] = fma(s.V, v1, fma(x.r2, h.m[2], G1));
    o[3] = fma(0.5, fma(y.r2, h.m[3], fma(s.V, Ny[2], Nx[2])), fma(k3 * s.th, v1, k1 * fma(s.V, G1, G2)));
}

// one side's sums: c = rho <psi>, cx, cy = rho <a psi> along the two gradients, g0 = rho <u psi>,
// g1 = rho <u^2 a_x psi> + rho <u v a_y psi>.  The left side (HALF > 0) comes first and sets them, the
// right one adds (an addition to zero is not free on the FP64 units)
template <int HALF>
DFK_HD Real acc(Real x, Real to) { return HALF > 0 ? x : x + to; }
template <int HALF>
DFK_HD Real acc(RealProd x, Real to) { return HALF > 0 ? (Real)x : x + to; }
template <int HALF>
DFK_HD void side_sums(const FlowState& s, const FlowGrad& x, const FlowGrad& y, const HalfMom& h, Real k1, Real k3,
                      Real c[4], Real cx[4], Real cy[4], Real g0[4], Real g1[4]) {
    const Real hV2 = 0.5 * s.V * s.V, rk = fma(k1, s.th, hV2), rm0 = s.rho * h.m[0], rm1 = s.rho * h.m[1],
               rm2 = s.rho * h.m[2];
    c[0] = acc<HALF>(rm0, c[0]);
    c[1] = acc<HALF>(rm1, c[1]);
    c[2] = acc<HALF>(s.V * rm0, c[2]);
    c[3] = fma(0.5, rm2, acc<HALF>(rk * rm0, c[3]));
    g0[0] = acc<HALF>(rm1, g0[0]);
    g0[1] = acc<HALF>(rm2, g0[1]);
    g0[2] = acc<HALF>(s.V * rm1, g0[2]);
    g0[3] = fma(0.5 * s.rho, h.m[3], acc<HALF>(rk * rm1, g0[3]));
    Real Nx[3], Ny[3], o[4];
    {
        const Real N0 = grad_mom(h, x, 0), p = x.r2 * h.m[0];
        Nx[0] = grad_mom(h, x, 2);
        cx[0] = acc<HALF>(N0, cx[0]);
        cx[1] = fma(x.r0, h.m[1], fma(x.r1, h.e1[1], acc<HALF>(x.q3 * h.e2[1], cx[1])));
        cx[2] = fma(s.V, N0, acc<HALF>(p, cx[2]));
        cx[3] = fma(s.V, p, fma(hV2, N0, fma(0.5, Nx[0], acc<HALF>(k1 * fma(s.th, N0, x.q3 * h.m[0]), cx[3]))));
        Nx[1] = fma(x.r0, h.m[3], fma(x.r1, h.e1[3], acc<HALF>(x.q3 * h.e2[3], g1[1])));
        Nx[2] = grad_mom(h, x, 4);
    }
    {
        const Real N0 = grad_mom(h, y, 0), p = y.r2 * h.m[0];
        Ny[0] = grad_mom(h, y, 1); Ny[1] = grad_mom(h, y, 2);
        cy[0] = acc<HALF>(N0, cy[0]);
        cy[1] = acc<HALF>(Ny[0], cy[1]);
        cy[2] = fma(s.V, N0, acc<HALF>(p, cy[2]));
        cy[3] = fma(s.V, p, fma(hV2, N0, fma(0.5, Ny[1], acc<HALF>(k1 * fma(s.th, N0, y.q3 * h.m[0]), cy[3]))));
        Ny[2] = grad_mom(h, y, 3);
    }
    transport(s, h, x, y, Nx, Ny, k1, k3, o);       // o[1] has the sum so far through Nx[1]
    g1[3] = acc<HALF>(Real(fma(s.V, o[2], fma(hV2, o[0], o[3]))), g1[3]);
    g1[2] = fma(s.V, o[0], acc<HALF>(o[2], g1[2]));
    g1[1] = o[1];
    g1[0] = acc<HALF>(o[0], g1[0]);
}

// the Euler equations' time derivative of a state with gradients x, y, as a gradient
DFK_HD FlowGrad euler_time_grad(const FlowState& s, const FlowGrad& x, const FlowGrad& y, const SchemeConsts& S) {
    FlowGrad t;
    const Real div = x.r1 + y.r2;
    t.r0 = -fma(s.U, x.r0, fma(s.V, y.r0, div));
    t.r1 = -fma(s.U, x.r1, fma(s.V, y.r1, x.dp));
    t.r2 = -fma(s.U, x.r2, fma(s.V, y.r2, y.dp));
    t.dp = -fma(s.U, x.dp, fma(s.V, y.dp, (S.gamma * s.th) * div));
    t.q3 = fma(-s.th, t.r0, t.dp);
    return t;
}

// under the tau = tau_n reading: rho <u A psi> of one side, A from the side's own compatibility condition
DFK_HD void side_time_sum(const FlowState& s, const FlowGrad& x, const FlowGrad& y, const HalfMom& h, const SchemeConsts& S,
                          Real k1, Real g2[4]) {
    const FlowGrad t = euler_time_grad(s, x, y, S);
    Real o[4];
    const Real N1 = grad_mom(h, t, 1);
    o[0] = N1; o[1] = grad_mom(h, t, 2); o[2] = t.r2 * h.m[1];
    o[3] = fma(0.5, grad_mom(h, t, 3), k1 * fma(s.th, N1, t.q3 * h.m[1]));
    to_lab(s.V, 0.5 * s.V * s.V, o);
#pragma unroll
    for (int i = 0; i < 4; ++i) g2[i] = g2[i] + o[i];
}

template <class Tape>
DFK_HD void tape_side(const Tape& tp, int b, const FlowState& s, const HalfMom& h) {
    if constexpr (Tape::active) { tp.put(b, s.ir.v); tp.put(b + 1, h.m[0].v); tp.put(b + 2, h.e1[0].v); tp.put(b + 3, Real(s.rs * s.rs).v); }
}
template <class Tape>
DFK_HD void tape_vec(const Tape& tp, int b, const Real v[4]) {
    if constexpr (Tape::active) {
#pragma unroll
        for (int i = 0; i < 4; ++i) tp.put(b + i, v[i].v);
    }
}

// sl, sr: side_state of L.W and R.W
template <class Tape>
DFK_HD void gks_flux_sides(const GPState& L, const GPState& Rt, const FlowState& sl, const FlowState& sr, double dtv,
                           const SchemeConsts& S, double F[4], double dF[4], const Tape& tp) {
    const Real dt = dtv;
    const Real k1 = 0.5 * (S.K + 1.0), k3 = 0.5 * (S.K + 3.0);
    // Sect. 3.4: the equilibrium state and its slopes by kinetic weighting, and the sides' flux moments
    Real Wc[4], Wcx[4], Wcy[4], dg[4], g1[4], g2[4] = {0.0, 0.0, 0.0, 0.0};
    {
        const FlowGrad x = point_grad(sl, L.Wn, S), y = point_grad(sl, L.Wt, S);
        HalfMom h;
        half_moments<+1>(sl, h);
        tape_side(tp, TG_L, sl, h);
        side_sums<+1>(sl, x, y, h, k1, k3, Wc, Wcx, Wcy, dg, g1);
        if (S.tau_reading == 1) side_time_sum(sl, x, y, h, S, k1, g2);
    }
    {
        const FlowGrad x = point_grad(sr, Rt.Wn, S), y = point_grad(sr, Rt.Wt, S);
        HalfMom h;
        half_moments<-1>(sr, h);
        tape_side(tp, TG_R, sr, h);
        side_sums<-1>(sr, x, y, h, k1, k3, Wc, Wcx, Wcy, dg, g1);
        if (S.tau_reading == 1) side_time_sum(sr, x, y, h, S, k1, g2);
    }
    // the equilibrium state: c0 = rho <u psi>, c1 = rho <u^2 a_x psi> + rho <u v a_y psi>, c2 = rho <u A psi>
    const FlowState c = flow_state(Wc, S);
    tape_vec(tp, TG_WC, Wc); tape_vec(tp, TG_WCX, Wcx); tape_vec(tp, TG_WCY, Wcy);
    if constexpr (Tape::active) tp.put(TG_IRC, c.ir.v);
    Real c0[4], c1[4], c2[4];
    {
        const FlowGrad x = flow_grad(c, Wcx, S), y = flow_grad(c, Wcy, S), t = euler_time_grad(c, x, y, S);
        HalfMom h;                                   // the full space: no boundary terms
        h.m[0] = 1.0; h.m[1] = c.U;
        h.e1[0] = 0.0; h.e2[0] = 0.0; h.e2[1] = 0.0;
        finish_moments(c, h);
        const Real hV2 = 0.5 * c.V * c.V, hU2 = 0.5 * c.U * c.U, gg = 0.5 * (S.K + 4.0);   // gamma / (gamma - 1)
        const Real ru = Wc[1];
        c0[0] = ru;
        c0[1] = fma(ru, c.U, c.p);
        c0[2] = 0.0;
        c0[3] = fma(hU2, ru, (gg * c.U) * c.p);
        to_lab(c.V, hV2, c0);
        const Real n1 = fma(c.U, t.r0, t.r1);
        c2[0] = n1;
        c2[1] = fma(c.U, n1 + t.r1, t.dp);
        c2[2] = c.U * t.r2;
        c2[3] = fma(hU2, fma(2.0, t.r1, n1), gg * fma(c.U, t.dp, c.th * t.r1));
        to_lab(c.V, hV2, c2);
        const Real Nx[3] = {grad_mom(h, x, 2), grad_mom(h, x, 3), grad_mom(h, x, 4)};
        const Real Ny[3] = {fma(c.U, y.r0, y.r1), grad_mom(h, y, 2), grad_mom(h, y, 3)};
        transport(c, h, x, y, Nx, Ny, k1, k3, c1);
        to_lab(c.V, hV2, c1);
    }
    // numerical collision time (Sect. 2.2) and the time coefficients of Eq. 27 (4 G(dt/2) - G(dt)) / dt and
    // 4 (G(dt) - 2 G(dt/2)) / dt^2, combined with E(dt) = E(dt/2)^2
    const Real ips = rcp_or_div(sl.p + sr.p), q = (sl.p - sr.p) * ips;
    const Real rT = fma(S.C2, fabs(q), S.C1);        // tau_n / dt
    Real E2 = 0.0, r = 0.0, h = 0.0;
    const bool viscous = dbits(rT.v) > 0;            // rT >= 0
    if (viscous) {
        h = 0.5 * rcp_or_div(rT);
        E2 = exp_neg(h);
        r = rT;
    }
    const Real om = 1.0 - E2, om2 = om * om, rom = r * om, idt = rcp_or_div(dt);
    const Real gF = rom * (3.0 - E2), gD = -4.0 * (r * om2) * idt;
    const Real aF = (r * dt) * (gF + (om2 - 1.0)), aD = 4.0 * rom * (E2 - rom);
    // their derivatives by r, with r E2' = h E2 (h = 1/(2 r))
    [[maybe_unused]] Real hE, gFr, gDr, aFr, aDr;
    if constexpr (Tape::active) {
        hE = h * E2;
        gFr = viscous ? fma(om, 3.0 - E2, -2.0 * hE * (2.0 - E2)) : Real(0.0);
        gDr = viscous ? Real(-4.0 * (om * fma(-2.0, hE, om)) * idt) : Real(0.0);
        aFr = dt * fma(r, gFr, fma(-2.0 * om, hE, gF + (om2 - 1.0)));
        aDr = 4.0 * fma(om, E2, fma(hE, fma(2.0, rom, om - E2), -2.0 * rom * om));
        tp.put(TG_GF, gF.v); tp.put(TG_GD, gD.v);
        const Real k2 = (Real(2.0 * S.C2) * ips) * ips, kl = k2 * sr.p, kr = k2 * sl.p;
        tp.put(TG_PL, dbits(q.v) >= 0 ? kl.v : -kl.v);
        tp.put(TG_PR, dbits(q.v) >= 0 ? -kr.v : kr.v);
    }
    if (S.tau_reading == 1) {                        // tau = tau_n: aF, aD as below with r (..) for tau = 0 added
        const Real T = r * dt, E1 = E2 * E2, TT = 2.0 * T * T, S3 = om * (3.0 - E2);
        const Real bF = TT * S3 * idt - 2.0 * T * E2 + T * E1 - T;
        const Real bD = 4.0 * (-TT * om2 + T * dt * E2 * om) * idt * idt;
        const Real cF = -T + T * gF, cD = 4.0 * T * T * om2 * idt * idt, dF1 = -T * T * S3 * idt;
        if constexpr (Tape::active) {
            tp.put(TG_AF, bF.v); tp.put(TG_AD, bD.v); tp.put(TG_T, T.v); tp.put(TG_CF, cF.v); tp.put(TG_CD, cD.v); tp.put(TG_BF, dF1.v);
        }
        // derivatives by r: (r^2 S3)' = r (gF + r S3')..., S3' = -2 E2' (2 - E2), r E2' = hE
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const Real d = dg[i] - c0[i];
            F[i] = (c0[i] + gF * d + bF * (c1[i] - g1[i]) - T * g1[i] + cF * c2[i] + dF1 * g2[i]).v;
            dF[i] = (c2[i] + gD * d + bD * (c1[i] - g1[i]) + cD * (g2[i] - c2[i])).v;
            if constexpr (Tape::active) {
                const Real rS = fma(-2.0 * hE, 2.0 - E2, 2.0 * S3);            // (r^2 S3)' / r
                const Real bFr = dt * (2.0 * r * rS - 2.0 * (E2 + hE) + E1 + 2.0 * hE * E2 - 1.0);
                const Real oo = 2.0 * rom * (om - hE);                          // (r^2 om^2)'
                const Real bDr = 4.0 * (-2.0 * oo + E2 * om + hE * (om - E2));
                const Real cFr = dt * (-1.0 + gF + r * gFr), cDr = 4.0 * oo, dFr = -dt * (r * rS);
                tp.put(TG_FR + i, (gFr * d + bFr * (c1[i] - g1[i]) - dt * g1[i] + cFr * c2[i] + dFr * g2[i]).v);
                tp.put(TG_DFR + i, (gDr * d + bDr * (c1[i] - g1[i]) + cDr * (g2[i] - c2[i])).v);
            }
        }
        return;
    }
    if constexpr (Tape::active) { tp.put(TG_AF, aF.v); tp.put(TG_AD, aD.v); }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const Real d = dg[i] - c0[i], e = c1[i] - g1[i];
        F[i] = fma(gF, d, fma(aF, e, c0[i])).v;
        dF[i] = fma(gD, d, fma(aD, e, c2[i])).v;
        if constexpr (Tape::active) {
            tp.put(TG_FR + i, fma(gFr, d, aFr * e).v);
            tp.put(TG_DFR + i, fma(gDr, d, aDr * e).v);
        }
    }
}

DFK_HD void gks_flux(const GPState& L, const GPState& R, double dt, const SchemeConsts& S, double F[4], double dF[4]) {
    gks_flux_sides(L, R, side_state(L.W, S), side_state(R.W, S), dt, S, F, dF, NoTape{});
}

// ------------------------------------------------------------------------------------------
// Lax-Friedrichs flux (Sect. 2.3) and its time derivative with frozen wave speed and
// W_t = -(A W_n + B W_t) on each side (Cauchy-Kovalevskaya)
// ------------------------------------------------------------------------------------------
// W_t from the primitive time derivative; 1/(gamma - 1) = (K + 2)/2
DFK_HD void lf_time(const FlowState& s, const FlowGrad& t, const SchemeConsts& S, Real T[4]) {
    T[0] = t.r0;
    T[1] = fma(s.U, t.r0, t.r1);
    T[2] = fma(s.V, t.r0, t.r2);
    T[3] = fma(0.5 * (S.K + 2.0), t.dp, fma(s.hq, t.r0, fma(s.U, t.r1, s.V * t.r2)));
}

// c = c^2 / c; zero at zero pressure, where 1/c is infinite
DFK_HD Real sound_speed(const FlowState& s, const SchemeConsts& S) {
    const Real c = (S.gamma * s.th) * (S.r2g * s.rs);
    return (dbits(s.th.v) << 1) == 0 ? Real(0.0) : c;
}

// One side's flux (F) and, unless VALUES, W_t (T) and the flux's derivative along it (D), in gradient form as
// the GKS flux: primitive gradients, the Euler equations' time derivative, back to conserved variables.
// sl, sr: side_state of L.W and R.W, which the DF factor shares
template <bool VALUES>
DFK_HD Real lf_side(const FlowState& s, const GPState& P, const SchemeConsts& S, Real F[4], Real T[4], Real D[4]) {
    const Real m = Real::raw(P.W[1]), E = Real::raw(P.W[3]), Ep = E + s.p;
    F[0] = m;
    F[1] = fma(m, s.U, s.p);
    F[2] = m * s.V;
    F[3] = s.U * Ep;
    if constexpr (!VALUES) {
        const FlowGrad t = euler_time_grad(s, point_grad(s, P.Wn, S), point_grad(s, P.Wt, S), S);
        lf_time(s, t, S, T);
        D[0] = T[1];
        D[1] = fma(s.U, T[1] + t.r1, t.dp);
        D[2] = fma(s.V, T[1], s.U * t.r2);
        D[3] = fma(Ep * s.ir, t.r1, s.U * (T[3] + t.dp));
    }
    return fabs(s.U) + sound_speed(s, S);
}
// VALUES: F alone (the Runge-Kutta stages use no time derivative); the slopes are not read
template <bool VALUES>
DFK_HD void lf_flux_sides(const GPState& L, const GPState& R, const FlowState& sl, const FlowState& sr, const SchemeConsts& S,
                          double F[4], double dF[4]) {
    Real Fl[4], Tl[4], Dl[4], Fr[4], Tr[4], Dr[4];
    const Real al = lf_side<VALUES>(sl, L, S, Fl, Tl, Dl), ar = lf_side<VALUES>(sr, R, S, Fr, Tr, Dr);
    const Real h = 0.5 * nn_max(al, ar);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        F[i] = fma(0.5, Fl[i] + Fr[i], -h * (Real::raw(R.W[i]) - Real::raw(L.W[i]))).v;
        if constexpr (!VALUES) dF[i] = fma(0.5, Dl[i] + Dr[i], -h * (Tr[i] - Tl[i])).v;
    }
}

DFK_HD void lf_flux(const GPState& L, const GPState& R, const SchemeConsts& S, double F[4], double dF[4]) {
    lf_flux_sides<false>(L, R, side_state(L.W, S), side_state(R.W, S), S, F, dF);
}

// DF factor (Sect. 3.2, Eq. 33) of a face's two cell averages in its local frame (df_states = 1), from their
// Maxwellians (maxw_pair): reciprocal square roots for the sound speeds, one division at the end
DFK_HD double df_alpha_maxw(const Maxw& l, const Maxw& r, const SchemeConsts& S) {
    // 1/c = sqrt(rho / (gamma p)) = sqrt(2/gamma) lambda / sqrt(lambda) on each side
    const double icl = S.r2g * (0.5 * l.tl) * l.isl, icr = S.r2g * (0.5 * r.tl) * r.isl;
    const double dn = l.U * icl - r.U * icr, dtg = l.V * icl - r.V * icr;
    // |p_l - p_r| (p_l + p_r) / (p_l p_r) = |p_l - p_r| (1/p_l + 1/p_r), 1/p = (rho/p) (1/rho)
    const double D = fabs(l.p - r.p) * (l.tl * l.ir + r.tl * r.ir) + dn * dn + dtg * dtg;
    return 1.0 / (1.0 + D * D);
}

DFK_HD double df_alpha(const double WL[4], const double WR[4], const SchemeConsts& S) {
    Maxw l, r;
    maxw_pair(WL, WR, S, l, r);
    return df_alpha_maxw(l, r, S);
}

// 0 < x <= +inf on the bit pattern (false for negatives, zeros and NaN)
DFK_HD bool positive_bits(double x) { const long long b = dbits(x); return b > 0 && b <= 0x7FF0000000000000LL; }

DFK_HD bool physical_state(const double W[4], double gm1) {
    if (!positive_bits(W[0])) return false;
    // p > 0 tested as rho p = (gamma - 1) (rho E - |rho u|^2 / 2) > 0: the same sign for rho > 0,
    // without a division
    double rp = gm1 * (W[0] * W[3] - 0.5 * (W[1] * W[1] + W[2] * W[2]));
    return positive_bits(rp);
}

}  // namespace dfk

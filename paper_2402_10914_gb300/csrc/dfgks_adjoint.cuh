// dfgks_adjoint.cuh -- hand-written reverse (vector-Jacobian) products of the building blocks in
// dfgks_device.cuh.  Each *_vjp routine recomputes what it needs of its forward counterpart and
// accumulates (+=) adjoints into its inputs.  Branch decisions (DF switch, fallback, the sign of
// |.|, the arguments selected by min/max) are those of the forward values; at an exact tie the
// derivative of the first argument is taken, and |x| has slope +1 at x = 0.
#pragma once
#include "dfgks_device.cuh"

namespace dfk {

// ------------------------------------------------------------------------------------------
// Characteristic basis
// ------------------------------------------------------------------------------------------
struct BasisBar { double u, v, c, ic, H, b1, b2, q2; };

DFK_HD void basis_bar_zero(BasisBar& b) { b.u = b.v = b.c = b.ic = b.H = b.b1 = b.b2 = b.q2 = 0.0; }

// adjoint of make_basis: accumulates into Wlb, Wrb (the two cell states)
DFK_HD void make_basis_vjp(const double Wl[4], const double Wr[4], const SchemeConsts& S, const BasisBar& Bb,
                           double Wlb[4], double Wrb[4]) {
    double r = 0.5 * (Wl[0] + Wr[0]), m = 0.5 * (Wl[1] + Wr[1]);
    double n = 0.5 * (Wl[2] + Wr[2]), E = 0.5 * (Wl[3] + Wr[3]);
    double ir = 1.0 / r, u = m * ir, v = n * ir, q2 = 0.5 * (u * u + v * v);
    double p = S.gm1 * (E - r * q2);
    double c = sqrt(S.gamma * p * ir), ic = 1.0 / c, H = (E + p) * ir, b1 = S.gm1 * ic * ic;
    double b1b = Bb.b1 + Bb.b2 * q2;
    double q2b = Bb.q2 + Bb.b2 * b1;
    double icb = Bb.ic + b1b * S.gm1 * 2.0 * ic;
    double cb = Bb.c - icb * ic * ic;
    double Eb = Bb.H * ir, pb = Bb.H * ir, irb = Bb.H * (E + p);
    double sb = cb * 0.5 / c;
    pb += sb * S.gamma * ir;
    irb += sb * S.gamma * p;
    Eb += pb * S.gm1;
    double rb = -pb * S.gm1 * q2;
    q2b += -pb * S.gm1 * r;
    double ub = Bb.u + q2b * u, vb = Bb.v + q2b * v;
    double mb = ub * ir, nb = vb * ir;
    irb += ub * m + vb * n;
    rb += -irb * ir * ir;
    const double g[4] = {rb, mb, nb, Eb};
    for (int k = 0; k < 4; ++k) { Wlb[k] += 0.5 * g[k]; Wrb[k] += 0.5 * g[k]; }
}

// adjoint of project (Q = L W): Wb += L^T Qb, basis adjoint accumulated
DFK_HD void project_vjp(const CharBasis& B, const double W[4], const double Qb[4], double Wb[4], BasisBar& Bb) {
    double kb = 0.5 * Qb[0] - Qb[1] + 0.5 * Qb[3];
    double mmb = 0.5 * Qb[0] - 0.5 * Qb[3];
    Wb[0] += Qb[1] - B.v * Qb[2];
    Bb.v += -Qb[2] * W[0];
    Wb[2] += Qb[2];
    // mm = (u W0 - W1) ic
    Bb.u += mmb * B.ic * W[0];
    Wb[0] += mmb * B.ic * B.u;
    Wb[1] += -mmb * B.ic;
    Bb.ic += mmb * (B.u * W[0] - W[1]);
    // k = b2 W0 - t
    Bb.b2 += kb * W[0];
    Wb[0] += kb * B.b2;
    double tb = -kb;
    // t = b1 (u W1 + v W2 - W3)
    Bb.b1 += tb * (B.u * W[1] + B.v * W[2] - W[3]);
    Bb.u += tb * B.b1 * W[1];
    Wb[1] += tb * B.b1 * B.u;
    Bb.v += tb * B.b1 * W[2];
    Wb[2] += tb * B.b1 * B.v;
    Wb[3] += -tb * B.b1;
}

// the two halves of the adjoint of back_project (W = R Q): Qb += R^T Wb, which does not depend on
// Q, and the basis adjoint, which is linear in Q
DFK_HD void back_project_T(const CharBasis& B, const double Wb[4], double Qb[4]) {
    double W0b = Wb[0] + Wb[2] * B.v + Wb[1] * B.u;
    double sb = Wb[3] * B.H + W0b, db = Wb[3] * B.u * B.c + Wb[1] * B.c;
    Qb[1] += Wb[3] * B.q2 + W0b;
    Qb[2] += Wb[3] * B.v + Wb[2];
    Qb[0] += sb - db;
    Qb[3] += sb + db;
}

DFK_HD void back_project_basis_vjp(const CharBasis& B, const double Q[4], const double Wb[4], BasisBar& Bb) {
    double s = Q[0] + Q[3], d = Q[3] - Q[0];
    double W0 = s + Q[1];
    Bb.H += Wb[3] * s;
    Bb.u += Wb[3] * B.c * d + Wb[1] * W0;
    Bb.c += Wb[3] * B.u * d + Wb[1] * d;
    Bb.q2 += Wb[3] * Q[1];
    Bb.v += Wb[3] * Q[2] + Wb[2] * W0;
}

// adjoint of back_project (W = R Q): Qb += R^T Wb, basis adjoint accumulated
DFK_HD void back_project_vjp(const CharBasis& B, const double Q[4], const double Wb[4], double Qb[4], BasisBar& Bb) {
    double s = Q[0] + Q[3], d = Q[3] - Q[0];
    double W0 = s + Q[1];
    double sb = 0.0, db = 0.0;
    // W3 = H s + u c d + q2 Q1 + v Q2
    Bb.H += Wb[3] * s;
    sb += Wb[3] * B.H;
    Bb.u += Wb[3] * B.c * d;
    Bb.c += Wb[3] * B.u * d;
    db += Wb[3] * B.u * B.c;
    Bb.q2 += Wb[3] * Q[1];
    Qb[1] += Wb[3] * B.q2;
    Bb.v += Wb[3] * Q[2];
    Qb[2] += Wb[3] * B.v;
    // W2 = v W0 + Q2
    Bb.v += Wb[2] * W0;
    Qb[2] += Wb[2];
    // W1 = u W0 + c d
    Bb.u += Wb[1] * W0;
    Bb.c += Wb[1] * d;
    db += Wb[1] * B.c;
    // W0 = s + Q1, with the uses in W1 and W2
    double W0b = Wb[0] + Wb[2] * B.v + Wb[1] * B.u;
    sb += W0b;
    Qb[1] += W0b;
    Qb[0] += sb - db;
    Qb[3] += sb + db;
}

// ------------------------------------------------------------------------------------------
// WENO-AO(5,3) and the DF quadratic
// ------------------------------------------------------------------------------------------
struct AOBar { double A1, A2, c3a3, c3a4, rmax, rmin; };

DFK_HD void ao_bar_zero(AOBar& b) { b.A1 = b.A2 = b.c3a3 = b.c3a4 = b.rmax = b.rmin = 0.0; }

// The outputs of a taped WENO-AO reconstruction (weno_ao_t), rebuilt from its tape
template <class Tape>
DFK_HD AO ao_from_tape(const Tape& tp, int base, const SchemeConsts& S) {
    const double iw = tp.get(base + AT_IW), c3 = tp.get(base + AT_C3);
    const double c0 = tp.get(base + AT_W) * iw - c3 * S.d[0], c1 = tp.get(base + AT_W + 1) * iw - c3 * S.d[1];
    const double c2 = tp.get(base + AT_W + 2) * iw - c3 * S.d[2];
    AO o;
    o.A1 = c0 * tp.get(base + AT_A1) + c1 * tp.get(base + AT_A1 + 1) + c2 * tp.get(base + AT_A1 + 2) + c3 * tp.get(base + AT_A1 + 3);
    o.A2 = c0 * tp.get(base + AT_A2) + c1 * tp.get(base + AT_A2 + 1) + c2 * tp.get(base + AT_A2 + 2) + c3 * tp.get(base + AT_A2 + 3);
    o.c3a3 = c3 * tp.get(base + AT_A3);
    o.c3a4 = c3 * tp.get(base + AT_A4);
    o.rmax = tp.get(base + AT_R + (int)tp.get(base + AT_KMAX));
    o.rmin = tp.get(base + AT_R + (int)tp.get(base + AT_KMIN));
    o.rs = 1.0;
    return o;
}

// reverse of weno_ao_t from its tape: qb += (d AO / d q)^T ob
template <class Tape>
DFK_HD void weno_ao_rev(const Tape& tp, int base, const SchemeConsts& S, const AOBar& ob, double qb[5]) {
    const double c13_3 = 13.0 / 3.0;
    double a1[4], a2[4], w[4], r[4], ie[4];
    for (int k = 0; k < 4; ++k) {
        a1[k] = tp.get(base + AT_A1 + k); a2[k] = tp.get(base + AT_A2 + k);
        w[k] = tp.get(base + AT_W + k); r[k] = tp.get(base + AT_R + k); ie[k] = tp.get(base + AT_IE + k);
    }
    const double a3 = tp.get(base + AT_A3), a4 = tp.get(base + AT_A4), iw = tp.get(base + AT_IW), c3 = tp.get(base + AT_C3);
    double c[4];
    for (int k = 0; k < 3; ++k) c[k] = w[k] * iw - c3 * S.d[k];
    c[3] = c3;
    double a1b[4], a2b[4], cb[4];
    for (int k = 0; k < 4; ++k) { a1b[k] = ob.A1 * c[k]; a2b[k] = ob.A2 * c[k]; cb[k] = ob.A1 * a1[k] + ob.A2 * a2[k]; }
    cb[3] += ob.c3a3 * a3 + ob.c3a4 * a4;
    double a3b = ob.c3a3 * c3, a4b = ob.c3a4 * c3;
    double wb[4], iwb = 0.0;
    for (int k = 0; k < 3; ++k) { wb[k] = cb[k] * iw; iwb += cb[k] * w[k]; cb[3] -= cb[k] * S.d[k]; }
    wb[3] = cb[3] * iw * S.inv_d3;
    iwb += cb[3] * w[3] * S.inv_d3;
    const double sumb = -iwb * iw * iw;
    double rb[4];
    for (int k = 0; k < 4; ++k) rb[k] = (wb[k] + sumb) * S.d[k] * 2.0 * r[k];
    rb[(int)tp.get(base + AT_KMAX)] += ob.rmax;
    rb[(int)tp.get(base + AT_KMIN)] += ob.rmin;
    double taub = 0.0, bb[4];
    for (int k = 0; k < 4; ++k) { double t = rb[k] * ie[k]; taub += t; bb[k] = -t * r[k]; }
    const double tb3 = taub * (1.0 / 3.0);
    for (int k = 0; k < 3; ++k) { const double sg = tp.get(base + AT_SG + k); bb[3] += tb3 * sg; bb[k] -= tb3 * sg; }
    for (int k = 0; k < 3; ++k) { a1b[k] += bb[k] * 2.0 * a1[k]; a2b[k] += bb[k] * 2.0 * c13_3 * a2[k]; }
    a1b[3] += bb[3] * (2.0 * a1[3] + 0.5 * a3);
    a3b += bb[3] * (0.5 * a1[3] + 2.0 * (3129.0 / 80.0) * a3);
    a2b[3] += bb[3] * (2.0 * c13_3 * a2[3] + (21.0 / 5.0) * a4);
    a4b += bb[3] * ((21.0 / 5.0) * a2[3] + 2.0 * (87617.0 / 140.0) * a4);
    qb[0] += 0.5 * a1b[0] + 0.5 * a2b[0] + (5.0 / 48.0) * a1b[3] - (1.0 / 16.0) * a2b[3] - (1.0 / 12.0) * a3b + (1.0 / 24.0) * a4b;
    qb[1] += -2.0 * a1b[0] - a2b[0] - 0.5 * a1b[1] + 0.5 * a2b[1] - (34.0 / 48.0) * a1b[3] + (12.0 / 16.0) * a2b[3]
           + (2.0 / 12.0) * a3b - (4.0 / 24.0) * a4b;
    qb[2] += 1.5 * a1b[0] + 0.5 * a2b[0] - a2b[1] - 1.5 * a1b[2] + 0.5 * a2b[2] - (22.0 / 16.0) * a2b[3] + (6.0 / 24.0) * a4b;
    qb[3] += 0.5 * a1b[1] + 0.5 * a2b[1] + 2.0 * a1b[2] - a2b[2] + (34.0 / 48.0) * a1b[3] + (12.0 / 16.0) * a2b[3]
           - (2.0 / 12.0) * a3b - (4.0 / 24.0) * a4b;
    qb[4] += -0.5 * a1b[2] + 0.5 * a2b[2] - (5.0 / 48.0) * a1b[3] - (1.0 / 16.0) * a2b[3] + (1.0 / 12.0) * a3b + (1.0 / 24.0) * a4b;
}

// o from a taped reconstruction (ratios unscaled, o.rs = 1)
DFK_HD void limiter_alpha_vjp(const AO& o, double outb, AOBar& ob) {
    double a1 = 1.0 + o.rmax * o.rmax, a2 = 1.0 + o.rmin * o.rmin, D = a1 + a2;
    ob.rmax += outb * (-2.0 * a2 / (D * D)) * 2.0 * o.rmax;
    ob.rmin += outb * (2.0 * a1 / (D * D)) * 2.0 * o.rmin;
}

DFK_HD void ao_at_right_edge_vjp(double valb, double slopeb, double& q0b, AOBar& ob) {
    q0b += valb;
    ob.A1 += 0.5 * valb + slopeb;
    ob.A2 += (1.0 / 6.0) * valb + slopeb;
    ob.c3a3 += 0.125 * valb + 0.75 * slopeb;
    ob.c3a4 += 0.05 * valb + 0.5 * slopeb;
}

DFK_HD void ao_at_gauss_vjp(const double valb[2], const double slopeb[2], double& q0b, AOBar& ob) {
    const double g = kGaussEta;
    double Eb = valb[0] + valb[1], Ob = valb[1] - valb[0], Esb = slopeb[0] + slopeb[1], Osb = slopeb[1] - slopeb[0];
    q0b += Eb;
    ob.c3a4 += -(1.0 / 180.0) * Eb + g * (1.0 / 3.0) * Osb;
    ob.A1 += g * Ob + Esb;
    ob.c3a3 += g * (1.0 / 12.0) * Ob + 0.25 * Esb;
    ob.A2 += 2.0 * g * Osb;
}

// a1 = (q3 - q1)/2, a2 = (q1 - 2 q2 + q3)/2 of the DF quadratic
DFK_HD void df_coeffs_vjp(double a1b, double a2b, double qb[5]) {
    qb[3] += 0.5 * a1b + 0.5 * a2b;
    qb[1] += -0.5 * a1b + 0.5 * a2b;
    qb[2] += -a2b;
}

DFK_HD void df_at_right_edge_vjp(double alpha, double valb, double slopeb, double qb[5]) {
    qb[2] += valb;
    df_coeffs_vjp(alpha * (0.5 * valb + slopeb), alpha * ((1.0 / 6.0) * valb + slopeb), qb);
}

DFK_HD void df_at_gauss_vjp(double alpha, const double valb[2], const double slopeb[2], double qb[5]) {
    const double g = kGaussEta;
    qb[2] += valb[0] + valb[1];
    double Ob = valb[1] - valb[0], Esb = slopeb[0] + slopeb[1], Osb = slopeb[1] - slopeb[0];
    df_coeffs_vjp(alpha * g * Ob + alpha * Esb, 2.0 * alpha * g * Osb, qb);
}

// ------------------------------------------------------------------------------------------
// GKS flux: reverse of the gradient form
//
// The moments' own derivatives are e1 and e2, and the marginal distribution g = phi at u = 0, a Gaussian in U of
// variance theta, obeys the heat equation dg/dtheta = g''/2, as every moment does.  So the adjoints of a side's
// m_0 .. m_4, phi and e2_0 go straight to U and theta,
//   U^ = sum m_k^ e1_k + 2 phi^ e2_0 + e2_0^ psi,  theta^ = sum m_k^ e2_k + phi^ psi + e2_0^ e2_0 (U^2/theta - 3)/(2 theta),
//   e2_0 = -phi U/(2 theta),  psi = dphi/dtheta = phi (U^2/theta - 1)/(2 theta),
// without going back through the recurrences, the Gaussian and the error function.  Bound by the FP64 units
// like the forward; the reverse of the flux written with slope coefficients took 2343 FP64 instructions per
// Gauss point, a tape of 172 values and that form's forward (1028 instructions).  10-step gradient on 256 x 256
// 72.9 -> 53.1 ms, reverse of a 67 x 83 stage 0.775 -> 0.620 ms (that one also reads a tape now).
// ------------------------------------------------------------------------------------------
struct GPStateBar { double W[4], Wn[4], Wt[4]; };
struct FlowBar { Real rho, U, V, p, th, hq; };
struct GradBar { Real r0, r1, r2, q3, dp; };

DFK_HD void zero(FlowBar& b) { b.rho = b.U = b.V = b.p = b.th = b.hq = 0.0; }
DFK_HD void zero(GradBar& b) { b.r0 = b.r1 = b.r2 = b.q3 = b.dp = 0.0; }

template <class Tape>
DFK_HD Real tape_real(const Tape& tp, int i) { return Real::raw(tp.get(i)); }

// a state of which 1/rho is known
DFK_HD FlowState flow_state_again(const Real W[4], Real ir, const SchemeConsts& S) {
    FlowState s;
    s.rho = W[0];
    s.ir = ir;
    s.U = W[1] * ir;
    s.V = W[2] * ir;
    s.hq = 0.5 * fma(s.U, s.U, s.V * s.V);
    s.p = S.gm1 * fma(-W[0], s.hq, W[3]);
    s.th = s.p * ir;
    return s;
}

// flow_state's reverse: the state adjoint to that of the conserved variables
DFK_HD void flow_state_rev(const FlowState& s, const FlowBar& b, const SchemeConsts& S, Real Wb[4]) {
    const Real pb = fma(b.th, s.ir, b.p), z = S.gm1 * pb, hqb = fma(-z, s.rho, b.hq);
    const Real Ub = fma(hqb, s.U, b.U), Vb = fma(hqb, s.V, b.V);
    Wb[0] = fma(-z, s.hq, fma(-s.ir, fma(b.th, s.th, fma(Ub, s.U, Vb * s.V)), b.rho));
    Wb[1] = Ub * s.ir;
    Wb[2] = Vb * s.ir;
    Wb[3] = z;
}

// flow_grad's reverse: a gradient's adjoint to that of the conserved gradient and of the state
DFK_HD void flow_grad_rev(const FlowState& s, const Real d0, const FlowGrad& g, const GradBar& b, const SchemeConsts& S,
                          Real db[4], FlowBar& sb) {
    const Real z = S.gm1 * (b.dp + b.q3);
    const Real r1b = fma(-s.U, z, b.r1), r2b = fma(-s.V, z, b.r2);
    sb.th = fma(-d0, b.q3, sb.th);
    sb.hq = fma(-d0, z, sb.hq);
    sb.U = fma(-g.r1, z, fma(-d0, r1b, sb.U));
    sb.V = fma(-g.r2, z, fma(-d0, r2b, sb.V));
    db[0] = fma(-s.th, b.q3, fma(-s.hq, z, fma(-s.U, r1b, fma(-s.V, r2b, b.r0))));
    db[1] = r1b;
    db[2] = r2b;
    db[3] = z;
}

// to_lab's reverse: the laboratory frame's adjoint b to the own frame's (a); w0, w2 are the own frame's values
DFK_HD void to_lab_rev(Real V, Real hV2, const Real b[4], Real w0, Real w2, Real a[4], Real& Vb) {
    Vb = fma(b[2], w0, fma(b[3], fma(V, w0, w2), Vb));
    a[0] = fma(hV2, b[3], fma(V, b[2], b[0]));
    a[1] = b[1];
    a[2] = fma(V, b[3], b[2]);
    a[3] = b[3];
}

// adjoints of m_0 .. m_4, phi and e2_0
struct MomAdj { Real m[5], phi, e; };

// reverse of N_k = r0 m_k + r1 e1_k + q3 e2_k for k = LO .. HI, the adjoints being Nb[k - LO]
template <int LO, int HI>
DFK_HD void grad_mom_rev(const HalfMom& h, const FlowGrad& g, const Real* Nb, GradBar& b, MomAdj& mb) {
#pragma unroll
    for (int k = LO; k <= HI; ++k) {
        const Real n = Nb[k - LO];
        b.r0 = fma(n, h.m[k], b.r0);
        b.r1 = fma(n, h.e1[k], b.r1);
        b.q3 = fma(n, h.e2[k], b.q3);
        mb.m[k] = fma(n, g.r0, mb.m[k]);
        const Real n1 = n * g.r1, n3 = n * g.q3;
        if (k == 0) { mb.phi = mb.phi + n1; mb.e = mb.e + n3; }
        if (k >= 1) mb.m[k - 1] = fma((double)k, n1, mb.m[k - 1]);
        if (k == 1) mb.phi = fma(0.5, n3, mb.phi);
        if (k >= 2) mb.m[k - 2] = fma(0.5 * k * (k - 1), n3, mb.m[k - 2]);
    }
}

// reverse of transport (own-frame adjoints a): the adjoints of N_2 .. N_4 of x are set, those of N_1 .. N_3 of y
// set, the rest accumulated.  Nx[0] = N_2 of x, Ny[j] = N_{1+j} of y
DFK_HD void transport_rev(const FlowState& s, const HalfMom& h, const FlowGrad& x, const FlowGrad& y, Real Nx0,
                          const Real Ny[3], Real k1, Real k3, const Real a[4], Real Nxb[3], Real Nyb[3], GradBar& xb,
                          GradBar& yb, MomAdj& mb, FlowBar& sb) {
    const Real ka = k1 * a[3], ha = 0.5 * a[3], kt = k3 * s.th;
    const Real v1 = y.r2 * h.m[1], G1 = fma(s.th, Ny[0], y.q3 * h.m[1]);
    const Real v1b = fma(kt, a[3], fma(s.V, a[2], a[0])), G1b = fma(s.V, ka, a[2]);
    Nxb[0] = fma(s.th, ka, a[0]);
    Nxb[1] = a[1];
    Nxb[2] = ha;
    Nyb[0] = fma(s.V, a[0], s.th * G1b);
    Nyb[1] = s.V * a[1];
    Nyb[2] = s.V * ha;
    xb.r2 = fma(a[2], h.m[2], xb.r2);
    xb.q3 = fma(ka, h.m[2], xb.q3);
    yb.r2 = fma(v1b, h.m[1], fma(a[1], h.m[2], fma(ha, h.m[3], yb.r2)));
    yb.q3 = fma(G1b, h.m[1], yb.q3);
    mb.m[1] = fma(v1b, y.r2, fma(G1b, y.q3, mb.m[1]));
    mb.m[2] = fma(a[2], x.r2, fma(ka, x.q3, fma(a[1], y.r2, mb.m[2])));
    mb.m[3] = fma(ha, y.r2, mb.m[3]);
    sb.V = fma(a[0], Ny[0], fma(a[1], Ny[1], fma(ha, Ny[2], fma(a[2], v1, fma(ka, G1, sb.V)))));
    sb.th = fma(k3 * v1, a[3], fma(ka, Nx0, fma(G1b, Ny[0], sb.th)));
}

// euler_time_grad's reverse: t's adjoint (q3 included) to those of the gradients and the state
DFK_HD void euler_time_grad_rev(const FlowState& s, const FlowGrad& x, const FlowGrad& y, const FlowGrad& t, const GradBar& tb,
                                const SchemeConsts& S, GradBar& xb, GradBar& yb, FlowBar& sb) {
    sb.th = fma(-t.r0, tb.q3, sb.th);
    const Real s0 = fma(s.th, tb.q3, -tb.r0), s1 = -tb.r1, s2 = -tb.r2, s3 = -(tb.dp + tb.q3);
    const Real gs = S.gamma * s3, div = x.r1 + y.r2, divb = fma(gs, s.th, s0);
    sb.th = fma(gs, div, sb.th);
    sb.U = fma(x.r0, s0, fma(x.r1, s1, fma(x.r2, s2, fma(x.dp, s3, sb.U))));
    sb.V = fma(y.r0, s0, fma(y.r1, s1, fma(y.r2, s2, fma(y.dp, s3, sb.V))));
    xb.r0 = fma(s.U, s0, xb.r0); yb.r0 = fma(s.V, s0, yb.r0);
    xb.r1 = fma(s.U, s1, xb.r1 + divb); yb.r1 = fma(s.V, s1, yb.r1);
    xb.r2 = fma(s.U, s2, xb.r2); yb.r2 = fma(s.V, s2, yb.r2 + divb);
    xb.dp = fma(s.U, s3, xb.dp + s1); yb.dp = fma(s.V, s3, yb.dp + s2);
}

// one side (SIGN +1 left, -1 right) from the adjoints of its sums (the equilibrium state, its gradients, dg, g1,
// g2) and of its pressure through tau_n
template <int SIGN, class Tape>
DFK_HD void gks_side_reverse(const Tape& tp, const GPState& P, const SchemeConsts& S, const Real Wcb[4], const Real Wcxb[4],
                             const Real Wcyb[4], const Real g0b[4], const Real g1b[4], const Real g2b[4], Real pb,
                             GPStateBar& Pb) {
    constexpr int base = SIGN > 0 ? TG_L : TG_R;
    const Real k1 = 0.5 * (S.K + 1.0), k3 = 0.5 * (S.K + 3.0);
    const Real W[4] = {Real::raw(P.W[0]), Real::raw(P.W[1]), Real::raw(P.W[2]), Real::raw(P.W[3])};
    const FlowState s = flow_state_again(W, tape_real(tp, base), S);
    const FlowGrad x = point_grad(s, P.Wn, S), y = point_grad(s, P.Wt, S);
    const Real i2th = tape_real(tp, base + 3);
    HalfMom h;
    h.m[0] = tape_real(tp, base + 1);
    h.e1[0] = tape_real(tp, base + 2);                    // phi
    h.m[1] = fma(s.U, h.m[0], s.th * h.e1[0]);
    h.e2[0] = -(h.e1[0] * s.U) * i2th;
    h.e2[1] = 0.5 * h.e1[0];
    finish_moments(s, h);
    FlowBar sb;
    zero(sb);
    sb.p = pb;
    MomAdj mb;
    GradBar xb, yb;
    zero(xb);
    zero(yb);
    const Real hV2 = 0.5 * s.V * s.V, kth = k1 * s.th;
    // c = rho <psi> and dg = rho <u psi>
    {
        Real a[4], b[4];
        to_lab_rev(s.V, hV2, Wcb, s.rho * h.m[0], 0.0, a, sb.V);
        to_lab_rev(s.V, hV2, g0b, s.rho * h.m[1], 0.0, b, sb.V);
        const Real A0 = fma(kth, a[3], a[0]), A1 = fma(kth, b[3], a[1] + b[0]), A2 = fma(0.5, a[3], b[1]), A3 = 0.5 * b[3];
        sb.rho = fma(A0, h.m[0], fma(A1, h.m[1], fma(A2, h.m[2], A3 * h.m[3])));
        sb.th = (k1 * s.rho) * fma(h.m[0], a[3], h.m[1] * b[3]);
        mb.m[0] = s.rho * A0; mb.m[1] = s.rho * A1; mb.m[2] = s.rho * A2; mb.m[3] = s.rho * A3;
        mb.m[4] = 0.0; mb.phi = 0.0; mb.e = 0.0;
    }
    // the two gradients' sums and their transport
    const Real Nx0 = grad_mom(h, x, 0), Nx2 = grad_mom(h, x, 2), Ny0 = grad_mom(h, y, 0);
    const Real Ny[3] = {grad_mom(h, y, 1), grad_mom(h, y, 2), grad_mom(h, y, 3)};
    Real Nxb[5], Nyb[4];
    {
        Real a[4];
        const Real v1 = y.r2 * h.m[1];
        const Real o0 = fma(s.V, Ny[0], Nx2) + v1, o2 = fma(s.V, v1, fma(x.r2, h.m[2], fma(s.th, Ny[0], y.q3 * h.m[1])));
        to_lab_rev(s.V, hV2, g1b, o0, o2, a, sb.V);
        transport_rev(s, h, x, y, Nx2, Ny, k1, k3, a, Nxb + 2, Nyb + 1, xb, yb, mb, sb);
    }
    {
        Real a[4];
        const Real p = x.r2 * h.m[0];
        to_lab_rev(s.V, hV2, Wcxb, Nx0, p, a, sb.V);
        const Real ka = k1 * a[3];
        Nxb[0] = fma(s.th, ka, a[0]);
        Nxb[1] = a[1];
        Nxb[2] = fma(0.5, a[3], Nxb[2]);
        xb.r2 = fma(a[2], h.m[0], xb.r2);
        xb.q3 = fma(ka, h.m[0], xb.q3);
        mb.m[0] = fma(a[2], x.r2, fma(ka, x.q3, mb.m[0]));
        sb.th = fma(ka, Nx0, sb.th);
    }
    {
        Real a[4];
        const Real p = y.r2 * h.m[0];
        to_lab_rev(s.V, hV2, Wcyb, Ny0, p, a, sb.V);
        const Real ka = k1 * a[3];
        Nyb[0] = fma(s.th, ka, a[0]);
        Nyb[1] = Nyb[1] + a[1];
        Nyb[2] = fma(0.5, a[3], Nyb[2]);
        yb.r2 = fma(a[2], h.m[0], yb.r2);
        yb.q3 = fma(ka, h.m[0], yb.q3);
        mb.m[0] = fma(a[2], y.r2, fma(ka, y.q3, mb.m[0]));
        sb.th = fma(ka, Ny0, sb.th);
    }
    grad_mom_rev<0, 4>(h, x, Nxb, xb, mb);
    grad_mom_rev<0, 3>(h, y, Nyb, yb, mb);
    if (S.tau_reading == 1) {                             // g2 = rho <u A psi>
        const FlowGrad t = euler_time_grad(s, x, y, S);
        GradBar tb;
        zero(tb);
        const Real N1 = grad_mom(h, t, 1), p = t.r2 * h.m[1];
        Real a[4], Ntb[3];
        to_lab_rev(s.V, hV2, g2b, N1, p, a, sb.V);
        const Real ka = k1 * a[3];
        Ntb[0] = fma(s.th, ka, a[0]);
        Ntb[1] = a[1];
        Ntb[2] = 0.5 * a[3];
        tb.r2 = a[2] * h.m[1];
        tb.q3 = ka * h.m[1];
        mb.m[1] = fma(a[2], t.r2, fma(ka, t.q3, mb.m[1]));
        sb.th = fma(ka, N1, sb.th);
        grad_mom_rev<1, 3>(h, t, Ntb, tb, mb);
        euler_time_grad_rev(s, x, y, t, tb, S, xb, yb, sb);
    }
    // moments to U and theta
    {
        const Real U2 = 2.0 * (s.U * s.U) * i2th;         // U^2 / theta
        const Real psi = (h.e1[0] * i2th) * (U2 - 1.0);
        Real u = fma(2.0 * mb.phi, h.e2[0], mb.e * psi), th = fma(mb.phi, psi, (mb.e * h.e2[0]) * (i2th * (U2 - 3.0)));
#pragma unroll
        for (int k = 0; k < 5; ++k) { u = fma(mb.m[k], h.e1[k], u); th = fma(mb.m[k], h.e2[k], th); }
        sb.U = sb.U + u;
        sb.th = sb.th + th;
    }
    Real d[4];
    flow_grad_rev(s, x.r0, x, xb, S, d, sb);
#pragma unroll
    for (int i = 0; i < 4; ++i) Pb.Wn[i] = d[i].v;
    flow_grad_rev(s, y.r0, y, yb, S, d, sb);
#pragma unroll
    for (int i = 0; i < 4; ++i) Pb.Wt[i] = d[i].v;
    flow_state_rev(s, sb, S, d);
#pragma unroll
    for (int i = 0; i < 4; ++i) Pb.W[i] = d[i].v;
}

// reverse of the GKS flux from its tape: sets the Gauss-point state adjoints Lb, Rb for the adjoints Fb, dFb
// (local frame) of F and dF
template <class Tape>
DFK_HD void gks_flux_reverse(const Tape& tp, const GPState& L, const GPState& R, const SchemeConsts& S, const double Fbv[4],
                             const double dFbv[4], GPStateBar& Lb, GPStateBar& Rb) {
    const Real k1 = 0.5 * (S.K + 1.0), k3 = 0.5 * (S.K + 3.0);
    // the final combination and tau_n / dt
    Real c0b[4], c1b[4], c2b[4], g0b[4], g1b[4], g2b[4], rTb = 0.0;
    {
        const Real gF = tape_real(tp, TG_GF), gD = tape_real(tp, TG_GD), aF = tape_real(tp, TG_AF), aD = tape_real(tp, TG_AD);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const Real Fb = Real::raw(Fbv[i]), Db = Real::raw(dFbv[i]);
            g0b[i] = fma(Fb, gF, Db * gD);
            c0b[i] = Fb - g0b[i];
            c1b[i] = fma(Fb, aF, Db * aD);
            g1b[i] = -c1b[i];
            c2b[i] = Db;
            rTb = fma(Fb, tape_real(tp, TG_FR + i), fma(Db, tape_real(tp, TG_DFR + i), rTb));
        }
        if (S.tau_reading == 1) {
            const Real T = tape_real(tp, TG_T), cF = tape_real(tp, TG_CF), cD = tape_real(tp, TG_CD), bF = tape_real(tp, TG_BF);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const Real Fb = Real::raw(Fbv[i]), Db = Real::raw(dFbv[i]);
                g1b[i] = fma(-Fb, T, g1b[i]);
                c2b[i] = fma(-Db, cD, fma(Fb, cF, Db));
                g2b[i] = fma(Fb, bF, Db * cD);
            }
        }
    }
    // the equilibrium state
    Real Wcb[4], Wcxb[4], Wcyb[4];
    {
        Real Wc[4], d[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) Wc[i] = tape_real(tp, TG_WC + i);
        const FlowState c = flow_state_again(Wc, tape_real(tp, TG_IRC), S);
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = tape_real(tp, TG_WCX + i);
        const FlowGrad x = flow_grad(c, d, S);
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = tape_real(tp, TG_WCY + i);
        const FlowGrad y = flow_grad(c, d, S);
        const FlowGrad t = euler_time_grad(c, x, y, S);
        HalfMom h;
        h.m[0] = 1.0; h.m[1] = c.U;
        h.e1[0] = 0.0; h.e2[0] = 0.0; h.e2[1] = 0.0;
        finish_moments(c, h);
        const Real hV2 = 0.5 * c.V * c.V, hU2 = 0.5 * c.U * c.U, gg = 0.5 * (S.K + 4.0), ru = Wc[1];
        FlowBar sb;
        zero(sb);
        Real rub, a[4];
        to_lab_rev(c.V, hV2, c0b, ru, 0.0, a, sb.V);
        {
            const Real g3 = gg * a[3];
            rub = fma(hU2, a[3], fma(c.U, a[1], a[0]));
            sb.U = fma(ru, fma(c.U, a[3], a[1]), g3 * c.p);
            sb.p = fma(g3, c.U, a[1]);
        }
        GradBar xb, yb, tb;
        zero(xb); zero(yb); zero(tb);
        const Real n1 = fma(c.U, t.r0, t.r1);
        to_lab_rev(c.V, hV2, c2b, n1, c.U * t.r2, a, sb.V);
        {
            const Real g3 = gg * a[3], U1 = c.U * a[1], H = hU2 * a[3];
            const Real n1b = a[0] + U1 + H;
            tb.r0 = c.U * n1b;
            tb.r1 = fma(2.0, H, U1) + fma(g3, c.th, n1b);
            tb.r2 = c.U * a[2];
            tb.dp = fma(g3, c.U, a[1]);
            sb.U = fma(n1 + t.r1, a[1], fma(t.r2, a[2], fma(c.U * a[3], fma(2.0, t.r1, n1), fma(g3, t.dp, fma(t.r0, n1b, sb.U)))));
            sb.th = fma(g3, t.r1, sb.th);
        }
        euler_time_grad_rev(c, x, y, t, tb, S, xb, yb, sb);
        MomAdj mb;
#pragma unroll
        for (int k = 0; k < 5; ++k) mb.m[k] = 0.0;
        mb.phi = 0.0; mb.e = 0.0;
        const Real Nx2 = grad_mom(h, x, 2), Ny[3] = {fma(c.U, y.r0, y.r1), grad_mom(h, y, 2), grad_mom(h, y, 3)};
        Real Nxb[3], Nyb[3];
        const Real v1 = y.r2 * h.m[1];
        const Real o0 = fma(c.V, Ny[0], Nx2) + v1, o2 = fma(c.V, v1, fma(x.r2, h.m[2], fma(c.th, Ny[0], y.q3 * h.m[1])));
        to_lab_rev(c.V, hV2, c1b, o0, o2, a, sb.V);
        transport_rev(c, h, x, y, Nx2, Ny, k1, k3, a, Nxb, Nyb, xb, yb, mb, sb);
        grad_mom_rev<2, 4>(h, x, Nxb, xb, mb);
        grad_mom_rev<1, 3>(h, y, Nyb, yb, mb);
        sb.U = sb.U + mb.m[1];
#pragma unroll
        for (int k = 2; k < 5; ++k) { sb.U = fma(mb.m[k], h.e1[k], sb.U); sb.th = fma(mb.m[k], h.e2[k], sb.th); }
        flow_grad_rev(c, x.r0, x, xb, S, Wcxb, sb);
        flow_grad_rev(c, y.r0, y, yb, S, Wcyb, sb);
        flow_state_rev(c, sb, S, Wcb);
        Wcb[1] = Wcb[1] + rub;
    }
    gks_side_reverse<+1>(tp, L, S, Wcb, Wcxb, Wcyb, g0b, g1b, g2b, rTb * tape_real(tp, TG_PL), Lb);
    gks_side_reverse<-1>(tp, R, S, Wcb, Wcxb, Wcyb, g0b, g1b, g2b, rTb * tape_real(tp, TG_PR), Rb);
}

// reverse of gks_flux: the forward evaluated again into a local tape, then its reverse; sets Lb, Rb
DFK_HD void gks_flux_vjp(const GPState& L, const GPState& R, double dt, const SchemeConsts& S,
                         const double Fb[4], const double dFb[4], GPStateBar& Lb, GPStateBar& Rb) {
    double t[TG_COUNT], F[4], dF[4];
    ArrayTape tp{t};
    gks_flux_sides(L, R, side_state(L.W, S), side_state(R.W, S), dt, S, F, dF, tp);
    gks_flux_reverse(tp, L, R, S, Fb, dFb, Lb, Rb);
}

// ------------------------------------------------------------------------------------------
// WENO-AO in undivided differences, the reverse of ao_weights and of its evaluations
//
// With z_k = r_k^2 and sum = 1 + sum_k d_k z_k the weights are c_3 = (1 + z_3)/sum, c_0, c_2 = d_0 (z_k - z_3)/sum and
// c_m = c_3 + d_1 (z_1 - z_3)/sum (ao_sum); the differences of one reconstruction are fb, ff, the second ones s0, s1, s2 and the third ones to, ti (outer and
// inner: t1, t2 of the forward for SGN +1, t3, t2 for the mirrored stencil), T = to + ti, U = SGN (ti - to).
// Bound by the FP64 units like the forward.  The sub-stencil polynomials' form (weno_ao_rev above, which stays with
// the other plain statements as what these routines are tested against; no kernel calls it) and a tape of 29 values a reconstruction instead of 6 took, with
// the forward: 400 x 400 L-F stage 5.76 -> 3.93 ms, 67 x 83 GKS stage 0.620 -> 0.483, 10-step GKS gradient on
// 256 x 256 53.1 -> 42.6.
// ------------------------------------------------------------------------------------------
struct AODiffBar { Real fb, ff, s0, s1, s2, a10, a11, a12, to, ti; };

// the weights of a reconstruction (SchemeConsts: d_0 = d_2)
struct AOCoeffs { Real r[4], c0, cm, c2, c3; };
DFK_HD AOCoeffs ao_coeffs(const AORatios& q, const SchemeConsts& S) {
    AOCoeffs c;
#pragma unroll
    for (int k = 0; k < 4; ++k) c.r[k] = q.tau * q.ie[k];
    const Real z3 = c.r[3] * c.r[3];
    c.c3 = fma(z3, q.iv, q.iv);
    const Real di = S.d[0] * q.iv;
    c.c0 = fma(c.r[0], c.r[0], -z3) * di;
    c.c2 = fma(c.r[2], c.r[2], -z3) * di;
    c.cm = fma(S.d[1] * q.iv, fma(c.r[1], c.r[1], -z3), c.c3);
    return c;
}

// four times the adjoints of z_k for those of the weights (the factors 2 of z = r^2 and of the squares in the
// smoothness indicators, once).  As in the forward, each is a difference of terms of its own sub-stencil's size
DFK_HD void ao_coeffs_rev(const AOCoeffs& c, const AORatios& q, Real c0b, Real cmb, Real c2b, Real c3b, const SchemeConsts& S, Real zb[4]) {
    const Real n = fma(c0b, c.c0, fma(cmb, c.cm, fma(c2b, c.c2, c3b * c.c3)));     // minus the sum's adjoint times the sum
    const Real iv = 4.0 * q.iv, di = S.d[0] * iv, em = cmb - n;
    zb[0] = di * (c0b - n);
    zb[1] = (S.d[1] * iv) * em;
    zb[2] = di * (c2b - n);
    zb[3] = iv * fma(S.d[0], fma(2.0, cmb, -(c0b + c2b)), fma(S.d[3], em, c3b));   // 1 - d_1 = 2 d_0 + d_3
}

// the limiter weight 2 (1 + z_min) / ((1 + z_max) + (1 + z_min)): adds to (four times) the adjoints of the z it was made of
// (the first attaining k, as the ratios' order is that of 1/(beta_k + eps))
DFK_HD void ao_limiter_rev(const AORatios& q, const AOCoeffs& c, Real wb, Real zb[4]) {
    int kmax = 0, kmin = 0;
    Real hi = q.ie[0], lo = q.ie[0], rh = c.r[0], rl = c.r[0];
#pragma unroll
    for (int k = 1; k < 4; ++k) {
        if (nn_less(hi, q.ie[k])) { hi = q.ie[k]; kmax = k; rh = c.r[k]; }
        if (nn_less(q.ie[k], lo)) { lo = q.ie[k]; kmin = k; rl = c.r[k]; }
    }
    const Real xh = fma(rh, rh, 1.0), xl = fma(rl, rl, 1.0), den = xh + xl;
    const Real g = wb * Real::raw(8.0 / Real(den * den).v);
    const Real hb = -(g * xl), lb = g * xh;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        zb[k] = zb[k] + (k == kmax ? hb : Real(0.0));
        zb[k] = zb[k] + (k == kmin ? lb : Real(0.0));
    }
}

// four times the adjoints of the z_k, and those of T, U so far, to the differences (b accumulates; b.a10, b.a11, b.a12
// hold the evaluation's share of the adjoints of a10 = fb + SGN s0/2, a11 = fb + SGN s1/2, a12 = ff - SGN s2/2)
template <int SGN>
DFK_HD void ao_ratios_rev(const AORatios& q, const AOCoeffs& c, const Real zb[4], Real s0, Real s1, Real s2, Real a10, Real a11,
                          Real a12, Real T, Real U, Real Tb, Real Ub, AODiffBar& b) {
    // r_k = tau / e_k; eb: twice the adjoints of e_k
    Real eb[4], g[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) { g[k] = zb[k] * c.r[k] * q.ie[k]; eb[k] = -(g[k] * c.r[k]); }
    const Real t3 = (1.0 / 3.0) * ((g[0] + g[1]) + (g[2] + g[3]));       // twice the adjoint of 3 tau
    // 3 tau = sum_k |e_3 - e_k|, the sign that of e_3 - e_k: e_3 >= e_k where 1/e_k >= 1/e_3
    int below = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const bool neg = nn_less(q.ie[k], q.ie[3]);
        below += neg;
        eb[k] = eb[k] - (neg ? -t3 : t3);
    }
    eb[3] = fma(t3, below < 2 ? (below ? Real(1.0) : Real(3.0)) : (below == 2 ? Real(-1.0) : Real(-3.0)), eb[3]);
    const Real h = 0.5 * SGN;
    const Real a10b = fma(eb[0], a10, b.a10), a12b = fma(eb[2], a12, b.a12);
    const Real m1b = eb[3] * fma(-1.0 / 12.0, T, a11), m2b = (13.0 / 12.0) * eb[3] * fma(-11.0 / 130.0, U, s1);
    const Real a11b = fma(eb[1], a11, m1b + b.a11);
    Tb = fma((781.0 / 2880.0) * eb[3], T, fma(-1.0 / 12.0, m1b, Tb));
    Ub = fma((1421461.0 / 1310400.0) * eb[3], U, fma(-11.0 / 130.0, m2b, Ub));
    b.fb = b.fb + (a10b + a11b);
    b.ff = b.ff + a12b;
    b.s0 = fma(h, a10b, fma((13.0 / 12.0) * eb[0], s0, b.s0));
    b.s1 = fma(h, a11b, fma((13.0 / 12.0) * eb[1], s1, b.s1 + m2b));
    b.s2 = fma(-h, a12b, fma((13.0 / 12.0) * eb[2], s2, b.s2));
    b.to = b.to + (SGN > 0 ? Tb - Ub : Tb + Ub);
    b.ti = b.ti + (SGN > 0 ? Tb + Ub : Tb - Ub);
}

// Reverse of project_diff and back_project_diff.  The adjoints of the products in DiffBasis are gathered here
// and folded to the basis in diff_basis_rev.
struct DiffBasisBar { Real b1, b1u, b1v, b2, ic, uic, v, u, hc, hH, huc, q2; };
DFK_HD void zero(DiffBasisBar& b) { b.b1 = b.b1u = b.b1v = b.b2 = b.ic = b.uic = b.v = b.u = b.hc = b.hH = b.huc = b.q2 = 0.0; }

// Wb += L^T Qb
DFK_HD void project_diff_rev(const DiffBasis& D, const Real W[4], const Real Qb[4], Real Wb[4], DiffBasisBar& b) {
    const Real kb = (Qb[0] + Qb[3]) - Qb[1], mb = Qb[0] - Qb[3];
    Wb[0] = fma(D.uic, mb, fma(D.b2, kb, fma(-D.v, Qb[2], Qb[1])));
    Wb[1] = fma(-D.b1u, kb, -(D.ic * mb));
    Wb[2] = fma(-D.b1v, kb, Qb[2]);
    Wb[3] = D.b1 * kb;
    b.b1 = fma(kb, W[3], b.b1);
    b.b1v = fma(-kb, W[2], b.b1v);
    b.b1u = fma(-kb, W[1], b.b1u);
    b.b2 = fma(kb, W[0], b.b2);
    b.uic = fma(mb, W[0], b.uic);
    b.ic = fma(-mb, W[1], b.ic);
    b.v = fma(-Qb[2], W[0], b.v);
}
// Qb = R^T Wb
DFK_HD void back_project_diff_T(const DiffBasis& D, const Real Wb[4], Real Qb[4]) {
    const Real w0 = fma(D.u, Wb[1], fma(D.v, Wb[2], Wb[0]));
    const Real s = fma(D.hH, Wb[3], 0.5 * w0), d = fma(D.huc, Wb[3], D.hc * Wb[1]);
    Qb[0] = s - d;
    Qb[1] = fma(D.q2, Wb[3], w0);
    Qb[2] = fma(D.v, Wb[3], Wb[2]);
    Qb[3] = s + d;
}
DFK_HD void back_project_diff_basis_rev(const Real Q[4], const Real Wb[4], DiffBasisBar& b) {
    const Real s = Q[0] + Q[3], d = Q[3] - Q[0], w0 = fma(0.5, s, Q[1]);
    b.u = fma(Wb[1], w0, b.u);
    b.hc = fma(Wb[1], d, b.hc);
    b.huc = fma(Wb[3], d, b.huc);
    b.hH = fma(Wb[3], s, b.hH);
    b.q2 = fma(Wb[3], Q[1], b.q2);
    b.v = fma(Wb[2], w0, fma(Wb[3], Q[2], b.v));
}
struct BasisAdj { Real u, v, c, ic, H, b1, b2, q2; };
DFK_HD BasisAdj diff_basis_rev(const DiffBasis& D, const DiffBasisBar& b) {
    BasisAdj o;
    o.u = fma(D.b1, b.b1u, fma(D.ic, b.uic, fma(D.hc, b.huc, b.u)));
    o.v = fma(D.b1, b.b1v, b.v);
    o.c = 0.5 * fma(D.u, b.huc, b.hc);
    o.ic = fma(D.u, b.uic, b.ic);
    o.H = 0.5 * b.hH;
    o.b1 = fma(D.u, b.b1u, fma(D.v, b.b1v, b.b1));
    o.b2 = b.b2;
    o.q2 = b.q2;
    return o;
}

// make_basis' reverse: half the adjoint of the mean state (each of the two cells'); r is the mean density.
// c and 1/c are functions of c^2 = gamma p / r
DFK_HD void make_basis_rev(const CharBasis& B, Real r, const BasisAdj& b, const SchemeConsts& S, Real g[4]) {
    const Real u = Real::raw(B.u), v = Real::raw(B.v), c = Real::raw(B.c), ic = Real::raw(B.ic), H = Real::raw(B.H),
               b1 = Real::raw(B.b1), q2 = Real::raw(B.q2);
    const Real ir = rcp_or_div(r);
    const Real b1b = fma(b.b2, q2, b.b1), icb = fma((2.0 * S.gm1) * ic, b1b, b.ic);
    const Real k = 0.5 * fma(-ic * ic, icb, b.c);                       // adjoint of c^2 is k / c
    const Real kg = (k * ic) * ir;
    const Real pb = fma(S.gamma, kg, b.H * ir), Eb = fma(S.gm1, pb, b.H * ir), z = S.gm1 * pb;
    const Real q2b = fma(-z, r, fma(b.b2, b1, b.q2));
    const Real ub = fma(q2b, u, b.u), vb = fma(q2b, v, b.v);
    const Real hr = 0.5 * ir;
    g[0] = -fma(0.5 * z, q2, hr * fma(b.H, H, fma(k, c, fma(ub, u, vb * v))));
    g[1] = hr * ub;
    g[2] = hr * vb;
    g[3] = 0.5 * Eb;
}

// ------------------------------------------------------------------------------------------
// Lax-Friedrichs flux
// ------------------------------------------------------------------------------------------
// one side's reverse: adjoints of its flux (Fb), its W_t (Tb) and the flux's derivative (Db), and of its wave
// speed |U| + c (ab); Wb holds the state's direct share and becomes the whole
DFK_HD void lf_side_reverse(const FlowState& s, const GPState& P, const FlowGrad& x, const FlowGrad& y, const FlowGrad& t,
                            const Real T[4], const SchemeConsts& S, const Real Fb[4], const Real Tb[4], const Real Db[4],
                            Real ab, Real Wb[4], GPStateBar& out) {
    const Real m = Real::raw(P.W[1]), Ep = Real::raw(P.W[3]) + s.p, H = Ep * s.ir;
    FlowBar sb;
    zero(sb);
    GradBar tb, xb, yb;
    zero(xb);
    zero(yb);
    // D = (T1, U (T1 + t1) + dp, V T1 + U t2, H t1 + U (T3 + dp))
    const Real T3b = fma(s.U, Db[3], Tb[3]), T1b = fma(s.U, Db[1], fma(s.V, Db[2], Tb[1] + Db[0]));
    // T = (t0, U t0 + t1, V t0 + t2, dp/(gamma-1) + hq t0 + U t1 + V t2)
    tb.r0 = fma(s.U, T1b, fma(s.V, Tb[2], fma(s.hq, T3b, Tb[0])));
    tb.r1 = fma(s.U, T3b, fma(H, Db[3], fma(s.U, Db[1], T1b)));
    tb.r2 = fma(s.V, T3b, fma(s.U, Db[2], Tb[2]));
    tb.q3 = 0.0;
    tb.dp = fma(0.5 * (S.K + 2.0), T3b, fma(s.U, Db[3], Db[1]));
    const Real Epb = fma(s.U, Fb[3], (t.r1 * Db[3]) * s.ir);            // of E + p, through H too
    sb.U = fma(T[1] + t.r1, Db[1], fma(t.r2, Db[2], fma(T[3] + t.dp, Db[3], fma(t.r0, T1b, fma(t.r1, T3b, fma(m, Fb[1], Ep * Fb[3]))))));
    sb.V = fma(T[1], Db[2], fma(t.r0, Tb[2], fma(t.r2, T3b, m * Fb[2])));
    sb.hq = t.r0 * T3b;
    sb.p = Fb[1] + Epb;
    // |U|'s slope: +1 at both zeros (the pattern of -0 is the smallest of the negative ones)
    sb.U = sb.U + ((unsigned long long)dbits(s.U.v) <= 1ULL << 63 ? ab : -ab);
    sb.th = (0.5 * S.gamma) * (S.r2g * s.rs) * ab;                      // dc/dtheta = gamma / (2 c)
    euler_time_grad_rev(s, x, y, t, tb, S, xb, yb, sb);
    Real d[4];
    flow_grad_rev(s, x.r0, x, xb, S, d, sb);
#pragma unroll
    for (int i = 0; i < 4; ++i) out.Wn[i] = d[i].v;
    flow_grad_rev(s, y.r0, y, yb, S, d, sb);
#pragma unroll
    for (int i = 0; i < 4; ++i) out.Wt[i] = d[i].v;
    flow_state_rev(s, sb, S, d);
    Wb[0] = fma(-H, (t.r1 * Db[3]) * s.ir, Wb[0] + d[0]);               // H's 1/rho
    Wb[1] = fma(s.U, Fb[1], fma(s.V, Fb[2], Fb[0] + (Wb[1] + d[1])));
    Wb[2] = Wb[2] + d[2];
    Wb[3] = Epb + (Wb[3] + d[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) out.W[i] = Wb[i].v;
}

// reverse of lf_flux; sets Lb, Rb.  In gradient form like the flux: with it and the forward's the reverse of a
// 400 x 400 stage went from 3.93 (products with the flux Jacobians) to 3.67 ms.
DFK_HD void lf_flux_vjp(const GPState& L, const GPState& R, const SchemeConsts& S, const double Fbv[4],
                        const double dFbv[4], GPStateBar& Lb, GPStateBar& Rb) {
    const FlowState sl = side_state(L.W, S), sr = side_state(R.W, S);
    const FlowGrad xl = point_grad(sl, L.Wn, S), yl = point_grad(sl, L.Wt, S), xr = point_grad(sr, R.Wn, S), yr = point_grad(sr, R.Wt, S);
    const FlowGrad tl = euler_time_grad(sl, xl, yl, S), tr = euler_time_grad(sr, xr, yr, S);
    const Real al = fabs(sl.U) + sound_speed(sl, S), ar = fabs(sr.U) + sound_speed(sr, S);
    const bool left = !nn_less(al, ar);           // the left speed on a tie (both >= 0)
    const Real h = 0.5 * (left ? al : ar);
    Real Tl[4], Tr[4];
    lf_time(sl, tl, S, Tl);
    lf_time(sr, tr, S, Tr);
    Real Fb[4], Db[4], Tb[4], Wb[4], sb = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const Real f = Real::raw(Fbv[i]), d = Real::raw(dFbv[i]);
        sb = fma(f, Real::raw(L.W[i]) - Real::raw(R.W[i]), fma(d, Tl[i] - Tr[i], sb));
        Fb[i] = 0.5 * f;
        Db[i] = 0.5 * d;
        Wb[i] = h * f;
        Tb[i] = h * d;
    }
    sb = 0.5 * sb;
    lf_side_reverse(sl, L, xl, yl, tl, Tl, S, Fb, Tb, Db, left ? sb : Real(0.0), Wb, Lb);
#pragma unroll
    for (int i = 0; i < 4; ++i) { Wb[i] = -(h * Real::raw(Fbv[i])); Tb[i] = -Tb[i]; }
    lf_side_reverse(sr, R, xr, yr, tr, Tr, S, Fb, Tb, Db, left ? Real(0.0) : sb, Wb, Rb);
}

}  // namespace dfk

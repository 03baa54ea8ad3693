// dfgks_adjoint.cu -- reverse (vector-Jacobian product) of the single-stage operator.
//
// With the forward records in place (face lines, Gauss-point states, fluxes), three kernels walk the
// sweeps backwards, both directions in one launch each where there is memory for both's adjoints:
//   ka_flux  : one thread per Gauss point.  Face adjoints from the cells' L, dL/dt and limited
//              dL/dt adjoints (Eq. 2 with A_m = 1/2), then the GKS / L-F flux adjoint into the
//              Gauss-point record adjoints, and the time-limiter weight's adjoint.  When the
//              forward sweep taped the GKS flux's intermediates, its reverse reads them instead
//              of recomputing the flux.
//   ka_faces : one thread per face side.  Evaluates the ratios of each tangential reconstruction
//              (or reads them from the forward sweep's tape), reverses it in differences,
//              and scatters (atomically) into the adjoints of
//              the five face lines and of the face basis; a Gauss point that fell back to the cell
//              average (flagged in the forward record) sends its adjoint to that cell.
//   ka_lines : one thread per face line.  The same for the eight normal reconstructions and the
//              limiter weight (the forward record names the reconstruction that set it), then
//              scatters into the ghosted cell adjoints.
// A final pass folds ghost-cell adjoints back into the interior cells they were copied from.
// alpha, dt and every branch decision are those of the forward pass.
#include "dfgks_adjoint.cuh"
#include "dfgks_bodies.cuh"

namespace dfk {

DFK_HD void aadd(double* p, double v) {
#ifdef __CUDA_ARCH__
    if (dbits(v) << 1) atomicAdd(p, v);         // not +-0, tested off the FP64 units
#else
    *p += v;
#endif
}

// TAPED: the GKS forward intermediates are read from the tape the forward sweep wrote
template <int DIR, int FLUX, bool TAPED = false>
DFK_HD void ka_flux_body(const Mesh& m, const SchemeConsts& S, const AdjointArgs& a, const double* __restrict__ gp,
                         long long gs, const double* __restrict__ fr, long long fs, double dt, double* __restrict__ lb,
                         long long ls, double* __restrict__ gb, int ax, int ay, int mm,
                         double* __restrict__ tape = nullptr) {
    Geo<DIR> g(m);
    int f = DIR == 0 ? ax : ay;
    int t = DIR == 0 ? ay : ax;
    if (f > g.nn || t >= g.nt) return;
    const long long fid = g.face(f, t), nf = g.nfaces();
    const long long dplane = (long long)m.nx * m.ny;
    // adjoints of the two cells' residuals (cells outside the mesh have none)
    double dL[4] = {0, 0, 0, 0}, ddL[4] = {0, 0, 0, 0}, ddLt[4] = {0, 0, 0, 0};
    for (int side = 0; side < 2; ++side) {
        const int n = f - 1 + side;
        if (n < 0 || n >= g.nn) continue;
        const long long c = DIR == 0 ? (long long)t * m.nx + n : (long long)n * m.nx + t;
        const double sg = side == 0 ? -1.0 : 1.0;    // F enters L of the left cell with -1/dn
        for (int k = 0; k < 4; ++k) {
            if (a.Lb) dL[k] += sg * a.Lb[k * dplane + c];
            if (a.dtLb) ddL[k] += sg * a.dtLb[k * dplane + c];
            if (a.dtLtb) ddLt[k] += sg * a.dtLtb[k * dplane + c];
        }
    }
    const double idn = g.idn;
    const double om = fr[FR_OMEGA * fs + fid];
    double Fb[4], dFb[4];
    for (int k = 0; k < 4; ++k) {
        Fb[k] = 0.5 * dL[k] * idn;                              // Gauss weight 1/2
        dFb[k] = 0.5 * (ddL[k] + om * ddLt[k]) * idn;
    }
    if (mm == 0 && S.time_limiter) {
        double wb = 0.0;
        for (int k = 0; k < 4; ++k) {
            double dFface = 0.5 * fr[(FR_DF + k) * fs + fid] + 0.5 * fr[(FR_DF + k) * fs + nf + fid];
            wb += dFface * ddLt[k] * idn;
        }
        lb[LR_TL * ls + g.line(f, t)] = wb;
    }
    to_local<DIR>(Fb);                                          // F = T^{-1} F~, T orthogonal
    to_local<DIR>(dFb);
    const long long eL = fid, eR = nf + fid;
    GPState L, R;
    for (int k = 0; k < 4; ++k) {
        L.W[k] = gp[(mm * 12 + k) * gs + eL];
        L.Wn[k] = gp[(mm * 12 + 4 + k) * gs + eL];
        L.Wt[k] = gp[(mm * 12 + 8 + k) * gs + eL];
        R.W[k] = gp[(mm * 12 + k) * gs + eR];
        R.Wn[k] = gp[(mm * 12 + 4 + k) * gs + eR];
        R.Wt[k] = gp[(mm * 12 + 8 + k) * gs + eR];
    }
    GPStateBar Lbar, Rbar;
    if (FLUX == 0 && TAPED) gks_flux_reverse(PlaneTape{tape + (long long)mm * nf + fid, fs}, L, R, S, Fb, dFb, Lbar, Rbar);
    else if (FLUX == 0) gks_flux_vjp(L, R, dt, S, Fb, dFb, Lbar, Rbar);
    else lf_flux_vjp(L, R, S, Fb, dFb, Lbar, Rbar);
    for (int k = 0; k < 4; ++k) {
        gb[(mm * 12 + k) * gs + eL] = Lbar.W[k];
        gb[(mm * 12 + 4 + k) * gs + eL] = Lbar.Wn[k];
        gb[(mm * 12 + 8 + k) * gs + eL] = Lbar.Wt[k];
        gb[(mm * 12 + k) * gs + eR] = Rbar.W[k];
        gb[(mm * 12 + 4 + k) * gs + eR] = Rbar.Wn[k];
        gb[(mm * 12 + 8 + k) * gs + eR] = Rbar.Wt[k];
    }
}

// the face basis of a line record
DFK_HD CharBasis line_basis(const double* __restrict__ lines, long long ls, long long l) {
    CharBasis B;
    B.u = lines[LR_U * ls + l]; B.v = lines[LR_V * ls + l]; B.c = lines[LR_C * ls + l];
    B.ic = lines[LR_IC * ls + l]; B.H = lines[LR_H * ls + l]; B.b1 = lines[LR_B1 * ls + l];
    B.b2 = lines[LR_B2 * ls + l]; B.q2 = lines[LR_Q2 * ls + l];
    return B;
}

// TAPED: the tangential reconstructions' ratios are read from the tape the forward sweep wrote
template <int DIR, bool TAPED = false>
DFK_HD void ka_faces_body(const Mesh& m, const SchemeConsts& S, const double* __restrict__ alpha,
                          const double* __restrict__ lines, long long ls, const double* __restrict__ gp,
                          const double* __restrict__ gb, long long gs, double* __restrict__ lb,
                          double* __restrict__ Wb, int ax, int ay, int side, double* __restrict__ ftape = nullptr) {
    Geo<DIR> g(m);
    int f = DIR == 0 ? ax : ay;
    int t = DIR == 0 ? ay : ax;
    if (f > g.nn || t >= g.nt) return;
    const long long l0 = g.line(f, t);
    const DiffBasis D = diff_basis(line_basis(lines, ls, l0));
    const int wbase = side == 0 ? LR_WL : LR_WR;
    const int nbase = side == 0 ? LR_WLN : LR_WRN;
    const int ncell = f - 1 + side;
    double al[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) al[b] = alpha[g.cell(m, ncell, t + Geo<DIR>::sigma * (b - 1))];
    const bool df = nn_less(nn_max(nn_max(al[0], al[1]), al[2]), S.alpha_thres);
    const Real idt = g.idtan;
    const long long e = (long long)side * g.nfaces() + g.face(f, t);
    const int fbits = (int)gp[GP_FB * gs + e];
    Real dW[4][4], F[4][4];
    {
        Real prev[4];
#pragma unroll
        for (int b = 0; b < 5; ++b) {
            const long long lbb = g.line(f, t + Geo<DIR>::sigma * (b - 2));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const Real w = Real::raw(lines[(wbase + k) * ls + lbb]);
                if (b > 0) dW[b - 1][k] = w - prev[k];
                prev[k] = w;
            }
            if (b > 0) project_diff(D, dW[b - 1], F[b - 1]);
        }
    }
    // Gauss-point adjoints -> characteristic value and tangential-slope adjoints (R^T, independent of the
    // reconstruction); a Gauss point that used the cell average sends its adjoint there.  The face line's normal
    // slope adjoint has no other contribution, so it is stored.
    Real wb[2][4], wtb[2][4], qvb[2][4], qtb[2][4], nb[4], centre[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) nb[k] = centre[k] = 0.0;
#pragma unroll
    for (int mm = 0; mm < 2; ++mm) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            wb[mm][k] = Real::raw(gb[(mm * 12 + k) * gs + e]);
            wtb[mm][k] = idt * Real::raw(gb[(mm * 12 + 8 + k) * gs + e]);
        }
        if ((fbits >> mm) & 1) {
            double wg[4] = {wb[mm][0].v, wb[mm][1].v, wb[mm][2].v, wb[mm][3].v};
            to_global<DIR>(wg);
            const long long c = g.cell(m, ncell, t);
#pragma unroll
            for (int k = 0; k < 4; ++k) { aadd(&Wb[k * m.plane + c], wg[k]); wb[mm][k] = wtb[mm][k] = 0.0; }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                nb[k] = nb[k] + Real::raw(gb[(mm * 12 + 4 + k) * gs + e]);
                centre[k] = centre[k] + wb[mm][k];
            }
        }
        back_project_diff_T(D, wb[mm], qvb[mm]);
        back_project_diff_T(D, wtb[mm], qtb[mm]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) lb[(nbase + k) * ls + l0] = nb[k].v;
    // per characteristic component: the coefficients, the evaluation's and the weights' reverse
    Real qv[2][4], qt[2][4], Fb[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const Real gg = kGaussEta;
        const Real s0 = F[1][k] - F[0][k], s1 = F[2][k] - F[1][k], s2 = F[3][k] - F[2][k];
        const Real a11 = fma(0.5, s1, F[1][k]);
        const Real Ob = gg * (qvb[1][k] - qvb[0][k]), Esb = qtb[0][k] + qtb[1][k], Osb = gg * (qtb[1][k] - qtb[0][k]);
        Real v[2], sl[2];
        AODiffBar b;
        b.fb = b.ff = b.to = b.ti = 0.0;
        if (df) {
            b.s0 = b.s2 = 0.0;
            const Real alpha1 = Real::raw(al[1]);
            df_diff_at_gauss(a11, s1, alpha1, v, sl);
            const Real a11b = alpha1 * (Ob + Esb);
            b.fb = a11b;
            b.s1 = fma(0.5, a11b, alpha1 * Osb);
        } else {
            const Real t1 = s1 - s0, t2 = s2 - s1, T = t1 + t2, U = t2 - t1;
            AORatios q;
            if constexpr (TAPED) q = tape_get_ratios(PlaneTape{ftape + e, gs}, k * RT_COUNT);
            else {
                const Real eps = (k == 0 || k == 3) ? Real(4.0 * S.eps) : Real(S.eps);
                q = ao_ratios(ao_weights<+1>(F[1][k], F[2][k], s0, s1, s2, second_difference_energy(s0, eps),
                                             second_difference_energy(s1, eps), second_difference_energy(s2, eps), a11, T, U,
                                             eps, S));
            }
            const AOCoeffs c = ao_coeffs(q, S);
            const Real a10 = fma(0.5, s0, F[1][k]), a12 = fma(-0.5, s2, F[2][k]);
            const Real c3T = c.c3 * T, c3U = c.c3 * U;
            {   // the values, for the basis (ao_diff_at_gauss)
                const Real B = fma(c.c0, a10, fma(c.cm, a11, c.c2 * a12)), E2 = fma(c.c0, s0, fma(c.cm, s1, c.c2 * s2));
                const Real O = gg * fma(-7.0 / 72.0, c3T, B), Es = fma(-1.0 / 12.0, c3T, B);
                const Real Os = gg * fma(-1.0 / 9.0, c3U, E2), E = (-1.0 / 4320.0) * c3U;
                v[0] = E - O; v[1] = E + O;
                sl[0] = Es - Os; sl[1] = Es + Os;
            }
            const Real Eb = qvb[0][k] + qvb[1][k], Bb = Ob + Esb;
            const Real c3Tb = fma(-7.0 / 72.0, Ob, (-1.0 / 12.0) * Esb), c3Ub = fma(-1.0 / 4320.0, Eb, (-1.0 / 9.0) * Osb);
            b.a10 = c.c0 * Bb; b.a11 = c.cm * Bb; b.a12 = c.c2 * Bb;
            b.s0 = c.c0 * Osb; b.s1 = c.cm * Osb; b.s2 = c.c2 * Osb;
            Real zb[4];
            ao_coeffs_rev(c, q, fma(Bb, a10, Osb * s0), fma(Bb, a11, Osb * s1), fma(Bb, a12, Osb * s2), fma(c3Tb, T, c3Ub * U), S, zb);
            ao_ratios_rev<+1>(q, c, zb, s0, s1, s2, a10, a11, a12, T, U, c.c3 * c3Tb, c.c3 * c3Ub, b);
        }
        // third differences to second, second to first
        const Real s0b = b.s0 - b.to, s1b = b.s1 + (b.to - b.ti), s2b = b.s2 + b.ti;
        Fb[0][k] = -s0b;
        Fb[1][k] = b.fb + (s0b - s1b);
        Fb[2][k] = b.ff + (s1b - s2b);
        Fb[3][k] = s2b;
        qv[0][k] = v[0]; qv[1][k] = v[1];
        qt[0][k] = sl[0]; qt[1][k] = sl[1];
    }
    DiffBasisBar Bb;
    zero(Bb);
#pragma unroll
    for (int mm = 0; mm < 2; ++mm) {          // zero adjoints (fallback) add nothing
        back_project_diff_basis_rev(qv[mm], wb[mm], Bb);
        back_project_diff_basis_rev(qt[mm], wtb[mm], Bb);
    }
    Real left[4];                             // adjoint of line b from the difference below it
#pragma unroll
    for (int k = 0; k < 4; ++k) left[k] = 0.0;
#pragma unroll
    for (int b = 0; b < 5; ++b) {
        Real w[4];
        if (b < 4) project_diff_rev(D, dW[b], Fb[b], w, Bb);
        const long long lbb = g.line(f, t + Geo<DIR>::sigma * (b - 2));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Real x = left[k];
            if (b < 4) x = b == 0 ? -w[k] : x - w[k];
            if (b == 2) x = x + centre[k];
            aadd(&lb[(wbase + k) * ls + lbb], x.v);
            if (b < 4) left[k] = w[k];
        }
    }
    const BasisAdj o = diff_basis_rev(D, Bb);
    aadd(&lb[LR_U * ls + l0], o.u.v); aadd(&lb[LR_V * ls + l0], o.v.v); aadd(&lb[LR_C * ls + l0], o.c.v);
    aadd(&lb[LR_IC * ls + l0], o.ic.v); aadd(&lb[LR_H * ls + l0], o.H.v); aadd(&lb[LR_B1 * ls + l0], o.b1.v);
    aadd(&lb[LR_B2 * ls + l0], o.b2.v); aadd(&lb[LR_Q2 * ls + l0], o.q2.v);
}

// one normal reconstruction's reverse (SGN +1: cell f-1's value at its right edge, -1: cell f's at its left): value
// and slope adjoints vb, sb (the slope per cell), limiter weight adjoint wb (0 unless this one set it); sets the
// value minus the cell average and the slope, and adds to b
template <int SGN>
DFK_HD void edge_reverse(const AORatios& q, bool df, Real alpha, Real vb, Real sb, double wb, Real fb, Real ff, Real s0, Real s1,
                         Real s2, Real to, Real ti, const SchemeConsts& S, Real& v, Real& sl, AODiffBar& b) {
    const bool lim = (dbits(wb) << 1) != 0;
    constexpr double h = 0.5 * SGN;
    if (df) {
        const Real ab = alpha * vb;
        b.ff = fma(alpha, sb, fma(h, ab, b.ff));
        b.s1 = fma(-1.0 / 6.0, ab, b.s1);
        v = alpha * fma(-1.0 / 6.0, s1, h * ff);
        sl = alpha * ff;
        if (!lim) return;
    }
    const AOCoeffs c = ao_coeffs(q, S);
    const Real a10 = fma(h, s0, fb), a11 = fma(h, s1, fb), a12 = fma(-h, s2, ff);
    const Real T = to + ti, U = SGN > 0 ? ti - to : to - ti;
    Real zb[4];
    if (!df) {
        const Real w = fma(1.0 / 30.0, to, (1.0 / 20.0) * ti), h12 = (1.0 / 12.0) * ti;
        const Real B = fma(c.c0, a10, fma(c.cm, a11, c.c2 * a12)), D = fma(c.c0, s0, fma(c.cm, s1, c.c2 * s2));
        const Real c3w = c.c3 * w;
        v = fma(1.0 / 12.0, D, SGN > 0 ? fma(h, B, -c3w) : fma(h, B, c3w));
        sl = fma(-c.c3, h12, fma(h, D, B));
        const Real xb = SGN > 0 ? -vb : vb;
        const Real Bb = fma(h, vb, sb), Db = fma(1.0 / 12.0, vb, h * sb);
        b.a10 = c.c0 * Bb; b.a11 = c.cm * Bb; b.a12 = c.c2 * Bb;
        b.s0 = fma(c.c0, Db, b.s0); b.s1 = fma(c.cm, Db, b.s1); b.s2 = fma(c.c2, Db, b.s2);
        b.to = fma((1.0 / 30.0) * c.c3, xb, b.to);
        b.ti = fma(c.c3, fma(1.0 / 20.0, xb, (-1.0 / 12.0) * sb), b.ti);
        ao_coeffs_rev(c, q, fma(Bb, a10, Db * s0), fma(Bb, a11, Db * s1), fma(Bb, a12, Db * s2), fma(xb, w, -(sb * h12)), S, zb);
    } else {
        b.a10 = b.a11 = b.a12 = 0.0;
        zb[0] = zb[1] = zb[2] = zb[3] = 0.0;
    }
    if (lim) ao_limiter_rev(q, c, Real::raw(wb), zb);
    ao_ratios_rev<SGN>(q, c, zb, s0, s1, s2, a10, a11, a12, T, U, 0.0, 0.0, b);
}

// TAPED: the normal reconstructions' ratios are read from the tape the forward sweep wrote
template <int DIR, bool TAPED = false>
DFK_HD void ka_lines_body(const Mesh& m, const SchemeConsts& S, const double* __restrict__ W,
                          const double* __restrict__ alpha, const double* __restrict__ lines,
                          const double* __restrict__ lb, long long ls, double* __restrict__ Wb, int ax, int ay,
                          double* __restrict__ ltape = nullptr) {
    Geo<DIR> g(m);
    int f = DIR == 0 ? ax : ay;
    int tt = DIR == 0 ? ay : ax;
    if (f > g.nn || tt >= g.nt + 4) return;
    const int t = tt - 2;
    const long long li = g.line(f, t);
    const CharBasis B = line_basis(lines, ls, li);
    const DiffBasis D = diff_basis(B);
    Real dW[5][4], F[5][4];
    Real density = 0.0;
    double al[6];
    {
        Real prev[4];
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            const long long c = g.cell(m, f - 3 + s, t);
            double w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = W[k * m.plane + c];
            to_local<DIR>(w);
            al[s] = alpha[c];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const Real x = Real::raw(w[k]);
                if (s > 0) dW[s - 1][k] = x - prev[k];
                prev[k] = x;
            }
            if (s == 2 || s == 3) density = fma(0.5, prev[0], density);
            if (s > 0) project_diff(D, dW[s - 1], F[s - 1]);
        }
    }
    const bool dfL = nn_less(nn_max(nn_max(al[1], al[2]), al[3]), S.alpha_thres);
    const bool dfR = nn_less(nn_max(nn_max(al[2], al[3]), al[4]), S.alpha_thres);
    const Real idn = g.idn;
    // the reconstruction that set the limiter weight in the forward pass (2k + side) and the
    // weight's adjoint
    const int tlk = S.time_limiter ? (int)lines[LR_TLK * ls + li] : -1;
    const double tlb = S.time_limiter ? lb[LR_TL * ls + li] : 0.0;
    Real WLb[4], WLnb[4], WRb[4], WRnb[4], qLb[4], qLnb[4], qRb[4], qRnb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        WLb[k] = Real::raw(lb[(LR_WL + k) * ls + li]); WLnb[k] = idn * Real::raw(lb[(LR_WLN + k) * ls + li]);
        WRb[k] = Real::raw(lb[(LR_WR + k) * ls + li]); WRnb[k] = idn * Real::raw(lb[(LR_WRN + k) * ls + li]);
    }
    back_project_diff_T(D, WLb, qLb);
    back_project_diff_T(D, WLnb, qLnb);
    back_project_diff_T(D, WRb, qRb);
    back_project_diff_T(D, WRnb, qRnb);
    Real qL[4], qLn[4], qR[4], qRn[4], Fb[5][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const Real f3 = F[2][k];
        const Real s1 = F[1][k] - F[0][k], s2 = f3 - F[1][k], s3 = F[3][k] - f3, s4 = F[4][k] - F[3][k];
        const Real t1 = s2 - s1, t2 = s3 - s2, t3 = s4 - s3;
        AORatios L, R;
        if constexpr (TAPED) {
            const PlaneTape T{ltape + li, ls};
            L = tape_get_ratios(T, 2 * k * RT_COUNT);
            R = tape_get_ratios(T, (2 * k + 1) * RT_COUNT);
        } else {
            const Real eps = (k == 0 || k == 3) ? Real(4.0 * S.eps) : Real(S.eps);
            const Real w1 = second_difference_energy(s1, eps), w2 = second_difference_energy(s2, eps);
            const Real w3 = second_difference_energy(s3, eps), w4 = second_difference_energy(s4, eps);
            L = ao_ratios(ao_weights<+1>(F[1][k], f3, s1, s2, s3, w1, w2, w3, fma(0.5, s2, F[1][k]), t1 + t2, t2 - t1, eps, S));
            R = ao_ratios(ao_weights<-1>(F[3][k], f3, s4, s3, s2, w4, w3, w2, fma(-0.5, s3, F[3][k]), t2 + t3, t3 - t2, eps, S));
        }
        AODiffBar l, r;                       // adjoints of F1, f3; s1, s2, s3; t1, t2 and of F3, f3; s4, s3, s2; t3, t2
        l.fb = l.ff = l.s0 = l.s1 = l.s2 = l.to = l.ti = 0.0;
        r = l;
        edge_reverse<+1>(L, dfL, Real::raw(al[2]), qLb[k], qLnb[k], tlk == 2 * k ? tlb : 0.0, F[1][k], f3, s1, s2, s3, t1, t2, S,
                         qL[k], qLn[k], l);
        edge_reverse<-1>(R, dfR, Real::raw(al[3]), qRb[k], qRnb[k], tlk == 2 * k + 1 ? tlb : 0.0, F[3][k], f3, s4, s3, s2, t3, t2,
                         S, qR[k], qRn[k], r);
        const Real tib = l.ti + r.ti;
        const Real s1b = l.s0 - l.to, s2b = (l.s1 + r.s2) + (l.to - tib), s3b = (l.s2 + r.s1) + (tib - r.to), s4b = r.s0 + r.to;
        Fb[0][k] = -s1b;
        Fb[1][k] = l.fb + (s1b - s2b);
        Fb[2][k] = (l.ff + r.ff) + (s2b - s3b);
        Fb[3][k] = r.fb + (s3b - s4b);
        Fb[4][k] = s4b;
    }
    DiffBasisBar Bb;
    zero(Bb);
    back_project_diff_basis_rev(qL, WLb, Bb);
    back_project_diff_basis_rev(qLn, WLnb, Bb);
    back_project_diff_basis_rev(qR, WRb, Bb);
    back_project_diff_basis_rev(qRn, WRnb, Bb);
    Real Wcb[6][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) Wcb[0][k] = 0.0;
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        Real w[4];
        project_diff_rev(D, dW[s], Fb[s], w, Bb);
#pragma unroll
        for (int k = 0; k < 4; ++k) { Wcb[s][k] = s == 0 ? -w[k] : Wcb[s][k] - w[k]; Wcb[s + 1][k] = w[k]; }
    }
    BasisAdj o = diff_basis_rev(D, Bb);
    o.u = o.u + Real::raw(lb[LR_U * ls + li]); o.v = o.v + Real::raw(lb[LR_V * ls + li]);
    o.c = o.c + Real::raw(lb[LR_C * ls + li]); o.ic = o.ic + Real::raw(lb[LR_IC * ls + li]);
    o.H = o.H + Real::raw(lb[LR_H * ls + li]); o.b1 = o.b1 + Real::raw(lb[LR_B1 * ls + li]);
    o.b2 = o.b2 + Real::raw(lb[LR_B2 * ls + li]); o.q2 = o.q2 + Real::raw(lb[LR_Q2 * ls + li]);
    Real gm[4];
    make_basis_rev(B, density, o, S, gm);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        Wcb[2][k] = Wcb[2][k] + (gm[k] + WLb[k]);
        Wcb[3][k] = Wcb[3][k] + (gm[k] + WRb[k]);
    }
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        double w[4] = {Wcb[s][0].v, Wcb[s][1].v, Wcb[s][2].v, Wcb[s][3].v};
        to_global<DIR>(w);                                     // the rotation is orthogonal
        const long long c = g.cell(m, f - 3 + s, t);
#pragma unroll
        for (int k = 0; k < 4; ++k) aadd(&Wb[k * m.plane + c], w[k]);
    }
}

// Reverse of the ghost fill: the y pass (all columns) first, then the x pass (interior rows).  Components
// [k0, k1): the kernels take one each, with the six ghost values loaded before they are added, as one thread's
// chain of dependent loads and stores is all the time there is (20 us a pass for four components in turn).
DFK_HD void fold_add(double* W, const long long d[2 * G], const long long o[2 * G], const bool neg[2 * G]) {
    double v[2 * G];
#pragma unroll
    for (int q = 0; q < 2 * G; ++q) v[q] = W[d[q]];
#pragma unroll
    for (int q = 2 * G - 1; q >= 0; --q) {
        W[d[q]] = 0.0;
        W[o[q]] += neg[q] ? -v[q] : v[q];
    }
}

DFK_HD void ka_fold_y_body(const Mesh& m, double* Wb, int i, int k0 = 0, int k1 = 4) {
    if (i >= m.nx + G) return;
    for (int k = k0; k < k1; ++k) {
        long long d[2 * G], o[2 * G];
        bool neg[2 * G];
#pragma unroll
        for (int gr = 0; gr < 2 * G; ++gr) {
            const int j = gr < G ? gr - G : m.ny + gr - G;
            bool mir;
            o[gr] = gid(m, i, ghost_src(j, m.ny, m.bc[2], m.bc[3], mir));
            d[gr] = gid(m, i, j);
            neg[gr] = mir && k == 2;
        }
        fold_add(Wb + k * m.plane, d, o, neg);
    }
}

DFK_HD void ka_fold_x_body(const Mesh& m, double* Wb, int j, int k0 = 0, int k1 = 4) {
    if (j >= m.ny) return;
    for (int k = k0; k < k1; ++k) {
        long long d[2 * G], o[2 * G];
        bool neg[2 * G];
#pragma unroll
        for (int gc = 0; gc < 2 * G; ++gc) {
            const int i = gc < G ? gc - G : m.nx + gc - G;
            bool mir;
            o[gc] = gid(m, ghost_src(i, m.nx, m.bc[0], m.bc[1], mir), j);
            d[gc] = gid(m, i, j);
            neg[gc] = mir && k == 1;
        }
        fold_add(Wb + k * m.plane, d, o, neg);
    }
}

DFK_HD void ka_accumulate_body(const Mesh& m, const double* __restrict__ Wbg, double* __restrict__ out, int i, int j) {
    if (i >= m.nx || j >= m.ny) return;
    const long long dp = (long long)m.nx * m.ny;
    for (int k = 0; k < 4; ++k) out[k * dp + (long long)j * m.nx + i] += Wbg[k * m.plane + gid(m, i, j)];
}

// ---- kernels: one thread per body invocation; blocks [0, nb0) take the x sweep, the rest the y sweep ----
struct ReverseDir {
    const double* lines; const double* gp; const double* fr; long long fs;
    double* lb; double* gb; double* tape; double* ltape; double* ftape;
};

__device__ __forceinline__ void reverse_at(int b, int lx, int& ax, int& ay) {
    const int i = b * (int)blockDim.x + (int)threadIdx.x;
    ax = i % lx;
    ay = i / lx;
}

template <int FLUX, bool TAPED>
__global__ void __launch_bounds__(128) ka_flux(Mesh m, SchemeConsts S, AdjointArgs a, ReverseDir X, ReverseDir Y, long long ls,
                                               long long gs, const double* dtp, int nb0) {
    int ax, ay;
    const int b = blockIdx.x;
    if (b < nb0) {
        reverse_at(b, faces_lx<0>(m), ax, ay);
        ka_flux_body<0, FLUX, TAPED>(m, S, a, X.gp, gs, X.fr, X.fs, *dtp, X.lb, ls, X.gb, ax, ay, blockIdx.y, X.tape);
    } else {
        reverse_at(b - nb0, faces_lx<1>(m), ax, ay);
        ka_flux_body<1, FLUX, TAPED>(m, S, a, Y.gp, gs, Y.fr, Y.fs, *dtp, Y.lb, ls, Y.gb, ax, ay, blockIdx.y, Y.tape);
    }
}

template <bool TAPED>
__global__ void __launch_bounds__(128) ka_faces(Mesh m, SchemeConsts S, const double* __restrict__ alpha, ReverseDir X, ReverseDir Y,
                                                long long ls, long long gs, double* __restrict__ Wb, int nb0) {
    int ax, ay;
    const int b = blockIdx.x;
    if (b < nb0) {
        reverse_at(b, faces_lx<0>(m), ax, ay);
        ka_faces_body<0, TAPED>(m, S, alpha, X.lines, ls, X.gp, X.gb, gs, X.lb, Wb, ax, ay, blockIdx.y, X.ftape);
    } else {
        reverse_at(b - nb0, faces_lx<1>(m), ax, ay);
        ka_faces_body<1, TAPED>(m, S, alpha, Y.lines, ls, Y.gp, Y.gb, gs, Y.lb, Wb, ax, ay, blockIdx.y, Y.ftape);
    }
}

template <bool TAPED>
__global__ void __launch_bounds__(128) ka_lines(Mesh m, SchemeConsts S, const double* __restrict__ W, const double* __restrict__ alpha,
                                                ReverseDir X, ReverseDir Y, long long ls, double* __restrict__ Wb, int nb0) {
    int ax, ay;
    const int b = blockIdx.x;
    if (b < nb0) {
        reverse_at(b, lines_lx<0>(m), ax, ay);
        ka_lines_body<0, TAPED>(m, S, W, alpha, X.lines, X.lb, ls, Wb, ax, ay, X.ltape);
    } else {
        reverse_at(b - nb0, lines_lx<1>(m), ax, ay);
        ka_lines_body<1, TAPED>(m, S, W, alpha, Y.lines, Y.lb, ls, Wb, ax, ay, Y.ltape);
    }
}

__global__ void ka_fold_y(Mesh m, double* Wb) { ka_fold_y_body(m, Wb, blockIdx.x * blockDim.x + threadIdx.x - G, blockIdx.y, blockIdx.y + 1); }
__global__ void ka_fold_x(Mesh m, double* Wb) { ka_fold_x_body(m, Wb, blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y, blockIdx.y + 1); }
__global__ void ka_accumulate_dense(Mesh m, const double* __restrict__ Wbg, double* __restrict__ out) {
    ka_accumulate_body(m, Wbg, out, blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y * blockDim.y + threadIdx.y);
}

void launch_adjoint(int dirs, const Mesh& m, const SchemeConsts& S, int flux, const AdjointArgs& a, const double* W,
                    const double* alpha, const double* dtp, const SweepBuffers B[2], double* const lb[2],
                    double* const gbuf[2], double* Wb, cudaStream_t s, KernelTimer* T) {
    // the forward sweep's 1-D grids (sweep_xy)
    const dim3 blk(kSweepThreads);
    const bool dx = dirs & 1, dy = dirs & 2;
    const int nf0 = dx ? (int)sweep_blocks(faces_lx<0>(m), faces_ly<0>(m)) : 0, nf1 = dy ? (int)sweep_blocks(faces_lx<1>(m), faces_ly<1>(m)) : 0;
    const int nl0 = dx ? (int)sweep_blocks(lines_lx<0>(m), lines_ly<0>(m)) : 0, nl1 = dy ? (int)sweep_blocks(lines_lx<1>(m), lines_ly<1>(m)) : 0;
    const dim3 gf(nf0 + nf1, 2), gl(nl0 + nl1);
    ReverseDir R[2];
    for (int d = 0; d < 2; ++d) {
        R[d] = {B[d].lines, B[d].gp, B[d].flux[d], B[d].flux_stride[d], lb[d], gbuf[d], B[d].tape[d], B[d].ltape, B[d].ftape};
        if (dirs & (1 << d)) cudaMemsetAsync(lb[d], 0, sizeof(double) * LR_COUNT * B[d].line_stride, s);
    }
    const int d0 = dx ? 0 : 1;
    const long long ls = B[d0].line_stride, gs = B[d0].gp_stride;
    if (T) T->begin(KK_FLUX);
    if (flux == 0 && B[d0].tape[d0]) ka_flux<0, true><<<gf, blk, 0, s>>>(m, S, a, R[0], R[1], ls, gs, dtp, nf0);
    else if (flux == 0) ka_flux<0, false><<<gf, blk, 0, s>>>(m, S, a, R[0], R[1], ls, gs, dtp, nf0);
    else ka_flux<1, false><<<gf, blk, 0, s>>>(m, S, a, R[0], R[1], ls, gs, dtp, nf0);
    if (T) { T->end(KK_FLUX, 1); T->begin(KK_FACES); }
    if (B[d0].ftape) ka_faces<true><<<gf, blk, 0, s>>>(m, S, alpha, R[0], R[1], ls, gs, Wb, nf0);
    else ka_faces<false><<<gf, blk, 0, s>>>(m, S, alpha, R[0], R[1], ls, gs, Wb, nf0);
    if (T) { T->end(KK_FACES, 1); T->begin(KK_LINES); }
    if (B[d0].ltape) ka_lines<true><<<gl, blk, 0, s>>>(m, S, W, alpha, R[0], R[1], ls, Wb, nl0);
    else ka_lines<false><<<gl, blk, 0, s>>>(m, S, W, alpha, R[0], R[1], ls, Wb, nl0);
    if (T) T->end(KK_LINES, 1);
}

void launch_adjoint_finish(const Mesh& m, double* Wbg, double* Wb_dense, cudaStream_t s) {
    ka_fold_y<<<dim3((m.nx + 2 * G + 31) / 32, 4), 32, 0, s>>>(m, Wbg);
    ka_fold_x<<<dim3((m.ny + 31) / 32, 4), 32, 0, s>>>(m, Wbg);
    dim3 blk(32, 8), grd((m.nx + 31) / 32, (m.ny + 7) / 8);
    ka_accumulate_dense<<<grd, blk, 0, s>>>(m, Wbg, Wb_dense);
}

// y <- a x + b y on dense arrays (step-adjoint combinations)
__global__ void ka_axpby(long long n, double a, const double* __restrict__ x, double b, double* __restrict__ y) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        y[q] = a * x[q] + b * y[q];
}
void launch_axpby(long long n, double a, const double* x, double b, double* y, cudaStream_t s) {
    long long blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    ka_axpby<<<(unsigned)blocks, 256, 0, s>>>(n, a, x, b, y);
}

}  // namespace dfk

// Host check of the reverse sweep's WENO-AO in differences (edge_reverse: weights, edge value and slope, limiter
// weight) against the reverse of the sub-stencil polynomials' form (weno_ao_rev), both mirror images, on smooth,
// rough, stepped and uniform stencils and on stencils so large that the weights leave their scaled form.
// Both are rounded at 2^-53 relative to stencil values at most ten times their differences, through at most
// four factors of beta^2: 1e-10 of the largest component is two orders above that.
#include "dfgks_adjoint.cu"
#include <cmath>
#include <cstdio>
#include <random>

using namespace dfk;

template <int SGN>
static double compare(const double q[5], double vb, double sb, double wb, bool df, double alpha, const SchemeConsts& S) {
    // textbook: the stencil as its own cell sees it, value and slope at its right edge
    double ref[5] = {0, 0, 0, 0, 0}, t[AT_COUNT], sq[5];
    for (int i = 0; i < 5; ++i) sq[i] = SGN > 0 ? q[i] : q[4 - i];
    const ArrayTape tp{t};
    const AO o = weno_ao_t(sq, S, tp, 0);
    AOBar ob;
    ao_bar_zero(ob);
    if (df) df_at_right_edge_vjp(alpha, vb, SGN * sb, ref);
    else ao_at_right_edge_vjp(vb, SGN * sb, ref[2], ob);
    if (wb != 0.0) limiter_alpha_vjp(o, wb, ob);
    if (!df || wb != 0.0) weno_ao_rev(tp, 0, S, ob, ref);
    // differences, unmirrored: fb, ff either side of the cell as the mirrored stencil names them
    const Real f0 = Real::raw(q[1] - q[0]), f1 = Real::raw(q[2] - q[1]), f2 = Real::raw(q[3] - q[2]), f3 = Real::raw(q[4] - q[3]);
    const Real a = f1 - f0, b = f2 - f1, c = f3 - f2, ta = b - a, tb = c - b, eps = S.eps;
    const Real fb = SGN > 0 ? f1 : f2, ff = SGN > 0 ? f2 : f1, s0 = SGN > 0 ? a : c, s2 = SGN > 0 ? c : a;
    const Real to = SGN > 0 ? ta : tb, ti = SGN > 0 ? tb : ta;
    const AORatios r = ao_ratios(ao_weights<SGN>(fb, ff, s0, b, s2, second_difference_energy(s0, eps), second_difference_energy(b, eps),
                                                 second_difference_energy(s2, eps), fma(0.5 * SGN, b, fb), ta + tb, tb - ta, eps, S));
    AODiffBar d;
    d.fb = d.ff = d.s0 = d.s1 = d.s2 = d.to = d.ti = 0.0;
    Real v, sl;
    edge_reverse<SGN>(r, df, alpha, vb, sb, wb, fb, ff, s0, b, s2, to, ti, S, v, sl, d);
    const double A = SGN > 0 ? d.s0.v : d.s2.v, C = SGN > 0 ? d.s2.v : d.s0.v, TA = SGN > 0 ? d.to.v : d.ti.v, TB = SGN > 0 ? d.ti.v : d.to.v;
    const double ab = A - TA, bb = d.s1.v + TA - TB, cb = C + TB;
    const double F[4] = {-ab, (SGN > 0 ? d.fb.v : d.ff.v) + ab - bb, (SGN > 0 ? d.ff.v : d.fb.v) + bb - cb, cb};
    double got[5];
    for (int i = 0; i < 5; ++i) got[i] = (i > 0 ? F[i - 1] : 0.0) - (i < 4 ? F[i] : 0.0);
    got[2] += vb;                                     // the value is taken relative to the cell average
    double worst = 0.0, scale = 1e-300;
    for (int i = 0; i < 5; ++i) scale = std::fmax(scale, std::fabs(ref[SGN > 0 ? i : 4 - i]));
    for (int i = 0; i < 5; ++i) {
        const double e = std::fabs(got[i] - ref[SGN > 0 ? i : 4 - i]) / scale;
        if (!(e <= worst)) worst = e;
    }
    return worst;
}

int main() {
    SchemeConsts S{};
    S.d[3] = 0.85; S.d[0] = 0.15 * 0.15 / 2; S.d[1] = 0.15 * 0.85; S.d[2] = S.d[0]; S.inv_d3 = 1.0 / 0.85; S.eps = 1e-6;
    std::mt19937_64 rng(7);
    auto U = [&](double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); };
    const char* names[] = {"smooth", "rough", "step", "uniform", "huge"};
    int bad = 0;
    for (int kind = 0; kind < 5; ++kind) {
        double worst = 0.0;
        for (int n = 0; n < 400; ++n) {
            double q[5];
            const double x0 = U(0, 6);
            for (int i = 0; i < 5; ++i)
                q[i] = kind == 0 ? std::sin(x0 + 0.3 * i) : kind == 1 ? U(-1, 1) : kind == 2 ? (i >= 1 + n % 4 ? 2.0 : 1.0) + 0.1 * U(-1, 1)
                     : kind == 3 ? 0.75 : 1e25 * U(-1, 1);
            const double vb = U(-1, 1), sb = U(-1, 1), wb = n % 3 == 0 ? 0.0 : U(-1, 1), al = U(0, 1);
            const bool df = n % 5 == 0;
            for (double e : {compare<+1>(q, vb, sb, wb, df, al, S), compare<-1>(q, vb, sb, wb, df, al, S)}) if (!(e <= worst)) worst = e;
        }
        const bool ok = worst <= 1e-10;
        bad += !ok;
        std::printf("%-8s %.3e %s\n", names[kind], worst, ok ? "ok" : "FAIL");
    }
    return bad ? 1 : 0;
}

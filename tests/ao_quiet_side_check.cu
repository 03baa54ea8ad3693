// Host check of the WENO-AO reconstruction beside a strong jump: cells on the quiet side must not take up rounding
// noise of the jump's size.  Stencils of smooth data of order 1 with one or two cells across a jump of 1e2 .. 1e12;
// the face line's two edges and the face side's Gauss points (line_component, face_component) against the
// sub-stencil polynomials in long double.
// With fewer than 64 roundings of quantities of the quiet data's size, values and slopes agree to 64 eps of it (plus
// as much of the reconstruction itself, where the weights let part of the jump in).
// Reverse: edge_reverse against the reverse of the sub-stencil form (weno_ao_rev), cell by cell, to 1e-10 of the
// largest adjoint (ao_reverse_check's bound), with cotangents of order 1.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include "dfgks_adjoint.cu"
using namespace dfk;

static SchemeConsts consts() {
    SchemeConsts S{};
    S.gamma = 1.4; S.gm1 = 0.4; S.K = 3.0; S.inv_K2 = 0.2;
    S.d[3] = 0.85; S.d[0] = S.d[2] = 0.15 * 0.15 / 2; S.d[1] = 0.15 * 0.85; S.inv_d3 = 1.0 / 0.85; S.eps = 1e-6;
    S.time_limiter = 1;
    return S;
}

// the AO polynomial of q about its centre: value minus the average and slope at x
typedef long double R;
static void ao(const R q[5], const SchemeConsts& S, R x, R& val, R& sl) {
    const R m2 = q[0], m1 = q[1], c = q[2], p1 = q[3], p2 = q[4];
    const R A1[4] = {0.5L * m2 - 2 * m1 + 1.5L * c, 0.5L * (p1 - m1), -1.5L * c + 2 * p1 - 0.5L * p2, (5 * (m2 - p2) - 34 * (m1 - p1)) / 48};
    const R A2[4] = {0.5L * (m2 - 2 * m1 + c), 0.5L * (m1 - 2 * c + p1), 0.5L * (c - 2 * p1 + p2), (-(m2 + p2) + 12 * (m1 + p1) - 22 * c) / 16};
    const R a3 = (-(m2 - p2) + 2 * (m1 - p1)) / 12, a4 = ((m2 + p2) - 4 * (m1 + p1) + 6 * c) / 24;
    R b[4];
    for (int k = 0; k < 4; ++k) b[k] = A1[k] * A1[k] + 13.0L / 3 * A2[k] * A2[k];
    b[3] += A1[3] * a3 / 2 + 21.0L / 5 * A2[3] * a4 + 3129.0L / 80 * a3 * a3 + 87617.0L / 140 * a4 * a4;
    const R tau = (fabsl(b[3] - b[0]) + fabsl(b[3] - b[1]) + fabsl(b[3] - b[2])) / 3;
    R z[4], sum = 1;
    for (int k = 0; k < 4; ++k) { const R r = tau / (b[k] + (R)S.eps); z[k] = r * r; sum += (R)S.d[k] * z[k]; }
    const R c3 = (1 + z[3]) / sum;
    R a1 = c3 * A1[3], a2 = c3 * A2[3];
    for (int k = 0; k < 3; ++k) { const R ck = (R)S.d[k] * (z[k] - z[3]) / sum; a1 += ck * A1[k]; a2 += ck * A2[k]; }
    val = a1 * x + a2 * (x * x - 1.0L / 12) + c3 * a3 * x * x * x + c3 * a4 * (x * x * x * x - 1.0L / 80);
    sl = a1 + 2 * a2 * x + 3 * c3 * a3 * x * x + 4 * c3 * a4 * x * x * x;
}

int main() {
    const SchemeConsts S = consts();
    std::mt19937_64 rng(3);
    auto U = [&](double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); };
    int bad = 0;
    for (double J : {1e2, 1e4, 1e6, 1e8, 1e12}) {
        double we = 0.0, wf = 0.0, wr = 0.0;
        auto worse = [](double& w, double e) { if (!(e <= w)) w = e; };
        for (int n = 0; n < 4000; ++n) {
            // six cells, smooth of order 1; the last (or first) one to three are across the jump
            double q[6];
            const double a = U(-1, 1), b = U(-0.5, 0.5), c = U(-0.1, 0.1);
            for (int i = 0; i < 6; ++i) q[i] = a + b * i + c * i * i;
            const int across = 1 + n % 3;
            const bool high = n & 4;
            for (int i = 0; i < across; ++i) q[high ? 5 - i : i] += J * U(0.5, 1.0);
            const double quiet = 1.0;
            // the face line between cells 2 and 3: both edges, of the cells on the quiet side
            Real f[5], o[4];
            for (int i = 0; i < 5; ++i) f[i] = Real::raw(q[i + 1] - q[i]);
            AOWeights L, Rr;
            line_component<false>(f, false, false, false, 0.0, 0.0, 1.0, S, o, L, Rr);
            const auto across_jump = [&](int i) { return high ? i > 5 - across : i < across; };
            for (int side = 0; side < 2; ++side) {
                if (across_jump(2 + side)) continue;
                R st[5], v, s;
                for (int i = 0; i < 5; ++i) st[i] = (R)q[side == 0 ? i : 5 - i] - (R)q[2 + side];
                ao(st, S, 0.5L, v, s);
                if (side) s = -s;
                worse(we, std::fabs((double)(o[2 * side].v - v)) / (quiet + std::fabs((double)v)));
                worse(we, std::fabs((double)(o[2 * side + 1].v - s)) / (quiet + std::fabs((double)s)));
            }
            // a face side of cells 0 .. 4 (or 1 .. 5), its Gauss points
            const int at = n % 2;
            if (!across_jump(at + 2)) {
                Real fs[4], g[4];
                for (int i = 0; i < 4; ++i) fs[i] = f[at + i];
                face_component(fs, false, false, 0.0, 1.0, S, g, NoTape{}, 0);
                R st[5], v, s;
                for (int i = 0; i < 5; ++i) st[i] = (R)q[at + i] - (R)q[at + 2];
                for (int m = 0; m < 2; ++m) {
                    ao(st, S, (m ? 1 : -1) * 0.28867513459481288225457L, v, s);
                    worse(wf, std::fabs((double)(g[m].v - v)) / (quiet + std::fabs((double)v)));
                    worse(wf, std::fabs((double)(g[2 + m].v - s)) / (quiet + std::fabs((double)s)));
                }
            }
            // the reverse of the edges, on stencils shifted so that the centre is their zero
            for (int side = 0; side < 2; ++side) {
                if (across_jump(2 + side)) continue;
                const double vb = U(-1, 1), sb = U(-1, 1);
                double sq[5], t[AT_COUNT], ref[5] = {0, 0, 0, 0, 0};
                for (int i = 0; i < 5; ++i) sq[i] = q[side == 0 ? i : 5 - i] - q[2 + side];
                const ArrayTape tp{t};
                weno_ao_t(sq, S, tp, 0);
                AOBar ob;
                ao_bar_zero(ob);
                ao_at_right_edge_vjp(vb, side ? -sb : sb, ref[2], ob);
                weno_ao_rev(tp, 0, S, ob, ref);
                // edge_reverse takes the unmirrored differences in the stencil's own order
                const Real fb = side ? f[3] : f[1], ff = f[2], s0 = side ? f[4] - f[3] : f[1] - f[0], s1 = side ? f[3] - f[2] : f[2] - f[1],
                           s2 = side ? f[2] - f[1] : f[3] - f[2];
                const Real to = side ? s0 - s1 : s1 - s0, ti = side ? s1 - s2 : s2 - s1, eps = S.eps;
                const Real w0 = second_difference_energy(s0, eps), w1 = second_difference_energy(s1, eps), w2 = second_difference_energy(s2, eps);
                AODiffBar d;
                d.fb = d.ff = d.s0 = d.s1 = d.s2 = d.to = d.ti = 0.0;
                Real v, sl;
                if (side == 0) edge_reverse<+1>(ao_ratios(ao_weights<+1>(fb, ff, s0, s1, s2, w0, w1, w2, fma(0.5, s1, fb), to + ti, ti - to, eps, S)),
                                                false, 0.0, vb, sb, 0.0, fb, ff, s0, s1, s2, to, ti, S, v, sl, d);
                else edge_reverse<-1>(ao_ratios(ao_weights<-1>(fb, ff, s0, s1, s2, w0, w1, w2, fma(-0.5, s1, fb), to + ti, to - ti, eps, S)),
                                      false, 0.0, vb, sb, 0.0, fb, ff, s0, s1, s2, to, ti, S, v, sl, d);
                // to the five cells, in the stencil's own order (differences of the mirrored one change sign)
                const double sg = side ? -1.0 : 1.0;
                const double s0b = d.s0.v - sg * d.to.v, s1b = d.s1.v + sg * (d.to.v - d.ti.v), s2b = d.s2.v + sg * d.ti.v;
                const double F[4] = {-s0b, sg * d.fb.v + s0b - s1b, sg * d.ff.v + s1b - s2b, s2b};
                double scale = 0.0;
                for (double x : ref) scale = std::fmax(scale, std::fabs(x));
                for (int i = 0; i < 5; ++i) {
                    const double got = (i > 0 ? F[i - 1] : 0.0) - (i < 4 ? F[i] : 0.0) + (i == 2 ? vb : 0.0);
                    worse(wr, std::fabs(got - ref[i]) / scale);
                }
            }
        }
        const double eps = 0x1p-52;
        const bool ok = we <= 64 * eps && wf <= 64 * eps && wr <= 1e-10;
        bad += !ok;
        std::printf("jump %.0e: edges %.1e, Gauss points %.1e, reverse %.1e %s\n", J, we, wf, wr, ok ? "ok" : "FAIL");
    }
    return bad ? 1 : 0;
}

// Host check: the WENO-AO reconstruction in undivided differences (ao_weights and its evaluations) against
// the sub-stencil polynomials of Sect. 3.1 in long double, over stencils of all magnitudes.  (In long double,
// because on constant data at 1e14 and above the polynomials' coefficients in double are rounding noise that
// counts against the smoothness epsilon; the differences are exact zeros there.)  With fewer than 64
// roundings the values and slopes agree to 128 eps max|q|.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "dfgks_device.cuh"
using namespace dfk;

static unsigned long long seed = 12345;
static double U() { seed = seed * 6364136223846793005ULL + 1442695040888963407ULL; return 2.0 * (double)(seed >> 11) * 0x1p-53 - 1.0; }

// value and slope at xi = 1/2, values and slopes at -/+ sqrt(3)/6, limiter fraction
static void reference(const double q[5], const SchemeConsts& S, double v[6], double& lim) {
    typedef long double R;
    const R m2 = q[0], m1 = q[1], c = q[2], p1 = q[3], p2 = q[4];
    const R A1[4] = {0.5L * m2 - 2 * m1 + 1.5L * c, 0.5L * (p1 - m1), -1.5L * c + 2 * p1 - 0.5L * p2,
                     (5 * (m2 - p2) - 34 * (m1 - p1)) / 48};
    const R A2[4] = {0.5L * (m2 - 2 * m1 + c), 0.5L * (m1 - 2 * c + p1), 0.5L * (c - 2 * p1 + p2),
                     (-(m2 + p2) + 12 * (m1 + p1) - 22 * c) / 16};
    const R a3 = (-(m2 - p2) + 2 * (m1 - p1)) / 12, a4 = ((m2 + p2) - 4 * (m1 + p1) + 6 * c) / 24;
    R b[4];
    for (int k = 0; k < 4; ++k) b[k] = A1[k] * A1[k] + 13.0L / 3 * A2[k] * A2[k];
    b[3] += A1[3] * a3 / 2 + 21.0L / 5 * A2[3] * a4 + 3129.0L / 80 * a3 * a3 + 87617.0L / 140 * a4 * a4;
    const R tau = (fabsl(b[3] - b[0]) + fabsl(b[3] - b[1]) + fabsl(b[3] - b[2])) / 3;
    R x[4], sum = 0, hi = 0, lo = 0;
    for (int k = 0; k < 4; ++k) {
        const R r = tau / (b[k] + (R)S.eps);
        x[k] = 1 + r * r;
        sum += (R)S.d[k] * x[k];
        hi = k ? std::max(hi, x[k]) : x[k];
        lo = k ? std::min(lo, x[k]) : x[k];
    }
    lim = (double)(2 * lo / (hi + lo));
    const R c3 = x[3] / sum;
    R a1 = c3 * A1[3], a2 = c3 * A2[3];
    for (int k = 0; k < 3; ++k) { const R ck = (R)S.d[k] * x[k] / sum - c3 * (R)S.d[k]; a1 += ck * A1[k]; a2 += ck * A2[k]; }
    const R g = 0.28867513459481288225457L;
    auto at = [&](R xi, double& val, double& sl) {
        val = (double)(c + a1 * xi + a2 * (xi * xi - 1.0L / 12) + c3 * a3 * xi * xi * xi + c3 * a4 * (xi * xi * xi * xi - 1.0L / 80));
        sl = (double)(a1 + 2 * a2 * xi + 3 * c3 * a3 * xi * xi + 4 * c3 * a4 * xi * xi * xi);
    };
    at(0.5L, v[0], v[1]);
    at(-g, v[2], v[4]);
    at(g, v[3], v[5]);
}

int main(int argc, char** argv) {
    if (argc != 2) return 2;
    const double scale = pow(10.0, atof(argv[1]));
    SchemeConsts S;
    S.d[3] = 0.85; S.d[0] = S.d[2] = 0.15 * 0.15 / 2.0; S.d[1] = 0.15 * 0.85; S.inv_d3 = 1.0 / 0.85; S.eps = 1e-6;
    double worst = 0.0, wlim = 0.0;
    for (int n = 0; n < 20000; ++n) {
        double q[5];
        const int kind = n % 4;      // rough, smooth, a jump, constant
        const double c = U(), a = U(), j = U();
        for (int i = 0; i < 5; ++i)
            q[i] = scale * (kind == 0 ? U() : kind == 1 ? c + 0.01 * a * i + 1e-4 * j * i * i + 1e-6 * U() : kind == 2 ? (i < 1 + n % 5 ? c : j) : c);
        double big = 0.0;
        for (double x : q) big = std::max(big, fabs(x));
        double v[6], w[6], lim;
        Real wr[4];
        reference(q, S, v, lim);
        for (int mir = 0; mir < 2; ++mir) {          // the stencil given as it is, and as the mirror of its reverse
            double p[5];
            for (int i = 0; i < 5; ++i) p[i] = mir ? q[4 - i] : q[i];
            Real f[4], s[3];
            for (int i = 0; i < 4; ++i) f[i] = p[i + 1] - p[i];
            for (int i = 0; i < 3; ++i) s[i] = f[i + 1] - f[i];
            const Real t1 = s[1] - s[0], t2 = s[2] - s[1];
            Real e[3];
            for (int i = 0; i < 3; ++i) e[i] = second_difference_energy(s[i], S.eps);
            if (!mir) {
                const Real a11 = fma(0.5, s[1], f[1]), T = t1 + t2, Uu = t2 - t1;
                const AOWeights A = ao_weights<+1>(f[1], f[2], s[0], s[1], s[2], e[0], e[1], e[2], a11, T, Uu, S.eps, S);
                ao_diff_at_gauss(A, a11, s[1], t1, t2, T, Uu, S, wr, wr + 2);
                for (int i = 0; i < 4; ++i) w[2 + i] = wr[i].v;
                for (int i = 0; i < 4; ++i) worst = std::max(worst, fabs(w[2 + i] + (i < 2 ? q[2] : 0.0) - v[2 + i]) / big);
                const double iv = ao_inverse_sum(A).v, y = Real(A.y0 * t1).v;
                const double val = 0.5 * f[2].v - s[1].v / 6.0 - iv * (S.d[0] / 3.0 * (y + 0.5 * t2.v * A.y2.v) + A.x3.v * (t1.v / 30.0 + t2.v / 20.0));
                worst = std::max(worst, fabs(q[2] + val - v[0]) / big);
                worst = std::max(worst, fabs(f[2].v - iv * (S.d[0] * y + A.x3.v * t2.v / 12.0) - v[1]) / big);
                wlim = std::max(wlim, fabs(2.0 * A.xmin.v / (A.xmax.v + A.xmin.v) - lim));
            } else {                                  // cell p[2], its right edge is q's left one
                const Real a11 = fma(-0.5, s[1], f[2]);
                const AOWeights A = ao_weights<-1>(f[2], f[1], s[2], s[1], s[0], e[2], e[1], e[0], a11, t1 + t2, t2 - t1, S.eps, S);
                const double iv = ao_inverse_sum(A).v, y = Real(A.y0 * t2).v;
                const double val = -0.5 * f[1].v - s[1].v / 6.0 + iv * (S.d[0] / 3.0 * (y + 0.5 * t1.v * A.y2.v) + A.x3.v * (t2.v / 30.0 + t1.v / 20.0));
                worst = std::max(worst, fabs(q[2] + val - v[0]) / big);
                worst = std::max(worst, fabs(-(f[1].v - iv * (S.d[0] * y + A.x3.v * t1.v / 12.0)) - v[1]) / big);
                wlim = std::max(wlim, fabs(2.0 * A.xmin.v / (A.xmax.v + A.xmin.v) - lim));
            }
        }
    }
    printf("scale %g: worst %.3e limiter %.3e\n", scale, worst, wlim);
    return worst <= 128 * 0x1p-52 && wlim <= 1e-9 ? 0 : 1;
}

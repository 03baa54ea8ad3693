// Host check of the reverses that the kernels call for the face basis and the projections of differences:
// project_diff_rev, back_project_diff_T with back_project_diff_basis_rev, diff_basis_rev and make_basis_rev, each
// chain from its outputs down to the two cell states, against central differences of its forward.
// Step 1e-6 of the argument: truncation 1e-12 and rounding 1e-10 relative, on adjoints of at least a thousandth
// of the largest one: 1e-6.
#include <cmath>
#include <cstdio>
#include <random>
#include "dfgks_adjoint.cuh"
using namespace dfk;

static std::mt19937_64 rng(2024);
static double U(double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); }
static void state(double W[4]) {
    const double rho = U(0.3, 2.0), u = U(-1, 1), v = U(-1, 1), p = U(0.2, 2.0);
    W[0] = rho; W[1] = rho * u; W[2] = rho * v; W[3] = p / 0.4 + 0.5 * rho * (u * u + v * v);
}
static void real4(const double* x, Real r[4]) { for (int i = 0; i < 4; ++i) r[i] = Real::raw(x[i]); }

// x = (left state, right state, vector); forward or back projection of the vector in their basis
static void forward(bool back, const double* x, const SchemeConsts& S, double* y) {
    const DiffBasis D = diff_basis(make_basis(x, x + 4, S));
    Real w[4], q[4];
    real4(x + 8, w);
    if (back) back_project_diff(D, w, q);
    else project_diff(D, w, q);
    for (int i = 0; i < 4; ++i) y[i] = q[i].v;
}
static void reverse(bool back, const double* x, const SchemeConsts& S, const double* yb, double* xb) {
    const CharBasis B = make_basis(x, x + 4, S);
    const DiffBasis D = diff_basis(B);
    Real w[4], q[4], wb[4], g[4];
    real4(x + 8, w);
    real4(yb, q);
    DiffBasisBar b;
    zero(b);
    if (back) {
        back_project_diff_T(D, q, wb);
        back_project_diff_basis_rev(w, q, b);
    } else {
        project_diff_rev(D, w, q, wb, b);
    }
    make_basis_rev(B, Real::raw(0.5 * (x[0] + x[4])), diff_basis_rev(D, b), S, g);
    for (int i = 0; i < 4; ++i) { xb[i] = xb[4 + i] = g[i].v; xb[8 + i] = wb[i].v; }
}

int main() {
    SchemeConsts S{};
    S.gamma = 1.4; S.gm1 = 0.4; S.K = 3.0; S.inv_K2 = 0.2; S.r2g = sqrt(2.0 / 1.4);
    int bad = 0;
    for (int back = 0; back < 2; ++back) {
        double worst = 0.0;
        for (int t = 0; t < 50; ++t) {
            double x[12], yb[4], xb[12], y1[4], y2[4], scale = 1e-30;
            state(x); state(x + 4);
            for (int i = 0; i < 4; ++i) { x[8 + i] = U(-1, 1); yb[i] = U(-1, 1); }
            reverse(back, x, S, yb, xb);
            for (double v : xb) scale = std::fmax(scale, std::fabs(v));
            for (int i = 0; i < 12; ++i) {
                const double h = 1e-6 * std::fmax(1.0, std::fabs(x[i])), keep = x[i];
                x[i] = keep + h; forward(back, x, S, y1);
                x[i] = keep - h; forward(back, x, S, y2);
                x[i] = keep;
                double fd = 0.0;
                for (int k = 0; k < 4; ++k) fd += yb[k] * (y1[k] - y2[k]) / (2 * h);
                const double e = std::fabs(fd - xb[i]) / std::fmax(std::fabs(fd), 1e-3 * scale);
                if (!(e <= worst)) worst = e;
            }
        }
        bad += !(worst <= 1e-6);
        std::printf("%s %.3e %s\n", back ? "back_project_diff" : "project_diff", worst, worst <= 1e-6 ? "ok" : "FAIL");
    }
    return bad ? 1 : 0;
}

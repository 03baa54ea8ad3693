// Host check that the taped sweeps stay inside the tapes the library lays out: both directions' ratio tapes (8
// reconstructions per face line, 4 per face side, RT_COUNT planes each) one after the other, both directions' GKS
// tapes likewise, all of exactly that size with guards around them.  A direction's forward may write its own tapes
// only; the reverse that reads them gives what the reverse that evaluates everything again gives.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <type_traits>
#include <vector>
#include "dfgks_adjoint.cu"
using namespace dfk;

static const double kGuard = -123456.789;

struct Case { int nx, ny, bc, flux, limiter; };

static int run(const Case& c) {
    Mesh m;
    m.nx = c.nx; m.ny = c.ny; m.P = (c.nx + 2 * G + 3) & ~3; m.NYg = c.ny + 2 * G; m.plane = (long long)m.P * m.NYg;
    m.dx = 1.0 / c.nx; m.dy = 0.8 / c.ny; m.rdx = 1.0 / m.dx; m.rdy = 1.0 / m.dy;
    for (int& b : m.bc) b = c.bc;
    m.dt_rule = 0; m.gi0 = 0; m.gj0 = 0; m.gnx = c.nx;
    SchemeConsts S{};
    S.gamma = 1.4; S.gm1 = 0.4; S.K = 3.0; S.inv_K2 = 0.2; S.r2g = sqrt(2.0 / 1.4);
    S.d[3] = 0.85; S.d[0] = 0.15 * 0.15 / 2; S.d[1] = 0.15 * 0.85; S.d[2] = S.d[0]; S.inv_d3 = 1.0 / 0.85;
    S.eps = 1e-6; S.alpha_thres = 0.5; S.C1 = 0.01; S.C2 = 5.0;
    S.time_limiter = c.limiter; S.tau_reading = 0; S.gp_fallback = 1; S.df_states = 0;
    const long long nfx = (long long)(m.nx + 1) * m.ny, nfy = (long long)(m.ny + 1) * m.nx;
    const long long nlx = (long long)(m.nx + 1) * (m.ny + 4), nly = (long long)(m.ny + 1) * (m.nx + 4);
    SweepBuffers B;
    B.line_stride = (std::max(nlx, nly) + 3) & ~3LL;
    B.gp_stride = (2 * std::max(nfx, nfy) + 3) & ~3LL;
    B.flux_stride[0] = (2 * nfx + 3) & ~3LL; B.flux_stride[1] = (2 * nfy + 3) & ~3LL;
    std::vector<double> W(4 * m.plane, 1.0), A(m.plane, 1.0), lines(LR_COUNT * B.line_stride), gp(GP_COUNT * B.gp_stride),
        fr0(FR_COUNT * B.flux_stride[0]), fr1(FR_COUNT * B.flux_stride[1]), lb(LR_COUNT * B.line_stride), gb(GP_COUNT * B.gp_stride);
    B.lines = lines.data(); B.gp = gp.data(); B.flux[0] = fr0.data(); B.flux[1] = fr1.data();
    std::mt19937_64 rng(17);
    auto U = [&](double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); };
    const long long N = (long long)c.nx * c.ny;
    std::vector<double> bars(12 * N);
    for (double& b : bars) b = U(-1, 1);
    for (int j = 0; j < m.ny; ++j) for (int i = 0; i < m.nx; ++i) {
        const long long g = gid(m, i, j);
        const double rho = U(0.5, 1.5), u = U(-0.5, 0.5), v = U(-0.5, 0.5), p = U(0.5, 1.5);
        W[g] = rho; W[m.plane + g] = rho * u; W[2 * m.plane + g] = rho * v; W[3 * m.plane + g] = p / 0.4 + 0.5 * rho * (u * u + v * v);
        A[g] = U(0, 1);
    }
    for (int j = 0; j < m.ny; ++j) for (int g = 0; g < 2 * G; ++g) ghost_x_body(m, W.data(), A.data(), g, j);
    for (int g = 0; g < 2 * G; ++g) for (int i = -G; i < m.nx + G; ++i) ghost_y_body(m, W.data(), A.data(), i, g);
    const AdjointArgs a = {bars.data(), bars.data() + 4 * N, bars.data() + 8 * N};
    const double dt = 0.002;

    const long long nr = 8 * RT_COUNT * B.line_stride + 4 * RT_COUNT * B.gp_stride, nk = TG_COUNT * std::max(B.flux_stride[0], B.flux_stride[1]);
    const long long pad = 4096;
    std::vector<double> arena(3 * pad + 2 * nr + 2 * nk, kGuard);
    double* const ratios = arena.data() + pad;
    double* const gks = ratios + 2 * nr + pad;
    int bad = 0;
    auto sweep = [&](auto dirc, bool taped, std::vector<double>& out) {
        constexpr int DIR = decltype(dirc)::value;
        double* lt = taped ? ratios + DIR * nr : nullptr;
        double* ft = taped ? lt + 8 * RT_COUNT * B.line_stride : nullptr;
        double* kt = taped && c.flux == 0 ? gks + DIR * nk : nullptr;
        const std::vector<double> before = arena;
        auto grid = [&](int lx, int ly, auto body) {                   // the kernels' grids, padded tail included
            const long long n = (long long)sweep_blocks(lx, ly) * kSweepThreads;
            for (long long i = 0; i < n; ++i) body((int)(i % lx), (int)(i / lx));
        };
        const int lx = lines_lx<DIR>(m), ly = lines_ly<DIR>(m), fx = faces_lx<DIR>(m), fy = faces_ly<DIR>(m);
        grid(lx, ly, [&](int x, int y) {
            if (lt) lines_body<DIR, true>(m, S, W.data(), A.data(), B.lines, B.line_stride, x, y, lt);
            else lines_body<DIR>(m, S, W.data(), A.data(), B.lines, B.line_stride, x, y);
        });
        for (int z = 0; z < 2; ++z) grid(fx, fy, [&](int x, int y) {
            int nfb;
            if (ft) faces_body<DIR, true>(m, S, W.data(), A.data(), B.lines, B.line_stride, B.gp, B.gp_stride, x, y, z, nfb, ft);
            else faces_body<DIR>(m, S, W.data(), A.data(), B.lines, B.line_stride, B.gp, B.gp_stride, x, y, z, nfb);
        });
        for (int z = 0; z < 2; ++z) grid(fx, fy, [&](int x, int y) {
            if (kt) flux_body<DIR, 0, false, true>(m, S, B.lines, B.line_stride, B.gp, B.gp_stride, B.flux[DIR], B.flux_stride[DIR], dt, x, y, z, kt);
            else if (c.flux == 0) flux_body<DIR, 0, false>(m, S, B.lines, B.line_stride, B.gp, B.gp_stride, B.flux[DIR], B.flux_stride[DIR], dt, x, y, z);
            else flux_body<DIR, 1, false>(m, S, B.lines, B.line_stride, B.gp, B.gp_stride, B.flux[DIR], B.flux_stride[DIR], dt, x, y, z);
        });
        for (size_t q = 0; q < arena.size(); ++q) {
            const double* p = arena.data() + q;
            const bool own = (lt && p >= lt && p < lt + nr) || (kt && p >= kt && p < kt + TG_COUNT * B.flux_stride[DIR]);
            if (!own && memcmp(p, &before[q], sizeof(double)) != 0) ++bad;
        }
        std::fill(lb.begin(), lb.end(), 0.0);
        std::fill(gb.begin(), gb.end(), 0.0);
        const std::vector<double> tapes = arena;
        for (int z = 0; z < 2; ++z) grid(fx, fy, [&](int x, int y) {
            if (kt) ka_flux_body<DIR, 0, true>(m, S, a, B.gp, B.gp_stride, B.flux[DIR], B.flux_stride[DIR], dt, lb.data(), B.line_stride, gb.data(), x, y, z, kt);
            else if (c.flux == 0) ka_flux_body<DIR, 0>(m, S, a, B.gp, B.gp_stride, B.flux[DIR], B.flux_stride[DIR], dt, lb.data(), B.line_stride, gb.data(), x, y, z);
            else ka_flux_body<DIR, 1>(m, S, a, B.gp, B.gp_stride, B.flux[DIR], B.flux_stride[DIR], dt, lb.data(), B.line_stride, gb.data(), x, y, z);
        });
        for (int z = 0; z < 2; ++z) grid(fx, fy, [&](int x, int y) {
            if (ft) ka_faces_body<DIR, true>(m, S, A.data(), B.lines, B.line_stride, B.gp, gb.data(), B.gp_stride, lb.data(), out.data(), x, y, z, ft);
            else ka_faces_body<DIR>(m, S, A.data(), B.lines, B.line_stride, B.gp, gb.data(), B.gp_stride, lb.data(), out.data(), x, y, z);
        });
        grid(lx, ly, [&](int x, int y) {
            if (lt) ka_lines_body<DIR, true>(m, S, W.data(), A.data(), B.lines, lb.data(), B.line_stride, out.data(), x, y, lt);
            else ka_lines_body<DIR>(m, S, W.data(), A.data(), B.lines, lb.data(), B.line_stride, out.data(), x, y);
        });
        if (memcmp(tapes.data(), arena.data(), arena.size() * sizeof(double)) != 0) ++bad;      // the reverse only reads them
    };
    std::vector<double> taped(4 * m.plane, 0.0), again(4 * m.plane, 0.0);
    sweep(std::integral_constant<int, 0>(), true, taped);
    sweep(std::integral_constant<int, 1>(), true, taped);
    sweep(std::integral_constant<int, 0>(), false, again);
    sweep(std::integral_constant<int, 1>(), false, again);
    double scale = 0.0, err = 0.0;
    for (size_t q = 0; q < again.size(); ++q) scale = std::fmax(scale, std::fabs(again[q]));
    for (size_t q = 0; q < again.size(); ++q) { const double e = std::fabs(taped[q] - again[q]) / scale; if (!(e <= err)) err = e; }
    const bool ok = bad == 0 && err <= 1e-12;
    std::printf("%d x %d bc %d flux %d: %d values outside their tape, taped against evaluated again %.2e %s\n", c.nx, c.ny, c.bc, c.flux, bad, err, ok ? "ok" : "FAIL");
    return ok ? 0 : 1;
}

int main() {
    int bad = 0;
    // GKS and L-F, odd sides, one row, one column, one cell, the smallest periodic and walled meshes
    for (const Case& c : {Case{13, 9, 0, 0, 1}, Case{9, 14, 1, 1, 1}, Case{11, 7, 2, 0, 0}, Case{1, 9, 1, 0, 1}, Case{12, 1, 1, 0, 1},
                          Case{1, 1, 1, 0, 1}, Case{3, 3, 0, 1, 0}, Case{3, 3, 2, 0, 1}}) bad += run(c);
    return bad ? 1 : 0;
}

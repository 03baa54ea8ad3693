// Host check of lf_flux_vjp where a normal velocity is zero: |U| has slope +1 at U = 0 whatever the zero's sign
// (the rule of dfgks_adjoint.cuh), so the adjoints of a state with momentum -0 are those of the state with +0.
// Both sides of the face, at rest and with tangential velocity, each side's wave speed being the larger one.
#include <cmath>
#include <cstdio>
#include "dfgks_adjoint.cuh"
using namespace dfk;

int main() {
    SchemeConsts S{};
    S.gamma = 1.4; S.gm1 = 0.4; S.K = 3.0; S.inv_K2 = 0.2; S.r2g = sqrt(2.0 / 1.4);
    int bad = 0, n = 0;
    for (int side = 0; side < 2; ++side)
        for (int other = 0; other < 2; ++other)              // the other side faster or slower
            for (double v : {0.0, 0.3}) {
                GPStateBar b[2][2];
                for (int minus = 0; minus < 2; ++minus) {
                    GPState P[2];
                    for (int s = 0; s < 2; ++s) {
                        const double rho = s == 0 ? 1.0 : 0.8, p = s == side ? 1.0 : (other ? 2.0 : 0.25);
                        const double u = s == side ? 0.0 : 0.4;
                        P[s].W[0] = rho; P[s].W[1] = rho * u; P[s].W[2] = rho * v;
                        P[s].W[3] = p / S.gm1 + 0.5 * rho * (u * u + v * v);
                        for (int k = 0; k < 4; ++k) { P[s].Wn[k] = 0.1 * (k + 1) - 0.3 * s; P[s].Wt[k] = 0.2 - 0.05 * k + 0.1 * s; }
                    }
                    P[side].W[1] = minus ? -0.0 : 0.0;
                    const double Fb[4] = {0.7, -0.4, 0.2, 0.9}, dFb[4] = {-0.3, 0.6, 0.5, -0.8};
                    lf_flux_vjp(P[0], P[1], S, Fb, dFb, b[minus][0], b[minus][1]);
                }
                for (int s = 0; s < 2; ++s)
                    for (int k = 0; k < 4; ++k) {
                        n += 3;
                        bad += b[0][s].W[k] != b[1][s].W[k];
                        bad += b[0][s].Wn[k] != b[1][s].Wn[k];
                        bad += b[0][s].Wt[k] != b[1][s].Wt[k];
                    }
                // and the slope is +1: a difference quotient towards positive velocities, where |U| = U
                if (!other) {                                // this side's wave speed is the larger one
                    double F1[4], D1[4], F0[4], D0[4];
                    GPState P[2];
                    for (int s = 0; s < 2; ++s) {
                        const double rho = s == 0 ? 1.0 : 0.8, p = s == side ? 1.0 : 0.25, u = s == side ? 0.0 : 0.4;
                        P[s].W[0] = rho; P[s].W[1] = rho * u; P[s].W[2] = rho * v;
                        P[s].W[3] = p / S.gm1 + 0.5 * rho * (u * u + v * v);
                        for (int k = 0; k < 4; ++k) { P[s].Wn[k] = 0.1 * (k + 1) - 0.3 * s; P[s].Wt[k] = 0.2 - 0.05 * k + 0.1 * s; }
                    }
                    const double Fb[4] = {0.7, -0.4, 0.2, 0.9}, dFb[4] = {-0.3, 0.6, 0.5, -0.8}, h = 1e-7;
                    lf_flux(P[0], P[1], S, F0, D0);
                    P[side].W[1] = h;
                    lf_flux(P[0], P[1], S, F1, D1);
                    double fd = 0.0;
                    for (int k = 0; k < 4; ++k) fd += (Fb[k] * (F1[k] - F0[k]) + dFb[k] * (D1[k] - D0[k])) / h;
                    // one-sided: error h/2 times a second derivative of order 10, and 1e-16/h of rounding
                    for (int minus = 0; minus < 2; ++minus) { ++n; bad += !(std::fabs(fd - b[minus][side].W[1]) <= 1e-5); }
                }
            }
    std::printf("%d of %d comparisons differ\n", bad, n);
    return bad ? 1 : 0;
}

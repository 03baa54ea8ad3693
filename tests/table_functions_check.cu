// Host check of the flux's table-driven functions against long double: exp(-y) for y < 700 and the pair
// exp(-x^2), erfc(|x|)/2 for all x, at table nodes, interval edges, the switch to the library functions, and
// random points.  exp(-y) is one rounding of T p + T after a polynomial in a reduced argument: 2 ulp is its
// bound; x^2 is rounded before it is used, which adds x^2 / 2 ulp, and erfcx adds two roundings and its fit's.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include "dfgks_device.cuh"
using namespace dfk;

int main() {
    const double eps = 0x1p-52;
    double w1 = 0, w2 = 0, w3 = 0;
    auto one = [&](double y) {
        const long double e = expl(-(long double)y);
        if (y < 700.0) w1 = std::max(w1, (double)(fabsl((long double)exp_neg(y).v - e) / e) / eps);
    };
    auto two = [&](double x) {
        Real G, t;
        gauss_erfc(x, G, t);
        const long double X = x, g = expl(-X * X), h = 0.5L * erfcl(fabsl(X));
        if (g < 1e-290L || h < 1e-290L) return;
        const double allow = 1.0 + 0.5 * x * x;
        w2 = std::max(w2, (double)(fabsl((long double)G.v - g) / g) / eps / allow);
        w3 = std::max(w3, (double)(fabsl((long double)t.v - h) / h) / eps / allow);
    };
    unsigned long long s = 99;
    auto U = [&]() { s = s * 6364136223846793005ULL + 1442695040888963407ULL; return (double)(s >> 11) * 0x1p-53; };
    for (int i = 0; i < 200000; ++i) { one(700.0 * U()); one(60.0 * U()); one(U()); two(14.0 * (U() - 0.5)); two(2.0 * (U() - 0.5)); }
    for (int i = 0; i <= 448; ++i)
        for (double d : {0.0, 1e-9, -1e-9}) { two(i / 64.0 + d); two(-i / 64.0 + d); one(std::max(0.0, (2 * i + 1) * 0.005415212346633780 + d)); }
    for (double x : {0.0, -0.0, 1e-300, 1e-17, 5.9999999999, 6.0, 6.0000000001, 25.0}) { two(x); two(-x); }
    one(0.0); one(699.9999999999);
    const bool tail = exp_neg(1e5).v == 0.0 && exp_neg(INFINITY).v == 0.0 && std::isnan(exp_neg(NAN).v);
    Real G, t;
    gauss_erfc(NAN, G, t);
    const bool nan = std::isnan(G.v) && std::isnan(t.v);
    printf("exp(-y) %.2f ulp; exp(-x^2) %.2f, erfc(|x|)/2 %.2f of (1 + x^2/2) ulp; tail %d nan %d\n", w1, w2, w3, tail, nan);
    return w1 <= 2.0 && w2 <= 2.0 && w3 <= 4.0 && tail && nan ? 0 : 1;
}

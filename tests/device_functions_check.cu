// The device's own forms of rcp, exp_neg and gauss_erfc (the host build of the header divides, and reads the tables
// through other pointers) against long double: at both ends of their ranges, at the switches between their forms, at
// table nodes and interval edges, and at random arguments.  Limits, in units of 2^-52 of the value unless said:
//   rcp          0.51 ulp of the result (one rounding; the step before it leaves 2^-60)
//   exp_neg      1.2 (one rounding of T p + T, p of a reduced argument)
//   exp(-x^2)    the same, and x^2's rounding, x^2 / 2
//   erfc(|x|)/2  that, the product's rounding 0.5, and 1.5 for erfcx
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>
#include "dfgks_device.cuh"
using namespace dfk;

__global__ void k_rcp(const double* x, double* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = rcp(Real::raw(x[i])).v;
}
__global__ void k_exp(const double* x, double* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = exp_neg(Real::raw(x[i])).v;
}
__global__ void k_gauss(const double* x, double* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    Real g, t;
    gauss_erfc(Real::raw(x[i]), g, t);
    y[i] = g.v;
    y[n + i] = t.v;
}

#define CK(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) { std::printf("%s\n", cudaGetErrorString(e_)); return 2; } } while (0)

int main() {
    unsigned long long s = 4242;
    auto U = [&]() { s = s * 6364136223846793005ULL + 1442695040888963407ULL; return (double)(s >> 11) * 0x1p-53; };
    std::vector<double> a, b, c;
    for (int i = 0; i < 400000; ++i) a.push_back((1.0 + U()) * std::pow(2.0, (int)(1980 * U()) - 990));     // 1e-298 .. 1e298
    for (int i = 0; i < 200000; ++i) a.push_back(0.5 + 1.5 * U());
    for (double m : {1e-300, 2e-300, 0.5, 1.0, 2.0, 1e299, 1e300})
        for (int k = -3; k <= 3; ++k) { const double x = m * (1.0 + k * 0x1p-52); if (x >= 1e-300 && x <= 1e300) a.push_back(x); }
    for (double& x : a) if (U() < 0.3) x = -x;
    for (int i = 0; i < 200000; ++i) { b.push_back(700.0 * U()); b.push_back(60.0 * U()); b.push_back(U()); }
    for (int n = 0; n <= 64640; n += 7)                                  // multiples of ln2/128, nodes and edges alike
        for (double d : {0.0, 1e-9, -1e-9}) b.push_back(std::min(699.999, std::max(0.0, n * 0.005415212348514945 + d)));
    for (double y : {0.0, 1e-300, 1e-17, 699.9999999999, 700.0, 700.0000000001, 708.0, 740.0, 1e5}) b.push_back(y);
    for (int i = 0; i < 300000; ++i) { c.push_back(14.0 * (U() - 0.5)); c.push_back(2.0 * (U() - 0.5)); }
    for (int i = 0; i <= 448; ++i)
        for (double d : {0.0, 1e-9, -1e-9}) { c.push_back(i / 64.0 + d); c.push_back(-i / 64.0 - d); }
    for (double x : {0.0, -0.0, 1e-300, 1e-17, 5.9999999999, 6.0, 6.0000000001, 25.0, 27.5}) { c.push_back(x); c.push_back(-x); }

    double *dx, *dy;
    const size_t most = std::max(a.size(), std::max(b.size(), c.size()));
    CK(cudaMalloc((void**)&dx, most * sizeof(double)));
    CK(cudaMalloc((void**)&dy, 2 * most * sizeof(double)));
    std::vector<double> y(2 * most);
    auto run = [&](void (*k)(const double*, double*, int), const std::vector<double>& x, int per) {
        const int n = (int)x.size();
        cudaError_t e = cudaMemcpy(dx, x.data(), n * sizeof(double), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return e;
        k<<<(n + 127) / 128, 128>>>(dx, dy, n);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        return cudaMemcpy(y.data(), dy, (size_t)per * n * sizeof(double), cudaMemcpyDeviceToHost);
    };
    const long double eps = 0x1p-52L;
    double wr = 0, we = 0, wg = 0, wt = 0;
    bool tails = true;
    auto worse = [](double& w, long double e) { if (!(e <= w)) w = (double)e; };
    CK(run(k_rcp, a, 1));
    for (size_t i = 0; i < a.size(); ++i) {
        const long double e = 1.0L / a[i];
        worse(wr, fabsl(y[i] - e) / std::ldexp(1.0, std::ilogb((double)fabsl(e)) - 52));
    }
    CK(run(k_exp, b, 1));
    for (size_t i = 0; i < b.size(); ++i) {
        const long double e = expl(-(long double)b[i]);
        if (b[i] < 700.0) worse(we, fabsl(y[i] - e) / e / eps);
        else if (e >= 1e-307L) tails = tails && fabsl(y[i] - e) / e <= 4 * eps;     // the library's exp
        else tails = tails && y[i] >= 0.0 && y[i] <= 1e-306;
    }
    CK(run(k_gauss, c, 2));
    const size_t n = c.size();
    for (size_t i = 0; i < n; ++i) {
        const long double X = c[i], g = expl(-X * X), h = 0.5L * erfcl(fabsl(X)), sq = 0.5L * X * X;
        if (fabsl(X) >= 6.0L) {                                          // the library's functions, t below 1e-17
            tails = tails && fabsl(y[i] - g) <= (4 + sq) * eps * g + 1e-300L && fabsl(y[n + i] - h) <= (16 + sq) * eps * h + 1e-300L;
            continue;
        }
        worse(wg, fabsl(y[i] - g) / g / eps - sq);
        worse(wt, fabsl(y[n + i] - h) / h / eps - sq);
    }
    cudaFree(dx);
    cudaFree(dy);
    const bool ok = wr <= 0.51 && we <= 1.2 && wg <= 1.2 && wt <= 3.2 && tails;
    std::printf("rcp %.4f ulp; exp_neg %.3f, exp(-x^2) %.3f + x^2/2, erfc(|x|)/2 %.3f + x^2/2 of 2^-52; tails %d %s\n", wr, we, wg, wt,
                (int)tails, ok ? "ok" : "FAIL");
    return ok ? 0 : 1;
}

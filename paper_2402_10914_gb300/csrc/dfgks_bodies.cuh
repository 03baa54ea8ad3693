// dfgks_bodies.cuh -- per-thread bodies of the step kernels (one face line, face side, Gauss point,
// cell or ghost cell), shared by the single-problem kernels (dfgks_kernels.cu) and the batched
// kernels (dfgks_batch.cu), so both run exactly the same arithmetic.  The bodies are also
// host-callable, so a test can run the GPU path's per-thread arithmetic on the CPU.
#pragma once
#include <float.h>
#include "dfgks_internal.h"

namespace dfk {

DFK_HD int ghost_src(int k, int n, int lo, int hi, bool& mir) {
    mir = false;
    if (k < 0) {
        if (lo == 0) return k + n;
        if (lo == 1) return 0;
        mir = true; return -1 - k;
    }
    if (k >= n) {
        if (hi == 0) return k - n;
        if (hi == 1) return n - 1;
        mir = true; return 2 * n - 1 - k;
    }
    return k;
}

template <int DIR>
struct Geo {
    int nn, nt;                  // cells along normal / tangential
    double dn, dtan;             // cell sizes along normal / tangential
    double idn, idtan;           // their reciprocals
    DFK_HD Geo(const Mesh& m) {
        nn = DIR == 0 ? m.nx : m.ny;
        nt = DIR == 0 ? m.ny : m.nx;
        dn = DIR == 0 ? m.dx : m.dy;
        dtan = DIR == 0 ? m.dy : m.dx;
        idn = DIR == 0 ? m.rdx : m.rdy;
        idtan = DIR == 0 ? m.rdy : m.rdx;
    }
    static constexpr int sigma = DIR == 0 ? 1 : -1;
    DFK_HD long long cell(const Mesh& m, int n, int t) const {
        return DIR == 0 ? gid(m, n, t) : gid(m, t, n);
    }
    // line (f, t), t in [-2, nt+2): contiguous along the thread-x direction
    DFK_HD long long line(int f, int t) const {
        return DIR == 0 ? (long long)(t + 2) * (nn + 1) + f : (long long)f * (nt + 4) + (t + 2);
    }
    // face (f, t), t in [0, nt)
    DFK_HD long long face(int f, int t) const {
        return DIR == 0 ? (long long)t * (nn + 1) + f : (long long)f * nt + t;
    }
    DFK_HD long long nfaces() const { return (long long)(nn + 1) * nt; }
};

// Index spaces of the sweep kernels, row-major, rows lx wide (the thread-x direction of the bodies):
// face lines (f, t+2) and face sides / Gauss points (f, t), with f the normal and t the tangential
// index, f along the rows for x-faces and t along the rows for y-faces.
template <int DIR> DFK_HD int lines_lx(const Mesh& m) { return DIR == 0 ? m.nx + 1 : m.nx + 4; }
template <int DIR> DFK_HD int lines_ly(const Mesh& m) { return DIR == 0 ? m.ny + 4 : m.ny + 1; }
template <int DIR> DFK_HD int faces_lx(const Mesh& m) { return DIR == 0 ? m.nx + 1 : m.nx; }
template <int DIR> DFK_HD int faces_ly(const Mesh& m) { return DIR == 0 ? m.ny : m.ny + 1; }

// The sweep kernels run on 1-D grids of one-warp blocks over such a space: thread i takes
// (i mod lx, i / lx), so only the grid's last warp is partly idle, where a 2-D grid of 32-wide rows
// would idle part of every row's last warp (15 of 416 lanes on a 401-face row).  Threads past the
// end get ay >= ly, which the bodies' bounds checks reject.
// One warp per block, because nothing is shared in a block and a launch's time is that of the SM with the most
// warps: with 128 threads a mesh of about 100 x 100 gives some SMs twice the work of others.  128 -> 32
// threads: 3 x 2 blocks of 100 x 100 cells 13.2 -> 11.6 ms per 4 steps, the reverse of a 67 x 83 stage
// 0.84 -> 0.77 ms, a 97 x 61 stage 0.177 -> 0.172 ms, a 400 x 400 step the same.
constexpr int kSweepThreads = 32;
inline unsigned sweep_blocks(int lx, int ly, int threads = kSweepThreads) { return (unsigned)(((long long)lx * ly + threads - 1) / threads); }

// Which sweep kernels take four threads per item (lines_quad, faces_quad) on a mesh that `beside` meshes of its size
// are swept at the same time as (itself included, the blocks of a decomposition on their streams): those whose whole
// items, of all these meshes, are at most two (lines) or three (sides) warps per SM.  A line's 785 FP64 instructions
// keep an SM's units 6 us per warp, a side's 440 3.5; the quads' 1250 and 640 take 10 and 5, against the 31 and
// 19 us that one thread takes however few there are: the quads win below three warps of lines and four of sides.
// Counting each block of a decomposition by itself costs 14 % in 4 x 4 blocks of 60 x 60 (1374 us a step, 1208 by the
// warps of eight) and 23 % in 2 x 2 of 50 x 50 (398, 323); blocks of 20 x 20 take the quads either way (433).
constexpr int kSMs = 152;
struct QuadSweeps { bool lines, faces; };
inline QuadSweeps quad_sweeps(const Mesh& m, int beside) {
    const long long nl = (long long)sweep_blocks(lines_lx<0>(m), lines_ly<0>(m)) + sweep_blocks(lines_lx<1>(m), lines_ly<1>(m));
    const long long nf = (long long)sweep_blocks(faces_lx<0>(m), faces_ly<0>(m)) + sweep_blocks(faces_lx<1>(m), faces_ly<1>(m));
    return {beside * nl <= 2 * kSMs, beside * 2 * nf <= 3 * kSMs};
}

__device__ __forceinline__ void sweep_xy(int lx, int& ax, int& ay) {
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    ax = i % lx;
    ay = i / lx;
}

__device__ __forceinline__ void warp_count_add(unsigned long long* dst, int v) {
    int s = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(dst, (unsigned long long)s);
}

DFK_HD void report_fail(DevState* st, long long key) {
#ifdef __CUDA_ARCH__
    atomicMin(&st->fail_key, (unsigned long long)key);
    if (atomicCAS(&st->err, 0, 5) == 0) st->fail_step = st->step;
    atomicExch(&st->halt, 1);
#else   // host build of the bodies (sequential)
    if ((unsigned long long)key < st->fail_key) st->fail_key = (unsigned long long)key;
    if (st->err == 0) { st->err = 5; st->fail_step = st->step; }
    st->halt = 1;
#endif
}

// number of cell (i, j) in positivity failures: j*nx + i in a whole mesh (Mesh::gi0)
DFK_HD long long fail_key(const Mesh& m, int i, int j) {
    const long long gnx = m.gnx > 0 ? m.gnx : m.nx;
    return (long long)(j + m.gj0) * gnx + (i + m.gi0);
}

DFK_HD bool state_ok(const double W[4], double gm1) {
    bool fin = isfinite(W[0]) && isfinite(W[1]) && isfinite(W[2]) && isfinite(W[3]);
    return fin && physical_state(W, gm1);
}

// CFL bound of one interior cell: min(dx/(|U|+c), dy/(|V|+c)), or 1/((|U|+c)/dx + (|V|+c)/dy)
__device__ __forceinline__ double cfl_cell(const Mesh& m, const double* W, double gamma, int c) {
    int i = c % m.nx, j = c / m.nx;
    long long g = gid(m, i, j);
    double r = W[g], U = W[m.plane + g] / r, V = W[2 * m.plane + g] / r;
    double p = (gamma - 1.0) * (W[3 * m.plane + g] - 0.5 * r * (U * U + V * V));
    double cs = sqrt(gamma * p / r);
    if (m.dt_rule) return 1.0 / ((fabs(U) + cs) / m.dx + (fabs(V) + cs) / m.dy);
    return fmin(m.dx / (fabs(U) + cs), m.dy / (fabs(V) + cs));
}

// block-wide minimum of v (all threads call); thread 0 of the block receives the result
__device__ __forceinline__ double block_min(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    __shared__ double red[32];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        v = (lane < (int)(blockDim.x >> 5)) ? red[lane] : DBL_MAX;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    }
    return v;
}

// one ghost cell of the x pass: ghost column gc in [0, 2G), interior row j (a side marked
// BC_EXTERNAL is left to the halo copy)
DFK_HD void ghost_x_body(const Mesh& m, double* W, double* alpha, int gc, int j) {
    if (gc >= 2 * G || j >= m.ny) return;
    if (m.bc[gc < G ? 0 : 1] == BC_EXTERNAL) return;
    int i = gc < G ? gc - G : m.nx + gc - G;
    bool mir;
    int s = ghost_src(i, m.nx, m.bc[0], m.bc[1], mir);
    long long d = gid(m, i, j), o = gid(m, s, j);
    if (W) {
#pragma unroll
        for (int k = 0; k < 4; ++k) W[k * m.plane + d] = W[k * m.plane + o];
        if (mir) W[1 * m.plane + d] = -W[1 * m.plane + d];
    }
    if (alpha) alpha[d] = alpha[o];
}

// one ghost cell of the y pass: column i in [-G, nx+G), ghost row gr in [0, 2G)
DFK_HD void ghost_y_body(const Mesh& m, double* W, double* alpha, int i, int gr) {
    if (i >= m.nx + G) return;
    if (m.bc[gr < G ? 2 : 3] == BC_EXTERNAL) return;
    int j = gr < G ? gr - G : m.ny + gr - G;
    bool mir;
    int s = ghost_src(j, m.ny, m.bc[2], m.bc[3], mir);
    long long d = gid(m, i, j), o = gid(m, i, s);
    if (W) {
#pragma unroll
        for (int k = 0; k < 4; ++k) W[k * m.plane + d] = W[k * m.plane + o];
        if (mir) W[2 * m.plane + d] = -W[2 * m.plane + d];
    }
    if (alpha) alpha[d] = alpha[o];
}

// one ghost cell of the y pass on a whole mesh (no side BC_EXTERNAL), from the interior cell that the two passes
// lead to: column i in [-G, nx+G), ghost row gr
DFK_HD void ghost_corner_body(const Mesh& m, double* W, double* alpha, int i, int gr) {
    if (i >= m.nx + G || gr >= 2 * G) return;
    const int j = gr < G ? gr - G : m.ny + gr - G;
    bool mx, my;
    const int si = ghost_src(i, m.nx, m.bc[0], m.bc[1], mx), sj = ghost_src(j, m.ny, m.bc[2], m.bc[3], my);
    const long long d = gid(m, i, j), o = gid(m, si, sj);
    if (W) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double v = W[k * m.plane + o];
            W[k * m.plane + d] = (k == 1 && mx) || (k == 2 && my) ? -v : v;
        }
    }
    if (alpha) alpha[d] = alpha[o];
}

// One characteristic variable of a face line from its first differences f: both sides' value (relative to the cell
// average) and slope, q = qL, qLn, qR, qRn, and their weights where they are used (L, R)
template <bool VALUES>
DFK_HD void line_component(const Real f[5], bool acoustic, bool dfL, bool dfR, double alL, double alR, Real idn,
                           const SchemeConsts& S, Real q[4], AOWeights& L, AOWeights& R) {
    const Real s1 = f[1] - f[0], s2 = f[2] - f[1], s3 = f[3] - f[2], s4 = f[4] - f[3];
    const Real f3 = f[2];
    if (!dfL || !dfR || (!VALUES && S.time_limiter)) {
        const Real eps = acoustic ? Real(4.0 * S.eps) : Real(S.eps);
        const Real t1 = s2 - s1, t2 = s3 - s2, t3 = s4 - s3;
        const Real w1 = second_difference_energy(s1, eps), w2 = second_difference_energy(s2, eps);
        const Real w3 = second_difference_energy(s3, eps), w4 = second_difference_energy(s4, eps);
        // both sides' evaluations without a branch, so that the two chains run side by side (a DF side's is overwritten
        // below): 20 L-F steps of 40 x 40 2.00 ms, 2.07 with a branch around each
        L = ao_weights<+1>(f[1], f3, s1, s2, s3, w1, w2, w3, fma(0.5, s2, f[1]), t1 + t2, t2 - t1, eps, S);
        ao_diff_at_edge<+1>(L, f[1], f3, s2, t1, t2, idn, S, q);
        R = ao_weights<-1>(f[3], f3, s4, s3, s2, w4, w3, w2, fma(-0.5, s3, f[3]), t2 + t3, t3 - t2, eps, S);
        ao_diff_at_edge<-1>(R, f[3], f3, s3, t3, t2, idn, S, q + 2);
    }
    // the central quadratics there
    const Real hf = 0.5 * f3, baseL = fma(-1.0 / 6.0, s2, hf), baseR = fma(-1.0 / 6.0, s3, -hf);
    if (dfL) { q[0] = Real::raw(alL) * baseL; q[1] = idn * (Real::raw(alL) * f3); }
    if (dfR) { q[2] = Real::raw(alR) * baseR; q[3] = idn * (Real::raw(alR) * f3); }
}

// the limiter fraction so far, (1 + rmax^2) / (1 + rmin^2) = hi / lo at its largest, and the reconstruction it is of
DFK_HD void limiter_update(Real xmax, Real xmin, int which, Real& hi, Real& lo, int& tlk) {
    if (nn_less(hi * xmin, xmax * lo)) { hi = xmax; lo = xmin; tlk = which; }
}

// one face line (normal reconstruction of both sides); returns the number of DF branches taken
// TAPE: also write the reconstructions' ratios for a reverse sweep (ltape, see SweepBuffers)
// VALUES: the face values alone, for sweeps whose consumers use neither slopes nor the limiter weight: the DF
// factors (alpha_only) and the L-F flux of the Runge-Kutta stages.  The slope and limiter fields stay unwritten.
template <int DIR, bool TAPE = false, bool VALUES = false>
DFK_HD int lines_body(const Mesh& m, const SchemeConsts& S, const double* __restrict__ W,
                                          const double* __restrict__ alpha, double* __restrict__ lines,
                                          long long ls, int ax, int ay, double* __restrict__ ltape = nullptr) {
    Geo<DIR> g(m);
    int f = DIR == 0 ? ax : ay;
    int tt = DIR == 0 ? ay : ax;                           // t + 2
    bool active = f <= g.nn && tt < g.nt + 4;
    int ndf = 0;
    if (active) {
        const int t = tt - 2;
        double Wc[6][4];
        double al[6];
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            long long c = g.cell(m, f - 3 + s, t);
#pragma unroll
            for (int k = 0; k < 4; ++k) Wc[s][k] = W[k * m.plane + c];
            to_local<DIR>(Wc[s]);
            al[s] = alpha[c];
        }
        CharBasis B = make_basis(Wc[2], Wc[3], S);
        const bool dfL = nn_less(nn_max(nn_max(al[1], al[2]), al[3]), S.alpha_thres);   // Eq. 34, cell f-1
        const bool dfR = nn_less(nn_max(nn_max(al[2], al[3]), al[4]), S.alpha_thres);   // Eq. 34, cell f
        ndf = (int)dfL + (int)dfR;
        const long long li = g.line(f, t);
        // the cell-average reading of the DF states, stored before the reconstructions so that
        // the two cell states need not stay live through them
        if (S.df_states) lines[LR_DFC * ls + li] = df_alpha(Wc[2], Wc[3], S);
        // the limiter weight so far as tn / td (1 until a reconstruction gives less); fractions are
        // compared by cross-multiplication, one division at the end
        double tn = 1.0, td = 1.0;
        int tlk = -1;                                     // the reconstruction that set it
        const DiffBasis D = diff_basis(B);
        const Real idn = g.idn;
        Real F[5][4];                               // first differences of the characteristic variables
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            Real dW[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) dW[k] = Real::raw(Wc[s + 1][k]) - Real::raw(Wc[s][k]);
            project_diff(D, dW, F[s]);
        }
        Real qL[4], qLn[4], qR[4], qRn[4];          // face value minus cell value, slope
        Real xhi = 1.0, xlo = 1.0;                  // limiter: (1 + rmax^2) / (1 + rmin^2), the largest so far
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const Real fk[5] = {F[0][k], F[1][k], F[2][k], F[3][k], F[4][k]};
            Real q[4];
            AOWeights L, R;
            line_component<VALUES>(fk, k == 0 || k == 3, dfL, dfR, al[2], al[3], idn, S, q, L, R);
            if constexpr (TAPE) {
                if (!dfL || !dfR || S.time_limiter) {
                    const PlaneTape T{ltape + li, ls};
                    tape_ratios(T, 2 * k * RT_COUNT, ao_ratios(L));
                    tape_ratios(T, (2 * k + 1) * RT_COUNT, ao_ratios(R));
                }
            }
            if (!VALUES && S.time_limiter) {
                limiter_update(L.xmax, L.xmin, 2 * k, xhi, xlo, tlk);
                limiter_update(R.xmax, R.xmin, 2 * k + 1, xhi, xlo, tlk);
            }
            qL[k] = q[0]; qLn[k] = q[1]; qR[k] = q[2]; qRn[k] = q[3];
        }
        tn = Real(2.0 * xlo).v;
        td = (xhi + xlo).v;
        Real w[16];
        back_project_diff(D, qL, w + LR_WL);
        back_project_diff(D, qR, w + LR_WR);
        if constexpr (!VALUES) {
            back_project_diff(D, qLn, w + LR_WLN);
            back_project_diff(D, qRn, w + LR_WRN);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            w[LR_WL + k] = w[LR_WL + k] + Real::raw(Wc[2][k]);
            w[LR_WR + k] = w[LR_WR + k] + Real::raw(Wc[3][k]);
        }
#pragma unroll
        for (int q = 0; q < 16; ++q)
            if (!VALUES || (q & 4) == 0) lines[q * ls + li] = w[q].v;       // LR_WLN, LR_WRN have bit 2
        if constexpr (!VALUES) {
            lines[LR_TL * ls + li] = tn / td;
            lines[LR_TLK * ls + li] = (double)tlk;
        }
        lines[LR_U * ls + li] = B.u;
        lines[LR_V * ls + li] = B.v;
        lines[LR_C * ls + li] = B.c;
        lines[LR_IC * ls + li] = B.ic;
        lines[LR_H * ls + li] = B.H;
        lines[LR_B1 * ls + li] = B.b1;
        lines[LR_B2 * ls + li] = B.b2;
        lines[LR_Q2 * ls + li] = B.q2;
    }
    return ndf;
}

// One characteristic variable of a face side from its first differences f: values (relative to the line's) and
// scaled slopes at the two Gauss points, q = v0, v1, slope0, slope1
template <class Tape>
DFK_HD void face_component(const Real f[4], bool acoustic, bool df, double alpha, Real idt, const SchemeConsts& S, Real q[4],
                           const Tape& tp, int base) {
    const Real s0 = f[1] - f[0], s1 = f[2] - f[1], s2 = f[3] - f[2];
    const Real a11 = fma(0.5, s1, f[1]);
    Real v[2], s[2];
    if (df) df_diff_at_gauss(a11, s1, Real::raw(alpha), v, s);
    else {
        const Real eps = acoustic ? Real(4.0 * S.eps) : Real(S.eps);
        const Real t1 = s1 - s0, t2 = s2 - s1, T = t1 + t2, U = t2 - t1;
        const AOWeights o = ao_weights<+1>(f[1], f[2], s0, s1, s2, second_difference_energy(s0, eps),
                                           second_difference_energy(s1, eps), second_difference_energy(s2, eps),
                                           a11, T, U, eps, S);
        if constexpr (Tape::active) tape_ratios(tp, base, ao_ratios(o));
        ao_diff_at_gauss(o, a11, s1, t1, t2, T, U, S, v, s);
    }
    q[0] = v[0]; q[1] = v[1];
    q[2] = s[0] * idt; q[3] = s[1] * idt;
}

// one face side (tangential reconstruction at both Gauss points, fallback); returns the number of
// DF branches taken and sets nfb to the number of fallbacks
// TAPE: also write the reconstructions' ratios for a reverse sweep (ftape, see SweepBuffers)
// VALUES: the Gauss-point values alone, without the two slopes (see lines_body)
template <int DIR, bool TAPE = false, bool VALUES = false>
DFK_HD int faces_body(const Mesh& m, const SchemeConsts& S, const double* __restrict__ W,
                                          const double* __restrict__ alpha, const double* __restrict__ lines,
                                          long long ls, double* __restrict__ gp, long long gs,
                                          int ax, int ay, int side, int& nfb,
                                          double* __restrict__ ftape = nullptr) {
    Geo<DIR> g(m);
    int f = DIR == 0 ? ax : ay;
    int t = DIR == 0 ? ay : ax;
    bool active = f <= g.nn && t < g.nt;
    int ndf = 0;
    nfb = 0;
    if (active) {
        const long long l0 = g.line(f, t);
        CharBasis B;
        B.u = lines[LR_U * ls + l0]; B.v = lines[LR_V * ls + l0]; B.c = lines[LR_C * ls + l0];
        B.ic = lines[LR_IC * ls + l0]; B.H = lines[LR_H * ls + l0]; B.b1 = lines[LR_B1 * ls + l0];
        B.b2 = lines[LR_B2 * ls + l0]; B.q2 = lines[LR_Q2 * ls + l0];
        const int wbase = side == 0 ? LR_WL : LR_WR;
        const int ncell = f - 1 + side;
        double al[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) al[b] = alpha[g.cell(m, ncell, t + Geo<DIR>::sigma * (b - 1))];
        const bool df = nn_less(nn_max(nn_max(al[0], al[1]), al[2]), S.alpha_thres);    // Eq. 34, tangential
        ndf = (int)df;
        double Wv[2][4], Wd[2][4];               // values and tangential slopes at the two Gauss points
        const long long e = (long long)side * g.nfaces() + g.face(f, t);
        double Wl[5][4];
#pragma unroll
        for (int b = 0; b < 5; ++b) {
            const long long lb = g.line(f, t + Geo<DIR>::sigma * (b - 2));
#pragma unroll
            for (int k = 0; k < 4; ++k) Wl[b][k] = lines[(wbase + k) * ls + lb];
        }
        const DiffBasis D = diff_basis(B);
        const Real idt = g.idtan;
        Real F[4][4], qv[2][4], qt[2][4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            Real dW[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) dW[k] = Real::raw(Wl[b + 1][k]) - Real::raw(Wl[b][k]);
            project_diff(D, dW, F[b]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const Real fk[4] = {F[0][k], F[1][k], F[2][k], F[3][k]};
            Real q[4];
            if constexpr (TAPE) face_component(fk, k == 0 || k == 3, df, al[1], idt, S, q, PlaneTape{ftape + e, gs}, k * RT_COUNT);
            else face_component(fk, k == 0 || k == 3, df, al[1], idt, S, q, NoTape{}, 0);
            qv[0][k] = q[0]; qv[1][k] = q[1];
            qt[0][k] = q[2]; qt[1][k] = q[3];
        }
#pragma unroll
        for (int mm = 0; mm < 2; ++mm) {
            Real w[4], d[4];
            back_project_diff(D, qv[mm], w);
            if constexpr (!VALUES) back_project_diff(D, qt[mm], d);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                Wv[mm][k] = (w[k] + Real::raw(Wl[2][k])).v;
                if constexpr (!VALUES) Wd[mm][k] = d[k].v;
            }
        }
        const int nbase = side == 0 ? LR_WLN : LR_WRN;
        int fbits = 0;
#pragma unroll
        for (int mm = 0; mm < 2; ++mm) {
            double Wg[4], Wt[4], Wn[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                Wg[k] = Wv[mm][k];
                if constexpr (!VALUES) { Wt[k] = Wd[mm][k]; Wn[k] = lines[(nbase + k) * ls + l0]; }
            }
            if (S.gp_fallback && !physical_state(Wg, S.gm1)) {
                long long c = g.cell(m, ncell, t);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    Wg[k] = W[k * m.plane + c];
                    if constexpr (!VALUES) { Wn[k] = 0.0; Wt[k] = 0.0; }
                }
                to_local<DIR>(Wg);
                ++nfb;
                fbits |= 1 << mm;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                gp[(mm * 12 + k) * gs + e] = Wg[k];
                if constexpr (!VALUES) {
                    gp[(mm * 12 + 4 + k) * gs + e] = Wn[k];
                    gp[(mm * 12 + 8 + k) * gs + e] = Wt[k];
                }
            }
        }
        gp[GP_FB * gs + e] = (double)fbits;
    }
    return ndf;
}

// ------------------------------------------------------------------------------------------
// Four threads per face line and per face side, one per characteristic variable, for meshes so small that a
// launch takes as long as one thread: a warp alone on its scheduler takes 12.7 cycles per instruction, 31 us for a
// line and 19 us for a side, whatever the mesh.  Differences and basis are formed by each thread of a quad; the
// results change hands in one 4 x 4 transposition, after which thread j back-projects the j-th vector.  The
// arithmetic is that of lines_body and faces_body operation by operation, so the results are the same bits.
// All 32 lanes take part in the exchanges: a quad past the end works on item 0 and writes nothing.
// 8 GKS steps of 100 x 4 1.77 -> 1.31 ms, 20 L-F steps of 40 x 40 3.82 -> 2.75 ms.
// ------------------------------------------------------------------------------------------
#ifdef __CUDACC__
// component k of project_diff
__device__ __forceinline__ Real project_diff_component(const DiffBasis& D, const Real W[4], int k) {
    const Real kk = fma(D.b1, W[3], fma(-D.b1v, W[2], fma(-D.b1u, W[1], D.b2 * W[0])));
    const Real mm = fma(-D.ic, W[1], D.uic * W[0]);
    const Real A = k == 2 ? -D.v : (k == 1 ? W[0] : kk), M = k == 2 ? W[0] : Real(1.0);
    const Real C = k == 2 ? W[2] : (k == 1 ? -kk : (k == 3 ? -mm : mm));
    return fma(A, M, C);
}
__device__ __forceinline__ Real pick(const Real q[4], int j) { return (j & 2) ? ((j & 1) ? q[3] : q[2]) : ((j & 1) ? q[1] : q[0]); }
// thread j of a quad holds q[0..3] of component j and gets the four components of q[j]
__device__ __forceinline__ void quad_transpose(Real q[4], int j) {
    Real r[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) r[x] = Real::raw(__shfl_xor_sync(0xffffffffu, pick(q, j ^ x).v, x));   // component j ^ x
#pragma unroll
    for (int c = 0; c < 4; ++c) q[c] = pick(r, c ^ j);
}
__device__ __forceinline__ Real quad_get(Real v, int c) { return Real::raw(__shfl_sync(0xffffffffu, v.v, ((int)threadIdx.x & 28) + c)); }

template <int DIR, bool VALUES>
__device__ __forceinline__ int lines_quad(const Mesh& m, const SchemeConsts& S, const double* __restrict__ W,
                                          const double* __restrict__ alpha, double* __restrict__ lines, long long ls,
                                          int ax, int ay) {
    Geo<DIR> g(m);
    const int j = threadIdx.x & 3;
    int f = DIR == 0 ? ax : ay, tt = DIR == 0 ? ay : ax;
    const bool active = f <= g.nn && tt < g.nt + 4;
    if (!active) f = tt = 0;
    const int t = tt - 2;
    double Wc[6][4], al[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        const long long c = g.cell(m, f - 3 + s, t);
#pragma unroll
        for (int k = 0; k < 4; ++k) Wc[s][k] = W[k * m.plane + c];
        to_local<DIR>(Wc[s]);
        al[s] = alpha[c];
    }
    const CharBasis B = make_basis(Wc[2], Wc[3], S);
    const bool dfL = nn_less(nn_max(nn_max(al[1], al[2]), al[3]), S.alpha_thres);
    const bool dfR = nn_less(nn_max(nn_max(al[2], al[3]), al[4]), S.alpha_thres);
    const long long li = g.line(f, t);
    if (S.df_states && active && j == 2) lines[LR_DFC * ls + li] = df_alpha(Wc[2], Wc[3], S);
    const DiffBasis D = diff_basis(B);
    Real F[5], q[4];
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        Real dW[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) dW[k] = Real::raw(Wc[s + 1][k]) - Real::raw(Wc[s][k]);
        F[s] = project_diff_component(D, dW, j);
    }
    AOWeights L, R;
    line_component<VALUES>(F, j == 0 || j == 3, dfL, dfR, al[2], al[3], g.idn, S, q, L, R);
    Real xhi = 1.0, xlo = 1.0;
    int tlk = -1;
    if (!VALUES && S.time_limiter) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            limiter_update(quad_get(L.xmax, k), quad_get(L.xmin, k), 2 * k, xhi, xlo, tlk);
            limiter_update(quad_get(R.xmax, k), quad_get(R.xmin, k), 2 * k + 1, xhi, xlo, tlk);
        }
    }
    quad_transpose(q, j);
    if (!active) return 0;
    if (!VALUES || (j & 1) == 0) {
        Real w[4];
        back_project_diff(D, q, w);
        if ((j & 1) == 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = w[k] + Real::raw(j == 0 ? Wc[2][k] : Wc[3][k]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) lines[(4 * j + k) * ls + li] = w[k].v;      // LR_WL, LR_WLN, LR_WR, LR_WRN
    }
    if (j == 0) {
        if (!VALUES) {
            lines[LR_TL * ls + li] = Real(2.0 * xlo).v / (xhi + xlo).v;
            lines[LR_TLK * ls + li] = (double)tlk;
        }
        return (int)dfL + (int)dfR;
    }
    if (j == 1) {
        lines[LR_U * ls + li] = B.u; lines[LR_V * ls + li] = B.v; lines[LR_C * ls + li] = B.c; lines[LR_IC * ls + li] = B.ic;
    } else if (j == 3) {
        lines[LR_H * ls + li] = B.H; lines[LR_B1 * ls + li] = B.b1; lines[LR_B2 * ls + li] = B.b2; lines[LR_Q2 * ls + li] = B.q2;
    }
    return 0;
}

template <int DIR, bool VALUES>
__device__ __forceinline__ int faces_quad(const Mesh& m, const SchemeConsts& S, const double* __restrict__ W,
                                          const double* __restrict__ alpha, const double* __restrict__ lines, long long ls,
                                          double* __restrict__ gp, long long gs, int ax, int ay, int side, int& nfb) {
    Geo<DIR> g(m);
    const int j = threadIdx.x & 3;
    int f = DIR == 0 ? ax : ay, t = DIR == 0 ? ay : ax;
    const bool active = f <= g.nn && t < g.nt;
    if (!active) f = t = 0;
    nfb = 0;
    const long long l0 = g.line(f, t);
    CharBasis B;
    B.u = lines[LR_U * ls + l0]; B.v = lines[LR_V * ls + l0]; B.c = lines[LR_C * ls + l0];
    B.ic = lines[LR_IC * ls + l0]; B.H = lines[LR_H * ls + l0]; B.b1 = lines[LR_B1 * ls + l0];
    B.b2 = lines[LR_B2 * ls + l0]; B.q2 = lines[LR_Q2 * ls + l0];
    const int wbase = side == 0 ? LR_WL : LR_WR, nbase = side == 0 ? LR_WLN : LR_WRN, ncell = f - 1 + side;
    double al[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) al[b] = alpha[g.cell(m, ncell, t + Geo<DIR>::sigma * (b - 1))];
    const bool df = nn_less(nn_max(nn_max(al[0], al[1]), al[2]), S.alpha_thres);
    const long long e = (long long)side * g.nfaces() + g.face(f, t);
    double Wl[5][4];
#pragma unroll
    for (int b = 0; b < 5; ++b) {
        const long long lb = g.line(f, t + Geo<DIR>::sigma * (b - 2));
#pragma unroll
        for (int k = 0; k < 4; ++k) Wl[b][k] = lines[(wbase + k) * ls + lb];
    }
    const DiffBasis D = diff_basis(B);
    Real F[4], q[4], w[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        Real dW[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) dW[k] = Real::raw(Wl[b + 1][k]) - Real::raw(Wl[b][k]);
        F[b] = project_diff_component(D, dW, j);
    }
    face_component(F, j == 0 || j == 3, df, al[1], g.idtan, S, q, NoTape{}, 0);
    quad_transpose(q, j);                      // threads 0, 1: the values at the two Gauss points; 2, 3: the slopes
    back_project_diff(D, q, w);
    double Wg[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) Wg[k] = j < 2 ? (w[k] + Real::raw(Wl[2][k])).v : w[k].v;
    const int bad = j < 2 && S.gp_fallback && !physical_state(Wg, S.gm1);
    const int b0 = __shfl_sync(0xffffffffu, bad, threadIdx.x & 28), b1 = __shfl_sync(0xffffffffu, bad, (threadIdx.x & 28) + 1);
    if (!active) return 0;
    const int mm = j & 1;
    const bool fell = mm == 0 ? b0 : b1;
    if (j < 2) {
        if (fell) {
            const long long c = g.cell(m, ncell, t);
#pragma unroll
            for (int k = 0; k < 4; ++k) Wg[k] = W[k * m.plane + c];
            to_local<DIR>(Wg);
            nfb = 1;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) gp[(mm * 12 + k) * gs + e] = Wg[k];
    } else if (!VALUES) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            gp[(mm * 12 + 4 + k) * gs + e] = fell ? 0.0 : lines[(nbase + k) * ls + l0];
            gp[(mm * 12 + 8 + k) * gs + e] = fell ? 0.0 : Wg[k];
        }
    }
    if (j != 0) return 0;
    gp[GP_FB * gs + e] = (double)(b0 | (b1 << 1));
    return (int)df;
}
#endif

// where one Gauss point's records live: side records eL / eR, its flux record e, its face line li
struct FluxSite { long long eL, eR, e, li; bool ok; };

template <int DIR>
DFK_HD FluxSite flux_site(const Mesh& m, int ax, int ay, int mm) {
    Geo<DIR> g(m);
    const int f = DIR == 0 ? ax : ay;
    const int t = DIR == 0 ? ay : ax;
    FluxSite s;
    s.ok = f <= g.nn && t < g.nt;
    if (!s.ok) { s.eL = s.eR = s.e = s.li = 0; return s; }
    const long long fid = g.face(f, t);
    s.eL = fid;
    s.eR = g.nfaces() + fid;
    s.e = (long long)mm * g.nfaces() + fid;
    s.li = g.line(f, t);
    return s;
}

// one Gauss point (flux, time derivative, DF factor, omega^t) of direction dir at a site
// VALUES (L-F): the flux and the DF factor alone, from records without slopes
template <int FLUX, bool ALPHA_ONLY, bool TAPE = false, bool VALUES = false>
DFK_HD void flux_point(int dir, const SchemeConsts& S, const FluxSite& site, const double* __restrict__ lines,
                       long long ls, const double* __restrict__ gp, long long gs, double* __restrict__ fr,
                       long long fs, double dt, int mm, double* __restrict__ tape = nullptr) {
    static_assert(!VALUES || FLUX == 1, "the GKS flux uses the slopes");
    GPState L, R;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        L.W[k] = gp[(mm * 12 + k) * gs + site.eL];
        R.W[k] = gp[(mm * 12 + k) * gs + site.eR];
        if constexpr (!VALUES && !ALPHA_ONLY) {
            L.Wn[k] = gp[(mm * 12 + 4 + k) * gs + site.eL];
            L.Wt[k] = gp[(mm * 12 + 8 + k) * gs + site.eL];
            R.Wn[k] = gp[(mm * 12 + 4 + k) * gs + site.eR];
            R.Wt[k] = gp[(mm * 12 + 8 + k) * gs + site.eR];
        }
    }
    const long long e = site.e;
    // the two sides' states serve the DF factor and the GKS flux.  The Gauss-point reading of Eq. 33 is
    // always evaluated (the default path stays branch-free); the cell-average reading, when selected,
    // overwrites it with its face line's value
    double F[4], dF[4];
    const FlowState sl = side_state(L.W, S), sr = side_state(R.W, S);
    fr[FR_ALPHA * fs + e] = df_alpha_sides(sl, sr, S).v;
    if (S.df_states) fr[FR_ALPHA * fs + e] = lines[LR_DFC * ls + site.li];
    if (ALPHA_ONLY) return;
    if constexpr (FLUX == 1) lf_flux_sides<VALUES>(L, R, sl, sr, S, F, dF);
    else if constexpr (TAPE) gks_flux_sides(L, R, sl, sr, dt, S, F, dF, PlaneTape{tape + e, fs});
    else gks_flux_sides(L, R, sl, sr, dt, S, F, dF, NoTape{});
    if (dir == 1) to_global<1>(F);
#pragma unroll
    for (int k = 0; k < 4; ++k) fr[(FR_F + k) * fs + e] = F[k];
    if constexpr (!VALUES) {
        if (dir == 1) to_global<1>(dF);
#pragma unroll
        for (int k = 0; k < 4; ++k) fr[(FR_DF + k) * fs + e] = dF[k];
        fr[FR_OMEGA * fs + e] = S.time_limiter ? lines[LR_TL * ls + site.li] : 1.0;
    }
}

// one Gauss point (flux, time derivative, DF factor, omega^t)
template <int DIR, int FLUX, bool ALPHA_ONLY, bool TAPE = false>
DFK_HD void flux_body(const Mesh& m, const SchemeConsts& S, const double* __restrict__ lines,
                                          long long ls, const double* __restrict__ gp, long long gs,
                                          double* __restrict__ fr, long long fs, double dt, int ax, int ay, int mm,
                         double* __restrict__ tape = nullptr) {
    const FluxSite site = flux_site<DIR>(m, ax, ay, mm);
    if (!site.ok) return;
    flux_point<FLUX, ALPHA_ONLY, TAPE>(DIR, S, site, lines, ls, gp, gs, fr, fs, dt, mm, tape);
}

// one cell: residual, limited time derivative, stage combination, alpha product, positivity.  Bound by the FP64
// units on 4 % of a step's time; a face's Gauss points summed before they are weighted and every operand in a
// vector register took 4 steps of 400 x 400 from 12.82 to 12.74 ms, a 1021 x 509 stage from 4.71 to 4.63.
template <int MODE>
DFK_HD void update_body(const Mesh& m, const SchemeConsts& S, const UpdateArgs& a,
                                            const double* __restrict__ frx, long long fsx,
                                            const double* __restrict__ fry, long long fsy,
                                            double dt, DevState* st, int i, int j) {
    if (i >= m.nx || j >= m.ny) return;
    const long long nfx = (long long)(m.nx + 1) * m.ny, nfy = (long long)(m.ny + 1) * m.nx;
    const long long fw = (long long)j * (m.nx + 1) + i, fe = fw + 1;
    const long long fsf = (long long)j * m.nx + i, fn = fsf + m.nx;
    // alpha product in the fixed order W(m1,m2), E, S, N
    Real ar = Real::raw(frx[FR_ALPHA * fsx + fw]) * Real::raw(frx[FR_ALPHA * fsx + nfx + fw]);
    ar = ar * Real::raw(frx[FR_ALPHA * fsx + fe]);
    ar = ar * Real::raw(frx[FR_ALPHA * fsx + nfx + fe]);
    ar = ar * Real::raw(fry[FR_ALPHA * fsy + fsf]);
    ar = ar * Real::raw(fry[FR_ALPHA * fsy + nfy + fsf]);
    ar = ar * Real::raw(fry[FR_ALPHA * fsy + fn]);
    ar = ar * Real::raw(fry[FR_ALPHA * fsy + nfy + fn]);
    const double an = ar.v;
    const long long g = gid(m, i, j);
    const long long dn = (long long)j * m.nx + i, dplane = (long long)m.nx * m.ny;
    if (MODE == UM_ALPHA) {
        if (a.alpha_out) a.alpha_out[a.alpha_dense ? dn : g] = an;
        return;
    }
    // Eq. 2: sums over a face's two Gauss points (weight 1/2 each), differences over the cell's faces
    Real L[4], dL[4], dLt[4];
    const Real hx = 0.5 * m.rdx, hy = 0.5 * m.rdy;
    const Real ow = Real::raw(frx[FR_OMEGA * fsx + fw]), oe = Real::raw(frx[FR_OMEGA * fsx + fe]);
    const Real os = Real::raw(fry[FR_OMEGA * fsy + fsf]), on = Real::raw(fry[FR_OMEGA * fsy + fn]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const auto face = [&](const double* fr, long long fs, long long nf, int field, long long f) {
            return Real::raw(fr[(field + k) * fs + f]) + Real::raw(fr[(field + k) * fs + nf + f]);
        };
        const Real FW = face(frx, fsx, nfx, FR_F, fw), FE = face(frx, fsx, nfx, FR_F, fe);
        const Real FS = face(fry, fsy, nfy, FR_F, fsf), FN = face(fry, fsy, nfy, FR_F, fn);
        const Real DW = face(frx, fsx, nfx, FR_DF, fw), DE = face(frx, fsx, nfx, FR_DF, fe);
        const Real DS = face(fry, fsy, nfy, FR_DF, fsf), DN = face(fry, fsy, nfy, FR_DF, fn);
        L[k] = fma(hx, FW - FE, hy * (FS - FN));
        dL[k] = fma(hx, DW - DE, hy * (DS - DN));
        dLt[k] = fma(hx, fma(ow, DW, -(oe * DE)), hy * fma(os, DS, -(on * DN)));
    }
    if (MODE == UM_RESIDUAL) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (a.L) a.L[k * dplane + dn] = L[k].v;
            if (a.dtL) a.dtL[k * dplane + dn] = dL[k].v;
            if (a.dtLt) a.dtLt[k * dplane + dn] = dLt[k].v;
        }
        if (a.alpha_out) a.alpha_out[a.alpha_dense ? dn : g] = an;
        return;
    }
    const Real t1 = dt, t2 = t1 * t1, third = (1.0 / 3.0) * t2;
    double Wo[4];
    if (MODE == UM_S2O4_1) {
        const Real h1 = 0.5 * t1, h2 = 0.5 * t2, e2 = 0.125 * t2;
        double Ws[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const Real w = Real::raw(a.Win[k * m.plane + g]);
            Ws[k] = fma(e2, dL[k], fma(h1, L[k], w)).v;
            a.acc[k * dplane + dn] = fma(-third, dLt[k], fma(h2, dL[k], fma(t1, L[k], w))).v;
            a.Wout[k * m.plane + g] = Ws[k];
        }
        if (!state_ok(Ws, S.gm1)) report_fail(st, fail_key(m, i, j));
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        Real w;
        if (MODE == UM_S2O4_2) w = fma(third, dLt[k], Real::raw(a.acc[k * dplane + dn]));
        else {
            const Real in = Real::raw(a.Win[k * m.plane + g]);
            if (MODE == UM_RK_1) w = fma(t1, L[k], in);
            else {
                const Real old = Real::raw(a.Wn[k * m.plane + g]), q = fma(t1, L[k], in);
                if (MODE == UM_RK_2) w = fma(0.75, old, 0.25 * q);
                else w = fma(1.0 / 3.0, old, (2.0 / 3.0) * q);                 // UM_RK_3
            }
        }
        Wo[k] = w.v;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) a.Wout[k * m.plane + g] = Wo[k];
    if ((MODE == UM_S2O4_2 || MODE == UM_RK_3) && a.alpha_out) a.alpha_out[a.alpha_dense ? dn : g] = an;
    if (!state_ok(Wo, S.gm1)) report_fail(st, fail_key(m, i, j));
}

}  // namespace dfk

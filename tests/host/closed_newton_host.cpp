// Whole closed-form fits (closed_newton.cuh: set-up, Newton iteration, and in FP32
// mode the rounding screen) on the host, and the residual of what they return from
// sums over the cells in long double, through extern "C" functions (one per
// arithmetic). In: rows of 10 raw moments. Out per row: 0 refused / 1 taken, the
// reported residual, the true one (both relative to n), 1 if the FP32 mode keeps
// the fit (rounds_alike), the square of 1 + the largest |mean| in thermal speeds
// (how an error of the moments about the mean grows in the residual), Newton
// iterations, evaluations, of which with the Gram sums.
#include "device_shim.h"
typedef int cudaError_t;
typedef void* cudaStream_t;
#include "../../paper_2109_06743_gb300/csrc/closed_newton.cuh"

using namespace vl;
using namespace vl::cf;
typedef long double LD;

static const FitCount kNoCount = {0, 0u, 0u, 0.f, 0.f, 0.f, 1.f, 0.f};

static void box_of(int N, double half, double tol, int max_iter, FitArgs& a) {
    std::memset(&a, 0, sizeof a);
    a.nv = N;
    a.tol = tol;
    a.max_iter = max_iter;
    for (int q = 0; q < 3; ++q) {
        a.vmin[q] = -half;
        a.vmax[q] = half;
        a.dv[q] = 2.0 * half / N;
        a.inv_dv[q] = 1.0 / a.dv[q];
    }
}

template <class T>
static void run(int N, double half, double tol, int max_iter, int cases, const double* in, double* out) {
    FitArgs a;
    box_of(N, half, tol, max_iter, a);
    const LD dv = 2.0L * half / N;
    for (int c = 0; c < cases; ++c) {
        double t[10], u0[3], sg[3], *o = out + 8 * c;
        for (int q = 0; q < 10; ++q) t[q] = in[10 * c + q];
        for (int q = 0; q < 8; ++q) o[q] = 0.0;
        FitBox<T> b;
        T Tt[10];
        typename Jac<T>::type eta0[10];
        float spread;
        Maxw<T> g;
        FitCount fc = kNoCount;
        if (!closed_setup<T>(t, a, u0, sg, b, Tt, eta0, spread)) continue;
        o[0] = closed_fit<T>(g, b, Tt, eta0, nullptr, t[0], a, fc) ? 1.0 : 0.0;
        o[5] = fc.iters;
        o[6] = fc.evals;
        o[7] = fc.grams;
        if (o[0] == 0.0) continue;
        o[1] = fc.res;
        o[3] = rounds_alike<T>(g, b, u0, sg, tol, a, fc) ? 1.0 : 0.0;
        LD D[10], R[10], m[3], p[6];
        for (auto& x : D) x = 0;
        for (int q = 0; q < 6; ++q) p[q] = wide_of(g.P[q]);
        for (int q = 0; q < 3; ++q) m[q] = wide_of(g.m[q]);
        for (int k = 0; k < N; ++k)
            for (int j = 0; j < N; ++j)
                for (int i = 0; i < N; ++i) {
                    const int ix[3] = {i, j, k};
                    LD w[3], d[3];
                    for (int q = 0; q < 3; ++q) {
                        w[q] = (dv * (ix[q] + 0.5L) - half - u0[q]) / sg[q];
                        d[q] = w[q] - m[q];
                    }
                    const LD q2 = p[0] * d[0] * d[0] + p[3] * d[1] * d[1] + p[5] * d[2] * d[2] +
                                  2 * (p[1] * d[0] * d[1] + p[2] * d[0] * d[2] + p[4] * d[1] * d[2]);
                    const LD M = dv * dv * dv * expl((LD)wide_of(g.L) - q2 / 2);
                    D[0] += M;
                    for (int x = 0, z = 4; x < 3; ++x) {
                        D[1 + x] += M * w[x];
                        for (int y = x; y < 3; ++y, ++z) D[z] += M * w[x] * w[y];
                    }
                }
        const LD n = t[0];
        R[0] = n;
        for (int x = 0, z = 4; x < 3; ++x) {
            R[1 + x] = (t[1 + x] - n * u0[x]) / sg[x];
            for (int y = x; y < 3; ++y, ++z)
                R[z] = ((LD)t[z] - (LD)u0[x] * t[1 + y] - (LD)u0[y] * t[1 + x] + n * u0[x] * u0[y]) / ((LD)sg[x] * sg[y]);
        }
        for (int q = 0; q < 10; ++q) o[2] = std::fmax(o[2], (double)fabsl((D[q] - R[q]) / n));
        double big = 0.0;
        for (int q = 0; q < 3; ++q) big = std::fmax(big, (double)fabsl(m[q]));
        o[4] = (1.0 + big) * (1.0 + big);
    }
}

// FP32 mode: the double-float fits against FP64 fits of the same targets to 4e-15 n.
// Out per row: 0 refused / 1 taken by both, the largest difference of L and of the
// means (in standard deviations), that of P (relative), and fit_slack.
extern "C" void closed_fit_apart(int N, double half, double tol, int max_iter, int cases, const double* in, double* out) {
    FitArgs a;
    box_of(N, half, tol, max_iter, a);
    FitArgs fine = a;
    fine.tol = 4e-15;
    for (int c = 0; c < cases; ++c) {
        double t[10], u0[3], sg[3], v0[3], s0[3], Td[10], ed[10], *o = out + 4 * c;
        for (int q = 0; q < 10; ++q) t[q] = in[10 * c + q];
        for (int q = 0; q < 4; ++q) o[q] = 0.0;
        FitBox<df2> b;
        FitBox<double> bd;
        df2 Tt[10];
        float eta0[10], spread;
        Maxw<df2> g;
        Maxw<double> gd;
        FitCount fc = kNoCount, fd = kNoCount;
        if (!closed_setup<df2>(t, a, u0, sg, b, Tt, eta0, spread) || !closed_setup<double>(t, fine, v0, s0, bd, Td, ed, spread) ||
            !closed_fit<df2>(g, b, Tt, eta0, nullptr, t[0], a, fc) || !closed_fit<double>(gd, bd, Td, ed, nullptr, t[0], fine, fd))
            continue;
        o[0] = 1.0;
        o[1] = std::fabs(wide_of(g.L) - gd.L);
        for (int q = 0; q < 3; ++q)
            o[1] = std::fmax(o[1], std::fabs((v0[q] - u0[q]) + s0[q] * gd.m[q] - sg[q] * wide_of(g.m[q])) / s0[q]);
        for (int x = 0; x < 3; ++x)
            for (int y = x; y < 3; ++y) {
                const int q = sym(x, y);
                const double f = (sg[x] / s0[x]) * (sg[y] / s0[y]);
                o[2] = std::fmax(o[2], std::fabs(wide_of(g.P[q]) / f - gd.P[q]) / std::sqrt(gd.P[sym(x, x)] * gd.P[sym(y, y)]));
            }
        o[3] = fit_slack(fc, tol);
    }
}

// Newton steps and evaluations of a fit from eta0 (out[0..2]: taken, steps,
// evaluations) and of the same fit from eta0 + dw first (out[3..5]); the steps that
// start alone takes with a cap of 40, or 0 where it fails (out[6]).
extern "C" void closed_fit_started(int N, double half, double tol, int max_iter, int cases, const double* in, const float* dw,
                                   double* out) {
    FitArgs a;
    box_of(N, half, tol, max_iter, a);
    for (int c = 0; c < cases; ++c) {
        double t[10], u0[3], sg[3], *o = out + 7 * c;
        for (int q = 0; q < 10; ++q) t[q] = in[10 * c + q];
        FitBox<df2> b;
        df2 Tt[10];
        float eta0[10], spread;
        Maxw<df2> g;
        for (int q = 0; q < 7; ++q) o[q] = 0.0;
        if (!closed_setup<df2>(t, a, u0, sg, b, Tt, eta0, spread)) continue;
        for (int start = 0; start < 2; ++start) {
            FitCount fc = kNoCount;
            o[3 * start] = closed_fit<df2>(g, b, Tt, eta0, start ? dw + 10 * c : nullptr, t[0], a, fc) ? 1.0 : 0.0;
            o[3 * start + 1] = fc.iters;
            o[3 * start + 2] = fc.evals;
        }
        float eta[10];
        FitCount fc = kNoCount;
        for (int q = 0; q < 10; ++q) eta[q] = eta0[q] + dw[10 * c + q];
        if (from_eta<df2>(eta, g) && closed_newton<df2>(g, b, N, Tt, t[0], tol, 40, fc)) o[6] = fc.iters;
    }
}

extern "C" void closed_fit_df2(int N, double half, double tol, int max_iter, int cases, const double* in, double* out) {
    run<df2>(N, half, tol, max_iter, cases, in, out);
}
extern "C" void closed_fit_f64(int N, double half, double tol, int max_iter, int cases, const double* in, double* out) {
    run<double>(N, half, tol, max_iter, cases, in, out);
}

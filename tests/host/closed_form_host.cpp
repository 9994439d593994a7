// closed_eval on the host against direct sums in long double, through two
// extern "C" functions (one per arithmetic). In: n_case rows of 13 doubles
// (density, mean of w about the box coordinates' origin [3], Theta [6] in
// velocity units xx xy xz yy yz zz, mean velocity [3]); the box is +-half on
// every axis with N cells. Out per row: 0 refused / 1 taken, then the largest
// error of the moments 1, d, d d relative to the density, and that of the
// Gram sums.
#include "device_shim.h"
#include "../../paper_2109_06743_gb300/csrc/closed_form.cuh"

using namespace vl;
using namespace vl::cf;
typedef long double LD;

static double val(df2 a) { return (double)a.hi + (double)a.lo; }
static double val(double a) { return a; }

template <class T>
static void run(int N, double half, int cases, const double* in, double* out) {
    for (int c = 0; c < cases; ++c) {
        const double *r = in + 13 * c, *th = r + 4, *u = r + 10;
        const double dv = 2.0 * half / N;
        const double sg[3] = {std::sqrt(th[0]), std::sqrt(th[3]), std::sqrt(th[5])};
        const double xy = th[1] / (sg[0] * sg[1]), xz = th[2] / (sg[0] * sg[2]), yz = th[4] / (sg[1] * sg[2]);
        const double det = 1 + 2 * xy * xz * yz - xy * xy - xz * xz - yz * yz;
        const double P[6] = {(1 - yz * yz) / det, (xz * yz - xy) / det, (xy * yz - xz) / det,
                             (1 - xz * xz) / det, (xy * xz - yz) / det, (1 - xy * xy) / det};
        const double K = std::pow(2 * M_PI, 1.5) * sg[0] * sg[1] * sg[2];
        Maxw<T> g;
        FitBox<T> b;
        g.L = num<T>(std::log(r[0]) - std::log(K) - 0.5 * std::log(det));
        b.K = num<T>(K);
        for (int q = 0; q < 6; ++q) g.P[q] = num<T>(P[q]);
        for (int a = 0; a < 3; ++a) {
            g.m[a] = num<T>(r[1 + a]);
            b.wc[a] = num<T>(-u[a] / sg[a]);
            b.h[a] = num<T>(dv / sg[a]);
        }
        Eval<T> e;
        double* o = out + 3 * c;
        o[0] = closed_eval<T>(g, b, N, true, e) ? 1.0 : 0.0;
        o[1] = o[2] = 0.0;
        if (o[0] == 0.0) continue;
        LD A[10], G[35], m[3], p[6], wc[3], h[3];
        for (auto& x : A) x = 0;
        for (auto& x : G) x = 0;
        for (int a = 0; a < 3; ++a) {
            m[a] = val(g.m[a]);
            wc[a] = val(b.wc[a]);
            h[a] = val(b.h[a]);
        }
        for (int q = 0; q < 6; ++q) p[q] = val(g.P[q]);
        for (int k = 0; k < N; ++k)
            for (int j = 0; j < N; ++j)
                for (int i = 0; i < N; ++i) {
                    const int ix[3] = {i, j, k};
                    LD d[3], pw[3][5];
                    for (int a = 0; a < 3; ++a) {
                        d[a] = wc[a] + h[a] * (ix[a] - (N - 1) / 2.0L) - m[a];
                        pw[a][0] = 1;
                        for (int q = 1; q < 5; ++q) pw[a][q] = pw[a][q - 1] * d[a];
                    }
                    const LD q = p[0] * d[0] * d[0] + p[3] * d[1] * d[1] + p[5] * d[2] * d[2] +
                                 2 * (p[1] * d[0] * d[1] + p[2] * d[0] * d[2] + p[4] * d[1] * d[2]);
                    const LD M = expl((LD)val(g.L) - q / 2);
                    for (int x = 0; x <= 4; ++x)
                        for (int y = 0; x + y <= 4; ++y)
                            for (int z = 0; x + y + z <= 4; ++z) G[mono4(x, y, z)] += M * pw[0][x] * pw[1][y] * pw[2][z];
                }
        const LD vol = (LD)val(b.K) / powl(2 * (LD)M_PIl, 1.5L) * h[0] * h[1] * h[2];
        for (auto& x : G) x *= vol;
        const double got[10] = {val(e.A0),    val(e.A1[0]), val(e.A1[1]), val(e.A1[2]), val(e.A2[0]),
                                val(e.A2[1]), val(e.A2[2]), val(e.A2[3]), val(e.A2[4]), val(e.A2[5])};
        for (int q = 0; q < 10; ++q) o[1] = std::fmax(o[1], (double)fabsl((got[q] - G[q]) / G[0]));
        for (int q = 0; q < 35; ++q) o[2] = std::fmax(o[2], (double)fabsl(((LD)e.C[q] - G[q]) / G[0]));
    }
}

extern "C" void closed_form_df2(int N, double half, int cases, const double* in, double* out) {
    run<df2>(N, half, cases, in, out);
}
extern "C" void closed_form_f64(int N, double half, int cases, const double* in, double* out) {
    run<double>(N, half, cases, in, out);
}

// The Newton fit of the discrete ten-moment Maxwellians (moment fitting,
// paper Sec. 2.2 and Algorithm 1) on the closed-form evaluation of
// closed_form.cuh: one thread per fit, both precisions.
//
// The iteration is that of the direct kernels (newton.cuh, newton64.cuh): the
// natural parameters eta of M = exp(eta . phi(w)), full Newton steps with the
// Gram matrix, the same start, tolerance and damping test. It is carried in
// the form M = exp(L - d.P d / 2), d = w - m, about the Maxwellian's own mean
// (a linear change of phi, which Newton's method does not see), so that a
// step (delta_0, delta_1, delta_2) is P <- P - 2 delta_2, m <- m + P^-1
// delta_1, L <- L + delta_0 + delta_1 . P^-1 delta_1 / 2.
//
// What the closed form refuses, a step that fails the descent test, a fit that
// does not converge and (FP32 mode) one whose line parameters would round
// differently (rounds_alike) go on a list; the direct kernels then fit those
// from their start as before. Results agree to the fit tolerance either way.
//
// Why one thread per fit: an evaluation is some 10 k operations with little
// parallelism inside (three axes, two sides), against 152 k for the direct
// sums by eight lanes; 65536 fits fill the chip 14 warps deep per SM.
// Measured (GB300), closed form and list: 65536 cold fits of 16^3 Harris ions
// 2.23 -> 0.44 ms (0.25 + 0.15, and theta), 65536 network-started fits of 12^3
// asymmetric-sheet electrons 2.11 -> 0.73-0.86 ms, 16384 fits in FP64 mode 5.08 -> 0.42
// ms. What bounds it: the slowest warps' chains of dependent operations (5.6
// cycles per instruction and warp, 10 warps per SM); blocks of 32 to 128 threads
// at 96 to 168 registers are all within 3%.
#pragma once

#include "closed_form.cuh"
#include "common.cuh"
#include "kernels.cuh"
#include "mlp_common.cuh"

namespace vl {
namespace cf {

constexpr int kCoefC = 16;

// dl = -J^-1 G, J the Gram matrix packed from the central sums C, by LDL^T
template <typename J>
CF_FN bool newton_direction(const J (&C)[35], const J (&G)[10], J (&dl)[10]) {
    J A[55], di[10];
    bool ok = true;
    CF_UNROLL
    for (int a = 0; a < 10; ++a)
        CF_UNROLL
        for (int b = 0; b <= a; ++b)
            A[tri(a, b)] = C[mono4(expo(a, 0) + expo(b, 0), expo(a, 1) + expo(b, 1), expo(a, 2) + expo(b, 2))];
    CF_UNROLL
    for (int j = 0; j < 10; ++j) {
        // row j: u_jk = a_jk - sum u_ji l_ki in place, then l_jk = u_jk / d_k
        CF_UNROLL
        for (int k = 0; k < j; ++k)
            CF_UNROLL
            for (int i = 0; i < k; ++i) A[tri(j, k)] -= A[tri(j, i)] * A[tri(k, i)];
        J d = A[tri(j, j)];
        CF_UNROLL
        for (int k = 0; k < j; ++k) {
            const J u = A[tri(j, k)];
            A[tri(j, k)] = u * di[k];
            d -= u * A[tri(j, k)];
        }
        ok = ok && d > J(0);
        di[j] = recip(d);
    }
    CF_UNROLL
    for (int i = 0; i < 10; ++i) {
        J s = -G[i];
        CF_UNROLL
        for (int k = 0; k < i; ++k) s -= A[tri(i, k)] * dl[k];
        dl[i] = s;
    }
    CF_UNROLL
    for (int i = 9; i >= 0; --i) {
        J s = dl[i] * di[i];
        CF_UNROLL
        for (int k = i + 1; k < 10; ++k) s -= A[tri(k, i)] * dl[k];
        dl[i] = s;
    }
    return ok;
}

// 3 x 3 symmetric inverse (xx, xy, xz, yy, yz, zz); false unless positive definite
template <typename J>
CF_FN bool inverse3(const J (&P)[6], J (&S)[6], J* det_out = nullptr) {
    const J c0 = P[3] * P[5] - P[4] * P[4], c1 = P[2] * P[4] - P[1] * P[5], c2 = P[1] * P[4] - P[2] * P[3],
            c5 = P[0] * P[3] - P[1] * P[1];
    const J det = P[0] * c0 + P[1] * c1 + P[2] * c2;
    const J id = recip(det);
    S[0] = c0 * id;
    S[1] = c1 * id;
    S[2] = c2 * id;
    S[3] = (P[0] * P[5] - P[2] * P[2]) * id;
    S[4] = (P[1] * P[2] - P[0] * P[4]) * id;
    S[5] = c5 * id;
    if (det_out) *det_out = det;
    return P[0] > J(0) && c5 > J(0) && det > J(0);
}

CF_FN float sq_root(float x) { return sqrtf(x); }
CF_FN double sq_root(double x) { return sqrt(x); }
CF_FN float log_of(float x) { return logf(x); }
CF_FN double log_of(double x) { return log(x); }

struct FitCount {
    int iters;              // Newton steps, evaluations and those with Gram sums, of every pass
    unsigned evals, grams;
    float last, before;     // size of the last Newton step and of the one before it
    float res, prev;        // residuals after and before the last step (relative to n)
    float omitted;          // largest Eval::omitted of the pass
};

// thresholds of the direct kernels: damping test above kDamp n, Gram sums with
// the next evaluation where another step is likely
CF_FN bool far_off(float rel, float) { return rel > 1e-3f; }
CF_FN bool far_off(double rel, double) { return rel > 1e-6; }
CF_FN bool more_steps(float rel, float, float) { return rel > 1e-5f; }
CF_FN bool more_steps(double rel, double tol, double) { return 100.0 * rel * rel > tol; }

// Newton iteration from g to max |D - Tt| <= tol n. Returns false when the
// fit is left to the direct kernels.
template <typename T>
CF_FN bool closed_newton(Maxw<T>& g, const FitBox<T>& b, int N, const T (&Tt)[10], double n, double tol,
                         int max_iter, FitCount& cnt) {
    typedef typename Jac<T>::type J;
    const J nj = (J)n, tolj = (J)(tol * n);
    bool gram = true, check = false;
    T L0 = num<T>(0.0);
    J gd = J(0);
    CF_LOOP
    for (int it = 0;; ++it) {
        Eval<T> e;
        if (!closed_eval<T>(g, b, N, gram, e)) return false;
        ++cnt.evals;
        cnt.grams += gram ? 1u : 0u;
        cnt.omitted = it == 0 ? e.omitted : fmaxf(cnt.omitted, e.omitted);
        // moments about w = 0, residual G
        T D[10], G[10];
        D[0] = e.A0;
        CF_UNROLL
        for (int a = 0; a < 3; ++a) D[1 + a] = add(e.A1[a], mul(g.m[a], e.A0));
        CF_UNROLL
        for (int a = 0; a < 3; ++a)
            CF_UNROLL
            for (int c = a; c < 3; ++c)
                D[4 + sym(a, c)] = add(e.A2[sym(a, c)], add(mul(g.m[a], D[1 + c]), mul(g.m[c], e.A1[a])));
        J gmax = J(0);
        bool fin = true;
        CF_UNROLL
        for (int q = 0; q < 10; ++q) {
            G[q] = sub(D[q], Tt[q]);
            const J v = fabs(jac(G[q]));
            fin = fin && v < J(1e30);
            gmax = v > gmax ? v : gmax;
        }
        if (!fin) return false;
        // dual L(eta) = D_0 - eta . T at a trial step far from the solution
        const J rel = gmax / nj;
        const bool far = far_off(rel, J(0));
        if (check || far) {
            T qT = mul(g.L, Tt[0]);
            CF_UNROLL
            for (int a = 0; a < 3; ++a)
                CF_UNROLL
                for (int c = a; c < 3; ++c) {
                    const T t2 = add(sub(Tt[4 + sym(a, c)], add(mul(g.m[a], Tt[1 + c]), mul(g.m[c], Tt[1 + a]))),
                                     mul(mul(g.m[a], g.m[c]), Tt[0]));
                    qT = sub(qT, scale(mul(g.P[sym(a, c)], t2), a == c ? 0.5f : 1.0f));
                }
            const T L1 = sub(e.A0, qT);
            if (check && !(jac(sub(L1, L0)) <= J(1e-4) * gd)) return false;
            L0 = L1;
        }
        if (gmax <= tolj) {
            cnt.res = (float)rel;
            return true;
        }
        if (it >= max_iter) return false;
        if (!gram) {
            // another step after all: the same evaluation with the Gram sums
            gram = true;
            check = false;
            --it;
            continue;
        }
        // residual about the mean, Newton direction there
        J Gj[10], Gc[10], m[3], dl[10];
        CF_UNROLL
        for (int q = 0; q < 10; ++q) Gj[q] = jac(G[q]);
        CF_UNROLL
        for (int a = 0; a < 3; ++a) m[a] = jac(g.m[a]);
        Gc[0] = Gj[0];
        CF_UNROLL
        for (int a = 0; a < 3; ++a) Gc[1 + a] = Gj[1 + a] - m[a] * Gj[0];
        CF_UNROLL
        for (int a = 0; a < 3; ++a)
            CF_UNROLL
            for (int c = a; c < 3; ++c)
                Gc[4 + sym(a, c)] = Gj[4 + sym(a, c)] - m[a] * Gj[1 + c] - m[c] * Gc[1 + a];
        if (!newton_direction<J>(e.C, Gc, dl)) return false;
        gd = J(0);
        J big = J(0);
        CF_UNROLL
        for (int q = 0; q < 10; ++q) {
            gd += Gc[q] * dl[q];
            const J v = fabs(dl[q]);
            big = v > big ? v : big;
        }
        cnt.before = it == 0 ? 0.f : cnt.last;
        cnt.last = (float)big;
        cnt.prev = (float)rel;
        check = far;
        gram = more_steps(rel, (J)tol, J(0));
        // the step
        const T z = num<T>(0.0);
        J P[6], S[6], dm[3];
        CF_UNROLL
        for (int a = 0; a < 3; ++a)
            CF_UNROLL
            for (int c = a; c < 3; ++c) {
                const int q = sym(a, c);
                g.P[q] = add(g.P[q], from(a == c ? J(-2) * dl[4 + q] : -dl[4 + q], z));
                P[q] = jac(g.P[q]);
            }
        if (!inverse3<J>(P, S)) return false;
        J dq = dl[0];
        CF_UNROLL
        for (int a = 0; a < 3; ++a) {
            dm[a] = S[sym(a, 0)] * dl[1] + S[sym(a, 1)] * dl[2] + S[sym(a, 2)] * dl[3];
            dq += J(0.5) * dm[a] * dl[1 + a];
            g.m[a] = add(g.m[a], from(dm[a], z));
        }
        g.L = add(g.L, from(dq, z));
        ++cnt.iters;
    }
}

// Scaled coordinates and start of one fit in J's arithmetic. u0 and sigma
// are the targets' mean and standard deviations rounded to J (any values
// define a valid change of variables: Tt below is transformed in FP64).
// eta0 is the continuous Maxwellian of the targets in w. False for targets a
// fit rejects (n <= 0 or not finite, Theta not positive definite).
template <typename T>
CF_FN bool closed_setup(const double (&t)[10], const FitArgs& a, double (&u0)[3], double (&sg)[3], FitBox<T>& b,
                        T (&Tt)[10], typename Jac<T>::type (&eta0)[10], float& spread) {
    typedef typename Jac<T>::type J;
    const double n = t[0];
    if (!(n > 0.0) || !(n < 1e300)) return false;
    bool fin = true;
    CF_UNROLL
    for (int q = 0; q < 10; ++q) fin = fin && fabs(t[q]) < 1e300;
    if (!fin) return false;
    const J nj = (J)n;
    J u[3], Th[6], s[3];
    CF_UNROLL
    for (int q = 0; q < 3; ++q) u[q] = (J)t[1 + q] / nj;
    CF_UNROLL
    for (int p = 0; p < 3; ++p)
        CF_UNROLL
        for (int q = p; q < 3; ++q) Th[sym(p, q)] = (J)t[4 + sym(p, q)] / nj - u[p] * u[q];
    J Pd[6];
    if (!(Th[3] > J(0) && Th[5] > J(0)) || !inverse3<J>(Th, Pd)) return false;
    // e-folds from the peak to the farthest corner, as fit_select counts them
    spread = 0.f;
    CF_UNROLL
    for (int q = 0; q < 3; ++q) {
        s[q] = sq_root(Th[sym(q, q)]);
        u0[q] = (double)u[q];
        sg[q] = (double)s[q];
        const double rs = 1.0 / sg[q];
        b.h[q] = num<T>(a.dv[q] * rs);
        b.wc[q] = num<T>((a.vmin[q] + 0.5 * a.nv * a.dv[q] - u0[q]) * rs);
        const float ext = fmaxf((float)(a.vmax[q] - u0[q]), (float)(u0[q] - a.vmin[q]));
        spread += ext * ext / (2.f * (float)Th[sym(q, q)]);
    }
    b.K = num<T>(15.749609945722417 * sg[0] * sg[1] * sg[2]);  // (2 pi)^(3/2) sigma_x sigma_y sigma_z
    Tt[0] = num<T>(n);
    const double rs[3] = {1.0 / sg[0], 1.0 / sg[1], 1.0 / sg[2]};
    CF_UNROLL
    for (int q = 0; q < 3; ++q) Tt[1 + q] = num<T>((t[1 + q] - n * u0[q]) * rs[q]);
    CF_UNROLL
    for (int p = 0; p < 3; ++p)
        CF_UNROLL
        for (int q = p; q < 3; ++q)
            Tt[4 + sym(p, q)] =
                num<T>((t[4 + sym(p, q)] - u0[p] * t[1 + q] - u0[q] * t[1 + p] + n * u0[p] * u0[q]) * (rs[p] * rs[q]));
    // the continuous Maxwellian of the targets
    J Cw[6], P[6], mw[3], det;
    CF_UNROLL
    for (int q = 0; q < 3; ++q) mw[q] = jac(Tt[1 + q]) / nj;
    CF_UNROLL
    for (int p = 0; p < 3; ++p)
        CF_UNROLL
        for (int q = p; q < 3; ++q) Cw[sym(p, q)] = jac(Tt[4 + sym(p, q)]) / nj - mw[p] * mw[q];
    if (!inverse3<J>(Cw, P, &det)) return false;
    J quad = J(0);
    CF_UNROLL
    for (int p = 0; p < 3; ++p) {
        eta0[1 + p] = P[sym(p, 0)] * mw[0] + P[sym(p, 1)] * mw[1] + P[sym(p, 2)] * mw[2];
        quad += mw[p] * eta0[1 + p];
    }
    eta0[0] = log_of(nj) - J(1.5) * log_of(J(6.283185307179586477)) - J(0.5) * (log_of(det) + J(2) * log_of(s[0] * s[1] * s[2])) -
              J(0.5) * quad;
    CF_UNROLL
    for (int p = 0; p < 3; ++p)
        CF_UNROLL
        for (int q = p; q < 3; ++q) eta0[4 + sym(p, q)] = (p == q ? J(-0.5) : J(-1)) * P[sym(p, q)];
    return true;
}

// M(w) = exp(eta . phi(w)) about its own mean; false unless a Gaussian
template <typename T>
CF_FN bool from_eta(const typename Jac<T>::type (&eta)[10], Maxw<T>& g) {
    typedef typename Jac<T>::type J;
    const T z = num<T>(0.0);
    const J P[6] = {J(-2) * eta[4], -eta[5], -eta[6], J(-2) * eta[7], -eta[8], J(-2) * eta[9]};
    J S[6], L = eta[0];
    if (!inverse3<J>(P, S)) return false;
    CF_UNROLL
    for (int q = 0; q < 6; ++q) g.P[q] = from(P[q], z);
    CF_UNROLL
    for (int p = 0; p < 3; ++p) {
        const J m = S[sym(p, 0)] * eta[1] + S[sym(p, 1)] * eta[2] + S[sym(p, 2)] * eta[3];
        L += J(0.5) * m * eta[1 + p];
        g.m[p] = from(m, z);
    }
    g.L = from(L, z);
    return true;
}

// The fit from the start eta0, or first from eta0 and the network's prediction dw
// if there is one (the guard of its inference writes NaN rows for the fits it
// rejects). One way out of the loop: with a return from inside it the lanes of a
// warp did not come together again (network-started fits 840 -> 1310 us).
CF_FN bool predicted(const float* dw) { return dw && fabsf(dw[0]) < 1e30f; }

template <typename T>
CF_FN bool closed_fit(Maxw<T>& g, const FitBox<T>& b, const T (&Tt)[10], const typename Jac<T>::type (&eta0)[10],
                      const float* dw, double n, const FitArgs& a, FitCount& fc) {
    typedef typename Jac<T>::type J;
    bool good = false;
    CF_LOOP
    for (int pass = predicted(dw) ? 0 : 1; pass < 2 && !good; ++pass) {
        J eta[10];
        CF_UNROLL
        for (int q = 0; q < 10; ++q) {
            const float d = pass == 0 ? dw[q] : 0.f;
            eta[q] = eta0[q] + (fabsf(d) < 1e30f ? (J)d : J(0));
        }
        good = from_eta<T>(eta, g) && closed_newton<T>(g, b, a.nv, Tt, n, a.tol, a.max_iter, fc);
    }
    return good;
}

// FP32 mode: the exchange rounds a fit's line parameters (fit.cu) to float,
// and one unit in the last place of L moves the whole Maxwellian by 5e-7. A fit
// with a parameter that close to a rounding boundary is decided by the direct
// kernel, so that f does not depend on which kernel made a fit.
//
// fit_slack: how far two fits of the same targets may lie apart, by the rounding
// of their sums, by a few 1e-6 of the last Newton step (FP32 Jacobian) and, where
// a residual lies at the tolerance, by one step more or less (measured against the
// direct kernels over 1.6e5 fits of the workloads: 5e-13, 1.8e-6 of the step, the
// residual or the step). Where the Gram sums leave out more than FP32 resolves
// (Eval::omitted; narrow Maxwellians near a face, two faces at once), the last step
// may leave a remainder of the size of the residual rather than 2e-6 of the step,
// and the direct kernel may need a step less: what is left out, times the step
// before.
CF_FN double fit_slack(const FitCount& fc, double tol) {
    const double last = fc.last, res = fc.res;
    double eps = 8e-13 + 2e-6 * last;
    if (fc.omitted > 1e-7f || res > 0.9 * tol) eps += res;
    if ((double)fc.prev < 1.1 * tol + 10.0 * fc.omitted * fc.before) eps += 2.2 * last;
    return eps;
}

// Off-diagonal parameters below 1/64 have a finer last place: it moves the
// Maxwellian by less than 1e-8, but a value that falls below zero makes the
// exchange rescale its cell, and that moves it by a rounding of f. They count down
// to 1/512, with the typical difference of two fits (1.5e-13) instead of the
// largest; below, the last place is lost in the exchange's own roundings. (Cells of
// 512 x 256 x 16^3 that differ from the direct kernels' after an exchange, of 1.6
// million: 5 without them, one by 9e-8; 1 with them, by 6e-9. Fits of 256 x 128 ions
// 429 -> 447 us.)
template <typename T>
CF_FN bool rounds_alike(const Maxw<T>& g, const FitBox<T>& b, const double (&u0)[3], const double (&sg)[3], double tol,
                        const FitArgs& a, const FitCount& fc) {
    const double eps = fit_slack(fc, tol);
    auto alike = [](double p, double d) { return (float)(p - d) == (float)(p + d); };
    const double e2 = 1.5 * eps, e4 = 3.0 * eps, es = (eps - 6.5e-13) / e4;
    auto small = [&](double p, double d) {
        return fabs(p) < 0.001953125 || alike(p, fabs(p) < 0.015625 ? d * es : d);
    };
    double h[3], P[6];
    bool ok = alike(wide_of(g.L), e2);
    CF_UNROLL
    for (int q = 0; q < 3; ++q) {
        h[q] = wide_of(b.h[q]);
        const double is = sg[q] * a.inv_dv[q];
        ok = ok && alike((u0[q] - a.vmin[q]) * a.inv_dv[q] - 0.5 + is * wide_of(g.m[q]), e2 * is);
    }
    CF_UNROLL
    for (int p = 0; p < 3; ++p)
        CF_UNROLL
        for (int q = p; q < 3; ++q) P[sym(p, q)] = h[p] * h[q] * wide_of(g.P[sym(p, q)]);
    const double iz = 1.0 / P[5], gx = -P[2] * iz, gy = -P[4] * iz;
    ok = ok && alike(0.5 * P[5], e2 * P[5]) && alike(P[0] + P[2] * gx, e4 * P[0]) && alike(P[3] + P[4] * gy, e4 * P[3]);
    return ok && small(gx, e4) && small(gy, e4) && small(P[1] + P[2] * gy, e4 * h[0] * h[1]);
}

#ifdef __CUDACC__

// Thread g fits Maxwellian g & 1 (0: the moments of f, 1: the fluid's,
// rescaled by n_V / n_F and written back) of cell g >> 1. Fits left to the
// direct kernels are appended to a.todo. With a.sel the kernel also reduces
// what chooses the direct kernel (see kernels.cuh).
template <typename T>
__global__ void __launch_bounds__(128, sizeof(typename Jac<T>::type) == 4 ? 3 : 2) closed_fit_kernel(FitArgs a) {
    typedef typename Jac<T>::type J;
    constexpr bool kF64 = sizeof(J) == 8;
    __shared__ unsigned long long cnt[VL_NSTATS];
    if (threadIdx.x < VL_NSTATS) cnt[threadIdx.x] = 0ull;
    __syncthreads();
    const long long fit = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool have = fit < 2 * a.ncell;
    FitCount fc = {0, 0u, 0u, 0.f, 0.f, 0.f, 1.f, 0.f};
    bool left = false, empty = false;
    unsigned warm = 0u;
    unsigned long long top = 0ull, wide = 0ull;
    if (have) {
        const long long cell = fit >> 1;
        const bool fl = (fit & 1) != 0;
        double t[10];
        const double nV = a.vmom[cell * 20];
        const double* src = fl ? a.fluid + cell * 10 : a.vmom + cell * 20;
        bool bad = !(src[0] >= 0.0);
#pragma unroll
        for (int q = 0; q < 10; ++q) {
            t[q] = src[q];
            bad = bad || !isfinite(t[q]);
        }
        if (bad && a.numeric) *reinterpret_cast<volatile int*>(a.numeric) = VL_ENUMERIC;
        if (fl) {
            const double sc = t[0] > 0.0 ? nV / t[0] : 0.0;
#pragma unroll
            for (int q = 0; q < 10; ++q) {
                t[q] *= sc;
                a.fluid[cell * 10 + q] = t[q];
            }
        }
        double u0[3], sg[3];
        FitBox<T> b;
        T Tt[10];
        J eta0[10];
        float spread = 0.f;
        double* coef = (fl ? a.coef_f : a.coef_v) + cell * kCoefC;
        bool good = false;
        // no density: invalid in either direct kernel as well. Written here, as cells a
        // species is absent from can be half the grid (32768 fits of 12^3, half of
        // them empty, 930 -> 325 us; by direct sums alone 820)
        empty = !(t[0] > 0.0) || !isfinite(t[0]);
        if (empty) {
            a.status[fit] = 2;
#pragma unroll
            for (int q = 0; q < kCoefC; ++q) coef[q] = 0.0;
        } else if (closed_setup<T>(t, a, u0, sg, b, Tt, eta0, spread)) {
            if (nV > 0.0 && isfinite(nV)) {
                top = (unsigned long long)__double_as_longlong(nV);
                if (spread > 60.f) wide = top;
            }
            Maxw<T> g;
            const float* dw = a.warm ? a.warm + fit * 10 : nullptr;
            const bool started = predicted(dw);
            good = closed_fit<T>(g, b, Tt, eta0, dw, t[0], a, fc);
            if (!kF64 && good) good = rounds_alike<T>(g, b, u0, sg, a.tol, a, fc);
            if (good) {
                warm = started ? 1u : 0u;
                coef[0] = wide_of(g.L);
                coef[1] = coef[2] = coef[3] = 0.0;
#pragma unroll
                for (int p = 0; p < 3; ++p) {
#pragma unroll
                    for (int q = p; q < 3; ++q) coef[4 + sym(p, q)] = (p == q ? -0.5 : -1.0) * wide_of(g.P[sym(p, q)]);
                    coef[10 + p] = u0[p] + sg[p] * wide_of(g.m[p]);
                    coef[13 + p] = sg[p];
                }
                a.status[fit] = 0;
                if (a.harvest) {
                    const unsigned long long slot = atomicAdd(a.harvest_count, 1ull);
                    if (slot < (unsigned long long)a.harvest_cap) {
                        float* smp = a.harvest + slot * mlp::kSample;
                        float x[mlp::kIn];
                        const bool ok = mlp::fit_inputs(t, a.vmin, a.dv, a.vmax, x);
                        for (int q = 0; q < mlp::kIn; ++q) smp[q] = x[q];
                        smp[22] = ok ? 1.f : 0.f;
                        smp[23] = 0.f;
                        // eta* about w = 0
                        T e0 = g.L;
#pragma unroll
                        for (int p = 0; p < 3; ++p) {
                            const T l = add(add(mul(g.P[sym(p, 0)], g.m[0]), mul(g.P[sym(p, 1)], g.m[1])),
                                            mul(g.P[sym(p, 2)], g.m[2]));
                            e0 = sub(e0, scale(mul(l, g.m[p]), 0.5f));
                            smp[mlp::kIn + 1 + p] = (float)jac(sub(l, from(eta0[1 + p], l)));
#pragma unroll
                            for (int q = p; q < 3; ++q)
                                smp[mlp::kIn + 4 + sym(p, q)] = (float)jac(
                                    sub(scale(g.P[sym(p, q)], p == q ? -0.5f : -1.f), from(eta0[4 + sym(p, q)], l)));
                        }
                        smp[mlp::kIn] = (float)jac(sub(e0, from(eta0[0], e0)));
                    }
                }
            }
        }
        left = !good && !empty;
        if (left) fc.iters = 0;  // the direct kernel's are the fit's; evaluations done are work done
    }
    if (kF64) {
        if (left) a.todo[atomicAdd(a.ntodo, 1u)] = (unsigned long long)fit;
    } else {
        // eight lanes hold four cells: V fits on the even ones, F on the odd
        const unsigned m = __ballot_sync(0xffffffffu, left) >> (threadIdx.x & 24);
        const int w = threadIdx.x & 7;
        if (w < 2) {
            const unsigned v = m >> w, keep = (v & 1u) | ((v >> 1) & 2u) | ((v >> 2) & 4u) | ((v >> 3) & 8u);
            if (keep) a.todo[atomicAdd(a.ntodo, 1u)] = (unsigned long long)((fit >> 3) * 2 + w) << 4 | keep;
        }
    }
    // CTA totals, then one atomic per counter
    constexpr unsigned kAll = 0xffffffffu;
    const unsigned it = __reduce_add_sync(kAll, (unsigned)fc.iters), ev = __reduce_add_sync(kAll, fc.evals),
                   gr = __reduce_add_sync(kAll, fc.grams), wa = __reduce_add_sync(kAll, warm),
                   em = __reduce_add_sync(kAll, empty ? 1u : 0u);
    if ((threadIdx.x & 31) == 0) {
        if (it) atomicAdd_block(&cnt[CNT_ITERS], (unsigned long long)it);
        if (ev) atomicAdd_block(&cnt[kF64 ? CNT_EVAL64_M : CNT_EVAL_M], (unsigned long long)ev);
        if (gr) atomicAdd_block(&cnt[kF64 ? CNT_EVAL64_G : CNT_EVAL_G], (unsigned long long)gr);
        if (wa) atomicAdd_block(&cnt[CNT_WARM], (unsigned long long)wa);
        if (em) atomicAdd_block(&cnt[CNT_INVALID], (unsigned long long)em);
    }
    if (a.sel) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            top = max(top, __shfl_xor_sync(kAll, top, o));
            wide = max(wide, __shfl_xor_sync(kAll, wide, o));
        }
        if ((threadIdx.x & 31) == 0) {
            if (top) atomicMax(&a.sel[0], top);
            if (wide) atomicMax(&a.sel[1], wide);
        }
    }
    __syncthreads();
    if (threadIdx.x < VL_NSTATS && cnt[threadIdx.x]) atomicAdd(&a.counters[threadIdx.x], cnt[threadIdx.x]);
}

#endif  // __CUDACC__

}  // namespace cf
}  // namespace vl

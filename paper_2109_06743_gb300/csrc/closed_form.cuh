// The discrete moments of a ten-moment Maxwellian on a velocity block in
// closed form (the moment fit's evaluation, paper Sec. 2.2 and Algorithm 1:
// the fitted Maxwellians' midpoint moments of degree <= 2 equal the targets).
//
// A Newton evaluation needs D_q = dv^3 sum_i M(v_i) phi_q(v_i) over the N^3
// cells. Summing the cells costs N^3 exponential recurrences; the sum over
// the whole lattice has a closed form, and what the box cuts off is small:
//   sum_box = sum_lattice - sum_x-out - sum_y-out - sum_z-out
//             + sum_xy-out + sum_xz-out + sum_yz-out - sum_xyz-out
// (inclusion and exclusion over the axes along which a cell lies outside).
//   * sum_lattice: Poisson summation. The zero mode is the Gaussian integral;
//     mode k adds the same integral with the mean moved by -2 pi i Sigma k
//     and the factor exp(-2 pi^2 k.Sigma k - 2 pi i k.mu), in index units.
//     Above 1.45 cells per standard deviation every mode is below rounding;
//     narrower Maxwellians take the modes up to |k|^2 = 5.
//   * sum_a-out: the marginal along axis a is a one-dimensional Gaussian,
//     summed over its few cells outside the box on either side by the
//     recurrence M <- M r, r <- r rr; along the other two axes the
//     conditional moments are linear and quadratic in the distance.
//   * the doubly and triply outside cells weigh the product of the tails
//     (1e-12 and less for a box of five standard deviations): FP32 sums over
//     the corners' first few cells.
// About 10 thousand operations instead of 37 N^3. closed_eval refuses (returns
// false) whatever it cannot give to rounding: means near or beyond a face,
// strongly correlated or very narrow covariances, heavy corners, narrow
// Maxwellians close to a face in FP32 mode; such fits take the direct sums
// (newton.cuh, newton64.cuh).
//
// T is the arithmetic: df2 (double-float pairs on the FP32 pipe, FP32 mode)
// or double (FP64 mode). J is that of the Jacobian (Gram matrix): float with
// df2, double with double. The functions also compile for the host, where
// the tests compare them with direct sums.
#pragma once

#include <math.h>

#include "df64.cuh"
#include "fit_index.cuh"

namespace vl {
namespace cf {

#ifdef __CUDACC__
#define CF_FN __device__ __forceinline__
#else
#define CF_FN inline
#endif
#ifdef __CUDA_ARCH__
#define CF_UNROLL _Pragma("unroll")
#define CF_LOOP _Pragma("unroll 1")
#else
#define CF_UNROLL
#define CF_LOOP
#endif

// ------------------------------------------------------------- arithmetic

template <typename T>
struct Jac;
template <>
struct Jac<df2> {
    typedef float type;
};
template <>
struct Jac<double> {
    typedef double type;
};

// sum of two pairs with the low parts added in FP32: the error is a few
// 2^-48 of the larger operand
CF_FN df2 add(df2 a, df2 b) {
    df2 s = df2_two_sum(a.hi, b.hi);
    return df2_qtwo_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
CF_FN df2 neg(df2 a) { return {-a.hi, -a.lo}; }
CF_FN df2 sub(df2 a, df2 b) { return add(a, neg(b)); }
CF_FN df2 mul(df2 a, df2 b) { return df2_mul(a, b); }
CF_FN df2 scale(df2 a, float b) { return df2_mulf(a, b); }
CF_FN float hi(df2 a) { return a.hi; }
CF_FN float jac(df2 a) { return a.hi + a.lo; }
// approximate reciprocal and reciprocal root (a few ulp)
#ifdef __CUDA_ARCH__
CF_FN float recip(float x) { return __fdividef(1.0f, x); }
CF_FN float rroot(float x) { return rsqrtf(x); }
#else
CF_FN float recip(float x) { return 1.0f / x; }
CF_FN float rroot(float x) { return 1.0f / sqrtf(x); }
#endif
CF_FN double recip(double x) { return 1.0 / x; }
// 1 / b: float reciprocal, then the remainder to second order
CF_FN df2 inv(df2 b) {
    const float r = recip(b.hi);
    const float e = fmaf(-b.lo, r, fmaf(-b.hi, r, 1.0f));
    return df2_qtwo_sum(r, r * fmaf(e, e, e));
}
// 1 / sqrt(b): with y near it and e = 1 - b y^2, y (1 + e/2 + 3 e^2/8)
CF_FN df2 rsqrt2(df2 b) {
    const float y = rroot(b.hi);
    const float y2 = __fmul_rn(y, y);
    const df2 q = df2_mul(b, df2{y2, fmaf(y, y, -y2)});
    const float e = __fsub_rn(__fsub_rn(1.0f, q.hi), q.lo);
    return df2_qtwo_sum(y, y * e * fmaf(0.375f, e, 0.5f));
}
CF_FN df2 expt(df2 a) { return df2_exp(a); }

CF_FN double add(double a, double b) { return a + b; }
CF_FN double neg(double a) { return -a; }
CF_FN double sub(double a, double b) { return a - b; }
CF_FN double mul(double a, double b) { return a * b; }
CF_FN double scale(double a, float b) { return a * (double)b; }
CF_FN float hi(double a) { return (float)a; }
CF_FN double jac(double a) { return a; }
CF_FN double inv(double b) { return 1.0 / b; }
CF_FN double rsqrt2(double b) { return 1.0 / sqrt(b); }
CF_FN double expt(double a) { return exp(a); }

template <typename T>
CF_FN T num(double x);
template <>
CF_FN df2 num<df2>(double x) { return {(float)x, (float)(x - (double)(float)x)}; }
template <>
CF_FN double num<double>(double x) { return x; }
// a value of the Jacobian's arithmetic in T
CF_FN df2 from(float x, df2) { return {x, 0.f}; }
CF_FN double from(double x, double) { return x; }
CF_FN double from(float x, double) { return (double)x; }

CF_FN double wide_of(df2 a) { return (double)a.hi + (double)a.lo; }
CF_FN double wide_of(double a) { return a; }
// a value in V: FP64, or FP32 without the rest
template <typename V, typename T>
CF_FN V plain(T a) {
    return sizeof(V) == 8 ? (V)wide_of(a) : (V)hi(a);
}

CF_FN float expj(float x) { return expf(x); }
CF_FN double expj(double x) { return exp(x); }

// (cos, sin)(2 pi x) for any x of moderate size: the nearest quarter turn is
// taken off exactly, the rest (|theta| <= pi/4) goes through Taylor series,
// whose terms beyond theta^8 need FP32 only
CF_FN void cossin(df2 x, df2& c, df2& s) {
    const float q = rintf(4.0f * x.hi);
    const df2 y = add(x, df2{-0.25f * q, 0.f});
    const df2 th = mul(y, num<df2>(6.283185307179586476925));
    const df2 t2 = mul(th, th);
    const float z = t2.hi;
    // cos = 1 - t2/2 (1 - t2/12 (1 - t2/30 (1 - t2/56 (...))))
    float tc = 1.0f - z * (1.0f / 90.0f) * (1.0f - z * (1.0f / 132.0f) * (1.0f - z * (1.0f / 182.0f)));
    df2 a = sub(df2{1.f, 0.f}, scale(mul(t2, num<df2>(1.0 / 56.0)), tc));
    a = sub(df2{1.f, 0.f}, mul(mul(t2, num<df2>(1.0 / 30.0)), a));
    a = sub(df2{1.f, 0.f}, mul(mul(t2, num<df2>(1.0 / 12.0)), a));
    const df2 co = sub(df2{1.f, 0.f}, mul(scale(t2, 0.5f), a));
    float ts = 1.0f - z * (1.0f / 110.0f) * (1.0f - z * (1.0f / 156.0f) * (1.0f - z * (1.0f / 210.0f)));
    df2 b = sub(df2{1.f, 0.f}, scale(mul(t2, num<df2>(1.0 / 72.0)), ts));
    b = sub(df2{1.f, 0.f}, mul(mul(t2, num<df2>(1.0 / 42.0)), b));
    b = sub(df2{1.f, 0.f}, mul(mul(t2, num<df2>(1.0 / 20.0)), b));
    b = sub(df2{1.f, 0.f}, mul(mul(t2, num<df2>(1.0 / 6.0)), b));
    const df2 si = mul(th, b);
    const int k = ((int)q) & 3;
    c = k == 0 ? co : (k == 1 ? neg(si) : (k == 2 ? neg(co) : si));
    s = k == 0 ? si : (k == 1 ? co : (k == 2 ? neg(si) : neg(co)));
}
CF_FN void cossin(double x, double& c, double& s) {
    const double r = x - rint(x);
#ifdef __CUDA_ARCH__
    sincospi(2.0 * r, &s, &c);
#else
    c = cos(6.283185307179586476925 * r);
    s = sin(6.283185307179586476925 * r);
#endif
}

// index of the pair (a, b) in xx, xy, xz, yy, yz, zz
CF_FN constexpr int sym(int a, int b) { return a <= b ? a * (5 - a) / 2 + b : b * (5 - b) / 2 + a; }

// ------------------------------------------------------------------- state

// M(w) = exp(L - (w - m).P (w - m) / 2), w the fit's scaled coordinates
template <typename T>
struct Maxw {
    T L, m[3], P[6];
};

// the box in scaled coordinates: centre wc, cell width h, and K =
// (2 pi)^(3/2) sigma_x sigma_y sigma_z (lattice sum times dv^3 = K exp(L) / sqrt(det P))
template <typename T>
struct FitBox {
    T wc[3], h[3], K;
};

// what an evaluation gives: A = moments 1, d, d d (d = w - m) times dv^3,
// the covariance S = P^-1, and the Gram sums C of degree <= 4 in d (mono4). C
// leaves out the doubly and triply outside cells, the tails' modes and the far
// modes; omitted is the largest weight (of degree <= 2) among them.
template <typename T>
struct Eval {
    T A0, A1[3], A2[6], S[6];
    typename Jac<T>::type C[35];
    float omitted;
};

// Adds a source: the moments of r t + z with z ~ N(0, S) and given power sums
// t_p of t. The lattice integral is (t_0, r = 0, S = Sigma), a tail has r the
// regression on the axis and S the conditional covariance, a Poisson mode
// r = s, t_p = amp Re((-i)^p exp(-i phi)).
template <typename T>
CF_FN void add_low(Eval<T>& e, T t0, T t1, T t2, const T (&r)[3], const T (&S)[6]) {
    e.A0 = add(e.A0, t0);
    CF_UNROLL
    for (int a = 0; a < 3; ++a) {
        e.A1[a] = add(e.A1[a], mul(r[a], t1));
        const T rt = mul(r[a], t2);
        CF_UNROLL
        for (int b = a; b < 3; ++b)
            e.A2[sym(a, b)] = add(e.A2[sym(a, b)], add(mul(rt, r[b]), mul(S[sym(a, b)], t0)));
    }
}

// adds moments 1, d, d d in a plain type
template <typename T, typename V>
CF_FN void add_moments(Eval<T>& e, const V (&m)[10]) {
    e.A0 = add(e.A0, num<T>(m[0]));
    CF_UNROLL
    for (int q = 0; q < 3; ++q) e.A1[q] = add(e.A1[q], num<T>(m[1 + q]));
    CF_UNROLL
    for (int q = 0; q < 6; ++q) e.A2[q] = add(e.A2[q], num<T>(m[4 + q]));
}

template <typename J>
CF_FN void add_gram(J (&C)[35], J t0, J t1, J t2, J t3, J t4, const J (&r)[3], const J (&S)[6]) {
    J B[6];
    CF_UNROLL
    for (int a = 0; a < 3; ++a)
        CF_UNROLL
        for (int b = a; b < 3; ++b) B[sym(a, b)] = r[a] * r[b];
    C[0] += t0;
    CF_UNROLL
    for (int a = 0; a < 3; ++a) {
        C[1 + a] += r[a] * t1;
        CF_UNROLL
        for (int b = a; b < 3; ++b) {
            C[4 + sym(a, b)] += B[sym(a, b)] * t2 + S[sym(a, b)] * t0;
            CF_UNROLL
            for (int c = b; c < 3; ++c) {
                const int x3 = (a == 0) + (b == 0) + (c == 0), y3 = (a == 1) + (b == 1) + (c == 1);
                C[mono4(x3, y3, 3 - x3 - y3)] +=
                    r[a] * B[sym(b, c)] * t3 + (r[a] * S[sym(b, c)] + r[b] * S[sym(a, c)] + r[c] * S[sym(a, b)]) * t1;
                CF_UNROLL
                for (int d = c; d < 3; ++d) {
                    const int x4 = x3 + (d == 0), y4 = y3 + (d == 1);
                    const J Bab = B[sym(a, b)], Bcd = B[sym(c, d)], Bac = B[sym(a, c)], Bbd = B[sym(b, d)],
                            Bad = B[sym(a, d)], Bbc = B[sym(b, c)];
                    const J Sab = S[sym(a, b)], Scd = S[sym(c, d)], Sac = S[sym(a, c)], Sbd = S[sym(b, d)],
                            Sad = S[sym(a, d)], Sbc = S[sym(b, c)];
                    C[mono4(x4, y4, 4 - x4 - y4)] +=
                        Bab * Bcd * t4 +
                        (Bab * Scd + Sab * Bcd + Bac * Sbd + Sac * Bbd + Bad * Sbc + Sad * Bbc) * t2 +
                        (Sab * Scd + Sac * Sbd + Sad * Sbc) * t0;
                }
            }
        }
    }
}

// the lattice integral's part of the Gram sums (odd degrees vanish)
template <typename J>
CF_FN void gram_main(J (&C)[35], J n, const J (&S)[6]) {
    C[0] = n;
    CF_UNROLL
    for (int a = 0; a < 3; ++a)
        CF_UNROLL
        for (int b = a; b < 3; ++b) {
            C[4 + sym(a, b)] = n * S[sym(a, b)];
            CF_UNROLL
            for (int c = b; c < 3; ++c)
                CF_UNROLL
                for (int d = c; d < 3; ++d) {
                    const int x = (a == 0) + (b == 0) + (c == 0) + (d == 0), y = (a == 1) + (b == 1) + (c == 1) + (d == 1);
                    C[mono4(x, y, 4 - x - y)] =
                        n * (S[sym(a, b)] * S[sym(c, d)] + S[sym(a, c)] * S[sym(b, d)] + S[sym(a, d)] * S[sym(b, c)]);
                }
        }
}

// ------------------------------------------------------------------- tails

// Power sums of one side of a marginal: cells at distance t + j h (j >= 0)
// from the mean with weights M, M r, M r (r rr), ... until they are below
// cut. Weights fall along the way (t is beyond 1.5 standard deviations), and
// so do M j and M j^2 times h^2 / t^2 and less: sums by Fast2Sum. Products
// are left unnormalised where only the pair's sum is read. Sums over j are
// returned as s[0..2] (T) and s3, s4 (FP32); false if the tail has no end.
CF_FN df2 mul_raw(df2 a, df2 b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    return {p, fmaf(a.lo, b.hi, e)};
}
struct Run {
    float s, e;
};
CF_FN void run_add(Run& a, float h, float l) {
    const float s = __fadd_rn(a.s, h);
    const float big = fmaxf(a.s, h), small = fminf(a.s, h);  // non-negative terms
    a.e = __fadd_rn(a.e, __fadd_rn(__fsub_rn(small, __fsub_rn(s, big)), l));
    a.s = s;
}
constexpr int kMaxTail = 96;  // cells of a tail (a wide Maxwellian's tail that is longer is refused)

CF_FN bool tail_sums(df2 M, df2 r, df2 rr, float cut, df2 (&s)[3], float& s3, float& s4) {
    Run a0 = {0.f, 0.f}, a1 = a0, a2 = a0;
    float j = 0.f, c3 = 0.f, c4 = 0.f;
    int n = 0;
    CF_LOOP
    for (; n < kMaxTail && M.hi > cut; ++n) {
        run_add(a0, M.hi, M.lo);
        const float p1 = __fmul_rn(M.hi, j);
        const float e1 = fmaf(M.lo, j, fmaf(M.hi, j, -p1));
        run_add(a1, p1, e1);
        const float p2 = __fmul_rn(p1, j);
        const float e2 = fmaf(e1, j, fmaf(p1, j, -p2));
        run_add(a2, p2, e2);
        const float p3 = p2 * j;
        c3 += p3;
        c4 = fmaf(p3, j, c4);
        M = mul_raw(M, r);
        r = mul_raw(r, rr);
        j += 1.0f;
    }
    s[0] = df2_qtwo_sum(a0.s, a0.e);
    s[1] = df2_qtwo_sum(a1.s, a1.e);
    s[2] = df2_qtwo_sum(a2.s, a2.e);
    s3 = c3;
    s4 = c4;
    return n < kMaxTail;
}
CF_FN bool tail_sums(double M, double r, double rr, float cut, double (&s)[3], double& s3, double& s4) {
    s[0] = s[1] = s[2] = s3 = s4 = 0.0;
    double j = 0.0;
    int n = 0;
    CF_LOOP
    for (; n < kMaxTail && M > (double)cut; ++n) {
        const double p1 = M * j, p2 = p1 * j, p3 = p2 * j;
        s[0] += M;
        s[1] += p1;
        s[2] += p2;
        s3 += p3;
        s4 += p3 * j;
        M *= r;
        r *= rr;
        j += 1.0;
    }
    return n < kMaxTail;
}

template <typename V>
CF_FN V pick(int a, V x, V y, V z) { return a == 0 ? x : (a == 1 ? y : z); }

template <typename V>
CF_FN V larger(V x, V y) { return x > y ? x : y; }

// ------------------------------------------------------------ doubly outside

// Power sums over the cells outside along axes a and b at once (all four
// corners), weights relative to the lattice integral: t[0..5] = 1, ta, tb,
// ta^2, ta tb, tb^2. (ap, am), (bp, bm): distances from the mean to the first
// cells outside on either side; Q the inverse of the marginal covariance;
// w4 the weights of the four corner cells (++, -+, +-, --). Rows and columns
// are walked outward by two-dimensional recurrences until they fall below
// cut. False where the weight does not fall outward (strong correlation).
//
// Two corners at a time, the two sides of a: they share the distances along b,
// and the one's chain of products hides the other's (with the screening of the
// triply outside corners below: 65536 fits of 16^3 Harris ions 438 -> 429 us,
// 16384 in FP64 441 -> 415). A corner then goes on with cells below cut while
// the other's are above it.
template <typename J>
CF_FN bool corner_sums(J ap, J am, J bp, J bm, J ha, J hb, J Qaa, J Qab, J Qbb, const J (&w4)[4], J cut, J (&t)[6]) {
    CF_UNROLL
    for (int q = 0; q < 6; ++q) t[q] = J(0);
    if (!(larger(larger(w4[0], w4[1]), larger(w4[2], w4[3])) > cut)) {
        // nothing to sum; the weight has to fall outward all the same
        bool ok = true;
        CF_UNROLL
        for (int c = 0; c < 4; ++c) {
            const J ta = (c & 1) ? am : ap, tb = (c & 2) ? bm : bp, qab = (c == 1 || c == 2) ? -Qab : Qab;
            ok = ok && Qaa * ta + qab * tb > J(0) && Qbb * tb + qab * ta > J(0);
        }
        return ok;
    }
    const J raa = expj(-Qaa * ha * ha), rbb = expj(-Qbb * hb * hb);
    const J ea = expj(-Qab * ha * hb), eb = expj(Qab * ha * hb);
    bool ok = true;
    CF_LOOP
    for (int side = 0; side < 2; ++side) {
        const J tb0 = side ? bm : bp;
        J w[2] = {side ? w4[2] : w4[0], side ? w4[3] : w4[1]};
        J ta[2] = {ap, am}, ra[2], rb[2], rab[2] = {side ? eb : ea, side ? ea : eb};
        CF_UNROLL
        for (int c = 0; c < 2; ++c) {
            const J qab = (c != side) ? -Qab : Qab;  // both distances counted positive
            // logarithms of the step ratios at the corner
            const J la = -(Qaa * ta[c] + qab * tb0) * ha, lb = -(Qbb * tb0 + qab * ta[c]) * hb;
            ok = ok && la < J(0) && lb < J(0);
            ra[c] = expj(la - J(0.5) * Qaa * ha * ha);
            rb[c] = expj(lb - J(0.5) * Qbb * hb * hb);
        }
        if (!ok) return false;
        J c0[2] = {J(0), J(0)}, c1a[2] = {J(0), J(0)}, c1b[2] = {J(0), J(0)}, c2a[2] = {J(0), J(0)},
          c2m[2] = {J(0), J(0)}, c2b[2] = {J(0), J(0)};
        CF_LOOP
        for (int i = 0; i < kMaxTail && larger(w[0], w[1]) > cut; ++i) {
            J v[2] = {w[0], w[1]}, r[2] = {rb[0], rb[1]}, tb = tb0;
            J s0[2] = {J(0), J(0)}, s1[2] = {J(0), J(0)}, s2[2] = {J(0), J(0)};
            CF_LOOP
            for (int j = 0; j < kMaxTail && larger(v[0], v[1]) > cut; ++j) {
                CF_UNROLL
                for (int c = 0; c < 2; ++c) {
                    const J vt = v[c] * tb;
                    s0[c] += v[c];
                    s1[c] += vt;
                    s2[c] += vt * tb;
                    v[c] *= r[c];
                    r[c] *= rbb;
                }
                tb += hb;
            }
            CF_UNROLL
            for (int c = 0; c < 2; ++c) {
                const J ts = ta[c] * s0[c];
                c0[c] += s0[c];
                c1a[c] += ts;
                c1b[c] += s1[c];
                c2a[c] += ta[c] * ts;
                c2m[c] += ta[c] * s1[c];
                c2b[c] += s2[c];
                w[c] *= ra[c];
                ra[c] *= raa;
                rb[c] *= rab[c];
                ta[c] += ha;
            }
        }
        t[0] += c0[0] + c0[1];
        t[1] += c1a[0] - c1a[1];
        t[2] += side ? -(c1b[0] + c1b[1]) : c1b[0] + c1b[1];
        t[3] += c2a[0] + c2a[1];
        t[4] += side ? c2m[1] - c2m[0] : c2m[0] - c2m[1];
        t[5] += c2b[0] + c2b[1];
    }
    return ok;
}

// a row of two corners from its cell v outward, ratio r to the next one
struct Two {
    float x, y;
};
CF_FN void light_row(Two v, Two r, float rr, float tb, float h, float cut, float (&s0)[2], float (&s1)[2], float (&s2)[2]) {
    s0[0] = s0[1] = s1[0] = s1[1] = s2[0] = s2[1] = 0.f;
    CF_LOOP
    for (int j = 0; j < kMaxTail && larger(v.x, v.y) > cut; ++j) {
        const float a = v.x * tb, b = v.y * tb;
        s0[0] += v.x;
        s0[1] += v.y;
        s1[0] += a;
        s1[1] += b;
        s2[0] = fmaf(a, tb, s2[0]);
        s2[1] = fmaf(b, tb, s2[1]);
        v.x *= r.x;
        v.y *= r.y;
        r.x *= rr;
        r.y *= rr;
        tb += h;
    }
}

// The same for heavy corners in FP64 mode: cells above heavy in FP64, lighter ones
// (1e-11 of the lattice integral: FP32 rounds them at 1e-17) and what a row or a
// corner has beyond them in FP32, whose chains are several times as short. All in
// FP64 the corners of strongly correlated fits took three quarters of the time
// (2048 fits of 16^3 1621 -> 1190 us, 24^3 2510 -> 1552).
template <typename J>
CF_FN bool corner_sums_mixed(J ap, J am, J bp, J bm, J ha, J hb, J Qaa, J Qab,
                             J Qbb, const J (&w4)[4], float cut, J (&t)[6]) {
    constexpr J heavy = J(1e-11);
    CF_UNROLL
    for (int q = 0; q < 6; ++q) t[q] = J(0);
    const J raa = expj(-Qaa * ha * ha), rbb = expj(-Qbb * hb * hb), ea = expj(-Qab * ha * hb), eb = expj(Qab * ha * hb);
    const float raaf = (float)raa, rbbf = (float)rbb, haf = (float)ha, hbf = (float)hb;
    bool ok = true;
    CF_LOOP
    for (int side = 0; side < 2; ++side) {
        const J tb0 = side ? bm : bp;
        J w[2] = {side ? w4[2] : w4[0], side ? w4[3] : w4[1]};
        J ta[2] = {ap, am}, ra[2], rb[2], rab[2] = {side ? eb : ea, side ? ea : eb};
        CF_UNROLL
        for (int c = 0; c < 2; ++c) {
            const J qab = (c != side) ? -Qab : Qab;
            const J la = -(Qaa * ta[c] + qab * tb0) * ha, lb = -(Qbb * tb0 + qab * ta[c]) * hb;
            ok = ok && la < J(0) && lb < J(0);
            ra[c] = expj(la - J(0.5) * Qaa * ha * ha);
            rb[c] = expj(lb - J(0.5) * Qbb * hb * hb);
        }
        if (!ok) return false;
        J c0[2] = {J(0), J(0)}, c1a[2] = {J(0), J(0)}, c1b[2] = {J(0), J(0)}, c2a[2] = {J(0), J(0)}, c2m[2] = {J(0), J(0)},
               c2b[2] = {J(0), J(0)};
        int i = 0;
        CF_LOOP
        for (; i < kMaxTail && larger(w[0], w[1]) > heavy; ++i) {
            J v[2] = {w[0], w[1]}, r[2] = {rb[0], rb[1]}, tb = tb0;
            J s0[2] = {J(0), J(0)}, s1[2] = {J(0), J(0)}, s2[2] = {J(0), J(0)};
            int j = 0;
            CF_LOOP
            for (; j < kMaxTail && larger(v[0], v[1]) > heavy; ++j) {
                CF_UNROLL
                for (int c = 0; c < 2; ++c) {
                    const J vt = v[c] * tb;
                    s0[c] += v[c];
                    s1[c] += vt;
                    s2[c] += vt * tb;
                    v[c] *= r[c];
                    r[c] *= rbb;
                }
                tb += hb;
            }
            float f0[2], f1[2], f2[2];
            light_row({(float)v[0], (float)v[1]}, {(float)r[0], (float)r[1]}, rbbf, (float)tb, hbf, cut, f0, f1, f2);
            CF_UNROLL
            for (int c = 0; c < 2; ++c) {
                s0[c] += f0[c];
                s1[c] += f1[c];
                const J ts = ta[c] * s0[c];
                c0[c] += s0[c];
                c1a[c] += ts;
                c1b[c] += s1[c];
                c2a[c] += ta[c] * ts;
                c2m[c] += ta[c] * s1[c];
                c2b[c] += s2[c] + f2[c];
                w[c] *= ra[c];
                ra[c] *= raa;
                rb[c] *= rab[c];
                ta[c] += ha;
            }
        }
        float wf[2], raf[2], rbf[2], rabf[2], taf[2];
        CF_UNROLL
        for (int c = 0; c < 2; ++c) {
            wf[c] = (float)w[c];
            raf[c] = (float)ra[c];
            rbf[c] = (float)rb[c];
            rabf[c] = (float)rab[c];
            taf[c] = (float)ta[c];
        }
        float d0[2] = {0.f, 0.f}, d1a[2] = {0.f, 0.f}, d1b[2] = {0.f, 0.f}, d2a[2] = {0.f, 0.f}, d2m[2] = {0.f, 0.f},
              d2b[2] = {0.f, 0.f};
        CF_LOOP
        for (; i < kMaxTail && larger(wf[0], wf[1]) > cut; ++i) {
            float f0[2], f1[2], f2[2];
            light_row({wf[0], wf[1]}, {rbf[0], rbf[1]}, rbbf, (float)tb0, hbf, cut, f0, f1, f2);
            CF_UNROLL
            for (int c = 0; c < 2; ++c) {
                const float ts = taf[c] * f0[c];
                d0[c] += f0[c];
                d1a[c] += ts;
                d1b[c] += f1[c];
                d2a[c] += taf[c] * ts;
                d2m[c] += taf[c] * f1[c];
                d2b[c] += f2[c];
                wf[c] *= raf[c];
                raf[c] *= raaf;
                rbf[c] *= rabf[c];
                taf[c] += haf;
            }
        }
        CF_UNROLL
        for (int c = 0; c < 2; ++c) {
            const J sa = c ? J(-1) : J(1), sb = side ? J(-1) : J(1);
            t[0] += c0[c] + d0[c];
            t[1] += sa * (c1a[c] + d1a[c]);
            t[2] += sb * (c1b[c] + d1b[c]);
            t[3] += c2a[c] + d2a[c];
            t[4] += sa * sb * (c2m[c] + d2m[c]);
            t[5] += c2b[c] + d2b[c];
        }
    }
    return ok;
}

// modes beyond |k|^2 = 2, one of each pair +-k, with |k|^2 <= 5
constexpr int kFarModes = 19;
CF_FN void far_mode(int q, int& x, int& y, int& z) {
    // (1, +-1, +-1); (2, 0, 0) and permutations; (2, +-1, 0) and permutations
    if (q < 4) {
        x = 1;
        y = (q & 1) ? -1 : 1;
        z = (q & 2) ? -1 : 1;
    } else if (q < 7) {
        x = q == 4 ? 2 : 0;
        y = q == 5 ? 2 : 0;
        z = q == 6 ? 2 : 0;
    } else {
        const int p = (q - 7) >> 1, s = (q & 1) ? 1 : -1;  // p: (2,1,0) (1,2,0) (2,0,1) (1,0,2) (0,2,1) (0,1,2)
        const int a = (p & 1) ? 1 : 2, b = s * (3 - a);
        x = p < 4 ? a : 0;
        y = p < 2 ? b : (p < 4 ? 0 : a);
        z = p < 2 ? 0 : b;
    }
}

// The Poisson modes along the two other axes of the cells outside along axis a:
// at signed distance t the cross section is a Gaussian with mean r t and
// covariance Sc, so mode k adds 2 amp Re exp(-i (phi + omega t)) times the
// moments of r t + N(-i s, Sc), s = 2 pi Sc k / h. f is minus the lattice
// integral, x the mean's offset from its cell, out gets 1, d, d d.
//
// They are the product of two small parts, so FP32 gives them where that
// product is small enough (Limits::tail). A narrow Maxwellian next to a face
// makes both parts large (0.7 cells per standard deviation, a face at 2: 1e-4 of
// the density, of which FP32 loses 4e-11): FP64 mode sums those in FP64, and FP32
// mode leaves such fits to the direct sums (an FP64 form of this kept for them cost
// every other fit 1 to 4% by its registers).
template <typename V>
struct Tail {
    V f, ca, iv, tp, tm, h, ih[3], x[3], r[3], S[6];
};

template <typename V, typename T>
CF_FN Tail<V> tail_of(T f, T ca, T iv, T tp, T tm, T h, const T (&ih)[3], const T (&x)[3], const T (&r)[3], const T (&S)[6]) {
    Tail<V> q = {plain<V>(f), plain<V>(ca), plain<V>(iv), plain<V>(tp), plain<V>(tm), plain<V>(h)};
    CF_UNROLL
    for (int c = 0; c < 3; ++c) {
        q.ih[c] = plain<V>(ih[c]);
        q.x[c] = plain<V>(x[c]);
        q.r[c] = plain<V>(r[c]);
    }
    CF_UNROLL
    for (int c = 0; c < 6; ++c) q.S[c] = plain<V>(S[c]);
    return q;
}

CF_FN void turn(float y, float& c, float& s) {
    y -= rintf(y);
    c = cosf(6.2831853f * y);
    s = sinf(6.2831853f * y);
}
CF_FN void turn(double y, double& c, double& s) { cossin(y, c, s); }

template <typename V>
CF_FN void tail_modes(int a, const Tail<V>& q, V cut, V (&out)[10]) {
    constexpr V two_pi = V(6.283185307179586476925);
    CF_UNROLL
    for (int d = 0; d < 10; ++d) out[d] = V(0);
    // first cells, and the ratios to the next ones
    const V t0[2] = {q.tp, q.tm}, rr = expj(-q.h * q.h * q.iv);
    V w0[2], r0[2];
    CF_UNROLL
    for (int side = 0; side < 2; ++side) {
        w0[side] = q.ca * expj(V(-0.5) * t0[side] * t0[side] * q.iv);
        r0[side] = expj(-(t0[side] + V(0.5) * q.h) * q.h * q.iv);
    }
    CF_LOOP
    for (int m = 0; m < 4; ++m) {
        const V kb = m == 1 ? V(0) : V(1), kc = m == 0 ? V(0) : (m == 3 ? V(-1) : V(1));
        const V k[3] = {a == 0 ? V(0) : kb, a == 1 ? V(0) : (a == 0 ? kb : kc), a == 2 ? V(0) : kc};
        V u[3], y[3], ex = V(0), om = V(0), ph = V(0);
        CF_UNROLL
        for (int d = 0; d < 3; ++d) u[d] = k[d] * q.ih[d];
        CF_UNROLL
        for (int d = 0; d < 3; ++d) {
            y[d] = q.S[sym(d, 0)] * u[0] + q.S[sym(d, 1)] * u[1] + q.S[sym(d, 2)] * u[2];
            ex += u[d] * y[d];
            om += u[d] * q.r[d];
            ph += k[d] * q.x[d];
        }
        ex *= V(19.739208802178717238);  // 2 pi^2
        if (ex > V(40)) continue;
        const V am = V(2) * q.f * expj(-ex);
        V cr, sr, c0 = V(0), s0 = V(0), c1 = V(0), s1 = V(0), c2 = V(0);
        turn(om * q.h, cr, sr);
        CF_LOOP
        for (int side = 0; side < 2; ++side) {
            V t = side ? t0[1] : t0[0], w = side ? w0[1] : w0[0], rt = side ? r0[1] : r0[0];
            if (!(w > cut)) continue;
            const V sg = side ? V(-1) : V(1);
            V c, s;
            turn(ph + om * sg * t, c, s);
            CF_LOOP
            for (int j = 0; j < 64 && w > cut; ++j) {
                const V wt = w * sg * t;
                c0 += w * c;
                s0 += w * s;
                c1 += wt * c;
                s1 += wt * s;
                c2 += wt * sg * t * c;
                const V cn = c * cr - sg * s * sr;
                s = s * cr + sg * c * sr;
                c = cn;
                w *= rt;
                rt *= rr;
                t += q.h;
            }
        }
        out[0] += am * c0;
        CF_UNROLL
        for (int d = 0; d < 3; ++d) {
            const V sd = two_pi * y[d];
            out[1 + d] += am * (q.r[d] * c1 - sd * s0);
            CF_UNROLL
            for (int e = d; e < 3; ++e) {
                const V se = two_pi * y[e];
                out[4 + sym(d, e)] +=
                    am * (q.r[d] * q.r[e] * c2 - (q.r[d] * se + sd * q.r[e]) * s1 + (q.S[sym(d, e)] - sd * se) * c0);
            }
        }
    }
}

// One far mode's moments 1, d, d d. A mode weighs 2 exp(-ex) (1 + 2 ex) of the
// density at most, of which FP32 loses some 4e-7.
template <typename V>
struct Far {
    V n, ih[3], x[3], S[6];
};
template <typename V>
CF_FN bool far_part(int q, const Far<V>& f, V (&out)[10]) {
    int k[3];
    far_mode(q, k[0], k[1], k[2]);
    V u[3], y[3], ex = V(0), ph = V(0);
    CF_UNROLL
    for (int a = 0; a < 3; ++a) {
        u[a] = V(k[a]) * f.ih[a];
        ph += V(k[a]) * f.x[a];
    }
    CF_UNROLL
    for (int a = 0; a < 3; ++a) {
        y[a] = f.S[sym(a, 0)] * u[0] + f.S[sym(a, 1)] * u[1] + f.S[sym(a, 2)] * u[2];
        ex += u[a] * y[a];
    }
    ex *= V(19.739208802178717238);  // 2 pi^2
    if (ex > V(48)) return false;
    V c, s;
    turn(ph, c, s);
    const V am = V(2) * f.n * expj(-ex);
    out[0] = am * c;
    CF_UNROLL
    for (int a = 0; a < 3; ++a) {
        y[a] *= V(6.283185307179586476925);
        out[1 + a] = -am * s * y[a];
        CF_UNROLL
        for (int b = 0; b <= a; ++b) out[4 + sym(a, b)] = am * c * (f.S[sym(a, b)] - y[a] * y[b]);
    }
    return true;
}
CF_FN float far_exponent(int q, const float (&ih)[3], const float (&S)[6]) {
    int k[3];
    far_mode(q, k[0], k[1], k[2]);
    float ex = 0.f;
    CF_UNROLL
    for (int a = 0; a < 3; ++a)
        CF_UNROLL
        for (int c = 0; c < 3; ++c) ex += (k[a] * ih[a]) * S[sym(a, c)] * (k[c] * ih[c]);
    return 19.7392088f * ex;
}
template <typename V, typename T>
CF_FN Far<V> far_of(const T& n, const T (&ih)[3], const T (&x)[3], const T (&S)[6]) {
    Far<V> f;
    f.n = plain<V>(n);
    CF_UNROLL
    for (int a = 0; a < 3; ++a) {
        f.ih[a] = plain<V>(ih[a]);
        f.x[a] = plain<V>(x[a]);
    }
    CF_UNROLL
    for (int q = 0; q < 6; ++q) f.S[q] = plain<V>(S[q]);
    return f;
}

// limits of a closed-form evaluation, relative to the density: what may be
// left out, and what may be summed in FP32
template <typename T>
struct Limits;
template <>
struct Limits<df2> {
    static constexpr float drop = 2e-15f;   // a neglected part
    static constexpr float cut = 1e-19f;    // smallest cell weight of a sum
    static constexpr float fp32 = 3e-7f;    // doubly outside cells (times t^2) summed in FP32
    static constexpr float tail = 3e-7f;    // tails' Poisson modes (times t^2; FP32 loses 4e-7 of it) in FP32
    static constexpr float far = 0.f;       // exponent of the far modes from which on FP32 does
};
template <>
struct Limits<double> {
    static constexpr float drop = 1e-16f;
    static constexpr float cut = 1e-21f;
    static constexpr float fp32 = 1e-10f;
    static constexpr float tail = 1e-9f;
    static constexpr float far = 26.f;
};

// Discrete moments (and with gram the Gram sums) of g over the N^3 cells of
// the box, about its own mean. False where the closed form does not apply.
template <typename T>
CF_FN bool closed_eval(const Maxw<T>& g, const FitBox<T>& b, int N, bool gram, Eval<T>& e) {
    typedef typename Jac<T>::type J;
    typedef Limits<T> Lim;
    const T* P = g.P;
    T (&S)[6] = e.S;
    // covariance by cofactors
    T det;
    {
        const T c0 = sub(mul(P[3], P[5]), mul(P[4], P[4])), c1 = sub(mul(P[2], P[4]), mul(P[1], P[5])),
                c2 = sub(mul(P[1], P[4]), mul(P[2], P[3])), c3 = sub(mul(P[0], P[5]), mul(P[2], P[2])),
                c4 = sub(mul(P[1], P[2]), mul(P[0], P[4])), c5 = sub(mul(P[0], P[3]), mul(P[1], P[1]));
        det = add(add(mul(P[0], c0), mul(P[1], c1)), mul(P[2], c2));
        if (!(hi(P[0]) > 0.f && hi(c5) > 0.f && hi(det) > 0.f && hi(det) < 1e30f)) return false;
        const T id = inv(det);
        S[0] = mul(c0, id);
        S[1] = mul(c1, id);
        S[2] = mul(c2, id);
        S[3] = mul(c3, id);
        S[4] = mul(c4, id);
        S[5] = mul(c5, id);
    }
    if (!(hi(g.L) > -80.f && hi(g.L) < 80.f)) return false;
    const T np = mul(mul(expt(g.L), b.K), rsqrt2(det));

    // FP32 view for the conditions
    float sf[6], pf[6], hf[3], tp[3], tm[3], sd[3];
    CF_UNROLL
    for (int q = 0; q < 6; ++q) {
        sf[q] = hi(S[q]);
        pf[q] = hi(P[q]);
    }
    CF_UNROLL
    for (int a = 0; a < 3; ++a) {
        hf[a] = hi(b.h[a]);
        const float off = hi(g.m[a]) - hi(b.wc[a]), edge = 0.5f * (float)(N + 1) * hf[a];
        tp[a] = edge - off;
        tm[a] = edge + off;
        sd[a] = sqrtf(sf[sym(a, a)]);
    }
    bool ok = true;
    CF_UNROLL
    for (int a = 0; a < 3; ++a) ok = ok && tp[a] > 1.5f * sd[a] && tm[a] > 1.5f * sd[a];
    if (!ok) return false;
    // smallest and largest index-space variances: k.Sigma k >= k_a^2 / P_aa
    // for every k, >= lam |k|^2 with lam Gershgorin's bound
    const float ih[3] = {1.f / hf[0], 1.f / hf[1], 1.f / hf[2]};
    const float kap = fminf(fminf(ih[0] * ih[0] / pf[0], ih[1] * ih[1] / pf[3]), ih[2] * ih[2] / pf[5]);
    float lam = 1e30f, top = 0.f;
    CF_UNROLL
    for (int a = 0; a < 3; ++a) {
        const int p = (a + 1) % 3, q = (a + 2) % 3;
        const float v = sf[sym(a, a)] * ih[a] * ih[a];
        lam = fminf(lam, v - fabsf(sf[sym(a, p)]) * ih[a] * ih[p] - fabsf(sf[sym(a, q)]) * ih[a] * ih[q]);
        top = fmaxf(top, v);
    }
    constexpr float kTwoPi2 = 19.7392088f;  // 2 pi^2
    const float modes1 = 6.f * (1.f + 39.5f * top) * expf(-kTwoPi2 * kap);
    const bool modes = modes1 > Lim::drop;
    if (modes && !(24.f * (1.f + 240.f * top) * expf(-6.f * kTwoPi2 * lam) <= 4.f * Lim::drop)) return false;
    e.omitted = modes ? 8.f * (1.f + 120.f * top) * expf(-3.f * kTwoPi2 * lam) : 0.f;

    // lattice integral
    const T zero = num<T>(0.0);
    e.A0 = np;
    CF_UNROLL
    for (int a = 0; a < 3; ++a) e.A1[a] = zero;
    CF_UNROLL
    for (int q = 0; q < 6; ++q) e.A2[q] = mul(S[q], np);
    if (gram) {
        CF_UNROLL
        for (int q = 0; q < 35; ++q) e.C[q] = J(0);
        J Sj[6];
        CF_UNROLL
        for (int q = 0; q < 6; ++q) Sj[q] = jac(S[q]);
        const J nj = jac(np);
        gram_main(e.C, nj, Sj);
    }

    // index of the mean, (m - wc)/h + (N - 1)/2, to the nearest cell
    T ihT[3], x[3];
    if (modes) {
        CF_UNROLL
        for (int a = 0; a < 3; ++a) {
            ihT[a] = inv(b.h[a]);
            x[a] = add(mul(sub(g.m[a], b.wc[a]), ihT[a]), from(0.5f * (float)(N - 1), zero));
            x[a] = add(x[a], from(-rintf(hi(x[a])), zero));
        }
    }

    // singly outside cells, axis by axis
    float out2 = 0.f;
    CF_LOOP
    for (int a = 0; a < 3; ++a) {
        const T va = pick(a, S[0], S[3], S[5]);
        const T h = pick(a, b.h[0], b.h[1], b.h[2]);
        const T off = sub(pick(a, g.m[0], g.m[1], g.m[2]), pick(a, b.wc[0], b.wc[1], b.wc[2]));
        const T edge = scale(h, 0.5f * (float)(N + 1));
        const T iv = inv(va);
        const T hiv = mul(h, iv);
        const T hh = mul(h, hiv);
        const T rr = expt(neg(hh));
        const T ca = mul(mul(h, rsqrt2(va)), num<T>(0.39894228040143267794));
        T t0 = zero, t1 = zero, t2 = zero;
        J t3 = J(0), t4 = J(0);
        CF_LOOP
        for (int side = 0; side < 2; ++side) {
            const T t = side ? add(edge, off) : sub(edge, off);
            const T x = mul(t, iv);
            const float q = 0.5f * hi(t) * hi(x);
            if (q > 60.f) continue;  // below every rounding
            const T M = mul(expt(scale(mul(t, x), -0.5f)), ca);
            const T r = expt(neg(add(mul(hiv, t), scale(hh, 0.5f))));
            T s[3];
            J s3, s4;
            if (!tail_sums(M, r, rr, Lim::cut, s, s3, s4)) return false;
            // distances t + j h
            const T u1 = add(mul(t, s[0]), mul(h, s[1]));
            const T u2 = add(mul(t, add(u1, mul(h, s[1]))), mul(mul(h, h), s[2]));
            t0 = add(t0, s[0]);
            t1 = side ? sub(t1, u1) : add(t1, u1);
            t2 = add(t2, u2);
            if (gram) {
                const J tj = jac(t), hj = jac(h), j0 = jac(s[0]), j1 = jac(s[1]) * hj, j2 = jac(s[2]) * hj * hj,
                        j3 = s3 * hj * hj * hj, j4 = s4 * hj * hj * hj * hj;
                const J u3 = tj * (tj * (tj * j0 + J(3) * j1) + J(3) * j2) + j3;
                t3 += side ? -u3 : u3;
                t4 += tj * (tj * (tj * (tj * j0 + J(4) * j1) + J(6) * j2) + J(4) * j3) + j4;
            }
        }
        const float f0 = hi(t0), f2 = hi(t2) * hi(iv);
        out2 = fmaxf(out2, fmaxf(f0, f2));
        if (!(f0 > 0.f)) continue;
        if (!(f0 < 0.25f)) return false;
        // regression of the other axes on this one and what remains
        T r[3], Sc[6];
        const T row[3] = {pick(a, S[0], S[1], S[2]), pick(a, S[1], S[3], S[4]), pick(a, S[2], S[4], S[5])};
        CF_UNROLL
        for (int c = 0; c < 3; ++c) r[c] = mul(row[c], iv);
        CF_UNROLL
        for (int c = 0; c < 3; ++c)
            CF_UNROLL
            for (int d = c; d < 3; ++d) Sc[sym(c, d)] = sub(S[sym(c, d)], mul(r[c], row[d]));
        const T nn = neg(np);
        const float weight = modes1 * fmaxf(f0, f2);
        e.omitted = fmaxf(e.omitted, weight);
        if (weight > Lim::tail) {
            if (sizeof(J) == 4) return false;
            double part[10];
            tail_modes<double>(a, tail_of<double>(nn, ca, iv, sub(edge, off), add(edge, off), h, ihT, x, r, Sc), (double)Lim::cut, part);
            add_moments(e, part);
        } else if (weight > Lim::drop) {
            float part[10];
            tail_modes<float>(a, tail_of<float>(nn, ca, iv, sub(edge, off), add(edge, off), h, ihT, x, r, Sc), Lim::cut, part);
            add_moments(e, part);
        }
        add_low(e, mul(nn, t0), mul(nn, t1), mul(nn, t2), r, Sc);
        if (gram) {
            const J nj = jac(nn);
            J rj[3], Sj[6];
            CF_UNROLL
            for (int c = 0; c < 3; ++c) rj[c] = jac(r[c]);
            CF_UNROLL
            for (int q = 0; q < 6; ++q) Sj[q] = jac(Sc[q]);
            add_gram<J>(e.C, nj * jac(t0), nj * jac(t1), nj * jac(t2), nj * t3, nj * t4, rj, Sj);
        }
    }
    // modes beyond tail_modes' four, and those of the doubly outside cells'
    // remaining axis, are left out
    if (modes) {
        if (24.f * (1.f + 160.f * top) * expf(-4.f * kTwoPi2 * lam) * out2 > 5.f * Lim::drop) return false;
    }

    // doubly outside cells
    CF_LOOP
    for (int p = 0; p < 3; ++p) {
        // axes a < b outside
        const int a = p == 2 ? 1 : 0;
        const float saa = p == 2 ? sf[3] : sf[0], sbb = p == 0 ? sf[3] : sf[5], sab = pick(p, sf[1], sf[2], sf[4]);
        const float d2 = saa * sbb - sab * sab;
        if (!(d2 > 0.f)) return false;
        const float Qaa = sbb / d2, Qab = -sab / d2, Qbb = saa / d2;
        const float ha = a ? hf[1] : hf[0], hb = p == 0 ? hf[1] : hf[2];
        const float ap = a ? tp[1] : tp[0], am = a ? tm[1] : tm[0], bp = p == 0 ? tp[1] : tp[2],
                    bm = p == 0 ? tm[1] : tm[2];
        const float norm = ha * hb * 0.15915494f / sqrtf(d2);
        float tf[6], w4[4], wtop = 0.f;
        CF_UNROLL
        for (int c = 0; c < 4; ++c) {
            const float ta = (c & 1) ? am : ap, tb = (c & 2) ? bm : bp, q2 = (c == 1 || c == 2) ? -2.f * Qab : 2.f * Qab;
            w4[c] = norm * expf(-0.5f * (Qaa * ta * ta + q2 * ta * tb + Qbb * tb * tb));
            wtop = fmaxf(wtop, w4[c]);
        }
        const T Taa = a ? S[3] : S[0], Tbb = p == 0 ? S[3] : S[5], Tab = pick(p, S[1], S[2], S[4]);
        if (sizeof(J) == 4 && wtop > 3e-10f) {
            // heavy corners: the FP32 exponent (about 16, to 1e-6) is not enough
            const T di = inv(sub(mul(Taa, Tbb), mul(Tab, Tab)));
            const T qaa = mul(Tbb, di), qbb = mul(Taa, di), qab = neg(mul(Tab, di));
            const T oa = sub(a ? g.m[1] : g.m[0], a ? b.wc[1] : b.wc[0]);
            const T ob = sub(p == 0 ? g.m[1] : g.m[2], p == 0 ? b.wc[1] : b.wc[2]);
            const T ea = scale(a ? b.h[1] : b.h[0], 0.5f * (float)(N + 1));
            const T eb = scale(p == 0 ? b.h[1] : b.h[2], 0.5f * (float)(N + 1));
            CF_UNROLL
            for (int c = 0; c < 4; ++c) {
                const T ta = (c & 1) ? add(ea, oa) : sub(ea, oa), tb = (c & 2) ? add(eb, ob) : sub(eb, ob);
                const T x = scale(mul(qab, tb), (c == 1 || c == 2) ? -2.f : 2.f);
                const T q = scale(add(mul(ta, add(mul(qaa, ta), x)), mul(qbb, mul(tb, tb))), 0.5f);
                const float qh = hi(q);
                w4[c] = norm * expf(-qh) * (1.f - hi(sub(q, from(qh, zero))));
            }
        }
        if (!corner_sums<float>(ap, am, bp, bm, ha, hb, Qaa, Qab, Qbb, w4, Lim::cut, tf)) return false;
        const float weight = fmaxf(tf[0], fmaxf(tf[3] / saa, tf[5] / sbb));
        e.omitted = fmaxf(e.omitted, weight);
        if (modes1 * weight > 5.f * Lim::drop) return false;
        if (!(tf[0] > 0.f)) continue;
        J t[6];
        if (sizeof(J) == 8 && weight > Lim::fp32) {
            const J Jaa = jac(Taa), Jbb = jac(Tbb), Jab = jac(Tab), dd = Jaa * Jbb - Jab * Jab;
            const T oa = sub(a ? g.m[1] : g.m[0], a ? b.wc[1] : b.wc[0]);
            const T ob = sub(p == 0 ? g.m[1] : g.m[2], p == 0 ? b.wc[1] : b.wc[2]);
            const J Ha = jac(a ? b.h[1] : b.h[0]), Hb = jac(p == 0 ? b.h[1] : b.h[2]);
            const J ea = J(0.5) * J(N + 1) * Ha, eb = J(0.5) * J(N + 1) * Hb;
            const J jap = ea - jac(oa), jam = ea + jac(oa), jbp = eb - jac(ob), jbm = eb + jac(ob);
            const J qaa = Jbb / dd, qab = -Jab / dd, qbb = Jaa / dd, nrm = Ha * Hb * J(0.15915494309189533577) / sqrt(dd);
            J j4[4];
            CF_UNROLL
            for (int c = 0; c < 4; ++c) {
                const J ta = (c & 1) ? jam : jap, tb = (c & 2) ? jbm : jbp, q2 = (c == 1 || c == 2) ? J(-2) * qab : J(2) * qab;
                j4[c] = nrm * expj(J(-0.5) * (qaa * ta * ta + q2 * ta * tb + qbb * tb * tb));
            }
            if (!corner_sums_mixed<J>(jap, jam, jbp, jbm, Ha, Hb, qaa, qab, qbb, j4, Lim::cut, t)) return false;
        } else {
            if (!(weight <= (sizeof(J) == 8 ? 1.f : Lim::fp32))) return false;
            CF_UNROLL
            for (int q = 0; q < 6; ++q) t[q] = J(tf[q]);
        }
        // the remaining axis: E[d_c | ta, tb] = ga ta + gb tb
        const J nj = jac(np);
        const J Sa = jac(pick(p, S[2], S[1], S[1])), Sb = jac(pick(p, S[4], S[4], S[2]));
        const J Jaa = jac(Taa), Jbb = jac(Tbb), Jab = jac(Tab);
        const J id = J(1) / (Jaa * Jbb - Jab * Jab);
        const J ga = (Sa * Jbb - Sb * Jab) * id, gb = (Sb * Jaa - Sa * Jab) * id;
        const J scc = jac(pick(p, S[5], S[3], S[0])) - ga * Sa - gb * Sb;
        const J ac = ga * t[3] + gb * t[4], bc = ga * t[4] + gb * t[5];
        const J cc = ga * ac + gb * bc + scc * t[0];
        const J d1c = ga * t[1] + gb * t[2];
        // first moments by axis, second moments by pair of axes
        const J f1[3] = {p == 2 ? d1c : t[1], p == 0 ? t[2] : (p == 1 ? d1c : t[1]), p == 0 ? d1c : t[2]};
        const J f2[6] = {p == 2 ? cc : t[3],          p == 0 ? t[4] : ac,           p == 0 ? ac : (p == 1 ? t[4] : bc),
                         p == 0 ? t[5] : (p == 1 ? cc : t[3]), p == 0 ? bc : (p == 1 ? bc : t[4]), p == 0 ? cc : t[5]};
        e.A0 = add(e.A0, from(nj * t[0], zero));
        CF_UNROLL
        for (int q = 0; q < 3; ++q) e.A1[q] = add(e.A1[q], from(nj * f1[q], zero));
        CF_UNROLL
        for (int q = 0; q < 6; ++q) e.A2[q] = add(e.A2[q], from(nj * f2[q], zero));
    }

    // triply outside cells: FP32 sums over the corners where they matter
    {
        const float norm = hf[0] * hf[1] * hf[2] * 0.063493636f * sqrtf(hi(det));
        float z0 = 0.f, z1[3] = {0.f, 0.f, 0.f}, z2[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        // all eight at once: outward the weight must fall, and which of them are
        // worth summing
        const float far2 = 2.f * logf(norm / Lim::cut);
        unsigned worth = 0u;
        bool fall = true;
        CF_UNROLL
        for (int c = 0; c < 8; ++c) {
            const float sx = (c & 1) ? -1.f : 1.f, sy = (c & 2) ? -1.f : 1.f, sz = (c & 4) ? -1.f : 1.f;
            const float x0 = (c & 1) ? tm[0] : tp[0], y0 = (c & 2) ? tm[1] : tp[1], zz = (c & 4) ? tm[2] : tp[2];
            const float pxy = sx * sy * pf[1], pxz = sx * sz * pf[2], pyz = sy * sz * pf[4];
            const float gx = pf[0] * x0 + pxy * y0 + pxz * zz, gy = pxy * x0 + pf[3] * y0 + pyz * zz,
                        gz = pxz * x0 + pyz * y0 + pf[5] * zz;
            fall = fall && gx > 0.f && gy > 0.f && gz > 0.f;
            if (gx * x0 + gy * y0 + gz * zz < far2) worth |= 1u << c;
        }
        if (!fall) return false;
        const float rzz = expf(-pf[5] * hf[2] * hf[2]);
        CF_LOOP
        for (int c = 0; c < 8; ++c) {
            if (!((worth >> c) & 1u)) continue;
            const float sx = (c & 1) ? -1.f : 1.f, sy = (c & 2) ? -1.f : 1.f, sz = (c & 4) ? -1.f : 1.f;
            const float x0 = (c & 1) ? tm[0] : tp[0], y0 = (c & 2) ? tm[1] : tp[1], zz = (c & 4) ? tm[2] : tp[2];
            const float pxy = sx * sy * pf[1], pxz = sx * sz * pf[2], pyz = sy * sz * pf[4];
            float x = x0;
            CF_LOOP
            for (int i = 0; i < kMaxTail; ++i, x += hf[0]) {
                float y = y0;
                bool any = false;
                CF_LOOP
                for (int j = 0; j < kMaxTail; ++j, y += hf[1]) {
                    const float gz0 = pxz * x + pyz * y + pf[5] * zz;
                    const float qq = 0.5f * ((pf[0] * x + pxy * y + pxz * zz) * x + (pxy * x + pf[3] * y + pyz * zz) * y +
                                             gz0 * zz);
                    float w = norm * expf(-qq), r = expf(-hf[2] * (gz0 + 0.5f * pf[5] * hf[2]));
                    if (!(w > Lim::cut)) break;
                    any = true;
                    float s0 = 0.f, s1 = 0.f, s2 = 0.f, z = zz;
                    CF_LOOP
                    for (int k = 0; k < kMaxTail && w > Lim::cut; ++k) {
                        s0 += w;
                        s1 = fmaf(w, z, s1);
                        s2 = fmaf(w * z, z, s2);
                        w *= r;
                        r *= rzz;
                        z += hf[2];
                    }
                    z0 += s0;
                    z1[0] = fmaf(sx * x, s0, z1[0]);
                    z1[1] = fmaf(sy * y, s0, z1[1]);
                    z1[2] = fmaf(sz, s1, z1[2]);
                    z2[0] = fmaf(x * x, s0, z2[0]);
                    z2[1] = fmaf(sx * sy * x * y, s0, z2[1]);
                    z2[2] = fmaf(sx * sz * x, s1, z2[2]);
                    z2[3] = fmaf(y * y, s0, z2[3]);
                    z2[4] = fmaf(sy * sz * y, s1, z2[4]);
                    z2[5] += s2;
                }
                if (!any) break;
            }
        }
        if (z0 > 0.f) {
            if (!(z0 < 0.1f * Lim::fp32)) return false;
            const float nf = -hi(np);
            e.A0 = add(e.A0, from(nf * z0, zero));
            CF_UNROLL
            for (int q = 0; q < 3; ++q) e.A1[q] = add(e.A1[q], from(nf * z1[q], zero));
            CF_UNROLL
            for (int q = 0; q < 6; ++q) e.A2[q] = add(e.A2[q], from(nf * z2[q], zero));
        }
    }

    // Poisson modes of a narrow Maxwellian
    if (modes) {
        CF_LOOP
        for (int q = 0; q < 9; ++q) {
            // axes, then the six face diagonals
            const float kx = (q == 0 || (q >= 3 && q < 7)) ? 1.f : 0.f;
            const float ky = (q == 1 || q == 3 || q >= 7) ? 1.f : (q == 4 ? -1.f : 0.f);
            const float kz = (q == 2 || q == 5 || q == 7) ? 1.f : ((q == 6 || q == 8) ? -1.f : 0.f);
            const T u[3] = {scale(ihT[0], kx), scale(ihT[1], ky), scale(ihT[2], kz)};
            T y[3];
            CF_UNROLL
            for (int a = 0; a < 3; ++a)
                y[a] = add(add(mul(S[sym(a, 0)], u[0]), mul(S[sym(a, 1)], u[1])), mul(S[sym(a, 2)], u[2]));
            const T kk = add(add(mul(u[0], y[0]), mul(u[1], y[1])), mul(u[2], y[2]));
            if (kTwoPi2 * hi(kk) > 48.f) continue;
            T cph, sph;
            cossin(add(add(scale(x[0], kx), scale(x[1], ky)), scale(x[2], kz)), cph, sph);
            const T amp = scale(mul(np, expt(mul(kk, num<T>(-19.739208802178717238)))), 2.f);
            const T two_pi = num<T>(6.283185307179586476925);
            T s[3];
            CF_UNROLL
            for (int a = 0; a < 3; ++a) s[a] = mul(y[a], two_pi);
            const T ac = mul(amp, cph), as = mul(amp, sph);
            add_low(e, ac, neg(as), neg(ac), s, S);
            if (gram) {
                const J cj = jac(ac), sj = jac(as);
                const J rj[3] = {jac(s[0]), jac(s[1]), jac(s[2])};
                J Sj[6];
                CF_UNROLL
                for (int r = 0; r < 6; ++r) Sj[r] = jac(S[r]);
                add_gram<J>(e.C, cj, -sj, -cj, sj, cj, rj, Sj);
            }
        }
    }
    if (modes && 3.f * kTwoPi2 * lam < 48.f) {
        const Far<float> ff = far_of<float>(np, ihT, x, S);
        CF_LOOP
        for (int q = 0; q < kFarModes; ++q) {
            if (sizeof(J) == 8 && far_exponent(q, ih, sf) < Lim::far) {
                double part[10];
                if (far_part<double>(q, far_of<double>(np, ihT, x, S), part)) add_moments(e, part);
            } else {
                float part[10];
                if (far_part<float>(q, ff, part)) add_moments(e, part);
            }
        }
    }
    return true;
}

}  // namespace cf
}  // namespace vl

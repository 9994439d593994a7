// Discrete ten-moment Maxwellian fit by Newton iteration (moment fitting,
// paper Sec. 2.2 and Algorithm 1; the discrete fit makes the midpoint
// moments of degree <= 2 of the sampled Maxwellian equal the targets).
//
// Unknowns: the natural parameters eta of M(v) = exp(eta . phi(w)),
// w_a = (v_a - u0_a)/sigma_a, phi = (1, w_a, w_a w_b (a <= b)); the equations
// D(eta) = sum_c M(v_c) phi(w_c) dv^3 = T are the gradient of a convex
// function whose Hessian is the Gram matrix sum M phi phi^T dv^3.
//
// GB300 layout: 8 lanes per cell, 4 cells per warp, and the four cells of a
// warp iterate in lockstep: every branch that decides how much work follows
// (converged, Jacobian needed, line-search step) is taken by a warp vote, and
// cells that are done sit out with their lanes idle, so the heavy block
// evaluations always run with every busy cell of the warp converged. The FP64
// pipe of GB300 runs at ~1/58 of the FP32 pipe, so everything that is
// evaluated per iteration is kept in double-float arithmetic (df64.cuh) on
// the FP32 pipe: the parameters, the index-space exponent, the line-start
// exponentials and the moment sums. FP64 is used once per fit for the
// targets and the output.
//   * Along a v_x line the exponent is quadratic in the cell index, so M is
//     generated by a two-term multiplicative recurrence; line starts follow
//     the same recurrence along v_y and are restarted (df64 exp) per plane.
//     One pass gives the double-float moments of degree <= 2 and, when the
//     Jacobian is wanted, FP32 sums of degree <= 4 from the same values.
//     The kernel's time follows its instruction count, so the edge pass
//     adds its running sums by Fast2Sum with operands ordered on the ALU
//     pipe and leaves products unnormalised where only the pair's sum is
//     read.
//   * Moment weights are centred on the cell nearest to the mean, which
//     keeps the conversion to w-space free of cancellation.
//   * The Jacobian (Gram matrix) is formed from the index sums by three
//     separable binomial transforms and solved by Cholesky in FP32: each
//     Newton step carries ~1e-6 relative error, so each iteration still gains
//     about six digits; the residual itself is double-float accurate.
//   * Cells that have not converged after six iterations (e.g. Maxwellians
//     cut by the velocity box) switch to an FP64 Jacobian ("precise mode").
//   * Blocks whose values span more than the float range (+-80 over the
//     block) start every recurrence at the cell nearest the mean instead
//     and run it outward, so the values that underflow are negligible ones;
//     blocks where that cannot be shown (a one-cell ratio outside e^+-80, a
//     line maximum that could overflow, a significant line whose start
//     underflowed) take a slow path with one FP64 exponential per cell.
#pragma once

#include "common.cuh"
#include "df64.cuh"
#include "fit_index.cuh"
#include "kernels.cuh"
#include "mlp_common.cuh"

namespace vl {

namespace {

constexpr int kG = 8;  // lanes per cell
constexpr int kCoefN = 16;

struct CellScratch {
    df2 eta[10], et[10], eta0[10], T[10];
    df2 m[10];          // index moments of degree <= 2
    df2 wc[3], h[3], wm[3];
    df2 step[10];       // Newton direction
    float g[35];        // FP32 index moments of degree <= 4
    float U[35], W[35]; // binomial transforms of g (Jacobian entries in w-space)
    float J[55];        // packed lower triangle of the Jacobian / its Cholesky factor
    float rhs[10];
    float shift[3];
    double tgt[10];
    double u0[3], sg[3];
    double dd[10];      // precise-mode step
    double Jd[100];     // precise-mode Gram matrix
};

// S = 1: 8 lanes per cell, four cells per warp (a unit is a warp). S = 4: a
// warp per cell, four lanes in the place of each of the 8; they share the
// lines of the lane's run and repeat the rest, so that every sum is formed in
// the same order and a fit has the same bits (a unit is a CTA of four warps).
template <int S>
__device__ __forceinline__ int glane() { return (threadIdx.x / S) & (kG - 1); }
template <int S>
__device__ __forceinline__ unsigned gmask() {
    return S == 1 ? 0xFFu << ((threadIdx.x & 31) & ~(kG - 1)) : 0xffffffffu;
}
template <int S>
__device__ __forceinline__ int gbase() { return S == 1 ? (threadIdx.x & 31) & ~(kG - 1) : 0; }
// one thread per cell
template <int S>
__device__ __forceinline__ bool glead() { return (threadIdx.x & (kG * S - 1)) == 0; }
// vote of the unit's four cells
template <int S>
__device__ __forceinline__ bool unit_any(bool x) {
    if constexpr (S == 1) return __any_sync(0xffffffffu, x) != 0;
    else return __syncthreads_or(x) != 0;
}

template <int S>
__device__ __forceinline__ float gbcastf(float v, int src) { return __shfl_sync(gmask<S>(), v, gbase<S>() + src * S); }
template <int S>
__device__ __forceinline__ double gbcastd(double v, int src) { return __shfl_sync(gmask<S>(), v, gbase<S>() + src * S); }

template <int S>
__device__ __forceinline__ float gsumf(float v) {
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) v += __shfl_xor_sync(gmask<S>(), v, o * S);
    return gbcastf<S>(v, 0);
}
template <int S>
__device__ __forceinline__ double gsumd(double v) {
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) v += __shfl_xor_sync(gmask<S>(), v, o * S);
    return gbcastd<S>(v, 0);
}

// running double-float sum: s plus the accumulated error terms e
struct acc2 {
    float s, e;
};
__device__ __forceinline__ void acc2_add(acc2& A, float hi, float lo) {
    float s = __fadd_rn(A.s, hi);
    float bb = __fsub_rn(s, A.s);
    float err = __fadd_rn(__fsub_rn(A.s, __fsub_rn(s, bb)), __fsub_rn(hi, bb));
    A.s = s;
    A.e = __fadd_rn(A.e, __fadd_rn(err, lo));
}
// A += c (hi + lo), c an exactly representable small number
__device__ __forceinline__ void acc2_addc(acc2& A, float hi, float lo, float c) {
    float p = __fmul_rn(hi, c);
    float e = fmaf(hi, c, -p);
    e = fmaf(lo, c, e);
    acc2_add(A, p, e);
}
// The same running sums by Fast2Sum (Dekker): when |big| >= |small|, s - big
// is exact and small - (s - big) is the exact error of s = big + small, so
// the result equals acc2_add's bit for bit with three FMA-pipe operations
// instead of six; the operands are ordered on the ALU pipe. _nn: a
// non-negative running sum and term (fmaxf / fminf); _mag: any signs (one
// magnitude compare, two selects).
__device__ __forceinline__ void acc2_add_nn(acc2& A, float hi, float lo) {
    const float s = __fadd_rn(A.s, hi);
    const float big = fmaxf(A.s, hi), small = fminf(A.s, hi);
    A.e = __fadd_rn(A.e, __fadd_rn(__fsub_rn(small, __fsub_rn(s, big)), lo));
    A.s = s;
}
__device__ __forceinline__ void acc2_add_mag(acc2& A, float hi, float lo) {
    const float s = __fadd_rn(A.s, hi);
    const bool ab = fabsf(A.s) >= fabsf(hi);
    const float big = ab ? A.s : hi, small = ab ? hi : A.s;
    A.e = __fadd_rn(A.e, __fadd_rn(__fsub_rn(small, __fsub_rn(s, big)), lo));
    A.s = s;
}
template <int S>
__device__ __forceinline__ df2 gsum_acc(acc2 a) {
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) {
        float s = __shfl_xor_sync(gmask<S>(), a.s, o * S);
        float e = __shfl_xor_sync(gmask<S>(), a.e, o * S);
        acc2_add(a, s, e);
    }
    df2 r = df2_qtwo_sum(a.s, a.e);
    return {gbcastf<S>(r.hi, 0), gbcastf<S>(r.lo, 0)};
}
// the line sums of lane s of the four that stand for one
__device__ __forceinline__ acc2 from_sub(acc2 a, int s) {
    const int src = (threadIdx.x & 28) + s;
    return {__shfl_sync(0xffffffffu, a.s, src), __shfl_sync(0xffffffffu, a.e, src)};
}
__device__ __forceinline__ float from_sub(float a, int s) {
    return __shfl_sync(0xffffffffu, a, (threadIdx.x & 28) + s);
}

// a * b as an unnormalised pair: p = fl(a.hi b.hi) and the FP32 sum of the
// rest (its exact rounding error and the cross terms), without the final
// renormalisation; the next product reads the low part through its own
// cross term, so a ratio chain of N steps keeps about N ulp(2^-24) of
// relative error in its low part
__device__ __forceinline__ df2 df2_mul_raw(df2 a, df2 b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return {p, e};
}
__device__ __forceinline__ df2 dmul(df2 a, df2 b) { return df2_mul(a, b); }
__device__ __forceinline__ df2 dadd(df2 a, df2 b) { return df2_add(a, b); }

// index-space exponent coefficients (centred indices c_a = i_a - (N-1)/2):
// kc = (k0, kx, ky, kz, kxx, kxy, kxz, kyy, kyz, kzz)
__device__ __noinline__ void index_coeffs(const df2* e, const df2* wc, const df2* h, df2* kc) {
    const df2 two = {2.f, 0.f};
    // k0 = q(wc)
    df2 k0 = e[0];
    k0 = dadd(k0, dmul(e[1], wc[0]));
    k0 = dadd(k0, dmul(e[2], wc[1]));
    k0 = dadd(k0, dmul(e[3], wc[2]));
    k0 = dadd(k0, dmul(e[4], dmul(wc[0], wc[0])));
    k0 = dadd(k0, dmul(e[5], dmul(wc[0], wc[1])));
    k0 = dadd(k0, dmul(e[6], dmul(wc[0], wc[2])));
    k0 = dadd(k0, dmul(e[7], dmul(wc[1], wc[1])));
    k0 = dadd(k0, dmul(e[8], dmul(wc[1], wc[2])));
    k0 = dadd(k0, dmul(e[9], dmul(wc[2], wc[2])));
    kc[0] = k0;
    kc[1] = dmul(h[0], dadd(dadd(e[1], dmul(two, dmul(e[4], wc[0]))), dadd(dmul(e[5], wc[1]), dmul(e[6], wc[2]))));
    kc[2] = dmul(h[1], dadd(dadd(e[2], dmul(two, dmul(e[7], wc[1]))), dadd(dmul(e[5], wc[0]), dmul(e[8], wc[2]))));
    kc[3] = dmul(h[2], dadd(dadd(e[3], dmul(two, dmul(e[9], wc[2]))), dadd(dmul(e[6], wc[0]), dmul(e[8], wc[1]))));
    kc[4] = dmul(e[4], dmul(h[0], h[0]));
    kc[5] = dmul(e[5], dmul(h[0], h[1]));
    kc[6] = dmul(e[6], dmul(h[0], h[2]));
    kc[7] = dmul(e[7], dmul(h[1], h[1]));
    kc[8] = dmul(e[8], dmul(h[1], h[2]));
    kc[9] = dmul(e[9], dmul(h[2], h[2]));
}

// Can float recurrences represent every value and one-cell step of the
// block? (the minimum of a concave quadratic over a box is at a corner;
// one-cell steps are linear in position, extreme at the corners)
template <int N, int S>
__device__ bool edge_ok(const df2* kcd) {
    const int gl = glane<S>();
    constexpr float hN = 0.5f * (N - 1);
    float k[10];
#pragma unroll
    for (int q = 0; q < 10; ++q) k[q] = kcd[q].hi;
    bool ok = k[4] < 0.f && fabsf(2.f * k[4]) < 80.f && fabsf(2.f * k[7]) < 80.f && fabsf(k[5]) < 80.f;
    // corners: 8 lanes, one corner each
    {
        float x = (gl & 1) ? hN : -hN, y = (gl & 2) ? hN : -hN, z = (gl & 4) ? hN : -hN;
        float q = k[0] + k[1] * x + k[2] * y + k[3] * z + k[4] * x * x + k[5] * x * y + k[6] * x * z + k[7] * y * y +
                  k[8] * y * z + k[9] * z * z;
        ok = ok && (q > -80.f) && (q < 80.f);
    }
    // one-cell steps along x at the extreme lines (both ends) and along y of
    // the line starts
    {
        float y = (gl & 1) ? hN : -hN, z = (gl & 2) ? hN : -hN, x = (gl & 4) ? hN - 1.f : -hN;
        float d = k[4] * (2.f * x + 1.f) + k[1] + k[5] * y + k[6] * z;
        ok = ok && fabsf(d) < 80.f;
        float yy = (gl & 4) ? hN - 1.f : -hN;
        float d2 = k[7] * (2.f * yy + 1.f) + k[2] - hN * k[5] + k[8] * z;
        ok = ok && fabsf(d2) < 80.f;
    }
    return __all_sync(gmask<S>(), ok);
}

__device__ __forceinline__ void gram_line(float* g, const float* T, float cj, float ck) {
    float pj[5], pk[5];
    pj[0] = pk[0] = 1.f;
#pragma unroll
    for (int q = 1; q < 5; ++q) {
        pj[q] = pj[q - 1] * cj;
        pk[q] = pk[q - 1] * ck;
    }
#pragma unroll
    for (int p = 0; p <= 4; ++p)
#pragma unroll
        for (int q = 0; q <= 4 - p; ++q)
#pragma unroll
            for (int r = 0; r <= 4 - p - q; ++r) g[mono4(p, q, r)] = fmaf(T[p], pj[q] * pk[r], g[mono4(p, q, r)]);
}

// The block's sums are accumulated per plane: over a lane's run of lines in
// one v_z plane the z weight sk is constant, so the line sums S_p (and the
// FP32 sums T_p of degree <= 4) are first summed with the powers of the y
// weight sj (P: S0, S1, S2, sj S0, sj S1, sj^2 S0; G[p][q] = sum T_p sj^q),
// and at the end of the run those times the powers of sk go into the block's
// ten moments m and 35 Gram sums g (the Gram part where GRAM and rt).
template <bool GRAM>
__device__ __forceinline__ void plane_add(acc2 (&P)[6], float (&G)[GRAM ? 15 : 1], acc2 S0, acc2 S1, acc2 S2,
                                          const float (&T)[5], float sj, bool rt = true) {
    acc2_add(P[0], S0.s, S0.e);
    acc2_add(P[1], S1.s, S1.e);
    acc2_add(P[2], S2.s, S2.e);
    acc2_addc(P[3], S0.s, S0.e, sj);
    acc2_addc(P[4], S1.s, S1.e, sj);
    acc2_addc(P[5], S0.s, S0.e, sj * sj);
    if (GRAM && rt) {
        float pj = 1.f;
#pragma unroll
        for (int q = 0; q <= 4; ++q) {
#pragma unroll
            for (int pp = 0; pp <= 4 - q; ++pp) G[tri4(pp, q)] = fmaf(T[pp], pj, G[tri4(pp, q)]);
            pj *= sj;
        }
    }
}

template <bool GRAM>
__device__ __forceinline__ void plane_flush(acc2 (&m)[10], float (&g)[GRAM ? 35 : 1], acc2 (&P)[6],
                                            float (&G)[GRAM ? 15 : 1], float sk, bool rt = true) {
    acc2_add(m[0], P[0].s, P[0].e);
    acc2_add(m[1], P[1].s, P[1].e);
    acc2_add(m[2], P[3].s, P[3].e);
    acc2_addc(m[3], P[0].s, P[0].e, sk);
    acc2_add(m[4], P[2].s, P[2].e);
    acc2_add(m[5], P[4].s, P[4].e);
    acc2_addc(m[6], P[1].s, P[1].e, sk);
    acc2_add(m[7], P[5].s, P[5].e);
    acc2_addc(m[8], P[3].s, P[3].e, sk);
    acc2_addc(m[9], P[0].s, P[0].e, sk * sk);
#pragma unroll
    for (int q = 0; q < 6; ++q) P[q] = {0.f, 0.f};
    if (GRAM && rt) {
        float pk = 1.f;
#pragma unroll
        for (int r = 0; r <= 4; ++r) {
#pragma unroll
            for (int pp = 0; pp <= 4 - r; ++pp)
#pragma unroll
                for (int q = 0; q <= 4 - r - pp; ++q) g[mono4(pp, q, r)] = fmaf(G[tri4(pp, q)], pk, g[mono4(pp, q, r)]);
            pk *= sk;
        }
#pragma unroll
        for (int q = 0; q < 15; ++q) G[q] = 0.f;
    }
}

// Fast path from the box edge: double-float recurrences for the index
// moments of degree <= 2 (cs.m) and, with GRAM, FP32 sums of degree <= 4
// (cs.g) from the high parts of the same values, in one pass over the block;
// every line starts at v_x's lowest cell and every run of line starts at
// v_y's lowest, so every value of the block must be in the float range.
template <int N, bool GRAM, int S>
__device__ __noinline__ void eval_edge(CellScratch& cs, const df2* kc) {
    const int gl = glane<S>();
    constexpr float hN = 0.5f * (N - 1);
    constexpr int R = (N * N) / kG;
    const int l0 = gl * R, l1 = l0 + R;
    // shifted indices are integers (the shift moves the centre to a cell)
    const float ci0 = -hN - cs.shift[0], shy = cs.shift[1], shz = cs.shift[2];
    const df2 two = {2.f, 0.f};
    const df2 e_in = df2_exp(dmul(two, kc[4]));
    const df2 e_j = df2_exp(dmul(two, kc[7]));
    const df2 e_xy = df2_exp(kc[5]);
    const df2 mhN = {-hN, 0.f};
    acc2 m[10], P[6];
#pragma unroll
    for (int q = 0; q < 10; ++q) m[q] = {0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 6; ++q) P[q] = {0.f, 0.f};
    float g[GRAM ? 35 : 1], G[GRAM ? 15 : 1];
#pragma unroll
    for (int q = 0; q < (GRAM ? 35 : 1); ++q) g[q] = 0.f;
#pragma unroll
    for (int q = 0; q < (GRAM ? 15 : 1); ++q) G[q] = 0.f;
    df2 Ms = {0.f, 0.f}, rs = {0.f, 0.f}, rl = {0.f, 0.f};
    if constexpr (S > 1) {
        // S lines at a time, one per lane: starts in turn by every lane, the
        // lines side by side, then their sums in turn
        const int sub = threadIdx.x & (S - 1);
#pragma unroll 1
        for (int lb = l0; lb < l1; lb += S) {
            df2 M = Ms, r = rs;
#pragma unroll 1
            for (int s = 0; s < S && lb + s < l1; ++s) {
                const int l = lb + s;
                const int j = l % N, k = l / N;
                const float cj = (float)j - hN, ck = (float)k - hN;
                if (l == l0 || j == 0) {
                    // B = kx + kxy cj + kxz ck; C = k0 + ky cj + kz ck + kyy cj^2 + kyz cj ck + kzz ck^2
                    df2 B = dadd(kc[1], dadd(df2_mulf(kc[5], cj), df2_mulf(kc[6], ck)));
                    df2 C = dadd(kc[0], dadd(df2_mulf(kc[2], cj), df2_mulf(kc[3], ck)));
                    C = dadd(C, dadd(df2_mulf(kc[7], cj * cj), dadd(df2_mulf(kc[8], cj * ck), df2_mulf(kc[9], ck * ck))));
                    // start value at c_x = -hN, first ratio, line-to-line ratio
                    Ms = df2_exp(dadd(df2_mulf(kc[4], hN * hN), dadd(dmul(B, mhN), C)));
                    rs = df2_exp(dadd(df2_mulf(kc[4], 2.f - N), B));
                    rl = df2_exp(dadd(dadd(kc[2], df2_mulf(kc[5], -hN)), dadd(df2_mulf(kc[7], 2.f * cj + 1.f), df2_mulf(kc[8], ck))));
                }
                if (s == sub) {
                    M = Ms;
                    r = rs;
                }
                Ms = df2_mul(Ms, rl);
                rl = df2_mul(rl, e_j);
                rs = df2_mul(rs, e_xy);
            }
            acc2 S0 = {0.f, 0.f}, S1 = {0.f, 0.f}, S2 = {0.f, 0.f};
            float T0 = 0.f, T1 = 0.f, T2 = 0.f, T3 = 0.f, T4 = 0.f;
            float ci = ci0;
        // as below: unrolled by 2 (measured: 4.5% faster than by 4, 10% faster than by 8)
#pragma unroll 2
            for (int i = 0; i < N; ++i) {
                // ordered Fast2Sum (S0, S2: non-negative terms; S1: any sign;
                // measured: Harris fit 11.95 -> 11.63 ms per step, TwoSum's bits)
                // of the weighted terms as chained products, each split exactly
                // by an FMA: M ci = p1 + e1, (p1 + e1) ci = p2 + e2 (no ci^2;
                // the Jacobian's sums of degree 3 and 4 continue the chain)
                acc2_add_nn(S0, M.hi, M.lo);
                const float p1 = __fmul_rn(M.hi, ci);
                float e1 = fmaf(M.hi, ci, -p1);
                e1 = fmaf(M.lo, ci, e1);
                acc2_add_mag(S1, p1, e1);
                const float p2 = __fmul_rn(p1, ci);
                float e2 = fmaf(p1, ci, -p2);
                e2 = fmaf(e1, ci, e2);
                acc2_add_nn(S2, p2, e2);
                if (GRAM) {
                    const float p3 = __fmul_rn(p2, ci);
                    T0 = __fadd_rn(T0, M.hi);
                    T1 = __fadd_rn(T1, p1);
                    T2 = __fadd_rn(T2, p2);
                    T3 = __fadd_rn(T3, p3);
                    T4 = fmaf(p3, ci, T4);
                }
                // unnormalised products where only the pair's sum is read (the
                // ratio always, the value without the Jacobian's FP32 sums of
                // its high part): three operations fewer each (measured: fit
                // 11.63 -> 11.06 ms per step; iterations unchanged)
                M = GRAM ? df2_mul(M, r) : df2_mul_raw(M, r);
                r = df2_mul_raw(r, e_in);
                ci += 1.f;
            }
#pragma unroll 1
            for (int s = 0; s < S && lb + s < l1; ++s) {
                const int l = lb + s, j = l % N, k = l / N;
                const float cj = (float)j - hN, ck = (float)k - hN;
                const float T[5] = {GRAM ? from_sub(T0, s) : 0.f, GRAM ? from_sub(T1, s) : 0.f,
                                    GRAM ? from_sub(T2, s) : 0.f, GRAM ? from_sub(T3, s) : 0.f,
                                    GRAM ? from_sub(T4, s) : 0.f};
                plane_add<GRAM>(P, G, from_sub(S0, s), from_sub(S1, s), from_sub(S2, s), T, cj - shy);
                if (j == N - 1 || l == l1 - 1) plane_flush<GRAM>(m, g, P, G, ck - shz);
            }
        }
    } else {
#pragma unroll 1
        for (int l = l0; l < l1; ++l) {
            const int j = l % N, k = l / N;
            const float cj = (float)j - hN, ck = (float)k - hN;
            if (l == l0 || j == 0) {
                // B = kx + kxy cj + kxz ck; C = k0 + ky cj + kz ck + kyy cj^2 + kyz cj ck + kzz ck^2
                df2 B = dadd(kc[1], dadd(df2_mulf(kc[5], cj), df2_mulf(kc[6], ck)));
                df2 C = dadd(kc[0], dadd(df2_mulf(kc[2], cj), df2_mulf(kc[3], ck)));
                C = dadd(C, dadd(df2_mulf(kc[7], cj * cj), dadd(df2_mulf(kc[8], cj * ck), df2_mulf(kc[9], ck * ck))));
                // start value at c_x = -hN, first ratio, line-to-line ratio
                Ms = df2_exp(dadd(df2_mulf(kc[4], hN * hN), dadd(dmul(B, mhN), C)));
                rs = df2_exp(dadd(df2_mulf(kc[4], 2.f - N), B));
                rl = df2_exp(dadd(dadd(kc[2], df2_mulf(kc[5], -hN)), dadd(df2_mulf(kc[7], 2.f * cj + 1.f), df2_mulf(kc[8], ck))));
            }
            acc2 S0 = {0.f, 0.f}, S1 = {0.f, 0.f}, S2 = {0.f, 0.f};
            float T0 = 0.f, T1 = 0.f, T2 = 0.f, T3 = 0.f, T4 = 0.f;
            df2 M = Ms, r = rs;
            float ci = ci0;
    // unrolled by 2 (measured: 4.5% faster than by 4, 10% faster than by 8)
#pragma unroll 2
            for (int i = 0; i < N; ++i) {
                // ordered Fast2Sum (S0, S2: non-negative terms; S1: any sign;
                // measured: Harris fit 11.95 -> 11.63 ms per step, TwoSum's bits)
                // of the weighted terms as chained products, each split exactly
                // by an FMA: M ci = p1 + e1, (p1 + e1) ci = p2 + e2 (no ci^2;
                // the Jacobian's sums of degree 3 and 4 continue the chain)
                acc2_add_nn(S0, M.hi, M.lo);
                const float p1 = __fmul_rn(M.hi, ci);
                float e1 = fmaf(M.hi, ci, -p1);
                e1 = fmaf(M.lo, ci, e1);
                acc2_add_mag(S1, p1, e1);
                const float p2 = __fmul_rn(p1, ci);
                float e2 = fmaf(p1, ci, -p2);
                e2 = fmaf(e1, ci, e2);
                acc2_add_nn(S2, p2, e2);
                if (GRAM) {
                    const float p3 = __fmul_rn(p2, ci);
                    T0 = __fadd_rn(T0, M.hi);
                    T1 = __fadd_rn(T1, p1);
                    T2 = __fadd_rn(T2, p2);
                    T3 = __fadd_rn(T3, p3);
                    T4 = fmaf(p3, ci, T4);
                }
                // unnormalised products where only the pair's sum is read (the
                // ratio always, the value without the Jacobian's FP32 sums of
                // its high part): three operations fewer each (measured: fit
                // 11.63 -> 11.06 ms per step; iterations unchanged)
                M = GRAM ? df2_mul(M, r) : df2_mul_raw(M, r);
                r = df2_mul_raw(r, e_in);
                ci += 1.f;
            }
            const float T[5] = {T0, T1, T2, T3, T4};
            plane_add<GRAM>(P, G, S0, S1, S2, T, cj - shy);
            if (j == N - 1 || l == l1 - 1) plane_flush<GRAM>(m, g, P, G, ck - shz);
            Ms = df2_mul(Ms, rl);
            rl = df2_mul(rl, e_j);
            rs = df2_mul(rs, e_xy);
        }
    }
#pragma unroll
    for (int q = 0; q < 10; ++q) {
        df2 v = gsum_acc<S>(m[q]);
        if (gl == 0) cs.m[q] = v;
    }
    if (GRAM) {
#pragma unroll
        for (int q = 0; q < 35; ++q) {
            float v = gsumf<S>(g[q]);
            if (gl == 0) cs.g[q] = v;
        }
    }
    __syncwarp(gmask<S>());
}

// Slow path: one FP64 exponential per cell (any exponent range).
template <int N, int S>
__device__ __noinline__ void eval_slow(CellScratch& cs, const df2* kcd, bool want_gram) {
    const int gl = glane<S>();
    constexpr double hN = 0.5 * (N - 1);
    double kc[10];
#pragma unroll
    for (int q = 0; q < 10; ++q) kc[q] = df2_to_d(kcd[q]);
    const double shx = cs.shift[0], shy = cs.shift[1], shz = cs.shift[2];
    double m[10];
    float g[35];
#pragma unroll
    for (int q = 0; q < 10; ++q) m[q] = 0.0;
#pragma unroll
    for (int q = 0; q < 35; ++q) g[q] = 0.f;
#pragma unroll 1
    for (int l = gl; l < N * N; l += kG) {
        const int j = l % N, k = l / N;
        const double cj = j - hN, ck = k - hN;
        const double B = kc[1] + kc[5] * cj + kc[6] * ck;
        const double C = kc[0] + kc[2] * cj + kc[3] * ck + kc[7] * cj * cj + kc[8] * cj * ck + kc[9] * ck * ck;
        double S0 = 0, S1 = 0, S2 = 0;
        float T[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int i = 0; i < N; ++i) {
            const double cq = i - hN;
            const double M = exp(C + cq * (B + kc[4] * cq));
            const double ci = cq - shx;
            S0 += M;
            S1 = fma(M, ci, S1);
            S2 = fma(M, ci * ci, S2);
            if (want_gram) {
                const float Mf = (float)M, cf = (float)ci;
                T[0] += Mf;
                T[1] = fmaf(Mf, cf, T[1]);
                T[2] = fmaf(Mf, cf * cf, T[2]);
                T[3] = fmaf(Mf, cf * cf * cf, T[3]);
                T[4] = fmaf(Mf, cf * cf * cf * cf, T[4]);
            }
        }
        const double sj = cj - shy, sk = ck - shz;
        m[0] += S0; m[1] += S1; m[2] += sj * S0; m[3] += sk * S0; m[4] += S2;
        m[5] += sj * S1; m[6] += sk * S1; m[7] += sj * sj * S0; m[8] += sj * sk * S0; m[9] += sk * sk * S0;
        if (want_gram) gram_line(g, T, (float)sj, (float)sk);
    }
#pragma unroll
    for (int q = 0; q < 10; ++q) {
        double v = gsumd<S>(m[q]);
        if (gl == 0) cs.m[q] = df2_d(v);
    }
    if (want_gram)
#pragma unroll
        for (int q = 0; q < 35; ++q) {
            float v = gsumf<S>(g[q]);
            if (gl == 0) cs.g[q] = v;
        }
    __syncwarp(gmask<S>());
}

// Evaluates the moments (and the Gram sums if gram) at eta; returns whether
// the fast path was taken (uniform over the group).
// the centre-out pass and the slow path for blocks beyond the float range
// (defined at the end of this file, away from the common path's code)
template <int N, int S>
__device__ __noinline__ bool evaluate_wide(CellScratch& cs, const df2* kc, bool gram);

// WIDE selects the kernel that holds the centre-out evaluation; it is a
// kernel of its own because holding that code slowed the common evaluation
// by about 5% (measured on the Harris workload, same iterations).
// In the WIDE kernel every block the centre-out pass can take takes it (not
// only those beyond the float range), so that the cells of a warp run the
// same code rather than both passes in turn (measured: instruction-fetch
// stalls dominated the mixed form).
template <int N, bool WIDE, int S>
__device__ __noinline__ bool evaluate(CellScratch& cs, const df2* eta, bool gram) {
    df2 kc[10];
    index_coeffs(eta, cs.wc, cs.h, kc);
    if constexpr (WIDE) return evaluate_wide<N, S>(cs, kc, gram);
    const bool fast = edge_ok<N, S>(kc);
    if (fast) {
        if (gram) eval_edge<N, true, S>(cs, kc);
        else eval_edge<N, false, S>(cs, kc);
        return true;
    }
    eval_slow<N, S>(cs, kc, gram);
    return false;
}

// evaluations of one fit (kept in registers, identical in all lanes)
struct FitWork {
    unsigned m, g, slow, precise, warm;
    __device__ __forceinline__ void add(bool fast, bool gram) {
        m += fast ? 1u : 0u;
        g += (fast && gram) ? 1u : 0u;
        slow += fast ? 0u : 1u;
    }
};

// w-space discrete moments D (10) from the index moments (double-float)
__device__ __noinline__ void w_moments(const CellScratch& cs, df2 vol, df2* D) {
    const df2* m = cs.m;
    const df2* w = cs.wm;
    const df2* h = cs.h;
    const df2 two = {2.f, 0.f};
    D[0] = m[0];
    D[1] = dadd(dmul(w[0], m[0]), dmul(h[0], m[1]));
    D[2] = dadd(dmul(w[1], m[0]), dmul(h[1], m[2]));
    D[3] = dadd(dmul(w[2], m[0]), dmul(h[2], m[3]));
    D[4] = dadd(dadd(dmul(dmul(w[0], w[0]), m[0]), dmul(dmul(two, dmul(w[0], h[0])), m[1])), dmul(dmul(h[0], h[0]), m[4]));
    D[5] = dadd(dadd(dmul(dmul(w[0], w[1]), m[0]), dmul(dmul(w[0], h[1]), m[2])),
                dadd(dmul(dmul(h[0], w[1]), m[1]), dmul(dmul(h[0], h[1]), m[5])));
    D[6] = dadd(dadd(dmul(dmul(w[0], w[2]), m[0]), dmul(dmul(w[0], h[2]), m[3])),
                dadd(dmul(dmul(h[0], w[2]), m[1]), dmul(dmul(h[0], h[2]), m[6])));
    D[7] = dadd(dadd(dmul(dmul(w[1], w[1]), m[0]), dmul(dmul(two, dmul(w[1], h[1])), m[2])), dmul(dmul(h[1], h[1]), m[7]));
    D[8] = dadd(dadd(dmul(dmul(w[1], w[2]), m[0]), dmul(dmul(w[1], h[2]), m[3])),
                dadd(dmul(dmul(h[1], w[2]), m[2]), dmul(dmul(h[1], h[2]), m[8])));
    D[9] = dadd(dadd(dmul(dmul(w[2], w[2]), m[0]), dmul(dmul(two, dmul(w[2], h[2])), m[3])), dmul(dmul(h[2], h[2]), m[9]));
#pragma unroll
    for (int q = 0; q < 10; ++q) D[q] = dmul(D[q], vol);
}

// coefficients c[A][p] = C(A, p) w^(A-p) h^p of (w + h xi)^A, packed by tri(A, p)
__device__ __forceinline__ void binom_coeffs(float w, float h, float* c) {
    float pw[5], ph[5];
    pw[0] = ph[0] = 1.f;
#pragma unroll
    for (int e = 1; e < 5; ++e) {
        pw[e] = pw[e - 1] * w;
        ph[e] = ph[e - 1] * h;
    }
#pragma unroll
    for (int A = 0; A <= 4; ++A)
#pragma unroll
        for (int p = 0; p <= A; ++p) c[tri(A, p)] = (float)binom4(A, p) * pw[A - p] * ph[p];
}

// Jacobian in w-space from the FP32 index sums g (degree <= 4): three
// separable binomial transforms (x, then y, then z), then the FP32 Cholesky
// solve J dl = rhs into cs.step. Lane 0 of the group, fully unrolled, in
// shared memory.
template <int S>
__device__ __noinline__ bool newton_step_f32(CellScratch& cs, float vol) {
    int ok = 1;
    if (glead<S>()) {
        float cx[15], cy[15], cz[15];
        binom_coeffs(cs.wm[0].hi, cs.h[0].hi, cx);
        binom_coeffs(cs.wm[1].hi, cs.h[1].hi, cy);
        binom_coeffs(cs.wm[2].hi, cs.h[2].hi, cz);
        float* g = cs.g;
        float* U = cs.U;
        float* W = cs.W;
        // x: U[A, q, r] = sum_p c_x[A][p] g[p, q, r]
#pragma unroll
        for (int A = 0; A <= 4; ++A)
#pragma unroll
            for (int q = 0; q <= 4 - A; ++q)
#pragma unroll
                for (int r = 0; r <= 4 - A - q; ++r) {
                    float sacc = 0.f;
#pragma unroll
                    for (int p = 0; p <= A; ++p) sacc = fmaf(cx[tri(A, p)], g[mono4(p, q, r)], sacc);
                    U[mono4(A, q, r)] = sacc;
                }
        // y: W[A, B, r] = sum_q c_y[B][q] U[A, q, r]
#pragma unroll
        for (int A = 0; A <= 4; ++A)
#pragma unroll
            for (int B = 0; B <= 4 - A; ++B)
#pragma unroll
                for (int r = 0; r <= 4 - A - B; ++r) {
                    float sacc = 0.f;
#pragma unroll
                    for (int q = 0; q <= B; ++q) sacc = fmaf(cy[tri(B, q)], U[mono4(A, q, r)], sacc);
                    W[mono4(A, B, r)] = sacc;
                }
        // z: U[A, B, C] = vol sum_r c_z[C][r] W[A, B, r]
#pragma unroll
        for (int A = 0; A <= 4; ++A)
#pragma unroll
            for (int B = 0; B <= 4 - A; ++B)
#pragma unroll
                for (int C = 0; C <= 4 - A - B; ++C) {
                    float sacc = 0.f;
#pragma unroll
                    for (int r = 0; r <= C; ++r) sacc = fmaf(cz[tri(C, r)], W[mono4(A, B, r)], sacc);
                    U[mono4(A, B, C)] = sacc * vol;
                }
        float* J = cs.J;
#pragma unroll
        for (int a = 0; a < 10; ++a)
#pragma unroll
            for (int b = 0; b <= a; ++b)
                J[tri(a, b)] = U[mono4(expo(a, 0) + expo(b, 0), expo(a, 1) + expo(b, 1), expo(a, 2) + expo(b, 2))];
        float inv[10];
#pragma unroll
        for (int i = 0; i < 10; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) {
                float sacc = J[tri(i, j)];
#pragma unroll
                for (int k = 0; k < j; ++k) sacc = fmaf(-J[tri(i, k)], J[tri(j, k)], sacc);
                if (i == j) {
                    ok &= sacc > 0.f ? 1 : 0;
                    const float d = sqrtf(fmaxf(sacc, 1e-30f));
                    J[tri(i, i)] = d;
                    inv[i] = 1.f / d;
                } else {
                    J[tri(i, j)] = sacc * inv[j];
                }
            }
        float y[10];
#pragma unroll
        for (int i = 0; i < 10; ++i) {
            float sacc = cs.rhs[i];
#pragma unroll
            for (int k = 0; k < i; ++k) sacc = fmaf(-J[tri(i, k)], y[k], sacc);
            y[i] = sacc * inv[i];
        }
#pragma unroll
        for (int i = 9; i >= 0; --i) {
            float sacc = y[i];
#pragma unroll
            for (int k = i + 1; k < 10; ++k) sacc = fmaf(-J[tri(k, i)], y[k], sacc);
            y[i] = sacc * inv[i];
        }
#pragma unroll
        for (int i = 0; i < 10; ++i) cs.step[i] = df2_f(y[i]);
    }
    __syncwarp(gmask<S>());
    return __shfl_sync(gmask<S>(), ok, gbase<S>()) != 0;
}

// Precise mode: Gram matrix in FP64 (one exponential per cell) and FP64
// Cholesky by lane 0 of the group; rhs = -G in FP64 (cs.dd on input).
template <int N, int S>
__device__ __noinline__ bool newton_step_f64(CellScratch& cs, const df2* eta, double vol) {
    const int gl = glane<S>();
    constexpr double hN = 0.5 * (N - 1);
    df2 kcd[10];
    index_coeffs(eta, cs.wc, cs.h, kcd);
    double kc[10], wc[3], h[3];
#pragma unroll
    for (int q = 0; q < 10; ++q) kc[q] = df2_to_d(kcd[q]);
    for (int q = 0; q < 3; ++q) {
        wc[q] = df2_to_d(cs.wc[q]);
        h[q] = df2_to_d(cs.h[q]);
    }
    double W[35];
#pragma unroll
    for (int q = 0; q < 35; ++q) W[q] = 0.0;
#pragma unroll 1
    for (int l = gl; l < N * N; l += kG) {
        const int j = l % N, k = l / N;
        const double cj = j - hN, ck = k - hN;
        const double B = kc[1] + kc[5] * cj + kc[6] * ck;
        const double C = kc[0] + kc[2] * cj + kc[3] * ck + kc[7] * cj * cj + kc[8] * cj * ck + kc[9] * ck * ck;
        double T[5] = {0, 0, 0, 0, 0};
#pragma unroll 1
        for (int i = 0; i < N; ++i) {
            const double ci = i - hN;
            const double M = exp(C + ci * (B + kc[4] * ci));
            const double w = wc[0] + h[0] * ci;
            double p = M;
            for (int q = 0; q < 5; ++q) {
                T[q] += p;
                p *= w;
            }
        }
        const double wy = wc[1] + h[1] * cj, wz = wc[2] + h[2] * ck;
        double py[5], pz[5];
        py[0] = pz[0] = 1.0;
#pragma unroll
        for (int q = 1; q < 5; ++q) {
            py[q] = py[q - 1] * wy;
            pz[q] = pz[q - 1] * wz;
        }
#pragma unroll
        for (int a = 0; a <= 4; ++a)
#pragma unroll
            for (int b = 0; b <= 4 - a; ++b)
#pragma unroll
                for (int c = 0; c <= 4 - a - b; ++c) W[mono4(a, b, c)] += T[a] * py[b] * pz[c];
    }
#pragma unroll
    for (int q = 0; q < 35; ++q) W[q] = gsumd<S>(W[q]) * vol;
    int ok = 1;
    if (glead<S>()) {
        const int E[10][3] = {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0},
                              {1, 1, 0}, {1, 0, 1}, {0, 2, 0}, {0, 1, 1}, {0, 0, 2}};
        double* J = cs.Jd;
        for (int a = 0; a < 10; ++a)
            for (int b = 0; b <= a; ++b)
                J[a * 10 + b] = W[mono4(E[a][0] + E[b][0], E[a][1] + E[b][1], E[a][2] + E[b][2])];
#pragma unroll 1
        for (int i = 0; i < 10 && ok; ++i)
#pragma unroll 1
            for (int j = 0; j <= i; ++j) {
                double s = J[i * 10 + j];
                for (int k = 0; k < j; ++k) s -= J[i * 10 + k] * J[j * 10 + k];
                if (i == j) {
                    if (!(s > 0.0)) {
                        ok = 0;
                        break;
                    }
                    J[i * 10 + i] = sqrt(s);
                } else {
                    J[i * 10 + j] = s / J[j * 10 + j];
                }
            }
        if (ok) {
            double y[10];
            for (int i = 0; i < 10; ++i) {
                double s = cs.dd[i];
                for (int k = 0; k < i; ++k) s -= J[i * 10 + k] * y[k];
                y[i] = s / J[i * 10 + i];
            }
            for (int i = 9; i >= 0; --i) {
                double s = y[i];
                for (int k = i + 1; k < 10; ++k) s -= J[k * 10 + i] * cs.dd[k];
                cs.dd[i] = s / J[i * 10 + i];
            }
        }
    }
    __syncwarp(gmask<S>());
    return __shfl_sync(gmask<S>(), ok, gbase<S>()) != 0;
}

// Fit set-up by the 8 lanes of a group (targets in cs.tgt): scaled
// coordinates, w-space targets and the start point (the continuous
// Maxwellian of the targets). Returns false, with zero coefficients written,
// for invalid targets (n <= 0 or non-finite, Theta not positive definite).
template <int N, int S>
__device__ __noinline__ bool fit_setup(CellScratch& cs, const FitArgs& a, double* coef, const float* warm) {
    const int gl = glane<S>();
    const unsigned msk = gmask<S>();
    const double* t = cs.tgt;
    const double n = t[0];
    auto write_zero = [&]() {
        if (!coef) return;
        coef[gl] = 0.0;
        coef[gl + 8] = 0.0;
    };
    if (!(n > 0.0) || !isfinite(n)) {
        write_zero();
        return false;
    }
    // scaled coordinates from FP32 estimates of u and Theta (any u0, sigma
    // define a valid change of variables; T below is transformed exactly)
    const float nf = (float)n;
    float u0f[3], Th[9];
    for (int q = 0; q < 3; ++q) u0f[q] = (float)t[1 + q] / nf;
    const int pk[3][3] = {{4, 5, 6}, {5, 7, 8}, {6, 8, 9}};
    for (int p = 0; p < 3; ++p)
        for (int q = 0; q < 3; ++q) Th[p * 3 + q] = (float)t[pk[p][q]] / nf - u0f[p] * u0f[q];
    {
        // positive definite?
        float l00 = Th[0];
        bool pd = l00 > 0.f;
        if (pd) {
            l00 = sqrtf(l00);
            float l10 = Th[3] / l00, l20 = Th[6] / l00, d1 = Th[4] - l10 * l10;
            pd = d1 > 0.f;
            if (pd) {
                float l11 = sqrtf(d1), l21 = (Th[7] - l20 * l10) / l11;
                pd = Th[8] - l20 * l20 - l21 * l21 > 0.f;
            }
        }
        if (!pd) {
            write_zero();
            return false;
        }
    }
    if (gl < 3) {
        const int q = gl;
        const double u0 = (double)u0f[q], sg = (double)sqrtf(Th[q * 4]);
        cs.u0[q] = u0;
        cs.sg[q] = sg;
        const double h = a.dv[q] / sg;
        const double wc = (a.vmin[q] + 0.5 * N * a.dv[q] - u0) / sg;
        float ic = rintf((float)((u0 - a.vmin[q]) / a.dv[q] - 0.5));
        ic = fminf(fmaxf(ic, 0.f), (float)(N - 1));
        const float sh = ic - 0.5f * (N - 1);
        cs.shift[q] = sh;
        cs.h[q] = df2_d(h);
        cs.wc[q] = df2_d(wc);
        cs.wm[q] = df2_d(wc + h * (double)sh);
    }
    // targets in w-space (FP64 once per fit): lane q computes T_q, lanes 0, 1 also T_8, T_9
    {
        const int ab[10][2] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 1}, {0, 2}, {1, 1}, {1, 2}, {2, 2}};
        const double u0[3] = {(double)u0f[0], (double)u0f[1], (double)u0f[2]};
        double sg[3];
        for (int q = 0; q < 3; ++q) sg[q] = (double)sqrtf(Th[q * 4]);
        for (int r = 0; r < 2; ++r) {
            const int c = gl + 8 * r;
            if (c >= 10) break;
            double v;
            if (c == 0) v = n;
            else if (c < 4) v = (t[c] - n * u0[c - 1]) / sg[c - 1];
            else {
                const int p = ab[c][0], q = ab[c][1];
                v = (t[pk[p][q]] - u0[p] * t[1 + q] - u0[q] * t[1 + p] + n * u0[p] * u0[q]) / (sg[p] * sg[q]);
            }
            cs.T[c] = df2_d(v);
        }
    }
    __syncwarp(msk);
    // start: continuous Maxwellian of the targets in w-space (FP32)
    {
        float Cw[9], P[9], mw[3];
        for (int p = 0; p < 3; ++p) mw[p] = cs.T[1 + p].hi / nf;
        const int sidx[3][3] = {{4, 5, 6}, {5, 7, 8}, {6, 8, 9}};
        for (int p = 0; p < 3; ++p)
            for (int q = 0; q < 3; ++q) Cw[p * 3 + q] = cs.T[sidx[p][q]].hi / nf - mw[p] * mw[q];
        float c00 = Cw[4] * Cw[8] - Cw[5] * Cw[7], c01 = Cw[5] * Cw[6] - Cw[3] * Cw[8], c02 = Cw[3] * Cw[7] - Cw[4] * Cw[6];
        float detC = Cw[0] * c00 + Cw[1] * c01 + Cw[2] * c02;
        float id = 1.f / detC;
        P[0] = c00 * id;
        P[1] = (Cw[2] * Cw[7] - Cw[1] * Cw[8]) * id;
        P[2] = (Cw[1] * Cw[5] - Cw[2] * Cw[4]) * id;
        P[4] = (Cw[0] * Cw[8] - Cw[2] * Cw[6]) * id;
        P[5] = (Cw[2] * Cw[3] - Cw[0] * Cw[5]) * id;
        P[8] = (Cw[0] * Cw[4] - Cw[1] * Cw[3]) * id;
        P[3] = P[1];
        P[6] = P[2];
        P[7] = P[5];
        float lam[3], quad = 0.f;
        for (int p = 0; p < 3; ++p) lam[p] = P[p * 3] * mw[0] + P[p * 3 + 1] * mw[1] + P[p * 3 + 2] * mw[2];
        for (int p = 0; p < 3; ++p) quad += mw[p] * lam[p];
        const float s3 = sqrtf(Th[0]) * sqrtf(Th[4]) * sqrtf(Th[8]);
        const float logdet = logf(detC) + 2.f * logf(s3);
        const float init[10] = {logf(nf) - 1.5f * logf(6.2831853f) - 0.5f * logdet - 0.5f * quad,
                                lam[0], lam[1], lam[2], -0.5f * P[0], -P[1], -P[2], -0.5f * P[4], -P[5], -0.5f * P[8]};
        for (int r = 0; r < 2; ++r) {
            const int c = gl + 8 * r;
            if (c >= 10) break;
            float v = 0.f;
#pragma unroll
            for (int q = 0; q < 10; ++q)
                if (q == c) v = init[q];
            cs.eta0[c] = df2_f(v);
            // warm start: the predicted correction eta* - eta_0 (if finite)
            const float dw = warm ? warm[c] : 0.f;
            cs.eta[c] = (dw == dw && fabsf(dw) < 1e30f) ? dadd(df2_f(v), df2_f(dw)) : df2_f(v);
        }
    }
    __syncwarp(msk);

    return true;
}

// Newton iteration from cs.eta by the 8 lanes of a group; all four groups of
// the warp call it together (active = false for a group that only keeps the
// others company). Returns whether the residual reached the tolerance; the
// number of Newton steps is added to *iters.
template <int N, bool WIDE, int S>
__device__ __noinline__ bool newton_loop(CellScratch& cs, const FitArgs& a, bool active, float nf, df2 vol,
                                         float tolf, int* iters, FitWork& work) {
    const int gl = glane<S>();
    const unsigned msk = gmask<S>();
    bool converged = false, have_gram = false;
    int nit = 0;
    if (active) {
        work.add(evaluate<N, WIDE, S>(cs, cs.eta, true), true);
        have_gram = true;
    }
    for (int it = 0;; ++it) {
        df2 G[10], L0 = {0.f, 0.f};
        float grel = 0.f;
        if (active) {
            df2 D[10];
            w_moments(cs, vol, D);
            float gmax = 0.f;
            bool fin = true;
#pragma unroll
            for (int q = 0; q < 10; ++q) {
                G[q] = dadd(D[q], df2_neg(cs.T[q]));
                const float v = fabsf(G[q].hi + G[q].lo);
                fin = fin && isfinite(v);
                gmax = fmaxf(gmax, v);
            }
            if (!fin || gmax <= tolf || it == a.max_iter) {
                converged = fin && gmax <= tolf;
                active = false;
                nit = it;
            }
            grel = gmax / nf;
            L0 = D[0];
        }
        if (!unit_any<S>(active)) break;
        const bool precise = it >= 6;
        // Jacobian at eta where the last evaluation did not form it
        const bool need_g = active && !precise && !have_gram;
        if (unit_any<S>(need_g)) {
            if (need_g) {
                work.add(evaluate<N, WIDE, S>(cs, cs.eta, true), true);
                have_gram = true;
            }
        }
        if (active) {
            bool ok;
            if (precise) {
                if (gl == 0)
                    for (int q = 0; q < 10; ++q) cs.dd[q] = -df2_to_d(G[q]);
                work.precise += 1u;
                __syncwarp(msk);
                ok = newton_step_f64<N, S>(cs, cs.eta, df2_to_d(vol));
                for (int r = 0; r < 2; ++r) {
                    const int c = gl + 8 * r;
                    if (c < 10) cs.step[c] = df2_d(cs.dd[c]);
                }
                __syncwarp(msk);
            } else {
                if (gl == 0)
                    for (int q = 0; q < 10; ++q) cs.rhs[q] = -(G[q].hi + G[q].lo);
                __syncwarp(msk);
                ok = newton_step_f32<S>(cs, vol.hi);
            }
            if (!ok) {
                active = false;
                nit = it;
            }
        }
        // damped step: backtracking on L(eta) = D_0 - eta . T while far away
        // (closer in, the decrease of L is below its double-float resolution
        // and the full Newton step is taken)
        const bool damp = active && grel > 1e-3f;
        float gd = 0.f;
        if (damp) {
#pragma unroll
            for (int q = 0; q < 10; ++q) {
                L0 = dadd(L0, df2_neg(dmul(cs.eta[q], cs.T[q])));
                gd = fmaf(G[q].hi, cs.step[q].hi, gd);
            }
        }
        // form the Jacobian with the next evaluation only where another Newton
        // step is likely: below 1e-5 of n one step from here converges in
        // almost every cell (measured: the Jacobian sums halve, the moment
        // evaluations grow by 0.2%, the fit time drops by 1.3%)
        const bool gram_next = unit_any<S>(active && grel > 1e-5f);
        float lamb = 1.f;
        bool pending = active;
        for (int ls = 0; ls < 12; ++ls) {
            if (pending) {
                for (int r = 0; r < 2; ++r) {
                    const int c = gl + 8 * r;
                    if (c < 10) cs.et[c] = dadd(cs.eta[c], df2_mulf(cs.step[c], lamb));
                }
                __syncwarp(msk);
                work.add(evaluate<N, WIDE, S>(cs, cs.et, gram_next), gram_next);
                if (!damp) {
                    pending = false;
                } else {
                    df2 L1 = dmul(cs.m[0], vol);
#pragma unroll
                    for (int q = 0; q < 10; ++q) L1 = dadd(L1, df2_neg(dmul(cs.et[q], cs.T[q])));
                    const df2 dL = dadd(L1, df2_neg(L0));
                    const float dlv = dL.hi + dL.lo;
                    if (isfinite(dlv) && dlv <= 1e-4f * lamb * gd) pending = false;
                    else lamb *= 0.5f;
                }
            }
            if (!unit_any<S>(pending)) break;
        }
        if (active) {
            have_gram = gram_next;
            for (int r = 0; r < 2; ++r) {
                const int c = gl + 8 * r;
                if (c < 10) cs.eta[c] = cs.et[c];
            }
            __syncwarp(msk);
        }
    }
    *iters += nit;
    return converged;
}

// the fitted exponent must be a Gaussian: -2 mu positive definite
__device__ __forceinline__ bool gaussian_exponent(const CellScratch& cs) {
    const float e4 = cs.eta[4].hi, e5 = cs.eta[5].hi, e6 = cs.eta[6].hi;
    const float e7 = cs.eta[7].hi, e8 = cs.eta[8].hi, e9 = cs.eta[9].hi;
    const float a00 = -2.f * e4, a10 = -e5, a20 = -e6, a11 = -2.f * e7, a21 = -e8, a22 = -2.f * e9;
    if (!(a00 > 0.f)) return false;
    const float l00 = sqrtf(a00), l10 = a10 / l00, l20 = a20 / l00, d1 = a11 - l10 * l10;
    if (!(d1 > 0.f)) return false;
    const float l11 = sqrtf(d1), l21 = (a21 - l20 * l10) / l11;
    return a22 - l20 * l20 - l21 * l21 > 0.f;
}

// The fallback of a fit that does not converge: the continuous Maxwellian of
// the targets in w-space, in FP64 (the start point eta0 is the same
// Maxwellian in FP32). C = covariance of w, m = mean of w:
// eta0 = log n - 3/2 log 2 pi - 1/2 log(det C s^2) - 1/2 m.P m, lambda = P m,
// quadratic part -1/2 w.P w, P = C^-1, s = sigma_x sigma_y sigma_z.
__device__ __noinline__ void continuous_eta_f64(const CellScratch& cs, double* eta) {
    const double n = df2_to_d(cs.T[0]);
    double mw[3], Cw[9];
    for (int p = 0; p < 3; ++p) mw[p] = df2_to_d(cs.T[1 + p]) / n;
    const int sidx[3][3] = {{4, 5, 6}, {5, 7, 8}, {6, 8, 9}};
    for (int p = 0; p < 3; ++p)
        for (int q = 0; q < 3; ++q) Cw[p * 3 + q] = df2_to_d(cs.T[sidx[p][q]]) / n - mw[p] * mw[q];
    const double c00 = Cw[4] * Cw[8] - Cw[5] * Cw[7], c01 = Cw[5] * Cw[6] - Cw[3] * Cw[8],
                 c02 = Cw[3] * Cw[7] - Cw[4] * Cw[6];
    const double detC = Cw[0] * c00 + Cw[1] * c01 + Cw[2] * c02;
    const double id = 1.0 / detC;
    double P[9];
    P[0] = c00 * id;
    P[1] = (Cw[2] * Cw[7] - Cw[1] * Cw[8]) * id;
    P[2] = (Cw[1] * Cw[5] - Cw[2] * Cw[4]) * id;
    P[4] = (Cw[0] * Cw[8] - Cw[2] * Cw[6]) * id;
    P[5] = (Cw[2] * Cw[3] - Cw[0] * Cw[5]) * id;
    P[8] = (Cw[0] * Cw[4] - Cw[1] * Cw[3]) * id;
    P[3] = P[1];
    P[6] = P[2];
    P[7] = P[5];
    double lam[3], quad = 0.0;
    for (int p = 0; p < 3; ++p) lam[p] = P[p * 3] * mw[0] + P[p * 3 + 1] * mw[1] + P[p * 3 + 2] * mw[2];
    for (int p = 0; p < 3; ++p) quad += mw[p] * lam[p];
    const double s3 = cs.sg[0] * cs.sg[1] * cs.sg[2];
    const double logdet = log(detC) + 2.0 * log(s3);
    eta[0] = log(n) - 1.5 * log(2.0 * 3.14159265358979323846) - 0.5 * logdet - 0.5 * quad;
    eta[1] = lam[0];
    eta[2] = lam[1];
    eta[3] = lam[2];
    eta[4] = -0.5 * P[0];
    eta[5] = -P[1];
    eta[6] = -P[2];
    eta[7] = -0.5 * P[4];
    eta[8] = -P[5];
    eta[9] = -0.5 * P[8];
}

// One fit by the 8 lanes of a group; all four groups of the warp call it
// together (have = false for a group without a cell). Starts from the MLP's
// prediction when warm is not null and falls back to the cold start (the
// continuous Maxwellian of the targets) if that run does not converge.
// Writes the coefficients (eta, u0, sigma) to coef (16 doubles, global; null:
// a fit that is only run along, nothing of it is kept),
// appends a training sample for a converged fit when harvesting, and returns
// the status: 0 converged, 1 fallback (continuous Maxwellian of the targets),
// 2 invalid targets.
template <int N, bool WIDE, int S>
__device__ int fit_cell(CellScratch& cs, const FitArgs& a, bool have, double* coef, const float* warm, int* iters,
                        FitWork& work) {
    const int gl = glane<S>();
    const unsigned msk = gmask<S>();
    *iters = 0;
    const bool valid = have && fit_setup<N, S>(cs, a, coef, warm);
    // the guard of the network's inference writes NaN rows for the fits it rejects
    if (valid && warm && warm[0] == warm[0] && fabsf(warm[0]) < 1e30f) work.warm += 1u;
    const double n = valid ? cs.tgt[0] : 1.0;
    const float nf = (float)n;
    const df2 vol = df2_d(a.dv[0] * a.dv[1] * a.dv[2]);
    const float tolf = (float)(a.tol * n);
    bool good = newton_loop<N, WIDE, S>(cs, a, valid, nf, vol, tolf, iters, work) && gaussian_exponent(cs);
    const bool retry = valid && warm != nullptr && !good;
    if (unit_any<S>(retry)) {
        if (retry) {
            for (int r = 0; r < 2; ++r) {
                const int c = gl + 8 * r;
                if (c < 10) cs.eta[c] = cs.eta0[c];
            }
            __syncwarp(msk);
        }
        const bool g2 = newton_loop<N, WIDE, S>(cs, a, retry, nf, vol, tolf, iters, work) && gaussian_exponent(cs);
        if (retry) good = g2;
    }
    if (!valid) return 2;
    double fb[10];
    if (!good) continuous_eta_f64(cs, fb);  // rare: every lane of the group forms it
    if (coef)
        for (int r = 0; r < 2; ++r) {
            const int c = gl + 8 * r;
            if (c < 10) coef[c] = good ? df2_to_d(cs.eta[c]) : fb[c];
            else if (c < 13) coef[c] = cs.u0[c - 10];
            else if (c < 16) coef[c] = cs.sg[c - 13];
        }
    if (good && coef && a.harvest) {
        unsigned long long slot = 0;
        if (glead<S>()) slot = atomicAdd(a.harvest_count, 1ull);
        slot = __shfl_sync(msk, slot, gbase<S>());
        if (slot < (unsigned long long)a.harvest_cap) {
            float* smp = a.harvest + slot * mlp::kSample;
            if (gl == 0) {
                float x[mlp::kIn];
                const bool ok = mlp::fit_inputs(cs.tgt, a.vmin, a.dv, a.vmax, x);
                for (int q = 0; q < mlp::kIn; ++q) smp[q] = x[q];
                smp[22] = ok ? 1.f : 0.f;
                smp[23] = 0.f;
            }
            for (int r = 0; r < 2; ++r) {
                const int c = gl + 8 * r;
                if (c < 10) {
                    const df2 d = dadd(cs.eta[c], df2_neg(cs.eta0[c]));
                    smp[mlp::kIn + c] = d.hi + d.lo;
                }
            }
        }
    }
    __syncwarp(msk);
    return good ? 0 : 1;
}

// Can the centre-out recurrences take every one-cell step of the block?
// The exponent is concave along x and y (a Maxwellian's quadratic form is negative
// definite), the step multipliers exp(2 k_xx), exp(2 k_yy), exp(+-k_xy) are
// finite, and the one-cell differences along x and along y stay within
// +-80 from one cell outside the box to one cell outside on the other side
// (differences are linear in position, extreme at the corners; 8 lanes,
// one corner each).
template <int N, int S>
__device__ bool centre_ok(const df2* kcd) {
    const int gl = glane<S>();
    constexpr float hN = 0.5f * (N - 1);
    float k[10];
#pragma unroll
    for (int q = 0; q < 10; ++q) k[q] = kcd[q].hi;
    bool ok = k[4] < 0.f && k[7] < 0.f && fabsf(2.f * k[4]) < 80.f && fabsf(2.f * k[7]) < 80.f &&
              fabsf(k[5]) < 80.f;
    {
        const float a = (gl & 1) ? hN : -hN - 1.f, b = (gl & 2) ? hN : -hN, c = (gl & 4) ? hN : -hN;
        // x step from x = a to a + 1 at (y, z) = (b, c)
        const float dx = k[4] * (2.f * a + 1.f) + k[1] + k[5] * b + k[6] * c;
        // y step from y = a to a + 1 at (x, z) = (b, c)
        const float dy = k[7] * (2.f * a + 1.f) + k[2] + k[5] * b + k[8] * c;
        ok = ok && fabsf(dx) < 80.f && fabsf(dy) < 80.f;
    }
    return __all_sync(gmask<S>(), ok);
}

// One v_x line of the centre-out path: the values from the start cell ic
// outward, right (ic .. N-1) then left (ic-1 .. 0), in one loop of N cells
// that turns at the right end; Mc is the value at ic, rR and rL the ratios
// to its right and left neighbours, and every further ratio is the previous
// one times exp(2 k_xx). Weights are the x indices relative to ic (integers,
// exact in FP32). The FP32 Jacobian sums are formed where rt is set.
template <int N, bool GRAM>
__device__ __forceinline__ void fast_line(acc2& S0, acc2& S1, acc2& S2, float (&T)[5], df2 Mc, df2 rR, df2 rL, df2 e_in,
                                          int ic, bool rt) {
    S0 = S1 = S2 = {0.f, 0.f};
    float T0 = 0.f, T1 = 0.f, T2 = 0.f, T3 = 0.f, T4 = 0.f;
    const df2 ML = df2_mul(Mc, rL), rLL = df2_mul(rL, e_in);
    const int turn = N - 1 - ic;
    df2 M = Mc, r = rR;
    float ci = 0.f, dc = 1.f;
// not unrolled: the wide kernel's code must stay small (instruction-fetch
// stalls; measured 8% faster per evaluation than unrolling by 4)
#pragma unroll 1
    for (int t = 0; t < N; ++t) {
        const float c2 = ci * ci;
        // TwoSum here: the ordered Fast2Sum of the edge pass measured about
        // 2% slower in the wide kernel
        acc2_add(S0, M.hi, M.lo);
        acc2_addc(S1, M.hi, M.lo, ci);
        acc2_addc(S2, M.hi, M.lo, c2);
        if (GRAM && rt) {
            T0 += M.hi;
            T1 = fmaf(M.hi, ci, T1);
            T2 = fmaf(M.hi, c2, T2);
            T3 = fmaf(M.hi, c2 * ci, T3);
            T4 = fmaf(M.hi, c2 * c2, T4);
        }
        // the ratio as an unnormalised pair, as in the edge pass
        const df2 Mn = df2_mul(M, r), rn = df2_mul_raw(r, e_in);
        const bool tt = t == turn;
        M = tt ? ML : Mn;
        r = tt ? rLL : rn;
        dc = tt ? -1.f : dc;
        ci = tt ? -1.f : ci + dc;
    }
    T[0] = T0;
    T[1] = T1;
    T[2] = T2;
    T[3] = T3;
    T[4] = T4;
}

// Float bound of one line's exponent q(c) = k_xx c^2 + B c + C over the box
// (c in [-hN, hN]): qhi, its maximum over the interval (an upper bound of
// the line's values), and qlo, its value at the cell nearest that maximum
// (one of the block's values); m_inv2kxx = -1 / (2 k_xx).
template <int N>
__device__ __forceinline__ void line_bounds(const df2* k, float m_inv2kxx, float cj, float ck, float& qhi,
                                            float& qlo) {
    constexpr float hN = 0.5f * (N - 1);
    const float B = k[1].hi + k[5].hi * cj + k[6].hi * ck;
    const float C = k[0].hi + k[2].hi * cj + k[3].hi * ck + k[7].hi * cj * cj + k[8].hi * cj * ck + k[9].hi * ck * ck;
    const float cs = fminf(fmaxf(B * m_inv2kxx, -hN), hN);
    qhi = (k[4].hi * cs + B) * cs + C;
    const float cn = rintf(cs + hN) - hN;
    qlo = (k[4].hi * cn + B) * cn + C;
}

// Fast path from the centre, for blocks whose values span more than the
// float range (a Maxwellian narrow against its velocity box): the same sums
// as eval_edge, in one pass over the block. Each lane owns R
// consecutive v_x lines; in each plane of its run it starts at the line
// nearest the mean's y index (one double-float exponential each for the
// value at the mean's x index and the ratios to the next cell in x and in
// y) and walks its lines outward in y, each line outward in x. Along any
// such walk the exponent is concave, so once values fall they keep falling:
// a value that underflows lies beyond its walk's maximum. The pass is valid
// (returned, uniform over the group) when no line's maximum can overflow
// (q < 80), the block's largest value is above e^-40, and every line whose
// start value is below 2^-100 (where the double-float pair loses its low
// part) has its maximum 45 e-folds below the block's largest value, i.e.
// contributes below 3e-20 of it. The Jacobian sums are formed where rt is
// set (GRAM is the storage for them).
template <int N, bool GRAM, int S>
__device__ __noinline__ bool eval_centre(CellScratch& cs, const df2* kc, bool rt) {
    const int gl = glane<S>();
    constexpr float hN = 0.5f * (N - 1);
    constexpr int R = (N * N) / kG;
    const int l0 = gl * R, l1 = l0 + R;
    const int ic = (int)(cs.shift[0] + hN), jc = (int)(cs.shift[1] + hN);
    const float cc = (float)ic - hN, shy = cs.shift[1], shz = cs.shift[2];
    const df2 two = {2.f, 0.f};
    const df2 e_in = df2_exp(dmul(two, kc[4]));
    const df2 e_j = df2_exp(dmul(two, kc[7]));
    const df2 e_xy = df2_exp(kc[5]);
    const df2 e_yx = df2_exp(df2_neg(kc[5]));
    const float m_inv2kxx = -0.5f / kc[4].hi;
    acc2 m[10], P[6];
#pragma unroll
    for (int q = 0; q < 10; ++q) m[q] = {0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 6; ++q) P[q] = {0.f, 0.f};
    float g[GRAM ? 35 : 1], G[GRAM ? 15 : 1];
#pragma unroll
    for (int q = 0; q < (GRAM ? 35 : 1); ++q) g[q] = 0.f;
#pragma unroll
    for (int q = 0; q < (GRAM ? 15 : 1); ++q) G[q] = 0.f;
    float qtop = -1e30f, qlost = -1e30f;
    bool over = false;
    constexpr float kPrecise = 7.8886091e-31f;  // 2^-100
    // one loop over the lane's R lines (one inlined copy of the line pass:
    // the kernel's code must stay within the instruction cache); a run of
    // lines in a plane starts with direct exponentials at the line nearest
    // the mean's y index, walks up to its last line, turns, and walks down
    int kk = l0 / N - 1, j = 0, dj = 1, left = 0, jb = 0, js = 0;
    float ck = 0.f, sk = 0.f;
    bool taint = false;
    df2 M0 = {0.f, 0.f}, rR0 = M0, rL0 = M0, rD0 = M0, Mc = M0, rV = M0, rR = M0, rL = M0, fxy = M0, fyx = M0;
    if constexpr (S > 1) {
        // S lines at a time, as in eval_edge
        const int sub = threadIdx.x & (S - 1);
#pragma unroll 1
        for (int tb = 0; tb < R; tb += S) {
            df2 Mo = M0, rRo = M0, rLo = M0;
            float sjs[S], sks[S];
            bool last[S];
#pragma unroll
            for (int s = 0; s < S; ++s) {
                sjs[s] = sks[s] = 0.f;
                last[s] = false;
                if (tb + s >= R) continue;
                if (left == 0) {
                    ++kk;
                    const int ja = max(l0 - kk * N, 0);
                    jb = min(l1 - 1 - kk * N, N - 1);
                    js = min(max(jc, ja), jb);
                    left = jb - ja + 1;
                    ck = (float)kk - hN;
                    sk = ck - shz;
                    const float cjs = (float)js - hN;
                    // exponent at (cc, cjs, ck) and its one-cell differences in x and y
                    const df2 B = dadd(kc[1], dadd(df2_mulf(kc[5], cjs), df2_mulf(kc[6], ck)));
                    df2 C = dadd(kc[0], dadd(df2_mulf(kc[2], cjs), df2_mulf(kc[3], ck)));
                    C = dadd(C, dadd(df2_mulf(kc[7], cjs * cjs), dadd(df2_mulf(kc[8], cjs * ck), df2_mulf(kc[9], ck * ck))));
                    const df2 q0 = dadd(C, df2_mulf(dadd(B, df2_mulf(kc[4], cc)), cc));
                    const df2 dX = dadd(B, df2_mulf(kc[4], 2.f * cc + 1.f));
                    const df2 dY =
                        dadd(dadd(kc[2], df2_mulf(kc[7], 2.f * cjs + 1.f)), dadd(df2_mulf(kc[5], cc), df2_mulf(kc[8], ck)));
                    M0 = df2_exp(q0);
                    rR0 = df2_exp(dX);
                    const df2 rU0 = df2_exp(dY);
                    // ratios to the left and down: exp(2 k_xx - dX), exp(2 k_yy - dY)
                    rL0 = df2_div(e_in, rR0);
                    rD0 = df2_div(e_j, rU0);
                    taint = !(M0.hi >= kPrecise);
                    Mc = M0;
                    rV = rU0;
                    rR = rR0;
                    rL = rL0;
                    fxy = e_xy;
                    fyx = e_yx;
                    j = js;
                    dj = 1;
                }
                const float cj = (float)j - hN;
                float qhi, qlo;
                line_bounds<N>(kc, m_inv2kxx, cj, ck, qhi, qlo);
                qtop = fmaxf(qtop, qlo);
                over = over || !(qhi < 80.f);
                if (taint || !(Mc.hi >= kPrecise)) qlost = fmaxf(qlost, qhi);
                if (s == sub) {
                    Mo = Mc;
                    rRo = rR;
                    rLo = rL;
                }
                sjs[s] = cj - shy;
                sks[s] = sk;
                --left;
                last[s] = left == 0;
                if (dj > 0 && j == jb) {
                    // turn: the downward walk starts one line below js
                    Mc = df2_mul(M0, rD0);
                    rV = df2_mul(rD0, e_j);
                    rR = df2_mul(rR0, e_yx);
                    rL = df2_mul(rL0, e_xy);
                    fxy = e_yx;
                    fyx = e_xy;
                    j = js - 1;
                    dj = -1;
                } else {
                    Mc = df2_mul(Mc, rV);
                    rV = df2_mul(rV, e_j);
                    rR = df2_mul(rR, fxy);
                    rL = df2_mul(rL, fyx);
                    j += dj;
                }
            }
            acc2 S0, S1, S2;
            float T[5];
            fast_line<N, GRAM>(S0, S1, S2, T, Mo, rRo, rLo, e_in, ic, rt);
#pragma unroll
            for (int s = 0; s < S; ++s) {
                if (tb + s >= R) continue;
                const float Ts[5] = {from_sub(T[0], s), from_sub(T[1], s), from_sub(T[2], s), from_sub(T[3], s),
                                     from_sub(T[4], s)};
                plane_add<GRAM>(P, G, from_sub(S0, s), from_sub(S1, s), from_sub(S2, s), Ts, sjs[s], rt);
                if (last[s]) plane_flush<GRAM>(m, g, P, G, sks[s], rt);
            }
        }
    } else {
#pragma unroll 1
        for (int t = 0; t < R; ++t) {
            if (left == 0) {
                ++kk;
                const int ja = max(l0 - kk * N, 0);
                jb = min(l1 - 1 - kk * N, N - 1);
                js = min(max(jc, ja), jb);
                left = jb - ja + 1;
                ck = (float)kk - hN;
                sk = ck - shz;
                const float cjs = (float)js - hN;
                // exponent at (cc, cjs, ck) and its one-cell differences in x and y
                const df2 B = dadd(kc[1], dadd(df2_mulf(kc[5], cjs), df2_mulf(kc[6], ck)));
                df2 C = dadd(kc[0], dadd(df2_mulf(kc[2], cjs), df2_mulf(kc[3], ck)));
                C = dadd(C, dadd(df2_mulf(kc[7], cjs * cjs), dadd(df2_mulf(kc[8], cjs * ck), df2_mulf(kc[9], ck * ck))));
                const df2 q0 = dadd(C, df2_mulf(dadd(B, df2_mulf(kc[4], cc)), cc));
                const df2 dX = dadd(B, df2_mulf(kc[4], 2.f * cc + 1.f));
                const df2 dY =
                    dadd(dadd(kc[2], df2_mulf(kc[7], 2.f * cjs + 1.f)), dadd(df2_mulf(kc[5], cc), df2_mulf(kc[8], ck)));
                M0 = df2_exp(q0);
                rR0 = df2_exp(dX);
                const df2 rU0 = df2_exp(dY);
                // ratios to the left and down: exp(2 k_xx - dX), exp(2 k_yy - dY)
                rL0 = df2_div(e_in, rR0);
                rD0 = df2_div(e_j, rU0);
                taint = !(M0.hi >= kPrecise);
                Mc = M0;
                rV = rU0;
                rR = rR0;
                rL = rL0;
                fxy = e_xy;
                fyx = e_yx;
                j = js;
                dj = 1;
            }
            const float cj = (float)j - hN;
            float qhi, qlo;
            line_bounds<N>(kc, m_inv2kxx, cj, ck, qhi, qlo);
            qtop = fmaxf(qtop, qlo);
            over = over || !(qhi < 80.f);
            if (taint || !(Mc.hi >= kPrecise)) qlost = fmaxf(qlost, qhi);
            acc2 S0, S1, S2;
            float T[5];
            fast_line<N, GRAM>(S0, S1, S2, T, Mc, rR, rL, e_in, ic, rt);
            plane_add<GRAM>(P, G, S0, S1, S2, T, cj - shy, rt);
            --left;
            if (left == 0) plane_flush<GRAM>(m, g, P, G, sk, rt);
            if (dj > 0 && j == jb) {
                // turn: the downward walk starts one line below js
                Mc = df2_mul(M0, rD0);
                rV = df2_mul(rD0, e_j);
                rR = df2_mul(rR0, e_yx);
                rL = df2_mul(rL0, e_xy);
                fxy = e_yx;
                fyx = e_xy;
                j = js - 1;
                dj = -1;
            } else {
                Mc = df2_mul(Mc, rV);
                rV = df2_mul(rV, e_j);
                rR = df2_mul(rR, fxy);
                rL = df2_mul(rL, fyx);
                j += dj;
            }
        }
    }
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) {
        qtop = fmaxf(qtop, __shfl_xor_sync(gmask<S>(), qtop, o * S));
        qlost = fmaxf(qlost, __shfl_xor_sync(gmask<S>(), qlost, o * S));
    }
    const bool ok = !__any_sync(gmask<S>(), over) && qtop > -40.f && qlost < qtop - 45.f;
#pragma unroll
    for (int q = 0; q < 10; ++q) {
        df2 v = gsum_acc<S>(m[q]);
        if (gl == 0) cs.m[q] = v;
    }
    if (GRAM && rt) {
#pragma unroll
        for (int q = 0; q < 35; ++q) {
            float v = gsumf<S>(g[q]);
            if (gl == 0) cs.g[q] = v;
        }
    }
    __syncwarp(gmask<S>());
    return ok;
}

// The WIDE kernel's evaluation: the centre-out pass where it is valid, else
// the edge pass where that is, else the slow path.
template <int N, int S>
__device__ __noinline__ bool evaluate_wide(CellScratch& cs, const df2* kc, bool gram) {
    bool fast = false;
    // one copy of the centre-out pass for both kinds of evaluation (the
    // Jacobian sums behind a flag uniform over the group): half the code of
    // two instantiations (measured: instruction-fetch stalls; 44.6 against
    // 45.8 ms per step on the asymmetric sheet with the same network)
    if (centre_ok<N, S>(kc)) fast = eval_centre<N, true, S>(cs, kc, gram);
    if (!fast && edge_ok<N, S>(kc)) {
        if (gram) eval_edge<N, true, S>(cs, kc);
        else eval_edge<N, false, S>(cs, kc);
        fast = true;
    }
    if (!fast) eval_slow<N, S>(cs, kc, gram);
    return fast;
}

// non-finite or negative targets (a numeric error upstream); empty cells
// (n = 0) are not
__device__ __forceinline__ bool bad_target_pair(double t0, double tq, bool first) {
    return !isfinite(tq) || (first && !(t0 >= 0.0));
}

// One fit by its lanes of a unit: targets, fit, counters. V targets are the
// moments of f, F targets the fluid moments rescaled by n_V / n_F (listed: the
// closed-form kernel has done that). keep = false: a fit that only runs along.
template <int N, bool WIDE, int S>
__device__ __forceinline__ void fit_of_unit(CellScratch& cs, const FitArgs& a, long long cell, bool fluid, bool have,
                                            bool keep, bool listed, unsigned long long* cnt) {
    const int gl = glane<S>();
    const unsigned msk = gmask<S>();
    bool bad = false;
    if (have) {
        const double* src = fluid ? a.fluid + cell * 10 : a.vmom + cell * 20;
        const double n0 = src[0];
        double scale = 1.0;
        if (fluid && !listed) scale = n0 > 0.0 ? a.vmom[cell * 20] / n0 : 0.0;
        for (int r = 0; r < 2; ++r) {
            const int c = gl + 8 * r;
            if (c < 10) {
                const double raw = src[c];
                bad = bad || bad_target_pair(n0, raw, c == 0);
                cs.tgt[c] = fluid && !listed ? raw * scale : raw;
            }
        }
    }
    __syncwarp(msk);
    if (have && fluid && !listed)
        for (int r = 0; r < 2; ++r) {
            const int c = gl + 8 * r;
            if (c < 10) a.fluid[cell * 10 + c] = cs.tgt[c];
        }
    __syncwarp(msk);
    FitWork work = {0u, 0u, 0u, 0u, 0u};
    int iters = 0;
    double* coef = keep ? (fluid ? a.coef_f : a.coef_v) + cell * kCoefN : nullptr;
    const float* warm = (have && a.warm) ? a.warm + cell * 20 + (fluid ? 10 : 0) : nullptr;
    const int st = fit_cell<N, WIDE, S>(cs, a, have, coef, warm, &iters, work);
    bad = __any_sync(msk, bad);
    if (keep && glead<S>()) {
        if (bad && a.numeric) *reinterpret_cast<volatile int*>(a.numeric) = VL_ENUMERIC;
        if (WIDE && !listed) atomicAdd_block(&cnt[CNT_WIDE_FITS], 1ull);
        a.status[cell * 2 + (fluid ? 1 : 0)] = st;
        atomicAdd_block(&cnt[CNT_ITERS], (unsigned long long)iters);
        if (st == 1) atomicAdd_block(&cnt[CNT_FALLBACK], 1ull);
        if (st == 2) atomicAdd_block(&cnt[CNT_INVALID], 1ull);
        atomicAdd_block(&cnt[CNT_EVAL_M], (unsigned long long)work.m);
        atomicAdd_block(&cnt[CNT_EVAL_G], (unsigned long long)work.g);
        atomicAdd_block(&cnt[CNT_EVAL_SLOW], (unsigned long long)work.slow);
        atomicAdd_block(&cnt[CNT_PRECISE], (unsigned long long)work.precise);
        if (work.warm) atomicAdd_block(&cnt[CNT_WARM], (unsigned long long)work.warm);
    }
    __syncwarp(msk);
}

// A unit is the V or the F fits of four consecutive cells, whose lanes vote on
// the work (newton_loop).
//
// newton_kernel: every fit of the species, a warp per unit. CTAs per SM the
// register budget is sized for (128 threads each): four for the common kernel
// (128 registers: measured 2.5% faster than three), three for the wide kernel
// (170 registers: 13% faster per Newton iteration on the asymmetric sheet than
// four, whose budget spills the centre-out pass)
template <int N, bool WIDE>
__global__ void __launch_bounds__(128, WIDE ? 3 : 4) newton_kernel(FitArgs a) {
    __shared__ CellScratch scratch[16];
    __shared__ unsigned long long cnt[VL_NSTATS];  // CTA totals, flushed once at the end
    if (a.select) {
        // chosen on the device: this kernel runs only if it is the one wanted
        const double nmax = __longlong_as_double((long long)a.select[0]);
        const double nwide = __longlong_as_double((long long)a.select[1]);
        if ((nwide > 1e-10 * nmax) != WIDE) return;
    }
    if (threadIdx.x < VL_NSTATS) cnt[threadIdx.x] = 0ull;
    __syncthreads();
    const int slot = threadIdx.x / kG;  // 16 fits per CTA
    const long long units = 2 * ((a.ncell + 3) / 4);
    for (long long u = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); u < units; u += (long long)gridDim.x * 4) {
        const long long cell = (u >> 1) * 4 + (slot & 3);
        const bool have = cell < a.ncell;  // a group past the last cell takes part with have = false
        fit_of_unit<N, WIDE, 1>(scratch[slot], a, cell, (u & 1) != 0, have, have, false, cnt);
    }
    __syncthreads();
    if (threadIdx.x < VL_NSTATS && threadIdx.x != CNT_CLIPPED && cnt[threadIdx.x])
        atomicAdd(&a.counters[threadIdx.x], cnt[threadIdx.x]);
}

// newton_list_kernel: the units holding fits the closed-form kernel left. The
// unit's other fits run along and are not kept: a fit has the same neighbours,
// hence the same bits, whoever asked for it. The list is usually short (a few
// units in a thousand), and then what counts is the latency of one fit, a chain
// of some 80 k instructions with eight lanes per cell: up to kShortList units
// each get a CTA, a warp per cell. A longer list is fitted a warp per unit, and a
// warp takes the next one when it is done: units take uneven time (131072 fits of
// 12^3, all left: narrow ones 111 ms by equal shares, 93 now, 99 without a closed-form
// attempt; correlated ones 47, 43 and 45).
constexpr long long kShortList = 912;  // two waves of 3 CTAs per SM
template <int N, bool WIDE>
__global__ void __launch_bounds__(128, 3) newton_list_kernel(FitArgs a) {
    __shared__ CellScratch scratch[16];
    __shared__ unsigned long long cnt[VL_NSTATS];
    const long long units = (long long)*a.ntodo;
    const double nmax = __longlong_as_double((long long)a.select[0]);
    const double nwide = __longlong_as_double((long long)a.select[1]);
    // chosen on the device: this kernel runs only if it is the one wanted
    if ((nwide > 1e-10 * nmax) != WIDE) return;
    // (the counter's fits are those of a species whose targets call for the wide kernel)
    if (WIDE && blockIdx.x == 0 && threadIdx.x == 0)
        atomicAdd(&a.counters[CNT_WIDE_FITS], 2ull * (unsigned long long)a.ncell);
    const bool brief = units <= kShortList;
    if ((brief ? (long long)blockIdx.x : (long long)blockIdx.x * 4) >= units) return;
    if (threadIdx.x < VL_NSTATS) cnt[threadIdx.x] = 0ull;
    __syncthreads();
    if (brief) {
        const int c = threadIdx.x >> 5;
        for (long long k = blockIdx.x; k < units; k += gridDim.x) {
            const unsigned long long entry = a.todo[k];
            const long long cell = (long long)(entry >> 5) * 4 + c;
            const bool have = cell < a.ncell, keep = have && ((entry >> c) & 1ull) != 0;
            fit_of_unit<N, WIDE, 4>(scratch[c], a, cell, ((entry >> 4) & 1ull) != 0, have, keep, true, cnt);
        }
    } else {
        const int slot = threadIdx.x / kG, c = slot & 3;
        for (;;) {
            unsigned long long k = 0;
            if ((threadIdx.x & 31) == 0) k = atomicAdd(a.next, 1ull);
            k = __shfl_sync(0xffffffffu, k, 0);
            if (k >= (unsigned long long)units) break;
            const unsigned long long entry = a.todo[k];
            const long long cell = (long long)(entry >> 5) * 4 + c;
            const bool have = cell < a.ncell, keep = have && ((entry >> c) & 1ull) != 0;
            fit_of_unit<N, WIDE, 1>(scratch[slot], a, cell, ((entry >> 4) & 1ull) != 0, have, keep, true, cnt);
        }
    }
    __syncthreads();
    if (threadIdx.x < VL_NSTATS && threadIdx.x != CNT_CLIPPED && cnt[threadIdx.x])
        atomicAdd(&a.counters[threadIdx.x], cnt[threadIdx.x]);
}

// newton_kernel: one CTA per four units (16 fits): fits take uneven time (one
// to several Newton iterations), so the hardware's CTA scheduler, which starts
// a new CTA wherever one finishes, balances the load better than a fixed
// persistent share per CTA (grids beyond 2^31 - 1 CTAs fall back to looping).
// Where the choice is the device's (a.select) both kernels are launched and the
// one not chosen returns at once. The list's length is on the device.
template <int N>
cudaError_t launch_n(const FitArgs& a, cudaStream_t st) {
    const long long quads = (a.ncell + 3) / 4;
    if constexpr (N >= kClosedMin) {
        if (a.ntodo) {
            const long long blocks = 2 * quads < kShortList ? 2 * quads : kShortList;
            newton_list_kernel<N, true><<<(unsigned)blocks, 128, 0, st>>>(a);
            newton_list_kernel<N, false><<<(unsigned)blocks, 128, 0, st>>>(a);
            count_launch(2);
            return cudaGetLastError();
        }
    }
    long long blocks = (2 * quads + 3) / 4;
    if (blocks > 0x7FFFFFFFLL) blocks = 0x7FFFFFFFLL;
    FitArgs b = a;
    if (a.wide >= 0) b.select = nullptr;
    if (a.wide != 0) {
        newton_kernel<N, true><<<(unsigned)blocks, 128, 0, st>>>(b);
        count_launch();
    }
    if (a.wide != 1) {
        newton_kernel<N, false><<<(unsigned)blocks, 128, 0, st>>>(b);
        count_launch();
    }
    return cudaGetLastError();
}

}  // namespace

}  // namespace vl

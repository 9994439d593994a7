// Fused spatial PFC sweeps in FP32, x then y (paper Sec. 2.1, the directional
// splitting of the Vlasov step; Sec. 3.3, reflecting walls), streamed along y:
// the pass pfc_advect_xy makes (out of place, f crosses HBM once).
//
// A CTA owns a strip of 8 cells per warp in x (up to four warps), 32
// contiguous velocity columns and a run of rows, and marches through the rows.
// A row of the strip with its x halo comes into a ring of shared-memory slots
// by TMA (centre, left and right halo as three boxes, so periodic images are
// ordinary boxes); each thread reads the window of its 8 cells in its column,
// forms their x-swept values in registers and feeds them to 8 running y sweeps
// (three or four values of state per cell), which emit one row of output per
// row of input. Mirror rows beyond a wall are read straight from global memory.
//
// Why: the tile form of the pass (16 x 16 cells, x-swept rows in shared memory)
// swept 20 rows per 16 in x, formed 10 fluxes per 8 outputs in y, passed every
// value through shared memory once more and stood at block-wide barriers
// between its phases: 68 instructions per value, issue- and barrier-bound. Here
// an x flux is formed 9/8 times, a y flux once, and warps only meet at the
// ring: 34 instructions per value, and the pass is bound by HBM (5.7 TB/s of
// the 6.8 a plain copy reaches) with the first and last rows of the CTAs' runs
// on top. Consecutive CTAs take the column chunks of the same cells, so that
// whole velocity blocks are read from HBM together.
// Measured, before -> after: 256 x 128 x 16^3 372 -> 187 us, 512 x 256 x 16^3
// 1274 -> 705, 128 x 64 x 20^3 (periodic) 228 -> 104; off the 16-cell tiles,
// 136 x 72 x 12^3 145 -> 41.
//
// The update of a cell is out = (f - phi) + phi', phi = alpha x its own flux
// and phi' that of the neighbour upwind, x = f + P U + Q D in the
// direction-independent form (U = min(f_{+} - f, 2f), D = max(f - f_{-}, -2f);
// (P, Q) = (A, B), or (-B, -A) for a negative displacement). A thread's
// direction selects which of two neighbouring cells gives f - phi and which phi'.
//
// FRAME: the two products are added in the order of the line's own direction
// and the multiplications by alpha are fused with the additions, the roundings
// of pfc_space_xy_kernel; without it, those of the FP64 tile kernel.
#include <cuda.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "f32x2.cuh"
#include "kernels.cuh"
#include "tc.cuh"

namespace vl {

namespace {

constexpr int kCols = 32;       // velocity columns of a CTA: one per lane
constexpr int kCells = 8;       // cells along x per thread
constexpr int kRing = 6;        // rows in flight (4: the same within 1%)
constexpr int kMaxWarps = 4;
constexpr int kMinRows = 4;
constexpr int kMaxHalo = 8;
constexpr uint32_t kPolls = 1u << 20;  // bound of a wait on a row (far beyond any real copy)

// displacement constants of one velocity index along an axis
struct Step {
    float alpha, P, Q;
    int s, fwd;
};
struct Tables {
    Step x[24], y[24];
};

struct MarchArgs {
    const void* f_in;
    void* f_out;
    int nx, ny, wall, hx, hy, rows;  // rows of a CTA's run
    unsigned long long* counters;
};

__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(tc::smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tc::smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void load_box(void* dst, const CUtensorMap* map, int c0, int c1, int c2, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(tc::smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(tc::smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ int wrap(int i, int n) {
    i %= n;
    return i < 0 ? i + n : i;
}

// U and D of a cell from its value and the differences above (a) and below
// (b); returns f + P U + Q D
template <bool FRAME>
__device__ __forceinline__ float limited(float f, float a, float b, float P, float Q, bool fwd) {
    const float f2 = __fadd_rn(f, f), U = fminf(a, f2), D = fmaxf(b, -f2);
    if (FRAME) return fmaf(fwd ? Q : P, fwd ? D : U, fmaf(fwd ? P : Q, fwd ? U : D, f));
    return fmaf(Q, D, fmaf(P, U, f));
}

}  // namespace

// CTAs of kMaxWarps per SM the registers are limited to, and the rows per CTA
// counted with (FRAME 5: 136 x 72 x 12^3 41.4 us, 4: 45.4; else 4: 128 x 64 x
// 16^3 59.8 us, 5: 63.6)
template <bool FRAME>
constexpr int kCtas = FRAME ? 5 : 4;

template <int N, bool FRAME>
__global__ void __launch_bounds__(32 * kMaxWarps, kCtas<FRAME>)
    pfc_space_march_kernel(const __grid_constant__ CUtensorMap centre, const __grid_constant__ CUtensorMap halo,
                           const __grid_constant__ Tables tab, MarchArgs a) {
    constexpr int V = N * N * N;
    constexpr uint32_t kBox = kCols * sizeof(float);  // bytes of a cell's columns
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint64_t* const full = reinterpret_cast<uint64_t*>(smem_raw);
    uint64_t* const empty = full + kRing;
    const int warps = blockDim.x >> 5, strip = warps * kCells, hx = a.hx, nx = a.nx, ny = a.ny;
    const int slot_cells = strip + 2 * hx;
    float* const ring = reinterpret_cast<float*>(smem_raw + 128);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the last strip of a row ends with the row and may repeat cells of the one before
    const int chunk = blockIdx.x, x0 = min((int)blockIdx.y * strip, nx - strip);
    const int ya = blockIdx.z * a.rows, yb = min(ny, ya + a.rows);
    if (threadIdx.x == 0)
        for (int q = 0; q < kRing; ++q) {
            tc::mbar_init(&full[q], 1);
            tc::mbar_init(&empty[q], (uint32_t)warps);
        }
    __syncthreads();

    // rows of the march: ya - hy .. yb - 1 + hy; those outside a walled domain
    // are mirror rows and do not go through the ring
    const int r0 = ya - a.hy, r1 = yb + a.hy;
    const int rf = a.wall ? max(r0, 0) : r0, rl = a.wall ? min(r1, ny) : r1;  // ring rows [rf, rl)
    const int nring = rl - rf;
    const uint32_t bytes = (uint32_t)slot_cells * kBox;
    const int xl = x0 == 0 ? nx - hx : x0 - hx, xr = x0 + strip == nx ? 0 : x0 + strip;  // hx <= 8 <= x0, nx
    auto issue = [&](int q) {  // one thread
        const int slot = q % kRing, row = wrap(rf + q, ny);
        float* const dst = ring + (size_t)slot * slot_cells * kCols;
        expect_tx(&full[slot], bytes);
        load_box(dst + hx * kCols, &centre, chunk * kCols, x0, row, &full[slot]);
        load_box(dst, &halo, chunk * kCols, xl, row, &full[slot]);
        load_box(dst + (hx + strip) * kCols, &halo, chunk * kCols, xr, row, &full[slot]);
    };
    int issued = 0;
    if (threadIdx.x == 0)
        for (; issued < kRing && issued < nring; ++issued) issue(issued);

    const int vi = chunk * kCols + lane;
    const int ix = vi % N, iy = (vi / N) % N, iz = vi / (N * N);
    const Step sx = tab.x[ix], sy = tab.y[iy];
    const bool fx = sx.fwd != 0, fy = sy.fwd != 0;
    // window of the 9 fluxes of 8 outputs: cells xw + off .. + 10
    const int xw = x0 + warp * kCells, off = fx ? -sx.s - 2 : sx.s - 1;
    const float* const src0 = ring + (hx + warp * kCells + off) * kCols + lane;
    const float* __restrict__ fin = reinterpret_cast<const float*>(a.f_in);
    // the step that reads row r emits row r + oro of this column
    const int oro = fy ? sy.s - 1 : -2 - sy.s;
    float* out = reinterpret_cast<float*>(a.f_out) + ((long long)(r0 + oro) * nx + xw) * V + vi;
    const long long ostride = (long long)nx * V;
    bool ok = true;

    // newest value, its difference below, and the kept terms of the cell below
    // (FRAME: f + P U + Q D and f - phi; else the one of phi and f - phi that
    // the next row needs, in h)
    float f[kCells], ap[kCells], h[kCells], h2[FRAME ? kCells : 1];
#pragma unroll
    for (int k = 0; k < kCells; ++k) f[k] = ap[k] = h[k] = 0.0f;
#pragma unroll
    for (int k = 0; k < (FRAME ? kCells : 1); ++k) h2[k] = 0.0f;
#pragma unroll 1
    for (int r = r0; r < r1; ++r, out += ostride) {
        float v[kCells + 3];
        if (a.wall && (r < 0 || r >= ny)) {
            const int row = r < 0 ? -1 - r : 2 * ny - 1 - r;
            const float* p = fin + (long long)row * nx * V + (iz * N + (N - 1 - iy)) * N + ix;
#pragma unroll
            for (int i = 0; i < kCells + 3; ++i) v[i] = __ldg(p + (long long)wrap(xw + off + i, nx) * V);
        } else {
            const int q = r - rf, slot = q % kRing;
            const uint32_t ph = (uint32_t)(q / kRing) & 1u;
            ok = tc::mbar_wait(&full[slot], ph, kPolls) && ok;
            const float* src = src0 + (size_t)slot * slot_cells * kCols;
#pragma unroll
            for (int i = 0; i < kCells + 3; ++i) v[i] = src[i * kCols];
            __syncwarp();
            if (lane == 0) arrive(&empty[slot]);
            // refill the slot of the row before this one, once every warp has
            // read it
            if (threadIdx.x == 0 && q > 0 && q - 1 + kRing < nring && ok) {
                const int b = (q - 1) % kRing;
                ok = tc::mbar_wait(&empty[b], (uint32_t)((q - 1) / kRing) & 1u, kPolls);
                if (ok) {
                    issue(q - 1 + kRing);
                    ++issued;
                }
            }
        }
        if (!__all_sync(0xffffffffu, ok)) break;
        // x: nine fluxes, eight outputs
        float n[kCells];
        {
            float hk = 0.0f, xk = 0.0f, tk = 0.0f;
#pragma unroll
            for (int i = 0; i <= kCells; ++i) {
                const float w = v[i + 1];
                const float x = limited<FRAME>(w, v[i + 2] - w, w - v[i], sx.P, sx.Q, fx);
                if (FRAME) {
                    const float t = fmaf(-sx.alpha, x, w);
                    if (i > 0) n[i - 1] = fmaf(sx.alpha, fx ? xk : x, fx ? t : tk);
                    xk = x;
                    tk = t;
                } else {
                    const float phi = __fmul_rn(sx.alpha, x), t = __fsub_rn(w, phi);
                    if (i > 0) n[i - 1] = __fadd_rn(fx ? t : phi, hk);
                    hk = fx ? phi : t;
                }
            }
        }
        // y: one flux per cell, two cells at a time
        const bool emit = r + oro >= ya && r + oro < yb;
        float o[kCells];
        const float2 al = x2::splat(sy.alpha), P = x2::splat(sy.P), Q = x2::splat(sy.Q);
#pragma unroll
        for (int k = 0; k < kCells; k += 2) {
            const float2 fk = make_float2(f[k], f[k + 1]), nk = make_float2(n[k], n[k + 1]);
            const float2 d = x2::sub(nk, fk), f2 = x2::add(fk, fk);
            const float2 U = make_float2(fminf(d.x, f2.x), fminf(d.y, f2.y));
            const float2 D = make_float2(fmaxf(ap[k], -f2.x), fmaxf(ap[k + 1], -f2.y));
            float2 e;
            if (FRAME) {
                const float2 t1 = make_float2(fy ? U.x : D.x, fy ? U.y : D.y);
                const float2 t2 = make_float2(fy ? D.x : U.x, fy ? D.y : U.y);
                const float2 x = x2::fma(fy ? Q : P, t2, x2::fma(fy ? P : Q, t1, fk));
                const float2 t = x2::fma(x2::neg(al), x, fk);
                e = x2::fma(al, make_float2(fy ? h[k] : x.x, fy ? h[k + 1] : x.y),
                            make_float2(fy ? t.x : h2[k], fy ? t.y : h2[k + 1]));
                h[k] = x.x;
                h[k + 1] = x.y;
                h2[k] = t.x;
                h2[k + 1] = t.y;
            } else {
                const float2 x = x2::fma(Q, D, x2::fma(P, U, fk));
                const float2 phi = x2::mul(al, x), t = x2::sub(fk, phi);
                e = x2::add(make_float2(fy ? t.x : phi.x, fy ? t.y : phi.y), make_float2(h[k], h[k + 1]));
                h[k] = fy ? phi.x : t.x;
                h[k + 1] = fy ? phi.y : t.y;
            }
            o[k] = e.x;
            o[k + 1] = e.y;
            ap[k] = d.x;
            ap[k + 1] = d.y;
        }
#pragma unroll
        for (int k = 0; k < kCells; ++k) f[k] = n[k];
        if (emit) {
#pragma unroll
            for (int k = 0; k < kCells; ++k) out[(long long)k * V] = o[k];
        }
    }
    // A row that did not come in time: count it, and let the copies still in
    // flight land before the shared memory goes away (bounded as well).
    if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) {
            atomicAdd(&a.counters[CNT_COPY_TIMEOUT], 1ull);
            for (int q = max(0, issued - kRing); q < issued; ++q)
                tc::mbar_wait(&full[q % kRing], (uint32_t)(q / kRing) & 1u, kPolls);
        }
        __syncthreads();
    }
}

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return (EncodeTiledFn) nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// f_in as a 3D tensor (velocity index, x, y), boxes of `cells` cells of a row
bool box_map(const SpaceXYArgs& a, int cells, CUtensorMap* m) {
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)a.V, (cuuint64_t)a.nx, (cuuint64_t)a.ny};
    const cuuint64_t strides[2] = {(cuuint64_t)a.V * 4, (cuuint64_t)a.V * 4 * a.nx};
    const cuuint32_t box[3] = {(cuuint32_t)kCols, (cuuint32_t)cells, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(a.f_in), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// displacement constants in FP64, reduced modulo the line length on periodic
// lines, as the single-axis sweeps form them
Step step_of(double vmin, double dv, double dt_over_h, int i, int n, bool wall) {
    const double c = (vmin + (i + 0.5) * dv) * dt_over_h;
    Step r;
    r.fwd = c >= 0.0;
    double ca = r.fwd ? c : -c;
    if (!wall) ca = std::fmod(ca, (double)n);
    if (!(ca <= (double)n)) ca = (double)n;
    r.s = (int)std::floor(ca);
    r.alpha = (float)(ca - r.s);
    const float A = (1.0f - r.alpha) * (2.0f - r.alpha) / 6.0f, B = (1.0f - r.alpha) * (1.0f + r.alpha) / 6.0f;
    r.P = r.fwd ? A : -B;
    r.Q = r.fwd ? B : -A;
    return r;
}

template <int N, bool FRAME>
cudaError_t launch_n(const SpaceXYArgs& s, cudaStream_t st) {
    // Warps of a strip: the fewest strips of 8 w cells plus the cost of their
    // halos (a halo cell is copied but not swept, hence half)
    const int groups = s.nx / kCells;
    int warps = 1;
    long long best = -1;
    for (int w = 1; w <= kMaxWarps && w <= groups; ++w) {
        const long long cost = (long long)((groups + w - 1) / w) * (kCells * w + s.hx);
        if (best < 0 || cost <= best) best = cost, warps = w;
    }
    const int strip = warps * kCells, strips = (groups + warps - 1) / warps;
    CUtensorMap centre, halo;
    if (!box_map(s, strip, &centre) || !box_map(s, s.hx, &halo)) return cudaErrorNotSupported;
    Tables tab;
    for (int i = 0; i < N; ++i) {
        tab.x[i] = step_of(s.vminx, s.dvx, s.cx, i, s.nx, false);
        tab.y[i] = step_of(s.vminy, s.dvy, s.cy, i, s.ny, s.wall != 0);
    }
    MarchArgs a;
    a.f_in = s.f_in;
    a.f_out = s.f_out;
    a.nx = s.nx;
    a.ny = s.ny;
    a.wall = s.wall;
    a.hx = s.hx;
    a.hy = s.hy;
    a.counters = s.counters;
    const size_t smem = 128 + (size_t)kRing * (strip + 2 * s.hx) * kCols * sizeof(float);
    auto* k = pfc_space_march_kernel<N, FRAME>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // Runs of rows: a run of n rows costs n + 2 hy + a start of about 8 rows;
    // the CTAs share the chip's slots, and the last ones leave it half empty
    // for half a run on average. Few runs repeat few halo rows, many fill the
    // chip on small grids.
    const double slots = 152.0 * kCtas<FRAME> * kMaxWarps / warps, cols = (double)(s.V / kCols) * strips;
    double least = 0.0;
    a.rows = s.ny;
    for (int runs = 1; runs <= std::max(1, s.ny / kMinRows) && runs <= 65535; ++runs) {
        const int rows = (s.ny + runs - 1) / runs;
        const double cost = (rows + 2 * s.hy + 8) * (std::max(1.0, cols * runs / slots) + 0.5);
        if (runs == 1 || cost < least) least = cost, a.rows = rows;
    }
    const dim3 grid((unsigned)(s.V / kCols), (unsigned)strips, (unsigned)((s.ny + a.rows - 1) / a.rows));
    k<<<grid, 32 * warps, smem, st>>>(centre, halo, tab, a);
    count_launch();
    return cudaGetLastError();
}

template <bool FRAME>
cudaError_t launch_t(const SpaceXYArgs& a, cudaStream_t st) {
    switch (a.nvx) {
        case 8: return launch_n<8, FRAME>(a, st);
        case 12: return launch_n<12, FRAME>(a, st);
        case 16: return launch_n<16, FRAME>(a, st);
        case 20: return launch_n<20, FRAME>(a, st);
        case 24: return launch_n<24, FRAME>(a, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace

// Can the streamed pass take the call? Rows of whole 8-cell groups (the halo
// boxes then never cross the grid's end), TMA's 16-byte alignment of f_in, and
// halos that fit the ring and, at a wall, the domain
bool march_fits(const SpaceXYArgs& a) {
    return a.nx % kCells == 0 && a.nx / kCells <= 65535 && a.hx <= kMaxHalo && a.hy <= kMaxHalo && a.hy <= a.ny &&
           a.V % kCols == 0 && a.V < (1LL << 31) && reinterpret_cast<uintptr_t>(a.f_in) % 16 == 0 &&
           a.counters != nullptr;
}

// Small grids of one or two groups of cells in x with long shifts, and 8 x 8 cells: a
// march starts with a ring to set up and 2 hy rows that emit nothing, and a few
// CTAs have little to hide them behind. us, march / tiles: 8 x 8 cells of 12^3 8.3 /
// 6.3 at half a cell, 12.5 / 8.4 at 6; 16 x 16 of 16^3 10.4 / 10.4 at 2 cells, 14.5 / 10.4
// at 4, 16.5 / 12.4 at 6; of 24^3 16.6 / 20.7 at 1, 26.7 / 22.7 at 4; 8 x 128 of 12^3 16.6 /
// 18.6 at 3, 20.7 / 18.6 at 5. Wider than high it is the other way: 64 x 8 of 12^3 14.5 /
// 18.6 at 6.
bool march_late(const SpaceXYArgs& a, long long ntiles) {
    if (a.nx > 16 || a.ny < a.nx) return false;
    if (ntiles <= 128 && (a.hx >= 5 || a.nx * a.ny <= 64)) return true;
    return ntiles <= 448 && a.hx >= 6;
}

cudaError_t launch_pfc_space_march(const SpaceXYArgs& a, bool frame, cudaStream_t st) {
    return frame ? launch_t<true>(a, st) : launch_t<false>(a, st);
}

}  // namespace vl

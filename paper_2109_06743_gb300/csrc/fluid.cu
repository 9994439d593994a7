// Ten-moment fluid step (paper Sec. 2.1 equations with the third moment from
// f, Sec. 2.2; CWENO of Kurganov and Levy 2000 and SSP-RK3 of Shu and Osher
// 1988, cited in Sec. 2.1). With FluidArgs.closure the same kernel runs the
// stand-alone fluid model of Sec. 2.3 (gradient heat-flux closure).
//
// Per species the state is U = (n, nu_a, E2_ab), E2 = P/m = int v v f. The
// equations divided by m read
//   dn/dt     + d_k nu_k    = 0
//   dnu_a/dt  + d_k E2_ka   = (q/m) (n E_a + (nu x B)_a)
//   dE2_ab/dt + d_k E3_kab  = (q/m) (nu_a E_b + nu_b E_a + C_ab + C_ba),
// C_ab = ((row a of E2) x B)_b, E3 = int v v v f taken from the Vlasov solver
// and reconstructed with the same CWENO polynomials as U. Fluxes are the
// central-upwind (local Lax-Friedrichs) flux with the ten-moment wave speed
// |u_d| + sqrt(3 Theta_dd) of the two neighbouring cells. The state stays in
// FP64; the reconstruction, fluxes and sources (the right-hand side L) are
// computed in R = double in FP64 mode and in R = float in FP32 mode (on GB300
// the FP64 pipe runs at ~1/58 of the FP32 pipe), and the Runge-Kutta
// combination U0 + dt L is formed in FP64.
//
// 2D3V: one CTA per tile of cells and stage (fluid_tile_kernel); 1D1V: one
// warp per 6 cells.
#include "common.cuh"
#include "kernels.cuh"

namespace vl {

__device__ __forceinline__ int s2(int a, int b) {
    return a == 0 ? b : (a == 1 ? (b == 0 ? 1 : b + 2) : (b == 0 ? 2 : (b == 1 ? 4 : 5)));
}

// index of the symmetric triple in xxx,xxy,xxz,xyy,xyz,xzz,yyy,yyz,yzz,zzz
__device__ __forceinline__ int s3(int a, int b, int c) {
    int x = (a == 0) + (b == 0) + (c == 0), y = (a == 1) + (b == 1) + (c == 1);
    // by number of x, then y
    if (x == 3) return 0;
    if (x == 2) return y == 1 ? 1 : 2;
    if (x == 1) return y == 2 ? 3 : (y == 1 ? 4 : 5);
    return y == 3 ? 6 : (y == 2 ? 7 : (y == 1 ? 8 : 9));
}

template <typename R>
__device__ __forceinline__ void cweno3_point(R um, R u0, R up, R* left, R* right) {
    const R eps = R(1e-6);
    R il = (u0 - um) * (u0 - um), ir = (up - u0) * (up - u0);
    R d2 = up - R(2) * u0 + um, d1 = up - um;
    R ic = (R(13) / R(3)) * d2 * d2 + R(0.25) * d1 * d1;
    R al = R(0.25) / ((eps + il) * (eps + il));
    R ar = R(0.25) / ((eps + ir) * (eps + ir));
    R ac = R(0.5) / ((eps + ic) * (eps + ic));
    R inv = R(1) / (al + ar + ac);
    R wl = al * inv, wr = ar * inv, wc = ac * inv;
    // values at xi = -1/2 and +1/2 of the linear left/right and the central
    // polynomial P_C = (P_opt - P_L/4 - P_R/4) / (1/2)
    R base = u0 - d2 / R(24) + R(0.125) * d2;
    R optl = base - R(0.25) * d1, optr = base + R(0.25) * d1;
    R ll = u0 - R(0.5) * (u0 - um), lr = u0 + R(0.5) * (u0 - um);
    R rl = u0 - R(0.5) * (up - u0), rr = u0 + R(0.5) * (up - u0);
    R cl = R(2) * optl - R(0.5) * ll - R(0.5) * rl;
    R cr = R(2) * optr - R(0.5) * lr - R(0.5) * rr;
    *left = wl * ll + wr * rl + wc * cl;
    *right = wl * lr + wr * rr + wc * cr;
}

// index of the flux of component k in direction dir: a state component (n:
// nu_d; nu_a: E2_da) or 10 + a third moment (E2_ab: E3_dab)
static __constant__ signed char kFluxVar[2][10] = {{1, 4, 5, 6, 10, 11, 12, 13, 14, 15},
                                                   {2, 5, 7, 8, 11, 13, 14, 16, 17, 18}};
// sign of a component under y -> -y (v_y -> -v_y): the state n nux nuy nuz xx
// xy xz yy yz zz, then the third moments xxx xxy xxz xyy xyz xzz yyy yyz yzz zzz
static __constant__ signed char kParity[20] = {1, 1, -1, 1, 1, -1, 1, 1, -1, 1, 1, -1, 1, 1, -1, 1, -1, 1, -1, 1};

// Gradient-closure model (Sec. 2.3): with zero heat flux the third moment
// is that of the Maxwellian with the state's n, u and E2,
//   E3_kab = u_k E2_ab + u_a E2_kb + u_b E2_ka - 2 n u_k u_a u_b,
// evaluated on the reconstructed interface states.
template <typename R>
__device__ __forceinline__ void closure_e3(const R* s, R* e3) {
    const R n = s[0];
    if (!(n > R(0))) {
#pragma unroll
        for (int k = 0; k < 10; ++k) e3[k] = R(0);
        return;
    }
    const R inv = R(1) / n;
    const R v[3] = {s[1] * inv, s[2] * inv, s[3] * inv};
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = a; b < 3; ++b)
#pragma unroll
            for (int k = b; k < 3; ++k)
                e3[s3(a, b, k)] = v[k] * s[4 + s2(a, b)] + v[a] * s[4 + s2(k, b)] + v[b] * s[4 + s2(k, a)] -
                                  R(2) * n * v[k] * v[a] * v[b];
}

// One RK stage over a tile of TX x TY cells, in shared-memory phases:
//   1. the stage input and the weighted third moments of the tile and two
//      halo cells per side (periodic images, mirror cells beyond a wall),
//      converted to R once;
//   2. the reconstruction of every component in every cell a flux of the tile
//      reads, once per direction (left and right interface values), and the
//      wave speeds; with CLOSURE the third moments of the interface states;
//   3. the flux differences, one (cell, component) per thread;
//   4. the sources, one thread per cell (with CLOSURE also the heat flux from
//      theta of the tile and its neighbours);
//   5. the Runge-Kutta combination, one (cell, component) per thread, so that
//      the FP64 state is read and written in contiguous runs.
// What bounds it: the reconstruction's arithmetic (four divisions a point).
// One thread per cell formed every point three times (for its own and both
// neighbours' fluxes) in one serial chain of about 20 k instructions, 60 us
// per stage however small the grid; here a point is formed 1.25-1.4 times and
// 256 threads share a tile. Measured (GB300): one FP32 step (three stages) of
// 128 x 64 cells 180 -> 37 us; the closure model's step of 64 x 64 cells in
// FP64, both species and fields, 1257 -> 330 us; same bits. Shapes: tile_shape
// (8 x 8 forms 1.25 points per point used, 8 x 4 1.38, 32 x 1 2.03).
constexpr int kTileThreads = 256;
template <typename R, int TX, int TY>
struct FluidTile {
    static constexpr int HX = TX + 4, HY = TY + 4;          // with halo
    static constexpr int PX = (TX + 2) * TY, PY = TX * (TY + 2);  // reconstructed points per direction
    R s[20][HX * HY];
    R x[20][2][PX], y[20][2][PY];  // [component][left, right interface value][point]
    R wx[PX], wy[PY];              // wave speeds
    R l[10][TX * TY];
};

template <typename R, bool CLOSURE, int TX, int TY>
__global__ void __launch_bounds__(kTileThreads) fluid_tile_kernel(FluidArgs a) {
    typedef FluidTile<R, TX, TY> Tile;
    constexpr int HX = Tile::HX, HY = Tile::HY, PX = Tile::PX, PY = Tile::PY, NV = CLOSURE ? 10 : 20;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Tile& t = *reinterpret_cast<Tile*>(smem_raw);
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int nx = a.nx, ny = a.ny;
    const bool use0 = a.wq0 != 0.0, use1 = a.wq1 != 0.0;
    const int tid = threadIdx.x;
    for (int e = tid; e < HX * HY * 10; e += kTileThreads) {
        const int k = e % 10, p = e / 10, lx = p % HX, ly = p / HX;
        if ((lx < 2 || lx >= TX + 2) && (ly < 2 || ly >= TY + 2)) continue;  // corners are not read
        int ix = x0 + lx - 2, iy = y0 + ly - 2;
        ix %= nx;
        if (ix < 0) ix += nx;
        bool mir = false;
        if (iy < 0 || iy >= ny) {
            if (a.bc_y == 1) {
                iy = iy < 0 ? -1 - iy : 2 * ny - 1 - iy;
                iy = iy < 0 ? 0 : iy;  // only rows beyond the last tile's own halo
                mir = true;
            } else {
                iy %= ny;
                if (iy < 0) iy += ny;
            }
        }
        const long long id = (long long)iy * nx + ix;
        R v = (R)a.Us[id * 10 + k];
        t.s[k][p] = mir ? v * (R)kParity[k] : v;
        if (!CLOSURE) {
            // Q = wq0 q0 + wq1 q1 (the weights are 0, 1/2 or 1, exact in R)
            v = R(0);
            if (use0) v += (R)a.wq0 * (R)a.q0[id * 20 + 10 + k];
            if (use1) v += (R)a.wq1 * (R)a.q1[id * 20 + 10 + k];
            t.s[10 + k][p] = mir ? v * (R)kParity[10 + k] : v;
        }
    }
    __syncthreads();
    for (int e = tid; e < NV * PX; e += kTileThreads) {
        const int k = e / PX, p = e % PX, c = (p / (TX + 2) + 2) * HX + p % (TX + 2) + 1;
        const R* u = t.s[k] + c;
        cweno3_point<R>(u[-1], u[0], u[1], &t.x[k][0][p], &t.x[k][1][p]);
    }
    for (int e = tid; e < NV * PY; e += kTileThreads) {
        const int k = e / PY, p = e % PY, c = (p / TX + 1) * HX + p % TX + 2;
        const R* u = t.s[k] + c;
        cweno3_point<R>(u[-HX], u[0], u[HX], &t.y[k][0][p], &t.y[k][1][p]);
    }
    // wave speeds |u_d| + sqrt(3 Theta_dd) from the cell averages
    for (int e = tid; e < PX + PY; e += kTileThreads) {
        const int dir = e < PX ? 0 : 1, p = dir ? e - PX : e;
        const int c = dir ? (p / TX + 1) * HX + p % TX + 2 : (p / (TX + 2) + 2) * HX + p % (TX + 2) + 1;
        const R n = t.s[0][c];
        R w = R(0);
        if (n > R(0)) {
            const R ud = t.s[1 + dir][c] / n;
            R th = t.s[dir ? 7 : 4][c] / n - ud * ud;
            if (th < R(0)) th = R(0);
            w = fabs(ud) + sqrt(R(3) * th);
        }
        if (dir) t.wy[p] = w;
        else t.wx[p] = w;
    }
    __syncthreads();
    if (CLOSURE) {
        for (int e = tid; e < 2 * (PX + PY); e += kTileThreads) {
            const int side = e & 1, q = e >> 1, dir = q < PX ? 0 : 1, p = dir ? q - PX : q;
            R s[10], e3[10];
#pragma unroll
            for (int k = 0; k < 10; ++k) s[k] = dir ? t.y[k][side][p] : t.x[k][side][p];
            closure_e3<R>(s, e3);
#pragma unroll
            for (int k = 0; k < 10; ++k) {
                if (dir) t.y[10 + k][side][p] = e3[k];
                else t.x[10 + k][side][p] = e3[k];
            }
        }
        __syncthreads();
    }
    // Walls: the interface beyond the last row is the wall itself (mirror
    // ghosts already give its flux).
    const R invhx = (R)a.invdx, invhy = (R)a.invdy;
    for (int e = tid; e < 10 * TX * TY; e += kTileThreads) {
        const int k = e / (TX * TY), cell = e % (TX * TY), cx = cell % TX, cy = cell / TX;
        R L = R(0);
#pragma unroll
        for (int dir = 0; dir < 2; ++dir) {
            const int p = dir ? (cy + 1) * TX + cx : cy * (TX + 2) + cx + 1, st = dir ? TX : 1;
            const R* ul = dir ? t.y[k][0] : t.x[k][0];
            const R* ur = dir ? t.y[k][1] : t.x[k][1];
            const int f = kFluxVar[dir][k];
            const R* fl = dir ? t.y[f][0] : t.x[f][0];
            const R* fr = dir ? t.y[f][1] : t.x[f][1];
            const R* ws = dir ? t.wy : t.wx;
            const R sm = fmax(ws[p - st], ws[p]), sp = fmax(ws[p], ws[p + st]);
            const R Hm = R(0.5) * (fr[p - st] + fl[p]) - R(0.5) * sm * (ul[p] - ur[p - st]);
            const R Hp = R(0.5) * (fr[p] + fl[p + st]) - R(0.5) * sp * (ul[p + st] - ur[p]);
            L -= (Hp - Hm) * (dir ? invhy : invhx);
        }
        t.l[k][cell] = L;
    }
    __syncthreads();
    for (int cell = tid; cell < TX * TY; cell += kTileThreads) {
        const int cx = cell % TX, cy = cell / TX, ix = x0 + cx, iy = y0 + cy;
        if (ix >= nx || iy >= ny) continue;
        const int c = (cy + 2) * HX + cx + 2;
        R u[10], eb[6], L[10];
#pragma unroll
        for (int k = 0; k < 10; ++k) {
            u[k] = t.s[k][c];
            L[k] = t.l[k][cell];
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) eb[k] = (R)a.eb[((long long)iy * nx + ix) * 6 + k];
        const R qm = (R)a.qm;
        const R* E = eb;
        const R* B = eb + 3;
        const R* nu = u + 1;
        L[1] += qm * (u[0] * E[0] + nu[1] * B[2] - nu[2] * B[1]);
        L[2] += qm * (u[0] * E[1] + nu[2] * B[0] - nu[0] * B[2]);
        L[3] += qm * (u[0] * E[2] + nu[0] * B[1] - nu[1] * B[0]);
        R M[3][3];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = 0; q < 3; ++q) M[p][q] = u[4 + s2(p, q)];
        R C[3][3];
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            C[p][0] = M[p][1] * B[2] - M[p][2] * B[1];
            C[p][1] = M[p][2] * B[0] - M[p][0] * B[2];
            C[p][2] = M[p][0] * B[1] - M[p][1] * B[0];
        }
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = p; q < 3; ++q) L[4 + s2(p, q)] += qm * (nu[p] * E[q] + nu[q] * E[p] + C[p][q] + C[q][p]);
        if (CLOSURE) {
            // heat flux of the closure: -(1/m) div Q = chi_k0 n v_t lap theta,
            // theta = E2 / n - u u, v_t = sqrt(tr(theta) / 3), five-point Laplacian
            R th[5][6];
            const int at[5] = {c, c - 1, c + 1, c - HX, c + HX};
#pragma unroll
            for (int o = 0; o < 5; ++o) {
                const R n = t.s[0][at[o]];
                const R inv = n > R(0) ? R(1) / n : R(0);
#pragma unroll
                for (int p = 0; p < 3; ++p)
#pragma unroll
                    for (int q = p; q < 3; ++q)
                        th[o][s2(p, q)] =
                            t.s[4 + s2(p, q)][at[o]] * inv - (t.s[1 + p][at[o]] * inv) * (t.s[1 + q][at[o]] * inv);
            }
            const R tr = th[0][0] + th[0][3] + th[0][5];
            const R vt = sqrt(tr > R(0) ? tr / R(3) : R(0));
            const R coef = (R)a.chi_k0 * u[0] * vt;
            const R ix2 = (R)a.invdx2, iy2 = (R)a.invdy2;
#pragma unroll
            for (int k = 0; k < 6; ++k)
                L[4 + k] += coef * ((th[2][k] - R(2) * th[0][k] + th[1][k]) * ix2 +
                                    (th[4][k] - R(2) * th[0][k] + th[3][k]) * iy2);
        }
#pragma unroll
        for (int k = 0; k < 10; ++k) t.l[k][cell] = L[k];
    }
    __syncthreads();
    for (int e = tid; e < 10 * TX * TY; e += kTileThreads) {
        const int k = e % 10, cell = e / 10, ix = x0 + cell % TX, iy = y0 + cell / TX;
        if (ix >= nx || iy >= ny) continue;
        const long long o = ((long long)iy * nx + ix) * 10 + k;
        const double us = a.Us[o];
        const double u0 = a.a0 != 0.0 ? a.U0[o] : 0.0;
        a.Uout[o] = a.a0 * u0 + a.a1 * (us + a.dt * (double)t.l[k][cell]);
    }
}

// 1D1V (three components n, nu, E2; periodic): one warp per 6 cells and stage.
// Four fields (n, nu, E2 and the third moment) are reconstructed in the 8 cells
// the 6 cells' fluxes read: one point a lane, each formed once. With a thread per
// cell every lane went through 18 points, some 2700 FP64 instructions in a row (39
// us a stage for 64 cells, 9 now).
constexpr int kCells1d = 6;
template <typename R>
__global__ void __launch_bounds__(32) fluid1d_stage_kernel(FluidArgs a) {
    constexpr int T = kCells1d;
    __shared__ R s[4][T + 4];              // n, nu, E2, E3 of cells x0 - 2 .. x0 + T + 1
    __shared__ R xl[4][T + 2], xr[4][T + 2], ws[T + 2];  // of cells x0 - 1 .. x0 + T
    const int lane = threadIdx.x, nx = a.nx, x0 = blockIdx.x * T;
    for (int e = lane; e < 4 * (T + 4); e += 32) {
        const int k = e / (T + 4);
        int c = (x0 + e % (T + 4) - 2) % nx;
        if (c < 0) c += nx;
        R v = R(0);
        if (k < 3) {
            v = (R)a.Us[(long long)c * 3 + k];
        } else {
            if (a.wq0 != 0.0) v += (R)a.wq0 * (R)a.q0[(long long)c * 4 + 3];
            if (a.wq1 != 0.0) v += (R)a.wq1 * (R)a.q1[(long long)c * 4 + 3];
        }
        s[k][e % (T + 4)] = v;
    }
    __syncwarp();
    {
        const int k = lane >> 3, p = lane & 7;
        cweno3_point<R>(s[k][p], s[k][p + 1], s[k][p + 2], &xl[k][p], &xr[k][p]);
    }
    if (lane < T + 2) {
        // wave speed |u| + sqrt(3 Theta)
        const R n = s[0][lane + 1], nu = s[1][lane + 1], e2 = s[2][lane + 1];
        R w = R(0);
        if (n > R(0)) {
            const R ud = nu / n;
            R th = e2 / n - ud * ud;
            if (th < R(0)) th = R(0);
            w = fabs(ud) + sqrt(R(3) * th);
        }
        ws[lane] = w;
    }
    __syncwarp();
    const int k = lane / T, c = lane % T, ix = x0 + c;
    if (k >= 3 || ix >= nx) return;
    const R sm = fmax(ws[c], ws[c + 1]), sp = fmax(ws[c + 1], ws[c + 2]);
    const R Hm = R(0.5) * (xr[k + 1][c] + xl[k + 1][c + 1]) - R(0.5) * sm * (xl[k][c + 1] - xr[k][c]);
    const R Hp = R(0.5) * (xr[k + 1][c + 1] + xl[k + 1][c + 2]) - R(0.5) * sp * (xl[k][c + 2] - xr[k][c + 1]);
    R L = R(0);
    L -= (Hp - Hm) * (R)a.invdx;
    const R E = (R)a.eb[(long long)ix * 6], qm = (R)a.qm;
    if (k == 1) L += qm * s[0][c + 2] * E;
    if (k == 2) L += qm * R(2) * s[1][c + 2] * E;
    const long long o = (long long)ix * 3 + k;
    const double us = a.Us[o];
    const double u0 = a.a0 != 0.0 ? a.U0[o] : 0.0;
    a.Uout[o] = a.a0 * u0 + a.a1 * (us + a.dt * (double)L);
}

template <typename R, bool CLOSURE, int TX, int TY>
static cudaError_t launch_tile(const FluidArgs& a, cudaStream_t st) {
    auto* k = fluid_tile_kernel<R, CLOSURE, TX, TY>;
    const int smem = (int)sizeof(FluidTile<R, TX, TY>);
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((a.nx + TX - 1) / TX), (unsigned)((a.ny + TY - 1) / TY));
    k<<<grid, kTileThreads, smem, st>>>(a);
    count_launch();
    return cudaGetLastError();
}

template <int TX, int TY>
static cudaError_t launch_shape(const FluidArgs& a, cudaStream_t st) {
    if (a.closure) return a.precision == 64 ? launch_tile<double, true, TX, TY>(a, st) : launch_tile<float, true, TX, TY>(a, st);
    return a.precision == 64 ? launch_tile<double, false, TX, TY>(a, st) : launch_tile<float, false, TX, TY>(a, st);
}

// The shape of the tiles: the one that forms fewest points on this grid, once the
// chip has work for two CTAs per SM, else 8 x 4 (more CTAs). A few rows or columns
// of cells fill 8 x 8 tiles badly: one FP64 step of 65535 x 1 cells 14.1 ms, in 32 x
// 1 tiles 3.1; 1 x 65535 14.2, in 1 x 32 3.1; 16384 x 3 3.7, in 8 x 4 2.1 (a thread per
// cell: 3.7, 3.7 and 2.7).
static int tile_shape(int nx, int ny) {
    constexpr int tx[4] = {8, 8, 32, 1}, ty[4] = {4, 8, 1, 32};
    int best = 0;
    long long least = 0;
    for (int q = 0; q < 4; ++q) {
        const long long tiles = (long long)((nx + tx[q] - 1) / tx[q]) * ((ny + ty[q] - 1) / ty[q]);
        const long long points = tiles * ((tx[q] + 2) * ty[q] + tx[q] * (ty[q] + 2));
        if (q == 0) least = points;
        if (q > 0 && tiles >= 2 * 152 && points <= least) least = points, best = q;
    }
    return best;
}

cudaError_t launch_fluid_stage(const FluidArgs& args, cudaStream_t st) {
    FluidArgs a = args;
    a.invdx = 1.0 / a.dx;
    a.invdy = 1.0 / a.dy;
    a.invdx2 = 1.0 / (a.dx * a.dx);
    a.invdy2 = 1.0 / (a.dy * a.dy);
    if (a.nvdim == 1) {
        const unsigned grid = (unsigned)((a.nx + kCells1d - 1) / kCells1d);
        if (a.precision == 64) fluid1d_stage_kernel<double><<<grid, 32, 0, st>>>(a);
        else fluid1d_stage_kernel<float><<<grid, 32, 0, st>>>(a);
        count_launch();
        return cudaGetLastError();
    }
    switch (tile_shape(a.nx, a.ny)) {
        case 0: return launch_shape<8, 4>(a, st);
        case 1: return launch_shape<8, 8>(a, st);
        case 2: return launch_shape<32, 1>(a, st);
        default: return launch_shape<1, 32>(a, st);
    }
}

}  // namespace vl

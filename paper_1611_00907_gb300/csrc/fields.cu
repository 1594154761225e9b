// Field kernels around the fused step: equilibrium initialisation (Eq. 14),
// macroscopic fields and FP64 reductions, natural-order populations, and
// the density gather used by checkpoints.
#include <cuda_fp16.h>

#include <algorithm>

#include "device_common.cuh"

namespace cplbm {

// ---------------------------------------------------------------------------
// Initial state f_i = f_i^eq(rho, u) (Eq. 14) at every fluid node, evaluated
// in FP64 whatever the storage and bound by the FP64 units: opposite
// directions share the even part of Eq. 14 and the factors are applied once,
// 35 FP64 instructions a node against 60 for the eight expressions written
// out.  It leaves the snapshot of the reductions behind as well, which took a
// pass of macro_kernel.  1500 x 1100 FP64: 203 + 320 -> 135 us.
// A block takes 64 x 4 nodes.
// ---------------------------------------------------------------------------
constexpr int INIT_X = 64, INIT_Y = 4;

template <class S>
__global__ void __launch_bounds__(INIT_X *INIT_Y)
    init_kernel(const Lattice L, const double *rho_in, const double *ux_in,
                const double *uy_in, double *prev, int *bad, int blocks_x, double pole)
{
    using pop_t = typename S::pop_t;
    using rho_t = typename S::rho_t;
    using real = typename S::real;
    const int by = blockIdx.x / blocks_x, bx = blockIdx.x - by * blocks_x;
    const int x = bx * INIT_X + threadIdx.x % INIT_X, r = by * INIT_Y + threadIdx.x / INIT_X;
    if (x >= L.nx || r >= L.nyf) return;
    const long long g = (long long)(r + L.walls) * L.nx + x;  // lattice index
    const double rho = rho_in[g];
    const double ux = ux_in ? ux_in[g] : 0.0, uy = uy_in ? uy_in[g] : 0.0;
    if (!(rho > 0.0 && rho < pole && isfinite(ux) && isfinite(uy)))
        atomicAdd(bad, 1);
    const double ref = S::offset ? L.rho_ref : 0.0;
    // f_i = w_i (rho (e +- 3 e_i.u) - ref), e = 1 + 4.5 (e_i.u)^2 - 1.5 u^2
    const double c = 1.0 - 1.5 * (ux * ux + uy * uy);
    const double sp = ux + uy, sm = ux - uy;
    const double r1 = rho * (1.0 / 9.0), r5 = rho * (1.0 / 36.0);
    pop_t *A = (pop_t *)L.pops + fidx(L, r, x);
    auto pair = [&](int i, double w, double rw, double u) {
        const double e = 4.5 * u * u + c, o = 3.0 * u;
        pop_t *p = A + (i - 1) * L.plane, *q = A + (opp(i) - 1) * L.plane;
        const double fp = S::offset ? rw * (e + o) - w * ref : rw * (e + o);
        const double fq = S::offset ? rw * (e - o) - w * ref : rw * (e - o);
        if (CPLBM_IN_POPS(L, p, 1)) st_real(p, (real)fp);
        if (CPLBM_IN_POPS(L, q, 1)) st_real(q, (real)fq);
    };
    pair(1, 1.0 / 9.0, r1, ux);
    pair(2, 1.0 / 9.0, r1, uy);
    pair(5, 1.0 / 36.0, r5, sp);
    pair(8, 1.0 / 36.0, r5, sm);
    const rho_t stored = (rho_t)(rho - ref);
    rho_t *q = (rho_t *)L.rho[0] + fidx(L, r, x);
    if (CPLBM_IN_RHO(L, 0, q, 1)) *q = stored;
    prev[g] = (double)((real)stored + (S::offset ? consts<real>(L).rho_ref : real(0)));
}

// Zero both generations of partial sums: block row k is generation k / 8,
// class k % 8.  One launch where sixteen memsets stood.
__global__ void clear_rings_kernel(const Lattice L, int words_per_entry)
{
    const int gen = blockIdx.y / R_COUNT, c = blockIdx.y % R_COUNT;
    const long long n = (long long)ring_elems(L, c) * words_per_entry;
    int *p = (int *)L.ring[gen][c];
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        p[i] = 0;
}

// ---------------------------------------------------------------------------
// Macroscopic fields (rho, v = u + F / (2 rho), mu) on the lattice rows of
// the output, plus optional FP64 reductions.  Tiled like the step so that
// mu and F come from the same stencil code.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void atomic_max_nonneg(double *addr, double v)
{
    // non-negative doubles order like their bit patterns
    atomicMax((unsigned long long *)addr, (unsigned long long)__double_as_longlong(v));
}

// A population: no store of the kernel touches it, so the loads of a thread's
// rows need not wait for the stores of the rows before (with them in order the
// reductions waited for memory eight times in a row: 2048 x 2048 FP32 314 us).
__device__ __forceinline__ double ld_stable(const double *p) { return __ldg(p); }
__device__ __forceinline__ float ld_stable(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ld_stable(const __half *p) { return __half2float(__ldg(p)); }
// Tests and comparisons of doubles on their bits: the FP64 units do the
// floating-point ones.  Non-negative doubles order like their bits.
__device__ __forceinline__ bool finite64(double v)
{
    return ((unsigned)__double2hiint(v) & 0x7FF00000u) != 0x7FF00000u;
}
__device__ __forceinline__ unsigned long long magnitude(double v)
{
    return (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
}
// FP64 values of FP32 results, exact, without the FP64 units, which do the
// type conversions too: the bits moved as in widen, those of subnormals after
// a scaling by 2^64.  (With a branch for them the field reads of 4096 x 4096
// FP32 took 460 us instead of 423; without them 420.)
__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(float v)
{
    const unsigned mag = __float_as_uint(v) & 0x7FFFFFFFu;
    if (mag >= 0x7F800000u) return (double)v;  // infinities, NaN
    const bool small = mag < 0x00800000u;      // zero, subnormal
    const unsigned m = __float_as_uint(small ? v * 0x1p64f : v) & 0x7FFFFFFFu;
    return __hiloint2double((int)((__float_as_uint(v) & 0x80000000u) |
                                  (m ? (m >> 3) + (small ? 0x34000000u : 0x38000000u) : 0u)),
                            (int)(m << 29));
}
// 1 / rho: IEEE division where rcp_nr has no answer (zero, infinite).  (The
// velocities' product with it, instead of a division, leaves the fields as far
// from 64-bit references as before, 1.5e-15 at 1500 x 1100; a remainder step
// that rounds it like the division took the fields' reads 9 % longer.)
__device__ __forceinline__ double inverse(double v)
{
    const unsigned e = (unsigned)__double2hiint(v) >> 20 & 0x7FFu;
    return e > 1 && e < 0x7FDu ? rcp_nr(v) : 1.0 / v;
}
// v / 3 correctly rounded (normal v): the rounded product, corrected by its
// exact remainder.
__device__ __forceinline__ float third(float v)
{
    const float q = v * (1.0f / 3.0f);
    return fmaf(fmaf(-3.0f, q, v), 1.0f / 3.0f, q);
}
// rho v = j + F / 2 of a node (momentum, force of Eq. 12 from the 12 grad).
__device__ __forceinline__ void half_force(const Consts<float> &, const float *f, float rho,
                                           float grx, float gry, float gmx, float gmy,
                                           double &px, double &py)
{
    const float c = 1.0f / 12.0f;
    const float Fx = -rho * (gmx * c) + third(grx * c), Fy = -rho * (gmy * c) + third(gry * c);
    const float jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8];
    const float jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8];
    px = to_f64(jx) + 0.5 * to_f64(Fx);
    py = to_f64(jy) + 0.5 * to_f64(Fy);
}
__device__ __forceinline__ void half_force(const Consts<double> &, const double *f, double rho,
                                           double grx, double gry, double gmx, double gmy,
                                           double &px, double &py)
{
    double jx, jy;
    momentum(f, jx, jy);
    const double r = rho * (-1.0 / 24.0);
    px = (1.0 / 72.0) * grx + (r * gmx + jx);
    py = (1.0 / 72.0) * gry + (r * gmy + jy);
}

// FP64 is bound by the FP64 units (about 70 FP64 instructions a node): 1500 x
// 1100, the four fields 367 -> 250 us; FP32 by instruction issue and latency
// (the division and the sums are FP64 in every storage): 4096 x 4096, density
// and velocity 829 -> 413 us with four blocks of 64 registers per SM (476 with
// three), the sums 847 -> 433.
template <class S, int TX, int TY>
__global__ void __launch_bounds__(256, sizeof(typename S::real) == 8 ? 3 : 4)
    macro_kernel(const Lattice L, int parity, int cur, double *o_rho, double *o_vx,
                 double *o_vy, double *o_mu, double *red, double *prev, int *bad,
                 long long tiles, int tiles_x)
{
    using real = typename S::real;
    using pop_t = typename S::pop_t;
    constexpr int WR = TX + 4, WM = TX + 2;
    constexpr int PER = TX * TY / 256;   // rows of a thread, one above the other
    static_assert(PER * 256 == TX * TY, "whole columns of rows");
    extern __shared__ unsigned char smem_raw[];
    real *s_rho = reinterpret_cast<real *>(smem_raw);
    real *s_mu = s_rho + (TY + 4) * WR;
    __shared__ double s_sum[4][256];
    __shared__ int s_bad;

    if (threadIdx.x == 0) s_bad = 0;
    const bool flow = o_vx || o_vy || red;   // otherwise no population is needed
    const Consts<real> &K = consts<real>(L);
    const real rho_ref = S::offset ? K.rho_ref : real(0);
    const pop_t *A = (const pop_t *)L.pops;
    double acc_m = 0.0, acc_x = 0.0, acc_y = 0.0;
    unsigned long long acc_d = 0;  // magnitude of a non-negative double
    int nbad = 0;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int X0 = (int)(tile % tiles_x) * TX, Y0 = (int)(tile / tiles_x) * TY;
        const int wx = min(TX, L.nx - X0), wy = min(TY, L.nyf - Y0);
        load_rho_tile<S, TX, TY>(L, cur, X0, Y0, s_rho);
        __syncthreads();
        if (flow || o_mu) {  // otherwise the density is all that is asked for
            mu_tile<S, TX, TY, true>(L, X0, Y0, s_rho, s_mu);
            __syncthreads();
        }

        // Tiles away from the lattice's edges read each direction at a constant
        // offset; the general addressing took a third of the instructions.
        const bool inside = X0 >= 1 && X0 + TX < L.nx && Y0 >= 1 && Y0 + TY < L.nyf;
        long long off[9];
#pragma unroll
        for (int i = 1; i < 9; ++i)
            off[i] = parity == 0 ? (i - 1) * L.plane
                                 : (opp(i) - 1) * L.plane - (long long)ey(i) * L.pitch - ex(i);
        // the snapshot's rows ahead of the work that needs them
        double before[PER];
        if (red && prev) {
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int x = threadIdx.x % TX, y = threadIdx.x / TX * PER + k;
                before[k] = x < wx && y < wy
                                ? prev[(long long)(Y0 + y + L.walls) * L.nx + X0 + x] : 0.0;
            }
        }
        // s_rho holds the stored form; rho_ref makes it absolute
        const int lx = threadIdx.x % TX, ly0 = threadIdx.x / TX * PER;
        const int cr0 = (ly0 + 1) * WR + lx + 2, cm0 = ly0 * WM + lx + 1;
        Row<real> rd = row_of(s_rho, cr0), rm = row_of(s_rho, cr0 + WR);
        Row<real> md = row_of(s_mu, cm0), mm = row_of(s_mu, cm0 + WM);
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int ly = ly0 + k;
            const Row<real> ru = row_of(s_rho, cr0 + (k + 2) * WR);
            const Row<real> mu = row_of(s_mu, cm0 + (k + 2) * WM);
            if (lx < wx && ly < wy) {
                const int x = X0 + lx, r = Y0 + ly;
                const long long g = (long long)(r + L.walls) * L.nx + x;
                const real rho = rm.c + rho_ref;
                const double rho64 = to_f64(rho);
                if (o_rho) o_rho[g] = rho64;
                if (o_mu) o_mu[g] = to_f64(mm.c);
                if (flow) {
                    real f[9];
                    if (inside) {
                        const pop_t *q = A + fidx(L, r, x);
#pragma unroll
                        for (int i = 1; i < 9; ++i)
                            f[i] = CPLBM_IN_POPS(L, q + off[i], 1) ? ld_stable(q + off[i]) : real(0);
                    } else {
#pragma unroll
                        for (int i = 1; i < 9; ++i) {
                            const pop_t *p = A + aa_read_index(L, parity, i, r, x);
                            f[i] = CPLBM_IN_POPS(L, p, 1) ? ld_stable(p) : real(0);
                        }
                    }
                    real grx, gry, gmx, gmy;
                    grad12(ru, rm, rd, grx, gry);
                    grad12(mu, mm, md, gmx, gmy);
                    double px, py;  // rho v
                    half_force(K, f, rho, grx, gry, gmx, gmy, px, py);
                    if (o_vx || o_vy) {
                        const double ir = inverse(rho64);
                        if (o_vx) o_vx[g] = px * ir;
                        if (o_vy) o_vy[g] = py * ir;
                    }
                    if (red) {
                        acc_m += rho64;
                        acc_x += px;
                        acc_y += py;
                        if (!(finite64(rho64) && finite64(px) && finite64(py))) ++nbad;
                        if (prev) {
                            const double d = rho64 - before[k];
                            if (finite64(d)) acc_d = max(acc_d, magnitude(d));
                            prev[g] = rho64;
                        }
                    }
                }
            }
            rd = rm;
            rm = ru;
            md = mm;
            mm = mu;
        }
        // Solid rows: rho by Eq. 28 and the wall mu from the shared tiles.
        if (L.walls && (o_rho || o_mu || o_vx || o_vy)) {
            for (int lx = threadIdx.x; lx < wx; lx += blockDim.x) {
                const int x = X0 + lx;
                if (Y0 == 0) {
                    const long long g = x;
                    if (o_rho) o_rho[g] = (double)(s_rho[1 * WR + lx + 2] + rho_ref);
                    if (o_mu) o_mu[g] = (double)s_mu[0 * WM + lx + 1];
                    if (o_vx) o_vx[g] = 0.0;
                    if (o_vy) o_vy[g] = 0.0;
                }
                if (Y0 + wy == L.nyf) {
                    const long long g = (long long)(L.ny - 1) * L.nx + x;
                    if (o_rho) o_rho[g] = (double)(s_rho[(wy + 2) * WR + lx + 2] + rho_ref);
                    if (o_mu) o_mu[g] = (double)s_mu[(wy + 1) * WM + lx + 1];
                    if (o_vx) o_vx[g] = 0.0;
                    if (o_vy) o_vy[g] = 0.0;
                }
            }
        }
        __syncthreads();  // the next tile reuses the shared memory
    }
    if (red) {
        // block reduction in a fixed order: the threads' sums by columns of
        // eight in the first warp, then across its lanes (FP64 additions on
        // one warp of the block instead of all eight)
        if (nbad) atomicAdd(&s_bad, nbad);
        s_sum[0][threadIdx.x] = acc_m;
        s_sum[1][threadIdx.x] = acc_x;
        s_sum[2][threadIdx.x] = acc_y;
        s_sum[3][threadIdx.x] = __longlong_as_double((long long)acc_d);
        __syncthreads();
        if (threadIdx.x < 32) {
            double m = 0, sx = 0, sy = 0, d = 0;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                const int t = threadIdx.x + 32 * w;
                m += s_sum[0][t];
                sx += s_sum[1][t];
                sy += s_sum[2][t];
                d = fmax(d, s_sum[3][t]);
            }
            for (int o = 16; o > 0; o >>= 1) {
                m += __shfl_down_sync(0xffffffffu, m, o);
                sx += __shfl_down_sync(0xffffffffu, sx, o);
                sy += __shfl_down_sync(0xffffffffu, sy, o);
                d = fmax(d, __shfl_down_sync(0xffffffffu, d, o));
            }
            if (threadIdx.x == 0) {
                atomicAdd(&red[0], m);
                atomicAdd(&red[1], sx);
                atomicAdd(&red[2], sy);
                atomic_max_nonneg(&red[3], d);
                if (s_bad) atomicAdd(bad, s_bad);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Natural-order FP64 populations [9][ny][nx] (solid rows untouched).
// ---------------------------------------------------------------------------
template <class S>
__global__ void populations_kernel(const Lattice L, int parity, int cur,
                                   double *f)
{
    using pop_t = typename S::pop_t;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (long long)L.nx * L.nyf) return;
    const int x = (int)(n % L.nx), r = (int)(n / L.nx);
    const long long N = (long long)L.nx * L.ny;
    const long long g = (long long)(r + L.walls) * L.nx + x;
    const double ref = S::offset ? L.rho_ref : 0.0;
    const pop_t *A = (const pop_t *)L.pops;
    double sum = 0.0;
    for (int i = 1; i < 9; ++i) {
        const pop_t *p = A + aa_read_index(L, parity, i, r, x);
        const double v = (CPLBM_IN_POPS(L, p, 1) ? (double)ld_real(p) : 0.0) +
                         wgt<double>(i) * ref;
        f[i * N + g] = v;
        sum += v;
    }
    f[g] = (double)load_rho<S>(L, cur, r, x) - sum;
}

// Stored-form density sum of every fluid node into dst (see load_rho).
template <class S>
__global__ void gather_rho_kernel(const Lattice L, int cur, void *dst)
{
    using rho_t = typename S::rho_t;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (long long)L.nx * L.nyf) return;
    const int x = (int)(n % L.nx), r = (int)(n / L.nx);
    ((rho_t *)dst)[fidx(L, r, x)] = (rho_t)load_rho_stored<S>(L, cur, r, x);
}

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
static inline unsigned blocks_for(long long n, int t)
{
    return (unsigned)((n + t - 1) / t);
}

template <class S>
static cudaError_t launch_init_t(const Lattice &L, const double *rho,
                                 const double *ux, const double *uy, double *prev,
                                 int *bad, cudaStream_t s)
{
    const int bx = (L.nx + INIT_X - 1) / INIT_X, by = (L.nyf + INIT_Y - 1) / INIT_Y;
    const double pole = (L.eos.kind == EOS_CS ? 4.0 : 1.0) / L.eos.b;
    init_kernel<S><<<(unsigned)bx * (unsigned)by, INIT_X * INIT_Y, 0, s>>>(L, rho, ux, uy, prev,
                                                                          bad, bx, pole);
    return cudaGetLastError();
}

// Four rounds of three blocks on each of 152 SMs.
constexpr long long MACRO_SUM_BLOCKS = 152 * 3 * 4;

template <class S, int TY>
static cudaError_t launch_macro_ty(const Lattice &L, int parity, int cur, double *rho,
                                   double *vx, double *vy, double *mu, double *red,
                                   double *prev, int *bad, cudaStream_t s)
{
    using real = typename S::real;
    constexpr int TX = FIELD_TILE_X;
    const size_t smem = sizeof(real) * ((TY + 4) * (TX + 4) + (TY + 2) * (TX + 2));
    const int tiles_x = (L.nx + TX - 1) / TX;
    const long long tiles = (long long)tiles_x * ((L.nyf + TY - 1) / TY);
    // The sums end in four atomics per block on the same four words: a bounded
    // number of blocks, each with several tiles of a large lattice.
    const unsigned grid = (unsigned)(red ? std::min(tiles, MACRO_SUM_BLOCKS) : tiles);
    macro_kernel<S, TX, TY><<<grid, 256, smem, s>>>(L, parity, cur, rho, vx, vy, mu, red, prev,
                                                    bad, tiles, tiles_x);
    return cudaGetLastError();
}

// Tiles of 64 x 16, or of 64 x 4 (a quarter of the work per block, half of
// it halo) while 64 x 16 would leave SMs without a block.
template <class S>
static cudaError_t launch_macro_t(const Lattice &L, int parity, int cur, double *rho, double *vx,
                                  double *vy, double *mu, double *red, double *prev, int *bad,
                                  cudaStream_t s)
{
    const long long tiles = (long long)((L.nx + FIELD_TILE_X - 1) / FIELD_TILE_X) *
                            ((L.nyf + FIELD_TILE_Y - 1) / FIELD_TILE_Y);
    return tiles < 152 ? launch_macro_ty<S, FIELD_TILE_Y_SMALL>(L, parity, cur, rho, vx, vy, mu,
                                                                red, prev, bad, s)
                       : launch_macro_ty<S, FIELD_TILE_Y>(L, parity, cur, rho, vx, vy, mu, red,
                                                          prev, bad, s);
}

template <class S>
static cudaError_t launch_pop_t(const Lattice &L, int parity, int cur,
                                double *f, cudaStream_t s)
{
    const long long n = (long long)L.nx * L.nyf;
    populations_kernel<S><<<blocks_for(n, 256), 256, 0, s>>>(L, parity, cur, f);
    return cudaGetLastError();
}

template <class S>
static cudaError_t launch_gather_t(const Lattice &L, int cur, void *dst,
                                   cudaStream_t s)
{
    const long long n = (long long)L.nx * L.nyf;
    gather_rho_kernel<S><<<blocks_for(n, 256), 256, 0, s>>>(L, cur, dst);
    return cudaGetLastError();
}

#define CPLBM_DISPATCH(prec, call)                                   \
    switch (prec) {                                                  \
    case P_F64: { using S = SF64; return call; }                     \
    case P_F32: { using S = SF32; return call; }                     \
    case P_F32_OFF: { using S = SF32Off; return call; }              \
    case P_F16_OFF: { using S = SF16Off; return call; }              \
    }                                                                \
    return cudaErrorInvalidValue;

cudaError_t launch_init(const Lattice &L, const double *rho, const double *ux,
                        const double *uy, double *prev, int *bad, cudaStream_t s)
{
    CPLBM_DISPATCH(L.precision, launch_init_t<S>(L, rho, ux, uy, prev, bad, s))
}

cudaError_t launch_clear_rings(const Lattice &L, cudaStream_t s)
{
    const int words = (int)rho_bytes(L.precision) / 4;
    const size_t most = std::max(ring_elems(L, R_L), ring_elems(L, R_B)) * words;
    const unsigned blocks = (unsigned)std::min<size_t>((most + 255) / 256, 64);
    clear_rings_kernel<<<dim3(blocks, 2 * R_COUNT), 256, 0, s>>>(L, words);
    return cudaGetLastError();
}

cudaError_t launch_macro(const Lattice &L, int parity, int cur, double *rho,
                         double *vx, double *vy, double *mu, double *red,
                         double *prev, int *bad, cudaStream_t s)
{
    CPLBM_DISPATCH(L.precision, launch_macro_t<S>(L, parity, cur, rho, vx, vy,
                                                  mu, red, prev, bad, s))
}

cudaError_t launch_populations(const Lattice &L, int parity, int cur,
                               double *f, cudaStream_t s)
{
    CPLBM_DISPATCH(L.precision, launch_pop_t<S>(L, parity, cur, f, s))
}

cudaError_t launch_gather_rho(const Lattice &L, int cur, void *dst,
                              cudaStream_t s)
{
    CPLBM_DISPATCH(L.precision, launch_gather_t<S>(L, cur, dst, s))
}

// The FP64 logarithm and reciprocal of the step kernels on n values
// (lbm_test_fp64_math).
__global__ void fp64_math_kernel(const double *__restrict__ x, int n,
                                 double *__restrict__ lg, double *__restrict__ rc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        lg[i] = log_tab(x[i]);
        rc[i] = rcp_nr(x[i]);
    }
}

cudaError_t launch_fp64_math(const double *x, int n, double *lg, double *rc,
                             cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    fp64_math_kernel<<<(n + 255) / 256, 256, 0, s>>>(x, n, lg, rc);
    return cudaGetLastError();
}

}  // namespace cplbm

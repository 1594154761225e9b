// Device building blocks of the chemical-potential LBM step (arXiv
// 1611.00907): D2Q9 lattice, storage types, the EOS chemical potentials,
// the AA-pattern addressing and the tile loaders shared by the fused step
// kernel and the field kernels.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "cplbm_internal.h"
#include "log_table.h"

namespace cplbm {

// ---------------------------------------------------------------------------
// D2Q9 lattice (Eq. 13-14).  e_0 = (0,0); e_1..4 = (1,0),(0,1),(-1,0),(0,-1);
// e_5..8 = (1,1),(-1,1),(-1,-1),(1,-1).
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int ex(int i)
{
    return (i == 1 || i == 5 || i == 8) ? 1 : (i == 3 || i == 6 || i == 7) ? -1 : 0;
}
__host__ __device__ constexpr int ey(int i)
{
    return (i == 2 || i == 5 || i == 6) ? 1 : (i == 4 || i == 7 || i == 8) ? -1 : 0;
}
__host__ __device__ constexpr int opp(int i)
{
    return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4) + 1 : ((i - 3) % 4) + 5);
}
static_assert(opp(1) == 3 && opp(2) == 4 && opp(3) == 1 && opp(4) == 2, "");
static_assert(opp(5) == 7 && opp(6) == 8 && opp(7) == 5 && opp(8) == 6, "");

template <class T>
__host__ __device__ constexpr T wgt(int i)
{
    return i == 0 ? T(4) / T(9) : (i <= 4 ? T(1) / T(9) : T(1) / T(36));
}

// ---------------------------------------------------------------------------
// Storage variants: population storage type, density storage type, the
// arithmetic type, and whether values are stored as offsets from the
// reference state (f_i - w_i rho_ref, rho - rho_ref).
// ---------------------------------------------------------------------------
struct SF64 {
    using pop_t = double; using rho_t = double; using real = double;
    static constexpr bool offset = false;
};
struct SF32 {
    using pop_t = float; using rho_t = float; using real = float;
    static constexpr bool offset = false;
};
struct SF32Off {
    using pop_t = float; using rho_t = float; using real = float;
    static constexpr bool offset = true;
};
struct SF16Off {
    using pop_t = __half; using rho_t = float; using real = float;
    static constexpr bool offset = true;
};

__device__ __forceinline__ double ld_real(const double *p) { return *p; }
__device__ __forceinline__ float ld_real(const float *p) { return *p; }
__device__ __forceinline__ float ld_real(const __half *p) { return __half2float(*p); }
__device__ __forceinline__ void st_real(double *p, double v) { *p = v; }
__device__ __forceinline__ void st_real(float *p, float v) { *p = v; }
__device__ __forceinline__ void st_real(__half *p, float v) { *p = __float2half_rn(v); }

// ---------------------------------------------------------------------------
// Bounds-checked build (CPLBM_CHECK_BOUNDS; a debug build that stands in for
// a memory checker): the global accesses of the step and field kernels are
// checked against the buffer they belong to first; an access outside it
// raises ERR_BOUNDS in L.err and is skipped (a load reads zero, a copy
// leaves its destination as it was).  TMA loads need no check: the tensor
// map bounds them.  In the normal build every check is the constant true,
// its arguments are not evaluated, and the accesses compile as before.
// n: elements accessed from p on.
// ---------------------------------------------------------------------------
#ifdef CPLBM_CHECK_BOUNDS
__device__ __forceinline__ bool in_buffer(const Lattice &L, const void *base, long long bytes,
                                          const void *p, long long size)
{
    const long long off = (const char *)p - (const char *)base;
    if (off >= 0 && off + size <= bytes) return true;
    if (L.err) atomicOr(L.err, ERR_BOUNDS);
    return false;
}
#define CPLBM_IN_POPS(L, p, n) \
    ::cplbm::in_buffer(L, (L).pops, (L).b_pops, p, (long long)(n) * sizeof(*(p)))
#define CPLBM_IN_RHO(L, k, p, n) \
    ::cplbm::in_buffer(L, (L).rho[k], (L).b_rho, p, (long long)(n) * sizeof(*(p)))
#define CPLBM_IN_RING(L, k, c, p, n) \
    ::cplbm::in_buffer(L, (L).ring[k][c], (L).b_ring[c], p, (long long)(n) * sizeof(*(p)))
#else
#define CPLBM_IN_POPS(L, p, n) true
#define CPLBM_IN_RHO(L, k, p, n) true
#define CPLBM_IN_RING(L, k, c, p, n) true
#endif

// ---------------------------------------------------------------------------
// Bulk chemical potential psi'(rho): Eq. 18 (vdW), Eq. 21 (RK/RKS), Eq. 24
// (PR), Eq. 27 (CS) without the -kappa lap(rho) term.
// ---------------------------------------------------------------------------
// FP64 reciprocal: the hardware's approximate reciprocal r (PTX
// rcp.approx.ftz.f64, which works on the upper 20 significand bits), then
// one cubic step r (1 + e + e^2) with the residual e = 1 - x r: what is left
// of the error is e^3, below 2^-56, a sixteenth of an ulp.  Three FP64-pipe
// instructions, one less than the two Newton-Raphson steps that reach the
// same (the GB300 FP64 pipe bounds the FP64 step).  Over 2.4 million samples
// of densities, pole distances and wide ranges the largest error is 0.508 ulp
// (0.500 after two Newton steps), the mean square the same to five digits, and
// 0.04 % of the values are not the correctly rounded ones; the fields of whole
// runs are equally far from 64-bit references either way, and two Newton steps
// cost FP64 steps 2.5 %.  Zero, infinite and NaN x give NaN.
__device__ __forceinline__ double rcp_nr(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// FP64 natural logarithm after Tang's table-driven method (P. T. P. Tang,
// ACM TOMS 16(4), 1990).  x = 2^m y with y in [1, 2); F = 1 + j/128 the
// breakpoint next to y, f = y - F (exact, |f| <= 2^-8), r = f/F from the
// tabulated 1/F; ln x = m ln 2 + ln F + ln(1 + r), the last by its Taylor
// series through r^7 (the rest is below 2^-59 of r).  The terms from r^5 on
// are r^5 T(r), T = 1/5 - r/6 + r^2/7, below 2^-42: T is summed in FP32,
// whose rounding moves the logarithm by less than 2^-58 of r, and goes to
// and from FP32 by moving bits (the GB300 FP64 pipe, which bounds the FP64
// step, does the type conversions too).  The exponent m becomes a double
// the same way.  ln 2 and ln F are
// tabulated as hi + lo with hi a multiple of 2^-32, so m ln2_hi + lnF_hi is
// exact: just below 1 the two cancel almost entirely, and only the small
// terms carry rounding errors.  For x in [1 - 2^-9, 1) (m = -1, j = 128) the
// series takes r = x - 1 directly.  Within about two ulp for positive
// normal x; zero, negative, subnormal, infinite and NaN x go to log().
__device__ __forceinline__ float narrow(double v)   // truncates; |v| < 2^-126: 0
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned mag = ((hi & 0x7FFFFFFFu) - 0x38000000u) << 3 | lo >> 29;
    return (hi & 0x7FFFFFFFu) < 0x38100000u ? 0.0f
                                            : __uint_as_float((hi & 0x80000000u) | mag);
}
__device__ __forceinline__ double widen(float v)    // exact; v zero or normal
{
    const unsigned b = __float_as_uint(v), mag = b & 0x7FFFFFFFu;
    return __hiloint2double((int)((b & 0x80000000u) | (mag ? (mag >> 3) + 0x38000000u : 0u)),
                            (int)(b << 29));
}
__device__ __forceinline__ double log_tab(double x)
{
    const int hi = __double2hiint(x);
    if ((unsigned)(hi - 0x00100000) >= 0x7FE00000u) return log(x);
    int m = (hi >> 20) - 1023;
    const int mant = hi & 0x000FFFFF;        // top 20 bits of the significand
    int j = (mant + (1 << 12)) >> 13;        // nearest multiple of 1/128: 0 .. 128
    double y = __hiloint2double(mant | 0x3FF00000, __double2loint(x));
    if (m == -1 && j == LOG_TABLE_N) {       // x in [1 - 2^-9, 1)
        y = x;
        m = 0;
        j = 0;
    }
    const double F = __hiloint2double(0x3FF00000 + (j << 13), 0);
    const double2 t = __ldg(&kLogTable[j]);  // {1/F, hi of ln F}
    const double r = (y - F) * t.x;
    const float rf = narrow(r);
    const double T = widen(fmaf(rf, fmaf(rf, 1.0f / 7.0f, -1.0f / 6.0f), 1.0f / 5.0f));
    double q = fma(T, r, -1.0 / 4.0);
    q = fma(q, r, 1.0 / 3.0);
    q = fma(q, r, -0.5);
    const double p = fma(r * r, q, r);       // ln(1 + r)
    const double dm = widen((float)m);
    return fma(dm, LN2_HI, t.y) + (fma(dm, LN2_LO, __ldg(&kLogTableLo[j])) + p);
}

// Reciprocal, division and logarithm of the arithmetic type: the FP32
// kernels use the hardware's approximate forms, whose few-ulp errors sit far
// below the FP32 storage error.  In the step kernels subnormal operands read
// as zero: one instruction each, where the scaling of subnormals takes three
// or four, which the issue-bound FP16-storage step paid for (2048 x 1026
// walled: 28.1 -> 26.7 us; results of normal operands are the same bits), so
// a step needs densities of 2^-126 = 1.2e-38 or more (below a quarter of that
// 1 / rho is infinite in FP32 anyway).  ANY: the logarithm of any density, for
// the field kernels, which read back whatever a lattice was given.  FP64: the
// reciprocal and logarithm above, within one or two ulp of IEEE division and
// log().
__device__ __forceinline__ float frcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double frcp(double x) { return rcp_nr(x); }
__device__ __forceinline__ float fdiv(float a, float b) { return a * frcp(b); }
__device__ __forceinline__ double fdiv(double a, double b) { return a * rcp_nr(b); }
template <bool ANY = false>
__device__ __forceinline__ float flog(float x)
{
    float l;
    if constexpr (ANY) asm("lg2.approx.f32 %0, %1;" : "=f"(l) : "f"(x));
    else asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(x));
    return l * 0.693147180559945f;
}
__device__ __forceinline__ double flog(double x) { return log_tab(x); }

template <bool ANY = false>
__device__ __forceinline__ float mu_bulk(const EosT<float> &e, float rho)
{
    switch (e.kind) {
    case EOS_VDW: {
        const float iq = fdiv(1.0f, 1.0f - e.b * rho);
        return e.RT * (flog<ANY>(rho * iq) + iq) - 2.0f * e.a * rho;
    }
    case EOS_CS: {
        const float h = e.quarter_b * rho;
        const float iq = fdiv(1.0f, 1.0f - h);
        return e.RT * ((3.0f - h) * (iq * iq * iq) + flog<ANY>(rho) + 1.0f) -
               2.0f * e.a * rho;
    }
    case EOS_PR: {
        const float br = e.b * rho;
        const float iq = fdiv(1.0f, 1.0f - br);
        return e.RT * flog<ANY>(rho * iq) -
               e.pr_c * flog(fdiv(e.pr_s2m1 + br, e.pr_s2p1 - br)) +
               e.RT * iq - fdiv(e.aalpha * rho, 1.0f + 2.0f * br - br * br);
    }
    default: {  // EOS_RKS
        const float br = e.b * rho;
        const float iq = fdiv(1.0f, 1.0f - br);
        return e.RT * (flog<ANY>(rho * iq) + iq) - e.rks_c * flog(1.0f + br) -
               fdiv(e.aalpha * rho, 1.0f + br);
    }
    }
}

// FP64: the same with fewer instructions.
template <bool = false>
__device__ __forceinline__ double mu_bulk(const EosT<double> &e, double rho)
{
    switch (e.kind) {
    case EOS_VDW: {
        const double iq = frcp(1.0 - e.b * rho);
        return e.RT * (flog(rho * iq) + iq) + e.m2a * rho;
    }
    case EOS_CS: {
        // (3 - h) / (1 - h)^3 = iq^2 (2 iq + 1) with iq = 1 / (1 - h)
        const double iq = frcp(1.0 - e.quarter_b * rho);
        return e.RT * (iq * iq * (2.0 * iq + 1.0) + flog(rho)) + (e.m2a * rho + e.RT);
    }
    case EOS_PR: {
        const double br = e.b * rho;
        const double iq = frcp(1.0 - br);
        return e.RT * (flog(rho * iq) + iq) -
               e.pr_c * flog(fdiv(e.pr_s2m1 + br, e.pr_s2p1 - br)) -
               fdiv(e.aalpha * rho, br * (2.0 - br) + 1.0);
    }
    default: {  // EOS_RKS
        const double br = e.b * rho;
        const double iq = frcp(1.0 - br), p = 1.0 + br;
        return e.RT * (flog(rho * iq) + iq) - e.rks_c * flog(p) - fdiv(e.aalpha * rho, p);
    }
    }
}

// Equation of state p0(rho): Eq. 16 (vdW), Eq. 19 (RK/RKS), Eq. 22 (PR),
// Eq. 25 (CS).  Used only by the pressure-tensor force of Eq. 5.
template <class T>
__device__ __forceinline__ T p0_bulk(const EosT<T> &e, T rho)
{
    const T br = e.b * rho;
    switch (e.kind) {
    case EOS_VDW:
        return fdiv(rho * e.RT, T(1) - br) - e.a * rho * rho;
    case EOS_CS: {
        const T h = e.quarter_b * rho, q = T(1) - h;
        return fdiv(rho * e.RT * (T(1) + h + h * h - h * h * h), q * q * q) -
               e.a * rho * rho;
    }
    case EOS_PR:
        return fdiv(rho * e.RT, T(1) - br) -
               fdiv(e.aalpha * rho * rho, T(1) + T(2) * br - br * br);
    default:  // EOS_RKS
        return fdiv(rho * e.RT, T(1) - br) - fdiv(e.aalpha * rho * rho, T(1) + br);
    }
}

// ---------------------------------------------------------------------------
// Asynchronous global -> shared copies of single elements (sm_80+ cp.async).
// A thread's copies become visible to that thread after cp_async_wait_all.
// ---------------------------------------------------------------------------
template <int BYTES>
__device__ __forceinline__ void cp_async(void *smem, const void *gmem)
{
    static_assert(BYTES == 4 || BYTES == 8 || BYTES == 16, "cp.async size");
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s),
                 "l"(gmem), "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}
// Wait until at most N of the thread's most recent copy groups are pending.
template <int N>
__device__ __forceinline__ void cp_async_wait_group()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------------------
// TMA (cp.async.bulk.tensor) loads completing on a shared-memory mbarrier.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_addr(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)),
                 "r"(count)
                 : "memory");
    // make the initialised barrier visible to the asynchronous proxy
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(
                     smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}
// Wait for phase `parity` of the barrier: poll while fewer than max_cycles
// SM clocks have passed; false when the limit was reached (max_cycles <= 0:
// at once, without polling).
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity,
                                          long long max_cycles)
{
    const unsigned a = smem_addr(bar);
    const long long t0 = clock64();
    while (clock64() - t0 < max_cycles) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n"
            " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map,
                                            int x, int y, unsigned long long *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];\n" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y),
        "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map,
                                            int x, int y, int z,
                                            unsigned long long *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z),
        "r"(smem_addr(bar))
        : "memory");
}

// ---------------------------------------------------------------------------
// Addressing.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int wrapi(int v, int n)
{
    return v < 0 ? v + n : (v >= n ? v - n : v);
}

// Index of population i (1..8) of fluid node (x, r) in the pops array.
__device__ __forceinline__ long long pidx(const Lattice &L, int i, int r, int x)
{
    return (long long)(i - 1) * L.plane + (long long)r * L.pitch + x;
}
__device__ __forceinline__ long long fidx(const Lattice &L, int r, int x)
{
    return (long long)r * L.pitch + x;
}
// Index of the partial sum of class c for the receiving node (r, x), whose
// tile is (bx, by): classes L and R keep one column per tile column, B and
// T one row per tile row, the corners one entry per tile.
__device__ __forceinline__ long long ring_index(const Lattice &L, int c, int bx,
                                                int by, int r, int x)
{
    if (c == R_L || c == R_R) return (long long)bx * L.nyf_pad + r;
    if (c == R_B || c == R_T) return (long long)by * L.pitch + x;
    return (long long)by * ((L.nx + 31) >> 5) + bx;
}

// Row r + dy of a fluid node; with walls, -1 / nyf mean the solid rows.
__device__ __forceinline__ bool row_is_solid(const Lattice &L, int r)
{
    return L.walls && (r < 0 || r >= L.nyf);
}
__device__ __forceinline__ int row_wrap(const Lattice &L, int r)
{
    return L.walls ? r : wrapi(r, L.nyf);
}

// AA pattern (in place).  Even step: node x reads f_i from its own slot i
// and writes f*_i into its own slot opp(i).  Odd step: node x reads f_i from
// slot opp(i) of x - e_i and writes f*_i into slot i of x + e_i.  Every slot
// a node reads is one it writes, so no two nodes touch the same slot in a
// step.  Halfway bounce-back (Sec. IV): on an odd step, a population whose
// source x - e_i is solid is read from slot i of x itself, where the even
// step left f*_opp(i); a population whose target x + e_i is solid is written
// to slot opp(i) of x, where the next even step reads it.
__device__ __forceinline__ long long aa_read_index(const Lattice &L, int parity,
                                                   int i, int r, int x)
{
    if (parity == 0) return pidx(L, i, r, x);
    const int rs = r - ey(i);
    if (row_is_solid(L, rs)) return pidx(L, i, r, x);
    return pidx(L, opp(i), row_wrap(L, rs), wrapi(x - ex(i), L.nx));
}
__device__ __forceinline__ long long aa_write_index(const Lattice &L,
                                                    int parity, int i, int r,
                                                    int x)
{
    if (parity == 0) return pidx(L, opp(i), r, x);
    const int rt = r + ey(i);
    if (row_is_solid(L, rt)) return pidx(L, opp(i), r, x);
    return pidx(L, i, row_wrap(L, rt), wrapi(x + ex(i), L.nx));
}

// Tile of a column or row: the compiled tile shapes are 32 or 64 wide and
// 16, 24 or 32 high, so no division by a variable is needed.
__device__ __forceinline__ int tile_x(const Lattice &L, int x) { return x >> (L.tx == 32 ? 5 : 6); }
__device__ __forceinline__ int tile_y(const Lattice &L, int r)
{
    return L.ty == 24 ? r / 24 : r >> (L.ty == 16 ? 4 : 5);
}

// ---------------------------------------------------------------------------
// Density of the current step at fluid node (x, r) in stored form (offset
// precisions: rho - rho_ref): the tile-local sum in rho[cur] plus the
// partial sums written by neighbouring tiles for nodes on the edge of their
// tile (see step.cu), always added in this order.
// ---------------------------------------------------------------------------
template <class S>
__device__ __forceinline__ typename S::real load_rho_stored(const Lattice &L,
                                                            int cur, int r,
                                                            int x)
{
    using rt = typename S::rho_t;
    using real = typename S::real;
    const rt *R = (const rt *)L.rho[cur];
    const rt *rp = R + fidx(L, r, x);
    real v = CPLBM_IN_RHO(L, cur, rp, 1) ? (real)*rp : real(0);
    const int bx = tile_x(L, x), by = tile_y(L, r);
    const int lx = x - bx * L.tx, ly = r - by * L.ty;
    const int wx = min(L.tx, L.nx - bx * L.tx);
    const int wy = min(L.ty, L.nyf - by * L.ty);
    const bool left = lx == 0, right = lx == wx - 1;
    const bool below = ly == 0 && !(L.walls && r == 0);
    const bool above = ly == wy - 1 && !(L.walls && r == L.nyf - 1);
    if (left | right | below | above) {
        rt *const *ring = (rt *const *)L.ring[cur];
        auto at = [&](int c) {
            const rt *q = ring[c] + ring_index(L, c, bx, by, r, x);
            return CPLBM_IN_RING(L, cur, c, q, 1) ? *q : rt(0);
        };
        if (left) v += (real)at(R_L);
        if (right) v += (real)at(R_R);
        if (below) {
            v += (real)at(R_B);
            if (left) v += (real)at(R_BL);
            if (right) v += (real)at(R_BR);
        }
        if (above) {
            v += (real)at(R_T);
            if (left) v += (real)at(R_TL);
            if (right) v += (real)at(R_TR);
        }
    }
    return v;
}

// Absolute density.
template <class S>
__device__ __forceinline__ typename S::real load_rho(const Lattice &L, int cur,
                                                     int r, int x)
{
    using real = typename S::real;
    const real v = load_rho_stored<S>(L, cur, r, x);
    return S::offset ? v + consts<real>(L).rho_ref : v;
}

// Fill s_rho[(TY + 4) x (TX + 4)] with the stored-form density of the tile
// at (X0, Y0) and a halo of two nodes; solid rows get the Eq. 28 average of
// the adjacent fluid row (the top row mirrors it from row nyf - 1).
template <class S, int TX, int TY>
__device__ void load_rho_tile(const Lattice &L, int cur, int X0, int Y0,
                              typename S::real *s_rho)
{
    using real = typename S::real;
    constexpr int W = TX + 4, H = TY + 4;
    const int wx = min(TX, L.nx - X0), wy = min(TY, L.nyf - Y0);
    // a halo that touches no edge of the lattice needs no wrap and no wall rule
    if (X0 >= 2 && X0 + TX + 2 <= L.nx && Y0 >= 2 && Y0 + TY + 2 <= L.nyf) {
        for (int k = threadIdx.x; k < W * H; k += blockDim.x)
            s_rho[k] = load_rho_stored<S>(L, cur, Y0 + k / W - 2, X0 + k % W - 2);
        return;
    }
    for (int k = threadIdx.x; k < W * H; k += blockDim.x) {
        const int lx = k % W, ly = k / W;
        if (lx > wx + 3 || ly > wy + 3) {  // beyond a ragged tile's halo
            s_rho[k] = real(0);
            continue;
        }
        // X0 - 2 <= x < X0 + wx + 2 <= nx + 2: one wrap suffices (nx >= 5)
        const int x = wrapi(X0 + lx - 2, L.nx);
        const int r = Y0 + ly - 2;
        real v;
        if (!L.walls) {
            v = load_rho_stored<S>(L, cur, wrapi(r, L.nyf), x);
        } else if (r >= 0 && r < L.nyf) {
            v = load_rho_stored<S>(L, cur, r, x);
        } else if (r == -1 || r == L.nyf) {
            // Eq. 28: rho(x, wall) = 2/3 rho(x, 1) + 1/6 rho(x-1, 1) + 1/6 rho(x+1, 1)
            // (the weights sum to one, so the stored form averages the same)
            const int rf = r < 0 ? 0 : L.nyf - 1;
            v = real(2.0 / 3.0) * load_rho_stored<S>(L, cur, rf, x) +
                real(1.0 / 6.0) * load_rho_stored<S>(L, cur, rf, wrapi(x - 1, L.nx)) +
                real(1.0 / 6.0) * load_rho_stored<S>(L, cur, rf, wrapi(x + 1, L.nx));
        } else {
            v = real(0);  // beyond a wall: never read
        }
        s_rho[k] = v;
    }
}

// Isotropic D2Q9 Laplacian and gradient on a shared-memory tile of row
// width W at linear index c.
template <class T, int W>
__device__ __forceinline__ T lap9(const T *s, int c)
{
    const T axial = s[c + 1] + s[c - 1] + s[c + W] + s[c - W];
    const T diag = (s[c + W + 1] + s[c + W - 1]) + (s[c - W + 1] + s[c - W - 1]);
    return (T(4) * axial + diag - T(20) * s[c]) * T(1.0 / 6.0);
}
template <class T, int W>
__device__ __forceinline__ void grad9(const T *s, int c, T &gx, T &gy)
{
    // 3 sum_i w_i phi(x + e_i) e_i = [4 (E - W) + (NE - NW + SE - SW)] / 12
    const T ne = s[c + W + 1], nw = s[c + W - 1];
    const T se = s[c - W + 1], sw = s[c - W - 1];
    gx = (T(4) * (s[c + 1] - s[c - 1]) + (ne - nw) + (se - sw)) * T(1.0 / 12.0);
    gy = (T(4) * (s[c + W] - s[c - W]) + (ne + nw) - (se + sw)) * T(1.0 / 12.0);
}

// One row of a field around column c of a stencil's window: the node, the
// sum and the difference of its east and west neighbours.  With rows u
// (above), m and d (below) the isotropic stencils without their factors are
//   12 grad_x = 4 D_m + D_u + D_d,   12 grad_y = 4 (C_u - C_d) + H_u - H_d,
//    6 lap    = 4 (H_m + C_u + C_d) + (H_u + H_d) - 20 C_m,
// which are grad9 / lap9 term by term; the factors sit in Consts.  A walk up
// the rows forms H and D once per row: 7 instructions for a gradient and 6
// for a Laplacian, against 12 and 9 from a 3 x 3 window.
template <class T> struct Row {
    T c, h, d;
};
template <class T>
__device__ __forceinline__ Row<T> row_of(const T *s, int i)
{
    const T w = s[i - 1], e = s[i + 1];
    return {s[i], e + w, e - w};
}
template <class T>
__device__ __forceinline__ T lap6(const Row<T> &u, const Row<T> &m, const Row<T> &d)
{
    return T(4) * (m.h + u.c + d.c) + (u.h + d.h) - T(20) * m.c;
}
template <class T>
__device__ __forceinline__ void grad12(const Row<T> &u, const Row<T> &m, const Row<T> &d,
                                       T &gx, T &gy)
{
    gx = T(4) * m.d + u.d + d.d;
    gy = T(4) * (u.c - d.c) + u.h - d.h;
}
// The same around linear index c of a shared-memory tile of row width W.
template <class T, int W>
__device__ __forceinline__ T lap6(const T *s, int c)
{
    return lap6(row_of(s, c + W), row_of(s, c), row_of(s, c - W));
}
template <class T, int W>
__device__ __forceinline__ void grad12(const T *s, int c, T &gx, T &gy)
{
    grad12(row_of(s, c + W), row_of(s, c), row_of(s, c - W), gx, gy);
}
// mu = psi'(rho) - kappa lap(rho) (Eq. 8) from the absolute density and 6 lap.
template <bool ANY = false>
__device__ __forceinline__ float mu_of(const Consts<float> &K, float rho, float l6)
{
    return mu_bulk<ANY>(K.eos, rho) - K.kappa * (l6 * (1.0f / 6.0f));
}
template <bool = false>
__device__ __forceinline__ double mu_of(const Consts<double> &K, double rho, double l6)
{
    return K.nk6 * l6 + mu_bulk(K.eos, rho);
}

// Fill s_mu[(TY + 2) x (TX + 2)] with mu on the tile and a one-node halo
// (Eq. 8) from the stored-form densities in s_rho; solid rows carry the
// surface values (Sec. IV, V).
template <class S, int TX, int TY, bool ANY = false>
__device__ void mu_tile(const Lattice &L, int X0, int Y0,
                        const typename S::real *s_rho, typename S::real *s_mu)
{
    using real = typename S::real;
    constexpr int W = TX + 2, H = TY + 2, WR = TX + 4;
    const Consts<real> &K = consts<real>(L);
    const real ref = S::offset ? K.rho_ref : real(0);
    const int wx = min(TX, L.nx - X0), wy = min(TY, L.nyf - Y0);
    for (int k = threadIdx.x; k < W * H; k += blockDim.x) {
        const int lx = k % W, ly = k / W;
        if (lx > wx + 1 || ly > wy + 1) {  // beyond a ragged tile's halo
            s_mu[k] = real(0);
            continue;
        }
        const int r = Y0 + ly - 1;
        const int c = (ly + 1) * WR + lx + 1;  // same node in s_rho
        real m;
        if (L.walls && r == -1) {
            m = K.mu_bottom;
        } else if (L.walls && r == L.nyf) {
            if (L.top_mode == 0) {
                const int cb = c - WR;  // fluid neighbour below (row nyf-1)
                m = mu_of<ANY>(K, s_rho[cb] + ref, lap6<real, WR>(s_rho, cb));
            } else {
                m = K.mu_top;
            }
        } else if (L.walls && (r < -1 || r > L.nyf)) {
            m = real(0);
        } else {
            m = mu_of<ANY>(K, s_rho[c] + ref, lap6<real, WR>(s_rho, c));
        }
        s_mu[k] = m;
    }
}

// ---------------------------------------------------------------------------
// BGK collision with the velocity-shift forcing (Eq. 13-14, Sec. II).
// ---------------------------------------------------------------------------
// m = sum f_i e_i + tau F of one node (populations f[1..8]) with the force
// of Eq. 12, F = -rho grad(mu) + grad(cs^2 rho), from the stencils 12 grad.
template <class T>
__device__ __forceinline__ void momentum(const T *f, T &jx, T &jy)
{
    const T d57 = f[5] - f[7], d86 = f[8] - f[6];
    jx = (f[1] - f[3]) + d57 + d86;
    jy = (f[2] - f[4]) + d57 - d86;
}
__device__ __forceinline__ void force_momentum(const Consts<float> &K, const float *f, float rho,
                                               float grx, float gry, float gmx, float gmy,
                                               float &mx, float &my)
{
    float jx, jy;
    momentum(f, jx, jy);
    const float c = 1.0f / 12.0f, third = 1.0f / 3.0f;
    const float Fx = grx * c * third - rho * (gmx * c);
    const float Fy = gry * c * third - rho * (gmy * c);
    mx = jx + K.tau * Fx;
    my = jy + K.tau * Fy;
}
__device__ __forceinline__ void force_momentum(const Consts<double> &K, const double *f,
                                               double rho, double grx, double gry, double gmx,
                                               double gmy, double &mx, double &my)
{
    double jx, jy;
    momentum(f, jx, jy);
    const double tr = K.nt12 * rho;
    mx = K.t36 * grx + (tr * gmx + jx);
    my = K.t36 * gry + (tr * gmy + jy);
}

// Collision of one node towards the equilibrium of velocity u = m / rho.
// f[1..8] are the node's stored populations (f_0 = drho - sum f_i is
// implicit), drho its stored density (rho - rho_ref) and rho the absolute
// one; fp[0..8] receive the post-collision values in stored form.  Eq. 14 in
// stored form is f_eq - w_i rho_ref = w_i (drho + rho P_i(u)), P_i = 3 e.u +
// 4.5 (e.u)^2 - 1.5 u^2; opposite directions share the even part of P.
//
// FP32: Eq. 13 as it stands, f + omega (f_eq - f).  Where the flow is
// uniform the same rounding repeats at every node and step and builds up; the
// shorter form below drifted by 3e-8 of the momentum per step in FP32 for
// tau = 1 (omega / 3 and omega / 12 both round up), and the FP32 kernels that
// carry the large lattices wait for memory, not for these instructions.
__device__ __forceinline__ void relax(const Consts<float> &K, const float *f, float drho,
                                      float rho, float mx, float my, float *fp)
{
    const float inv_rho = frcp(rho), omega = K.omega;
    const float ux = mx * inv_rho, uy = my * inv_rho;
    const float usq = 1.5f * (ux * ux + uy * uy);
    const float w1 = 1.0f / 9.0f, w5 = 1.0f / 36.0f;
    {
        const float ex2 = 4.5f * ux * ux - usq, ey2 = 4.5f * uy * uy - usq;
        const float ax = w1 * (drho + rho * ex2), bx = w1 * rho * 3.0f * ux;
        const float ay = w1 * (drho + rho * ey2), by = w1 * rho * 3.0f * uy;
        fp[1] = f[1] + omega * ((ax + bx) - f[1]);
        fp[3] = f[3] + omega * ((ax - bx) - f[3]);
        fp[2] = f[2] + omega * ((ay + by) - f[2]);
        fp[4] = f[4] + omega * ((ay - by) - f[4]);
    }
    {
        const float sp = ux + uy, sm = ux - uy;
        const float ep = 4.5f * sp * sp - usq, em = 4.5f * sm * sm - usq;
        const float a5 = w5 * (drho + rho * ep), b5 = w5 * rho * 3.0f * sp;
        const float a8 = w5 * (drho + rho * em), b8 = w5 * rho * 3.0f * sm;
        fp[5] = f[5] + omega * ((a5 + b5) - f[5]);
        fp[7] = f[7] + omega * ((a5 - b5) - f[7]);
        fp[8] = f[8] + omega * ((a8 + b8) - f[8]);
        fp[6] = f[6] + omega * ((a8 - b8) - f[6]);
    }
    // The rest population takes what the moving ones leave of the density:
    // in exact arithmetic this equals f_0 + omega (f_0^eq - f_0) with
    // f_0 = drho - sum_{i>0} f_i, and it keeps the collision's mass exact
    // instead of biased by the rounding of f_eq.
    fp[0] = drho - (((fp[1] + fp[2]) + (fp[3] + fp[4])) +
                    ((fp[5] + fp[6]) + (fp[7] + fp[8])));
}
// FP64, where every instruction of the narrow pipe counts: with e_ab =
// m_a u_b the even part of omega f_eq is, along an axis, omega/9 (drho +
// 3 e_xx - 1.5 e_yy) and, along a diagonal, omega/36 (drho + 3 (e_xx + e_yy)
// +- 9 e_xy), and the odd part omega w_i 3 m.e_i: two fused multiply-adds
// per population finish f* = (1 - omega) f + even + odd.  The FP64 step is
// bound by that pipe (82 % busy); this form, the shared row sums of the
// stencils, log_tab and rcp_nr together took a 1024 x 1024 periodic CS step
// from 325 to 252 us.
__device__ __forceinline__ void relax(const Consts<double> &K, const double *f, double drho,
                                      double rho, double mx, double my, double *fp)
{
    const double ir = frcp(rho);
    const double ux = mx * ir, uy = my * ir;
    const double exx = mx * ux, eyy = my * uy, exy = mx * uy;
    const double t = K.o9 * drho;
    {
        const double ax = K.o3 * exx + (K.no6 * eyy + t);
        const double ay = K.o3 * eyy + (K.no6 * exx + t);
        fp[1] = K.o3 * mx + (K.om1 * f[1] + ax);
        fp[3] = -K.o3 * mx + (K.om1 * f[3] + ax);
        fp[2] = K.o3 * my + (K.om1 * f[2] + ay);
        fp[4] = -K.o3 * my + (K.om1 * f[4] + ay);
    }
    {
        const double sp = mx + my, sm = mx - my;
        const double s = K.o12 * (exx + eyy) + 0.25 * t;
        const double ap = K.o4 * exy + s, am = -K.o4 * exy + s;
        fp[5] = K.o12 * sp + (K.om1 * f[5] + ap);
        fp[7] = -K.o12 * sp + (K.om1 * f[7] + ap);
        fp[8] = K.o12 * sm + (K.om1 * f[8] + am);
        fp[6] = -K.o12 * sm + (K.om1 * f[6] + am);
    }
    fp[0] = drho - (((fp[1] + fp[2]) + (fp[3] + fp[4])) +
                    ((fp[5] + fp[6]) + (fp[7] + fp[8])));
}

}  // namespace cplbm

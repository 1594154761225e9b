// Many steps of a small lattice, or of a batch of small ones, in one launch:
// every CTA keeps its rectangle of the lattice in shared memory for the
// whole call and exchanges only a three-node rim with its neighbours in each
// step.  Single steps, larger lattices and FP16 storage run on the tile
// kernels (step_impl.cuh).
//
// Why.  A lattice of a few hundred thousand nodes is a microsecond of work
// for the whole GPU, but the tile kernels pay a launch, the loads' latency
// and the drain of the grid in every step (9 us for 256 x 128 FP32), and
// their tiles leave most SMs idle (64 x 64 FP64: four tiles of 32 x 32, each
// bound by the FP64 pipe of its own SM, 57 us).  Here the lattice is cut so
// that every SM gets one rectangle, of any size, and a step costs the
// arithmetic of that rectangle plus one trip through L2.  Measured per step,
// tile kernels (default shape, 16-step graphs) -> here: FP32 64 x 64 20.9 ->
// 1.7 us, 256 x 128 6.7 -> 2.5, 512 x 512 7.5 -> 5.2, 704 x 704 9.6 -> 8.2;
// FP64 64 x 64 47 -> 5.6 us, 256 x 256 39 -> 21, 500 x 200 40 -> 28, 512 x 512
// 74 -> 64.  What bounds it: up to some 30 000 nodes the exchange and the
// barriers (about 1.5 us), beyond that FP64 the FP64 units, FP32 issue.
//
// State in shared memory (tile w x h, cell of node (x, y) at row y + 3,
// column x + 4 of a plane):
//   F[0..8]  post-collision populations in the in-place (AA) order of the
//            tile kernels: an even step of the call leaves f*_i in slot
//            opp(i) of its node, an odd one in slot i of x + e_i, so that
//            every slot a node reads is one it writes and no barrier stands
//            between the two;
//   R        stored density on the tile and two nodes around it (three
//            columns beside the rows next to a wall, for Eq. 28);
//   M        mu on the tile and one node around it.
// A step: mu, then force and collision, publish the rim, receive the
// neighbours' rims, then the next density, which needs all populations that
// stream into the tile and the two nodes around it: the rims are three
// nodes wide.
//
// Exchange.  A published value is one 64-bit word, the FP32 value beside a
// 32-bit tag that numbers the step (FP64: two words of 32 bits and a tag
// each), written and read with single relaxed 64-bit accesses.  The receiver
// polls the words themselves until they carry the step's tag, so there are
// no flags and no fences: one trip to L2 and back instead of four.  Two
// generations of words alternate.  A CTA overwrites the words of step k in
// step k + 2, after it has received its neighbours' words of step k + 1,
// which each of them published only after it had received all words of
// step k (a block barrier stands between).  The launch is cooperative, so
// all CTAs are resident and every wait ends; it is bounded all the same
// (Lattice::wait_cycles).  A CTA stores its part of the state, populations and
// density, once it has received every rim of the call; one that gives up
// raises ERR_WAIT_TIMEOUT and stores nothing.  Others may have finished by
// then, and the host counts the steps of the call: a lattice whose time-out
// has been reported is inconsistent until it is initialised or loaded again.
#pragma once
#include <type_traits>

#include "resident.h"
#include "step_impl.cuh"

namespace cplbm {

// ---------------------------------------------------------------------------
// Exchange words.
// ---------------------------------------------------------------------------
template <class real> struct Word;
template <> struct Word<float> {
    using type = unsigned long long;
    static __device__ __forceinline__ void put(type *p, float v, unsigned tag)
    {
        const unsigned long long w = (unsigned long long)tag << 32 | __float_as_uint(v);
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;\n" ::"l"(p), "l"(w) : "memory");
    }
    static __device__ __forceinline__ type get(const type *p)
    {
        type w;
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];\n" : "=l"(w) : "l"(p) : "memory");
        return w;
    }
    static __device__ __forceinline__ bool is(type w, unsigned tag)
    {
        return (unsigned)(w >> 32) == tag;
    }
    static __device__ __forceinline__ float value(type w) { return __uint_as_float((unsigned)w); }
};
template <> struct Word<double> {
    using type = ulonglong2;
    static __device__ __forceinline__ void put(type *p, double v, unsigned tag)
    {
        const unsigned long long t = (unsigned long long)tag << 32;
        const unsigned long long a = t | (unsigned)__double2loint(v);
        const unsigned long long b = t | (unsigned)__double2hiint(v);
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};\n" ::"l"(p), "l"(a), "l"(b)
                     : "memory");
    }
    static __device__ __forceinline__ type get(const type *p)
    {
        type w;
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];\n"
                     : "=l"(w.x), "=l"(w.y) : "l"(p) : "memory");
        return w;
    }
    static __device__ __forceinline__ bool is(type w, unsigned tag)
    {
        return (unsigned)(w.x >> 32) == tag && (unsigned)(w.y >> 32) == tag;
    }
    static __device__ __forceinline__ double value(type w)
    {
        return __hiloint2double((int)(unsigned)w.y, (int)(unsigned)w.x);
    }
};

#ifdef CPLBM_CHECK_BOUNDS
#define CPLBM_IN_XCHG(L, p) ::cplbm::in_buffer(L, (L).xchg, (L).b_xchg, p, sizeof(*(p)))
#else
#define CPLBM_IN_XCHG(L, p) true
#endif

// ---------------------------------------------------------------------------
// A thread's nodes of one column, (x, y) .. (x, y + N - 1), N one or two.
// FP32 computes on packed pairs with the functions of the two-nodes-per-lane
// path: two nodes per thread, or, on tiles of at most a node per thread, one
// (the other half of each pair idle), which halves the chain of shared-memory
// accesses that a step of a small tile waits for.  FP64: one, since an FP64
// instruction holds the SM quarter's FP64 unit for the same time however few
// lanes are active, so on small tiles it is the number of instructions per
// thread that counts.  i: index of the lower node in a field of row width W.
// ---------------------------------------------------------------------------
struct Rows2 {
    Row2 d, m, u;
};
template <int N>
__device__ __forceinline__ Rows2 rows2(const float *s, int i, int W)
{
    Row<float> r[4];
#pragma unroll
    for (int j = 0; j < 2 + N; ++j) r[j] = row_of(s, i + (j - 1) * W);
    if (N == 1) r[3] = r[2];
    auto two = [&](int a) {
        return Row2{make_float2(r[a].c, r[a + 1].c), make_float2(r[a].h, r[a + 1].h),
                    make_float2(r[a].d, r[a + 1].d)};
    };
    return {two(0), two(1), two(2)};
}
template <int N>
__device__ __forceinline__ void column_mu(const Consts<float> &K, float ref, const float *R,
                                          int i, int W, float (&mu)[N])
{
    const Rows2 r = rows2<N>(R, i, W);
    const float2 m = pfma(p2(-K.kappa), lap2(r.u, r.m, r.d),
                          mu_bulk2(K.eos, padd(r.m.c, p2(ref))));
    mu[0] = m.x;
    if constexpr (N == 2) mu[1] = m.y;
}
__device__ __forceinline__ void column_mu(const Consts<double> &K, double ref, const double *R,
                                          int i, int W, double (&mu)[1])
{
    mu[0] = mu_of(K, R[i] + ref,
                  lap6(row_of(R, i + W), row_of(R, i), row_of(R, i - W)));
}
template <int N>
__device__ __forceinline__ void column_collide(const Consts<float> &K, float ref, const float *R,
                                               int i, int W, const float *M, int j, int MW,
                                               const float (&f)[N][9], float (&fp)[N][9])
{
    const Rows2 r = rows2<N>(R, i, W), m = rows2<N>(M, j, MW);
    float2 grx, gry, gmx, gmy, g[9], gp[9];
    grad2(r.u, r.m, r.d, grx, gry);
    grad2(m.u, m.m, m.d, gmx, gmy);
    const float2 drho = r.m.c, rho = padd(drho, p2(ref)), third = p2(1.0f / 3.0f);
    const float2 Fx = psub(pmul(grx, third), pmul(rho, gmx));
    const float2 Fy = psub(pmul(gry, third), pmul(rho, gmy));
#pragma unroll
    for (int k = 1; k < 9; ++k) g[k] = make_float2(f[0][k], f[N - 1][k]);
    collide2(g, drho, rho, Fx, Fy, p2(K.tau), p2(K.omega), gp);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        fp[0][k] = gp[k].x;
        if constexpr (N == 2) fp[1][k] = gp[k].y;
    }
}
__device__ __forceinline__ void column_collide(const Consts<double> &K, double ref,
                                               const double *R, int i, int W, const double *M,
                                               int j, int MW, const double (&f)[1][9],
                                               double (&fp)[1][9])
{
    double grx, gry, gmx, gmy, mx, my;
    grad12(row_of(R, i + W), row_of(R, i), row_of(R, i - W), grx, gry);
    grad12(row_of(M, j + MW), row_of(M, j), row_of(M, j - MW), gmx, gmy);
    const double drho = R[i], rho = drho + ref;
    force_momentum(K, f[0], rho, grx, gry, gmx, gmy, mx, my);
    relax(K, f[0], drho, rho, mx, my, fp[0]);
}

// Density v of node (r, x) as a whole into generation gen: the partial sums
// that load_rho_stored would add to it become zero.
template <class rt>
__device__ __forceinline__ void store_rho_whole(const Lattice &L, int gen, int r, int x, rt v)
{
    put_rho(L, gen, (rt *)L.rho[gen], fidx(L, r, x), v);
    const int bx = tile_x(L, x), by = tile_y(L, r);
    const int lx = x - bx * L.tx, ly = r - by * L.ty;
    const bool left = lx == 0, right = lx == min(L.tx, L.nx - bx * L.tx) - 1;
    const bool below = ly == 0 && !(L.walls && r == 0);
    const bool above = ly == min(L.ty, L.nyf - by * L.ty) - 1 && !(L.walls && r == L.nyf - 1);
    rt *const *ring = (rt *const *)L.ring[gen];
    auto clear = [&](int c) { put_ring(L, gen, ring, c, ring_index(L, c, bx, by, r, x), rt(0)); };
    if (left) clear(R_L);
    if (right) clear(R_R);
    if (below) {
        clear(R_B);
        if (left) clear(R_BL);
        if (right) clear(R_BR);
    }
    if (above) {
        clear(R_T);
        if (left) clear(R_TL);
        if (right) clear(R_TR);
    }
}

// n / w for 0 <= n < 2^20, w >= 1, with iw = 1 / w in FP32: the product is
// off by less than 2^-3 of the distance between quotients' edges.
__device__ __forceinline__ int div_by(int n, float iw) { return (int)(((float)n + 0.5f) * iw); }

// A node of another tile whose populations a thread receives in every step:
// its words' offset in a generation, its cell, the populations needed, and
// whether its row is the first or last fluid row of a walled lattice.
struct RimNode {
    long long at;
    int cell;
    unsigned need;     // bit i: population i; 0: none
    bool b, t;
};

// WALLS: the variant of lattices with walls (batches: of any lattice).
template <class S, int NT, int N, bool BATCH, bool WALLS>
__global__ void __launch_bounds__(NT, 1) resident_kernel(const ResidentArgs A)
{
    using real = typename S::real;
    using pop_t = typename S::pop_t;
    using rho_t = typename S::rho_t;
    using WD = Word<real>;
    static_assert(N == 1 || sizeof(real) == 4, "FP64: one node per thread");
    static_assert(sizeof(pop_t) == sizeof(real) && sizeof(rho_t) == sizeof(real),
                  "populations kept as stored");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Lattice sL;
    int x0, y0, w, h;
    if (BATCH) {
        const ResidentTile t = A.tiles[blockIdx.x];
        const int *src = reinterpret_cast<const int *>(A.lats + t.inst);
        for (int q = threadIdx.x; q < (int)(sizeof(Lattice) / sizeof(int)); q += NT)
            reinterpret_cast<int *>(&sL)[q] = src[q];
        x0 = t.x0;
        y0 = t.y0;
        w = t.w;
        h = t.h;
        __syncthreads();
    } else {
        const int by = blockIdx.x / A.gx, bx = blockIdx.x - by * A.gx;
        x0 = bx * A.w;
        y0 = by * A.h;
        w = min(A.w, A.L.nx - x0);
        h = min(A.h, A.L.nyf - y0);
    }
    const Lattice &L = BATCH ? sL : A.L;
    const Geo g(w, h);
    const int fw = g.fw, fp_ = g.fp, rw = g.rw, mw = g.mw;
    real *const F = reinterpret_cast<real *>(smem_raw);
    real *const R = F + 9 * fp_;
    real *const M = R + rw * (h + 5);
    const Consts<real> &K = consts<real>(L);
    const real ref = S::offset ? K.rho_ref : real(0);
    const bool walls = WALLS && L.walls != 0;
    const bool wb = walls && y0 == 0, wt = walls && y0 + h == L.nyf;
    const int tid = threadIdx.x;
    typename WD::type *const X = (typename WD::type *)L.xchg;

    auto cell = [&](int x, int y) { return (y + RIM) * fw + x + HX; };
    auto fluid = [&](int y) { return !walls || (unsigned)(y0 + y) < (unsigned)L.nyf; };
    auto first_row = [&](int y) { return walls && y0 + y == 0; };
    auto last_row = [&](int y) { return walls && y0 + y == L.nyf - 1; };
    // nodes whose density a step needs
    auto in_r = [&](int x, int y) {
        if (!fluid(y) || y < -2 || y > h + 1) return false;
        const int e = (wb && y == 0) || (wt && y == h - 1) ? 3 : 2;
        return x >= -e && x < w + e;
    };
    // population i of the node at cell c before a collision: the place a
    // step of kind S (0 even, 1 odd in the call) reads it from; b, t: the
    // node's row is the first / last fluid row of a walled lattice
    auto pull = [&](int kind, int i, int c, bool b, bool t) -> real & {
        const bool own = kind == 0 || (ey(i) > 0 && b) || (ey(i) < 0 && t);
        return own ? F[i * fp_ + c] : F[opp(i) * fp_ + c - (ey(i) * fw + ex(i))];
    };

    // 1. The state: populations of the tile in natural order (the place an
    //    even step reads), the density around it.
    const float iw = 1.0f / (float)w;
    {
        const pop_t *P = (const pop_t *)L.pops;
        for (int n = tid; n < w * h; n += NT) {
            const int y = div_by(n, iw), x = n - y * w, c = cell(x, y);
#pragma unroll
            for (int i = 1; i < 9; ++i) {
                const pop_t *q = P + aa_read_index(L, A.parity, i, y0 + y, x0 + x);
                F[i * fp_ + c] = CPLBM_IN_POPS(L, q, 1) ? (real)*q : real(0);
            }
        }
        const float irw = 1.0f / (float)rw;
        for (int n = tid; n < rw * (h + 4); n += NT) {
            const int y = div_by(n, irw) - 2, x = n - (y + 2) * rw - 3;
            if (!fluid(y)) {
                R[n] = real(0.1);  // an ordinary density: enters only values no one reads
                continue;
            }
            R[n] = load_rho_stored<S>(L, A.parity, walls ? y0 + y : wrapi(y0 + y, L.nyf),
                                      wrapi(x0 + x, L.nx));
        }
    }
    // the rim nodes of this thread (the plan's tiles have at most RIM_NODES
    // per thread)
    RimNode rim[RIM_NODES];
    {
        const int side = walls ? HX : RIM;    // halo columns that may be needed
        const int hw = w + 2 * side, nrow = RIM * hw, nhalo = 2 * nrow + 2 * side * h;
        const float ihw = 1.0f / (float)hw, ih = 1.0f / (float)h;
#pragma unroll
        for (int s = 0; s < RIM_NODES; ++s) {
            const int n = tid + s * NT;
            int x, y;
            if (n < 2 * nrow) {
                const int q = div_by(n, ihw);
                x = n - q * hw - side;
                y = q < RIM ? q - RIM : h + q - RIM;
            } else {
                const int q = n - 2 * nrow, col = div_by(q, ih);
                y = q - col * h;
                x = col < side ? col - side : w + col - side;
            }
            RimNode &e = rim[s];
            e.need = 0;
            if (n >= nhalo || !fluid(y)) continue;
            e.b = first_row(y);
            e.t = last_row(y);
            e.cell = cell(x, y);
            e.at = fidx(L, walls ? y0 + y : wrapi(y0 + y, L.nyf), wrapi(x0 + x, L.nx));
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const bool back = (ey(i) < 0 && e.b) || (ey(i) > 0 && e.t);  // bounces back
                if (back ? in_r(x, y) : in_r(x + ex(i), y + ey(i))) e.need |= 1u << i;
            }
        }
    }
    __syncthreads();

    const int cols = (h + N - 1) / N, mcols = (h + 2 + N - 1) / N, nrx = w + 4;
    const float imw = 1.0f / (float)mw, inrx = 1.0f / (float)nrx;
    auto step = [&](auto kind_c, int k) -> bool {
        constexpr int kind = decltype(kind_c)::value;
        const unsigned tag = A.tag + (unsigned)k;
        const bool last = k == A.nsteps - 1;
        typename WD::type *const Xk = X + (long long)(tag & 1u) * 9 * L.plane;

        // 2. Eq. 28 on the solid rows, then mu on the tile and one node
        //    around it.
        if (wb || wt) {
            for (int n = tid; n < 2 * nrx; n += NT) {
                const bool top = n >= nrx;
                if (!(top ? wt : wb)) continue;
                const int x = n - (top ? nrx : 0) - 2;
                const real *s = R + ((top ? h - 1 : 0) + 2) * rw + x + 3;
                R[((top ? h : -1) + 2) * rw + x + 3] = real(2.0 / 3.0) * s[0] +
                                                      real(1.0 / 6.0) * s[-1] +
                                                      real(1.0 / 6.0) * s[1];
            }
            __syncthreads();
        }
        for (int n = tid; n < mw * mcols; n += NT) {
            const int yy = div_by(n, imw), x = n - yy * mw - 1, y = N * yy - 1;
            real m[N];
            column_mu(K, ref, R, (y + 2) * rw + x + 3, rw, m);
            real *q = M + (y + 1) * mw + x + 1;
#pragma unroll
            for (int j = 0; j < N; ++j)
                q[j * mw] = wb && y + j == -1 ? K.mu_bottom : (wt && y + j == h ? K.mu_top : m[j]);
        }
        __syncthreads();
        if (wt && L.top_mode == 0) {  // the top row copies its fluid neighbour
            for (int x = tid; x < mw; x += NT) M[(h + 1) * mw + x] = M[h * mw + x];
            __syncthreads();
        }

        // 3. Force, collision, in-place streaming; the rim goes out.
        for (int n = tid; n < w * cols; n += NT) {
            const int yy = div_by(n, iw), x = n - yy * w, y = N * yy;
            const int c = cell(x, y);
            real f[N][9], fp[N][9];
#pragma unroll
            for (int j = 0; j < N; ++j)
#pragma unroll
                for (int i = 1; i < 9; ++i)
                    f[j][i] = pull(kind, i, c + j * fw, first_row(y + j), last_row(y + j));
            column_collide(K, ref, R, (y + 2) * rw + x + 3, rw, M, (y + 1) * mw + x + 1, mw, f,
                           fp);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                if (j > 0 && y + j >= h) break;
                const int yj = y + j, cj = c + j * fw;
                const bool b = first_row(yj), t = last_row(yj);
                F[cj] = fp[j][0];
                // kind 0: slot opp(i) of the node; kind 1: slot i of x + e_i,
                // or opp(i) of the node where that is solid
#pragma unroll
                for (int i = 1; i < 9; ++i) pull(kind, opp(i), cj, b, t) = fp[j][i];
                const int mx = walls ? HX : RIM;
                if (yj < RIM || yj >= h - RIM || x < mx || x >= w - mx) {
                    typename WD::type *q = Xk + fidx(L, y0 + yj, x0 + x);
#pragma unroll
                    for (int i = 0; i < 9; ++i, q += L.plane)
                        if (CPLBM_IN_XCHG(L, q)) WD::put(q, fp[j][i], tag);
                }
            }
        }

        // 4. The neighbours' rims: the populations that stream into a node
        //    whose density the next step needs.  (No barrier since step 3:
        //    the slots written here are read by no node of this tile there.)
        bool ok = true;
#pragma unroll
        for (int s = 0; s < RIM_NODES; ++s) {
            const RimNode &e = rim[s];
            unsigned need = e.need;
            const typename WD::type *q = Xk + e.at;
            const long long t0 = clock64();
            while (need) {
                if (clock64() - t0 >= L.wait_cycles) {
                    ok = false;
                    break;
                }
                typename WD::type v[9];
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    if (need >> i & 1)
                        v[i] = CPLBM_IN_XCHG(L, q + i * L.plane) ? WD::get(q + i * L.plane)
                                                                 : typename WD::type{};
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    if ((need >> i & 1) && WD::is(v[i], tag)) {
                        need &= ~(1u << i);
                        if (i == 0) F[e.cell] = WD::value(v[0]);
                        else pull(kind, opp(i), e.cell, e.b, e.t) = WD::value(v[i]);
                    }
            }
        }
        if (__syncthreads_or(!ok)) return false;
        if (last) {  // every rim of the call is here: the populations back
            pop_t *P = (pop_t *)L.pops;
            for (int n = tid; n < w * h; n += NT) {
                const int y = div_by(n, iw), x = n - y * w, c = cell(x, y);
#pragma unroll
                for (int i = 1; i < 9; ++i) {
                    pop_t *q = P + aa_write_index(L, (A.parity + k) & 1, i, y0 + y, x0 + x);
                    if (CPLBM_IN_POPS(L, q, 1))
                        *q = (pop_t)pull(kind, opp(i), c, first_row(y), last_row(y));
                }
            }
        }

        // 5. The next density (tile-kernel order of the sum).
        constexpr int next = kind ^ 1;
        auto density = [&](int x, int y) {
            const int c = cell(x, y);
            const bool b = first_row(y), t = last_row(y);
            const real same = F[c] + pull(next, 1, c, b, t) + pull(next, 3, c, b, t);
            const real up = pull(next, 2, c, b, t) + pull(next, 5, c, b, t) + pull(next, 6, c, b, t);
            const real down = pull(next, 4, c, b, t) + pull(next, 8, c, b, t) + pull(next, 7, c, b, t);
            R[(y + 2) * rw + x + 3] = same + up + down;
        };
        for (int n = tid; n < nrx * (h + 4); n += NT) {
            const int yy = div_by(n, inrx), x = n - yy * nrx - 2, y = yy - 2;
            if (fluid(y)) density(x, y);
        }
        if (WALLS && tid < 4) {  // beside the rows next to a wall
            const bool top = tid & 2;
            if (top ? wt : wb) density(tid & 1 ? w + 2 : -3, top ? h - 1 : 0);
        }
        __syncthreads();
        return true;
    };
    for (int k = 0; k < A.nsteps; k += 2) {
        if (!step(std::integral_constant<int, 0>{}, k) ||
            (k + 1 < A.nsteps && !step(std::integral_constant<int, 1>{}, k + 1))) {
            if (tid == 0 && L.err) atomicOr(L.err, ERR_WAIT_TIMEOUT);
            return;
        }
    }

    // 6. The density back as a whole; the last step stored the populations.
    const int gen = (A.parity + A.nsteps) & 1;
    for (int n = tid; n < w * h; n += NT) {
        const int y = div_by(n, iw), x = n - y * w;
        store_rho_whole(L, gen, y0 + y, x0 + x, (rho_t)R[(y + 2) * rw + x + 3]);
    }
}

// Launch of one precision: threads 256, or RESIDENT_THREADS with two FP32
// nodes per thread (ResidentPlan::threads).
template <class S>
cudaError_t launch_resident_t(const ResidentArgs &a, bool batch, int grid, int threads,
                              size_t smem, cudaStream_t s)
{
    constexpr int NT = resident_threads(sizeof(typename S::real) == 8),
                  N = sizeof(typename S::real) == 8 ? 1 : 2;
    void *const kern[2][3] = {{(void *)resident_kernel<S, 256, 1, false, false>,
                               (void *)resident_kernel<S, 256, 1, false, true>,
                               (void *)resident_kernel<S, 256, 1, true, true>},
                              {(void *)resident_kernel<S, NT, N, false, false>,
                               (void *)resident_kernel<S, NT, N, false, true>,
                               (void *)resident_kernel<S, NT, N, true, true>}};
    void *k = kern[threads == NT][batch ? 2 : a.L.walls ? 1 : 0];
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)RESIDENT_SMEM);
    if (e != cudaSuccess) return e;
    void *args[] = {const_cast<ResidentArgs *>(&a)};
    return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(threads), args, smem, s);
}

}  // namespace cplbm

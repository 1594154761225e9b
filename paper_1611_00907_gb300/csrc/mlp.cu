// Small BF16 multilayer perceptron with FP32 accumulation for the learned
// warm start: hand-written inference and training kernels on the tensor
// cores (mma.sync m16n8k16 BF16 -> FP32).
//
// Network: 16 inputs (the caller's features, zero-padded) -> 3 hidden layers
// of 128 tanh units -> 16 outputs (zero-padded; linear).  Each layer keeps
// FP32 master weights (Adam state beside them) and two BF16 copies, for the
// forward product and for back-propagation.
//
// Everything here is latency: the network is 37 000 parameters, an iteration
// of 1024 samples 0.2 GFLOP.  A CTA takes 16 samples at a time, so that a
// thousand samples are 64 CTAs, and its eight warps split each layer's
// outputs; a warp's weights go straight from L2 to registers, in the order
// the MMA wants them (fragment order, written by the Adam kernel), all loads
// ahead of the first product.  Activations and deltas stay in padded shared
// memory and reach the MMA by ldmatrix, transposed for the weight gradients.
// Training is full-batch gradient descent: a CTA back-propagates its samples
// and adds its weight gradients into FP32 accumulators (pairs per reduction);
// the Adam kernel then updates every weight.  1024 samples: 161 us an
// iteration with 64 samples and four warps per CTA, weights and activations
// read from unpadded shared memory; now 14 us, a chain of eight products with
// their barriers, the gradient's reductions and the Adam pass, whose launches
// overlap by programmatic dependent launch.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <new>
#include <string>

#include "../../include/cplbm.h"
#include "cplbm_internal.h"  // dev_alloc / dev_free
#include "trace.h"

namespace cplbm_mlp {

constexpr int DIN = 16, H = 128, DOUT = 16, NL = 4;
constexpr int SAMPLES = 16, WARPS = 8, THREADS = 32 * WARPS;
constexpr int MAX_CTAS = 152;   // one per SM; more samples take several rounds
__host__ __device__ constexpr int layer_k(int l) { return l == 0 ? DIN : H; }
__host__ __device__ constexpr int layer_n(int l) { return l == NL - 1 ? DOUT : H; }

// Groups of SAMPLES samples.  (Counted in groups, the loops over them stay
// within an int for every B.)
__host__ __device__ constexpr int groups(int B) { return B / SAMPLES + (B % SAMPLES != 0); }

// Offsets of layer l's weights [k][n] and biases in the flat parameter
// arrays (FP32 masters, gradients, Adam moments share the layout).
__host__ __device__ constexpr int w_off(int l)
{
    return l == 0 ? 0 : w_off(l - 1) + layer_k(l - 1) * layer_n(l - 1);
}
constexpr int NW = w_off(NL);
__host__ __device__ constexpr int b_off(int l)
{
    return l == 0 ? NW : b_off(l - 1) + layer_n(l - 1);
}
constexpr int NPARAM = b_off(NL);

struct Params {
    const __nv_bfloat16 *wt;  // forward weights in fragment order, BF16, at w_off(l)
    const __nv_bfloat16 *w;   // back-propagation weights likewise
    const float *p;           // FP32 masters (biases read from here)
};

// Fragment order of a B operand of mma.m16n8k16 (PTX ISA; lane = 4 g + t):
// output column `col`, contraction index `kk` of KK.  A lane's four values of
// a 16-deep step lie together, two steps side by side where there are two,
// so that a lane's share of a column tile is a run of 16-byte words.
__host__ __device__ constexpr int frag_pos(int col, int kk, int KK)
{
    const int j = col / 8, g = col % 8, step = kk / 16, r = kk % 16;
    const int lane = 4 * g + (r % 8) / 2, e = (r & 1) + (r >= 8 ? 2 : 0);
    return KK == 16 ? (j * 32 + lane) * 4 + e
                    : ((j * (KK / 32) + step / 2) * 32 + lane) * 8 + (step & 1) * 4 + e;
}

// ---------------------------------------------------------------------------
// mma.m16n8k16 BF16 -> FP32 and its fragments.
// ---------------------------------------------------------------------------
struct FragA {
    unsigned r[4];
};
__device__ __forceinline__ void mma(float (&acc)[4], const FragA &a, unsigned b0, unsigned b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
        : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3])
        : "r"(a.r[0]), "r"(a.r[1]), "r"(a.r[2]), "r"(a.r[3]), "r"(b0), "r"(b1));
}
template <bool TRANS>
__device__ __forceinline__ FragA ldmatrix4(const __nv_bfloat16 *p)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(p);
    FragA f;
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                     : "=r"(f.r[0]), "=r"(f.r[1]), "=r"(f.r[2]), "=r"(f.r[3]) : "r"(s) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                     : "=r"(f.r[0]), "=r"(f.r[1]), "=r"(f.r[2]), "=r"(f.r[3]) : "r"(s) : "memory");
    return f;
}
// A operand from row-major [16][...] at column k0 (row stride LD).
template <int LD>
__device__ __forceinline__ FragA frag_a(const __nv_bfloat16 *m, int k0)
{
    const int lane = threadIdx.x & 31;
    return ldmatrix4<false>(m + (lane & 15) * LD + k0 + (lane >> 4) * 8);
}
// A operand of the transpose: rows are columns k0 .. k0 + 15 of m, the
// contraction runs over m's 16 rows.
template <int LD>
__device__ __forceinline__ FragA frag_at(const __nv_bfloat16 *m, int k0)
{
    const int lane = threadIdx.x & 31;
    return ldmatrix4<true>(m + ((lane & 7) + (lane >> 4) * 8) * LD + k0 + ((lane >> 3) & 1) * 8);
}
// B operands of two column tiles n0, n0 + 8 of m [16][...], contraction over
// its rows: {b0, b1} of the first tile, then of the second.
template <int LD>
__device__ __forceinline__ FragA frag_b2(const __nv_bfloat16 *m, int n0)
{
    const int lane = threadIdx.x & 31;
    return ldmatrix4<true>(m + ((lane & 7) + ((lane >> 3) & 1) * 8) * LD + n0 + (lane >> 4) * 8);
}

// Rows of 16 and 128 values, padded so that the eight rows an ldmatrix reads
// lie in different banks.
constexpr int LD16 = 24, LD128 = 136;

struct Smem {
    __nv_bfloat16 in[SAMPLES * LD16];           // input of layer 0, [s][k]
    __nv_bfloat16 act[NL - 1][SAMPLES * LD128]; // inputs of layers 1 .. 3
    __nv_bfloat16 dout[SAMPLES * LD16];         // output delta [s][n]
    __nv_bfloat16 dlt[2][SAMPLES * LD128];      // deltas of the hidden layers
    float out[SAMPLES * DOUT];
};

// A warp's weights: its two column tiles of each 128-column layer (layer 3's
// forward product has two tiles in all: one each for the first two warps).
struct Weights {
    uint2 in[2];          // layer 0 forward (16 deep)
    uint4 f1[2][4], f2[2][4], f3[4];
    uint2 b3[2];          // back-propagation through layer 3 (16 deep)
    uint4 b2[2][4], b1[2][4];
};
__device__ __forceinline__ uint4 load16(const __nv_bfloat16 *w, int tile, int k2)
{
    return reinterpret_cast<const uint4 *>(w)[(tile * 4 + k2) * 32 + (threadIdx.x & 31)];
}
template <bool BACK>
__device__ __forceinline__ void load_weights(const Params &P, Weights &W)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int j = 2 * warp + q;
        W.in[q] = reinterpret_cast<const uint2 *>(P.wt + w_off(0))[j * 32 + lane];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            W.f1[q][k] = load16(P.wt + w_off(1), j, k);
            W.f2[q][k] = load16(P.wt + w_off(2), j, k);
        }
    }
    if (warp < 2)
#pragma unroll
        for (int k = 0; k < 4; ++k) W.f3[k] = load16(P.wt + w_off(3), warp, k);
    if (BACK) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int j = 2 * warp + q;
            W.b3[q] = reinterpret_cast<const uint2 *>(P.w + w_off(3))[j * 32 + lane];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                W.b2[q][k] = load16(P.w + w_off(2), j, k);
                W.b1[q][k] = load16(P.w + w_off(1), j, k);
            }
        }
    }
}

// acc[q] = (16 x 128 at m) * (the warp's column tile q), contraction in
// ascending order.
template <int NT>
__device__ __forceinline__ void product(const __nv_bfloat16 *m, const uint4 (*w)[4],
                                        float (&acc)[NT][4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const FragA a0 = frag_a<LD128>(m, 32 * k), a1 = frag_a<LD128>(m, 32 * k + 16);
#pragma unroll
        for (int q = 0; q < NT; ++q) mma(acc[q], a0, w[q][k].x, w[q][k].y);
#pragma unroll
        for (int q = 0; q < NT; ++q) mma(acc[q], a1, w[q][k].z, w[q][k].w);
    }
}
// Two adjacent values as a BF16 pair at row r, column c of m.
__device__ __forceinline__ void put2(__nv_bfloat16 *m, int r, int c, float x, float y)
{
    *reinterpret_cast<__nv_bfloat162 *>(m + r * LD128 + c) = __floats2bfloat162_rn(x, y);
}
__device__ __forceinline__ float2 get2(const __nv_bfloat16 *m, int r, int c)
{
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(m + r * LD128 + c));
}
// tanh(acc + bias) of the warp's tiles into m.
__device__ __forceinline__ void activate(const float (&acc)[2][4], const float2 (&bias)[2],
                                         __nv_bfloat16 *m)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int c = ((threadIdx.x >> 5) * 2 + q) * 8 + 2 * t;
        put2(m, g, c, tanhf(acc[q][0] + bias[q].x), tanhf(acc[q][1] + bias[q].y));
        put2(m, g + 8, c, tanhf(acc[q][2] + bias[q].x), tanhf(acc[q][3] + bias[q].y));
    }
}
struct Biases {
    float2 h[NL - 1][2], out;
};
__device__ __forceinline__ void load_biases(const Params &P, Biases &B)
{
    const int warp = threadIdx.x >> 5, t = threadIdx.x & 3;
#pragma unroll
    for (int l = 0; l < NL - 1; ++l)
#pragma unroll
        for (int q = 0; q < 2; ++q)
            B.h[l][q] = *reinterpret_cast<const float2 *>(P.p + b_off(l) + (2 * warp + q) * 8 + 2 * t);
    if (warp < 2) B.out = *reinterpret_cast<const float2 *>(P.p + b_off(NL - 1) + warp * 8 + 2 * t);
}

// Forward pass of the CTA's 16 samples from s0 on: every layer's input and
// the FP32 outputs in S.  Ends with a barrier.
__device__ __forceinline__ void forward(const Weights &W, const Biases &Bs, Smem &S,
                                        const float *X, int nin, int B, int s0)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {
        const int s = threadIdx.x / DIN, k = threadIdx.x % DIN;
        const float v = s0 + s < B && k < nin ? X[(long long)(s0 + s) * nin + k] : 0.f;
        S.in[s * LD16 + k] = __float2bfloat16(v);
    }
    __syncthreads();
    {
        float acc[2][4] = {};
        const FragA a = frag_a<LD16>(S.in, 0);
        mma(acc[0], a, W.in[0].x, W.in[0].y);
        mma(acc[1], a, W.in[1].x, W.in[1].y);
        activate(acc, Bs.h[0], S.act[0]);
    }
    __syncthreads();
    {
        float acc[2][4] = {};
        product<2>(S.act[0], W.f1, acc);
        activate(acc, Bs.h[1], S.act[1]);
    }
    __syncthreads();
    {
        float acc[2][4] = {};
        product<2>(S.act[1], W.f2, acc);
        activate(acc, Bs.h[2], S.act[2]);
    }
    __syncthreads();
    if (warp < 2) {
        float acc[1][4] = {};
        product<1>(S.act[2], &W.f3, acc);
        const int g = lane >> 2, c = warp * 8 + 2 * (lane & 3);
        float *o = S.out + g * DOUT + c;
        o[0] = acc[0][0] + Bs.out.x;
        o[1] = acc[0][1] + Bs.out.y;
        o[8 * DOUT] = acc[0][2] + Bs.out.x;
        o[8 * DOUT + 1] = acc[0][3] + Bs.out.y;
    }
    __syncthreads();
}

// Programmatic dependent launch: a kernel lets its successor start while it
// runs, and touches memory only once its predecessor has ended.
__device__ __forceinline__ void after_predecessor()
{
    asm volatile("griddepcontrol.launch_dependents;\n griddepcontrol.wait;\n" ::: "memory");
}

__global__ void __launch_bounds__(THREADS, 1)
    mlp_infer_kernel(Params P, const float *X, int nin, float *Y, int nout, int B)
{
    __shared__ __align__(16) Smem S;
    Weights W;
    Biases Bs;
    load_weights<false>(P, W);
    load_biases(P, Bs);
    for (int q = blockIdx.x; q < groups(B); q += gridDim.x) {
        const int s0 = q * SAMPLES;
        forward(W, Bs, S, X, nin, B, s0);
        const int s = threadIdx.x / DOUT, c = threadIdx.x % DOUT;
        if (s0 + s < B && c < nout) Y[(long long)(s0 + s) * nout + c] = S.out[threadIdx.x];
        __syncthreads();
    }
}

__device__ __forceinline__ void add2(float *p, float x, float y)
{
    asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};\n" ::"l"(p), "f"(x), "f"(y)
                 : "memory");
}
// Weight gradient dW[k][n] += sum_s a[s][k] d[s][n] of the rows k0 .. k0 + 15
// and the column tiles n0 .. n0 + 8 (NT - 1) of a layer with N columns.
template <int LDA, int LDD, int N, int NT>
__device__ __forceinline__ void weight_grad(const __nv_bfloat16 *a, const __nv_bfloat16 *d,
                                            int k0, int n0, float *grad)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const FragA at = frag_at<LDA>(a, k0);
    float *o = grad + (k0 + g) * N + n0 + 2 * t;
#pragma unroll
    for (int q = 0; q < NT; q += 2) {
        const FragA b = frag_b2<LDD>(d, n0 + 8 * q);
        float x[4] = {}, y[4] = {};
        mma(x, at, b.r[0], b.r[1]);
        mma(y, at, b.r[2], b.r[3]);
        add2(o + 8 * q, x[0], x[1]);
        add2(o + 8 * q + 8 * N, x[2], x[3]);
        add2(o + 8 * q + 8, y[0], y[1]);
        add2(o + 8 * q + 8 + 8 * N, y[2], y[3]);
    }
}
// Delta of a hidden layer from acc = (delta above) W^T: acc (1 - a^2), a the
// layer's output; samples beyond B have a zero delta above.
__device__ __forceinline__ void hidden_delta(const float (&acc)[2][4], const __nv_bfloat16 *a,
                                             __nv_bfloat16 *d)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int c = ((threadIdx.x >> 5) * 2 + q) * 8 + 2 * t;
        const float2 u = get2(a, g, c), v = get2(a, g + 8, c);
        put2(d, g, c, acc[q][0] * (1.f - u.x * u.x), acc[q][1] * (1.f - u.y * u.y));
        put2(d, g + 8, c, acc[q][2] * (1.f - v.x * v.x), acc[q][3] * (1.f - v.y * v.y));
    }
}
// Bias gradient: column sums of a hidden layer's delta.
__device__ __forceinline__ void bias_grad(const __nv_bfloat16 *d, float *grad)
{
    if (threadIdx.x >= H) return;
    float sum = 0.f;
#pragma unroll
    for (int s = 0; s < SAMPLES; ++s) sum += __bfloat162float(d[s * LD128 + threadIdx.x]);
    atomicAdd(&grad[threadIdx.x], sum);
}

// Forward, mean-squared-error gradient, back-propagation and weight
// gradients of the CTA's samples; gradients are added into grad (FP32, the
// parameter layout) and, where it is wanted, the squared error into *loss.
__global__ void __launch_bounds__(THREADS, 1)
    mlp_train_kernel(Params P, const float *X, int nin, const float *T, int nout,
                     int B, float *grad, float *loss)
{
    __shared__ __align__(16) Smem S;
    Weights W;
    Biases Bs;
    const int warp = threadIdx.x >> 5;
    after_predecessor();
    load_weights<true>(P, W);
    load_biases(P, Bs);
    for (int q = blockIdx.x; q < groups(B); q += gridDim.x) {
        const int s0 = q * SAMPLES;
        forward(W, Bs, S, X, nin, B, s0);
        {   // output delta: d(mean sq error)/dy = 2 (y - t) / (B nout)
            const int s = threadIdx.x / DOUT, c = threadIdx.x % DOUT, gs = s0 + s;
            float d = 0.f, se = 0.f;
            if (gs < B && c < nout) {
                const float e = S.out[threadIdx.x] - T[(long long)gs * nout + c];
                se = e * e;
                d = 2.f * e / (float)(B * nout);
            }
            S.dout[s * LD16 + c] = __float2bfloat16(d);
            d += __shfl_xor_sync(0xffffffffu, d, 16);  // the warp's two samples
            if ((threadIdx.x & 16) == 0) atomicAdd(&grad[b_off(NL - 1) + c], d);
            if (loss) {
                for (int o = 16; o > 0; o >>= 1) se += __shfl_down_sync(0xffffffffu, se, o);
                if ((threadIdx.x & 31) == 0) atomicAdd(loss, se);
            }
        }
        __syncthreads();
        {
            float acc[2][4] = {};
            const FragA a = frag_a<LD16>(S.dout, 0);
            mma(acc[0], a, W.b3[0].x, W.b3[0].y);
            mma(acc[1], a, W.b3[1].x, W.b3[1].y);
            hidden_delta(acc, S.act[2], S.dlt[0]);
        }
        weight_grad<LD128, LD16, DOUT, 2>(S.act[2], S.dout, warp * 16, 0, grad + w_off(3));
        __syncthreads();
        {
            float acc[2][4] = {};
            product<2>(S.dlt[0], W.b2, acc);
            hidden_delta(acc, S.act[1], S.dlt[1]);
        }
        weight_grad<LD128, LD128, H, 16>(S.act[1], S.dlt[0], warp * 16, 0, grad + w_off(2));
        bias_grad(S.dlt[0], grad + b_off(2));
        __syncthreads();
        {
            float acc[2][4] = {};
            product<2>(S.dlt[1], W.b1, acc);
            // every warp has finished with the first delta (barrier above)
            hidden_delta(acc, S.act[0], S.dlt[0]);
        }
        weight_grad<LD128, LD128, H, 16>(S.act[0], S.dlt[1], warp * 16, 0, grad + w_off(1));
        bias_grad(S.dlt[1], grad + b_off(1));
        __syncthreads();
        weight_grad<LD16, LD128, H, 2>(S.in, S.dlt[0], 0, warp * 16, grad + w_off(0));
        bias_grad(S.dlt[0], grad + b_off(0));
        __syncthreads();  // the next samples reuse S
    }
}

// Adam step on the FP32 masters, then the BF16 copies; clears grad.
__global__ void mlp_adam_kernel(float *p, float *grad, float *m, float *v,
                                __nv_bfloat16 *wt, __nv_bfloat16 *w, float lr,
                                float b1, float b2, float eps, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    after_predecessor();
    if (i >= NPARAM) return;
    const float g = grad[i];
    m[i] = b1 * m[i] + (1.f - b1) * g;
    v[i] = b2 * v[i] + (1.f - b2) * g * g;
    p[i] -= lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
    grad[i] = 0.f;
    if (i < NW) {
        int l = 0;
        while (l + 1 < NL && i >= w_off(l + 1)) ++l;
        const int K = layer_k(l), N = layer_n(l), local = i - w_off(l);
        const int k = local / N, n = local % N;
        const __nv_bfloat16 b = __float2bfloat16(p[i]);
        w[w_off(l) + frag_pos(k, n, N)] = b;
        wt[w_off(l) + frag_pos(n, k, K)] = b;
    }
}

}  // namespace cplbm_mlp

using namespace cplbm_mlp;
using cplbm::dev_alloc;
using cplbm::dev_free;

struct lbm_mlp {
    float *p = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    float *loss = nullptr;
    __nv_bfloat16 *wt = nullptr, *w = nullptr;
    int device = 0;
    long long steps = 0;
    std::string err;
};

namespace {
thread_local std::string g_mlp_err;

lbm_status mfail(lbm_mlp *m, lbm_status s, const char *msg, cudaError_t e)
{
    std::string t = msg;
    if (e != cudaSuccess) t += std::string(": ") + cudaGetErrorString(e);
    (m ? m->err : g_mlp_err) = t;
    return s;
}

#define MCUDA(m, call, msg)                                        \
    do {                                                           \
        cudaError_t e_ = (call);                                   \
        if (e_ != cudaSuccess) return mfail((m), LBM_ERR_CUDA, msg, e_); \
    } while (0)

Params params_of(const lbm_mlp *m) { return Params{m->wt, m->w, m->p}; }

int ctas(int B) { return std::min(groups(B), MAX_CTAS); }

// A launch that may start while its predecessor on the stream still runs
// (the kernel waits for it, after_predecessor).
template <class... K, class... A>
cudaError_t launch_after(void (*kern)(K...), int grid, int block, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, K(args)...);
}
}  // namespace

extern "C" {

int lbm_mlp_param_count(void) { return NPARAM; }

lbm_status lbm_mlp_create(int device, const float *init, lbm_mlp **out)
{
    if (out) *out = nullptr;
    if (!out || !init) {
        g_mlp_err = "null argument";
        return LBM_ERR_ARG;
    }
    lbm_mlp *m = new (std::nothrow) lbm_mlp();
    if (!m) return LBM_ERR_OOM;
    m->device = device;
    cudaError_t e = cudaSetDevice(device);
    const size_t fb = NPARAM * sizeof(float);
    if (e == cudaSuccess) e = dev_alloc((void **)&m->p, fb);
    if (e == cudaSuccess) e = dev_alloc((void **)&m->grad, fb);
    if (e == cudaSuccess) e = dev_alloc((void **)&m->m, fb);
    if (e == cudaSuccess) e = dev_alloc((void **)&m->v, fb);
    if (e == cudaSuccess) e = dev_alloc((void **)&m->loss, sizeof(float));
    if (e == cudaSuccess) e = dev_alloc((void **)&m->wt, NW * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = dev_alloc((void **)&m->w, NW * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMemcpy(m->p, init, fb, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(m->grad, 0, fb);
    if (e == cudaSuccess) e = cudaMemset(m->m, 0, fb);
    if (e == cudaSuccess) e = cudaMemset(m->v, 0, fb);
    if (e == cudaSuccess) {
        // BF16 copies of the initial weights: an Adam step with lr = 0
        mlp_adam_kernel<<<(NPARAM + 255) / 256, 256>>>(m->p, m->grad, m->m, m->v,
                                                       m->wt, m->w, 0.f, 0.9f,
                                                       0.999f, 1e-8f, 1.f, 1.f);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        g_mlp_err = std::string("mlp create: ") + cudaGetErrorString(e);
        lbm_mlp_destroy(m);
        return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
    }
    *out = m;
    return LBM_OK;
}

lbm_status lbm_mlp_train(lbm_mlp *m, const float *X, int nin, const float *T,
                         int nout, int B, int iters, float lr, float *loss_out)
{
    CPLBM_TRACE("lbm_mlp_train");
    if (!m) return LBM_ERR_ARG;
    if (!X || !T || B <= 0 || nin < 1 || nin > DIN || nout < 1 || nout > DOUT ||
        iters < 0 || !(lr >= 0))
        return mfail(m, LBM_ERR_ARG, "bad training arguments", cudaSuccess);
    MCUDA(m, cudaSetDevice(m->device), "cudaSetDevice");
    float loss = 0.f;
    MCUDA(m, cudaMemsetAsync(m->loss, 0, sizeof(float)), "memset");
    for (int it = 0; it < iters; ++it) {
        // the error of the last forward pass is the one reported
        MCUDA(m, launch_after(mlp_train_kernel, ctas(B), THREADS, params_of(m), X, nin, T, nout,
                              B, m->grad, it + 1 == iters ? m->loss : nullptr),
              "mlp train launch");
        ++m->steps;
        const float c1 = 1.f - std::pow(0.9f, (float)m->steps);
        const float c2 = 1.f - std::pow(0.999f, (float)m->steps);
        MCUDA(m, launch_after(mlp_adam_kernel, (NPARAM + 255) / 256, 256, m->p, m->grad, m->m,
                              m->v, m->wt, m->w, lr, 0.9f, 0.999f, 1e-8f, c1, c2),
              "mlp adam launch");
    }
    MCUDA(m, cudaMemcpy(&loss, m->loss, sizeof(float), cudaMemcpyDeviceToHost),
          "loss copy");
    if (loss_out) *loss_out = loss / (float)(B * nout);
    return LBM_OK;
}

lbm_status lbm_mlp_gradient(lbm_mlp *m, const float *X, int nin, const float *T,
                            int nout, int B, float *grad, float *loss_out)
{
    CPLBM_TRACE("lbm_mlp_gradient");
    if (!m) return LBM_ERR_ARG;
    if (!X || !T || !grad || B <= 0 || nin < 1 || nin > DIN || nout < 1 || nout > DOUT)
        return mfail(m, LBM_ERR_ARG, "bad gradient arguments", cudaSuccess);
    MCUDA(m, cudaSetDevice(m->device), "cudaSetDevice");
    // the training pass without the optimiser step: the accumulated full-batch
    // gradient is copied out and the accumulator cleared again
    MCUDA(m, cudaMemsetAsync(m->grad, 0, NPARAM * sizeof(float)), "memset");
    MCUDA(m, cudaMemsetAsync(m->loss, 0, sizeof(float)), "memset");
    mlp_train_kernel<<<ctas(B), THREADS>>>(params_of(m), X, nin, T, nout, B, m->grad, m->loss);
    MCUDA(m, cudaGetLastError(), "mlp gradient launch");
    float loss = 0.f;
    MCUDA(m, cudaMemcpy(grad, m->grad, NPARAM * sizeof(float), cudaMemcpyDeviceToHost),
          "gradient copy");
    MCUDA(m, cudaMemcpy(&loss, m->loss, sizeof(float), cudaMemcpyDeviceToHost),
          "loss copy");
    MCUDA(m, cudaMemset(m->grad, 0, NPARAM * sizeof(float)), "memset");
    if (loss_out) *loss_out = loss / (float)(B * nout);
    return LBM_OK;
}

lbm_status lbm_mlp_predict(lbm_mlp *m, const float *X, int nin, float *Y,
                           int nout, int B)
{
    CPLBM_TRACE("lbm_mlp_predict");
    if (!m) return LBM_ERR_ARG;
    if (!X || !Y || B <= 0 || nin < 1 || nin > DIN || nout < 1 || nout > DOUT)
        return mfail(m, LBM_ERR_ARG, "bad prediction arguments", cudaSuccess);
    MCUDA(m, cudaSetDevice(m->device), "cudaSetDevice");
    mlp_infer_kernel<<<ctas(B), THREADS>>>(params_of(m), X, nin, Y, nout, B);
    MCUDA(m, cudaGetLastError(), "mlp infer launch");
    MCUDA(m, cudaDeviceSynchronize(), "mlp infer");
    return LBM_OK;
}

lbm_status lbm_mlp_get_params(lbm_mlp *m, float *out)
{
    if (!m || !out) return LBM_ERR_ARG;
    MCUDA(m, cudaMemcpy(out, m->p, NPARAM * sizeof(float), cudaMemcpyDeviceToHost),
          "params copy");
    return LBM_OK;
}

void lbm_mlp_destroy(lbm_mlp *m)
{
    if (!m) return;
    dev_free(m->p);
    dev_free(m->grad);
    dev_free(m->m);
    dev_free(m->v);
    dev_free(m->loss);
    dev_free(m->wt);
    dev_free(m->w);
    delete m;
}

const char *lbm_mlp_last_error(const lbm_mlp *m)
{
    return m ? m->err.c_str() : g_mlp_err.c_str();
}

}  // extern "C"

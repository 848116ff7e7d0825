// Small multilayer perceptron n_in -> H -> H -> n_out (SiLU) trained and run
// on the GPU with BF16 inputs and FP32 accumulation: the learned residual on
// the Taylor predictor.  The paper has no learned component; the network is a
// workload-side addition documented with the design.
//
// Every product is one GEMM kernel on the tensor cores, mma.sync m16n8k16 with
// bf16 operands and fp32 accumulators; ldmatrix absorbs the transposes of the
// backward pass, the epilogues bias, activation and its derivative.  Weight
// gradients, sums over the batch, have a kernel of their own.  Elementwise kernels form
// the mean-squared-error gradient, sum bias gradients and take the Adam step (Kingma & Ba 2015) on an FP32 master copy of
// the parameters, refreshed into bf16 after every step.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <numeric>
#include <random>
#include <utility>
#include <vector>

#include "common.cuh"

namespace mh {
namespace {

using bf16 = __nv_bfloat16;

constexpr int kTM = 64, kTN = 64, kTK = 32, kPad16 = 8;
constexpr int kSplitRows = 256;      // least rows of one part of a bias gradient

__device__ __forceinline__ float silu(float z) { return z / (1.0f + __expf(-z)); }
__device__ __forceinline__ float dsilu(float z)
{
    const float s = 1.0f / (1.0f + __expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

// What a GEMM does with its sums.
enum { kStore = 0,       // c = sum
       kBias = 1,        // c = sum + bias
       kBiasSilu = 2,    // c = z = sum + bias, h = bf16(silu(z))
       kDsilu = 3,       // h = bf16(sum * silu'(c)), c read
       kSilu = 4 };      // h = bf16(silu(sum + bias)): inference, which reads no z again

// Rows x cols bf16 tile src[r * ld + c] to shared memory [rows][cols + kPad16], zero
// outside rmax x cmax.  128 threads; vec: 16-byte loads (base and ld allow them).
template <int rows, int cols>
__device__ __forceinline__ void stage(bf16 (*dst)[cols + kPad16], const bf16 *__restrict__ src, int64_t ld, int rmax,
                                      int cmax, bool vec)
{
    constexpr int per_row = cols / 8;
#pragma unroll
    for (int e = threadIdx.x; e < rows * per_row; e += 128) {
        const int r = e / per_row, c = (e % per_row) * 8;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (r < rmax) {
            const bf16 *q = src + r * ld + c;
            if (vec && c + 8 <= cmax) {
                v = *reinterpret_cast<const uint4 *>(q);
            } else {
                __align__(16) bf16 w[8];           // read as one 16-byte word below
#pragma unroll
                for (int k = 0; k < 8; ++k) w[k] = c + k < cmax ? q[k] : __float2bfloat16(0.0f);
                v = *reinterpret_cast<const uint4 *>(w);
            }
        }
        *reinterpret_cast<uint4 *>(&dst[r][c]) = v;
    }
}

template <bool trans>
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], const bf16 *p)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    if (trans)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}

// C[M x N] (fp32, row stride ldc) = A[M x K] B[K x N] with bf16 operands:
//   A(m, k) = TA ? a[k * lda + m] : a[m * lda + k]
//   B(k, n) = TB ? b[n * ldb + k] : b[k * ldb + n]
// Tiles keep the operands' own order in shared memory; ldmatrix transposes on the
// way to the fragments.
// The network's layers are bound by their activations' traffic (65537 x 128
// FP32 and BF16 values written or read per layer), so bias, SiLU and its
// derivative are applied here instead of in passes of their own.
template <bool TA, bool TB, int EPI>
__global__ void __launch_bounds__(128) k_gemm_bf16(int M, int N, int K, const bf16 *__restrict__ a, int lda,
                                                   const bf16 *__restrict__ b, int ldb, float *__restrict__ c,
                                                   int ldc, const float *__restrict__ bias,
                                                   bf16 *__restrict__ h, bool veca, bool vecb)
{
    constexpr int AR = TA ? kTK : kTM, AC = TA ? kTM : kTK, BR = TB ? kTN : kTK, BC = TB ? kTK : kTN;
    __shared__ __align__(16) bf16 As[AR][AC + kPad16];
    __shared__ __align__(16) bf16 Bs[BR][BC + kPad16];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.x * kTM, n0 = blockIdx.y * kTN;     // rows on x: up to 2^31 tiles
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int g = lane >> 2, t = lane & 3;
    const int lr = lane & 7, lq = lane >> 3;                   // ldmatrix: row and matrix of this lane's address
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
    for (int k0 = 0; k0 < K; k0 += kTK) {
        const int kn = K - k0;
        if (TA)
            stage<AR, AC>(As, a + (int64_t)k0 * lda + m0, lda, kn, M - m0, veca);
        else
            stage<AR, AC>(As, a + (int64_t)m0 * lda + k0, lda, M - m0, kn, veca);
        if (TB)
            stage<BR, BC>(Bs, b + (int64_t)n0 * ldb + k0, ldb, N - n0, kn, vecb);
        else
            stage<BR, BC>(Bs, b + (int64_t)k0 * ldb + n0, ldb, kn, N - n0, vecb);
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < kTK; ks += 16) {
            uint32_t af[2][4], bq[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                // matrices: (m 0-7, k 0-7), (m 8-15, k 0-7), (m 0-7, k 8-15), (m 8-15, k 8-15)
                const int m = wm + 16 * i + (lq & 1) * 8, k = ks + (lq >> 1) * 8;
                ldmatrix4<TA>(af[i], TA ? &As[k + lr][m] : &As[m + lr][k]);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                // matrices: (n 0-7, k 0-7), (n 0-7, k 8-15), (n 8-15, k 0-7), (n 8-15, k 8-15)
                const int n = wn + 16 * j + (lq >> 1) * 8, k = ks + (lq & 1) * 8;
                ldmatrix4<!TB>(bq[j], TB ? &Bs[n + lr][k] : &Bs[k + lr][n]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    asm volatile(
                        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                        : "+f"(acc[i][j][0]), "+f"(acc[i][j][1]), "+f"(acc[i][j][2]), "+f"(acc[i][j][3])
                        : "r"(af[i][0]), "r"(af[i][1]), "r"(af[i][2]), "r"(af[i][3]), "r"(bq[j / 2][2 * (j & 1)]),
                          "r"(bq[j / 2][2 * (j & 1) + 1]));
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int m = m0 + wm + 16 * i + g + (q >= 2 ? 8 : 0);
                const int n = n0 + wn + 8 * j + 2 * t + (q & 1);
                if (m >= M || n >= N) continue;
                const int64_t e = (int64_t)m * ldc + n;
                if (EPI == kDsilu) {
                    h[e] = __float2bfloat16(acc[i][j][q] * dsilu(c[e]));
                } else {
                    const float z = EPI == kStore ? acc[i][j][q] : acc[i][j][q] + bias[n];
                    if (EPI != kSilu) c[e] = z;
                    if (EPI == kBiasSilu || EPI == kSilu) h[e] = __float2bfloat16(silu(z));
                }
            }
}

// Weight gradients C[M x N] = A^T B, sums over the batch of up to 2^24 rows: one
// chain of products per output element in row order, as k_gemm_bf16 takes them
// (the tensor core rounds each step towards zero, so cutting the chain changes the
// weights' gradients of 65537 rows by 7e-5 of their size).  Small output tiles put the
// chains on as many SMs as there are tiles and the rows come through a ring of
// asynchronous copies.  Bound by the ring: ~630 cycles per 64-row stage, of which the
// chain's four dependent products take 82 (20.4 each, measured); the rest is the
// copies' latency with three stages in flight and a barrier per stage.  All weights of
// the network in one launch: the gradients of 65537 rows took 8 ms each on one to four
// SMs with a barrier and element-wise loads every 16 rows, 313 us now.
constexpr int kWT = 32, kWK = 64, kWStages = 4;

struct WGrad {
    const bf16 *a, *b;
    float *c;
    int M, N, lda, ldb, tiles_n, first;    // first: the first CTA of this gradient
    bool vec;
};
struct WGrads {
    WGrad g[3];
    int64_t K;
};

__device__ __forceinline__ void copy_rows(bf16 (*dst)[kWT + kPad16], const bf16 *src, int ld, int cmax, int64_t rmax,
                                          bool vec)
{
    // kWK rows of kWT columns: 4 chunks of 8 per row, 128 threads
#pragma unroll
    for (int q = 0; q < kWK * (kWT / 8) / 128; ++q) {
        const int e = threadIdx.x + q * 128, r = e >> 2, c = (e & 3) * 8;
        const bf16 *p = src + (int64_t)r * ld + c;
        if (vec) {
            const unsigned d = (unsigned)__cvta_generic_to_shared(&dst[r][c]);
            const bool in = r < rmax && c < cmax;              // ld is a multiple of 8; else 16 zero bytes
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(in ? p : src), "r"(in ? 16 : 0)
                         : "memory");
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                dst[r][c + k] = r < rmax && c + k < cmax ? p[k] : __float2bfloat16(0.0f);
        }
    }
}

__global__ void __launch_bounds__(128) k_wgrad(WGrads w)
{
    __shared__ __align__(16) bf16 As[kWStages][kWK][kWT + kPad16];
    __shared__ __align__(16) bf16 Bs[kWStages][kWK][kWT + kPad16];
    const int which = (int)blockIdx.x >= w.g[2].first ? 2 : (int)blockIdx.x >= w.g[1].first ? 1 : 0;
    const WGrad &q = w.g[which];
    const int tile = blockIdx.x - q.first;
    const int m0 = tile / q.tiles_n * kWT, n0 = tile % q.tiles_n * kWT;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wm = (warp >> 1) * 16, wn = (warp & 1) * 16;
    const int g = lane >> 2, t = lane & 3, lr = lane & 7, lq = lane >> 3;
    float acc[2][4] = {{0.0f, 0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f, 0.0f}};
    const int64_t steps = (w.K + kWK - 1) / kWK;
    auto fetch = [&](int64_t s) {
        if (s < steps) {
            // whole rows: the padding columns hold zeros
            copy_rows(As[s % kWStages], q.a + s * kWK * q.lda + m0, q.lda, q.lda - m0, w.K - s * kWK, q.vec);
            copy_rows(Bs[s % kWStages], q.b + s * kWK * q.ldb + n0, q.ldb, q.ldb - n0, w.K - s * kWK, q.vec);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int s = 0; s < kWStages - 1; ++s) fetch(s);
    for (int64_t s = 0; s < steps; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kWStages - 2) : "memory");
        __syncthreads();                       // step s has landed; step s - 1 is read
        fetch(s + kWStages - 1);
        const auto &A = As[s % kWStages];
        const auto &B = Bs[s % kWStages];
        uint32_t af[kWK / 16][4], bq[kWK / 16][4];
#pragma unroll
        for (int ks = 0; ks < kWK / 16; ++ks) {
            ldmatrix4<true>(af[ks], &A[ks * 16 + (lq >> 1) * 8 + lr][wm + (lq & 1) * 8]);
            ldmatrix4<true>(bq[ks], &B[ks * 16 + (lq & 1) * 8 + lr][wn + (lq >> 1) * 8]);
        }
#pragma unroll
        for (int ks = 0; ks < kWK / 16; ++ks)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                asm volatile(
                    "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                    "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                    : "+f"(acc[j][0]), "+f"(acc[j][1]), "+f"(acc[j][2]), "+f"(acc[j][3])
                    : "r"(af[ks][0]), "r"(af[ks][1]), "r"(af[ks][2]), "r"(af[ks][3]), "r"(bq[ks][2 * j]),
                      "r"(bq[ks][2 * j + 1]));
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int m = m0 + wm + g + (e >= 2 ? 8 : 0), n = n0 + wn + 8 * j + 2 * t + (e & 1);
            if (m < q.M && n < q.N) q.c[(int64_t)m * q.N + n] = acc[j][e];
        }
}

// out[e] = sum of the parts, one warp per e, in a fixed order
__global__ void k_sum_parts(int64_t n, int parts, const float *__restrict__ x, float *__restrict__ out)
{
    const int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (e >= n) return;
    float s = 0.0f;
    for (int p = threadIdx.x & 31; p < parts; p += 32) s += x[p * n + e];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) out[e] = s;
}

// dY = bf16(2 (Y - T) / (B n_out)), rows of O values with stride ld; per-block partial
// sums of (Y - T)^2 (double).
__global__ void k_mse(int64_t n, int64_t denom, const float *Y, const float *T, bf16 *dY, int O, int ld, double *part)
{
    __shared__ double red[256];
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double s = 0.0;
    if (e < n) {
        const float d = Y[e] - T[e];
        dY[e / O * ld + e % O] = __float2bfloat16(2.0f * d / (float)denom);
        s = (double)d * (double)d;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

__global__ void k_sum_double(int64_t n, const double *x, double *out)
{
    __shared__ double red[256];
    double s = 0.0;
    for (int64_t k = threadIdx.x; k < n; k += blockDim.x) s += x[k];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

// out[part][n] = sum of X[b][n] over the part's rows b (bf16 inputs, fp32 sums in a
// fixed order): 64 columns by four row groups per CTA.
__global__ void __launch_bounds__(256) k_colsum(int64_t B, int N, int ld, int rows, const bf16 *__restrict__ X,
                                                float *__restrict__ out)
{
    __shared__ float red[4][64];
    const int c = threadIdx.x & 63, rg = threadIdx.x >> 6;
    const int n = blockIdx.x * 64 + c;
    const int64_t b0 = (int64_t)blockIdx.y * rows, b1 = min(B, b0 + rows);
    float s = 0.0f;
    if (n < N)
        for (int64_t b = b0 + rg; b < b1; b += 4) s += __bfloat162float(X[b * ld + n]);
    red[rg][c] = s;
    __syncthreads();
    if (rg == 0 && n < N) out[(int64_t)blockIdx.y * N + n] = (red[0][c] + red[1][c]) + (red[2][c] + red[3][c]);
}

// rows of src (fp32, width w) gathered by idx (or 0..n-1) into bf16 / fp32 dst
// (dst16 with row stride ld)
__global__ void k_gather(int64_t n, int w, const float *src, const int *idx, bf16 *dst16, int ld, float *dst32)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * w) return;
    const int64_t r = e / w, c = e - r * w;
    const int64_t s = idx ? (int64_t)idx[r] : r;
    const float v = src[s * w + c];
    if (dst16) dst16[r * ld + c] = __float2bfloat16(v);
    if (dst32) dst32[e] = v;
}

__global__ void k_adam(int64_t n, float *p, const float *g, float *m, float *v, bf16 *p16, float lr,
                       float b1, float b2, float eps, float c1, float c2)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const float gr = g[e];
    const float mm = b1 * m[e] + (1.0f - b1) * gr;
    const float vv = b2 * v[e] + (1.0f - b2) * gr * gr;
    m[e] = mm;
    v[e] = vv;
    const float q = p[e] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    p[e] = q;
    p16[e] = __float2bfloat16(q);
}

__global__ void k_to_bf16(int64_t n, const float *x, bf16 *y)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) y[e] = __float2bfloat16(x[e]);
}

inline unsigned nb(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

inline int pad8(int n) { return (n + 7) / 8 * 8; }
inline bool vec16(const bf16 *p, int ld) { return ld % 8 == 0 && reinterpret_cast<uintptr_t>(p) % 16 == 0; }

// Parts of a bias gradient over B rows: two CTAs per SM, kSplitRows rows at least.
// (One thread per column took 7 ms at 65537 rows, 256 parts 13 us.)
inline int split_parts(int64_t B) { return (int)std::max<int64_t>(1, std::min<int64_t>(B / kSplitRows, 304)); }

template <bool TA, bool TB, int EPI>
int gemm(int M, int N, int K, const bf16 *a, int lda, const bf16 *b, int ldb, float *c, int ldc, cudaStream_t st,
         const float *bias = nullptr, bf16 *h = nullptr)
{
    dim3 grid((M + kTM - 1) / kTM, (N + kTN - 1) / kTN);
    k_gemm_bf16<TA, TB, EPI><<<grid, 128, 0, st>>>(M, N, K, a, lda, b, ldb, c, ldc, bias, h, vec16(a, lda),
                                                   vec16(b, ldb));
    MH_LAUNCHED("k_gemm_bf16");
    return MH_OK;
}

}  // namespace
}  // namespace mh

using namespace mh;

struct mh_mlp {
    int n_in = 0, H = 0, n_out = 0;
    int64_t n_params = 0;
    int64_t oW1 = 0, ob1 = 0, oW2 = 0, ob2 = 0, oW3 = 0, ob3 = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    bf16 *p16 = nullptr;
    int64_t t = 0;
    int64_t cap = 0;                 // rows of X16, H1, H2: all that inference needs
    int64_t cap_train = 0;           // rows of the other buffers
    bf16 *X16 = nullptr, *H1 = nullptr, *H2 = nullptr, *dY16 = nullptr, *dZ2 = nullptr, *dZ1 = nullptr;
    float *Z1 = nullptr, *Z2 = nullptr, *Y = nullptr, *T = nullptr;
    double *lpart = nullptr, *lsum = nullptr;
    float *gpart = nullptr;          // parts of the bias gradient being formed
    int *idx = nullptr;
    int64_t idx_cap = 0;
};

namespace {

template <typename T>
void drop(T *&p)
{
    if (p) cudaFree(p);
    p = nullptr;
}

void free_train(mh_mlp *n)
{
    drop(n->dY16); drop(n->dZ2); drop(n->dZ1); drop(n->Z1); drop(n->Z2); drop(n->Y); drop(n->T);
    drop(n->lpart); drop(n->lsum); drop(n->gpart);
    n->cap_train = 0;
}

void free_ws(mh_mlp *n)
{
    free_train(n);
    drop(n->X16); drop(n->H1); drop(n->H2);
    n->cap = 0;
}

// Workspace of a pass over `rows` rows: inference, or with the gradient's buffers too.
int ensure_ws(mh_mlp *n, int64_t rows, bool train, cudaStream_t st)
{
    const int64_t H = n->H;
    if (rows > n->cap) {
        MH_CUDA(cudaStreamSynchronize(st));
        drop(n->X16); drop(n->H1); drop(n->H2);
        n->cap = 0;
        MH_CUDA(cudaMalloc((void **)&n->X16, rows * pad8(n->n_in) * sizeof(bf16)));
        MH_CUDA(cudaMalloc((void **)&n->H1, rows * H * sizeof(bf16)));
        MH_CUDA(cudaMalloc((void **)&n->H2, rows * H * sizeof(bf16)));
        // the padding columns of X16 (and dY16) stay zero
        MH_CUDA(cudaMemsetAsync(n->X16, 0, rows * pad8(n->n_in) * sizeof(bf16), st));
        n->cap = rows;
    }
    if (train && rows > n->cap_train) {
        MH_CUDA(cudaStreamSynchronize(st));
        free_train(n);
        MH_CUDA(cudaMalloc((void **)&n->dY16, rows * pad8(n->n_out) * sizeof(bf16)));
        MH_CUDA(cudaMalloc((void **)&n->dZ2, rows * H * sizeof(bf16)));
        MH_CUDA(cudaMalloc((void **)&n->dZ1, rows * H * sizeof(bf16)));
        MH_CUDA(cudaMalloc((void **)&n->Z1, rows * H * sizeof(float)));
        MH_CUDA(cudaMalloc((void **)&n->Z2, rows * H * sizeof(float)));
        MH_CUDA(cudaMalloc((void **)&n->Y, rows * n->n_out * sizeof(float)));
        MH_CUDA(cudaMalloc((void **)&n->T, rows * n->n_out * sizeof(float)));
        const int64_t gp = (int64_t)split_parts(rows) * std::max(n->H, n->n_out);
        MH_CUDA(cudaMalloc((void **)&n->gpart, gp * sizeof(float)));
        MH_CUDA(cudaMalloc((void **)&n->lpart, (nb(rows * n->n_out) + 1) * sizeof(double)));
        MH_CUDA(cudaMalloc((void **)&n->lsum, sizeof(double)));
        MH_CUDA(cudaMemsetAsync(n->dY16, 0, rows * pad8(n->n_out) * sizeof(bf16), st));
        n->cap_train = rows;
    }
    return MH_OK;
}

// Forward over rows already gathered into X16; Y (fp32) receives the outputs.  EPI:
// kBiasSilu keeps the pre-activations Z1, Z2 for the gradient, kSilu does not.
template <int EPI>
int forward_ws(mh_mlp *n, int64_t B, float *Y, cudaStream_t st)
{
    const int H = n->H;
    const bf16 *W1 = n->p16 + n->oW1, *W2 = n->p16 + n->oW2, *W3 = n->p16 + n->oW3;
    if (int rc = gemm<false, true, EPI>((int)B, H, n->n_in, n->X16, pad8(n->n_in), W1, n->n_in, n->Z1, H, st,
                                        n->p + n->ob1, n->H1))
        return rc;
    if (int rc = gemm<false, true, EPI>((int)B, H, H, n->H1, H, W2, H, n->Z2, H, st, n->p + n->ob2, n->H2)) return rc;
    return gemm<false, true, kBias>((int)B, n->n_out, H, n->H2, H, W3, H, Y, n->n_out, st, n->p + n->ob3);
}

// A bias gradient, the column sums of a over the batch: parts side by side, then added in order.
int bias_grad(mh_mlp *n, int M, int64_t B, const bf16 *a, int lda, float *gb, cudaStream_t st)
{
    const int parts = split_parts(B), rows = (int)((B + parts - 1) / parts);
    k_colsum<<<dim3((M + 63) / 64, parts), 256, 0, st>>>(B, M, lda, rows, a, n->gpart);
    MH_LAUNCHED("k_colsum");
    k_sum_parts<<<nb((int64_t)M * 32), 256, 0, st>>>(M, parts, n->gpart, gb);
    MH_LAUNCHED("k_sum_parts");
    return MH_OK;
}

// Loss (device scalar lsum, sum of squares) and gradients into g, for rows in X16 / T / Y.
int backward_ws(mh_mlp *n, int64_t B, cudaStream_t st)
{
    const int H = n->H, O = n->n_out, lo = pad8(O);
    const bf16 *W2 = n->p16 + n->oW2, *W3 = n->p16 + n->oW3;
    const int64_t ny = B * O;
    k_mse<<<nb(ny), 256, 0, st>>>(ny, ny, n->Y, n->T, n->dY16, O, lo, n->lpart);
    MH_LAUNCHED("k_mse");
    k_sum_double<<<1, 256, 0, st>>>(nb(ny), n->lpart, n->lsum);
    MH_LAUNCHED("k_sum_double");
    // back-propagated errors
    if (int rc = gemm<false, false, kDsilu>((int)B, H, O, n->dY16, lo, W3, H, n->Z2, H, st, nullptr, n->dZ2)) return rc;
    if (int rc = gemm<false, false, kDsilu>((int)B, H, H, n->dZ2, H, W2, H, n->Z1, H, st, nullptr, n->dZ1)) return rc;
    // gradients of all three layers
    WGrads w;
    w.K = B;
    int first = 0;
    auto layer = [&](int k, int M, int N, const bf16 *a, int lda, const bf16 *b, int ldb, float *c) {
        const int tn = (N + kWT - 1) / kWT;
        w.g[k] = WGrad{a, b, c, M, N, lda, ldb, tn, first, vec16(a, lda) && vec16(b, ldb)};
        first += (M + kWT - 1) / kWT * tn;
    };
    layer(0, H, H, n->dZ2, H, n->H1, H, n->g + n->oW2);
    layer(1, H, n->n_in, n->dZ1, H, n->X16, pad8(n->n_in), n->g + n->oW1);
    layer(2, O, H, n->dY16, lo, n->H2, H, n->g + n->oW3);
    k_wgrad<<<first, 128, 0, st>>>(w);
    MH_LAUNCHED("k_wgrad");
    if (int rc = bias_grad(n, O, B, n->dY16, lo, n->g + n->ob3, st)) return rc;
    if (int rc = bias_grad(n, H, B, n->dZ2, H, n->g + n->ob2, st)) return rc;
    return bias_grad(n, H, B, n->dZ1, H, n->g + n->ob1, st);
}

int check_net(const mh_mlp *n)
{
    if (!n) { set_error("NULL mh_mlp handle"); return MH_EINVAL; }
    return MH_OK;
}

}  // namespace

namespace mh {
// Inference for the learned predictor (learned.cu): Y[n x n_out] from X[n x n_in] (fp32, device).
int mlp_infer(mh_mlp *n, const float *X, float *Y, int64_t rows, cudaStream_t st)
{
    // rows per pass: 256 MB of X16, H1 and H2 (H = 128: 2^18 rows in 147 MB), whole tiles
    const int64_t row_bytes = (int64_t)sizeof(bf16) * (pad8(n->n_in) + 2 * n->H);
    const int64_t chunk = std::min<int64_t>(1 << 18, (256ll << 20) / row_bytes / kTM * kTM);
    if (int rc = ensure_ws(n, std::min(rows, chunk), false, st)) return rc;
    for (int64_t r0 = 0; r0 < rows; r0 += chunk) {
        const int64_t B = std::min(chunk, rows - r0);
        k_gather<<<nb(B * n->n_in), 256, 0, st>>>(B, n->n_in, X + r0 * n->n_in, nullptr, n->X16, pad8(n->n_in),
                                                       nullptr);
        MH_LAUNCHED("k_gather");
        if (int rc = forward_ws<kSilu>(n, B, Y + r0 * n->n_out, st)) return rc;
    }
    return MH_OK;
}
int mlp_dims(const mh_mlp *n, int *n_in, int *n_out)
{
    if (!n) return MH_EINVAL;
    *n_in = n->n_in;
    *n_out = n->n_out;
    return MH_OK;
}
}  // namespace mh

extern "C" {

int mh_mlp_create(mh_mlp **out, int n_in, int n_hidden, int n_out, uint64_t seed)
{
    if (!out) { set_error("mh_mlp_create: out is NULL"); return MH_EINVAL; }
    *out = nullptr;
    if (n_in < 1 || n_in > 4096 || n_hidden < 1 || n_hidden > 4096 || n_out < 1 || n_out > 4096) {
        set_error("mh_mlp_create: sizes must be in [1, 4096]");
        return MH_EINVAL;
    }
    mh_mlp *n = new (std::nothrow) mh_mlp();
    if (!n) { set_error("mh_mlp_create: host allocation failed"); return MH_ENOMEM; }
    n->n_in = n_in;
    n->H = n_hidden;
    n->n_out = n_out;
    n->oW1 = 0;
    n->ob1 = n->oW1 + (int64_t)n_hidden * n_in;
    n->oW2 = n->ob1 + n_hidden;
    n->ob2 = n->oW2 + (int64_t)n_hidden * n_hidden;
    n->oW3 = n->ob2 + n_hidden;
    n->ob3 = n->oW3 + (int64_t)n_out * n_hidden;
    n->n_params = n->ob3 + n_out;
    // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights, zero biases
    std::vector<float> h(n->n_params, 0.0f);
    std::mt19937_64 rng(seed);
    std::uniform_real_distribution<float> u(-1.0f, 1.0f);
    auto fill = [&](int64_t off, int64_t count, int fan_in) {
        const float sc = 1.0f / std::sqrt((float)fan_in);
        for (int64_t k = 0; k < count; ++k) h[off + k] = sc * u(rng);
    };
    fill(n->oW1, (int64_t)n_hidden * n_in, n_in);
    fill(n->oW2, (int64_t)n_hidden * n_hidden, n_hidden);
    fill(n->oW3, (int64_t)n_out * n_hidden, n_hidden);
    cudaError_t e = cudaMalloc((void **)&n->p, n->n_params * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void **)&n->g, n->n_params * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void **)&n->m, n->n_params * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void **)&n->v, n->n_params * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void **)&n->p16, n->n_params * sizeof(bf16));
    if (e == cudaSuccess) e = cudaMemcpy(n->p, h.data(), n->n_params * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(n->m, 0, n->n_params * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(n->v, 0, n->n_params * sizeof(float));
    if (e == cudaSuccess) {
        k_to_bf16<<<nb(n->n_params), 256>>>(n->n_params, n->p, n->p16);
        e = cudaDeviceSynchronize();
    }
    if (e != cudaSuccess) {
        int rc = cuda_fail(e, "mh_mlp_create");
        mh_mlp_destroy(n);
        return rc;
    }
    *out = n;
    return MH_OK;
}

void mh_mlp_destroy(mh_mlp *n)
{
    if (!n) return;
    cudaDeviceSynchronize();
    free_ws(n);
    void *ptrs[] = {n->p, n->g, n->m, n->v, n->p16, n->idx};
    for (void *q : ptrs)
        if (q) cudaFree(q);
    delete n;
}

int mh_mlp_num_params(const mh_mlp *n, int64_t *count)
{
    if (int rc = check_net(n)) return rc;
    if (count) *count = n->n_params;
    return MH_OK;
}

int mh_mlp_get_params(mh_mlp *n, float *host, int64_t count)
{
    if (int rc = check_net(n)) return rc;
    if (!host || count != n->n_params) { set_error("mh_mlp_get_params: need n_params floats"); return MH_EINVAL; }
    MH_CUDA(cudaDeviceSynchronize());
    MH_CUDA(cudaMemcpy(host, n->p, count * sizeof(float), cudaMemcpyDeviceToHost));
    return MH_OK;
}

int mh_mlp_set_params(mh_mlp *n, const float *host, int64_t count)
{
    if (int rc = check_net(n)) return rc;
    if (!host || count != n->n_params) { set_error("mh_mlp_set_params: need n_params floats"); return MH_EINVAL; }
    MH_CUDA(cudaDeviceSynchronize());
    MH_CUDA(cudaMemcpy(n->p, host, count * sizeof(float), cudaMemcpyHostToDevice));
    MH_CUDA(cudaMemset(n->m, 0, count * sizeof(float)));
    MH_CUDA(cudaMemset(n->v, 0, count * sizeof(float)));
    n->t = 0;
    k_to_bf16<<<nb(count), 256>>>(count, n->p, n->p16);
    MH_LAUNCHED("k_to_bf16");
    MH_CUDA(cudaDeviceSynchronize());
    return MH_OK;
}

int mh_mlp_forward(mh_mlp *n, const float *x, float *y, int64_t rows, void *stream)
{
    if (int rc = check_net(n)) return rc;
    if (!x || !y || rows < 1) { set_error("mh_mlp_forward: device x, y and rows >= 1 required"); return MH_EINVAL; }
    return mlp_infer(n, x, y, rows, (cudaStream_t)stream);
}

int mh_mlp_loss_grad(mh_mlp *n, const float *x, const float *t, int64_t rows, double *loss, float *grad_host,
                     void *stream)
{
    if (int rc = check_net(n)) return rc;
    if (!x || !t || rows < 1 || rows > (1 << 24)) { set_error("mh_mlp_loss_grad: device x, t and 1 <= rows <= 2^24"); return MH_EINVAL; }
    cudaStream_t st = (cudaStream_t)stream;
    if (int rc = ensure_ws(n, rows, true, st)) return rc;
    k_gather<<<nb(rows * n->n_in), 256, 0, st>>>(rows, n->n_in, x, nullptr, n->X16, pad8(n->n_in), nullptr);
    MH_LAUNCHED("k_gather");
    k_gather<<<nb(rows * n->n_out), 256, 0, st>>>(rows, n->n_out, t, nullptr, nullptr, 0, n->T);
    MH_LAUNCHED("k_gather");
    if (int rc = forward_ws<kBiasSilu>(n, rows, n->Y, st)) return rc;
    if (int rc = backward_ws(n, rows, st)) return rc;
    double ls = 0.0;
    MH_CUDA(cudaMemcpyAsync(&ls, n->lsum, sizeof(double), cudaMemcpyDeviceToHost, st));
    if (grad_host) MH_CUDA(cudaMemcpyAsync(grad_host, n->g, n->n_params * sizeof(float), cudaMemcpyDeviceToHost, st));
    MH_CUDA(cudaStreamSynchronize(st));
    if (loss) *loss = ls / (double)(rows * n->n_out);
    return MH_OK;
}

int mh_mlp_train(mh_mlp *n, const float *x, const float *t, int64_t rows, int epochs, int batch, float lr,
                 uint64_t seed, double *final_loss, void *stream)
{
    if (int rc = check_net(n)) return rc;
    if (!x || !t || rows < 1 || epochs < 1 || batch < 1 || batch > (1 << 20) || !(lr > 0.0f)) {
        set_error("mh_mlp_train: device x, t; rows, epochs, batch >= 1; lr > 0");
        return MH_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t B = std::min<int64_t>(batch, rows);
    if (int rc = ensure_ws(n, B, true, st)) return rc;
    if (rows > n->idx_cap) {
        MH_CUDA(cudaStreamSynchronize(st));
        if (n->idx) cudaFree(n->idx);
        n->idx = nullptr;
        MH_CUDA(cudaMalloc((void **)&n->idx, rows * sizeof(int)));
        n->idx_cap = rows;
    }
    std::vector<int> perm(rows);
    std::iota(perm.begin(), perm.end(), 0);
    std::mt19937_64 rng(seed);
    double last = 0.0;
    for (int ep = 0; ep < epochs; ++ep) {
        std::shuffle(perm.begin(), perm.end(), rng);
        MH_CUDA(cudaMemcpyAsync(n->idx, perm.data(), rows * sizeof(int), cudaMemcpyHostToDevice, st));
        double ep_sum = 0.0;
        int64_t ep_rows = 0;
        for (int64_t r0 = 0; r0 + B <= rows; r0 += B) {      // the ragged tail is left to the next epoch's order
            k_gather<<<nb(B * n->n_in), 256, 0, st>>>(B, n->n_in, x, n->idx + r0, n->X16, pad8(n->n_in), nullptr);
            MH_LAUNCHED("k_gather");
            k_gather<<<nb(B * n->n_out), 256, 0, st>>>(B, n->n_out, t, n->idx + r0, nullptr, 0, n->T);
            MH_LAUNCHED("k_gather");
            if (int rc = forward_ws<kBiasSilu>(n, B, n->Y, st)) return rc;
            if (int rc = backward_ws(n, B, st)) return rc;
            n->t += 1;
            const float c1 = 1.0f - std::pow(0.9f, (float)n->t), c2 = 1.0f - std::pow(0.999f, (float)n->t);
            k_adam<<<nb(n->n_params), 256, 0, st>>>(n->n_params, n->p, n->g, n->m, n->v, n->p16, lr, 0.9f, 0.999f,
                                                    1e-8f, c1, c2);
            MH_LAUNCHED("k_adam");
            double ls = 0.0;
            if (r0 + 2 * B > rows) {           // last batch of the epoch: read its loss
                MH_CUDA(cudaMemcpyAsync(&ls, n->lsum, sizeof(double), cudaMemcpyDeviceToHost, st));
                MH_CUDA(cudaStreamSynchronize(st));
                ep_sum += ls;
                ep_rows += B;
            }
        }
        if (ep_rows) last = ep_sum / (double)(ep_rows * n->n_out);
    }
    MH_CUDA(cudaStreamSynchronize(st));
    if (final_loss) *final_loss = last;
    return MH_OK;
}

}  // extern "C"

// ttm_mlp.cu -- the learned warm start: an MLP K -> 128 -> 128 -> 3 with
// GELU activations (tanh form) and a normalised output u_hat = y / |y|
// that predicts the maximising direction of the form C . u^{(x)n} from the
// components scaled to unit Frobenius norm. Loss per sample:
// 1 - (u_hat . u*)^2 (independent of the sign of u*).
//
// Training runs on the GPU with the kernels below, seven launches a step:
// the minibatch gather, the two hidden layers (product, bias and GELU), the
// head (output layer, normalised-output loss, its gradient and the gradient
// at the second layer's pre-activations), the product back to the first
// layer, all weight and bias gradients in one launch, and the reduction of
// those with Adam. Parameters are one flat FP32 array:
// W1 [H][K], b1 [H], W2 [H][H], b2 [H], W3 [3][H], b3 [3].
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "mlp_mma.cuh"
#include "ttm_internal.h"

namespace ttm {

constexpr int kH = kMlpH;

__host__ __device__ inline int64_t mlp_num_params(int K) { return (int64_t)kH * K + kH + kH * kH + kH + 3 * kH + 3; }

// ------------------------------------------------------------- kernels --

__device__ __forceinline__ float gelu_t(float x)
{
    const float c = 0.7978845608028654f;  // sqrt(2 / pi)
    return 0.5f * x * (1.f + tanhf(c * (x + 0.044715f * x * x * x)));
}

__device__ __forceinline__ float gelu_t_grad(float x)
{
    const float c = 0.7978845608028654f;
    const float t = tanhf(c * (x + 0.044715f * x * x * x));
    return 0.5f * (1.f + t) + 0.5f * x * (1.f - t * t) * c * (1.f + 3.f * 0.044715f * x * x);
}

// Epilogues of k_gemm: a layer's pre-activation (plus bias) and GELU, or the
// gradient at a layer's pre-activations (in place of them)
enum GemmEpi { EPI_GELU = 0, EPI_GELU_GRAD = 1 };

// act[M][N] and out from op(B): acc = A op(B), A [M][K] row-major,
// op(B)[k][n] = TB ? B[n ldb + k] : B[k ldb + n].
//   EPI_GELU:      act = acc + bias, out = GELU(act)
//   EPI_GELU_GRAD: act = acc * GELU'(act) (out unused)
// 64 x 64 tiles, k steps of 16. FP32: 4 x 4 values per thread. BF16: the
// operands are rounded (nearest even) as they are staged and multiplied on
// the tensor cores (mma.sync m16n8k16, FP32 accumulate); warp w owns rows
// 16 (w >> 1) .. +16 and columns 32 (w & 1) .. +32 (shared rows of 24 BF16
// keep the fragment loads of a warp in distinct banks).
// A step's products are 4096 x 128 x 128 at most, 128 CTAs of 8 k steps: what
// bounds them is the latency of the loads, so the next step's operands are
// in registers while this one is multiplied, and lanes run along k where k
// is the contiguous index.
template <bool TB, int EPI, bool BF16>
__global__ void __launch_bounds__(256) k_gemm(int M, int N, int K, const float* __restrict__ A, int lda,
                                              const float* __restrict__ B, int ldb, const float* __restrict__ bias,
                                              float* act, float* __restrict__ out)
{
    __shared__ float As[BF16 ? 1 : 16][65], Bs[BF16 ? 1 : 16][65];
    __shared__ __align__(16) __nv_bfloat16 Ah[BF16 ? 64 : 1][24], Bh[BF16 ? 64 : 1][24];
    const int tid = threadIdx.x;
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const int ak = tid & 15, am = tid >> 4;                            // element (k, row) of A, rows + 16 i
    const int bk = TB ? tid & 15 : tid >> 6, bn = TB ? tid >> 4 : tid & 63;
    float pa[4], pb[4];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int m = m0 + am + 16 * i, k = k0 + ak;
            pa[i] = m < M && k < K ? A[(int64_t)m * lda + k] : 0.f;
            const int n = n0 + (TB ? bn + 16 * i : bn), kb = k0 + (TB ? bk : bk + 4 * i);
            pb[i] = n < N && kb < K ? (TB ? B[(int64_t)n * ldb + kb] : B[(int64_t)kb * ldb + n]) : 0.f;
        }
    };
    float acc[4][4] = {};
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int mm = am + 16 * i, nn = TB ? bn + 16 * i : bn, kb = TB ? bk : bk + 4 * i;
            if constexpr (BF16) {
                Ah[mm][ak] = __float2bfloat16_rn(pa[i]);
                Bh[nn][kb] = __float2bfloat16_rn(pb[i]);
            } else {
                As[ak][mm] = pa[i];
                Bs[kb][nn] = pb[i];
            }
        }
        __syncthreads();
        if (k0 + 16 < K) fetch(k0 + 16);
        if constexpr (BF16) {
            const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
            const int wm = (warp >> 1) * 16, wn = (warp & 1) * 32;
            uint32_t af[4];
            af[0] = ld_b32(&Ah[wm + g][2 * t]);
            af[1] = ld_b32(&Ah[wm + g + 8][2 * t]);
            af[2] = ld_b32(&Ah[wm + g][2 * t + 8]);
            af[3] = ld_b32(&Ah[wm + g + 8][2 * t + 8]);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int nn = wn + 8 * j + g;
                mma_bf16(acc[j], af, ld_b32(&Bh[nn][2 * t]), ld_b32(&Bh[nn][2 * t + 8]));
            }
        } else {
            const int tx = tid % 16, ty = tid / 16;
#pragma unroll
            for (int kk = 0; kk < 16; kk++) {
                float a[4], b[4];
#pragma unroll
                for (int i = 0; i < 4; i++) { a[i] = As[kk][ty * 4 + i]; b[i] = Bs[kk][tx + 16 * i]; }
#pragma unroll
                for (int i = 0; i < 4; i++)
#pragma unroll
                    for (int j = 0; j < 4; j++) acc[i][j] += a[i] * b[j];
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
            int m, n;
            if constexpr (BF16) {
                // accumulator (i, 2h + q): row g + 8h, column 8i + 2t + q of the warp tile
                const int lane = tid & 31, warp = tid >> 5;
                m = m0 + (warp >> 1) * 16 + (lane >> 2) + 8 * (j >> 1);
                n = n0 + (warp & 1) * 32 + 8 * i + 2 * (lane & 3) + (j & 1);
            } else {
                m = m0 + (tid / 16) * 4 + i;
                n = n0 + tid % 16 + 16 * j;
            }
            if (m >= M || n >= N) continue;
            const int64_t o = (int64_t)m * N + n;
            if constexpr (EPI == EPI_GELU) {
                const float v = acc[i][j] + bias[n];
                act[o] = v;
                out[o] = gelu_t(v);
            } else {
                act[o] = acc[i][j] * gelu_t_grad(act[o]);
            }
        }
}

// The output layer and its way back, one warp per row: y = W3 h2 + b3,
// u_hat = y / |y|; with targets the per-sample loss 1 - (u_hat . u*)^2,
// dy = (I - u_hat u_hat^T)(-2 (u_hat . u*) u*) / |y| * scale and, in place of
// a2, the gradient (dy W3) * GELU'(a2) at the second layer's
// pre-activations. BF16: operands of both products rounded to BF16.
// (As a 64 x 64-tiled product with N = 3 the output layer took 18 us of a
// 4096-row step, 3 of 64 columns in use.)
template <bool BF16>
__global__ void __launch_bounds__(256) k_mlp_head(const float* __restrict__ h2, float* __restrict__ a2,
                                                  const float* __restrict__ W3, const float* __restrict__ b3,
                                                  const float* __restrict__ U, int64_t n, float scale,
                                                  float* __restrict__ u_out, float* __restrict__ dy,
                                                  float* __restrict__ loss)
{
    auto rnd = [](float v) { return BF16 ? __bfloat162float(__float2bfloat16_rn(v)) : v; };
    const int lane = threadIdx.x & 31;
    float w[3][kH / 32];
#pragma unroll
    for (int c = 0; c < 3; c++)
#pragma unroll
        for (int q = 0; q < kH / 32; q++) w[c][q] = rnd(W3[c * kH + lane + 32 * q]);
    for (int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); i < n; i += (int64_t)gridDim.x * 8) {
        float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < kH / 32; q++) {
            const float h = rnd(h2[i * kH + lane + 32 * q]);
#pragma unroll
            for (int c = 0; c < 3; c++) v[c] += h * w[c][q];
        }
#pragma unroll
        for (int c = 0; c < 3; c++) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
            v[c] += b3[c];
        }
        const float ny = sqrtf(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
        const float inv = ny > 0.f ? 1.f / ny : 0.f;
        const float uh[3] = {v[0] * inv, v[1] * inv, v[2] * inv};
        if (u_out && lane < 3) u_out[i * 3 + lane] = uh[lane];
        if (!U) continue;
        const float us[3] = {U[i * 3], U[i * 3 + 1], U[i * 3 + 2]};
        const float dot = uh[0] * us[0] + uh[1] * us[1] + uh[2] * us[2];
        const float gu[3] = {-2.f * dot * us[0], -2.f * dot * us[1], -2.f * dot * us[2]};
        const float ug = uh[0] * gu[0] + uh[1] * gu[1] + uh[2] * gu[2];
        float d[3];
#pragma unroll
        for (int c = 0; c < 3; c++) d[c] = (gu[c] - ug * uh[c]) * inv * scale;
        if (lane < 3) dy[i * 3 + lane] = d[lane];
        if (lane == 0) loss[i] = 1.f - dot * dot;
#pragma unroll
        for (int q = 0; q < kH / 32; q++) {
            const int64_t o = i * kH + lane + 32 * q;
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < 3; c++) s += rnd(d[c]) * w[c][q];
            a2[o] = s * gelu_t_grad(a2[o]);
        }
    }
}

// All weight and bias gradients of a step, split over the rows: CTA
// (tile, s) adds rows [s chunk, (s + 1) chunk) of D^T H for a 64 x 64 tile of
// one layer's W (and D's column sums for its b) into part[s][np], in the
// layout of the parameters; k_grad_reduce adds the splits in order.
// Without the split these products are 2 to 4 CTAs that walk all rows: 0.7 ms
// each at 4096 rows under ncu, and 0.2 ms for each column sum on one CTA,
// nearly all of a step. An epoch of 16 steps of 4096 rows (K = 28) took
// 26.2 ms; with the splits (8 x 64 CTAs) and the fused epilogues it takes
// 1.46 ms, its shuffle on the host included. The parameters after that epoch
// are as far from float64 as before on eight sets of inputs (1.1e-7 of their
// norm), though single ones differ either way.
struct GradJob {
    const float *D, *H;   // [rows][M], [rows][N]
    int M, N;
    int64_t off_w, off_b;
};
struct GradJobs { GradJob j[3]; };

template <bool BF16>
__global__ void __launch_bounds__(256) k_wgrad(GradJobs jobs, int tiles1, int rows, int chunk, int64_t np,
                                               float* __restrict__ part)
{
    __shared__ float As[BF16 ? 1 : 16][65], Bs[BF16 ? 1 : 16][65];
    __shared__ __align__(16) __nv_bfloat16 Ah[BF16 ? 64 : 1][24], Bh[BF16 ? 64 : 1][24];
    __shared__ float colsum[4][64];
    const int tid = threadIdx.x;
    // tiles: 2 of W3 (3 x H), 4 of W2 (H x H), then tiles1 of W1 (H x K)
    const int b = blockIdx.x;
    const GradJob J = b < 2 ? jobs.j[2] : (b < 6 ? jobs.j[1] : jobs.j[0]);
    const int tile = b < 2 ? b : (b < 6 ? b - 2 : b - 6);
    const int tn = b < 6 ? 2 : tiles1 / 2;
    const int m0 = (tile / tn) * 64, n0 = (tile % tn) * 64;
    const int r0 = blockIdx.y * chunk, r1 = min(rows, r0 + chunk);
    const int kk0 = tid >> 6, mm = tid & 63;
    const bool am = m0 + mm < J.M, bn = n0 + mm < J.N;
    float pa[4], pb[4], bsum = 0.f;
    auto fetch = [&](int r) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int k = r + kk0 + 4 * i;
            pa[i] = am && k < r1 ? J.D[(int64_t)k * J.M + m0 + mm] : 0.f;
            pb[i] = bn && k < r1 ? J.H[(int64_t)k * J.N + n0 + mm] : 0.f;
        }
    };
    float acc[4][4] = {};
    fetch(r0);
    for (int r = r0; r < r1; r += 16) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            bsum += pa[i];
            if constexpr (BF16) {
                Ah[mm][kk0 + 4 * i] = __float2bfloat16_rn(pa[i]);
                Bh[mm][kk0 + 4 * i] = __float2bfloat16_rn(pb[i]);
            } else {
                As[kk0 + 4 * i][mm] = pa[i];
                Bs[kk0 + 4 * i][mm] = pb[i];
            }
        }
        __syncthreads();
        if (r + 16 < r1) fetch(r + 16);
        if constexpr (BF16) {
            const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
            const int wm = (warp >> 1) * 16, wn = (warp & 1) * 32;
            uint32_t af[4];
            af[0] = ld_b32(&Ah[wm + g][2 * t]);
            af[1] = ld_b32(&Ah[wm + g + 8][2 * t]);
            af[2] = ld_b32(&Ah[wm + g][2 * t + 8]);
            af[3] = ld_b32(&Ah[wm + g + 8][2 * t + 8]);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int nn = wn + 8 * j + g;
                mma_bf16(acc[j], af, ld_b32(&Bh[nn][2 * t]), ld_b32(&Bh[nn][2 * t + 8]));
            }
        } else {
            const int tx = tid % 16, ty = tid / 16;
#pragma unroll
            for (int kk = 0; kk < 16; kk++) {
                float x[4], y[4];
#pragma unroll
                for (int i = 0; i < 4; i++) { x[i] = As[kk][ty * 4 + i]; y[i] = Bs[kk][tx + 16 * i]; }
#pragma unroll
                for (int i = 0; i < 4; i++)
#pragma unroll
                    for (int j = 0; j < 4; j++) acc[i][j] += x[i] * y[j];
            }
        }
        __syncthreads();
    }
    float* dst = part + (int64_t)blockIdx.y * np;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
            int m, n;
            if constexpr (BF16) {
                const int lane = tid & 31, warp = tid >> 5;
                m = m0 + (warp >> 1) * 16 + (lane >> 2) + 8 * (j >> 1);
                n = n0 + (warp & 1) * 32 + 8 * i + 2 * (lane & 3) + (j & 1);
            } else {
                m = m0 + (tid / 16) * 4 + i;
                n = n0 + tid % 16 + 16 * j;
            }
            if (m < J.M && n < J.N) dst[J.off_w + (int64_t)m * J.N + n] = acc[i][j];
        }
    if (n0 == 0) {
        colsum[kk0][mm] = bsum;
        __syncthreads();
        if (tid < 64 && m0 + tid < J.M)
            dst[J.off_b + m0 + tid] = colsum[0][tid] + colsum[1][tid] + colsum[2][tid] + colsum[3][tid];
    }
}

struct AdamStep {
    float *p, *m, *v;  // p == nullptr: no update
    float lr, b1, b2, eps, c1, c2;
};

// g (+)= the splits of part in order; then, with a step, Adam on the parameters
__global__ void k_grad_reduce(const float* __restrict__ part, int splits, int64_t np, float* __restrict__ g, int acc,
                              AdamStep ad)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    float s = acc ? g[i] : 0.f;
#pragma unroll 8
    for (int k = 0; k < splits; k++) s += part[(int64_t)k * np + i];
    g[i] = s;
    if (!ad.p) return;
    const float mi = ad.b1 * ad.m[i] + (1.f - ad.b1) * s;
    const float vi = ad.b2 * ad.v[i] + (1.f - ad.b2) * s * s;
    ad.m[i] = mi;
    ad.v[i] = vi;
    ad.p[i] -= ad.lr * (mi / ad.c1) / (sqrtf(vi / ad.c2) + ad.eps);
}

// rows idx[i] of X (K wide) and U (3 wide) into contiguous batch buffers
__global__ void k_gather_rows(const float* __restrict__ X, const float* __restrict__ U, const int64_t* __restrict__ idx,
                              int64_t n, int K, float* __restrict__ Xb, float* __restrict__ Ub)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * (K + 3); t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / (K + 3);
        const int c = (int)(t - i * (K + 3));
        const int64_t s = idx[i];
        if (c < K) Xb[i * K + c] = X[s * K + c];
        else Ub[i * 3 + (c - K)] = U[s * 3 + (c - K)];
    }
}

__global__ void k_sum_partial(const float* __restrict__ v, int64_t n, double* __restrict__ out)
{
    __shared__ double s[256];
    double a = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) a += v[i];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = s[0];
}

// Standalone BF16 inference: u_hat of n rows of X [n][K] into U [n][3].
// Each warp stages 32 rows in shared memory and runs the tensor-core MLP.
template <int KX>
__global__ void __launch_bounds__(256) k_mlp_infer(const unsigned char* __restrict__ image, const float* __restrict__ X,
                                                   int K, int64_t n, float* __restrict__ U)
{
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char* img = smem;
    __nv_bfloat16* sx_all = reinterpret_cast<__nv_bfloat16*>(smem + kMlpImageBytes);
    float* sy_all = reinterpret_cast<float*>(smem + kMlpImageBytes + sizeof(__nv_bfloat16) * 8 * 32 * kW1S);
    mlp_image_to_smem(image, img);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __nv_bfloat16* sx = sx_all + warp * 32 * kW1S;
    float* sy = sy_all + warp * 32 * 4;
    const float* b3 = reinterpret_cast<const float*>(img + kMlpOffB3);
    const int64_t groups = (n + 31) / 32;
    for (int64_t gi = (int64_t)blockIdx.x * 8 + warp; gi < groups; gi += (int64_t)gridDim.x * 8) {
        const int64_t row = gi * 32 + lane;
        for (int k = 0; k < KX; k++)
            sx[lane * kW1S + k] = __float2bfloat16_rn(row < n && k < K ? X[row * K + k] : 0.f);
        __syncwarp();
        mlp_warp_bf16<KX>(sx, img, sy);
        __syncwarp();
        if (row < n) {
            float y0 = sy[lane * 4] + b3[0], y1 = sy[lane * 4 + 1] + b3[1], y2 = sy[lane * 4 + 2] + b3[2];
            const float nn = sqrtf(y0 * y0 + y1 * y1 + y2 * y2);
            const float inv = nn > 0.f ? 1.f / nn : 0.f;
            U[row * 3] = y0 * inv;
            U[row * 3 + 1] = y1 * inv;
            U[row * 3 + 2] = y2 * inv;
        }
        __syncwarp();
    }
}

// Training pairs from maps: X[i] = C(v_i) / ||C(v_i)||_F (zero if the norm
// is zero), U[i] = orientation at v_i; C [K][V] (order n, graded-lex).
__global__ void k_make_pairs(const float* __restrict__ C, int n_order, int K, int64_t V,
                             const float* __restrict__ orient, const int64_t* __restrict__ idx, int64_t n,
                             float* __restrict__ X, float* __restrict__ U)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = idx[i];
        float f2 = 0.f;
        int k = 0;
        for (int a = n_order; a >= 0; a--)
            for (int b = n_order - a; b >= 0; b--, k++) {
                const int c = n_order - a - b;
                float mult = 1.f;
                for (int q = 2; q <= n_order; q++) mult *= (float)q;
                for (int q = 2; q <= a; q++) mult /= (float)q;
                for (int q = 2; q <= b; q++) mult /= (float)q;
                for (int q = 2; q <= c; q++) mult /= (float)q;
                const float x = C[(int64_t)k * V + v];
                f2 += mult * x * x;
            }
        const float inv = f2 > 0.f ? rsqrtf(f2) : 0.f;
        for (k = 0; k < K; k++) X[i * K + k] = C[(int64_t)k * V + v] * inv;
        for (int c = 0; c < 3; c++) U[i * 3 + c] = orient[(int64_t)c * V + v];
    }
}

// ---------------------------------------------------------------- host --

// counter-based SplitMix64 for the initial weights
static uint64_t splitmix(uint64_t z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
static double u01(uint64_t seed, uint64_t i) { return (splitmix(seed ^ (i * 0xD1B54A32D192ED03ull)) >> 11) * 0x1.0p-53; }

// FP32 -> BF16 with round to nearest even (finite inputs)
static uint16_t bf16_rne(float f)
{
    uint32_t u;
    std::memcpy(&u, &f, 4);
    u += 0x7FFFu + ((u >> 16) & 1u);
    return (uint16_t)(u >> 16);
}

void mlp_refresh_image(ttm_mlp* M)
{
    if (!M->image_dirty && M->image.p) return;
    const int K = M->K;
    std::vector<float> p(M->np);
    TTM_CUDA_TRY(cudaMemcpy(p.data(), M->params.p, M->np * sizeof(float), cudaMemcpyDeviceToHost));
    std::vector<unsigned char> img(kMlpImageBytes, 0);
    uint16_t* W1 = reinterpret_cast<uint16_t*>(img.data() + kMlpOffW1);
    uint16_t* W2 = reinterpret_cast<uint16_t*>(img.data() + kMlpOffW2);
    uint16_t* W3 = reinterpret_cast<uint16_t*>(img.data() + kMlpOffW3);
    float* b1 = reinterpret_cast<float*>(img.data() + kMlpOffB1);
    float* b2 = reinterpret_cast<float*>(img.data() + kMlpOffB2);
    float* b3 = reinterpret_cast<float*>(img.data() + kMlpOffB3);
    const float* pW1 = p.data();
    const float* pb1 = pW1 + (size_t)kH * K;
    const float* pW2 = pb1 + kH;
    const float* pb2 = pW2 + (size_t)kH * kH;
    const float* pW3 = pb2 + kH;
    const float* pb3 = pW3 + 3 * kH;
    for (int j = 0; j < kH; j++) {
        for (int k = 0; k < K; k++) W1[j * kW1S + k] = bf16_rne(pW1[(size_t)j * K + k]);
        for (int k = 0; k < kH; k++) W2[j * kW2S + k] = bf16_rne(pW2[(size_t)j * kH + k]);
        b1[j] = pb1[j];
        b2[j] = pb2[j];
    }
    for (int o = 0; o < 3; o++) {
        for (int k = 0; k < kH; k++) W3[o * kW2S + k] = bf16_rne(pW3[o * kH + k]);
        b3[o] = pb3[o];
    }
    if (!M->image.p) M->image.alloc(kMlpImageBytes);
    TTM_CUDA_TRY(cudaMemcpy(M->image.p, img.data(), kMlpImageBytes, cudaMemcpyHostToDevice));
    M->image_dirty = false;
}

}  // namespace ttm

namespace ttm {

// row splits of the weight gradients: at least 64 rows each (four k steps),
// at most 64 splits (8 tiles x 64 splits are 3.4 CTAs per SM)
constexpr int kGradSplits = 64;

static void mlp_scratch(ttm_mlp* M, int64_t rows)
{
    if (rows <= M->cap) return;
    const int K = M->K;
    M->xb.alloc(rows * K * sizeof(float));
    M->ub.alloc(rows * 3 * sizeof(float));
    M->a1.alloc(rows * kH * sizeof(float));
    M->h1.alloc(rows * kH * sizeof(float));
    M->a2.alloc(rows * kH * sizeof(float));
    M->h2.alloc(rows * kH * sizeof(float));
    M->dy.alloc(rows * 3 * sizeof(float));
    M->loss.alloc(rows * sizeof(float));
    M->part.alloc(256 * sizeof(double));
    M->gpart.alloc((size_t)kGradSplits * M->np * sizeof(float));
    M->cap = rows;
}

struct MlpView {
    const float *W1, *b1, *W2, *b2, *W3, *b3;
};
static MlpView view(const float* p, int K)
{
    MlpView v;
    v.W1 = p;
    v.b1 = v.W1 + (size_t)kH * K;
    v.W2 = v.b1 + kH;
    v.b2 = v.W2 + (size_t)kH * kH;
    v.W3 = v.b2 + kH;
    v.b3 = v.W3 + 3 * kH;
    return v;
}

template <bool TB, int EPI>
static void gemm(bool bf16, int M, int N, int K, const float* A, int lda, const float* B, int ldb, const float* bias,
                 float* act, float* out, cudaStream_t st)
{
    const dim3 grid((unsigned)ceil_div(N, 64), (unsigned)ceil_div(M, 64));
    if (bf16) k_gemm<TB, EPI, true><<<grid, 256, 0, st>>>(M, N, K, A, lda, B, ldb, bias, act, out);
    else k_gemm<TB, EPI, false><<<grid, 256, 0, st>>>(M, N, K, A, lda, B, ldb, bias, act, out);
    TTM_LAUNCH_CHECK();
}

// forward of `rows` rows: fills a1..h2 (a2 then holds the gradient at the
// second layer's pre-activations if there are targets); u_out gets u_hat if
// not null; with targets fills loss and dy (scaled by dscale)
static void mlp_forward_rows(ttm_mlp* M, const float* X, const float* U, int64_t rows, float* u_out, float dscale,
                             cudaStream_t st)
{
    const int K = M->K;
    MlpView w = view(M->params.as<float>(), K);
    float *a1 = M->a1.as<float>(), *h1 = M->h1.as<float>(), *a2 = M->a2.as<float>(), *h2 = M->h2.as<float>();
    gemm<true, EPI_GELU>(M->bf16, (int)rows, kH, K, X, K, w.W1, K, w.b1, a1, h1, st);
    gemm<true, EPI_GELU>(M->bf16, (int)rows, kH, kH, h1, kH, w.W2, kH, w.b2, a2, h2, st);
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(rows, 8), 1024);
    if (M->bf16)
        k_mlp_head<true><<<grid, 256, 0, st>>>(h2, a2, w.W3, w.b3, U, rows, dscale, u_out, M->dy.as<float>(),
                                               M->loss.as<float>());
    else
        k_mlp_head<false><<<grid, 256, 0, st>>>(h2, a2, w.W3, w.b3, U, rows, dscale, u_out, M->dy.as<float>(),
                                                M->loss.as<float>());
    TTM_LAUNCH_CHECK();
}

// gradient of the loss of the rows in the last forward (dy already scaled),
// into g (accumulated if acc), then the Adam step if ad.p is set
static void mlp_backward_rows(ttm_mlp* M, const float* X, int64_t rows, float* g, bool acc, const AdamStep& ad,
                              cudaStream_t st)
{
    const int K = M->K;
    MlpView w = view(M->params.as<float>(), K);
    float *a1 = M->a1.as<float>(), *h1 = M->h1.as<float>(), *d2 = M->a2.as<float>(), *h2 = M->h2.as<float>();
    // d1 = (d2 W2) * GELU'(a1), in place of a1
    gemm<false, EPI_GELU_GRAD>(M->bf16, (int)rows, kH, kH, d2, kH, w.W2, kH, nullptr, a1, nullptr, st);
    const int64_t o_b1 = (int64_t)kH * K, o_W2 = o_b1 + kH, o_b2 = o_W2 + kH * kH, o_W3 = o_b2 + kH, o_b3 = o_W3 + 3 * kH;
    GradJobs jobs;
    jobs.j[0] = GradJob{a1, X, kH, K, 0, o_b1};
    jobs.j[1] = GradJob{d2, h1, kH, kH, o_W2, o_b2};
    jobs.j[2] = GradJob{M->dy.as<float>(), h2, 3, kH, o_W3, o_b3};
    const int chunk = (int)std::max<int64_t>(64, ceil_div(ceil_div(rows, kGradSplits), 16) * 16);
    const int splits = (int)ceil_div(rows, chunk);
    const int tiles1 = 2 * (int)ceil_div(K, 64);
    const dim3 grid((unsigned)(6 + tiles1), (unsigned)splits);
    float* part = M->gpart.as<float>();
    if (M->bf16) k_wgrad<true><<<grid, 256, 0, st>>>(jobs, tiles1, (int)rows, chunk, M->np, part);
    else k_wgrad<false><<<grid, 256, 0, st>>>(jobs, tiles1, (int)rows, chunk, M->np, part);
    TTM_LAUNCH_CHECK();
    k_grad_reduce<<<(unsigned)ceil_div(M->np, 128), 128, 0, st>>>(part, splits, M->np, g, acc, ad);
    TTM_LAUNCH_CHECK();
}

static double sum_loss(ttm_mlp* M, int64_t rows, cudaStream_t st)
{
    k_sum_partial<<<256, 256, 0, st>>>(M->loss.as<float>(), rows, M->part.as<double>());
    TTM_LAUNCH_CHECK();
    std::vector<double> h(256);
    TTM_CUDA_TRY(cudaMemcpyAsync(h.data(), M->part.p, 256 * sizeof(double), cudaMemcpyDeviceToHost, st));
    TTM_CUDA_TRY(cudaStreamSynchronize(st));
    double s = 0.0;
    for (double x : h) s += x;
    return s;
}

}  // namespace ttm

using namespace ttm;

extern "C" int64_t ttm_mlp_num_params(int n_inputs) { return n_inputs > 0 ? mlp_num_params(n_inputs) : 0; }

extern "C" ttm_status ttm_mlp_create(ttm_ctx* ctx, int n_inputs, uint64_t seed, ttm_mlp** out)
{
    if (!ctx || !out || n_inputs <= 0 || n_inputs > 128) return TTM_E_INVALID_ARG;
    ttm_mlp* M = new ttm_mlp();
    try {
        TTM_CUDA_TRY(cudaSetDevice(ctx->device));
        M->ctx = ctx;
        M->K = n_inputs;
        M->np = mlp_num_params(n_inputs);
        M->params.alloc(M->np * sizeof(float));
        M->grad.alloc(M->np * sizeof(float));
        M->m.alloc(M->np * sizeof(float));
        M->v.alloc(M->np * sizeof(float));
        // weights ~ N(0, 1/fan_in) by Box-Muller on SplitMix64 counters, biases 0
        std::vector<float> h(M->np, 0.f);
        const int K = n_inputs;
        auto fill = [&](size_t off, int64_t count, int fan_in, uint64_t stream) {
            const double sd = 1.0 / std::sqrt((double)fan_in);
            for (int64_t i = 0; i < count; i++) {
                double u1 = u01(seed + stream, 2 * i), u2 = u01(seed + stream, 2 * i + 1);
                double z = std::sqrt(-2.0 * std::log1p(-u1)) * std::cos(2.0 * M_PI * u2);
                h[off + i] = (float)(sd * z);
            }
        };
        fill(0, (int64_t)kH * K, K, 1);
        fill((size_t)kH * K + kH, (int64_t)kH * kH, kH, 2);
        fill((size_t)kH * K + kH + kH * kH + kH, 3 * kH, kH, 3);
        TTM_CUDA_TRY(cudaMemcpy(M->params.p, h.data(), M->np * sizeof(float), cudaMemcpyHostToDevice));
        TTM_CUDA_TRY(cudaMemset(M->m.p, 0, M->np * sizeof(float)));
        TTM_CUDA_TRY(cudaMemset(M->v.p, 0, M->np * sizeof(float)));
        *out = M;
        return TTM_OK;
    } catch (const Error& e) {
        delete M;
        return (ttm_status)fail(ctx, e);
    }
}

extern "C" void ttm_mlp_destroy(ttm_mlp* mlp) { delete mlp; }

extern "C" int ttm_mlp_inputs(const ttm_mlp* mlp) { return mlp ? mlp->K : 0; }

extern "C" ttm_status ttm_mlp_get_params(const ttm_mlp* mlp, float* h_params)
{
    if (!mlp || !h_params) return TTM_E_INVALID_ARG;
    try {
        TTM_CUDA_TRY(cudaMemcpy(h_params, mlp->params.p, mlp->np * sizeof(float), cudaMemcpyDeviceToHost));
        return TTM_OK;
    } catch (const Error& e) {
        return (ttm_status)fail(mlp->ctx, e);
    }
}

extern "C" ttm_status ttm_mlp_set_params(ttm_mlp* mlp, const float* h_params)
{
    if (!mlp || !h_params) return TTM_E_INVALID_ARG;
    try {
        TTM_CUDA_TRY(cudaMemcpy(mlp->params.p, h_params, mlp->np * sizeof(float), cudaMemcpyHostToDevice));
        TTM_CUDA_TRY(cudaMemset(mlp->m.p, 0, mlp->np * sizeof(float)));
        TTM_CUDA_TRY(cudaMemset(mlp->v.p, 0, mlp->np * sizeof(float)));
        mlp->step = 0;
        mlp->image_dirty = true;
        return TTM_OK;
    } catch (const Error& e) {
        return (ttm_status)fail(mlp->ctx, e);
    }
}

extern "C" ttm_status ttm_mlp_forward(ttm_mlp* mlp, const float* d_X, int64_t n, float* d_U, void* stream)
{
    if (!mlp || !d_X || !d_U || n < 0) return TTM_E_INVALID_ARG;
    try {
        cudaStream_t st = (cudaStream_t)stream;
        const int64_t chunk = 65536;
        mlp_scratch(mlp, std::min<int64_t>(std::max<int64_t>(n, 1), chunk));
        for (int64_t s = 0; s < n; s += chunk) {
            const int64_t r = std::min(chunk, n - s);
            mlp_forward_rows(mlp, d_X + s * mlp->K, nullptr, r, d_U + s * 3, 1.f, st);
        }
        return TTM_OK;
    } catch (const Error& e) {
        return (ttm_status)fail(mlp->ctx, e);
    }
}

extern "C" ttm_status ttm_mlp_loss_grad(ttm_mlp* mlp, const float* d_X, const float* d_U, int64_t n, float* d_grad,
                                        double* h_loss, void* stream)
{
    if (!mlp || !d_X || !d_U || !d_grad || n <= 0) return TTM_E_INVALID_ARG;
    try {
        cudaStream_t st = (cudaStream_t)stream;
        const int64_t chunk = 65536;
        mlp_scratch(mlp, std::min(n, chunk));
        double L = 0.0;
        for (int64_t s = 0; s < n; s += chunk) {
            const int64_t r = std::min(chunk, n - s);
            mlp_forward_rows(mlp, d_X + s * mlp->K, d_U + s * 3, r, nullptr, 1.f, st);
            mlp_backward_rows(mlp, d_X + s * mlp->K, r, d_grad, s > 0, AdamStep{}, st);
            L += sum_loss(mlp, r, st);
        }
        if (h_loss) *h_loss = L;
        return TTM_OK;
    } catch (const Error& e) {
        return (ttm_status)fail(mlp->ctx, e);
    }
}

extern "C" ttm_status ttm_mlp_train(ttm_mlp* mlp, const float* d_X, const float* d_U, int64_t n, int epochs, int batch,
                                    float lr, uint64_t seed, double* h_last_loss, void* stream)
{
    if (!mlp || !d_X || !d_U || n <= 0 || epochs <= 0 || batch <= 0 || !(lr > 0)) return TTM_E_INVALID_ARG;
    try {
        cudaStream_t st = (cudaStream_t)stream;
        const int64_t B = std::min<int64_t>(batch, n);
        mlp_scratch(mlp, B);
        const int K = mlp->K;
        std::vector<int64_t> perm(n);
        DevBuf dperm;
        dperm.alloc(n * sizeof(int64_t));
        double last = 0.0;
        for (int ep = 0; ep < epochs; ep++) {
            // Fisher-Yates with SplitMix64 counters
            for (int64_t i = 0; i < n; i++) perm[i] = i;
            for (int64_t i = n - 1; i > 0; i--) {
                int64_t j = (int64_t)(u01(seed + 17 + ep, i) * (double)(i + 1));
                if (j > i) j = i;
                std::swap(perm[i], perm[j]);
            }
            TTM_CUDA_TRY(cudaMemcpyAsync(dperm.p, perm.data(), n * sizeof(int64_t), cudaMemcpyHostToDevice, st));
            double ep_loss = 0.0;
            for (int64_t b0 = 0; b0 + B <= n; b0 += B) {
                k_gather_rows<<<512, 256, 0, st>>>(d_X, d_U, dperm.as<int64_t>() + b0, B, K, mlp->xb.as<float>(),
                                                   mlp->ub.as<float>());
                TTM_LAUNCH_CHECK();
                // mean loss over the batch
                mlp_forward_rows(mlp, mlp->xb.as<float>(), mlp->ub.as<float>(), B, nullptr, 1.f / (float)B, st);
                mlp->step++;
                const float b1 = 0.9f, b2 = 0.999f;
                const float c1 = 1.f - std::pow(b1, (float)mlp->step), c2 = 1.f - std::pow(b2, (float)mlp->step);
                mlp_backward_rows(mlp, mlp->xb.as<float>(), B, mlp->grad.as<float>(), false,
                                  AdamStep{mlp->params.as<float>(), mlp->m.as<float>(), mlp->v.as<float>(), lr, b1,
                                           b2, 1e-8f, c1, c2},
                                  st);
                if (b0 + 2 * B > n) ep_loss = sum_loss(mlp, B, st) / (double)B;
            }
            last = ep_loss;
        }
        TTM_CUDA_TRY(cudaStreamSynchronize(st));
        mlp->image_dirty = true;
        if (h_last_loss) *h_last_loss = last;
        return TTM_OK;
    } catch (const Error& e) {
        return (ttm_status)fail(mlp->ctx, e);
    }
}

// file: "TTMMLP1\0", int32 K, int32 H, int64 nparams, float params[]
extern "C" ttm_status ttm_mlp_save(const ttm_mlp* mlp, const char* path)
{
    if (!mlp || !path) return TTM_E_INVALID_ARG;
    std::vector<float> h(mlp->np);
    ttm_status s = ttm_mlp_get_params(mlp, h.data());
    if (s != TTM_OK) return s;
    FILE* f = std::fopen(path, "wb");
    if (!f) return TTM_E_INVALID_ARG;
    const char magic[8] = {'T', 'T', 'M', 'M', 'L', 'P', '1', 0};
    int32_t K = mlp->K, H = kH;
    int64_t np = mlp->np;
    bool ok = std::fwrite(magic, 1, 8, f) == 8 && std::fwrite(&K, 4, 1, f) == 1 && std::fwrite(&H, 4, 1, f) == 1 &&
              std::fwrite(&np, 8, 1, f) == 1 && std::fwrite(h.data(), sizeof(float), np, f) == (size_t)np;
    std::fclose(f);
    return ok ? TTM_OK : TTM_E_INTERNAL;
}

extern "C" ttm_status ttm_mlp_load(ttm_ctx* ctx, const char* path, ttm_mlp** out)
{
    if (!ctx || !path || !out) return TTM_E_INVALID_ARG;
    FILE* f = std::fopen(path, "rb");
    if (!f) return TTM_E_INVALID_ARG;
    char magic[8];
    int32_t K = 0, H = 0;
    int64_t np = 0;
    bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, "TTMMLP1", 7) == 0 && std::fread(&K, 4, 1, f) == 1 &&
              std::fread(&H, 4, 1, f) == 1 && std::fread(&np, 8, 1, f) == 1 && H == kH && K > 0 && K <= 128 &&
              np == mlp_num_params(K);
    std::vector<float> h;
    if (ok) {
        h.resize(np);
        ok = std::fread(h.data(), sizeof(float), np, f) == (size_t)np;
    }
    std::fclose(f);
    if (!ok) return TTM_E_INVALID_ARG;
    ttm_status s = ttm_mlp_create(ctx, K, 0, out);
    if (s != TTM_OK) return s;
    return ttm_mlp_set_params(*out, h.data());
}

extern "C" ttm_status ttm_mlp_infer(ttm_mlp* mlp, const float* d_X, int64_t n, float* d_U, void* stream)
{
    if (!mlp || !d_X || !d_U || n < 0) return TTM_E_INVALID_ARG;
    try {
        TTM_CUDA_TRY(cudaSetDevice(mlp->ctx->device));
        mlp_refresh_image(mlp);
        if (n == 0) return TTM_OK;
        const size_t smem = kMlpImageBytes + sizeof(__nv_bfloat16) * 8 * 32 * kW1S + sizeof(float) * 8 * 32 * 4;
        const int64_t groups = (n + 31) / 32;
        const int grid = (int)std::min<int64_t>((groups + 7) / 8, (int64_t)mlp->ctx->num_sms * 8);
        cudaStream_t st = (cudaStream_t)stream;
        if (mlp_kx(mlp->K) == 16) {
            TTM_CUDA_TRY(cudaFuncSetAttribute(k_mlp_infer<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_mlp_infer<16><<<grid, 256, smem, st>>>(mlp->image.as<unsigned char>(), d_X, mlp->K, n, d_U);
        } else if (mlp_kx(mlp->K) == 32) {
            TTM_CUDA_TRY(cudaFuncSetAttribute(k_mlp_infer<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_mlp_infer<32><<<grid, 256, smem, st>>>(mlp->image.as<unsigned char>(), d_X, mlp->K, n, d_U);
        } else {
            throw Error{E_UNSUPPORTED, "tensor-core inference takes at most 32 inputs"};
        }
        TTM_LAUNCH_CHECK();
        return TTM_OK;
    } catch (const Error& e) {
        return (ttm_status)fail(mlp->ctx, e);
    }
}

extern "C" ttm_status ttm_mlp_make_pairs(ttm_ctx* ctx, const float* d_C, int order_n, int64_t V, const float* d_orient,
                                         const int64_t* d_idx, int64_t n, float* d_X, float* d_U, void* stream)
{
    if (!ctx) return TTM_E_INVALID_ARG;
    try {
        TTM_REQUIRE(d_C && d_orient && d_idx && d_X && d_U && V > 0 && n >= 0, E_INVALID_ARG, "bad argument");
        TTM_REQUIRE(order_n >= 1 && order_n <= 12, E_UNSUPPORTED, "order out of range");
        TTM_CUDA_TRY(cudaSetDevice(ctx->device));
        if (n == 0) return TTM_OK;
        const int K = (order_n + 1) * (order_n + 2) / 2;
        k_make_pairs<<<(unsigned)std::min<int64_t>(ceil_div(n, 256), 4096), 256, 0, (cudaStream_t)stream>>>(
            d_C, order_n, K, V, d_orient, d_idx, n, d_X, d_U);
        TTM_LAUNCH_CHECK();
        return TTM_OK;
    } catch (const Error& e) {
        return (ttm_status)fail(ctx, e);
    }
}

extern "C" ttm_status ttm_mlp_set_precision(ttm_mlp* mlp, int mode)
{
    if (!mlp || (mode != TTM_MLP_FP32 && mode != TTM_MLP_BF16)) return TTM_E_INVALID_ARG;
    mlp->bf16 = mode == TTM_MLP_BF16;
    return TTM_OK;
}

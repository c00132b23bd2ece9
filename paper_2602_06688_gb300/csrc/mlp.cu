// Learned nonlinear reconstructor: a 3-layer perceptron (slopes -> modes)
// with GELU, trained by the project's own forward/backward kernels and Adam.
// Not in the paper (its reconstructor is the linear Modalrec): a nonlinear
// alternative trained on simulated pairs, with BF16 weights, FP32
// accumulation and batch 256 (the 8 m and 39 m learned workloads).
//
// Layout.  Widths are padded to multiples of 128 (zero pads stay zero: their
// inputs and output gradients are zero) and the batch to a multiple of 128,
// so every contraction is one tensor-core GEMM  C = A . B^T  with both
// operands K-major bf16 (specula_gemm_bf16):
//   forward   Z_l = H_{l-1} W_l^T          A = H_{l-1} [B][in],  B = W_l [out][in]
//   dW_l      dW_l = dZ_l^T H_{l-1}        A = dZ_l^T [out][B],  B = H_{l-1}^T [in][B]
//   dH_{l-1}  dH = dZ_l W_l                A = dZ_l [B][out],    B = W_l^T [in][out]
// The element-wise kernels that produce H, dZ and the bf16 weights also
// write their transposed copies (32 x 32 shared-memory tiles), so no GEMM
// needs an MN-major operand.  FP32 master weights and Adam moments; bf16
// copies refreshed after every update.  Reductions (bias gradients, loss)
// run in a fixed order: bit-reproducible.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "internal.h"

namespace specula {

constexpr int TT = 32;   // transpose tile
// Thread rows of a tile kernel: one element per thread.  The training step's
// kernels cover 256 rows by about 1000 columns, so the time is that of a few
// rounds of loads; four elements per thread were four times the rounds
// (gelu' of 256 x 1024 from 16 partials: 13.8 us).  Matrices of more than four waves
// of such blocks take eight rows, four elements per thread (tile_rows): their time is
// that of the blocks (4096 x 2560 inputs: 41 us with 32 rows, 28 with 8; bias and GELU of
// 4096 x 1024: 26, 23).
constexpr int TY = 32, TYL = 8;
static int tile_rows(int R, int C, int sms) {
  return (long long)(R / TT) * (C / TT) > 8LL * sms ? TYL : TY;
}

__device__ __forceinline__ float gelu_f(float z) {
  return 0.5f * z * (1.0f + erff(z * (float)M_SQRT1_2));
}
__device__ __forceinline__ float gelu_grad_f(float z) {
  const float inv_sqrt_2pi = 0.5f * (float)M_2_SQRTPI * (float)M_SQRT1_2;   // 1/sqrt(2 pi)
  return 0.5f * (1.0f + erff(z * (float)M_SQRT1_2)) + z * expf(-0.5f * z * z) * inv_sqrt_2pi;
}

// Tiled writer of a bf16 matrix and, where outT is given, its transpose.  Block (32, RY), grid
// (C/32, R/32); the value function is evaluated once per element.
template <int RY, class F>
__device__ __forceinline__ void tile_bf16_pair(int R, int C, __nv_bfloat16 *out,
                                               __nv_bfloat16 *outT, F value) {
  __shared__ __nv_bfloat16 tile[TT][TT + 2];
  const int c0 = blockIdx.x * TT, r0 = blockIdx.y * TT;
#pragma unroll
  for (int k = 0; k < TT / RY; ++k) {
    const int dr = threadIdx.y + RY * k, r = r0 + dr, c = c0 + threadIdx.x;
    __nv_bfloat16 v = __float2bfloat16_rn(0.f);
    if (r < R && c < C) {
      v = __float2bfloat16_rn(value(r, c));
      out[(size_t)r * C + c] = v;
    }
    tile[dr][threadIdx.x] = v;
  }
  if (!outT) return;   // the whole launch
  __syncthreads();
#pragma unroll
  for (int k = 0; k < TT / RY; ++k) {
    const int dc = threadIdx.y + RY * k, c = c0 + dc, r = r0 + threadIdx.x;
    if (r < R && c < C) outT[(size_t)c * R + r] = tile[threadIdx.x][dc];
  }
}

// X [B][n_in] float -> Xb [Bp][in_pad] and XbT [in_pad][Bp] (zero pads)
template <int RY>
__global__ void __launch_bounds__(TT * RY) k_pack_input(const float *__restrict__ X, int B,
                                                       int n_in, int Bp, int in_pad,
                                                       __nv_bfloat16 *Xb, __nv_bfloat16 *XbT) {
  pdl_wait();
  tile_bf16_pair<RY>(Bp, in_pad, Xb, XbT, [&](int r, int c) {
    return (r < B && c < n_in) ? X[(size_t)r * n_in + c] : 0.f;
  });
}

// A GEMM's result as its split-K partials part[s][R][C], added in split order.
// The kernel that consumes a product adds them itself: a separate reduction
// wrote and re-read every product once more (nine launches of a training step).
struct Partials {
  const float *p;
  int splits;
  size_t n;   // R C
};
__device__ __forceinline__ float partial_sum(const Partials &P, size_t e) {
  // eight loads in flight, added in order
  float v = 0.f;
  int s = 0;
  for (; s + 8 <= P.splits; s += 8) {
    float x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = __ldg(P.p + (size_t)(s + u) * P.n + e);
#pragma unroll
    for (int u = 0; u < 8; ++u) v += x[u];
  }
  if (s < P.splits) {
    float x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = s + u < P.splits ? __ldg(P.p + (size_t)(s + u) * P.n + e) : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (s + u < P.splits) v += x[u];
  }
  return v;
}

// Z = sum of partials + bias; H = gelu(Z) and its transpose in bf16
template <int RY>
__global__ void __launch_bounds__(TT * RY) k_bias_gelu(const Partials P,
                                                      const float *__restrict__ bias,
                                                      float *__restrict__ Z, int R, int C,
                                                      __nv_bfloat16 *H, __nv_bfloat16 *HT) {
  pdl_wait();
  tile_bf16_pair<RY>(R, C, H, HT, [&](int r, int c) {
    const size_t e = (size_t)r * C + c;
    const float z = partial_sum(P, e) + bias[c];
    Z[e] = z;
    return gelu_f(z);
  });
}

// Y = sum of partials + bias (padded, for the backward pass) and, when given,
// the caller's [B][n_out]
__global__ void __launch_bounds__(256) k_output(const Partials P, const float *__restrict__ bias,
                                                int C, float *__restrict__ Y, int B, int n_out,
                                                float *__restrict__ out) {
  pdl_wait();
  const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (e >= P.n) return;
  const int r = (int)(e / C), c = (int)(e - (size_t)r * C);
  const float y = partial_sum(P, e) + bias[c];
  Y[e] = y;
  if (out && r < B && c < n_out) out[(size_t)r * n_out + c] = y;
}

// dA = (sum of partials) gelu'(Z); bf16 dZ and its transpose
template <int RY>
__global__ void __launch_bounds__(TT * RY) k_gelu_back(const Partials P,
                                                      const float *__restrict__ Z, float *dA,
                                                      int R, int C, __nv_bfloat16 *dZb,
                                                      __nv_bfloat16 *dZbT) {
  pdl_wait();
  tile_bf16_pair<RY>(R, C, dZb, dZbT, [&](int r, int c) {
    const size_t e = (size_t)r * C + c;
    const float d = partial_sum(P, e) * gelu_grad_f(Z[e]);
    dA[e] = d;
    return d;
  });
}

// The bias gradients, the column sums of dZ, where the weight gradients' launch does
// not take them along
__global__ void __launch_bounds__(128) k_bias_grad(const ColSums S) {
  pdl_wait();
  column_sums(S, blockIdx.x * 4 + (threadIdx.x >> 5), gridDim.x * 4);
}

// dY = scale (Y - T) on the B x n_out block, zero on pads, in bf16 with its
// transpose; loss = inv_count x the squared residuals' sum, each block's in part,
// added by the block that finishes last (done counts, wrapping to zero)
__global__ void __launch_bounds__(TT * TY) k_loss_grad(
    const float *__restrict__ Y, const float *__restrict__ T, int B, int n_out, int Bp,
    int out_pad, float scale, float *dYf, __nv_bfloat16 *dYb, __nv_bfloat16 *dYbT, unsigned *done,
    float *__restrict__ part, float inv_count, float *__restrict__ loss) {
  pdl_wait();
  __shared__ float s_sq[2][TY];
  float sq = 0.f;
  tile_bf16_pair<TY>(Bp, out_pad, dYb, dYbT, [&](int r, int c) {
    float d = 0.f;
    if (r < B && c < n_out) d = Y[(size_t)r * out_pad + c] - T[(size_t)r * n_out + c];
    sq += d * d;
    const float g = scale * d;
    dYf[(size_t)r * out_pad + c] = g;
    return g;
  });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  if (threadIdx.x == 0) s_sq[0][threadIdx.y] = sq;
  __syncthreads();
  __shared__ bool s_end;
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    float s = 0.f;
    for (int y = 0; y < TY; ++y) s += s_sq[0][y];
    __stcg(part + blockIdx.y * gridDim.x + blockIdx.x, s);
    __threadfence();
    const unsigned last = gridDim.x * gridDim.y - 1;
    s_end = atomicInc(done, last) == last;
  }
  __syncthreads();
  if (!s_end) return;
  __threadfence();
  const int n = gridDim.x * gridDim.y, t = threadIdx.y * TT + threadIdx.x;
  float s = 0.f;
  for (int i = t; i < n; i += TT * TY) s += __ldcg(part + i);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0) s_sq[1][threadIdx.y] = s;
  __syncthreads();
  if (t == 0) {
    s = 0.f;
    for (int y = 0; y < TY; ++y) s += s_sq[1][y];
    *loss = s * inv_count;
  }
}

__device__ __forceinline__ void adam_step(float &p, float &m, float &v, float g, float lr_t,
                                          float b1, float b2, float eps) {
  m = b1 * m + (1.f - b1) * g;
  v = b2 * v + (1.f - b2) * g * g;
  p -= lr_t * m / (sqrtf(v) + eps);
}

// Adam on every layer's weights and biases in one launch; the updated
// weights' bf16 copy and its transpose come from the same registers (three
// launches per layer and one more pass over the weights before).  Blocks
// [first[l], first[l + 1]) are layer l's 32 x 128 weight tiles, a row of
// four-float loads per warp; the rest 256 bias entries each.  Bound by L2: 32
// bytes per weight.
constexpr int kAdamC = 128;
struct AdamLayer {
  float *W, *mW, *vW, *b, *mb, *vb;
  const float *gW, *gb;
  __nv_bfloat16 *Wb, *WbT;
  int R, C;
};
struct AdamArgs {
  AdamLayer L[3];
  int first[4], bias_first[4];
};
__global__ void __launch_bounds__(TT * 8) k_adam(const AdamArgs A, float lr_t, float b1, float b2,
                                                 float eps) {
  pdl_wait();
  __shared__ __nv_bfloat16 tile[kAdamC][TT + 2];   // transposed
  const int blk = blockIdx.x, lane = threadIdx.x, warp = threadIdx.y;
  if (blk >= A.first[3]) {
    const int q = blk - A.first[3];
    const int l = q >= A.bias_first[2] ? 2 : (q >= A.bias_first[1] ? 1 : 0);
    const AdamLayer &L = A.L[l];
    const int i = (q - A.bias_first[l]) * (TT * 8) + warp * TT + lane;
    if (i < L.R) adam_step(L.b[i], L.mb[i], L.vb[i], L.gb[i], lr_t, b1, b2, eps);
    return;
  }
  const int l = blk >= A.first[2] ? 2 : (blk >= A.first[1] ? 1 : 0);
  const AdamLayer &L = A.L[l];
  const int tiles_c = L.C / kAdamC, q = blk - A.first[l];   // widths are multiples of 128
  const int r0 = q / tiles_c * TT, c0 = q % tiles_c * kAdamC;
  constexpr int NR = TT / 8;
  float4 p[NR], m[NR], v[NR], g[NR];
#pragma unroll
  for (int k = 0; k < NR; ++k) {
    const size_t e = (size_t)(r0 + warp + 8 * k) * L.C + c0 + 4 * lane;
    p[k] = *reinterpret_cast<const float4 *>(L.W + e);
    m[k] = *reinterpret_cast<const float4 *>(L.mW + e);
    v[k] = *reinterpret_cast<const float4 *>(L.vW + e);
    g[k] = __ldg(reinterpret_cast<const float4 *>(L.gW + e));
  }
#pragma unroll
  for (int k = 0; k < NR; ++k) {
    const int dr = warp + 8 * k;
    const size_t e = (size_t)(r0 + dr) * L.C + c0 + 4 * lane;
    adam_step(p[k].x, m[k].x, v[k].x, g[k].x, lr_t, b1, b2, eps);
    adam_step(p[k].y, m[k].y, v[k].y, g[k].y, lr_t, b1, b2, eps);
    adam_step(p[k].z, m[k].z, v[k].z, g[k].z, lr_t, b1, b2, eps);
    adam_step(p[k].w, m[k].w, v[k].w, g[k].w, lr_t, b1, b2, eps);
    *reinterpret_cast<float4 *>(L.W + e) = p[k];
    *reinterpret_cast<float4 *>(L.mW + e) = m[k];
    *reinterpret_cast<float4 *>(L.vW + e) = v[k];
    __nv_bfloat162 w[2] = {__floats2bfloat162_rn(p[k].x, p[k].y),
                           __floats2bfloat162_rn(p[k].z, p[k].w)};
    *reinterpret_cast<uint2 *>(L.Wb + e) = *reinterpret_cast<const uint2 *>(w);
    tile[4 * lane][dr] = w[0].x;
    tile[4 * lane + 1][dr] = w[0].y;
    tile[4 * lane + 2][dr] = w[1].x;
    tile[4 * lane + 3][dr] = w[1].y;
  }
  if (!L.WbT) return;   // the first layer's: nothing multiplies by it
  __syncthreads();
  // a column's 32 rows are 64 bytes: two columns per warp
  const int half = lane / 16, pr = 2 * (lane % 16);
#pragma unroll
  for (int k = 0; k < kAdamC / 16; ++k) {
    const int c = 16 * k + 2 * warp + half;
    *reinterpret_cast<uint32_t *>(L.WbT + (size_t)(c0 + c) * L.R + r0 + pr) =
        *reinterpret_cast<const uint32_t *>(&tile[c][pr]);
  }
}

__global__ void __launch_bounds__(TT * TY) k_cast_w(const float *__restrict__ W, int R, int C, __nv_bfloat16 *Wb,
                         __nv_bfloat16 *WbT) {
  tile_bf16_pair<TY>(R, C, Wb, WbT, [&](int r, int c) { return W[(size_t)r * C + c]; });
}

// column mean and standard deviation of X [R][C] (float64 sums, rows in order)
__global__ void k_col_stats(const float *__restrict__ X, int R, int C, float *__restrict__ mean,
                            float *__restrict__ stdv) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= C) return;
  double s = 0.0, s2 = 0.0;
  for (int r = 0; r < R; ++r) {
    const double v = X[(size_t)r * C + c];
    s += v;
    s2 += v * v;
  }
  const double m = s / R;
  const double var = s2 / R - m * m;
  mean[c] = (float)m;
  stdv[c] = (float)sqrt(var > 0.0 ? var : 0.0);
}

// out[r][c] = (X[r][c] - shift[c]) * mul[c]
__global__ void k_affine_cols(const float *__restrict__ X, size_t n, int C,
                              const float *__restrict__ shift, const float *__restrict__ mul,
                              float *__restrict__ out) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n;
       e += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % C);
    out[e] = (X[e] - shift[c]) * mul[c];
  }
}

}  // namespace specula

using namespace specula;

extern "C" int specula_col_stats(specula_ctx *ctx, const float *X_dev, int32_t rows,
                                 int32_t cols, float *mean_dev, float *std_dev, void *stream) {
  if (!ctx || !X_dev || !mean_dev || !std_dev || rows < 1 || cols < 1) return SPECULA_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  SPECULA_LAUNCH(ctx, SPECULA_K_MLP, st,
                 k_col_stats<<<(cols + 127) / 128, 128, 0, st>>>(X_dev, rows, cols, mean_dev,
                                                                 std_dev));
  return SPECULA_OK;
}

extern "C" int specula_affine_cols(specula_ctx *ctx, const float *X_dev, int64_t rows,
                                   int32_t cols, const float *shift_dev, const float *mul_dev,
                                   float *out_dev, void *stream) {
  if (!ctx || !X_dev || !shift_dev || !mul_dev || !out_dev || rows < 1 || cols < 1)
    return SPECULA_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t n = (size_t)rows * cols;
  SPECULA_LAUNCH(ctx, SPECULA_K_MLP, st,
                 k_affine_cols<<<(unsigned)std::min<size_t>((n + 255) / 256, 8192), 256, 0, st>>>(
                     X_dev, n, cols, shift_dev, mul_dev, out_dev));
  return SPECULA_OK;
}

struct specula_mlp {
  specula_ctx *ctx = nullptr;
  int device = 0;  // copied from ctx so destroy never dereferences it
  int n[4];        // true widths: n_in, h1, h2, n_out
  int np[4];       // padded widths
  int bmax;        // padded batch capacity
  int t = 0;       // Adam steps taken
  int last_b = 0;  // batch of the last forward
  DevBuf W[3], b[3], mW[3], vW[3], mb[3], vb[3], Wb[3], WbT[3], gW[3], gb[3];
  DevBuf Xb, XbT, Z[2], H[2], HT[2], Y, dYf, dYb, dYbT, dA[2], dZb[2], dZbT[2];
  DevBuf work, part, loss;
  DevBuf done;     // finished-block count of the loss kernel
  DevBuf Hi[2];    // inference activations, [kInferMax][np] float32
  size_t work_floats = 0;
};

static inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

// ---- inference for a few vectors (specula_mlp_infer) ---------------------------
// A batch of a few slope vectors leaves the tensor-core GEMMs (128-row tiles)
// mostly padding, and the time goes to reading the bf16 weights.  Each layer
// instead streams them once against every input vector in float32, then adds
// the bias and applies GELU; activations stay float32.  A CTA of four warps
// takes two output rows, each warp a quarter of K: eight 16-byte weight loads
// in flight per lane and every activation load used for both rows.  (One warp
// per row with scalar activation loads took 51 us for 13344-2048-2048-4000,
// 1.5 TB/s: four times the load instructions and half the bytes in flight;
// now 19.7 us.)  A hidden layer's CTAs start under the layer before and send their
// weight rows to L2 first.  The first layer's start when the kernel before the
// network has left.  (Under the last layer of the call before: 18.6 us, but then every
// kernel that reads the network's output starts while it is being written.)
constexpr int kInferMax = 4;
constexpr int kGemvWarps = 4, kGemvRows = 2;

__device__ __forceinline__ uint4 ld_stream_w(const uint4 *p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
// Activations: plain loads.  A layer's CTAs are resident while the layer before
// still writes them, and the non-coherent path (ld.global.nc, what __ldg and const
// __restrict__ give) is only defined for memory that is not written during the
// kernel's life.
__device__ __forceinline__ float4 ld_act4(const float *p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ float ld_act(const float *p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// out[b][o] = act(sum_k W[o][k] x[b][k] + bias[o]), o < n_out, b < nb;
// W bf16 [.][ldw]; x float [nb][ldx] with k < K read, by 16-byte loads when
// VX (ldx % 4 == 0 and x aligned); grid ceil(n_out / 2), block 128.
template <int NB, bool GELU, bool VX>
__global__ void __launch_bounds__(kGemvWarps * 32) k_mlp_gemv(
    const __nv_bfloat16 *__restrict__ W, int ldw, const float *x, int ldx, int K, int n_out, int nb,
    const float *__restrict__ bias, float *out, int ldo) {
  // the last layer (no GELU) does not: a kernel behind the network starts once its
  // CTAs have left, as behind any other kernel
  if constexpr (GELU) pdl_trigger();
  __shared__ float s_w[kGemvWarps][kGemvRows * NB];
  const int o0 = blockIdx.x * kGemvRows;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the weights do not depend on the layer before: on their way to L2 while it runs
  if (warp < kGemvRows && lane == 0 && o0 + warp < n_out && K >= 8)
    prefetch_l2(W + (size_t)(o0 + warp) * ldw, (uint32_t)(K / 8 * 16));
  pdl_wait();
  const uint4 *w8[kGemvRows];
#pragma unroll
  for (int i = 0; i < kGemvRows; ++i)
    w8[i] = reinterpret_cast<const uint4 *>(W + (size_t)min(o0 + i, n_out - 1) * ldw);
  const int k8 = K / 8;
  const int seg = (k8 + kGemvWarps - 1) / kGemvWarps;
  const int lo = warp * seg, hi = min(k8, lo + seg);
  float acc[kGemvRows][NB];
#pragma unroll
  for (int i = 0; i < kGemvRows; ++i)
#pragma unroll
    for (int q = 0; q < NB; ++q) acc[i][q] = 0.f;
  constexpr int UL = 4;
  for (int j0 = lo + lane; j0 < hi; j0 += UL * 32) {
    uint4 wv[UL][kGemvRows];
#pragma unroll
    for (int u = 0; u < UL; ++u)
#pragma unroll
      for (int i = 0; i < kGemvRows; ++i)
        wv[u][i] = j0 + 32 * u < hi ? ld_stream_w(w8[i] + j0 + 32 * u) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < UL; ++u) {
      const int j = j0 + 32 * u;
      if (j < hi) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
          if (q < nb) {
            const float *xp = x + (size_t)q * ldx + 8 * j;
            float xv[8];
            if constexpr (VX) {
              const float4 a = ld_act4(xp), c = ld_act4(xp + 4);
              xv[0] = a.x; xv[1] = a.y; xv[2] = a.z; xv[3] = a.w;
              xv[4] = c.x; xv[5] = c.y; xv[6] = c.z; xv[7] = c.w;
            } else {
#pragma unroll
              for (int e = 0; e < 8; ++e) xv[e] = ld_act(xp + e);
            }
#pragma unroll
            for (int i = 0; i < kGemvRows; ++i) {
              const uint4 w = wv[u][i];
              acc[i][q] += bf16_lo(w.x) * xv[0] + bf16_hi(w.x) * xv[1] + bf16_lo(w.y) * xv[2] +
                           bf16_hi(w.y) * xv[3] + bf16_lo(w.z) * xv[4] + bf16_hi(w.z) * xv[5] +
                           bf16_lo(w.w) * xv[6] + bf16_hi(w.w) * xv[7];
            }
          }
        }
      }
    }
  }
  // the K % 8 tail, by the last warp
  const int kt = 8 * k8 + lane;
  if (warp == kGemvWarps - 1 && kt < K) {
#pragma unroll
    for (int i = 0; i < kGemvRows; ++i) {
      const float wk = __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(w8[i])[kt]);
#pragma unroll
      for (int q = 0; q < NB; ++q)
        if (q < nb) acc[i][q] += wk * ld_act(x + (size_t)q * ldx + kt);
    }
  }
#pragma unroll
  for (int i = 0; i < kGemvRows; ++i)
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      float v = acc[i][q];
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
      if (lane == 0) s_w[warp][q * kGemvRows + i] = v;
    }
  __syncthreads();
  const int i = threadIdx.x % kGemvRows, q = threadIdx.x / kGemvRows;
  if (q < nb && q < NB && o0 + i < n_out) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kGemvWarps; ++w) v += s_w[w][threadIdx.x];
    v += bias[o0 + i];
    out[(size_t)q * ldo + o0 + i] = GELU ? gelu_f(v) : v;
  }
}

static int mlp_splits(int M, int N, int K) {
  const int tiles = (M / 128) * (N / 128);
  int want = std::max(1, (2 * 152 + tiles / 2) / std::max(tiles, 1));
  return gemm_splits(K, want);
}

// C = A B^T left as split-K partials in the workspace, for the kernel that
// follows on the stream to add
static int mlp_gemm(specula_mlp *p, const void *A, const void *B, int M, int N, int K,
                    Partials *out, cudaStream_t st) {
  const int s = mlp_splits(M, N, K);
  if ((size_t)s * M * N > p->work_floats) return SPECULA_EINVAL;
  *out = Partials{p->work.as<float>(), s, (size_t)M * N};
  return gemm_bf16_partials(p->ctx, A, B, M, N, K, s, p->work.as<float>(), st);
}

// Padded batch up to which the weight gradients run in one launch
constexpr int kDwGroupK = 4096;

// Weight gradients dW_l = dZ_l^T H_{l-1}, l = 0 .. 2 (M = np[l + 1], N = np[l]), over
// the padded batch.  The products are short (four K blocks at a batch of 256) and
// bound by what they write: one launch over all the layers' 128 x 128 tiles, a
// tile's K slices added in registers, so the sums are those of the split-K
// products to the last bit.  Beyond kDwGroupK each layer's own launch, its K split
// over the SMs, and their sum: gW holds the gradient whatever the batch, so a replayed
// graph's Adam or get_grad needs no state of the host's.  Own launches (their sums
// left to Adam then) / one launch, a step of 2512-1024-1024-500:
// 123 / 95 us at 256 rows, 294 / 263 at 2048; of 300-128-128-60, four tiles in all:
// 98 / 74 at 1024, 225 / 169 at 4096 (the bias gradients in it, as below).
static int mlp_gemm_dw(specula_mlp *p, const void *const *A, const void *const *B, int batch,
                       int Bp, cudaStream_t st) {
  const bool group = Bp <= kDwGroupK;
  int M[3], N[3], splits[3], s;
  float *out[3];
  for (int l = 0; l < 3; ++l) {
    M[l] = p->np[l + 1];
    N[l] = p->np[l];
    out[l] = p->gW[l].as<float>();
    splits[l] = mlp_splits(M[l], N[l], Bp);
    if (!group && (size_t)splits[l] * M[l] * N[l] > p->work_floats) return SPECULA_EINVAL;
  }
  // the bias gradients in the same launch, by warps that the products leave idle: a
  // block that summed its tile column last made each producer of dZ 4 us longer
  // (a step of 2512-1024-1024-500 at 256 rows 95 -> 82 us)
  ColSums cs;
  cs.n = 3;
  cs.rows = batch;
  const DevBuf *D[3] = {&p->dA[0], &p->dA[1], &p->dYf};
  for (int l = 0; l < 3; ++l) {
    cs.cols[l] = M[l];
    cs.D[l] = D[l]->as<float>();
    cs.sum[l] = p->gb[l].as<float>();
  }
  if (group) return gemm_bf16_group(p->ctx, 3, A, B, M, N, Bp, splits, out, cs, st);
  SPECULA_LAUNCH_PDL(p->ctx, SPECULA_K_MLP, st, k_bias_grad, (M[0] + M[1] + M[2]) / 128, 128, 0,
                     cs);
  for (int l = 2; l >= 0; --l)
    if ((s = gemm_bf16_tn(p->ctx, A[l], B[l], M[l], N[l], Bp, out[l], splits[l],
                          p->work.as<float>(), st)))
      return s;
  return SPECULA_OK;
}

static int cast_layer(specula_mlp *p, int l, cudaStream_t st) {
  const int R = p->np[l + 1], C = p->np[l];
  dim3 g((C + TT - 1) / TT, (R + TT - 1) / TT);
  SPECULA_LAUNCH(p->ctx, SPECULA_K_MLP, st,
                 k_cast_w<<<g, dim3(TT, TY), 0, st>>>(p->W[l].as<float>(), R, C,
                                                    p->Wb[l].as<__nv_bfloat16>(),
                                                    p->WbT[l].as<__nv_bfloat16>()));
  return SPECULA_OK;
}

extern "C" int specula_mlp_create(specula_ctx *ctx, int32_t n_in, int32_t n_h1, int32_t n_h2,
                                  int32_t n_out, int32_t batch_max, specula_mlp **out) {
  if (!ctx || !out || n_in < 1 || n_out < 1 || batch_max < 1) return SPECULA_EINVAL;
  if (n_h1 < 128 || n_h2 < 128 || n_h1 % 128 || n_h2 % 128) return SPECULA_EUNSUPPORTED;
  if (n_in > 65536 || n_out > 65536 || batch_max > 65536) return SPECULA_EUNSUPPORTED;
  *out = nullptr;
  SPECULA_CK(cudaSetDevice(ctx->device));
  std::unique_ptr<specula_mlp> p(new specula_mlp());
  p->ctx = ctx;
  p->device = ctx->device;
  p->n[0] = n_in; p->n[1] = n_h1; p->n[2] = n_h2; p->n[3] = n_out;
  p->np[0] = round_up(n_in, 128); p->np[1] = n_h1; p->np[2] = n_h2; p->np[3] = round_up(n_out, 128);
  p->bmax = round_up(batch_max, 128);
  const int Bp = p->bmax;
  int s;
  for (int l = 0; l < 3; ++l) {
    const size_t nw = (size_t)p->np[l + 1] * p->np[l], nb = p->np[l + 1];
    if ((s = p->W[l].alloc(nw * 4)) || (s = p->mW[l].alloc(nw * 4)) || (s = p->vW[l].alloc(nw * 4)) ||
        (s = p->gW[l].alloc(nw * 4)) || (s = p->Wb[l].alloc(nw * 2)) || (l > 0 && (s = p->WbT[l].alloc(nw * 2))) ||
        (s = p->b[l].alloc(nb * 4)) || (s = p->mb[l].alloc(nb * 4)) || (s = p->vb[l].alloc(nb * 4)) ||
        (s = p->gb[l].alloc(nb * 4)))
      return s;
    SPECULA_CK(cudaMemset(p->W[l].p, 0, nw * 4));
    SPECULA_CK(cudaMemset(p->mW[l].p, 0, nw * 4));
    SPECULA_CK(cudaMemset(p->vW[l].p, 0, nw * 4));
    SPECULA_CK(cudaMemset(p->gW[l].p, 0, nw * 4));
    SPECULA_CK(cudaMemset(p->b[l].p, 0, nb * 4));
    SPECULA_CK(cudaMemset(p->mb[l].p, 0, nb * 4));
    SPECULA_CK(cudaMemset(p->vb[l].p, 0, nb * 4));
    SPECULA_CK(cudaMemset(p->gb[l].p, 0, nb * 4));
  }
  const int in = p->np[0], h1 = p->np[1], h2 = p->np[2], o = p->np[3];
  if ((s = p->Xb.alloc((size_t)Bp * in * 2)) || (s = p->XbT.alloc((size_t)Bp * in * 2)) ||
      (s = p->Z[0].alloc((size_t)Bp * h1 * 4)) || (s = p->Z[1].alloc((size_t)Bp * h2 * 4)) ||
      (s = p->H[0].alloc((size_t)Bp * h1 * 2)) || (s = p->H[1].alloc((size_t)Bp * h2 * 2)) ||
      (s = p->HT[0].alloc((size_t)Bp * h1 * 2)) || (s = p->HT[1].alloc((size_t)Bp * h2 * 2)) ||
      (s = p->Y.alloc((size_t)Bp * o * 4)) || (s = p->dYf.alloc((size_t)Bp * o * 4)) ||
      (s = p->dA[0].alloc((size_t)Bp * h1 * 4)) || (s = p->dA[1].alloc((size_t)Bp * h2 * 4)) ||
      (s = p->dYb.alloc((size_t)Bp * o * 2)) || (s = p->dYbT.alloc((size_t)Bp * o * 2)) ||
      (s = p->dZb[0].alloc((size_t)Bp * h1 * 2)) || (s = p->dZb[1].alloc((size_t)Bp * h2 * 2)) ||
      (s = p->dZbT[0].alloc((size_t)Bp * h1 * 2)) || (s = p->dZbT[1].alloc((size_t)Bp * h2 * 2)))
    return s;
  // split-K workspace: the largest of a step's GEMMs that use it, for every padded
  // batch up to the capacity
  size_t wf = 1;
  for (int b = 128; b <= Bp; b += 128) {
    const int shapes[8][3] = {{b, h1, in}, {b, h2, h1}, {b, o, h2},  {b, h2, o},
                              {b, h1, h2}, {h1, in, b}, {h2, h1, b}, {o, h2, b}};
    // (the last three, the weight gradients, only beyond kDwGroupK)
    for (int i = 0; i < (b > kDwGroupK ? 8 : 5); ++i) {
      const auto &sh = shapes[i];
      wf = std::max(wf, (size_t)mlp_splits(sh[0], sh[1], sh[2]) * sh[0] * sh[1]);
    }
  }
  p->work_floats = wf;
  if ((s = p->work.alloc(wf * 4))) return s;
  if ((s = p->Hi[0].alloc((size_t)kInferMax * h1 * 4)) ||
      (s = p->Hi[1].alloc((size_t)kInferMax * h2 * 4)))
    return s;
  const int tiles = ((o + TT - 1) / TT) * ((Bp + TT - 1) / TT);
  if ((s = p->part.alloc((size_t)tiles * 4)) || (s = p->loss.alloc(4)) ||
      (s = p->done.alloc(4)))
    return s;
  SPECULA_CK(cudaMemset(p->done.p, 0, p->done.bytes));
  for (int l = 0; l < 3; ++l)
    if ((s = cast_layer(p.get(), l, 0))) return s;
  SPECULA_CK(cudaDeviceSynchronize());
  *out = p.release();
  return SPECULA_OK;
}

extern "C" int specula_mlp_destroy(specula_mlp *mlp) {
  if (!mlp) return SPECULA_EINVAL;
  cudaSetDevice(mlp->device);
  cudaDeviceSynchronize();
  delete mlp;
  return SPECULA_OK;
}

extern "C" int specula_mlp_set_layer(specula_mlp *p, int32_t layer, const float *W_host,
                                     const float *b_host) {
  if (!p || layer < 0 || layer > 2 || !W_host || !b_host) return SPECULA_EINVAL;
  SPECULA_CK(cudaSetDevice(p->ctx->device));
  const int R = p->n[layer + 1], C = p->n[layer], RP = p->np[layer + 1], CP = p->np[layer];
  std::vector<float> w((size_t)RP * CP, 0.f), b(RP, 0.f);
  for (int r = 0; r < R; ++r)
    for (int c = 0; c < C; ++c) w[(size_t)r * CP + c] = W_host[(size_t)r * C + c];
  for (int r = 0; r < R; ++r) b[r] = b_host[r];
  SPECULA_CK(cudaMemcpy(p->W[layer].p, w.data(), w.size() * 4, cudaMemcpyHostToDevice));
  SPECULA_CK(cudaMemcpy(p->b[layer].p, b.data(), b.size() * 4, cudaMemcpyHostToDevice));
  for (DevBuf *z : {&p->mW[layer], &p->vW[layer]}) SPECULA_CK(cudaMemset(z->p, 0, z->bytes));
  for (DevBuf *z : {&p->mb[layer], &p->vb[layer]}) SPECULA_CK(cudaMemset(z->p, 0, z->bytes));
  p->t = 0;
  int s = cast_layer(p, layer, 0);
  if (s) return s;
  SPECULA_CK(cudaDeviceSynchronize());
  return SPECULA_OK;
}

static int copy_out(specula_mlp *p, int layer, const DevBuf &W, const DevBuf &b, float *W_host,
                    float *b_host) {
  SPECULA_CK(cudaSetDevice(p->ctx->device));
  SPECULA_CK(cudaDeviceSynchronize());
  const int R = p->n[layer + 1], C = p->n[layer], CP = p->np[layer];
  SPECULA_CK(cudaMemcpy2D(W_host, (size_t)C * 4, W.p, (size_t)CP * 4, (size_t)C * 4, R,
                          cudaMemcpyDeviceToHost));
  SPECULA_CK(cudaMemcpy(b_host, b.p, (size_t)R * 4, cudaMemcpyDeviceToHost));
  return SPECULA_OK;
}

extern "C" int specula_mlp_get_layer(specula_mlp *p, int32_t layer, float *W_host,
                                     float *b_host) {
  if (!p || layer < 0 || layer > 2 || !W_host || !b_host) return SPECULA_EINVAL;
  return copy_out(p, layer, p->W[layer], p->b[layer], W_host, b_host);
}

extern "C" int specula_mlp_get_grad(specula_mlp *p, int32_t layer, float *dW_host,
                                    float *db_host) {
  if (!p || layer < 0 || layer > 2 || !dW_host || !db_host) return SPECULA_EINVAL;
  return copy_out(p, layer, p->gW[layer], p->gb[layer], dW_host, db_host);
}

extern "C" int specula_mlp_forward(specula_mlp *p, const float *X_dev, int32_t batch,
                                   float *Y_dev, void *stream) {
  if (!p || !X_dev || batch < 1) return SPECULA_EINVAL;
  const int Bp = round_up(batch, 128);
  if (Bp > p->bmax) return SPECULA_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  specula_ctx *ctx = p->ctx;
  const int in = p->np[0], h1 = p->np[1], h2 = p->np[2], o = p->np[3];
  int sms = 0, s;
  SPECULA_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  int ry = tile_rows(Bp, in, sms);
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_MLP, st, (ry == TY ? k_pack_input<TY> : k_pack_input<TYL>),
                     dim3(in / TT, Bp / TT), dim3(TT, ry), 0, X_dev, batch, p->n[0], Bp, in,
                     p->Xb.as<__nv_bfloat16>(), p->XbT.as<__nv_bfloat16>());
  const void *Hin = p->Xb.p;
  Partials P;
  for (int l = 0; l < 2; ++l) {
    const int K = p->np[l], N = p->np[l + 1];
    if ((s = mlp_gemm(p, Hin, p->Wb[l].p, Bp, N, K, &P, st))) return s;
    ry = tile_rows(Bp, N, sms);
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_MLP, st, (ry == TY ? k_bias_gelu<TY> : k_bias_gelu<TYL>),
                       dim3(N / TT, Bp / TT), dim3(TT, ry), 0, P, p->b[l].as<float>(),
                       p->Z[l].as<float>(), Bp, N,
                       p->H[l].as<__nv_bfloat16>(), p->HT[l].as<__nv_bfloat16>());
    Hin = p->H[l].p;
  }
  if ((s = mlp_gemm(p, Hin, p->Wb[2].p, Bp, o, h2, &P, st))) return s;
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_MLP, st, k_output, (unsigned)((P.n + 255) / 256), 256, 0, P,
                     p->b[2].as<float>(), o, p->Y.as<float>(), batch, p->n[3], Y_dev);
  p->last_b = batch;
  (void)h1;
  return SPECULA_OK;
}

extern "C" int specula_mlp_infer(specula_mlp *p, const float *X_dev, int32_t batch,
                                 float *Y_dev, void *stream) {
  if (!p || !X_dev || !Y_dev || batch < 1) return SPECULA_EINVAL;
  if (batch > kInferMax) return specula_mlp_forward(p, X_dev, batch, Y_dev, stream);
  cudaStream_t st = (cudaStream_t)stream;
  specula_ctx *ctx = p->ctx;
  const __nv_bfloat16 *W0 = p->Wb[0].as<__nv_bfloat16>(), *W1 = p->Wb[1].as<__nv_bfloat16>(),
                      *W2 = p->Wb[2].as<__nv_bfloat16>();
  float *H0 = p->Hi[0].as<float>(), *H1 = p->Hi[1].as<float>();
  const int h1 = p->n[1], h2 = p->n[2];
  const bool vx = p->n[0] % 4 == 0 && (uintptr_t)X_dev % 16 == 0;
  auto grid = [](int n) { return (unsigned)((n + kGemvRows - 1) / kGemvRows); };
#define SPECULA_GEMV1(NB, VX)                                                                \
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_MLP, st, (k_mlp_gemv<NB, true, VX>), grid(h1),                \
                     kGemvWarps * 32, 0, W0, p->np[0], X_dev, p->n[0], p->n[0], h1, batch,        \
                     p->b[0].as<float>(), H0, h1)
#define SPECULA_GEMV(NB)                                                                     \
  do {                                                                                       \
    if (vx)                                                                                  \
      SPECULA_GEMV1(NB, true);                                                               \
    else                                                                                     \
      SPECULA_GEMV1(NB, false);                                                              \
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_MLP, st, (k_mlp_gemv<NB, true, true>), grid(h2),            \
                       kGemvWarps * 32, 0, W1, p->np[1], H0, h1, h1, h2, batch,                   \
                       p->b[1].as<float>(), H1, h2); \
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_MLP, st, (k_mlp_gemv<NB, false, true>), grid(p->n[3]),      \
                       kGemvWarps * 32, 0, W2, p->np[2], H1, h2, h2, p->n[3], batch,              \
                       p->b[2].as<float>(), Y_dev, p->n[3]); \
  } while (0)
  if (batch == 1)
    SPECULA_GEMV(1);
  else
    SPECULA_GEMV(kInferMax);
#undef SPECULA_GEMV1
#undef SPECULA_GEMV
  return SPECULA_OK;
}

extern "C" int specula_mlp_backward(specula_mlp *p, const float *T_dev, int32_t batch,
                                    float *loss_dev, void *stream) {
  if (!p || !T_dev || batch < 1 || batch != p->last_b) return SPECULA_EINVAL;
  const int Bp = round_up(batch, 128);
  cudaStream_t st = (cudaStream_t)stream;
  specula_ctx *ctx = p->ctx;
  const int h1 = p->np[1], h2 = p->np[2], o = p->np[3];
  const float scale = 2.0f / ((float)batch * (float)p->n[3]);
  const dim3 gl(o / TT, Bp / TT);
  int sms = 0, s;
  SPECULA_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_MLP, st, k_loss_grad, gl, dim3(TT, TY), 0, p->Y.as<float>(), T_dev,
                     batch, p->n[3], Bp, o, scale, p->dYf.as<float>(), p->dYb.as<__nv_bfloat16>(),
                     p->dYbT.as<__nv_bfloat16>(), p->done.as<unsigned>(), p->part.as<float>(),
                     1.0f / ((float)batch * (float)p->n[3]),
                     loss_dev ? loss_dev : p->loss.as<float>());
  Partials P;
  if ((s = mlp_gemm(p, p->dYb.p, p->WbT[2].p, Bp, h2, o, &P, st))) return s;
  for (int l = 1; l >= 0; --l) {
    const int N = p->np[l + 1];
    const int ry = tile_rows(Bp, N, sms);
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_MLP, st, (ry == TY ? k_gelu_back<TY> : k_gelu_back<TYL>),
                       dim3(N / TT, Bp / TT), dim3(TT, ry), 0, P,
                       p->Z[l].as<float>(), p->dA[l].as<float>(), Bp, N,
                       p->dZb[l].as<__nv_bfloat16>(), p->dZbT[l].as<__nv_bfloat16>());
    if (l == 1)
      if ((s = mlp_gemm(p, p->dZb[1].p, p->WbT[1].p, Bp, h1, h2, &P, st))) return s;
  }
  const void *dT[3] = {p->dZbT[0].p, p->dZbT[1].p, p->dYbT.p};
  const void *HinT[3] = {p->XbT.p, p->HT[0].p, p->HT[1].p};
  return mlp_gemm_dw(p, dT, HinT, batch, Bp, st);
}

extern "C" int specula_mlp_adam(specula_mlp *p, float lr, float b1, float b2, float eps,
                                void *stream) {
  if (!p || !(lr > 0) || !(b1 >= 0 && b1 < 1) || !(b2 >= 0 && b2 < 1) || !(eps > 0))
    return SPECULA_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  p->t += 1;
  const double lr_t = lr * sqrt(1.0 - pow((double)b2, p->t)) / (1.0 - pow((double)b1, p->t));
  AdamArgs A;
  A.first[0] = A.bias_first[0] = 0;
  for (int l = 0; l < 3; ++l) {
    const int R = p->np[l + 1], C = p->np[l];
    A.L[l] = AdamLayer{p->W[l].as<float>(),  p->mW[l].as<float>(), p->vW[l].as<float>(),
                       p->b[l].as<float>(),  p->mb[l].as<float>(), p->vb[l].as<float>(),
                       p->gW[l].as<float>(), p->gb[l].as<float>(),
                       p->Wb[l].as<__nv_bfloat16>(), p->WbT[l].as<__nv_bfloat16>(), R, C};
    A.first[l + 1] = A.first[l] + (R / TT) * (C / kAdamC);
    A.bias_first[l + 1] = A.bias_first[l] + (R + TT * 8 - 1) / (TT * 8);
  }
  SPECULA_LAUNCH_PDL(p->ctx, SPECULA_K_MLP, st, k_adam, A.first[3] + A.bias_first[3], dim3(TT, 8),
                     0, A, (float)lr_t, b1, b2, eps);
  return SPECULA_OK;
}

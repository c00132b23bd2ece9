// Closed adaptive-optics loop pieces (the SOUL example's DM, IirFilter
// integrator and delayed connection, App. B, Listing 2; Sect. 2.2 for the
// ":-1" delayed input): the modal mirror's shape, the residual phase with its
// statistics, and the integrator update.  Per step k of a loop:
//   residual = phi_atm(t_k) - B^T c_{k-1},   m = R (slopes(residual) - ref),
//   c_k = (1 - leak) c_{k-1} + gain m.
// Every sum runs in a fixed order (no float atomics), so a loop is
// bit-reproducible.
#include <cooperative_groups.h>

#include "internal.h"

namespace cg = cooperative_groups;

namespace specula {

constexpr int kDmWarps = 8;
constexpr int kDmUnroll = 8;
constexpr int kDmMaxCluster = 8;
constexpr int kLoopThreads = 256;

__device__ __forceinline__ void dm_axpy(float4 &a, float c, float4 v) {
  a.x += c * v.x;
  a.y += c * v.y;
  a.z += c * v.z;
  a.w += c * v.w;
}

// Four pixels per lane of a tile of 4 LT: neighbours by one 16-byte access (VEC) or LT
// apart by four of 4 bytes.
template <bool VEC, int LT> struct DmPixels {
  int i[4];
  __device__ DmPixels(int tile, int ln, int n) {
#pragma unroll
    for (int k = 0; k < 4; ++k) i[k] = tile * 4 * LT + (VEC ? 4 * ln : ln + LT * k);
  }
  // (pixels past the grid repeat the last, or the last four)
  __device__ __forceinline__ float4 load(const float *row, int n) const {
    if constexpr (VEC)
      return __ldg(reinterpret_cast<const float4 *>(row + min(i[0], n - 4)));
    else
      return make_float4(__ldg(row + min(i[0], n - 1)), __ldg(row + min(i[1], n - 1)),
                         __ldg(row + min(i[2], n - 1)), __ldg(row + min(i[3], n - 1)));
  }
  __device__ __forceinline__ void store(float *phase, int n, float4 v) const {
    if constexpr (VEC) {
      if (i[0] < n) *reinterpret_cast<float4 *>(phase + i[0]) = v;
    } else {
      if (i[0] < n) phase[i[0]] = v.x;
      if (i[1] < n) phase[i[1]] = v.y;
      if (i[2] < n) phase[i[2]] = v.z;
      if (i[3] < n) phase[i[3]] = v.w;
    }
  }
};

// phase[p] = sum over j of cmd[j] B[j][p].  Bound by reading B once: one
// thread per pixel over all modes kept 5 KB in flight per SM (500 modes of
// 160^2 pixels: 33 us for 51 MB).  A CTA of eight warps takes 4 LT pixels, the modes
// split over the warps, over 32 / LT parts of a warp and, on small pupils, over a
// cluster of CTAs; eight rows' loads in flight per lane.  Each part adds its
// modes in order, then the parts' and the CTAs' sums are added in order.
template <bool VEC, int LT>
__global__ void __launch_bounds__(kDmWarps * 32, 4) k_dm_shape(const float *__restrict__ B,
                                                            const float *__restrict__ cmd,
                                                            float *__restrict__ phase,
                                                            int n_modes, int n_pix2) {
  __shared__ float4 s_p[kDmWarps][32];
  pdl_wait();
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int SUB = 32 / LT, NP = kDmWarps * SUB;   // parts of the modes per CTA
  const int ln = lane % LT;
  const DmPixels<VEC, LT> px(blockIdx.x / cs, ln, n_pix2);
  const int part = rank * NP + warp * SUB + lane / LT, parts = cs * NP;
  int j = (int)((long long)n_modes * part / parts);
  const int j1 = (int)((long long)n_modes * (part + 1) / parts);
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (; j + kDmUnroll <= j1; j += kDmUnroll) {
    float4 v[kDmUnroll];
#pragma unroll
    for (int u = 0; u < kDmUnroll; ++u) v[u] = px.load(B + (size_t)(j + u) * n_pix2, n_pix2);
#pragma unroll
    for (int u = 0; u < kDmUnroll; ++u) dm_axpy(acc, __ldg(cmd + j + u), v[u]);
  }
  if (j < j1) {   // the rest's loads in flight together too
    float4 v[kDmUnroll];
#pragma unroll
    for (int u = 0; u < kDmUnroll; ++u)
      if (j + u < j1) v[u] = px.load(B + (size_t)(j + u) * n_pix2, n_pix2);
#pragma unroll
    for (int u = 0; u < kDmUnroll; ++u)
      if (j + u < j1) dm_axpy(acc, __ldg(cmd + j + u), v[u]);
  }
  s_p[warp][lane] = acc;
  __syncthreads();
  if (warp == 0) {
    acc = s_p[0][ln];
#pragma unroll
    for (int i = 1; i < NP; ++i) dm_axpy(acc, 1.f, s_p[i / SUB][i % SUB * LT + ln]);
    if (lane < LT) s_p[0][lane] = acc;
  }
  if (cs > 1) {
    cl.sync();
    if (rank == 0 && warp == 0) {
      for (int c = 1; c < cs; ++c) dm_axpy(acc, 1.f, cl.map_shared_rank(&s_p[0][0], c)[ln]);
    }
    cl.sync();   // no CTA leaves before its sums are read
  }
  if (rank == 0 && warp == 0 && lane < LT) px.store(phase, n_pix2, acc);
}

// The same for few modes: a warp takes 128 pixels and every mode, eight modes' loads in
// flight, and adds the sums of the same eight parts in the same order, so the result
// is k_dm_shape's to the last bit; up to eight modes one chain, as parts of one
// product round twice.
template <bool VEC>
__global__ void __launch_bounds__(kDmWarps * 32) k_dm_few(const float *__restrict__ B,
                                                          const float *__restrict__ cmd,
                                                          float *__restrict__ phase, int n_modes,
                                                          int n_pix2) {
  pdl_wait();
  const DmPixels<VEC, 32> px(blockIdx.x * kDmWarps + (threadIdx.x >> 5), threadIdx.x & 31, n_pix2);
  const int parts = n_modes <= kDmUnroll ? 1 : kDmWarps;
  float4 sum = make_float4(0.f, 0.f, 0.f, 0.f), acc = sum;
  int part = 1, next = n_modes / parts;   // modes below `next` are in the part so far
  for (int j = 0; j < n_modes; j += kDmUnroll) {
    float4 v[kDmUnroll];
#pragma unroll
    for (int u = 0; u < kDmUnroll; ++u)
      if (j + u < n_modes) v[u] = px.load(B + (size_t)(j + u) * n_pix2, n_pix2);
#pragma unroll
    for (int u = 0; u < kDmUnroll; ++u)
      if (j + u < n_modes) {
        if (j + u == next) {
          dm_axpy(sum, 1.f, acc);
          acc = make_float4(0.f, 0.f, 0.f, 0.f);
          ++part;
          next = n_modes * part / parts;
        }
        dm_axpy(acc, __ldg(cmd + j + u), v[u]);
      }
  }
  dm_axpy(sum, 1.f, acc);
  px.store(phase, n_pix2, sum);
}

// residual = atm - dm over the grid, and its statistics: float64 sums over
// the pupil (weights amp) of w, w r, w r^2, w cos(k r), w sin(k r), k =
// lambda_wfs / lambda_sci, per CTA in a fixed order; the CTA that finishes
// last adds the CTAs' sums in a fixed order and writes
//   stats[0] = sqrt(sum w r^2 / sum w - mean^2),
//   stats[1] = |sum w e^{ikr}|^2 / (sum w)^2.
// Up to kLoopMaxBlocks CTAs, one pixel per thread on the 8 m pupil: float64
// runs at 2 operations per clock and SM, so 13 CTAs of 8 pixels per thread
// took 13 us, and the statistics in a kernel of one thread 6.5 us.
__device__ __forceinline__ void loop_block_sum(double (&a)[5], double (*s_p)[kLoopThreads / 32]) {
  // five butterflies at once: each level halves the values a lane carries, nine
  // additions instead of 25 with the same pairs (value 4 and zeros in the upper half)
  const int lane = threadIdx.x & 31;
  const bool u = lane & 16, h = lane & 8, t = lane & 4;
  double b[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double hi = i == 0 ? a[4] : 0.0;
    b[i] = (u ? hi : a[i]) + __shfl_xor_sync(0xffffffffu, u ? a[i] : hi, 16);
  }
  double c[2], d;
#pragma unroll
  for (int i = 0; i < 2; ++i)
    c[i] = (h ? b[2 + i] : b[i]) + __shfl_xor_sync(0xffffffffu, h ? b[i] : b[2 + i], 8);
  d = (t ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, t ? c[0] : c[1], 4);
  d += __shfl_xor_sync(0xffffffffu, d, 2);
  d += __shfl_xor_sync(0xffffffffu, d, 1);
  const int q = (u ? 4 : 0) + (h ? 2 : 0) + (t ? 1 : 0);
  if (lane % 4 == 0 && q < 5) s_p[q][threadIdx.x >> 5] = d;
  __syncthreads();
}

__global__ void __launch_bounds__(kLoopThreads) k_loop_residual(
    const float *__restrict__ amp, const float *__restrict__ atm, const float *__restrict__ dm,
    float *__restrict__ resid, double *__restrict__ part, unsigned *__restrict__ done,
    double *__restrict__ stats, int n_pix2, float k) {
  pdl_wait();
  __shared__ double s_p[5][kLoopThreads / 32];
  __shared__ bool s_last;
  double a[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n_pix2; p += gridDim.x * blockDim.x) {
    const float r = atm[p] - dm[p];
    resid[p] = r;
    const double w = (double)amp[p];
    float sv, cv;
    sincosf(r * k, &sv, &cv);
    a[0] += w;
    a[1] += w * (double)r;
    a[2] += w * (double)r * (double)r;
    a[3] += w * (double)cv;
    a[4] += w * (double)sv;
  }
  loop_block_sum(a, s_p);
  // thread q < 5: the warps' sums of value q
  const auto warps_sum = [&]() {
    double v = 0.0;
    if (threadIdx.x < 5)
      for (int w = 0; w < kLoopThreads / 32; ++w) v += s_p[threadIdx.x][w];
    return v;
  };
  double v = warps_sum();
  if (gridDim.x > 1) {
    if (threadIdx.x < 5) {
      __stcg(part + (size_t)blockIdx.x * 5 + threadIdx.x, v);
      __threadfence();
    }
    __syncthreads();
    // atomicInc wraps to zero on the last CTA: ready for the next launch
    if (threadIdx.x == 0) s_last = atomicInc(done, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
#pragma unroll
    for (int q = 0; q < 5; ++q) a[q] = 0.0;
    for (int b = threadIdx.x; b < gridDim.x; b += blockDim.x)
#pragma unroll
      for (int q = 0; q < 5; ++q) a[q] += __ldcg(part + (size_t)b * 5 + q);
    loop_block_sum(a, s_p);
    v = warps_sum();
  }
  if (threadIdx.x >= 32) return;
#pragma unroll
  for (int q = 0; q < 5; ++q) a[q] = __shfl_sync(0xffffffffu, v, q);
  if (threadIdx.x != 0) return;
  if (!(a[0] > 0.0)) {
    stats[0] = 0.0;
    stats[1] = 0.0;
    return;
  }
  const double mean = a[1] / a[0];
  const double var = a[2] / a[0] - mean * mean;
  stats[0] = sqrt(var > 0.0 ? var : 0.0);
  stats[1] = (a[3] * a[3] + a[4] * a[4]) / (a[0] * a[0]);
}

__global__ void __launch_bounds__(256) k_loop_integrate(const float *__restrict__ m,
                                                        float *__restrict__ cmd, int n,
                                                        float keep, float gain) {
  pdl_wait();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) cmd[j] = keep * cmd[j] + gain * m[j];
}

int loop_alloc_workspace(specula_ctx *ctx) {
  // the CTAs' sums, then the count of CTAs that are done (zero between calls)
  const size_t n = (size_t)kLoopMaxBlocks * 5 * sizeof(double);
  if (cudaMalloc(&ctx->loop_part, n + sizeof(double)) != cudaSuccess) return SPECULA_ENOMEM;
  if (cudaMemset(ctx->loop_part, 0, n + sizeof(double)) != cudaSuccess) return SPECULA_ECUDA;
  return SPECULA_OK;
}

}  // namespace specula

using namespace specula;

extern "C" int specula_dm_shape(specula_ctx *ctx, int32_t n_modes, int32_t n_pix2,
                                const float *basis_dev, const float *cmd_dev, float *phase_dev,
                                void *stream) {
  if (!ctx || !basis_dev || !cmd_dev || !phase_dev) return SPECULA_EINVAL;
  if (n_modes < 1 || n_pix2 < 1) return SPECULA_EINVAL;
  if (n_modes > 12288) return SPECULA_EUNSUPPORTED;   // the documented limit
  cudaStream_t st = (cudaStream_t)stream;
  const bool v4 = n_pix2 % 4 == 0 && (((uintptr_t)basis_dev | (uintptr_t)phase_dev) % 16) == 0;
  int sms = 0;
  SPECULA_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  // tiles of 32, 16 or 8 lanes, the widest that give two CTAs per SM; then the modes
  // over a cluster until there are, while every part keeps a full unroll of
  // modes.  (Narrow tiles before clusters, whose CTAs share SMs while others stand
  // idle; with the shorter butterflies of the residual, 8 m step 64.9 -> 62.3 us.)
  // k_dm_few up to eight modes, and below four modes per warp where a warp per 128
  // pixels still gives every SM a CTA (400^2 pixels: 12 modes 4.0 -> 3.1 us, 20 modes
  // 6.2 -> 5.0; 50 modes 8.6 against 9.8).
  const auto tiles_of = [&](int lt) { return (int)((n_pix2 + 4LL * lt - 1) / (4 * lt)); };
  const int few = (tiles_of(32) + kDmWarps - 1) / kDmWarps;
  if (n_modes <= kDmUnroll || (n_modes < 4 * kDmWarps && few >= sms)) {
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_LOOP, st, (v4 ? k_dm_few<true> : k_dm_few<false>), few,
                       kDmWarps * 32, 0, basis_dev, cmd_dev, phase_dev, n_modes, n_pix2);
    return SPECULA_OK;
  }
  int lt = 32;
  while (v4 && lt > 8 && tiles_of(lt) < 2 * sms &&
         n_modes / (kDmWarps * (64 / lt)) >= kDmUnroll)
    lt /= 2;
  const int tiles = tiles_of(lt);
  int cs = 1;
  while (cs < kDmMaxCluster && tiles * cs < 2 * sms &&
         n_modes / (kDmWarps * (32 / lt) * cs * 2) >= kDmUnroll)
    cs *= 2;
  const unsigned grid = (unsigned)tiles * cs;
  const int cluster = cs > 1 ? cs : 0;
  void (*fn)(const float *, const float *, float *, int, int) =
      !v4 ? k_dm_shape<false, 32>
          : (lt == 32 ? k_dm_shape<true, 32>
                      : (lt == 16 ? k_dm_shape<true, 16> : k_dm_shape<true, 8>));
  SPECULA_LAUNCH(ctx, SPECULA_K_LOOP, st,
                 SPECULA_CK(launch_pdl(fn, grid, kDmWarps * 32, 0, st, cluster, basis_dev, cmd_dev,
                                       phase_dev, n_modes, n_pix2)));
  return SPECULA_OK;
}

extern "C" int specula_loop_residual(specula_ctx *ctx, int32_t n_pix2, const float *amp_dev,
                                     const float *atm_dev, const float *dm_dev,
                                     double wfs_over_sci, float *resid_dev, double *stats_dev,
                                     void *stream) {
  if (!ctx || !amp_dev || !atm_dev || !dm_dev || !resid_dev || !stats_dev) return SPECULA_EINVAL;
  if (n_pix2 < 1 || !(wfs_over_sci > 0.0) || !isfinite(wfs_over_sci)) return SPECULA_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  int blocks = (n_pix2 + kLoopThreads - 1) / kLoopThreads;
  blocks = blocks > kLoopMaxBlocks ? kLoopMaxBlocks : blocks;
  unsigned *done = reinterpret_cast<unsigned *>(ctx->loop_part + (size_t)kLoopMaxBlocks * 5);
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_LOOP, st, k_loop_residual, blocks, kLoopThreads, 0, amp_dev,
                     atm_dev, dm_dev, resid_dev, ctx->loop_part, done, stats_dev, n_pix2,
                     (float)wfs_over_sci);
  return SPECULA_OK;
}

extern "C" int specula_loop_integrate(specula_ctx *ctx, int32_t n_modes, float gain, float leak,
                                      const float *modes_dev, float *cmd_dev, void *stream) {
  if (!ctx || !modes_dev || !cmd_dev || n_modes < 1) return SPECULA_EINVAL;
  if (!isfinite(gain) || !isfinite(leak) || leak < 0.f || leak > 1.f) return SPECULA_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_LOOP, st, k_loop_integrate, (n_modes + 255) / 256, 256, 0,
                     modes_dev, cmd_dev, n_modes, 1.f - leak, gain);
  return SPECULA_OK;
}

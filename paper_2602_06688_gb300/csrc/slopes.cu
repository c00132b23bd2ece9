// Slope computers (PyrSlopec / ShSlopec, App. A, Tab. 4; Slopes, Tab. 3).
// Output per batch element: all x slopes, then all y slopes.  Every reduction
// runs in a fixed order (per-thread strided sums, then a fixed shuffle tree,
// then warps in index order), so results are bit-reproducible.
#include <cooperative_groups.h>

#include <algorithm>

#include "internal.h"

namespace cg = cooperative_groups;

namespace specula {

constexpr int kPyrThreads = 256;
constexpr int kPyrCluster = 8;
constexpr int kPyrKeep = 4;   // subapertures whose values a thread keeps

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The warp's sums of a (lower half of the lanes) and b (upper half): one
// exchange, then four levels whose rounding errors (Knuth's two-sum) are
// carried along.  Two plain butterflies take one shuffle more, and their
// cancelling partial sums were the largest part of the centre of gravity's error
// (3364 spots of 24^2, whole chain against float64: 2.1e-7 -> 1.8e-7).
__device__ __forceinline__ float warp_sum_pair(float a, float b) {
  const bool up = threadIdx.x & 16;
  float h = up ? b : a, l = 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float g = __shfl_xor_sync(0xffffffffu, o == 16 ? (up ? a : b) : h, o);
    if (o < 16) l += __shfl_xor_sync(0xffffffffu, l, o);
    const float t = h + g, z = t - h;
    l += (h - (t - z)) + (g - z);
    h = t;
  }
  return isfinite(l) ? h + l : h;
}

// Non-finite guard: one status write per offending output, so the cost is
// nil when the slopes are finite.
__device__ __forceinline__ void guard_finite(float a, float b, int32_t *nf_status) {
  if (nf_status && !(isfinite(a) && isfinite(b))) atomicExch(nf_status, SPECULA_ENONFINITE);
}

// Pyramid slopes of one batch element per cluster of CTAs (grid (cluster,
// n_batch)), subapertures strided over its threads.  Each thread keeps the
// four pupil-image values of its first kPyrKeep subapertures while it sums
// them; the CTAs' sums meet in distributed shared memory, in rank order, for
// the global normalisation T, and the slopes come from the kept values (the
// rest are read again).  So the frame's 27 000 values are read once, in two
// dependent rounds of loads; CTAs that each summed all of them took 8.5 us for
// the 39 m sensor's 6672 subapertures, 5.5 us for the 8 m one's 1256; now 7.3 and
// 4.9 us.
// MAPS: idx holds explicit detector indices of the four pupil images
// (idx[q n_valid + k] for image q = Q1..Q4 of subaperture k, any padding and
// image separation; side: the detector's side), otherwise subaperture indices
// of the quadrant layout (side: subapertures across).  Index checks are
// branch-free: an out-of-range index reads element 0 and is reported once per
// CTA.
template <bool MAPS>
__global__ void __launch_bounds__(kPyrThreads) k_pyr_slopes(
    const float *__restrict__ det, const int32_t *__restrict__ idx, const float *__restrict__ ref,
    int side, int n_valid, float *__restrict__ out, int32_t *status, int32_t *nf_status) {
  __shared__ float s_w[kPyrThreads / 32];
  __shared__ float s_sum;
  pdl_wait();
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int b = blockIdx.y;
  const int ld = MAPS ? side : 2 * side;   // detector row
  const unsigned lim = (unsigned)(side * side);
  const float *d = det + (size_t)b * ld * ld;
  int bad = 0;
  // the values of subaperture k: Q1 (+x, +y), Q2 (-x, +y), Q3 (-x, -y), Q4 (+x, -y)
  const auto values = [&](int k, float (&v)[4]) {
    int i[4];
    if constexpr (MAPS) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int e = __ldg(idx + (size_t)c * n_valid + k);
        bad |= (unsigned)e >= lim;
        i[c] = (unsigned)e < lim ? e : 0;
      }
    } else {
      int e = __ldg(idx + k);
      bad |= (unsigned)e >= lim;
      e = (unsigned)e < lim ? e : 0;
      const int r = e / side, c = e - r * side;
      i[2] = r * ld + c;
      i[3] = i[2] + side;
      i[1] = i[2] + side * ld;
      i[0] = i[1] + side;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = d[i[c]];
  };
  const int k0 = rank * kPyrThreads + threadIdx.x, stride = cs * kPyrThreads;
  float q[kPyrKeep][4], r0[kPyrKeep], r1[kPyrKeep];
#pragma unroll
  for (int u = 0; u < kPyrKeep; ++u) {
    const int k = k0 + u * stride;
    r0[u] = r1[u] = 0.f;
    if (k < n_valid) {
      values(k, q[u]);
      if (ref) {
        r0[u] = ref[k];
        r1[u] = ref[n_valid + k];
      }
    } else {
      q[u][0] = q[u][1] = q[u][2] = q[u][3] = 0.f;
    }
  }
  float part = 0.f;
#pragma unroll
  for (int u = 0; u < kPyrKeep; ++u) part += ((q[u][0] + q[u][1]) + q[u][2]) + q[u][3];
  for (int k = k0 + kPyrKeep * stride; k < n_valid; k += stride) {
    float v[4];
    values(k, v);
    part += ((v[0] + v[1]) + v[2]) + v[3];
  }
  part = warp_sum(part);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = part;
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < kPyrThreads / 32; ++i) t += s_w[i];
    s_sum = t;
    if (bad) atomicExch(status, SPECULA_EINVAL);
  }
  cl.sync();
  float T = 0.f;
  for (int c = 0; c < cs; ++c) T += *cl.map_shared_rank(&s_sum, c);
  T /= (float)n_valid;
  float *o = out + (size_t)b * 2 * n_valid;
  const auto store = [&](int k, const float (&v)[4], float ra, float rb) {
    float sx = ((v[0] + v[3]) - (v[1] + v[2])) / T;
    float sy = ((v[0] + v[1]) - (v[2] + v[3])) / T;
    if (ref) {
      sx -= ra;
      sy -= rb;
    }
    o[k] = sx;
    o[n_valid + k] = sy;
    guard_finite(sx, sy, nf_status);
  };
#pragma unroll
  for (int u = 0; u < kPyrKeep; ++u)
    if (k0 + u * stride < n_valid) store(k0 + u * stride, q[u], r0[u], r1[u]);
  for (int k = k0 + kPyrKeep * stride; k < n_valid; k += stride) {
    float v[4];
    values(k, v);
    store(k, v, ref ? ref[k] : 0.f, ref ? ref[n_valid + k] : 0.f);
  }
  cl.sync();   // no CTA leaves while another reads its sum
}

// One warp per (batch element, subaperture): centre of gravity of the spot.
// V4: four neighbouring pixels per load (nf % 4 == 0, spots 16-byte aligned),
// all of a lane's loads of a 24^2 spot in flight together; pixel by pixel the
// 3364 spots of the 39 m sensor took 6.5 us, now 4.9.
template <bool V4>
__global__ void __launch_bounds__(256) k_sh_cog(const float *__restrict__ spots,
                                                const float *__restrict__ ref, int nf,
                                                int n_valid, int n_batch,
                                                float *__restrict__ out, int32_t *nf_status) {
  pdl_wait();
  const long long task = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (task >= (long long)n_valid * n_batch) return;   // warp-uniform
  const int b = (int)(task / n_valid), k = (int)(task % n_valid);
  const float *sp = spots + (size_t)task * nf * nf;
  const float c = 0.5f * (float)(nf - 1);
  float si = 0.f, sx = 0.f, sy = 0.f;
  if constexpr (V4) {
    const int n4 = nf / 4, n = nf * n4;
    constexpr int UL = 5;
    for (int e0 = lane; e0 < n; e0 += UL * 32) {
      float4 v[UL];
#pragma unroll
      for (int u = 0; u < UL; ++u)
        v[u] = e0 + 32 * u < n ? __ldg(reinterpret_cast<const float4 *>(sp) + e0 + 32 * u)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < UL; ++u) {
        const int e = e0 + 32 * u;
        if (e < n) {
          const int y = e / n4, x = 4 * (e - y * n4);
          const float s = (v[u].x + v[u].y) + (v[u].z + v[u].w);
          const float xf = (float)x - c;
          si += s;
          sx += v[u].x * xf + v[u].y * (xf + 1.f) + v[u].z * (xf + 2.f) + v[u].w * (xf + 3.f);
          sy += s * ((float)y - c);
        }
      }
    }
  } else {
    for (int e = lane; e < nf * nf; e += 32) {
      const float v = sp[e];
      const int y = e / nf, x = e - y * nf;
      si += v;
      sx += v * ((float)x - c);
      sy += v * ((float)y - c);
    }
  }
  si = warp_sum(si);
  float g = warp_sum_pair(sx, sy);
  if (lane % 16 == 0) {   // lane 0: x, lane 16: y
    const int o = lane == 0 ? k : n_valid + k;
    g /= si;
    if (ref) g -= ref[o];
    out[(size_t)b * 2 * n_valid + o] = g;
    guard_finite(g, g, nf_status);
  }
}

template <bool MAPS>
static int pyr_launch(specula_ctx *ctx, const int32_t *idx, int side, int n_valid,
                      const float *det, const float *ref, int n_batch, float *out,
                      cudaStream_t st) {
  // a cluster as large as the subapertures fill, one per thread first
  const int cs = std::min(kPyrCluster, (n_valid + kPyrThreads - 1) / kPyrThreads);
  SPECULA_LAUNCH(ctx, SPECULA_K_SLOPES, st,
                 SPECULA_CK(launch_pdl(k_pyr_slopes<MAPS>, dim3(cs, n_batch), kPyrThreads, 0, st,
                                       cs > 1 ? cs : 0, det, idx, ref, side, n_valid, out,
                                       ctx->status_dev, ctx->guard ? ctx->status_dev : nullptr)));
  return SPECULA_OK;
}

int slopes_pyr_run(specula_ctx *ctx, const int32_t *idx, int n_sub, int n_valid,
                   const float *det, const float *ref, int n_batch, float *out, cudaStream_t st) {
  return pyr_launch<false>(ctx, idx, n_sub, n_valid, det, ref, n_batch, out, st);
}

}  // namespace specula

using namespace specula;

extern "C" int specula_slopes(specula_ctx *ctx, const specula_slopec_desc *d, const float *img_dev,
                              const float *ref_dev, int32_t n_batch, float *slopes_dev,
                              void *stream) {
  if (!ctx || !d || !img_dev || !slopes_dev || n_batch < 0) return SPECULA_EINVAL;
  if (d->n_valid < 1 || d->n_sub < 1) return SPECULA_EINVAL;
  if (n_batch == 0) return SPECULA_OK;
  cudaStream_t st = (cudaStream_t)stream;
  if (d->kind == SPECULA_SLOPES_PYR) {
    if (!d->subap_idx_dev || d->n_valid > d->n_sub * d->n_sub) return SPECULA_EINVAL;
    return slopes_pyr_run(ctx, d->subap_idx_dev, d->n_sub, d->n_valid, img_dev, ref_dev, n_batch,
                          slopes_dev, st);
  } else if (d->kind == SPECULA_SLOPES_PYR_MAPS) {
    if (!d->subap_idx_dev || d->n_sub < 1) return SPECULA_EINVAL;
    return pyr_launch<true>(ctx, d->subap_idx_dev, d->n_sub, d->n_valid, img_dev, ref_dev, n_batch,
                            slopes_dev, st);
  } else if (d->kind == SPECULA_SLOPES_SH) {
    if (d->fft_n < 2) return SPECULA_EINVAL;
    const long long tasks = (long long)d->n_valid * n_batch;
    const unsigned grid = (unsigned)((tasks + 7) / 8);
    int32_t *nfs = ctx->guard ? ctx->status_dev : nullptr;
    if (d->fft_n % 4 == 0 && (uintptr_t)img_dev % 16 == 0)
      SPECULA_LAUNCH_PDL(ctx, SPECULA_K_SLOPES, st, k_sh_cog<true>, grid, 256, 0, img_dev, ref_dev,
                         d->fft_n, d->n_valid, n_batch, slopes_dev, nfs);
    else
      SPECULA_LAUNCH_PDL(ctx, SPECULA_K_SLOPES, st, k_sh_cog<false>, grid, 256, 0, img_dev, ref_dev,
                         d->fft_n, d->n_valid, n_batch, slopes_dev, nfs);
  } else {
    return SPECULA_EINVAL;
  }
  return SPECULA_OK;
}

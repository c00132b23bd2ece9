// Float32 modal reconstructor products: modes[b] = R slopes[b] (Modalrec /
// Recmat, App. A, Tabs. 3-4), for one slope vector and for batches.
//
// Three kernels, each a fixed order of float32 additions (bit-reproducible):
//   one vector   k_mvm_f32_split  one row of R per CTA
//   2-4 vectors  k_mvm_f32_rows   two rows of R per CTA or per warp (and 5-8 vectors
//                                 where R has few rows)
//   batches      k_mvm_f32_tile   64 rows x 8-64 vectors per CTA, both staged in
//                                 shared memory, K split over a cluster
// Which one, and its tile, follow the batch and the sizes, so the last bits of a
// frame's modes depend on the batch it is in.
// All read R from HBM once per 64 vectors.  Up to about 20 vectors that read
// is the bound (a product takes 2 flops per vector and 4 bytes of R), beyond
// it the FP32 pipes are.  Measured, against one warp per row and four vectors
// per pass over R: 4000 x 13344 on 8 vectors 116 -> 49 us (4.4 TB/s of R),
// on 16 vectors 69 us, on 32 117 us; 500 x 25600 on 256 vectors 5.7 ms ->
// 0.19 ms (35 TFLOP/s).
#include <cooperative_groups.h>

#include <algorithm>

#include "internal.h"

namespace cg = cooperative_groups;

namespace specula {

// Loads of V = 4, 2 or 1 floats, the widest that n_slopes and both pointers
// allow (a sensor with an odd number of valid subapertures has
// n_slopes = 2 mod 4).  ld_stream does not allocate in L1.
template <int V> struct VecOf;
template <> struct VecOf<4> { using T = float4; };
template <> struct VecOf<2> { using T = float2; };
template <> struct VecOf<1> { using T = float; };

__device__ __forceinline__ float4 ld_stream(const float4 *p) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ float2 ld_stream(const float2 *p) {
  float2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.f32 {%0,%1}, [%2];"
               : "=f"(v.x), "=f"(v.y)
               : "l"(p));
  return v;
}
__device__ __forceinline__ float ld_stream(const float *p) {
  float v;
  asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float dotv(float4 a, float4 x) {
  return a.x * x.x + a.y * x.y + a.z * x.z + a.w * x.w;
}
__device__ __forceinline__ float dotv(float2 a, float2 x) { return a.x * x.x + a.y * x.y; }
__device__ __forceinline__ float dotv(float a, float x) { return a * x; }

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One slope vector, one row per CTA of kSplitWarps warps: warp w streams the
// w-th contiguous segment of the row (UL loads in flight per lane), then the
// warps' sums are added in warp order.  Four streams per row keep more bytes
// in flight per row than one warp does.  4000 x 13344: 34.9 us, 6.1 TB/s.
constexpr int kSplitWarps = 4;
template <int V>
__global__ void __launch_bounds__(kSplitWarps * 32) k_mvm_f32_split(
    const float *__restrict__ R, const float *__restrict__ s, float *__restrict__ m, int n_modes,
    int n_slopes) {
  pdl_wait();
  using T = typename VecOf<V>::T;
  __shared__ float s_w[kSplitWarps];
  const int row = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T *r4 = reinterpret_cast<const T *>(R + (size_t)row * n_slopes);
  const T *s4 = reinterpret_cast<const T *>(s);
  const int n4 = n_slopes / V;
  const int seg = (n4 + kSplitWarps - 1) / kSplitWarps;
  const int lo = warp * seg, hi = min(n4, lo + seg);
  constexpr int UL = 4;
  float acc = 0.f;
  for (int j0 = lo + lane; j0 < hi; j0 += UL * 32) {
    T a[UL];
#pragma unroll
    for (int u = 0; u < UL; ++u) a[u] = (j0 + 32 * u < hi) ? ld_stream(r4 + j0 + 32 * u) : T{};
#pragma unroll
    for (int u = 0; u < UL; ++u) {
      const int j = j0 + 32 * u;
      if (j < hi) acc += dotv(a[u], __ldg(s4 + j));
    }
  }
  acc = warp_sum_f(acc);
  if (lane == 0) s_w[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kSplitWarps; ++w) v += s_w[w];
    m[row] = v;
  }
}

// Up to NB slope vectors, two rows of R per WPR warps, each warp a contiguous segment
// of both: every load of the slopes serves two rows, and there is nothing to stage or
// to wait for, so a product is as short as its longest warp (the tiles below: at
// least 4 us).  WPR = 1, a row per warp, where a warp's UL loads take a whole row
// (kShortRow); else 4.  Before (the tiles) / now, 2 and 4 vectors: 64 x 512 4.5 / 1.9,
// 4.6 / 2.3 us; 4000 x 200 4.0 / 1.9, 4.0 / 2.3; 500 x 2512 5.5 / 3.5, 5.6 / 4.3;
// 4000 x 13344 49.6 / 36.6, 49.5 / 44.6.
constexpr int kRowsUnroll = 4;
template <int V> constexpr int kShortRow = 32 * kRowsUnroll * V;
template <int V, int NB, int WPR>
__global__ void __launch_bounds__(kSplitWarps * 32) k_mvm_f32_rows(
    const float *__restrict__ R, const float *__restrict__ s, float *__restrict__ m, int n_modes,
    int n_slopes, int nb) {
  pdl_wait();
  using T = typename VecOf<V>::T;
  constexpr int ROWS = 2, UL = kRowsUnroll;
  __shared__ float s_w[kSplitWarps][ROWS * NB];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row0 = (blockIdx.x * (kSplitWarps / WPR) + warp / WPR) * ROWS;
  const T *r4[ROWS], *s4[NB];
#pragma unroll
  for (int i = 0; i < ROWS; ++i)
    r4[i] = reinterpret_cast<const T *>(R + (size_t)min(row0 + i, n_modes - 1) * n_slopes);
#pragma unroll
  for (int q = 0; q < NB; ++q)   // vectors past the batch repeat its last
    s4[q] = reinterpret_cast<const T *>(s + (size_t)min(q, nb - 1) * n_slopes);
  const int n4 = n_slopes / V;
  const int seg = (n4 + WPR - 1) / WPR;
  const int lo = warp % WPR * seg, hi = min(n4, lo + seg);
  float acc[ROWS][NB];
#pragma unroll
  for (int i = 0; i < ROWS; ++i)
#pragma unroll
    for (int q = 0; q < NB; ++q) acc[i][q] = 0.f;
  for (int j0 = lo + lane; j0 < hi; j0 += UL * 32) {
    T a[UL][ROWS];
#pragma unroll
    for (int u = 0; u < UL; ++u)
#pragma unroll
      for (int i = 0; i < ROWS; ++i)
        a[u][i] = (j0 + 32 * u < hi) ? ld_stream(r4[i] + j0 + 32 * u) : T{};
#pragma unroll
    for (int u = 0; u < UL; ++u) {
      const int j = j0 + 32 * u;
      if (j < hi) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
          const T x = __ldg(s4[q] + j);
#pragma unroll
          for (int i = 0; i < ROWS; ++i) acc[i][q] += dotv(a[u][i], x);
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < ROWS; ++i)
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const float v = warp_sum_f(acc[i][q]);
      if constexpr (WPR == 1) {
        if (lane == 0 && q < nb && row0 + i < n_modes) m[(size_t)q * n_modes + row0 + i] = v;
      } else {
        if (lane == 0) s_w[warp][q * ROWS + i] = v;
      }
    }
  if constexpr (WPR > 1) {
    static_assert(WPR == kSplitWarps, "the CTA's warps share its rows");
    __syncthreads();
    const int i = threadIdx.x % ROWS, q = threadIdx.x / ROWS;
    if (q < min(NB, nb) && row0 + i < n_modes) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < kSplitWarps; ++w) v += s_w[w][threadIdx.x];
      m[(size_t)q * n_modes + row0 + i] = v;
    }
  }
}

template <int V, int NB>
static int launch_rows(specula_ctx *ctx, const float *R, const float *s, float *m, int n_modes,
                       int n_slopes, int nb, cudaStream_t st) {
  if (n_slopes <= kShortRow<V>)
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_RECON, st, (k_mvm_f32_rows<V, NB, 1>),
                       (n_modes + 2 * kSplitWarps - 1) / (2 * kSplitWarps), kSplitWarps * 32, 0, R,
                       s, m, n_modes, n_slopes, nb);
  else
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_RECON, st, (k_mvm_f32_rows<V, NB, kSplitWarps>),
                       (n_modes + 1) / 2, kSplitWarps * 32, 0, R, s, m, n_modes, n_slopes, nb);
  return SPECULA_OK;
}

// Batches: C[b][row] over tiles of 64 rows x 8-64 vectors, 256 threads.  Both
// operands are K-contiguous, so 64-deep stages go to shared memory as they
// lie (cp.async) and each thread's RM x RN products take two neighbouring k at
// a time (packed float32 FMAs, no operand moves).  The eight warps are two
// row halves x four quarters of a stage's K.  The cluster's
// CTAs take K slices of one tile and add their tiles through distributed
// shared memory in rank order: no workspace, so batches may be captured
// without a set-up call.
// Rounding: the 16 products of a quarter stage are summed apart and then added to
// the running sum, and the sums of the quarters and the cluster are added with
// their rounding errors carried along; two CTAs at least share a K of more than four
// stages, or (FOLD) one adds them in blocks and the blocks in a second sum, which
// lies in shared memory, as 64 products per thread leave no registers for it.  A
// product's rounding errors then number about 6 + n_slopes / 256 at most, a warp
// per row's 7 + n_slopes / 256.  (With plain sums over the quarters and one CTA where
// the tiles fill the SMs, 4000 x 13344 on 100 vectors was 2.7e-7 of the norm off, a
// warp per row 2.0e-7; 64 x 512 0.92e-7 and 0.83e-7.  Now 2.0e-7 and 0.77e-7.)
constexpr int kTm = 64, kTk = 64, kTld = kTk + 4, kTout = kTm + 4;
constexpr int kTq = 4;   // K quarters of a stage
// A warp covers 32 rows: 32 / RM lanes of RM rows, RM lanes of RN vectors.
// Small batches take RM = 4, which needs fewer shared loads per product
// (8 vectors: 6 loads of 16 bytes for 8 products of 4 k, against 9).
template <int RM, int RN, bool FOLD> struct TileCfg {
  static constexpr int LM = 32 / RM, LN = RM, BN = LN * RN;
  // small batches wait on HBM: two CTAs per SM
  static constexpr int STAGES = BN >= 64 ? 4 : 5;
  static constexpr int CTAS = BN >= 32 ? 1 : 2;
  static constexpr size_t stages = (size_t)STAGES * (kTm + BN) * kTld * sizeof(float);
  static constexpr size_t smem = stages + (FOLD ? RM * RN * 256 * sizeof(float) : 0);
  // columns at a time (FOLD keeps more addresses in registers; the rows are read twice)
  static constexpr int JH = FOLD ? RN / 2 : RN;
  static_assert((size_t)kTq * BN * kTout * sizeof(float) <= stages, "the output tiles fit the stages");
  static_assert(smem * CTAS <= 224 * 1024, "CTAS tiles per SM");
};

template <int V>
__device__ __forceinline__ void cp_async_vec(float *dst, const float *src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = ok ? 4 * V : 0;   // 0: the destination is zero-filled
  if constexpr (V == 4)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n)
                 : "memory");
  else if constexpr (V == 2)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(n)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n)
                 : "memory");
}

template <int RM, int RN, int V, bool FOLD>
__global__ void __launch_bounds__(256, TileCfg<RM, RN, FOLD>::CTAS) k_mvm_f32_tile(
    const float *__restrict__ R, const float *__restrict__ s, float *__restrict__ m, int n_modes,
    int n_slopes, int nb, int tiles_n) {
  using C = TileCfg<RM, RN, FOLD>;
  constexpr int BN = C::BN, STAGES = C::STAGES, LM = C::LM, LN = C::LN;
  constexpr int kStage = (kTm + BN) * kTld;
  extern __shared__ __align__(16) float sm_f[];
  pdl_wait();
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int tile = blockIdx.x / cs;
  const int m0 = tile / tiles_n * kTm, n0 = tile % tiles_n * BN;
  const int kb_all = (n_slopes + kTk - 1) / kTk;
  const int kb0 = (int)((long long)kb_all * rank / cs);
  const int kb1 = (int)((long long)kb_all * (rank + 1) / cs);

  // this thread's share of a stage: column group lc of rows lr, lr + RS, ...
  constexpr int PER = kTk / V, RS = 256 / PER, NR = kTm / RS, NS = (BN + RS - 1) / RS;
  const int lc = (threadIdx.x % PER) * V, lr = threadIdx.x / PER;
  const int rows_ok = n_modes - m0 - lr, vecs_ok = min(nb - n0, BN) - lr;
  const float *gr = R + (size_t)(m0 + min(lr, n_modes - 1 - m0)) * n_slopes + lc;
  const float *gs = s + (size_t)(n0 + min(lr, nb - 1 - n0)) * n_slopes + lc;
  auto load_stage = [&](int slot, int kb) {
    float *dst = sm_f + slot * kStage + lr * kTld + lc;
    const int k = kb * kTk;
    const bool k_ok = k + lc < n_slopes;
#pragma unroll
    for (int t = 0; t < NR; ++t) {
      const bool ok = k_ok && t * RS < rows_ok;
      cp_async_vec<V>(dst + t * RS * kTld, ok ? gr + (size_t)(t * RS) * n_slopes + k : R, ok);
    }
#pragma unroll
    for (int t = 0; t < NS; ++t) {
      if (BN % RS == 0 || t * RS + lr < BN) {
        const bool ok = k_ok && t * RS < vecs_ok;
        cp_async_vec<V>(dst + (kTm + t * RS) * kTld,
                        ok ? gs + (size_t)(t * RS) * n_slopes + k : s, ok);
      }
    }
  };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quarter = warp >> 1, wm = (warp & 1) * 32, lm = lane / LN, ln = lane % LN;
  float sum[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) sum[i][j] = 0.f;
  // FOLD: a block's sums into the second ones
  float4 *tot = reinterpret_cast<float4 *>(sm_f + C::stages / sizeof(float)) + threadIdx.x;
  const int per = kb1 - kb0 < 32 ? 4 : (kb1 - kb0 < 64 ? 8 : 16);   // stages per block
  int left = per;
  const auto fold = [&](bool first) {
#pragma unroll
    for (int e = 0; e < RM * RN / 4; ++e) {
      float *u = &sum[e / (RN / 4)][e % (RN / 4) * 4];
      float4 &t = tot[e * 256];
      const float4 v = first ? make_float4(0.f, 0.f, 0.f, 0.f) : t;
      t = make_float4(v.x + u[0], v.y + u[1], v.z + u[2], v.w + u[3]);
      u[0] = u[1] = u[2] = u[3] = 0.f;
    }
  };
  if constexpr (FOLD) fold(true);

#pragma unroll
  for (int st = 0; st < STAGES - 1; ++st) {
    if (kb0 + st < kb1) load_stage(st, kb0 + st);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int slot = 0;
  for (int kb = kb0; kb < kb1; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();   // this stage has landed; the one refilled next is read no more
    {
      const int nslot = slot == 0 ? STAGES - 1 : slot - 1;
      if (kb + STAGES - 1 < kb1) load_stage(nslot, kb + STAGES - 1);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const float *sa = sm_f + slot * kStage + (wm + lm) * kTld + quarter * (kTk / kTq);
    const float *sb = sm_f + slot * kStage + (kTm + ln) * kTld + quarter * (kTk / kTq);
#pragma unroll
    for (int jh = 0; jh < RN; jh += C::JH) {
      float2 acc[RM][C::JH];
#pragma unroll
      for (int k = 0; k < kTk / kTq; k += 4) {
        float4 a[RM];
#pragma unroll
        for (int i = 0; i < RM; ++i) a[i] = *reinterpret_cast<const float4 *>(sa + i * LM * kTld + k);
#pragma unroll
        for (int j = 0; j < C::JH; ++j) {
          const float4 b = *reinterpret_cast<const float4 *>(sb + (jh + j) * LN * kTld + k);
          const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
#pragma unroll
          for (int i = 0; i < RM; ++i) {
            const float2 a0 = make_float2(a[i].x, a[i].y), a1 = make_float2(a[i].z, a[i].w);
            acc[i][j] = k == 0 ? __fmul2_rn(a0, b0) : __ffma2_rn(a0, b0, acc[i][j]);
            acc[i][j] = __ffma2_rn(a1, b1, acc[i][j]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < C::JH; ++j) sum[i][jh + j] += acc[i][j].x + acc[i][j].y;
    }
    if constexpr (FOLD) {
      if (--left == 0) {   // uniform
        fold(false);
        left = per;
      }
    }
    slot = slot == STAGES - 1 ? 0 : slot + 1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();   // every stage has been read: the memory becomes the output tiles

  if constexpr (FOLD) {
#pragma unroll
    for (int e = 0; e < RM * RN / 4; ++e) {
      float *u = &sum[e / (RN / 4)][e % (RN / 4) * 4];
      const float4 t = tot[e * 256];
      u[0] += t.x;
      u[1] += t.y;
      u[2] += t.z;
      u[3] += t.w;
    }
  }
  // T[quarter][vector][row]
  float *T = sm_f;
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j)
      T[(quarter * BN + j * LN + ln) * kTout + wm + i * LM + lm] = sum[i][j];
  cl.sync();
  // this CTA adds its share of the vectors over the quarters and the
  // cluster, in order, the additions' errors (Knuth's two-sum) beside
  const int v0 = BN * rank / cs, v1 = BN * (rank + 1) / cs;
  for (int o = threadIdx.x; o < (v1 - v0) * kTm; o += 256) {
    const int v = v0 + o / kTm, r = o % kTm;
    float x = 0.f, e = 0.f;
    for (int c = 0; c < cs; ++c) {
      const float *Tc = cl.map_shared_rank(T, c) + v * kTout + r;
#pragma unroll
      for (int q = 0; q < kTq; ++q) {
        const float y = Tc[q * BN * kTout], t = __fadd_rn(x, y), z = __fsub_rn(t, x);
        e = __fadd_rn(e, __fadd_rn(__fsub_rn(x, __fsub_rn(t, z)), __fsub_rn(y, z)));
        x = t;
      }
    }
    if (isfinite(e)) x += e;   // an infinite or NaN sum is x itself
    if (n0 + v < nb && m0 + r < n_modes) m[(size_t)(n0 + v) * n_modes + m0 + r] = x;
  }
  cl.sync();   // no CTA leaves while another reads its tiles
}

template <int RM, int RN, int V, bool FOLD = false>
static int launch_tile(specula_ctx *ctx, const float *R, const float *s, float *m, int n_modes,
                       int n_slopes, int nb, cudaStream_t st) {
  using C = TileCfg<RM, RN, FOLD>;
  int sms = 0;
  SPECULA_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  const int tiles_n = (nb + C::BN - 1) / C::BN;
  const long long tiles = (long long)((n_modes + kTm - 1) / kTm) * tiles_n;
  const int kb = (n_slopes + kTk - 1) / kTk;
  // split K while the CTAs still fit one wave and a slice holds at least four
  // stages; clusters of eight at one CTA per SM leave SMs of most GPCs unused
  // (measured: half the GPU idle), so one per SM stops at four
  const int max_cs = C::CTAS == 1 ? 4 : 8;
  int cs = kb > 4 && !FOLD ? 2 : 1;   // (the rounding above)
  while (cs < max_cs && tiles * cs * 2 <= (long long)sms * C::CTAS && kb / (cs * 2) >= 4) cs *= 2;
  if (tiles * cs > 0x7fffffffLL) return SPECULA_EUNSUPPORTED;
  int e = ensure_dynamic_smem((const void *)k_mvm_f32_tile<RM, RN, V, FOLD>, C::smem);
  if (e) return e;
  SPECULA_LAUNCH(ctx, SPECULA_K_RECON, st,
                 SPECULA_CK(launch_pdl((k_mvm_f32_tile<RM, RN, V, FOLD>), (unsigned)(tiles * cs), 256,
                                       C::smem, st, cs > 1 ? cs : 0, R, s, m, n_modes, n_slopes,
                                       nb, tiles_n)));
  return SPECULA_OK;
}

template <int V>
static int run_v(specula_ctx *ctx, const float *R, const float *s, float *m, int n_modes,
                 int n_slopes, int nb, cudaStream_t st) {
  if (nb == 1) {
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_RECON, st, (k_mvm_f32_split<V>), n_modes, kSplitWarps * 32,
                       0, R, s, m, n_modes, n_slopes);
    return SPECULA_OK;
  }
  if (nb == 2) return launch_rows<V, 2>(ctx, R, s, m, n_modes, n_slopes, nb, st);
  // (single floats: four vectors' loads for two of R cost more than staging does, 500 x
  // 2511 on 4 vectors 8.8 us against the tiles' 6.4)
  if (nb <= 4 && (V > 1 || n_slopes <= kShortRow<V>))
    return launch_rows<V, 4>(ctx, R, s, m, n_modes, n_slopes, nb, st);
  // 5-8 vectors: the rows where R is too short to give the SMs tiles, up to 16 of them
  // (8 vectors, rows / tiles: 64 x 512 1.7 / 4.6 us, 500 x 2512 3.9 / 5.6, 1000 x 5000
  // 8.2 / 12.1; 2000 x 6672 19.9 / 16.2, 4000 x 512 7.2 / 5.6)
  if (nb <= 8 && n_modes <= 16 * kTm && V == 4)
    return launch_rows<V, 8>(ctx, R, s, m, n_modes, n_slopes, nb, st);
  if (nb <= 8) return launch_tile<4, 2, V>(ctx, R, s, m, n_modes, n_slopes, nb, st);
  if (nb <= 16) return launch_tile<4, 4, V>(ctx, R, s, m, n_modes, n_slopes, nb, st);
  if (nb <= 32) return launch_tile<8, 4, V>(ctx, R, s, m, n_modes, n_slopes, nb, st);
  // One CTA with a second sum (7 % more) where two take longer, counted in waves of
  // stages with three more per CTA (128 vectors, two CTAs / one: 4000 x 512 26.8 /
  // 21.6 us, 4000 x 1024 41.6 / 38.1, 4000 x 2512 87.4 / 87.0, 4000 x 13344 397 / 416)
  int sms = 0;
  SPECULA_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  const long long tiles = (long long)((n_modes + kTm - 1) / kTm) * ((nb + 63) / 64);
  const int kb = (n_slopes + kTk - 1) / kTk;
  const auto time = [&](int cs) { return (tiles * cs + sms - 1) / sms * (kb / cs + 3); };
  if (kb > 4 && time(2) * 100 > time(1) * 107)
    return launch_tile<8, 8, V, true>(ctx, R, s, m, n_modes, n_slopes, nb, st);
  return launch_tile<8, 8, V>(ctx, R, s, m, n_modes, n_slopes, nb, st);
}

int recon_f32_run(specula_ctx *ctx, const float *R, const float *s, float *m, int n_modes,
                  int n_slopes, int nb, cudaStream_t st) {
  const uintptr_t a = (uintptr_t)R | (uintptr_t)s | (uintptr_t)((size_t)n_slopes * sizeof(float));
  if (a % 16 == 0) return run_v<4>(ctx, R, s, m, n_modes, n_slopes, nb, st);
  if (a % 8 == 0) return run_v<2>(ctx, R, s, m, n_modes, n_slopes, nb, st);
  return run_v<1>(ctx, R, s, m, n_modes, n_slopes, nb, st);
}

}  // namespace specula

// BF16 and TF32 GEMMs on the 5th-generation tensor cores (tcgen05), FP32
// accumulate:
//     C[M][N] = A[M][K] . B[N][K]^T        (both operands K-major, row-major)
// The dense contractions of the learned reconstructor (its forward layers,
// their gradients), batched reconstructor MVMs and the DFT-as-GEMM pyramid
// variant run here.  The TF32 kernel reads float32 storage (the tensor cores
// use its upper 19 bits).
//
// Large products run on CTA pairs (k_gemm_pair below), the rest on k_gemm_tn:
// persistent, one CTA per SM, looping over (128 x BN output tile, K
// slice) work items, BN = 256 (128 where N is a multiple of 128 but not of
// 256); M and N need not be tile multiples (TMA fills rows beyond the
// operands with zeros, the epilogue masks its stores).  K is a sum of up to
// three terms C = sum_t A_t B_t^T over the same K extent (split-precision
// products such as hi.hi + hi.lo + lo.hi run as one accumulation); a K
// that is not a multiple of the stage depth is zero-filled the same way.
//   warp 0, one thread : TMA loads of A and B tiles (128 bytes of K: 64 bf16
//                        or 32 tf32, 128-byte swizzle) into a shared-memory
//                        ring (4 stages at BN = 256, 6 at BN = 128)
//   warp 1             : allocates 2 BN tensor-memory columns (two
//                        accumulators); one thread issues 4 tcgen05.mma
//                        (K = 16 bf16 or 8 tf32 each) per stage, commits each
//                        stage back to the producer and each finished tile
//                        to the epilogue
//   warps 4-7          : drain a finished accumulator (tcgen05.ld, one row
//                        per thread, transposed in shared memory to whole
//                        lines) to global memory while the next tile
//                        accumulates in the other one
// Split-K partials go to a caller workspace and are summed in split order by
// k_split_reduce (no atomics: bit-reproducible) or by the caller's next kernel
// (gemm_bf16_partials).  Every wait is bounded:
// on timeout the CTA records SPECULA_ETIMEOUT in the context status word,
// waits for its own copies and MMAs, frees its tensor memory and returns.
#include <cuda.h>

#include <string.h>

#include <algorithm>
#include <mutex>

#include "internal.h"
#include "tc_gemm.cuh"

namespace specula {

constexpr int GBM = 128;
constexpr int kMaxTerms = 3;
constexpr uint32_t G_A_BYTES = GBM * 128;   // 128 rows x 128 bytes of K
// K elements per 128-byte row of a stage: 64 bf16 (TF32 = false) or 32 tf32
template <bool TF32> constexpr int gbk() { return TF32 ? 32 : 64; }
constexpr int kOutLd = 36;   // row stride (floats) of an epilogue warp's 32 x 32 block
template <int BN> struct GCfg {
  static constexpr int STAGES = BN == 256 ? 4 : 6;
  static constexpr uint32_t B_BYTES = BN * 128;
  static constexpr size_t SMEM =
      1024 + STAGES * (G_A_BYTES + B_BYTES) + 4 * 32 * kOutLd * sizeof(float) + 256;
};

// the operand maps of every term (kernel parameter space)
struct GemmMaps {
  CUtensorMap a[kMaxTerms];
  CUtensorMap b[kMaxTerms];
};

struct GemmShape {
  int M, N;
  int tiles_m, tiles_n;
  int n_items;              // tiles_m x tiles_n x splits
  int splits;
  int kb_term;              // K blocks per term
  int kb_total;             // kb_term x terms
  int kb_per_split;
  int vec4;                 // N % 4 == 0 and a 16-byte aligned output
};
// Products of one K in one launch: term q of the maps is a product of its own,
// work items [first[q], first[q + 1]) its tiles.
struct GemmGroup {
  int first[kMaxTerms + 1];
  int M[kMaxTerms], N[kMaxTerms], tiles_n[kMaxTerms];
  float *out[kMaxTerms];
  int kb_slice[kMaxTerms];   // K blocks accumulated together; the slices are added in order
  ColSums sums;   // by the two warps of each CTA that have no other part
};

__device__ __forceinline__ bool wait_noabort(uint64_t *bar, uint32_t parity) {
  return tc::mbar_wait(bar, parity, nullptr);
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}

// work item -> (m0, n0, split).  Tiles are taken in bands of kBand tile
// columns, row by row within a band: the CTAs running together (one per
// SM) then read a block of about 19 x 8 tiles, whose A rows and B columns
// (70 MB at K = 8192) stay in L2, instead of every row of A per wave.
constexpr int kBand = 8;
__device__ __forceinline__ void gemm_item(const GemmShape &g, int w, int BN, int &m0, int &n0,
                                          int &split, int bm = GBM) {
  const int tiles = g.tiles_m * g.tiles_n;
  split = w / tiles;
  const int t = w - split * tiles;
  const int band = t / (kBand * g.tiles_m);
  const int nb0 = band * kBand;
  const int gw = min(kBand, g.tiles_n - nb0);
  const int r = t - band * kBand * g.tiles_m;
  const int tm = r / gw;
  m0 = tm * bm;
  n0 = (nb0 + (r - tm * gw)) * BN;
}

// the same for a group: split is the product, whose K blocks are its term's
__device__ __forceinline__ void gemm_item(const GemmGroup &g, int w, int BN, int &m0, int &n0,
                                          int &q) {
  q = 0;
  while (q + 1 < kMaxTerms && w >= g.first[q + 1]) ++q;
  const int t = w - g.first[q], tm = t / g.tiles_n[q];
  m0 = tm * GBM;
  n0 = (t - tm * g.tiles_n[q]) * BN;
}

// One epilogue warp's 32 rows of a tile (load(c0, v): 32 columns of this lane's row) to
// dst [M][N] from (row0, n0) on: 32 x 32 blocks through shared memory, so that
// rows go out as whole 128-byte lines (one row per lane wrote 32 half sectors per
// store).
template <int BN, int UNROLL, class Load>
__device__ __forceinline__ void store_tile(Load load, float *blk, int lane, int row0, int n0,
                                           int M, int N, int vec4, float *__restrict__ dst) {
#pragma unroll UNROLL
  for (int c0 = 0; c0 < BN; c0 += 32) {
    float v[32];
    load(c0, v);
    const int col = n0 + c0;
    if (col >= N) break;   // warp-uniform
#pragma unroll
    for (int q = 0; q < 8; ++q)
      *reinterpret_cast<float4 *>(blk + lane * kOutLd + 4 * q) =
          make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    __syncwarp();
    if (vec4) {   // N % 4 == 0: four columns are inside together
      const int r = lane >> 3, c = (lane & 7) * 4;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int row = row0 + r + 4 * q;
        if (row < M && col + c < N)
          *reinterpret_cast<float4 *>(dst + (size_t)row * N + col + c) =
              *reinterpret_cast<const float4 *>(blk + (r + 4 * q) * kOutLd + c);
      }
    } else {
      for (int r = 0; r < 32; ++r)
        if (row0 + r < M && col + lane < N)
          dst[(size_t)(row0 + r) * N + col + lane] = blk[r * kOutLd + lane];
    }
    __syncwarp();
  }
}

template <bool TF32, int BN, bool GROUP>
__global__ void __launch_bounds__(256, 1) k_gemm_tn(const __grid_constant__ GemmMaps maps,
                                                    const GemmShape g, const GemmGroup gg,
                                                    float *__restrict__ out, int32_t *status) {
  const auto item = [&](int w, int &m0, int &n0, int &split) {
    if constexpr (GROUP)
      gemm_item(gg, w, BN, m0, n0, split);
    else
      gemm_item(g, w, BN, m0, n0, split);
  };
  using C = GCfg<BN>;
  constexpr int NACC = GROUP ? 4 : 2;   // accumulators in tensor memory
  constexpr uint32_t TMEM_COLS = NACC * BN;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = tc::smem_u32(smem_raw);
  uint8_t *base = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  uint8_t *sA = base;
  uint8_t *sB = base + C::STAGES * G_A_BYTES;
  float *s_out = reinterpret_cast<float *>(sB + C::STAGES * C::B_BYTES);
  uint64_t *full = reinterpret_cast<uint64_t *>(s_out + 4 * 32 * kOutLd);
  uint64_t *empty = full + C::STAGES;
  uint64_t *acc_full = empty + C::STAGES;   // [NACC]
  uint64_t *acc_empty = acc_full + NACC;    // [NACC]
  uint64_t *done = acc_empty + NACC;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      tc::mbar_init(full + s, 1);
      tc::mbar_init(empty + s, 1);
    }
    for (int b = 0; b < NACC; ++b) {
      tc::mbar_init(acc_full + b, 1);
      tc::mbar_init(acc_empty + b, 4);   // one arrival per epilogue warp
    }
    tc::mbar_init(done, 1);
    *abort_flag = 0;
    tc::mbar_fence_init();
  }
  if (warp == 1) tc::tmem_alloc(tmem_slot, TMEM_COLS);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();   // barriers and tensor memory are set up under the kernel before
  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;   // stage fills issued (ring position)
      bool ok = true;
      for (int w = blockIdx.x; w < g.n_items && ok; w += gridDim.x) {
        int m0, n0, split;
        item(w, m0, n0, split);
        const int kb0 = split * g.kb_per_split;
        const int nk = min(g.kb_per_split, g.kb_total - kb0);
        for (int i = 0; i < nk; ++i, ++it) {
          const uint32_t s = it % C::STAGES;
          if (it >= (uint32_t)C::STAGES &&
              !tc::mbar_wait(empty + s, ((it / C::STAGES) & 1) ^ 1, abort_flag)) {
            *abort_flag = 1;
            ok = false;
            break;
          }
          const int gk = kb0 + i, term = gk / g.kb_term;
          const int kx = (gk - term * g.kb_term) * gbk<TF32>();
          tc::mbar_arrive_expect_tx(full + s, G_A_BYTES + C::B_BYTES);
          tc::tma_load_2d(sA + s * G_A_BYTES, &maps.a[term], full + s, kx, m0);
          tc::tma_load_2d(sB + s * C::B_BYTES, &maps.b[term], full + s, kx, n0);
        }
      }
      // every issued copy lands before the CTA may leave
      for (uint32_t s = 0; s < (uint32_t)C::STAGES && s < it; ++s) {
        const uint32_t last = s + ((it - 1 - s) / C::STAGES) * C::STAGES;
        wait_noabort(full + s, (last / C::STAGES) & 1);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc =
          TF32 ? tc::idesc_tf32_f32(GBM, BN) : tc::idesc_bf16_f32(GBM, BN);
      uint32_t it = 0;
      int j = 0;   // accumulations of this CTA so far
      bool ok = true;
      for (int w = blockIdx.x; w < g.n_items && ok; w += gridDim.x) {
        int m0, n0, split;
        item(w, m0, n0, split);
        const int nk = min(g.kb_per_split, g.kb_total - split * g.kb_per_split);
        const int per = GROUP ? gg.kb_slice[split] : nk;
        for (int i0 = 0; i0 < nk && ok; i0 += per, ++j) {
          const int buf = j % NACC, n = min(per, nk - i0);
          // the epilogue has drained this accumulator's previous use
          if (j >= NACC && !tc::mbar_wait(acc_empty + buf, (j / NACC - 1) & 1, abort_flag)) {
            *abort_flag = 1;
            ok = false;
            break;
          }
          tc::fence_after();
          const uint32_t d = tmem + (uint32_t)(buf * BN);
          for (int i = 0; i < n; ++i, ++it) {
            const uint32_t s = it % C::STAGES;
            if (!tc::mbar_wait(full + s, (it / C::STAGES) & 1, abort_flag)) {
              *abort_flag = 1;
              ok = false;
              break;
            }
            tc::fence_after();
            const uint64_t ad = tc::desc_sw128(tc::smem_u32(sA + s * G_A_BYTES));
            const uint64_t bd = tc::desc_sw128(tc::smem_u32(sB + s * C::B_BYTES));
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {   // +32 bytes of K per step (16 bf16 or 8 tf32)
              if constexpr (TF32)
                tc::mma_tf32(d, ad + 2 * kk, bd + 2 * kk, idesc, (i | kk) ? 1u : 0u);
              else
                tc::mma_bf16(d, ad + 2 * kk, bd + 2 * kk, idesc, (i | kk) ? 1u : 0u);
            }
            tc::mma_commit(empty + s);
          }
          if (ok) tc::mma_commit(acc_full + buf);
        }
      }
      tc::mma_commit(done);      // arrives once every MMA issued has finished
      wait_noabort(done, 0);     // before the tensor memory is freed
    }
  } else if (warp < 4) {
    if constexpr (GROUP) column_sums(gg.sums, 2 * blockIdx.x + warp - 2, 2 * gridDim.x);
  } else {
    const int wl = warp - 4;   // tensor-memory lanes 32 wl .. 32 wl + 31
    const uint32_t lanes = tmem + ((uint32_t)(wl * 32) << 16);
    float *blk = s_out + wl * 32 * kOutLd;
    int j = 0;
    bool go = true;
    // the next accumulator, once it is finished; released by the lambda below
    const auto finished = [&]() {
      go = tc::mbar_wait(acc_full + j % NACC, (j / NACC) & 1, abort_flag);
      go = __all_sync(0xffffffffu, go);
      if (!go) *abort_flag = 1;
      tc::fence_after();
      return lanes + (uint32_t)(j % NACC * BN);
    };
    const auto release = [&]() {
      tc::fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty + j % NACC);
      ++j;
    };
    for (int w = blockIdx.x; w < g.n_items && go; w += gridDim.x) {
      int m0, n0, split;
      item(w, m0, n0, split);
      const int row0 = m0 + wl * 32;
      if constexpr (GROUP) {
        // the slices' sums, in order, in registers
        float sum[BN];
#pragma unroll
        for (int c = 0; c < BN; ++c) sum[c] = 0.f;
        for (int i0 = 0; i0 < g.kb_per_split; i0 += gg.kb_slice[split]) {
          const uint32_t acc = finished();
          if (!go) break;
#pragma unroll
          for (int c0 = 0; c0 < BN; c0 += 32) {
            float v[32];
            tc::tmem_ld32(acc + (uint32_t)c0, v);
#pragma unroll
            for (int c = 0; c < 32; ++c) sum[c0 + c] += v[c];
          }
          release();
        }
        if (!go) break;
        store_tile<BN, BN / 32>(
            [&](int c0, float (&v)[32]) {
#pragma unroll
              for (int c = 0; c < 32; ++c) v[c] = sum[c0 + c];
            },
            blk, lane, row0, n0, gg.M[split], gg.N[split], g.vec4, gg.out[split]);
      } else {
        const uint32_t acc = finished();
        if (!go) break;
        store_tile<BN, 1>([&](int c0, float (&v)[32]) { tc::tmem_ld32(acc + (uint32_t)c0, v); },
                          blk, lane, row0, n0, g.M, g.N, g.vec4, out + (size_t)split * g.M * g.N);
        release();
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after();
    tc::tmem_dealloc(tmem, TMEM_COLS);
  }
  if (threadIdx.x == 0 && *abort_flag) atomicExch(status, SPECULA_ETIMEOUT);
}

// The same over CTA pairs (cta_group::2): a pair owns 256 x 256 tiles, each CTA
// 128 rows of A, 128 rows of B and 128 rows of the accumulator; one thread of the
// leader issues the MMAs for both.  An SM's port from L2 (64 bytes per clock) was what
// bounded the single-CTA form: 48 KB per 128 x 256 x 64 step, 768 clocks for 512
// of the tensor cores, measured 60 bytes per clock; a pair's CTA takes 32 KB
// for the same step.  4000 x 13344 on 2048 frames in split bf16 (three terms, five
// slices, their sum included): 481 -> 413 us, 1.59 PFLOP/s; on 512 frames one term
// 74 -> 66 us.  Bit-identical.
constexpr int kPairM = 2 * GBM, kPairN = 256, kPairStages = 6;
constexpr uint32_t kPairStage = 2 * G_A_BYTES;   // 128 rows of A and of B
constexpr size_t kPairSmem =
    1024 + kPairStages * kPairStage + 4 * 32 * kOutLd * sizeof(float) + 256;
template <bool TF32>
__global__ void __launch_bounds__(256, 1) k_gemm_pair(const __grid_constant__ GemmMaps maps,
                                                      const GemmShape g, float *__restrict__ out,
                                                      int32_t *status) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = tc::smem_u32(smem_raw);
  uint8_t *base = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  float *s_out = reinterpret_cast<float *>(base + kPairStages * kPairStage);
  uint64_t *full = reinterpret_cast<uint64_t *>(s_out + 4 * 32 * kOutLd);   // the leader's count
  uint64_t *empty = full + kPairStages;
  uint64_t *acc_full = empty + kPairStages;   // [2]
  uint64_t *acc_empty = acc_full + 2;         // [2], the leader's count
  uint64_t *done = acc_empty + 2;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)tc::cluster_rank();
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kPairStages; ++s) {
      tc::mbar_init(full + s, 1);
      tc::mbar_init(empty + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(acc_full + b, 1);
      tc::mbar_init(acc_empty + b, 8);   // the epilogue warps of both CTAs
    }
    tc::mbar_init(done, 1);
    *abort_flag = 0;
    tc::mbar_fence_init();
  }
  if (warp == 1) tc::tmem_alloc_pair(tmem_slot, 2 * kPairN);
  tc::fence_before();
  __syncthreads();
  tc::cluster_sync();   // both CTAs' barriers are initialised
  tc::fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();
  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int w = pair; w < g.n_items && ok; w += pairs) {
        int m0, n0, split;
        gemm_item(g, w, kPairN, m0, n0, split, kPairM);
        const int kb0 = split * g.kb_per_split;
        const int nk = min(g.kb_per_split, g.kb_total - kb0);
        for (int i = 0; i < nk; ++i, ++it) {
          const uint32_t s = it % kPairStages;
          if (it >= (uint32_t)kPairStages &&
              !tc::mbar_wait(empty + s, ((it / kPairStages) & 1) ^ 1, abort_flag)) {
            *abort_flag = 1;
            ok = false;
            break;
          }
          const int gk = kb0 + i, term = gk / g.kb_term;
          const int kx = (gk - term * g.kb_term) * gbk<TF32>();
          if (rank == 0) tc::mbar_arrive_expect_tx(full + s, 2 * kPairStage);
          const uint32_t bar = tc::leader_addr(full + s);
          uint8_t *st = base + s * kPairStage;
          tc::tma_load_2d_pair(st, &maps.a[term], bar, kx, m0 + rank * GBM);
          tc::tma_load_2d_pair(st + G_A_BYTES, &maps.b[term], bar, kx, n0 + rank * GBM);
        }
      }
      // every issued copy has landed and been read before the CTA may leave
      for (uint32_t s = 0; s < (uint32_t)kPairStages && s < it; ++s) {
        const uint32_t last = s + ((it - 1 - s) / kPairStages) * kPairStages;
        wait_noabort(empty + s, (last / kPairStages) & 1);
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc =
          TF32 ? tc::idesc_tf32_f32(kPairM, kPairN) : tc::idesc_bf16_f32(kPairM, kPairN);
      uint32_t it = 0;
      int j = 0;
      bool ok = true;
      for (int w = pair; w < g.n_items && ok; w += pairs, ++j) {
        int m0, n0, split;
        gemm_item(g, w, kPairN, m0, n0, split, kPairM);
        const int nk = min(g.kb_per_split, g.kb_total - split * g.kb_per_split);
        const int buf = j & 1;
        // both CTAs have drained this accumulator's previous tile
        if (j >= 2 && !tc::mbar_wait(acc_empty + buf, ((j >> 1) - 1) & 1, abort_flag)) {
          *abort_flag = 1;
          break;
        }
        tc::fence_after();
        const uint32_t d = tmem + (uint32_t)(buf * kPairN);
        for (int i = 0; i < nk; ++i, ++it) {
          const uint32_t s = it % kPairStages;
          if (!tc::mbar_wait(full + s, (it / kPairStages) & 1, abort_flag)) {
            *abort_flag = 1;
            ok = false;
            break;
          }
          tc::fence_after();
          const uint64_t ad = tc::desc_sw128(tc::smem_u32(base + s * kPairStage));
          const uint64_t bd = tc::desc_sw128(tc::smem_u32(base + s * kPairStage + G_A_BYTES));
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            tc::mma_pair<TF32>(d, ad + 2 * kk, bd + 2 * kk, idesc, (i | kk) ? 1u : 0u);
          tc::mma_commit_pair(empty + s);
        }
        if (ok) tc::mma_commit_pair(acc_full + buf);
      }
      tc::mma_commit_leader(done);   // arrives once every MMA issued has finished
      wait_noabort(done, 0);         // before the tensor memory is freed
    }
  } else if (warp >= 4) {
    const int wl = warp - 4;
    int j = 0;
    for (int w = pair; w < g.n_items; w += pairs, ++j) {
      int m0, n0, split;
      gemm_item(g, w, kPairN, m0, n0, split, kPairM);
      const int buf = j & 1;
      bool go = tc::mbar_wait(acc_full + buf, (j >> 1) & 1, abort_flag);
      go = __all_sync(0xffffffffu, go);
      if (!go) {
        *abort_flag = 1;
        break;
      }
      tc::fence_after();
      const uint32_t acc = tmem + ((uint32_t)(wl * 32) << 16) + (uint32_t)(buf * kPairN);
      store_tile<kPairN, 1>([&](int c0, float (&v)[32]) { tc::tmem_ld32(acc + (uint32_t)c0, v); },
                            s_out + wl * 32 * kOutLd, lane, m0 + rank * GBM + wl * 32, n0, g.M,
                            g.N, g.vec4, out + (size_t)split * g.M * g.N);
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive_cluster(tc::leader_addr(acc_empty + buf));
    }
  }
  __syncwarp();
  tc::fence_before();
  __syncthreads();
  tc::cluster_sync();   // neither CTA's memory is used by the other from here on
  if (warp == 1) {
    tc::fence_after();
    tc::tmem_dealloc_pair(tmem, 2 * kPairN);
  }
  if (threadIdx.x == 0 && *abort_flag) atomicExch(status, SPECULA_ETIMEOUT);
  tc::cluster_sync();
}

// out[e] = sum of part[s][e] over the splits, in order, eight splits' loads in
// flight; V = 4 floats per load where n and the pointers allow and the threads still
// give every SM a CTA (a few partials of 32 x 500: 6.8 us by four floats in 16 CTAs, 4.0 by
// one in 63).
template <int V>
__global__ void __launch_bounds__(256) k_split_reduce(const float *__restrict__ part, int splits,
                                                      size_t n, float *__restrict__ out) {
  pdl_wait();
  const size_t nv = n / V;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nv;
       e += (size_t)gridDim.x * blockDim.x) {
    float v[V];
#pragma unroll
    for (int q = 0; q < V; ++q) v[q] = 0.f;
#pragma unroll 8
    for (int s = 0; s < splits; ++s) {
      if constexpr (V == 4) {
        const float4 x = __ldcs(reinterpret_cast<const float4 *>(part + (size_t)s * n) + e);
        v[0] += x.x;
        v[1] += x.y;
        v[2] += x.z;
        v[3] += x.w;
      } else {
        v[0] += part[(size_t)s * n + e];
      }
    }
    if constexpr (V == 4)
      reinterpret_cast<float4 *>(out)[e] = make_float4(v[0], v[1], v[2], v[3]);
    else
      out[e] = v[0];
  }
}

// ---- host --------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static std::mutex mu;
  static EncodeTiledFn fn = nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// rows x K row-major (bf16, or float32 read as tf32), box of 128 bytes of K
// x box_rows, 128-byte swizzle
static int make_map(CUtensorMap *m, const void *ptr, int rows, int K, int box_rows,
                    bool tf32 = false) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return SPECULA_ECUDA;
  const int es_bytes = tf32 ? 4 : 2;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)K * es_bytes};
  cuuint32_t box[2] = {(cuuint32_t)(128 / es_bytes), (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  CUresult r = fn(m, tf32 ? CU_TENSOR_MAP_DATA_TYPE_TFLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                  const_cast<void *>(ptr), dims, strides,
                  box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? SPECULA_OK : SPECULA_ECUDA;
}

int gemm_check(const void *A, const void *B, int M, int N, int K, bool tf32) {
  if (!A || !B || M < 1 || N < 1 || K < 1) return SPECULA_EINVAL;
  if (K % (tf32 ? 4 : 8)) return SPECULA_EUNSUPPORTED;   // rows of a multiple of 16 bytes (TMA)
  if ((uintptr_t)A % 16 || (uintptr_t)B % 16) return SPECULA_EINVAL;
  return SPECULA_OK;
}

// splits that keep every K slice of kb blocks non-empty
static int splits_for(int kb, int want) {
  int s = std::max(1, std::min(want, kb));
  const int per = (kb + s - 1) / s;
  return (kb + per - 1) / per;
}

int gemm_splits(int K, int want, bool tf32) {
  const int k = tf32 ? gbk<true>() : gbk<false>();
  return splits_for((K + k - 1) / k, want);
}

// output tile width: 128 where N is a multiple of 128 but not of 256 (no
// zero columns computed), else 256
static int gemm_bn(int N) { return (N % 128 == 0 && N % 256 != 0) ? 128 : 256; }

static int sm_count() {
  static int sms[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (dev >= 64) return 0;
  if (!sms[dev] && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev))
    return 0;
  return sms[dev];
}

static int gemm_split_reduce(specula_ctx *ctx, const float *part, int splits, size_t n, float *C,
                             cudaStream_t st) {
  const bool v4 = n % 4 == 0 && (((uintptr_t)part | (uintptr_t)C) % 16) == 0 &&
                  n / 4 >= (size_t)256 * sm_count();
  const size_t threads = v4 ? n / 4 : n;
  const unsigned grid = (unsigned)std::min<size_t>((threads + 255) / 256, 8192);
  if (v4)
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_GEMM, st, k_split_reduce<4>, grid, 256, 0, part, splits, n,
                       C);
  else
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_GEMM, st, k_split_reduce<1>, grid, 256, 0, part, splits, n,
                       C);
  return SPECULA_OK;
}

// Whether a product runs on CTA pairs: K long enough that loading bounds it (4096 x
// 4096 at 16 K blocks takes 37.5 us either way), no more than an eighth of the rows
// padding, and the pairs' waves shorter in all.  A K block of a tile takes 512
// clocks on a pair and 768 on a single CTA (k_gemm_pair), so a second wave with few tiles
// in it costs more than the pairs give: 1152 x 4096 is 144 tiles, one wave of single
// CTAs, or 80 pair tiles, two waves of 76 (K = 4096: 26.1 against 45.3 us); 2048 x 4000
// at 209 blocks takes 139 us on pairs against 169.
static bool gemm_pairs(int M, int tiles_n, int splits, int kb_per_split, int sms) {
  const int tiles_m = (M + GBM - 1) / GBM;
  const long long cols = (long long)tiles_n * splits;
  const auto waves = [](long long items, int slots) { return (items + slots - 1) / slots; };
  return sms >= 2 && (tiles_m % 2 == 0 || tiles_m >= 8) && kb_per_split >= 16 &&
         512 * waves((tiles_m + 1) / 2 * cols, sms / 2) < 768 * waves(tiles_m * cols, sms);
}

template <bool TF32, int BN>
static int gemm_launch(specula_ctx *ctx, int n_terms, const void *const *A, const void *const *B,
                       int M, int N, int K, float *C, int splits, float *work,
                       cudaStream_t st, bool partials) {
  using Cfg = GCfg<BN>;
  int s;
  const int sms = sm_count();
  if (sms < 1) return SPECULA_ECUDA;
  GemmShape g;
  g.M = M;
  g.N = N;
  g.kb_term = (K + gbk<TF32>() - 1) / gbk<TF32>();
  g.kb_total = g.kb_term * n_terms;
  g.splits = splits_for(g.kb_total, splits);
  g.kb_per_split = (g.kb_total + g.splits - 1) / g.splits;
  g.tiles_n = (N + BN - 1) / BN;
  const bool pairs =
      BN == kPairN && gemm_pairs(M, g.tiles_n, g.splits, g.kb_per_split, sms);
  const int bm = pairs ? kPairM : GBM;
  g.tiles_m = (M + bm - 1) / bm;
  g.n_items = g.tiles_m * g.tiles_n * g.splits;
  const bool to_work = partials || g.splits > 1;
  if (to_work && !work) return SPECULA_EINVAL;
  if (partials && g.splits != splits) return SPECULA_EINVAL;
  float *dst = to_work ? work : C;
  g.vec4 = (N % 4 == 0) && ((uintptr_t)dst % 16 == 0);
  GemmMaps maps;
  memset(&maps, 0, sizeof(maps));
  for (int t = 0; t < n_terms; ++t) {
    if ((s = make_map(&maps.a[t], A[t], M, K, GBM, TF32))) return s;
    if ((s = make_map(&maps.b[t], B[t], N, K, pairs ? GBM : BN, TF32))) return s;
  }
  const void *fn = pairs ? (const void *)k_gemm_pair<TF32> : (const void *)k_gemm_tn<TF32, BN, false>;
  if ((s = ensure_dynamic_smem(fn, pairs ? kPairSmem : Cfg::SMEM))) return s;
  const int grid = std::min(g.n_items, sms);
  if (pairs)
    SPECULA_LAUNCH(ctx, SPECULA_K_GEMM, st,
                   SPECULA_CK(launch_pdl(k_gemm_pair<TF32>, 2 * std::min(g.n_items, sms / 2), 256,
                                         kPairSmem, st, 2, maps, g, dst, ctx->status_dev)));
  else
    SPECULA_LAUNCH_PDL(ctx, SPECULA_K_GEMM, st, (k_gemm_tn<TF32, BN, false>), grid, 256, Cfg::SMEM,
                     maps, g, GemmGroup{}, dst, ctx->status_dev);
  if (g.splits > 1 && !partials)
    return gemm_split_reduce(ctx, work, g.splits, (size_t)M * N, C, st);
  return SPECULA_OK;
}

template <bool TF32>
static int gemm_terms(specula_ctx *ctx, int n_terms, const void *const *A, const void *const *B,
                      int M, int N, int K, float *C, int splits, float *work, cudaStream_t st,
                      bool partials = false) {
  if (!ctx || (!C && !partials) || n_terms < 1 || n_terms > kMaxTerms || splits < 1)
    return SPECULA_EINVAL;
  for (int t = 0; t < n_terms; ++t) {
    const int s = gemm_check(A[t], B[t], M, N, K, TF32);
    if (s) return s;
  }
  if (gemm_bn(N) == 128)
    return gemm_launch<TF32, 128>(ctx, n_terms, A, B, M, N, K, C, splits, work, st, partials);
  return gemm_launch<TF32, 256>(ctx, n_terms, A, B, M, N, K, C, splits, work, st, partials);
}

int gemm_bf16_tn(specula_ctx *ctx, const void *A, const void *B, int M, int N, int K, float *C,
                 int splits, float *work, cudaStream_t st) {
  return gemm_terms<false>(ctx, 1, &A, &B, M, N, K, C, splits, work, st);
}

int gemm_bf16_partials(specula_ctx *ctx, const void *A, const void *B, int M, int N, int K,
                       int splits, float *work, cudaStream_t st) {
  return gemm_terms<false>(ctx, 1, &A, &B, M, N, K, nullptr, splits, work, st, true);
}

int gemm_bf16_group(specula_ctx *ctx, int n, const void *const *A, const void *const *B,
                    const int *M, const int *N, int K, const int *splits, float *const *C,
                    const ColSums &cs, cudaStream_t st) {
  constexpr int BN = 128;
  if (!ctx || n < 1 || n > kMaxTerms) return SPECULA_EINVAL;
  GemmMaps maps;
  memset(&maps, 0, sizeof(maps));
  GemmShape g{};
  GemmGroup gg{};
  gg.sums = cs;
  int s;
  if ((s = ensure_dynamic_smem((const void *)k_gemm_tn<false, BN, true>, GCfg<BN>::SMEM))) return s;
  const int sms = sm_count();
  if (sms < 1) return SPECULA_ECUDA;
  g.kb_term = g.kb_per_split = (K + gbk<false>() - 1) / gbk<false>();
  g.kb_total = g.kb_term * n;
  g.vec4 = 1;
  for (int q = 0; q < kMaxTerms; ++q) {
    gg.first[q + 1] = gg.first[q];
    if (q >= n) continue;
    if ((s = gemm_check(A[q], B[q], M[q], N[q], K, false))) return s;
    if ((s = make_map(&maps.a[q], A[q], M[q], K, GBM))) return s;
    if ((s = make_map(&maps.b[q], B[q], N[q], K, BN))) return s;
    gg.M[q] = M[q];
    gg.N[q] = N[q];
    gg.out[q] = C[q];
    gg.kb_slice[q] = (g.kb_term + splits[q] - 1) / splits[q];
    gg.tiles_n[q] = (N[q] + BN - 1) / BN;
    gg.first[q + 1] += (M[q] + GBM - 1) / GBM * gg.tiles_n[q];
    if (N[q] % 4 || (uintptr_t)C[q] % 16) g.vec4 = 0;
  }
  g.n_items = gg.first[kMaxTerms];
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_GEMM, st, (k_gemm_tn<false, BN, true>),
                     std::min(g.n_items, sms), 256, GCfg<BN>::SMEM, maps, g, gg, (float *)nullptr,
                     ctx->status_dev);
  return SPECULA_OK;
}

int gemm_bf16_terms(specula_ctx *ctx, int n_terms, const void *const *A, const void *const *B,
                    int M, int N, int K, float *C, int splits, float *work, cudaStream_t st) {
  return gemm_terms<false>(ctx, n_terms, A, B, M, N, K, C, splits, work, st);
}

int gemm_tf32_tn(specula_ctx *ctx, const float *A, const float *B, int M, int N, int K, float *C,
                 int splits, float *work, cudaStream_t st) {
  const void *a = A, *b = B;
  return gemm_terms<true>(ctx, 1, &a, &b, M, N, K, C, splits, work, st);
}

}  // namespace specula

using namespace specula;

extern "C" int specula_gemm_bf16(specula_ctx *ctx, const void *A_dev, const void *B_dev,
                                 int32_t M, int32_t N, int32_t K, float *C_dev, int32_t splits,
                                 float *work_dev, void *stream) {
  if (!ctx || !C_dev || splits < 1) return SPECULA_EINVAL;
  return gemm_bf16_tn(ctx, A_dev, B_dev, M, N, K, C_dev, splits, work_dev,
                      (cudaStream_t)stream);
}

extern "C" int specula_gemm_tf32(specula_ctx *ctx, const float *A_dev, const float *B_dev,
                                 int32_t M, int32_t N, int32_t K, float *C_dev, int32_t splits,
                                 float *work_dev, void *stream) {
  if (!ctx || !C_dev || splits < 1) return SPECULA_EINVAL;
  return gemm_tf32_tn(ctx, A_dev, B_dev, M, N, K, C_dev, splits, work_dev,
                      (cudaStream_t)stream);
}

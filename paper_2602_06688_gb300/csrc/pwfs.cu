// Modulated pyramid wavefront sensor image (ModulatedPyramid + CCD binning,
// App. A, Tab. 4; parameters of App. B, Listing 2).
//
// Per modulation point m the sensor computes, on the N x N padded grid
// (N = 2 n_pix), I_m = |IDFT2( M . DFT2( pad(E . tilt_m) ) )|^2 with centred
// transforms.  The centred forward transform is an unshifted FFT between an
// input phase p(n) = exp(i pi (N-1) n / N) and an output phase; the output
// phase cancels against the input phase of the centred inverse, whose own
// output phase disappears in |.|^2.  So the GPU evaluates
//     I_m = |IFFT2( M . FFT2( pad(E . tilt_m . p_x p_y) ) )|^2 / N^4,
// with tilt_m . p folded into per-axis tables gx[m][i], gy[m][j] and the
// 1/N^2 folded into the per-axis mask tables.
//
// Pipeline, one chunk of K (batch element, modulation point) items at a time
// so that the intermediates stay L2-resident:
//   F  k_field          E = amp exp(i phase) once per batch element
//   A  k_rows_fwd       E . gx . gy, row FFT of the n_pix non-zero rows
//                       (input half zero: pruned)              -> rows ws
//   B  k_cols           per column tile (staged with cp.async): column FFT
//                       (pruned) -> mask -> inverse column FFT  -> cols ws
//   C  k_rows_inv_part  per (bin strip, item): row inverse FFT -> |.|^2 /
//                       n_mod -> b x b bins              -> part[b][m] ws
//   D  k_bin_reduce     once a batch element's n_mod items are done: the
//                       detector = sum over m in order (no atomics:
//                       bit-reproducible)
//
// Each N-point transform is a two-level split N = N1 x N2 evaluated by one
// group of G lanes: step 1, lane n1 < N1 holds x[n1 + N1 n2] (n2 < N2) and
// does an N2-point register DFT, multiplies by W_N^{n1 k2}; the values are
// exchanged through shared memory; step 2, lane k2 < N2 does an N1-point
// register DFT and holds X[N2 k1 + k2].  With N2 % 4 == 0 the non-zero half
// of a zero-padded input (indices N/4 .. 3N/4) is exactly registers
// N2/4 .. 3N2/4 of every lane, so zero inputs are never loaded.  The
// inter-step twiddles are read through the read-only cache: lane n1 reads
// table[k2][n1], so a warp's reads are consecutive for each k2.
#include <math.h>

#include <algorithm>

#include "fft_regs.cuh"
#include "internal.h"
#include "pwfs_common.cuh"

namespace specula {

int pwfs_init_device() {
  return upload_codelet_twiddles() == cudaSuccess ? SPECULA_OK : SPECULA_ECUDA;
}

__device__ __forceinline__ void cp_async8(void *smem_dst, const void *gsrc) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}
// a read-only load that does not allocate in L1 (data read once per CTA)
__device__ __forceinline__ float2 ld_stream2(const float2 *p) {
  float2 v;
  asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}

// --------------------------------------------------------------------------
// F: field of the batch elements b0 .. b0 + gridDim.y - 1 into slots b % nbw.
__global__ void __launch_bounds__(256) k_field(const float *__restrict__ amp,
                                               const float *__restrict__ phase,
                                               float2 *__restrict__ field, int npix2, int b0,
                                               int nbw, float phase_scale) {
  pdl_wait();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= npix2) return;
  const int b = b0 + blockIdx.y;
  float sv, cv;
  sincosf(phase[(size_t)b * npix2 + e] * phase_scale, &sv, &cv);
  const float a = amp[e];
  field[(size_t)(b % nbw) * npix2 + e] = make_float2(a * cv, a * sv);
}

// --------------------------------------------------------------------------
// A: E . gx . gy and the row FFT of the non-zero rows.
// grid (ceil(n_pix / VPC), ceil(n_items / ka)); block VPC * G threads.
template <int N1, int N2>
__global__ void __launch_bounds__(256, 2) k_rows_fwd(
    const float2 *__restrict__ field, const float2 *__restrict__ gx,
    const float2 *__restrict__ gy, const float2 *__restrict__ twA, float2 *__restrict__ rows_out,
    int n_pix, int n_mod, int nbw, int item0, int n_items, int ka) {
  using S = Split<N1, N2>;
  constexpr int N = S::N, G = S::G, S1 = S::S1;
  constexpr int Q0 = N2 / 4, QH = N2 / 2;
  extern __shared__ float2 smem[];
  const int vpc = blockDim.x / G;
  const int vec = threadIdx.x / G, lane = threadIdx.x % G;
  float2 *xb = smem + vec * S::XB;
  const int j = blockIdx.x * vpc + vec;
  const bool row_ok = j < n_pix;
  const bool in_lane = row_ok && lane < N1;

  float2 e[QH];
  int cur_b = -1;
  const int it_begin = blockIdx.y * ka;
  for (int q = 0; q < ka; ++q) {
    const int it = it_begin + q;
    if (it >= n_items) break;
    const int gi = item0 + it;
    const int b = gi / n_mod, m = gi - b * n_mod;
    if (b != cur_b) {
      cur_b = b;
      const float2 *src = field + ((size_t)(b % nbw) * n_pix + (row_ok ? j : 0)) * n_pix + lane;
#pragma unroll
      for (int h = 0; h < QH; ++h) e[h] = in_lane ? src[N1 * h] : make_float2(0.f, 0.f);
    }
    float2 r[N2];
    const float2 gyv = row_ok ? gy[(size_t)m * n_pix + j] : make_float2(0.f, 0.f);
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) r[n2] = make_float2(0.f, 0.f);
    if (in_lane) {
      const float2 *g = gx + (size_t)m * n_pix + lane;
#pragma unroll
      for (int h = 0; h < QH; ++h) r[Q0 + h] = cmul(cmul(e[h], __ldg(g + N1 * h)), gyv);
    }
    RegDFT<N2, false>::run(r);
    __syncwarp();
    if (lane < N1) {
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2)
        xb[k2 * S1 + lane] = cmulc(r[k2], __ldg(twA + k2 * N1 + lane));
    }
    __syncwarp();
    if (lane < N2) {
      float2 r2[N1];
#pragma unroll
      for (int n1 = 0; n1 < N1; ++n1) r2[n1] = xb[lane * S1 + n1];
      RegDFT<N1, false>::run(r2);
      if (row_ok) {
        float2 *dst = rows_out + ((size_t)it * n_pix + j) * N + lane;
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) dst[N2 * k1] = r2[k1];
      }
    }
  }
}

// --------------------------------------------------------------------------
// B: per tile of TC columns: column FFT (rows n_pix non-zero) -> pyramid
// mask -> inverse column FFT, in a column-major shared tile whose column
// stride CS = 2 (mod 16) complex keeps the row-wise staging conflict-free.
// grid (N / TC, n_items); block TC * G threads.
template <int N1, int N2, int TC>
struct ColsCfg {
  using S = Split<N1, N2>;
  static constexpr int CS = round_cs(imax3(S::N, N2 * S::S1, N1 * S::S2));
  static constexpr size_t smem = (size_t)(TC * CS) * sizeof(float2);
};

template <int N1, int N2, int TC>
__global__ void __launch_bounds__(256, 3) k_cols(
    const float2 *__restrict__ rows_in, float2 *__restrict__ cols_out,
    const float2 *__restrict__ twA, const float2 *__restrict__ twB,
    const float2 *__restrict__ mask, int n_pix) {
  using S = Split<N1, N2>;
  constexpr int N = S::N, G = S::G, S1 = S::S1, S2 = S::S2;
  constexpr int CS = ColsCfg<N1, N2, TC>::CS;
  constexpr int Q0 = N2 / 4, QH = N2 / 2;
  extern __shared__ float2 smem[];
  float2 *s_tile = smem;
  const int it = blockIdx.y;
  const int col0 = blockIdx.x * TC;
  constexpr int off = N / 4;
  // all staging loads in flight at once (asynchronous copies into the tile)
  const float2 *src = rows_in + (size_t)it * n_pix * N + col0;
  for (int e = threadIdx.x; e < n_pix * TC; e += blockDim.x) {
    const int c = e % TC, jj = e / TC;
    cp_async8(s_tile + c * CS + off + jj, src + (size_t)jj * N + c);
  }
  const int vec = threadIdx.x / G, lane = threadIdx.x % G;
  const float2 mk = __ldg(mask + col0 + vec);
  cp_async_wait_all();
  __syncthreads();

  float2 *col = s_tile + vec * CS;

  // forward, standard split; non-zero input rows are registers Q0..Q0+QH-1
  float2 r[N2];
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) r[n2] = make_float2(0.f, 0.f);
  if (lane < N1) {
#pragma unroll
    for (int h = 0; h < QH; ++h) r[Q0 + h] = col[lane + N1 * (Q0 + h)];
  }
  RegDFT<N2, false>::run(r);
  __syncwarp();
  if (lane < N1) {
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2)
      col[k2 * S1 + lane] = cmulc(r[k2], __ldg(twA + k2 * N1 + lane));
  }
  __syncwarp();
  float2 r2[N1];
  if (lane < N2) {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) r2[n1] = col[lane * S1 + n1];
  } else {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) r2[n1] = make_float2(0.f, 0.f);
  }
  RegDFT<N1, false>::run(r2);
  // lane k2 holds F[v = N2 k1 + k2] of column k = col0 + vec
  if (lane < N2) {
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1)
      r2[k1] = cmul(r2[k1], cmul(__ldg(mask + N2 * k1 + lane), mk));
  }
  // inverse, swapped split: lane n1' = k2 (< N2), registers n2' = k1 (< N1)
  RegDFT<N1, true>::run(r2);
  __syncwarp();
  if (lane < N2) {
#pragma unroll
    for (int k2 = 0; k2 < N1; ++k2)
      col[k2 * S2 + lane] = cmul(r2[k2], __ldg(twB + k2 * N2 + lane));
  }
  __syncwarp();
  float2 r3[N2];
  if (lane < N1) {
#pragma unroll
    for (int n1 = 0; n1 < N2; ++n1) r3[n1] = col[lane * S2 + n1];
  } else {
#pragma unroll
    for (int n1 = 0; n1 < N2; ++n1) r3[n1] = make_float2(0.f, 0.f);
  }
  RegDFT<N2, true>::run(r3);
  __syncwarp();
  if (lane < N1) {
#pragma unroll
    for (int k1 = 0; k1 < N2; ++k1) col[N1 * k1 + lane] = r3[k1];   // y = N1 k1' + k2'
  }
  __syncthreads();
  float2 *dst = cols_out + (size_t)it * N * N + col0;
  for (int e = threadIdx.x; e < N * TC; e += blockDim.x) {
    const int c = e % TC, y = e / TC;
    dst[(size_t)y * N + c] = s_tile[c * CS + y];
  }
}

// --------------------------------------------------------------------------
// C: per (bin strip, item): row inverse FFTs, |.|^2 scaled by 1/n_mod, and
// the b x b bins of the strip into part[b % nbw][m].  Each warp's intensity
// row reuses its own exchange buffer.  grid (N / bsz, n_items);
// block round32(bsz G).
template <int N1, int N2>
__global__ void __launch_bounds__(256, 2) k_rows_inv_part(
    const float2 *__restrict__ cols_in, const float2 *__restrict__ twA, float *__restrict__ part,
    int bsz, float scale, int n_mod, int nbw, int item0) {
  using S = Split<N1, N2>;
  constexpr int N = S::N, G = S::G, S1 = S::S1;
  extern __shared__ float2 smem[];
  const int vec = threadIdx.x / G, lane = threadIdx.x % G;
  const bool act = vec < bsz;
  const int it = blockIdx.y;
  const int y = blockIdx.x * bsz + (act ? vec : 0);
  float2 *xb = smem + vec * S::XB;
  float2 r[N2];
  if (act && lane < N1) {
    const float2 *src = cols_in + ((size_t)it * N + y) * N + lane;
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) r[n2] = src[N1 * n2];
  } else {
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) r[n2] = make_float2(0.f, 0.f);
  }
  RegDFT<N2, true>::run(r);
  if (lane < N1) {
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) xb[k2 * S1 + lane] = cmul(r[k2], __ldg(twA + k2 * N1 + lane));
  }
  __syncwarp();
  float2 r2[N1];
  if (lane < N2) {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) r2[n1] = xb[lane * S1 + n1];
  }
  __syncwarp();
  float *s_row = reinterpret_cast<float *>(xb);   // this warp's intensity row
  if (act && lane < N2) {
    RegDFT<N1, true>::run(r2);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1)
      s_row[N2 * k1 + lane] = (r2[k1].x * r2[k1].x + r2[k1].y * r2[k1].y) * scale;
  }
  __syncthreads();
  const int nd = N / bsz;
  const int gi = item0 + it;
  const int b = gi / n_mod, m = gi - b * n_mod;
  float *dst = part + (((size_t)(b % nbw) * n_mod + m) * nd + blockIdx.x) * nd;
  const float *s_I = reinterpret_cast<const float *>(smem);
  constexpr int RS = 2 * S::XB;   // row stride of the intensity rows (floats)
  for (int q = threadIdx.x; q < nd; q += blockDim.x) {
    float v = 0.f;
    for (int rr = 0; rr < bsz; ++rr)
      for (int xx = 0; xx < bsz; ++xx) v += s_I[rr * RS + q * bsz + xx];
    dst[q] = v;
  }
}

// --------------------------------------------------------------------------
// Two-pass form.  The pyramid mask is separable, M(u, v) = Mx(u) My(v), and
// so is the centred 2D transform, hence
//     IDFT2(M . DFT2(P)) = (IDFT_y My DFT_y) (IDFT_x Mx DFT_x) P :
// the x filter acts on each row alone and the y filter on each column alone.
// Pass R filters the n_pix non-zero rows of every item (forward row FFT of
// the pruned input, x mask, inverse row FFT); pass K filters every column
// (forward FFT of its n_pix non-zero entries, y mask, inverse FFT), squares,
// scales by 1/n_mod and bins, so the N x N intermediate of the three-pass
// form is never written.  Between the two, a slot's filtered rows are held
// column-major ([slot][x][row]): pass R transposes its rows on the way out,
// and pass K reads each column as one contiguous run, coalesced, straight
// into registers.  The inverse row transform's output phase depends
// on x only and vanishes in |.|^2.

// How a CTA's threads share its transforms.
// Splits with N1 <= 32: a warp runs P = 32 / N1 transforms side by side: in
// the outer stages lane (p, n1) = (lane / N1, lane % N1) holds N2 values of
// transform p, in the middle stage lane (c, k2) = (lane / N2, lane % N2) holds
// N1 values of transform PB i + c, i = 0 .. IT-1.  So 320 = 10 x 32 keeps 30 of
// 32 lanes busy in the outer stages and all in the middle one (as 20 x 16 with
// a warp per transform: 20 and 16), 128 = 8 x 16 all.
// Square splits with N1 = N2 > 32 (1600 = 40 x 40): thread t holds values t % N1
// of transform t / N1 in every stage, four transforms on five warps, and the
// stages are separated by CTA barriers instead of warp ones.  40 values per
// thread leave 15 warps per SM; as 32 x 50, a warp per transform, the 50-point
// transforms took 220 registers (8 warps) and the middle stage two lane strides
// of 50 / 64.
// XS: stride (complex) of the exchange buffers; where a warp holds lanes of
// several transforms XS = N1 (mod 16) puts the lanes of an outer stage on
// consecutive banks, else it is odd.
template <int N1, int N2> struct Pack {
  static constexpr int N = N1 * N2;
  static constexpr bool CTA = N1 > 32;
  static constexpr int S1 = N1 | 1, S2 = N2 | 1;   // exchange strides (odd: no conflicts)
  static constexpr int P = CTA ? 1 : 32 / N1;
  static constexpr int PB = CTA ? 1 : 32 / N2;
  static constexpr int IT = (P + PB - 1) / PB;
  static constexpr bool FULL = PB * N2 == 32 && IT * PB == P;   // no idle lane in the middle
  static constexpr int base = imax3(N, N2 * S1, N1 * S2);
  static constexpr bool MANY = CTA || P > 1;
  static constexpr int XS = MANY ? base + ((N1 - base) % 16 + 16) % 16 : (base | 1);
  // the row pass: a one-transform warp's buffer stays even (16-byte loads)
  static constexpr int XSR = MANY ? XS : base;
  static_assert(N2 <= 32 || (CTA && N1 == N2), "wide splits are square");
  // transforms of a CTA of `threads`
  static __host__ __device__ constexpr int vecs(int threads) {
    return CTA ? threads / N1 : threads / 32 * P;
  }
  static __device__ __forceinline__ void sync() {
    if constexpr (CTA) __syncthreads();
    else __syncwarp();
  }
};

// Middle stage of the CTA's transforms (buffers at sm, sm + STRIDE, ...):
// N1-point DFT, mask, inverse, twiddle of the swapped split, in place.
template <int N1, int N2, int STRIDE>
__device__ __forceinline__ void packed_mid(float2 *sm, const float2 *__restrict__ mask,
                                           const float2 *__restrict__ twB) {
  using K = Pack<N1, N2>;
  const int lane = threadIdx.x % 32, k2 = K::CTA ? threadIdx.x % N2 : lane % N2;
#pragma unroll
  for (int i = 0; i < K::IT; ++i) {
    const int c = i * K::PB + lane / N2;   // transform of the warp
    const bool act = K::CTA || K::FULL || (lane < K::PB * N2 && c < K::P);
    // idle lanes repeat another's work
    float2 *xb = sm + (K::CTA ? threadIdx.x / N2
                              : threadIdx.x / 32 * K::P + min(c, K::P - 1)) * STRIDE;
    float2 r2[N1];
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) r2[n1] = xb[k2 * K::S1 + n1];
    RegDFT<N1, false>::run(r2);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) r2[k1] = cmul(r2[k1], __ldg(mask + N2 * k1 + k2));
    RegDFT<N1, true>::run(r2);
    K::sync();
    if (act) {
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1)
        xb[k1 * K::S2 + k2] = cmul(r2[k1], __ldg(twB + k1 * N2 + k2));
    }
  }
}

// Points m and n_mod - m share cos(theta), hence the x factor of the tilt;
// their y factors are constant along a row and commute with the row filter.
// So the row filter runs once per distinct cosine ("slot" c = 0 .. nc-1,
// representative m = c) without the y factor, and the column pass applies
// each item's own y factor gy[m][row] to its input.
// R: grid (ceil(n_pix / (warps P)), ceil(n_slots / ka)); writes rows_out[slot][x][row].
// PAD: the padding N / n_pix.  The pupil sits at padded offset PadRegs::OFF,
// so only registers LO .. HI of a lane can be non-zero: the others are neither
// loaded nor added (RegDFTZ).  With pad 2 and N2 % 4 == 0 the pupil is exactly
// registers N2/4 .. 3 N2/4 of every lane; otherwise each lane checks its first
// and last ones.
// Splits with up to 32 values per lane run four warps per CTA, five CTAs per
// SM at 96 registers (4 P rows per CTA: the transposed output goes out as
// whole 32-byte sectors), and reload the field row for every slot (caching it
// across slots needs 32 more registers: spills at that bound); smaller
// ones (N2 <= 16) run 256 threads, two CTAs per SM, with the cached row; 40-value
// threads 160 (four transforms), three CTAs per SM.
template <int N1, int N2, int PAD> struct PadRegs {
  static constexpr int N = N1 * N2, NP = N / PAD, OFF = (N - NP) / 2;
  static constexpr int LO = OFF / N1, HI = (OFF + NP - 1) / N1 + 1;
  static constexpr bool ALIGNED = OFF % N1 == 0 && NP % N1 == 0;
  static constexpr nzmask NZ = nz_range(LO, HI);
  static_assert(N % PAD == 0, "whole pupil side");
};

template <int N1, int N2> struct RowFiltLaunch {
  static constexpr int threads = N2 > 32 ? 4 * N1 : (N2 > 16 ? 128 : 256);
  static constexpr int min_blocks = N2 > 32 ? 3 : (N2 > 16 ? 5 : 2);
  static constexpr bool reload = N2 > 16;
};
template <int N1, int N2, int PAD>
__global__ void __launch_bounds__(RowFiltLaunch<N1, N2>::threads,
                                  RowFiltLaunch<N1, N2>::min_blocks) k_rowfilt(
    const float2 *__restrict__ field, const float2 *__restrict__ gx,
    const float2 *__restrict__ twA, const float2 *__restrict__ twB,
    const float2 *__restrict__ mask, float2 *__restrict__ rows_out, int n_pix, int nc, int nbw,
    int slot0, int n_slots, int ka, int s0) {
  pdl_wait();
  using P = PadRegs<N1, N2, PAD>;
  using K = Pack<N1, N2>;
  constexpr int N = K::N, S1 = K::S1, S2 = K::S2;
  constexpr int LO = P::LO, NR = P::HI - P::LO;
  extern __shared__ __align__(16) float2 smem[];
  const int vpc = K::vecs(blockDim.x);   // rows per CTA
  const int wlane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int lane = K::CTA ? threadIdx.x % N1 : wlane % N1;
  const bool outer = K::CTA || wlane / N1 < K::P;   // this lane takes part in the outer stages
  const int vec = K::CTA ? threadIdx.x / N1 : warp * K::P + (outer ? wlane / N1 : 0);
  constexpr int XBF = K::XSR;
  float2 *xb = smem + vec * XBF;
  // where vector v's output row sits in its buffer: 4 v complex in, as far
  // as the buffer's slack allows, and even, so that with an even XBF two
  // adjacent columns of a row are one aligned 16-byte load
  auto row_tile_off = [](int v) { return min(4 * v, (XBF - N) & ~1); };
  // lanes that take no part and rows past the pupil repeat valid ones; their
  // values are not stored
  const int j = min(blockIdx.x * vpc + vec, n_pix - 1);
  // the pupil column of register LO + h is lane + N1 (LO + h) - OFF
  const auto in_pupil = [&](int h) {
    const int i = lane + N1 * (LO + h) - P::OFF;
    return P::ALIGNED || ((h > 0 || i >= 0) && (h < NR - 1 || i < n_pix));
  };
  constexpr bool kReload = RowFiltLaunch<N1, N2>::reload || !P::ALIGNED;
  float2 e[kReload ? 1 : NR];
  int cur_b = -1;
  const int it_begin = blockIdx.y * ka;
  for (int q = 0; q < ka; ++q) {
    const int it = it_begin + q;
    if (it >= n_slots) break;
    const int gi = slot0 + it;
    const int b = gi / nc, c = s0 + (gi - b * nc);   // nc slots per element from s0
    const float2 *src = field + ((size_t)(b % nbw) * n_pix + j) * n_pix +
                        (lane + N1 * LO - P::OFF);
    if constexpr (!kReload) {
      if (b != cur_b) {
        cur_b = b;
#pragma unroll
        for (int h = 0; h < NR; ++h) e[h] = src[N1 * h];
      }
    }
    // forward row transform, pruned input (standard split)
    float2 r[N2];
    {
      const float2 *g = gx + (size_t)c * n_pix + (lane + N1 * LO - P::OFF);
      float2 f[NR];
#pragma unroll
      for (int h = 0; h < NR; ++h) {
        if constexpr (kReload)
          f[h] = in_pupil(h) ? src[N1 * h] : make_float2(0.f, 0.f);
        else
          f[h] = e[h];
      }
#pragma unroll
      for (int h = 0; h < NR; ++h)
        r[LO + h] = in_pupil(h) ? cmul(f[h], __ldg(g + N1 * h)) : make_float2(0.f, 0.f);
    }
    RegDFTZ<N2, false, P::NZ>::run(r);
    K::sync();
    if (outer) {
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) xb[k2 * S1 + lane] = cmulc(r[k2], __ldg(twA + k2 * N1 + lane));
    }
    K::sync();
    // the x mask between the forward and the inverse transform (swapped split)
    packed_mid<N1, N2, XBF>(smem, mask, twB);
    K::sync();
    float2 r3[N2];
#pragma unroll
    for (int n1 = 0; n1 < N2; ++n1) r3[n1] = xb[lane * S2 + n1];
    RegDFT<N2, true>::run(r3);
    // The slot's block is column-major (rows_out[it][x][row]), so that the
    // column pass loads a column coalesced.  Each vector puts its row in
    // its own exchange buffer (T_v, offset a few complex per vector against
    // bank conflicts), and the CTA writes one run of vpc rows per column x,
    // as 16-byte row pairs where the rows allow.
    K::sync();   // this vector's last-stage loads are done
    if (outer) {
#pragma unroll
      for (int k1 = 0; k1 < N2; ++k1) xb[N1 * k1 + lane + row_tile_off(vec)] = r3[k1];   // x = N1 k1 + lane
    }
    __syncthreads();
    {
      const int j0 = blockIdx.x * vpc;
      float2 *dst = rows_out + ((size_t)it * N) * n_pix + j0;
      if ((vpc & 1) == 0 && (n_pix & 1) == 0) {
        const int hp = vpc / 2, h = threadIdx.x % hp;   // rows 2h and 2h + 1
        const int xt = threadIdx.x / hp, nxt = blockDim.x / hp;
        if (j0 + 2 * h < n_pix && xt < nxt) {           // n_pix even: both rows exist
          const float2 *ta = smem + (2 * h) * XBF + row_tile_off(2 * h);
          const float2 *tb = smem + (2 * h + 1) * XBF + row_tile_off(2 * h + 1);
          if constexpr (XBF % 2 == 0) {
            // columns x and x + 1 of both rows: two 16-byte loads, two stores
            for (int x = 2 * xt; x < N; x += 2 * nxt) {
              const float4 a = *reinterpret_cast<const float4 *>(ta + x);
              const float4 c = *reinterpret_cast<const float4 *>(tb + x);
              *reinterpret_cast<float4 *>(dst + (size_t)x * n_pix + 2 * h) =
                  make_float4(a.x, a.y, c.x, c.y);
              *reinterpret_cast<float4 *>(dst + (size_t)(x + 1) * n_pix + 2 * h) =
                  make_float4(a.z, a.w, c.z, c.w);
            }
          } else {
            for (int x = xt; x < N; x += nxt) {
              const float2 a = ta[x], c = tb[x];
              *reinterpret_cast<float4 *>(dst + (size_t)x * n_pix + 2 * h) =
                  make_float4(a.x, a.y, c.x, c.y);
            }
          }
        }
      } else {
        const int v = threadIdx.x % vpc, xt = threadIdx.x / vpc, nxt = blockDim.x / vpc;
        if (j0 + v < n_pix && xt < nxt) {
          const float2 *tv = smem + v * XBF + row_tile_off(v);
          for (int x = xt; x < N; x += nxt) dst[(size_t)x * n_pix + v] = tv[x];
        }
      }
    }
    if (q + 1 < ka && it + 1 < n_slots) __syncthreads();   // the buffers are the next slot's
  }
}

// K: per tile of up to tc columns (whole detector pixels, at most P per
// warp), read from rows_in[slot][x][row]: the item's y tilt, column filter,
// |.|^2 / n_mod, b x b bins ->
// part[b % nbw][m][ybin][xbin].  grid (ceil(N / tc), 2 n_slots): y = 2 p + w is
// item m = c (w = 0) or m = n_mod - c (w = 1, when distinct) of slot p.
//
// Tiles of at most 160 threads (five columns for the 39 m pupil's bin side 5,
// twelve for the 8 m pupil's 4) take the variant bounded at 160 threads x 4
// CTAs per SM: 96 registers per thread, so the twiddle loads can be issued
// earlier.
template <int N1, int N2, int PAD, int MAXT>
__global__ void __launch_bounds__(MAXT, N2 > 32 ? 3 : (MAXT <= 160 ? 4 : (MAXT <= 256 ? 3 : 2)))
    k_colfilt_bin(
    const float2 *__restrict__ rows_in, const float2 *__restrict__ gy,
    const float2 *__restrict__ twA, const float2 *__restrict__ twB,
    const float2 *__restrict__ mask, float *__restrict__ part, int n_pix, int fp, int fq,
    float scale, int n_mod, int nc, int nbw, int slot0, int tc, int s0) {
  pdl_wait();
  using P = PadRegs<N1, N2, PAD>;
  using K = Pack<N1, N2>;
  constexpr int N = K::N, S1 = K::S1, S2 = K::S2, CS = K::XS;
  constexpr int LO = P::LO, NR = P::HI - P::LO;
  extern __shared__ __align__(16) float2 smem_k[];
  float2 *s_tile = smem_k;
  const int it = blockIdx.y >> 1;              // slot within the chunk
  const int gs = slot0 + it;
  const int b = gs / nc, cslot = s0 + (gs - b * nc);   // nc slots per element from s0
  const int m = (blockIdx.y & 1) ? n_mod - cslot : cslot;
  if ((blockIdx.y & 1) && (cslot == 0 || 2 * cslot == n_mod)) return;   // no second item
  const int col0 = blockIdx.x * tc, ncol = min(tc, N - col0);
  const int wlane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int lane = K::CTA ? threadIdx.x % N1 : wlane % N1;
  const bool outer = K::CTA || wlane / N1 < K::P;   // this lane takes part in the outer stages
  const int vec = K::CTA ? threadIdx.x / N1 : warp * K::P + (outer ? wlane / N1 : 0);
  // this vector's column x = col0 + vec: n_pix contiguous rows of the
  // slot's column-major block, loaded coalesced straight into registers and
  // past L1 (which keeps the twiddle, mask and tilt tables)
  // (lanes that take no part and columns past the tile repeat valid ones;
  // their values are not stored, or not binned)
  const float2 *cx = rows_in + ((size_t)it * N + min(col0 + vec, N - 1)) * n_pix;
  float2 r[N2];
  {
    const int row0 = lane + N1 * LO - P::OFF;   // pupil row of register LO
    const float2 *g = gy + (size_t)m * n_pix + row0;
    const float2 *w = cx + row0;
    float2 e[NR];
    bool ok[NR];
#pragma unroll
    for (int h = 0; h < NR; ++h) {
      const int row = row0 + N1 * h;
      ok[h] = P::ALIGNED || ((h > 0 || row >= 0) && (h < NR - 1 || row < n_pix));
      e[h] = ok[h] ? ld_stream2(w + N1 * h) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int h = 0; h < NR; ++h) {
      r[LO + h] = ok[h] ? cmul(e[h], __ldg(g + N1 * h)) : make_float2(0.f, 0.f);
    }
  }
  float2 *col = s_tile + vec * CS;   // this vector's exchange buffer
  RegDFTZ<N2, false, P::NZ>::run(r);
  if (outer) {
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) col[k2 * S1 + lane] = cmulc(r[k2], __ldg(twA + k2 * N1 + lane));
  }
  K::sync();
  packed_mid<N1, N2, CS>(s_tile, mask, twB);
  K::sync();
  float2 r3[N2];
#pragma unroll
  for (int n1 = 0; n1 < N2; ++n1) r3[n1] = col[lane * S2 + n1];
  RegDFT<N2, true>::run(r3);
  K::sync();
  float *colI = reinterpret_cast<float *>(col);   // this column's intensity, y = N1 k1 + lane
  if (outer) {
#pragma unroll
    for (int k1 = 0; k1 < N2; ++k1)
      colI[N1 * k1 + lane] = (r3[k1].x * r3[k1].x + r3[k1].y * r3[k1].y) * scale;
  }
  __syncthreads();
  float *dst = part + ((size_t)(b % nbw) * n_mod + m) * (N * fq / fp) * (N * fq / fp);
  const float *s_I = reinterpret_cast<const float *>(smem_k);
  if (fq != 1) {
    // fractional detector pixels of fp / fq grid pixels (area-weighted
    // rebinning): output pixel o covers [o fp, (o + 1) fp) and grid pixel i
    // covers [i fq, (i + 1) fq) in units of 1 / fq; the weight is their
    // overlap, an integer, and the sum is divided by fq^2 once.  The tile's
    // ncol = k fp columns hold exactly its k fq output columns.
    const int nd = N * fq / fp, nxo = ncol / fp * fq, xo0 = col0 / fp * fq;
    const float inv = 1.0f / (float)(fq * fq);
    for (int q = threadIdx.x; q < nd * nxo; q += blockDim.x) {
      const int yo = q / nxo, X = xo0 + (q - yo * nxo);
      const int px0 = X * fp / fq, px1 = ((X + 1) * fp + fq - 1) / fq;
      const int py0 = yo * fp / fq, py1 = ((yo + 1) * fp + fq - 1) / fq;
      float v = 0.f;
      for (int py = py0; py < py1; ++py) {
        const int wy = min((py + 1) * fq, (yo + 1) * fp) - max(py * fq, yo * fp);
        for (int px = px0; px < px1; ++px) {
          const int wx = min((px + 1) * fq, (X + 1) * fp) - max(px * fq, X * fp);
          v += (float)(wx * wy) * s_I[(size_t)(px - col0) * 2 * CS + py];
        }
      }
      dst[(size_t)yo * nd + X] = v * inv;
    }
    return;
  }
  const int bsz = fp, nd = N / bsz, nbx = ncol / bsz;
  if (bsz == 5 && nbx == 1) {
    // the 39 m pupil's 5 x 5 bins, one bin column per tile: unrolled sums
    for (int yb = threadIdx.x; yb < nd; yb += blockDim.x) {
      const float *c0 = s_I + yb * 5;
      float v = 0.f;
#pragma unroll
      for (int rr = 0; rr < 5; ++rr)
#pragma unroll
        for (int cc = 0; cc < 5; ++cc) v += c0[cc * 2 * CS + rr];
      dst[(size_t)yb * nd + col0 / 5] = v;
    }
    return;
  }
  for (int q = threadIdx.x; q < nd * nbx; q += blockDim.x) {
    const int yb = q / nbx, xb = q - yb * nbx;
    float v = 0.f;
    for (int rr = 0; rr < bsz; ++rr)
      for (int cc = 0; cc < bsz; ++cc) v += s_I[(size_t)(xb * bsz + cc) * 2 * CS + yb * bsz + rr];
    dst[(size_t)yb * nd + col0 / bsz + xb] = v;
  }
}

// --------------------------------------------------------------------------
// D: det[b] = sum over m = 0 .. n_mod-1 of part[b % nbw][m], in order.
// grid (ceil(nd^2 / 256), number of batch elements from b0).
__global__ void __launch_bounds__(256) k_bin_reduce(const float *__restrict__ part,
                                                    float *__restrict__ det, int nd2, int n_mod,
                                                    int nbw, int b0, float alpha, float beta) {
  pdl_wait();
  const int pix = blockIdx.x * blockDim.x + threadIdx.x;
  if (pix >= nd2) return;
  const int b = b0 + blockIdx.y;
  const float *src = part + (size_t)(b % nbw) * n_mod * nd2 + pix;
  // sixteen loads in flight, then the adds in order m = 0, 1, ...
  float v = 0.f;
  int m = 0;
  for (; m + 16 <= n_mod; m += 16) {
    float x[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) x[u] = src[(size_t)(m + u) * nd2];
#pragma unroll
    for (int u = 0; u < 16; ++u) v += x[u];
  }
  for (; m < n_mod; ++m) v += src[(size_t)m * nd2];
  // det = alpha v (beta = 0) or beta det + alpha v (accumulating images)
  float *d = det + (size_t)b * nd2 + pix;
  *d = beta == 0.f ? alpha * v : beta * *d + alpha * v;
}

// --------------------------------------------------------------------------
// host side

constexpr int kColsTile = 8;

// f(integral_constant<int, pad>) for the paddings the two-pass kernels of a
// split are built for: those that divide N, but not pad 2 at 660 and 1600 (the
// plan refuses it).
template <int N1, int N2, class F> static void for_pad(int pad, F &&f) {
  constexpr int N = N1 * N2;
  if constexpr (N2 % 4 == 0 && N1 <= 32)
    if (pad == 2) f(std::integral_constant<int, 2>{});
  if constexpr (N % 3 == 0)
    if (pad == 3) f(std::integral_constant<int, 3>{});
  if constexpr (N % 4 == 0)
    if (pad == 4) f(std::integral_constant<int, 4>{});
}

template <int N1, int N2>
static int configure(PwfsPlan *p) {
  using S = Split<N1, N2>;
  {
    const int nd = p->pad * p->n_sub;
    int a = S::N, b = nd;
    while (b) {
      const int t = a % b;
      a = b;
      b = t;
    }
    p->fp = S::N / a;
    p->fq = nd / a;
    p->G = S::G;
  }
  int s;
  if constexpr (S::WIDE) {
    // wide splits: the two-pass form only
    p->blockA = p->blockB = p->blockC = 0;
    p->smemA = p->smemB = p->smemC = 0;
  } else {
    const int bsz = p->fq == 1 ? p->fp : 0;   // whole bins only below the two-pass form
    p->blockA = 256;
    const int vpcA = 256 / S::G;
    p->smemA = (size_t)(vpcA * S::XB) * sizeof(float2);
    p->blockB = kColsTile * S::G;
    p->smemB = ColsCfg<N1, N2, kColsTile>::smem;
    const int thrC = ((bsz * S::G + 31) / 32) * 32;
    if (thrC > 256) return SPECULA_EUNSUPPORTED;   // bin side too large for one CTA strip
    p->blockC = bsz ? thrC : 0;                     // 0: no three-pass form (fractional bins)
    const int nvecC = thrC / S::G;
    p->smemC = (size_t)(nvecC * S::XB) * sizeof(float2);
    if (p->smemA > 227 * 1024 || p->smemB > 227 * 1024 || p->smemC > 227 * 1024)
      return SPECULA_EUNSUPPORTED;
    if ((s = ensure_dynamic_smem((const void *)k_rows_fwd<N1, N2>, p->smemA)) ||
        (s = ensure_dynamic_smem((const void *)k_cols<N1, N2, kColsTile>, p->smemB)) ||
        (s = ensure_dynamic_smem((const void *)k_rows_inv_part<N1, N2>, p->smemC)))
      return s;
  }
  return SPECULA_OK;
}

// Two-pass form (its own split of N: N1, N2): column tiles of whole detector
// pixels, so every detector pixel lies in one CTA.  The number of warps is the
// one that leaves the fewest lanes idle (a tile narrower than its warps, a
// last tile that is not full), up to five of 32-value lanes and eight of
// shorter ones (eleven where a detector pixel is a fraction of grid pixels:
// the SOUL example's 11-column tiles); five for 1600's four columns.
template <int N1, int N2>
static int configure_two(PwfsPlan *p) {
  using K = Pack<N1, N2>;
  int s = SPECULA_OK;
  p->two_ok = false;
  p->blockR = RowFiltLaunch<N1, N2>::threads;
  p->smemR = (size_t)K::vecs(p->blockR) * K::XSR * sizeof(float2);
  // a detector pixel's columns at the three-pass split's lanes per transform
  // fit one CTA: the geometries that the plan takes
  if (p->fp * p->G > (K::CTA ? 128 : (p->fq != 1 ? 352 : 256))) return SPECULA_OK;
  if constexpr (K::CTA) {
    p->blockK = 4 * N1;
    p->tcK = 4 / p->fp * p->fp;   // fp <= 4 from the line above
  } else {
    const int fit = (p->fp + K::P - 1) / K::P;   // warps that hold one detector pixel
    const int most = p->fq != 1 ? 11 : std::max(fit, N2 >= 32 ? 5 : 8);
    int best = 0, cost = 0;   // lane columns issued for the N columns of an item
    for (int w = fit; w <= most; ++w) {
      const int tc = w * K::P / p->fp * p->fp;
      const int c = (K::N + tc - 1) / tc * w;
      if (!best || c <= cost) best = w, cost = c;
    }
    if (!best || best * 32 > (p->fq != 1 ? 352 : 256)) return SPECULA_OK;
    p->blockK = best * 32;
    p->tcK = best * K::P / p->fp * p->fp;
  }
  p->smemK = (size_t)K::vecs(p->blockK) * K::XS * sizeof(float2);
  if (p->smemR > 227 * 1024 || p->smemK > 227 * 1024) return SPECULA_OK;
  for_pad<N1, N2>(p->pad, [&](auto pc) {
    constexpr int PAD = decltype(pc)::value;
    if ((s = ensure_dynamic_smem((const void *)k_rowfilt<N1, N2, PAD>, p->smemR))) return;
    if constexpr (K::CTA) {
      s = ensure_dynamic_smem((const void *)k_colfilt_bin<N1, N2, PAD, 160>, p->smemK);
    } else if (!(s = ensure_dynamic_smem((const void *)k_colfilt_bin<N1, N2, PAD, 256>,
                                         p->smemK)) &&
               !(s = ensure_dynamic_smem((const void *)k_colfilt_bin<N1, N2, PAD, 160>,
                                         p->smemK))) {
      s = ensure_dynamic_smem((const void *)k_colfilt_bin<N1, N2, PAD, 352>, p->smemK);
    }
  });
  if (s) return s;
  p->two_ok = true;
  return SPECULA_OK;
}

// Two-pass form, one chunk of `chunk` row-filter slots (batch element,
// distinct cosine) at a time; each slot feeds one or two column items.
template <int N1, int N2>
static int run_split2(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase,
                      int n_batch, float *det, cudaStream_t st) {
  using K = Pack<N1, N2>;
  const int Np = p->n_pix;
  const int nd = p->pad * p->n_sub;   // detector side
  // the imaged cosine slots [s0, s0 + nc) of every batch element
  const int s0 = p->slot_lo;
  const int nc = (p->slot_hi < 0 ? p->nc : p->slot_hi) - s0;
  const int total = n_batch * nc;
  const int vpc = K::vecs(p->blockR);
  const float scale = 1.0f / (float)p->n_mod;
  // The workspace has a field and a partial detector for each of nbw batch
  // elements, the most that `chunk` slots of the whole circle touch; of a slot
  // range's fewer slots per element as many as touch no more.
  const int chunk = std::min(p->chunk, (p->nbw - 1) * nc);
  int field_done = -1, det_done = -1;
  for (int j0 = 0; j0 < total; j0 += chunk) {
    const int nj = std::min(chunk, total - j0);
    const int b0 = j0 / nc, b1 = (j0 + nj - 1) / nc;
    const int fb = std::max(b0, field_done + 1);
    if (fb <= b1) {
      dim3 gF((Np * Np + 255) / 256, b1 - fb + 1);
      SPECULA_LAUNCH_PDL(ctx, SPECULA_K_PWFS_FIELD, st, k_field, gF, 256, 0, amp, phase,
                         p->field.as<float2>(), Np * Np, fb, p->nbw, p->run_phase_scale);
      field_done = b1;
    }
    dim3 gR((Np + vpc - 1) / vpc, (nj + p->ka - 1) / p->ka);
    dim3 gK((K::N + p->tcK - 1) / p->tcK, 2 * nj);
    int s = SPECULA_EUNSUPPORTED;
    for_pad<N1, N2>(p->pad, [&](auto pc) {
      constexpr int PAD = decltype(pc)::value;
      s = [&]() -> int {
        SPECULA_LAUNCH_PDL(ctx, SPECULA_K_PWFS_ROWFILT, st, (k_rowfilt<N1, N2, PAD>), gR,
                           p->blockR, p->smemR, p->field.as<float2>(), p->gx.as<float2>(),
                           p->tpA.as<float2>(), p->tpB.as<float2>(), p->mask.as<float2>(),
                           p->rows.as<float2>(), Np, nc, p->nbw, j0, nj, p->ka, s0);
#define SPECULA_COLFILT(MAXT_)                                                                 \
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_PWFS_COLFILT, st, (k_colfilt_bin<N1, N2, PAD, MAXT_>), gK,    \
                     p->blockK, p->smemK, p->rows.as<float2>(), p->gy.as<float2>(),               \
                     p->tpA.as<float2>(), p->tpB.as<float2>(), p->mask.as<float2>(),              \
                     p->part.as<float>(), Np, p->fp, p->fq, scale, p->n_mod, nc, p->nbw, j0,      \
                     p->tcK, s0)
        if constexpr (K::CTA) {
          SPECULA_COLFILT(160);
        } else {
          if (p->blockK > 256)    // tiles of fractional detector pixels
            SPECULA_COLFILT(352);
          else if (p->blockK <= 160)
            SPECULA_COLFILT(160);
          else
            SPECULA_COLFILT(256);
        }
#undef SPECULA_COLFILT
        return SPECULA_OK;
      }();
    });
    if (s) return s;
    const int complete = (j0 + nj) / nc - 1;
    if (complete > det_done) {
      dim3 gD((nd * nd + 255) / 256, complete - det_done);
      SPECULA_LAUNCH_PDL(ctx, SPECULA_K_PWFS_BIN, st, k_bin_reduce, gD, 256, 0,
                         p->part.as<float>(), det, nd * nd, p->n_mod, p->nbw, det_done + 1,
                         p->run_alpha, p->run_beta);
      det_done = complete;
    }
  }
  return SPECULA_OK;
}

template <int N1, int N2>
static int run_split(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase,
                     int n_batch, float *det, cudaStream_t st) {
  using S = Split<N1, N2>;
  if constexpr (S::WIDE) {
    return SPECULA_EUNSUPPORTED;   // the three-pass kernels hold N2 <= 32
  } else {
    const int Np = p->n_pix;
    const int bsz = Np / p->n_sub;
    const int nd = S::N / bsz;
    const int total = n_batch * p->n_mod;
    const int vpcA = p->blockA / S::G;
    const float scale = 1.0f / (float)p->n_mod;
    int field_done = -1;   // highest batch element whose field is in its slot
    int det_done = -1;     // highest batch element whose detector is written
    for (int i0 = 0; i0 < total; i0 += p->chunk) {
      const int ni = std::min(p->chunk, total - i0);
      const int b0 = i0 / p->n_mod, b1 = (i0 + ni - 1) / p->n_mod;
      const int fb = std::max(b0, field_done + 1);
      if (fb <= b1) {
        dim3 gF((Np * Np + 255) / 256, b1 - fb + 1);
        SPECULA_LAUNCH_PDL(ctx, SPECULA_K_PWFS_FIELD, st, k_field, gF, 256, 0, amp, phase,
                           p->field.as<float2>(), Np * Np, fb, p->nbw, p->run_phase_scale);
        field_done = b1;
      }
      dim3 gA((Np + vpcA - 1) / vpcA, (ni + p->ka - 1) / p->ka);
      {
        SPECULA_LAUNCH(ctx, SPECULA_K_PWFS_ROWS_FWD, st,
                       k_rows_fwd<N1, N2><<<gA, p->blockA, p->smemA, st>>>(
                           p->field.as<float2>(), p->gx.as<float2>(), p->gy.as<float2>(),
                           p->twA.as<float2>(), p->rows.as<float2>(), Np, p->n_mod, p->nbw, i0,
                           ni, p->ka));
        dim3 gB(S::N / kColsTile, ni);
        SPECULA_LAUNCH(ctx, SPECULA_K_PWFS_COLS, st,
                       k_cols<N1, N2, kColsTile><<<gB, p->blockB, p->smemB, st>>>(
                           p->rows.as<float2>(), p->cols.as<float2>(), p->twA.as<float2>(),
                           p->twB.as<float2>(), p->mask.as<float2>(), Np));
        dim3 gC(S::N / bsz, ni);
        SPECULA_LAUNCH(ctx, SPECULA_K_PWFS_ROWS_INV, st,
                       k_rows_inv_part<N1, N2><<<gC, p->blockC, p->smemC, st>>>(
                           p->cols.as<float2>(), p->twA.as<float2>(), p->part.as<float>(), bsz,
                           scale, p->n_mod, p->nbw, i0));
      }
      // batch elements whose last modulation point is in this chunk
      const int complete = (i0 + ni) / p->n_mod - 1;
      if (complete > det_done) {
        dim3 gD((nd * nd + 255) / 256, complete - det_done);
        SPECULA_LAUNCH_PDL(ctx, SPECULA_K_PWFS_BIN, st, k_bin_reduce, gD, 256, 0,
                           p->part.as<float>(), det, nd * nd, p->n_mod, p->nbw, det_done + 1,
                           p->run_alpha, p->run_beta);
        det_done = complete;
      }
    }
    return SPECULA_OK;
  }
}

bool pwfs_split_for(int N, int *N1, int *N2) {
  switch (N) {
    case 64: *N1 = 8; *N2 = 8; return true;
    case 128: *N1 = 8; *N2 = 16; return true;
    case 240: *N1 = 15; *N2 = 16; return true;
    case 320: *N1 = 20; *N2 = 16; return true;
    case 660: *N1 = 30; *N2 = 22; return true;   // 22 = 2 x 11, prime-factor form
    case 960: *N1 = 30; *N2 = 32; return true;
    case 1600: *N1 = 32; *N2 = 50; return true;   // no kernel's: the two-pass form takes 40 x 40
    default: return false;
  }
}

int pwfs_set_tiles(PwfsPlan *p, int chunk, int ka, int passes) {
  if (passes < 2 || passes > 4) return SPECULA_EINVAL;
  if (passes == 2 && !p->two_ok) return SPECULA_EUNSUPPORTED;
  if (passes == 3 && (p->pad != 2 || !p->blockC)) return SPECULA_EUNSUPPORTED;   // pad-2, whole bins
  if (passes == 4 && !p->pair_ok) return SPECULA_EUNSUPPORTED;
  const int nd = p->pad * p->n_sub;   // detector side
  // batch elements one chunk can touch: chunk items (three-pass) or chunk
  // row-filter slots, nc per batch element (two-pass); the paired form runs
  // whole batch elements, chunk / nc (at least one) per launch
  const int per_b = passes == 3 ? p->n_mod : p->nc;
  if (passes == 4) chunk = std::max(1, chunk / p->nc) * p->nc;
  const int nbw = passes == 4 ? chunk / p->nc : (chunk + per_b - 1) / per_b + 1;
  const size_t need_field = (size_t)nbw * p->n_pix * p->n_pix * sizeof(float2);
  // two complex of padding: the paired form's column staging window may
  // read one entry past the last row
  const size_t need_rows = ((size_t)chunk * p->n_pix * p->N + 2) * sizeof(float2);
  const size_t need_cols = passes == 3 ? (size_t)chunk * p->N * p->N * sizeof(float2) : 0;
  const size_t need_part = (size_t)nbw * p->n_mod * nd * nd * sizeof(float);
  int s;
  if (need_rows > p->rows.bytes || need_cols > p->cols.bytes || need_field > p->field.bytes ||
      need_part > p->part.bytes) {
    cudaDeviceSynchronize();   // the old workspace may still be in use
    if ((s = p->field.alloc(std::max(need_field, p->field.bytes)))) return s;
    if ((s = p->rows.alloc(std::max(need_rows, p->rows.bytes)))) return s;
    if (need_cols > p->cols.bytes && (s = p->cols.alloc(need_cols))) return s;
    if ((s = p->part.alloc(std::max(need_part, p->part.bytes)))) return s;
    // items outside an imaged slot range are never written: they read as 0
    SPECULA_CK(cudaMemset(p->part.p, 0, p->part.bytes));
  }
  p->chunk = chunk;
  p->ka = ka;
  p->nbw = nbw;
  p->passes = passes;
  return SPECULA_OK;
}

int pwfs_bin_reduce(specula_ctx *ctx, const float *part, float *det, int nd2, int n_mod,
                    float alpha, float beta, cudaStream_t st) {
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_PWFS_BIN, st, k_bin_reduce, dim3((nd2 + 255) / 256, 1), 256, 0,
                     part, det, nd2, n_mod, 1, 0, alpha, beta);
  return SPECULA_OK;
}

int pwfs_field_launch(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase,
                      int fb, int nb, cudaStream_t st) {
  const int Np = p->n_pix;
  dim3 gF((Np * Np + 255) / 256, nb);
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_PWFS_FIELD, st, k_field, gF, 256, 0, amp, phase,
                     p->field.as<float2>(), Np * Np, fb, p->nbw, p->run_phase_scale);
  return SPECULA_OK;
}

int pwfs_bin_reduce_range(specula_ctx *ctx, PwfsPlan *p, float *det, int nd2, int b0, int nb,
                          cudaStream_t st) {
  dim3 gD((nd2 + 255) / 256, nb);
  SPECULA_LAUNCH_PDL(ctx, SPECULA_K_PWFS_BIN, st, k_bin_reduce, gD, 256, 0, p->part.as<float>(),
                     det, nd2, p->n_mod, p->nbw, b0, p->run_alpha, p->run_beta);
  return SPECULA_OK;
}

int pwfs_run(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase, int n_batch,
             float *det, cudaStream_t st) {
  if (p->slot_hi >= 0 && (p->form != SPECULA_PWFS_FORM_TILT || p->passes == 3))
    return SPECULA_EUNSUPPORTED;   // slot ranges: the two-pass tilt forms only
  if (p->form == SPECULA_PWFS_FORM_SHIFTED)
    return pwfs_shifted_run(ctx, p, amp, phase, n_batch, det, st);
  if (p->form == SPECULA_PWFS_FORM_DFTGEMM_BF16 || p->form == SPECULA_PWFS_FORM_DFTGEMM_TF32)
    return pwfs_dftgemm_run(ctx, p, amp, phase, n_batch, det, st);
  if (p->passes == 4) return pwfs_pair_run(ctx, p, amp, phase, n_batch, det, st);
  if (p->passes == 2) {
    switch (p->N) {
      case 64: return run_split2<8, 8>(ctx, p, amp, phase, n_batch, det, st);
      case 128: return run_split2<8, 16>(ctx, p, amp, phase, n_batch, det, st);
      case 240: return run_split2<15, 16>(ctx, p, amp, phase, n_batch, det, st);
      case 320:
        return p->M1 == 16 ? run_split2<16, 20>(ctx, p, amp, phase, n_batch, det, st)
                           : run_split2<10, 32>(ctx, p, amp, phase, n_batch, det, st);
      case 660: return run_split2<30, 22>(ctx, p, amp, phase, n_batch, det, st);
      case 960: return run_split2<30, 32>(ctx, p, amp, phase, n_batch, det, st);
      case 1600: return run_split2<40, 40>(ctx, p, amp, phase, n_batch, det, st);
      default: return SPECULA_EUNSUPPORTED;
    }
  }
  switch (p->N) {
    case 64: return run_split<8, 8>(ctx, p, amp, phase, n_batch, det, st);
    case 128: return run_split<8, 16>(ctx, p, amp, phase, n_batch, det, st);
    case 240: return run_split<15, 16>(ctx, p, amp, phase, n_batch, det, st);
    case 320: return run_split<20, 16>(ctx, p, amp, phase, n_batch, det, st);
    case 660: return run_split<30, 22>(ctx, p, amp, phase, n_batch, det, st);
    case 960: return run_split<30, 32>(ctx, p, amp, phase, n_batch, det, st);
    case 1600: return run_split<32, 50>(ctx, p, amp, phase, n_batch, det, st);
    default: return SPECULA_EUNSUPPORTED;
  }
}

// Time the plan's present tiling and each candidate on the caller's buffers (set-up
// call: may reallocate the workspace and synchronises) and keep the fastest; the
// present one stays unless another is also faster in a second, longer run of the two.
// Candidates: a list of small chunks, and whole batch elements (nc, 2 nc, 4 nc, ...
// slots) for batches whose slots go beyond the list, where the plan's own default is
// one of them and the list's last, nearly empty waves cost most (8 m image, batch 16:
// 157 us untuned, 184 with the list alone; batch 256: 2443 and 2773, tuned now 2354).
int pwfs_autotune(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase,
                  int n_batch, float *det, cudaStream_t st, int reps, size_t max_ws_bytes,
                  int *best_chunk, int *best_ka, int *best_passes) {
  static const int kChunks[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64};
  constexpr int kListEnd = 64, kMaxChunk = 4096;   // what specula_pwfs_set_tiles takes
  const size_t per_item = ((size_t)p->n_pix * p->N + (size_t)p->N * p->N) * sizeof(float2);
  const auto item_bytes = [&](int passes) {
    return passes != 3 ? (size_t)p->n_pix * p->N * sizeof(float2) : per_item;
  };
  const int total = n_batch * p->n_mod;
  cudaEvent_t e0, e1;
  SPECULA_CK(cudaEventCreate(&e0));
  SPECULA_CK(cudaEventCreate(&e1));
  const auto run = [&](int chunk, int ka, int passes, int n, float *ms) -> int {
    int s = pwfs_set_tiles(p, chunk, ka, passes);
    if (!s) s = pwfs_run(ctx, p, amp, phase, n_batch, det, st);   // warm-up
    if (s) return s;
    cudaEventRecord(e0, st);
    for (int r = 0; r < n; ++r)
      if ((s = pwfs_run(ctx, p, amp, phase, n_batch, det, st))) return s;
    cudaEventRecord(e1, st);
    if (cudaEventSynchronize(e1) != cudaSuccess) return SPECULA_ECUDA;
    cudaEventElapsedTime(ms, e0, e1);
    return SPECULA_OK;
  };
  int status = SPECULA_OK;
  float best = 1e30f;
  int bc = p->chunk, bk = p->ka, bp = p->passes;
  const int c0 = bc, k0 = bk, p0 = bp;
  const bool keep_ok = (size_t)c0 * item_bytes(p0) <= max_ws_bytes;
  const auto consider = [&](int chunk, int ka, int passes) -> int {
    float ms = 0.f;
    const int s = run(chunk, ka, passes, reps, &ms);
    if (!s && ms < best) { best = ms; bc = p->chunk; bk = ka; bp = passes; }
    return s;
  };
  // ka sets the row pass's grid depth (slots per warp): values that fill
  // whole waves of CTAs can win (the ELT frame: ka 5, 300 CTAs on 304
  // slots), so the search goes to 8
  const auto consider_kas = [&](int chunk, int passes) -> int {
    for (int ka = 1; ka <= std::min(passes == 4 ? 1 : 8, chunk); ++ka) {
      const int s = consider(chunk, ka, passes);
      if (s) return s;
    }
    return SPECULA_OK;
  };
  if (keep_ok && (status = consider(c0, k0, p0))) goto done;
  for (int passes = 2; passes <= 4; ++passes) {
    if (passes == 2 && !p->two_ok) continue;
    if (passes == 3 && p->pad != 2) continue;
    if (passes == 4 && !p->pair_ok) continue;
    const size_t item = item_bytes(passes);
    if (passes != 4)
      for (int c : kChunks) {
        if (c != 1 && (c > total || (size_t)c * item > max_ws_bytes)) break;
        if ((status = consider_kas(c, passes))) goto done;
      }
    if (passes == 4 || (passes == 2 && (long long)n_batch * p->nc > kListEnd))
      for (int c = 1; c <= n_batch && (long long)c * p->nc <= kMaxChunk; c *= 2) {
        if ((size_t)c * p->nc * item > max_ws_bytes && (c != 1 || passes == 2)) break;
        if ((status = consider_kas(c * p->nc, passes))) goto done;
      }
  }
  if (keep_ok && (bc != c0 || bk != k0 || bp != p0)) {
    float now = 0.f, other = 0.f;
    if ((status = run(c0, k0, p0, 4 * reps, &now)) ||
        (status = run(bc, bk, bp, 4 * reps, &other)))
      goto done;
    if (now <= other) { bc = c0; bk = k0; bp = p0; }
  }
  status = pwfs_set_tiles(p, bc, bk, bp);
  *best_chunk = bc;
  *best_ka = bk;
  *best_passes = bp;
done:
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return status;
}

// The three-pass form's split (none for 1600), and the two-pass form's: the
// same but for 1600 = 40 x 40 and 320 = 10 x 32, at padding 4 16 x 20: there the
// rounding of the 10 x 32 twiddles that the few bright frequencies meet made the
// whole image 7e-8 too faint (r.m.s. error 1.33e-7 over 32 images of 80 px pupils;
// 20 x 16 1.04e-7, 16 x 20 1.02e-7; 64 images of 7 points 159, 255 and 196 us).
template <int N1, int N2, int M1 = N1, int M2 = N2>
static int configure_both(PwfsPlan *p) {
  p->M1 = M1;
  p->M2 = M2;
  const int s = configure<N1, N2>(p);
  return s ? s : configure_two<M1, M2>(p);
}

static int configure_for(PwfsPlan *p) {
  switch (p->N) {
    case 64: return configure_both<8, 8>(p);
    case 128: return configure_both<8, 16>(p);
    case 240: return configure_both<15, 16>(p);
    case 320:
      return p->pad == 4 ? configure_both<20, 16, 16, 20>(p) : configure_both<20, 16, 10, 32>(p);
    case 660: return configure_both<30, 22>(p);
    case 960: return configure_both<30, 32>(p);
    case 1600: return configure_both<32, 50, 40, 40>(p);
    default: return SPECULA_EUNSUPPORTED;
  }
}

PwfsPlan *pwfs_plan_find(specula_ctx *ctx, const specula_pupil_desc *pupil,
                         const specula_pwfs_desc *d) {
  for (auto &p : ctx->pwfs)
    if (p->n_pix == pupil->n_pix && p->pad == d->pad && p->n_mod == d->n_mod &&
        p->n_sub == d->n_sub && p->pup_dist == d->pup_dist_px && p->mod_amp == d->mod_amp)
      return p.get();
  return nullptr;
}

// exp(i * pi * num / den) with num reduced exactly modulo 2 den
static inline void exp_ipi(long long num, long long den, double *c, double *s) {
  long long r = num % (2 * den);
  if (r < 0) r += 2 * den;
  const double a = M_PI * (double)r / (double)den;
  *c = cos(a);
  *s = sin(a);
}

// inter-step twiddles (cos, sin)(2 pi (a b mod N) / N)
void pwfs_host_twiddles(int N, int N1, int N2, std::vector<float2> *twA,
                        std::vector<float2> *twB) {
  twA->resize(N);
  twB->resize(N);
  for (int a = 0; a < N2; ++a)
    for (int b = 0; b < N1; ++b) {
      double c, sn;
      exp_ipi(2LL * ((long long)a * b % N), N, &c, &sn);
      (*twA)[a * N1 + b] = (*twB)[b * N2 + a] = make_float2((float)c, (float)sn);
    }
}

void pwfs_host_tables(int Np, int N, int N1, int N2, int n_mod, double mod_amp, int pup_dist,
                      PwfsTablesHost *t) {
  const int off = (N - Np) / 2;
  // modulation tilt x centred-DFT input phase, per axis, float64 -> float32
  std::vector<float2> gx((size_t)n_mod * Np), gy((size_t)n_mod * Np);
  for (int m = 0; m < n_mod; ++m) {
    const double th = 2.0 * M_PI * m / n_mod;
    const double ct = cos(th), sn = sin(th);
    for (int i = 0; i < Np; ++i) {
      const double x = (double)i - (Np - 1) / 2.0;
      double pc, ps;
      exp_ipi((long long)(N - 1) * (off + i), N, &pc, &ps);
      const double ax = 2.0 * M_PI * mod_amp * x * ct / Np;
      const double ay = 2.0 * M_PI * mod_amp * x * sn / Np;
      const double cx = cos(ax), sx = sin(ax), cy = cos(ay), sy = sin(ay);
      gx[(size_t)m * Np + i] = make_float2((float)(cx * pc - sx * ps), (float)(cx * ps + sx * pc));
      gy[(size_t)m * Np + i] = make_float2((float)(cy * pc - sy * ps), (float)(cy * ps + sy * pc));
    }
  }
  // pyramid mask per axis: exp(-2 pi i c |u| / N) / N, c = pup_dist / 2,
  // u = k - (N-1)/2: angle = -pi pup_dist |2k - N + 1| / (2N)
  std::vector<float2> mk(N);
  for (int k = 0; k < N; ++k) {
    long long a = 2LL * k - N + 1;
    if (a < 0) a = -a;
    double c, sn;
    exp_ipi(-(long long)pup_dist * a, 2LL * N, &c, &sn);
    mk[k] = make_float2((float)(c / N), (float)(sn / N));
  }
  t->gx = std::move(gx);
  t->gy = std::move(gy);
  t->mask = std::move(mk);
  pwfs_host_twiddles(N, N1, N2, &t->twA, &t->twB);
}

int pwfs_plan_build(specula_ctx *ctx, const specula_pupil_desc *pupil,
                    const specula_pwfs_desc *d, PwfsPlan **out) {
  const int Np = pupil->n_pix, N = d->pad * Np;
  int N1, N2;
  if (!pwfs_split_for(N, &N1, &N2)) return SPECULA_EUNSUPPORTED;
  if (N2 % 4 && d->pad == 2) return SPECULA_EUNSUPPORTED;   // pruned pad-2 loads need N2 % 4 == 0
  std::unique_ptr<PwfsPlan> p(new PwfsPlan());
  p->n_pix = Np; p->pad = d->pad; p->n_mod = d->n_mod; p->n_sub = d->n_sub;
  p->pup_dist = d->pup_dist_px; p->mod_amp = d->mod_amp;
  p->N = N; p->N1 = N1; p->N2 = N2;
  // distinct cosines of the modulation angles 2 pi m / n_mod: m and n_mod - m
  p->nc = d->n_mod / 2 + 1;
  int s = configure_for(p.get());
  if (!s) s = pwfs_pair_configure(p.get());
  if (s) return s;
  PwfsTablesHost T;
  pwfs_host_tables(Np, N, N1, N2, d->n_mod, d->mod_amp, d->pup_dist_px, &T);
  if ((s = pwfs_pair_tables(p.get(), T))) return s;
  const std::vector<float2> &gx = T.gx, &gy = T.gy, &mk = T.mask, &ta = T.twA, &tb = T.twB;
  if ((s = p->gx.upload(gx.data(), gx.size() * sizeof(float2)))) return s;
  if ((s = p->gy.upload(gy.data(), gy.size() * sizeof(float2)))) return s;
  if ((s = p->mask.upload(mk.data(), mk.size() * sizeof(float2)))) return s;
  if (p->blockA) {   // the three-pass form's split (and the shifted form's)
    if ((s = p->twA.upload(ta.data(), ta.size() * sizeof(float2)))) return s;
    if ((s = p->twB.upload(tb.data(), tb.size() * sizeof(float2)))) return s;
  }
  std::vector<float2> pa, pb;
  pwfs_host_twiddles(N, p->M1, p->M2, &pa, &pb);
  if ((s = p->tpA.upload(pa.data(), pa.size() * sizeof(float2)))) return s;
  if ((s = p->tpB.upload(pb.data(), pb.size() * sizeof(float2)))) return s;

  // Default chunk.  Two-pass form: as many row-filter slots as keep the rows
  // workspace within kRowsBytes, a size that L2 (129 MB) still holds between
  // the passes, in whole batch elements where one fits (at most
  // kChunkElements) and in equal parts of one where not.  Small chunks end
  // each launch on a nearly empty last wave: 4 of the 39 m image's 25 slots
  // per launch (120 row and 1536 column CTAs at a time) cost its frame 303 us
  // against 253 us in one chunk; the ANDES image in 13 chunks 604 us, 402 us
  // in one.
  // Three-pass form: both intermediates near 48 MB.
  constexpr size_t kRowsBytes = (size_t)100 << 20;
  constexpr int kChunkElements = 32;
  int chunk;
  if (p->two_ok) {
    const size_t slot = (size_t)Np * N * sizeof(float2);
    const int fit = (int)std::max<size_t>(1, kRowsBytes / slot);
    if (fit >= p->nc) {
      chunk = std::min(fit / p->nc, kChunkElements) * p->nc;
    } else {
      const int parts = (p->nc + fit - 1) / fit;
      chunk = (p->nc + parts - 1) / parts;
    }
    chunk = std::min(chunk, 4096);
  } else {
    const size_t per_item = ((size_t)Np * N + (size_t)N * N) * sizeof(float2);
    chunk = (int)std::min<size_t>(64, std::max<size_t>(1, (48u << 20) / per_item));
  }
  if ((s = pwfs_set_tiles(p.get(), chunk, 1, p->two_ok ? 2 : 3))) return s;
  *out = p.get();
  ctx->pwfs.push_back(std::move(p));
  return SPECULA_OK;
}

}  // namespace specula

// Von Karman phase screens by the FFT method with subharmonics (set-up call;
// AtmoEvolution, App. A, Tab. 4; Listing 2 `L0`, `Cn2`, `seed`).
//
//   Phi(f) = 0.023 r0^(-5/3) (|f|^2 + L0^-2)^(-11/6), Phi(0) = 0  [rad^2 m^2]
//   screen[y][x] = Re sum_k c_k sqrt(Phi(f_k)) df exp(2 pi i f_k . (x, y) pitch)
//                + subharmonics - their spatial mean
//
// A set-up cost, not per frame: float64, and pairs of float32 in the batched form.
// The single screen from given noise: spectral weighting, a radix-2 Stockham FFT along rows in shared memory, a
// tiled transpose, the second row pass, and a final kernel that adds the
// separable subharmonic sum and rounds to float32 once.
#include <math.h>

#include <algorithm>
#include <vector>

#include "float_pair.cuh"
#include "internal.h"
#include "philox.cuh"

namespace specula {

// A[ky][kx] = noise[ky][kx] * sqrt(Phi(f)) * df
__global__ void k_psd_weight(const double2 *__restrict__ noise, double2 *__restrict__ A, int M,
                             double Md, double coef, double k0) {
  const int kx = blockIdx.x * blockDim.x + threadIdx.x, ky = blockIdx.y;
  if (kx >= M) return;
  const int sx = kx >= M / 2 ? kx - M : kx, sy = ky >= M / 2 ? ky - M : ky;
  const double fx = (double)sx / Md, fy = (double)sy / Md;
  const double f2 = fx * fx + fy * fy;
  double a = 0.0;
  if (f2 > 0.0) a = sqrt(coef * pow(f2 + k0, -11.0 / 6.0)) / Md;
  const double2 c = noise[(size_t)ky * M + kx];
  A[(size_t)ky * M + kx] = make_double2(c.x * a, c.y * a);
}

// In-place unnormalised inverse DFT of each row (exp(+2 pi i k n / M)),
// radix-2 Stockham in shared memory.  One CTA per row.
__global__ void k_fft_rows_f64(double2 *__restrict__ data, const double2 *__restrict__ tw, int M,
                               int logM) {
  extern __shared__ double2 sm[];
  double2 *a = sm, *b = sm + M;
  double2 *row = data + (size_t)blockIdx.x * M;
  for (int i = threadIdx.x; i < M; i += blockDim.x) a[i] = row[i];
  __syncthreads();
  // Stockham: stage with half-size Ls, stride; out[j*2Ls + k] etc.
  int L = 1;
  for (int s = 0; s < logM; ++s) {
    const int Ls = L;  // current sub-transform length
    L <<= 1;
    const int half = M / 2;
    for (int q = threadIdx.x; q < half; q += blockDim.x) {
      const int k = q % Ls;        // index within sub-transform
      const int j = q / Ls;        // which sub-transform pair
      const double2 u = a[j * Ls + k];
      const double2 v0 = a[j * Ls + k + half];
      // twiddle exp(+2 pi i k / L) = tw[k * (M / L)]
      const double2 w = tw[k * (M / L)];
      const double2 v = make_double2(v0.x * w.x - v0.y * w.y, v0.x * w.y + v0.y * w.x);
      b[j * L + k] = make_double2(u.x + v.x, u.y + v.y);
      b[j * L + k + Ls] = make_double2(u.x - v.x, u.y - v.y);
    }
    __syncthreads();
    double2 *t = a; a = b; b = t;
  }
  for (int i = threadIdx.x; i < M; i += blockDim.x) row[i] = a[i];
}

__global__ void k_transpose_f64(const double2 *__restrict__ in, double2 *__restrict__ out, int M) {
  __shared__ double2 tile[32][33];
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y)
    tile[r][threadIdx.x] = in[(size_t)(by + r) * M + bx + threadIdx.x];
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y)
    out[(size_t)(bx + r) * M + by + threadIdx.x] = tile[threadIdx.x][r];
}

// screen[y][x] = Re(T[x][y]) + sum_{p,a,b} Re(C[p][b][a] tx[p][a][x] tx[p][b][y]) - mean
__global__ void k_screen_final(const double2 *__restrict__ T, const double2 *__restrict__ tab,
                               const double2 *__restrict__ coef, double sub_mean, int M,
                               int levels, float *__restrict__ out) {
  __shared__ double2 tile[32][33];
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  // T is stored transposed: T[x][y]
  for (int r = threadIdx.y; r < 32; r += blockDim.y)
    tile[r][threadIdx.x] = T[(size_t)(bx + r) * M + by + threadIdx.x];
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int y = by + r, x = bx + threadIdx.x;
    double v = tile[threadIdx.x][r].x;
    double sub = 0.0;
    for (int p = 0; p < levels; ++p)
      for (int bb = 0; bb < 3; ++bb)
        for (int aa = 0; aa < 3; ++aa) {
          if (aa == 1 && bb == 1) continue;
          const double2 ex = tab[((size_t)p * 3 + aa) * M + x];
          const double2 ey = tab[((size_t)p * 3 + bb) * M + y];
          const double2 e = make_double2(ex.x * ey.x - ex.y * ey.y, ex.x * ey.y + ex.y * ey.x);
          const double2 c = coef[(p * 3 + bb) * 3 + aa];
          sub += c.x * e.x - c.y * e.y;
        }
    out[(size_t)y * M + x] = (float)(v + (sub - sub_mean));
  }
}

// ---- Box-Muller in float64 ------------------------------------------------------
// (r cos 2 pi v, r sin 2 pi v), r = sqrt(-2 ln u), with the uniforms u, v =
// (x + 1/2) 2^-32 of two Philox words: the values of specula_rng_complex and the
// batched screens' subharmonic coefficients (their grids take float32 pairs).
// float64 runs at 2 operations per clock and SM here, so the functions
// are written for these arguments, 33-bit integers over 2^33: table lookups
// after exact integer range reduction and short polynomials (the table-driven
// method of Tang, ACM TOMS 16, 378, 1990, for the logarithm; addition theorems
// for sine and cosine; Goldschmidt's iteration for the square root), about 39
// float64 operations per pair where log, sqrt and sincospi take about twice
// that.  Largest errors on the CPU over 6 million arguments: radius 1.7e-16
// relative, angle 2.1e-16; a normal's, against 113-bit arithmetic over half a million,
// 3.6e-16 of the radius (7.3e-16 with log, cos and sin of the rounded angle).
constexpr int kLogFirst = 90, kLogCount = 91;   // j = 90 .. 180
// c = 128 / j rounded, and 2 ln c and 2 n ln 2 as multiples of 2^-40, whose sums
// are exact, with their remainders
static __device__ double2 d_bm_log[kLogCount];  // (c, 2 ln c high)
static __device__ double d_bm_log_lo[kLogCount];
static __device__ double2 d_bm_exp[34];
static __device__ double2 d_bm_trig[257];       // (cos, sin) 2 pi k / 256
// the same as pairs of float32 for the batched screens (float_pair.cuh)
static __device__ BmLog d_bmp_log[kBmCount];
static __device__ fpair d_bmp_exp[34];
static __device__ cpair d_bmp_trig[257];

int screens_init_device() {
  double2 lg[kLogCount], ex[34], tr[257];
  double lo[kLogCount];
  const auto high = [](long double v) { return rint((double)(v * 0x1p40L)) * 0x1p-40; };
  for (int j = 0; j < kLogCount; ++j) {
    const double c = 128.0 / (double)(kLogFirst + j);
    const long double l = 2.0L * logl((long double)c);
    lg[j] = make_double2(c, high(l));
    lo[j] = (double)(l - (long double)lg[j].y);
  }
  for (int n = 0; n < 34; ++n) {
    const long double l = 2.0L * n * logl(2.0L);
    ex[n].x = high(l);
    ex[n].y = (double)(l - (long double)ex[n].x);
  }
  for (int k = 0; k <= 256; ++k) {
    // reduced to an eighth of a turn: the argument's rounding stays below 2^-54
    const int a = k % 64, q = (k / 64) % 4;
    const double x = M_PI * (a <= 32 ? a : 64 - a) / 128.0;
    const double c = a <= 32 ? cos(x) : sin(x), s = a <= 32 ? sin(x) : cos(x);
    const double cq[4] = {c, -s, -c, s}, sq[4] = {s, c, -s, -c};
    tr[k] = make_double2(cq[q], sq[q]);
  }
  BmLog plg[kBmCount];
  fpair pex[34];
  cpair ptr[257];
  const auto pair = [](long double v) {
    const float h = (float)v;
    return fpair{h, (float)(v - (long double)h)};
  };
  for (int j = 0; j < kBmCount; ++j) {
    const double c = rint(128.0 / (double)(kBmFirst + j) * 2048.0) / 2048.0;
    const fpair l = pair(2.0L * logl((long double)c));
    plg[j] = BmLog{(float)c, l.h, l.l, 0.f};
  }
  for (int n = 0; n < 34; ++n) pex[n] = pair(2.0L * n * logl(2.0L));
  for (int k = 0; k <= 256; ++k) ptr[k] = cpair{pair(tr[k].x), pair(tr[k].y)};
  SPECULA_CK(cudaMemcpyToSymbol(d_bmp_log, plg, sizeof(plg)));
  SPECULA_CK(cudaMemcpyToSymbol(d_bmp_exp, pex, sizeof(pex)));
  SPECULA_CK(cudaMemcpyToSymbol(d_bmp_trig, ptr, sizeof(ptr)));
  SPECULA_CK(cudaMemcpyToSymbol(d_bm_log, lg, sizeof(lg)));
  SPECULA_CK(cudaMemcpyToSymbol(d_bm_log_lo, lo, sizeof(lo)));
  SPECULA_CK(cudaMemcpyToSymbol(d_bm_exp, ex, sizeof(ex)));
  SPECULA_CK(cudaMemcpyToSymbol(d_bm_trig, tr, sizeof(tr)));
  return SPECULA_OK;
}

// sqrt(-2 ln((x + 1/2) 2^-32)).  With m = 2 x + 1 = f 2^k, f in [1, 2) or, from
// 181/128 on, halved: -2 ln u = 2 (33 - k) ln 2 + 2 ln c - 2 ln(1 + r), r = f c - 1,
// c = 128 / j for the nearest j / 128 to f, |r| <= 0.5 / 90; near u = 1 both
// table terms are zero, so small results keep their relative accuracy.
__device__ __forceinline__ double bm_radius(uint32_t x) {
  const int k = 32 - __clz(x);   // bit length of x: m has its top bit there
  const uint64_t m = 2ull * x + 1ull;
  const uint64_t mant = (m << (52 - k)) & 0xFFFFFFFFFFFFFull;
  const int j1 = 128 + (((int)(mant >> 44) + 1) >> 1);
  const bool half = j1 > 180;
  const int j = half ? 64 + (((int)(mant >> 45) + 1) >> 1) : j1;
  const double f = __longlong_as_double((long long)(mant | ((half ? 1022ull : 1023ull) << 52)));
  const double2 cl = __ldg(d_bm_log + (j - kLogFirst));
  const double2 en = __ldg(d_bm_exp + (33 - k - (half ? 1 : 0)));
  const double lo = en.y + __ldg(d_bm_log_lo + (j - kLogFirst));
  const double r = fma(f, cl.x, -1.0), r2 = r * r;
  double p = fma(r, -2.0 / 7.0, 1.0 / 3.0);
  p = fma(r, p, -2.0 / 5.0);
  p = fma(r, p, 0.5);
  p = fma(r, p, -2.0 / 3.0);
  p = fma(r, p, 1.0);
  const double t = (en.x + cl.y) + fma(-2.0, r, fma(r2, p, lo));
  const double y = (double)rsqrtf((float)t);
  double g = t * y, h = 0.5 * y;
  const double e = fma(-g, h, 0.5);
  g = fma(g, e, g);
  h = fma(h, e, h);
  return fma(fma(-g, g, t), h, g);
}

// (cos, sin) of 2 pi (x + 1/2) 2^-32: the nearest k / 256 of a turn from the
// table, the rest |theta| <= pi / 256 by Taylor polynomials to theta^7
__device__ __forceinline__ double2 bm_angle(uint32_t x) {
  const uint32_t k = (uint32_t)(((uint64_t)x + (1u << 23)) >> 24);
  const int q = (int)(2ll * x + 1ll - ((long long)k << 25));   // 2^33 of a turn
  const double th = (__longlong_as_double(0x4338000000000000ll + q) - 6755399441055744.0) *
                    (2.0 * M_PI / 8589934592.0);
  const double2 cs = __ldg(d_bm_trig + k);
  const double t2 = th * th;
  const double s = fma(th * t2, fma(t2, fma(t2, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), th);
  const double c1 = t2 * fma(t2, fma(t2, -1.0 / 720.0, 1.0 / 24.0), -0.5);   // cos - 1
  return make_double2(fma(cs.x, c1, fma(-cs.y, s, cs.x)), fma(cs.y, c1, fma(cs.x, s, cs.y)));
}

// four standard normals for counter (pair index, sample, stream): words 0 / 1
// and 2 / 3, each (r cos, r sin)
__device__ __forceinline__ void normals4(uint64_t pair, uint32_t sample, uint32_t stream,
                                         uint64_t seed, double g[4]) {
  uint32_t c[4] = {(uint32_t)pair, (uint32_t)(pair >> 32), sample, stream};
  philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double r = bm_radius(c[2 * i]);
    const double2 a = bm_angle(c[2 * i + 1]);
    g[2 * i] = r * a.x;
    g[2 * i + 1] = r * a.y;
  }
}

// the same four normals as pairs of float32
__device__ __forceinline__ void normals4_pair(uint64_t pair, uint32_t sample, uint32_t stream,
                                              uint64_t seed, cpair g[2]) {
  uint32_t c[4] = {(uint32_t)pair, (uint32_t)(pair >> 32), sample, stream};
  philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const fpair r = bm_radius(c[2 * i], d_bmp_log, d_bmp_exp);
    const cpair a = bm_angle(c[2 * i + 1], d_bmp_trig);
    g[i] = cpair{fp_mul(r, a.re), fp_mul(r, a.im)};
  }
}

// n complex normals per sample: element 2i, 2i+1 from counter i
__global__ void k_rng_complex(uint64_t seed, int sample0, int stream_id, long long n,
                              double2 *__restrict__ out) {
  const long long pair = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  if (2 * pair >= n) return;
  double g[4];
  normals4((uint64_t)pair, (uint32_t)(sample0 + b), (uint32_t)stream_id, seed, g);
  out[(size_t)b * n + 2 * pair] = make_double2(g[0], g[1]);
  if (2 * pair + 1 < n) out[(size_t)b * n + 2 * pair + 1] = make_double2(g[2], g[3]);
}

// ---- batched screens ---------------------------------------------------------------
// The result is rounded to float32 once; until then values are pairs of float32
// (float_pair.cuh, about 48 bits; the tables are made in float64).  The float64
// rate, 2 fused multiply-adds per clock and SM, bounded the same passes in float64:
// 256 screens of 256^2 took 2.5 ms there (pass 1 1.63, pass 2 0.81); now 0.46 ms
// (0.55 while pass 2 took its columns in five dependent rounds of loads and their
// subharmonics in float64 on eight threads).
// Error against float64 unchanged to nine digits (2.5e-8 of the screen's norm, the
// final rounding; 0 to 15 values in a million round the other way).
//  * The spectral amplitude depends on (|kx|, |ky|) and not on the screen: one
//    quadrant table per call.  It is divided by a power of two that takes the
//    largest near 1, so that the pairs' exponents never leave their range; the
//    rounded result is multiplied by it again.
//  * Only the real part is wanted: Re IDFT(a) = IDFT(h), h the Hermitian part
//    of a, so the row transforms run for ky = 0 .. M/2 only and the column
//    transforms take two real columns at a time: half the transforms.
//  * The subharmonics are separable: per column nine products, per pixel six.
// Pass 1 (k_screen_rows) draws rows ky and -ky, combines and transforms them;
// pass 2 (k_screen_cols) transforms the columns, adds the subharmonics and
// rounds to float32 once.

__device__ __forceinline__ double2 dmul(double2 a, double2 w) {
  return make_double2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
}
__device__ __forceinline__ double2 dadd(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ cpair ldg_cpair(const cpair *p) {
  const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
  return cpair{{v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ void dft4(cpair (&x)[4]) {   // natural order, sign +
  const cpair a = cp_add(x[0], x[2]), b = cp_sub(x[0], x[2]);
  const cpair c = cp_add(x[1], x[3]), e = cp_sub(x[1], x[3]);
  x[0] = cp_add(a, c);
  x[2] = cp_sub(a, c);
  x[1] = cpair{fp_sub(b.re, e.im), fp_add(b.im, e.re)};
  x[3] = cpair{fp_add(b.re, e.im), fp_sub(b.im, e.re)};
}

// M = 2^LOGM point inverse DFT (sign +) of one vector by M/4 threads: radix-4 Stockham
// passes in place in buf, the values in registers between a pass's two barriers.  All
// threads of the CTA call it.  load(i): input i of the
// first pass, called before the first barrier; store(i, v): output i, called
// after the last barrier (every load and exchange of the CTA is done).  tw[m]
// = exp(2 pi i m / M).  Odd LOGM ends with a radix-2 pass.
template <int LOGM, class Load, class Store>
__device__ __forceinline__ void dft(cpair *buf, int t, const cpair *__restrict__ tw,
                                     Load load, Store store) {
  constexpr int M = 1 << LOGM, P4 = LOGM / 2;
  cpair x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) x[q] = load(t + q * (M / 4));
#pragma unroll
  for (int s = 0; s < P4; ++s) {
    const int L = 1 << (2 * s);
    const int k = t & (L - 1);
    if (s > 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = buf[t + q * (M / 4)];
#pragma unroll
      for (int q = 1; q < 4; ++q) x[q] = cp_mul(x[q], ldg_cpair(tw + q * k * (M / (4 * L))));
    }
    dft4(x);
    __syncthreads();   // every input of this pass is in registers
    if (s == P4 - 1 && LOGM % 2 == 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) store(t + q * (M / 4), x[q]);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) buf[(t - k) * 4 + k + q * L] = x[q];
      __syncthreads();
    }
  }
  if constexpr (LOGM % 2 == 1) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {   // L = M/2: output i and i + M/2 from inputs i, i + M/2
      const int i = t + h * (M / 4);
      x[2 * h] = buf[i];
      x[2 * h + 1] = cp_mul(buf[i + M / 2], ldg_cpair(tw + i));
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = t + h * (M / 4);
      store(i, cp_add(x[2 * h], x[2 * h + 1]));
      store(i + M / 2, cp_sub(x[2 * h], x[2 * h + 1]));
    }
  }
}

constexpr int kScrThreads = 256;
constexpr int kSubLevels = 3;

// small CTAs: the float64 work spreads over every SM (with 256 threads 27 us at M =
// 256, now 17; one warp per CTA in k_screen_sub_coef: 18.6 -> 12.2 us for 64 screens)
constexpr int kTabThreads = 64;
// tw[m] = exp(2 pi i m / M), m < M; per level p: sub[p][x] = exp(2 pi i x /
// (M 3^(p+1))), subp the same in pairs; amp[j][i] = inv_s sqrt(Phi) df / 2 at
// |ky| = j, |kx| = i <= M/2 (the half of the Hermitian part).
__global__ void __launch_bounds__(kTabThreads) k_screen_tables(cpair *__restrict__ tw,
                                                       double2 *__restrict__ sub,
                                                       cpair *__restrict__ subp,
                                                       fpair *__restrict__ amp, int M, double Md,
                                                       double coef, double k0, double inv_s) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int H = M / 2 + 1;
  if (e < M) {
    double sn, cs;
    sincospi(2.0 * (double)e / (double)M, &sn, &cs);
    tw[e] = cpair{fp_from(cs), fp_from(sn)};
    double w = 1.0;
    for (int p = 0; p < kSubLevels; ++p) {
      w *= 3.0;
      sincospi(2.0 * (double)e / ((double)M * w), &sn, &cs);
      sub[(size_t)p * M + e] = make_double2(cs, sn);
      subp[(size_t)p * M + e] = cpair{fp_from(cs), fp_from(sn)};
    }
  }
  if (e < H * H) {
    const double fx = (double)(e % H) / Md, fy = (double)(e / H) / Md;
    const double f2 = fx * fx + fy * fy;
    amp[e] = fp_from(
        f2 > 0.0 ? inv_s * (0.5 * (sqrt(coef * pow(f2 + k0, -11.0 / 6.0)) / Md)) : 0.0);
  }
}

// mean[p] = mean over x of sub[p][x]: one CTA per level, strided sums, then a
// fixed tree.
__global__ void __launch_bounds__(256) k_screen_sub_mean(const double2 *__restrict__ sub, int M,
                                                         double2 *__restrict__ mean) {
  __shared__ double2 s_v[256];
  double2 v = make_double2(0.0, 0.0);
  for (int x = threadIdx.x; x < M; x += 256) v = dadd(v, sub[(size_t)blockIdx.x * M + x]);
  s_v[threadIdx.x] = v;
  for (int o = 128; o > 0; o >>= 1) {
    __syncthreads();
    if (threadIdx.x < o) s_v[threadIdx.x] = dadd(s_v[threadIdx.x], s_v[threadIdx.x + o]);
  }
  if (threadIdx.x == 0) mean[blockIdx.x] = make_double2(s_v[0].x / M, s_v[0].y / M);
}

// One warp per screen: its 27 subharmonic coefficients (Philox stream 1,
// element e = (p * 3 + b) * 3 + a, frequencies (a - 1, b - 1) df / 3^(p+1))
// and the spatial mean of their sum.
__global__ void __launch_bounds__(32) k_screen_sub_coef(const double2 *__restrict__ mean,
                                                         double Md, double psd, double k0,
                                                         double inv_s, uint64_t seed, int sample0,
                                                         cpair *__restrict__ coef,
                                                         fpair *__restrict__ sub_mean) {
  __shared__ double2 s_c[28];
  const int lane = threadIdx.x, b = blockIdx.x;
  if (lane < 14) {
    double g[4];
    normals4((uint64_t)lane, (uint32_t)(sample0 + b), 1u, seed, g);
    s_c[2 * lane] = make_double2(g[0], g[1]);
    s_c[2 * lane + 1] = make_double2(g[2], g[3]);
  }
  __syncwarp();
  double m = 0.0;
  if (lane < 27) {
    const int p = lane / 9, bb = (lane / 3) % 3, a = lane % 3;
    const double df = 1.0 / (Md * (p == 0 ? 3.0 : (p == 1 ? 9.0 : 27.0)));
    const double fx = (a - 1) * df, fy = (bb - 1) * df, f2 = fx * fx + fy * fy;
    const double amp = f2 > 0.0 ? inv_s * (sqrt(psd * pow(f2 + k0, -11.0 / 6.0)) * df) : 0.0;
    const double2 c = make_double2(s_c[lane].x * amp, s_c[lane].y * amp);
    coef[(size_t)b * 27 + lane] = cpair{fp_from(c.x), fp_from(c.y)};
    const double2 e = mean[p];
    const double2 mx = a == 1 ? make_double2(1.0, 0.0) : make_double2(e.x, a == 2 ? e.y : -e.y);
    const double2 my = bb == 1 ? make_double2(1.0, 0.0) : make_double2(e.x, bb == 2 ? e.y : -e.y);
    const double2 mm = dmul(mx, my);
    m = c.x * mm.x - c.y * mm.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
  if (lane == 0) sub_mean[b] = fp_from(m);
}

template <int LOGM> struct ScrCfg {
  static constexpr int M = 1 << LOGM, H = M / 2 + 1;
  static constexpr int TPR = M / 4;                       // threads per transform
  // rows per CTA of pass 1
  static constexpr int RPB = TPR >= kScrThreads ? 1 : kScrThreads / TPR;
  static constexpr size_t smem1 = (size_t)RPB * 2 * M * sizeof(cpair);
  // pass 2: TB transforms per CTA, two columns each (eight columns give the
  // row tiles whole 128-byte lines; fewer where M/4 threads fill a CTA)
  static constexpr int TB0 = TPR >= 1024 ? 1 : (TPR >= 512 ? 2 : (TPR >= 64 ? 4 : 256 / TPR));
  static constexpr int TB = TB0 * 2 > M ? M / 2 : TB0;
  static constexpr int W = 2 * TB, LD = H | 1;
  static constexpr size_t smem2 =
      ((size_t)W * LD > (size_t)TB * M ? (size_t)W * LD : (size_t)TB * M) * sizeof(cpair) +
      (size_t)W * 10 * sizeof(fpair);
};

// Pass 1: rows ky = 0 .. M/2 of the Hermitian part, transformed along kx.
// grid (ceil(H / RPB), n_screens).
template <int LOGM>
__global__ void __launch_bounds__(ScrCfg<LOGM>::RPB *ScrCfg<LOGM>::TPR) k_screen_rows(
    const cpair *__restrict__ tw, const fpair *__restrict__ amp, uint64_t seed, int sample0,
    cpair *__restrict__ rows) {
  using C = ScrCfg<LOGM>;
  constexpr int M = C::M, TPR = C::TPR;
  extern __shared__ __align__(16) cpair sm_c[];
  const int v = threadIdx.x / TPR, t = threadIdx.x % TPR, b = blockIdx.y;
  const int ky = blockIdx.x * C::RPB + v;
  const bool ok = ky < C::H;
  cpair *c1 = sm_c + (size_t)v * 2 * M, *c2 = c1 + M;   // noise rows ky and -ky
  const int kyn = ky == 0 ? 0 : M - ky;
  if (ok) {
    for (int i = t; i < M; i += TPR) {   // M/2 counters per row, two rows
      const bool second = i >= M / 2;
      const int pr = second ? i - M / 2 : i;
      cpair g[2];
      normals4_pair((uint64_t)(second ? kyn : ky) * (M / 2) + pr, (uint32_t)(sample0 + b), 0u,
                    seed, g);
      cpair *d = (second ? c2 : c1) + 2 * pr;
      d[0] = g[0];
      d[1] = g[1];
    }
  }
  __syncthreads();
  const fpair *am = amp + (size_t)(ok ? ky : 0) * C::H;
  cpair *dst = rows + ((size_t)b * C::H + (ok ? ky : 0)) * M;
  dft<LOGM>(
      c1, t, tw,
      [&](int i) {
        const float2 a = __ldg(reinterpret_cast<const float2 *>(am + (i > M / 2 ? M - i : i)));
        const cpair p = c1[i], q = c2[i == 0 ? 0 : M - i];
        return cpair{fp_mul(fpair{a.x, a.y}, fp_add(p.re, q.re)),
                     fp_mul(fpair{a.x, a.y}, fp_sub(p.im, q.im))};
      },
      [&](int i, cpair z) {
        if (ok) dst[i] = z;
      });
}

// Pass 2: W columns of one screen, two at a time.  grid (M / W, n_screens).
template <int LOGM>
__global__ void __launch_bounds__(ScrCfg<LOGM>::TB *ScrCfg<LOGM>::TPR) k_screen_cols(
    const cpair *__restrict__ rows, const cpair *__restrict__ tw,
    const cpair *__restrict__ subp, const cpair *__restrict__ coef,
    const fpair *__restrict__ sub_mean, float s1, float s2, float *__restrict__ out) {
  using C = ScrCfg<LOGM>;
  constexpr int M = C::M, TPR = C::TPR, W = C::W, LD = C::LD, NT = C::TB * TPR;
  extern __shared__ __align__(16) cpair sm_c[];
  const int v = threadIdx.x / TPR, t = threadIdx.x % TPR, b = blockIdx.y;
  const int x0 = blockIdx.x * W;
  fpair *s_sub = reinterpret_cast<fpair *>(
      sm_c + ((size_t)W * LD > (size_t)C::TB * M ? (size_t)W * LD : (size_t)C::TB * M));
  // the columns' half spectra, column-major: four loads of a thread in flight, and
  // the row M/2
  const cpair *src = rows + (size_t)b * C::H * M + x0;
  cpair in[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int e = threadIdx.x + i * NT;
    in[i] = src[(size_t)(e / W) * M + e % W];
  }
  if (threadIdx.x < W) sm_c[(size_t)threadIdx.x * LD + M / 2] = src[(size_t)(M / 2) * M + threadIdx.x];
  // column x's subharmonics: s_sub[c][2p] cos + s_sub[c][2p + 1] sin of level
  // p's row phase, plus s_sub[c][6], the sum of the levels' s_k[c]
  fpair *s_k = s_sub + W * 7;
  for (int i = threadIdx.x; i < kSubLevels * W; i += NT) {
    const int c = i % W, p = i / W;
    const cpair *cf = coef + (size_t)b * 27 + p * 9;
    const cpair e = ldg_cpair(subp + (size_t)p * M + x0 + c), en = cpair{e.re, fp_neg(e.im)};
    cpair G[3];
#pragma unroll
    for (int bb = 0; bb < 3; ++bb) {
      const cpair *q = cf + bb * 3;
      G[bb] = cp_add(cp_mul(ldg_cpair(q), en), cp_mul(ldg_cpair(q + 2), e));
      if (bb != 1) G[bb] = cp_add(G[bb], ldg_cpair(q + 1));
    }
    const fpair sc = fp_add(G[2].re, G[0].re), ss = fp_sub(G[0].im, G[2].im);
    s_sub[c * 7 + 2 * p] = fp_norm(sc.h, sc.l);
    s_sub[c * 7 + 2 * p + 1] = fp_norm(ss.h, ss.l);
    s_k[c * kSubLevels + p] = G[1].re;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int e = threadIdx.x + i * NT;
    sm_c[(size_t)(e % W) * LD + e / W] = in[i];
  }
  __syncthreads();
  if (threadIdx.x < W) {   // read after the transforms' barriers
    fpair k = fp_neg(sub_mean[b]);
#pragma unroll
    for (int p = 0; p < kSubLevels; ++p) k = fp_add(k, s_k[threadIdx.x * kSubLevels + p]);
    s_sub[threadIdx.x * 7 + 6] = fp_norm(k.h, k.l);
  }
  const cpair *r1 = sm_c + (size_t)(2 * v) * LD, *r2 = r1 + LD;
  const fpair *u1 = s_sub + (2 * v) * 7, *u2 = u1 + 7;
  float *tile = reinterpret_cast<float *>(sm_c);
  constexpr int TLD = M + 1;
  dft<LOGM>(
      sm_c + (size_t)v * M, t, tw,
      [&](int i) {
        if (i == 0 || i == M / 2) return cpair{r1[i].re, r2[i].re};
        const int k = i < M / 2 ? i : M - i;
        const cpair a = r1[k], c = r2[k];
        // conjugates above M/2
        return i < M / 2 ? cpair{fp_sub(a.re, c.im), fp_add(a.im, c.re)}
                         : cpair{fp_add(a.re, c.im), fp_sub(c.re, a.im)};
      },
      [&](int y, cpair z) {
        fpair v1 = fp_add(z.re, u1[6]), v2 = fp_add(z.im, u2[6]);
#pragma unroll
        for (int p = 0; p < kSubLevels; ++p) {
          const cpair e = ldg_cpair(subp + (size_t)p * M + y);
          v1 = fp_add(v1, fp_dot(u1[2 * p], e.re, u1[2 * p + 1], e.im));
          v2 = fp_add(v2, fp_dot(u2[2 * p], e.re, u2[2 * p + 1], e.im));
        }
        tile[(2 * v) * TLD + y] = __fadd_rn(v1.h, v1.l) * s1 * s2;
        tile[(2 * v + 1) * TLD + y] = __fadd_rn(v2.h, v2.l) * s1 * s2;
      });
  __syncthreads();
  float *dst = out + (size_t)b * M * M + x0;
  for (int e = threadIdx.x; e < M * W; e += NT) {
    const int c = e % W, y = e / W;
    dst[(size_t)y * M + c] = tile[c * TLD + y];
  }
}

// Bytes of the half spectra of one screen, and the most a group of screens
// takes: a group stays in L2 between the two passes.
static size_t screen_bytes(int M) { return (size_t)(M / 2 + 1) * M * sizeof(cpair); }
constexpr size_t kScreenGroupBytes = (size_t)80 << 20;

template <int LOGM>
static int screen_batch(specula_ctx *ctx, int n_screens, double pitch_m, double r0_m, double L0_m,
                        uint64_t seed, int sample0, float *out, cudaStream_t st) {
  using C = ScrCfg<LOGM>;
  constexpr int M = C::M, H = C::H;
  const double Md = (double)M * pitch_m;
  const double coef = 0.023 * pow(r0_m, -5.0 / 3.0);
  const double k0 = isinf(L0_m) ? 0.0 : 1.0 / (L0_m * L0_m);
  const int groups = (int)(((size_t)n_screens * screen_bytes(M) + kScreenGroupBytes - 1) /
                           kScreenGroupBytes);
  const int G = std::min(n_screens, std::max(1, (n_screens + groups - 1) / groups));
  // the power of two that takes the largest amplitude to [1, 2), in two factors
  // of at most 2^126
  int ex = 0;
  frexp(0.5 * sqrt(coef * pow(1.0 / (Md * Md) + k0, -11.0 / 6.0)) / Md, &ex);
  ex = std::max(-252, std::min(252, ex - 1));
  const double inv_s = ldexp(1.0, -ex);
  const float s1 = (float)ldexp(1.0, ex / 2), s2 = (float)ldexp(1.0, ex - ex / 2);
  // workspace, kept by the context: half spectra, twiddles, subharmonic row
  // phases (in pairs and in float64) and their means, coefficients, amplitude
  // quadrant; entries of 16 bytes but the last two
  static_assert(sizeof(cpair) == sizeof(double2) && sizeof(fpair) == sizeof(double), "");
  const size_t nd2 = (size_t)G * H * M + M + (size_t)2 * kSubLevels * M + 4 + (size_t)G * 27;
  const size_t need = nd2 * sizeof(double2) + ((size_t)G + (size_t)H * H) * sizeof(double);
  int s;
  if (ctx->screen_ws.bytes < need && (s = ctx->screen_ws.alloc(need))) return s;
  cpair *rows = ctx->screen_ws.as<cpair>(), *tw = rows + (size_t)G * H * M, *subp = tw + M;
  double2 *sub = reinterpret_cast<double2 *>(subp + (size_t)kSubLevels * M);
  double2 *mean = sub + (size_t)kSubLevels * M;
  cpair *cf = reinterpret_cast<cpair *>(mean + 4);
  fpair *sm = reinterpret_cast<fpair *>(cf + (size_t)G * 27), *amp = sm + G;
  if ((s = ensure_dynamic_smem((const void *)k_screen_rows<LOGM>, C::smem1)) ||
      (s = ensure_dynamic_smem((const void *)k_screen_cols<LOGM>, C::smem2)))
    return s;
  SPECULA_LAUNCH(ctx, SPECULA_K_CALIB, st,
                 k_screen_tables<<<(std::max(H * H, M) + kTabThreads - 1) / kTabThreads, kTabThreads, 0, st>>>(
                     tw, sub, subp, amp, M, Md, coef, k0, inv_s));
  SPECULA_LAUNCH(ctx, SPECULA_K_CALIB, st,
                 k_screen_sub_mean<<<kSubLevels, 256, 0, st>>>(sub, M, mean));
  for (int g0 = 0; g0 < n_screens; g0 += G) {
    const int ng = std::min(G, n_screens - g0);
    SPECULA_LAUNCH(ctx, SPECULA_K_CALIB, st,
                   k_screen_sub_coef<<<ng, 32, 0, st>>>(mean, Md, coef, k0, inv_s, seed, sample0 + g0,
                                                       cf, sm));
    SPECULA_LAUNCH(ctx, SPECULA_K_CALIB, st,
                   k_screen_rows<LOGM><<<dim3((H + C::RPB - 1) / C::RPB, ng), C::RPB * C::TPR,
                                         C::smem1, st>>>(tw, amp, seed, sample0 + g0, rows));
    SPECULA_LAUNCH(ctx, SPECULA_K_CALIB, st,
                   k_screen_cols<LOGM><<<dim3(M / C::W, ng), C::TB * C::TPR, C::smem2, st>>>(
                       rows, tw, subp, cf, sm, s1, s2, out + (size_t)g0 * M * M));
  }
  // the workspace is the context's, whatever stream its next call runs on
  SPECULA_CK(cudaStreamSynchronize(st));
  return SPECULA_OK;
}

// phase[b][j][i] = scale[b] * screen[b][j + o][i + o], o = (side - n) / 2
__global__ void k_random_phase(const float *__restrict__ scr, int side, int n,
                               const float *__restrict__ scale, float *__restrict__ phase) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, b = blockIdx.z;
  if (i >= n) return;
  const int o = (side - n) / 2;
  phase[((size_t)b * n + j) * n + i] =
      scale[b] * scr[((size_t)b * side + j + o) * side + i + o];
}

}  // namespace specula

using namespace specula;

static double psd_host(double fx, double fy, double r0, double L0) {
  const double f2 = fx * fx + fy * fy;
  if (!(f2 > 0)) return 0.0;
  const double k0 = isinf(L0) ? 0.0 : 1.0 / (L0 * L0);
  return 0.023 * pow(r0, -5.0 / 3.0) * pow(f2 + k0, -11.0 / 6.0);
}

extern "C" int specula_screen_generate(specula_ctx *ctx, int32_t side, double pitch_m,
                                       double r0_m, double L0_m, const double *noise_dev,
                                       const double *noise_sub_host, float *screen_dev,
                                       void *stream) {
  if (!ctx || !noise_dev || !noise_sub_host || !screen_dev) return SPECULA_EINVAL;
  if (side < 32 || side > 4096 || (side & (side - 1))) return SPECULA_EINVAL;
  if (!(pitch_m > 0) || !(r0_m > 0) || !(L0_m > 0)) return SPECULA_EINVAL;
  SPECULA_CK(cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  const int M = side;
  int logM = 0;
  while ((1 << logM) < M) ++logM;
  const double Md = (double)M * pitch_m;
  const double df = 1.0 / Md;
  const double coef = 0.023 * pow(r0_m, -5.0 / 3.0);
  const double k0 = isinf(L0_m) ? 0.0 : 1.0 / (L0_m * L0_m);
  const int levels = 3;

  // host tables: FFT twiddles exp(+2 pi i k / M); subharmonic exponentials and
  // coefficients; the spatial mean of the subharmonic sum
  std::vector<double2> tw(M / 2);
  for (int k = 0; k < M / 2; ++k) {
    const double a = 2.0 * M_PI * (double)k / (double)M;
    tw[k] = make_double2(cos(a), sin(a));
  }
  std::vector<double2> tab((size_t)levels * 3 * M), coefs(levels * 9);
  std::vector<double2> tmean(levels * 3);
  double sub_mean = 0.0;
  for (int p = 0; p < levels; ++p) {
    const double dfp = df / pow(3.0, p + 1);
    for (int a = 0; a < 3; ++a) {
      const double f = (a - 1) * dfp;
      double sr = 0, si = 0;
      for (int x = 0; x < M; ++x) {
        const double ang = 2.0 * M_PI * f * ((double)x * pitch_m);
        const double2 e = make_double2(cos(ang), sin(ang));
        tab[((size_t)p * 3 + a) * M + x] = e;
        sr += e.x;
        si += e.y;
      }
      tmean[p * 3 + a] = make_double2(sr / M, si / M);
    }
    for (int b = 0; b < 3; ++b)
      for (int a = 0; a < 3; ++a) {
        double2 c = make_double2(0, 0);
        if (!(a == 1 && b == 1)) {
          const double amp = sqrt(psd_host((a - 1) * dfp, (b - 1) * dfp, r0_m, L0_m)) * dfp;
          const double *n = noise_sub_host + 2 * ((p * 3 + b) * 3 + a);
          c = make_double2(n[0] * amp, n[1] * amp);
          const double2 mx = tmean[p * 3 + a], my = tmean[p * 3 + b];
          const double2 e = make_double2(mx.x * my.x - mx.y * my.y, mx.x * my.y + mx.y * my.x);
          sub_mean += c.x * e.x - c.y * e.y;
        }
        coefs[(p * 3 + b) * 3 + a] = c;
      }
  }

  DevBuf A, B, dtw, dtab, dcoef;
  int s;
  if ((s = A.alloc((size_t)M * M * sizeof(double2)))) return s;
  if ((s = B.alloc((size_t)M * M * sizeof(double2)))) return s;
  if ((s = dtw.upload(tw.data(), tw.size() * sizeof(double2)))) return s;
  if ((s = dtab.upload(tab.data(), tab.size() * sizeof(double2)))) return s;
  if ((s = dcoef.upload(coefs.data(), coefs.size() * sizeof(double2)))) return s;

  k_psd_weight<<<dim3((M + 255) / 256, M), 256, 0, st>>>((const double2 *)noise_dev,
                                                          A.as<double2>(), M, Md, coef, k0);
  SPECULA_CK_LAUNCH();
  const size_t sm = 2 * (size_t)M * sizeof(double2);
  if ((s = ensure_dynamic_smem((const void *)k_fft_rows_f64, sm))) return s;
  k_fft_rows_f64<<<M, 256, sm, st>>>(A.as<double2>(), dtw.as<double2>(), M, logM);
  SPECULA_CK_LAUNCH();
  k_transpose_f64<<<dim3(M / 32, M / 32), dim3(32, 8), 0, st>>>(A.as<double2>(), B.as<double2>(), M);
  SPECULA_CK_LAUNCH();
  k_fft_rows_f64<<<M, 256, sm, st>>>(B.as<double2>(), dtw.as<double2>(), M, logM);
  SPECULA_CK_LAUNCH();
  k_screen_final<<<dim3(M / 32, M / 32), dim3(32, 8), 0, st>>>(
      B.as<double2>(), dtab.as<double2>(), dcoef.as<double2>(), sub_mean, M, levels, screen_dev);
  SPECULA_CK_LAUNCH();
  // the temporaries are freed on return; wait for the kernels that use them
  SPECULA_CK(cudaStreamSynchronize(st));
  return SPECULA_OK;
}

extern "C" int specula_rng_complex(specula_ctx *ctx, uint64_t seed, int32_t sample0,
                                   int32_t n_samples, int32_t stream_id, int64_t n_per_sample,
                                   double *out_dev, void *stream) {
  if (!ctx || !out_dev || n_samples < 1 || n_per_sample < 1 || sample0 < 0 || stream_id < 0)
    return SPECULA_EINVAL;
  if (n_samples > 65535) return SPECULA_EUNSUPPORTED;
  const long long pairs = (n_per_sample + 1) / 2;
  dim3 grid((unsigned)((pairs + 255) / 256), n_samples);
  cudaStream_t st = (cudaStream_t)stream;
  SPECULA_LAUNCH(ctx, SPECULA_K_CALIB, st,
                 k_rng_complex<<<grid, 256, 0, st>>>(seed, sample0, stream_id, n_per_sample,
                                                     (double2 *)out_dev));
  return SPECULA_OK;
}

extern "C" int specula_screen_generate_batch(specula_ctx *ctx, int32_t n_screens, int32_t side,
                                             double pitch_m, double r0_m, double L0_m,
                                             uint64_t seed, int32_t sample0, float *screens_dev,
                                             void *stream) {
  if (!ctx || !screens_dev || n_screens < 1 || sample0 < 0) return SPECULA_EINVAL;
  if (side < 32 || side > 4096 || (side & (side - 1))) return SPECULA_EINVAL;
  if (!(pitch_m > 0) || !(r0_m > 0) || !(L0_m > 0)) return SPECULA_EINVAL;
  SPECULA_CK(cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  switch (side) {
#define SPECULA_SCREENS(LOGM_)                                                                 \
  case 1 << LOGM_:                                                                             \
    return screen_batch<LOGM_>(ctx, n_screens, pitch_m, r0_m, L0_m, seed, sample0, screens_dev, \
                               st)
    SPECULA_SCREENS(5);
    SPECULA_SCREENS(6);
    SPECULA_SCREENS(7);
    SPECULA_SCREENS(8);
    SPECULA_SCREENS(9);
    SPECULA_SCREENS(10);
    SPECULA_SCREENS(11);
    SPECULA_SCREENS(12);
#undef SPECULA_SCREENS
    default: return SPECULA_EINVAL;
  }
}

extern "C" int specula_random_phase(specula_ctx *ctx, const float *screens_dev, int32_t n,
                                    int32_t side, int32_t n_pix, const float *scale_dev,
                                    float *phase_dev, void *stream) {
  if (!ctx || !screens_dev || !scale_dev || !phase_dev || n < 1 || n_pix < 1 || side < n_pix)
    return SPECULA_EINVAL;
  if (n > 65535) return SPECULA_EUNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  dim3 grid((n_pix + 127) / 128, n_pix, n);
  SPECULA_LAUNCH(ctx, SPECULA_K_ATMO, st,
                 k_random_phase<<<grid, 128, 0, st>>>(screens_dev, side, n_pix, scale_dev,
                                                      phase_dev));
  return SPECULA_OK;
}

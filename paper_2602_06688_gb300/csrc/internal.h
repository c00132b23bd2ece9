// Internal declarations shared by the translation units of libspecula_gb300.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <memory>
#include <utility>
#include <vector>

#include "../../include/specula_gb300.h"

namespace specula {
// the CUDA error behind the calling thread's last SPECULA_ECUDA (api.cu)
void note_cuda_error(cudaError_t e, const char *file, int line);
}

#define SPECULA_CK(call)                                   \
  do {                                                     \
    cudaError_t e_ = (call);                               \
    if (e_ != cudaSuccess) {                               \
      specula::note_cuda_error(e_, __FILE__, __LINE__);    \
      return SPECULA_ECUDA;                                \
    }                                                      \
  } while (0)

#define SPECULA_CK_LAUNCH()                                \
  do {                                                     \
    cudaError_t e_ = cudaGetLastError();                   \
    if (e_ != cudaSuccess) {                               \
      specula::note_cuda_error(e_, __FILE__, __LINE__);    \
      return SPECULA_ECUDA;                                \
    }                                                      \
  } while (0)

namespace specula {

// Every buffer the library allocates carries kGuardBytes of a fixed pattern
// past its end.  A kernel that writes past its workspace lands there rather
// than in a neighbouring allocation, which would not fault;
// specula_check_guards compares the bands (api.cu keeps the live buffers).
constexpr size_t kGuardBytes = 256;
constexpr unsigned char kGuardByte = 0xA5;
struct DevBuf;
void guard_register(DevBuf *b);
void guard_unregister(DevBuf *b);

// A device buffer owned by a plan.
struct DevBuf {
  void *p = nullptr;
  size_t bytes = 0;
  int device = -1;
  DevBuf() = default;
  DevBuf(const DevBuf &) = delete;
  DevBuf &operator=(const DevBuf &) = delete;
  ~DevBuf() { release(); }
  void release() {
    if (!p) return;
    guard_unregister(this);
    cudaFree(p);
    p = nullptr;
  }
  int alloc(size_t n) {
    release();
    bytes = n;
    if (n == 0) return SPECULA_OK;
    if (cudaMalloc(&p, n + kGuardBytes) != cudaSuccess) {
      p = nullptr;
      return SPECULA_ENOMEM;
    }
    if (cudaGetDevice(&device) != cudaSuccess ||
        cudaMemset(static_cast<char *>(p) + n, kGuardByte, kGuardBytes) != cudaSuccess) {
      cudaFree(p);
      p = nullptr;
      return SPECULA_ECUDA;
    }
    guard_register(this);
    return SPECULA_OK;
  }
  int upload(const void *h, size_t n) {
    int s = alloc(n);
    if (s) return s;
    return cudaMemcpy(p, h, n, cudaMemcpyHostToDevice) == cudaSuccess ? SPECULA_OK : SPECULA_ECUDA;
  }
  template <class T> T *as() const { return static_cast<T *>(p); }
};

// Pyramid plan: tables and the per-chunk intermediate workspace.
struct PwfsPlan {
  int n_pix, pad, n_mod, n_sub, pup_dist;
  double mod_amp;
  int N, N1, N2;
  int chunk;            // modulation items per pipeline chunk
  int ka;               // items per row group in the row-forward pass
  int nbw;              // field slots: batch elements one chunk can touch
  int blockA, blockB, blockC;
  size_t smemA, smemB, smemC;
  int passes;           // 2: row filter + column filter/bins; 3: rows, cols, rows
  int nc;               // row-filter slots per batch element (distinct cosines)
  int slot_lo = 0;      // cosine slots [slot_lo, slot_hi) imaged (slot_hi < 0: all)
  int slot_hi = -1;
  bool two_ok;          // the two-pass form fits this geometry
  int G = 32;           // lanes per transform of the split N1 x N2
  int M1 = 0, M2 = 0;   // the two-pass form's split of N
  int blockR, blockK;   // two-pass blocks
  size_t smemR, smemK;
  int tcK = 0;          // columns of a column-pass tile
  // a detector pixel is fp / fq grid pixels (N / (pad n_sub) in lowest
  // terms; fq = 1: fp x fp binning, else area-weighted rebinning)
  int fp = 1, fq = 1;
  DevBuf gx, gy;        // [n_mod][n_pix] float2: tilt x pre-phase (x and y parts)
  DevBuf mask;          // [N] float2: pyramid mask factor per axis, x (1/N)
  DevBuf twA, twB;      // [N] float2: inter-step twiddles (cos, sin)
  DevBuf tpA, tpB;      // the same for the two-pass form's split
  DevBuf field;         // [nbw][n_pix][n_pix] float2: E = amp exp(i phase)
  DevBuf rows;          // [chunk][n_pix][N] float2: after the row transform
  DevBuf cols;          // [chunk][N][N] float2: after the column pass (three-pass form)
  DevBuf part;          // [chunk][nd][nd] float: binned intensity per item
  // per-call settings of the polychromatic image (defaults: a plain image):
  // the phase is multiplied by run_phase_scale and the detector becomes
  // run_beta det + run_alpha image
  float run_phase_scale = 1.f, run_alpha = 1.f, run_beta = 0.f;
  // shifted-mask form (SPECULA_PWFS_FORM_SHIFTED)
  int form = 0;
  int sm_blockK = 0, sm_chunk = 0;
  size_t sm_smemK = 0, sm_smemR = 0, sm_smemC = 0;
  DevBuf sm_pre;        // [Np] float2: centred-DFT input phase over the pupil
  DevBuf sm_mx, sm_my;  // [nc][N], [n_mod][N] float2: shifted mask factors / N
  DevBuf sm_frows;      // [Np][N] float2: after the forward row transform
  DevBuf sm_fspec;      // [N][N] float2: the field's spectrum
  DevBuf sm_rows;       // [sm_chunk][N][N] float2 (+2): after the inverse row transform
  DevBuf sm_part;       // [n_mod][nd][nd] float: binned intensity per point
  // two-pass form with packed-pair arithmetic (passes == 4, pwfs_pair.cu)
  bool pair_ok = false;
  int pair_blockR = 0, pair_blockK = 0;
  size_t pair_smemR = 0, pair_smemK = 0;
  DevBuf twA2, twB2;    // [N] float4 (re, re, im, im): inter-step twiddles
  DevBuf mask2;         // [N] float4: mask factor per axis, x (1/N)
  DevBuf gx2;           // [n_mod][n_pix] float4: x factor of the tilt x pre-phase
  DevBuf pair_units;    // [n_pair_units] int4: (slot a, point a, slot b, point b or -1)
  DevBuf gyp;           // [n_pair_units][n_pix] float4: the units' y factors (re_a, re_b, im_a, im_b)
  int n_pair_units = 0;
  int pair_units_for = -1;   // the slot range the unit table was built for
  std::vector<float2> gy_host;
  // DFT-as-GEMM forms (pwfs_dftgemm.cu)
  int dg_form = -1;     // the form the operator below was built for
  int dg_M1 = 0, dg_M2 = 0;
  DevBuf dg_B;          // [2N][6 n_pix] split operator (bf16 or float32/tf32)
  DevBuf dg_A1, dg_A2;  // split operands of the row and column GEMMs
  DevBuf dg_C1, dg_C2;  // [M][2N] float32 products
  DevBuf dg_work;       // split-K partials of the row GEMM
};

struct ShPlan {
  int n_pix, n_sub, sub_pix, fft_n;
  double obsc = 0.0;   // the pupil's obscuration (the valid list depends on it)
  int n_valid;
  int sub_lo = 0, sub_hi = -1;   // imaged valid subapertures [sub_lo, sub_hi) (-1: all)
  DevBuf valid;         // [n_valid] int32
  DevBuf pre;           // [fft_n] float2: centred-DFT input phase
  DevBuf tw;            // [fft_n] float2 twiddles
};

}  // namespace specula

// capacity of the per-context extraction coordinate table
#define SPECULA_ATMO_MAX_LAYERS 64
#define SPECULA_ATMO_MAX_PIX 8192

struct specula_ctx {
  int device = 0;
  int32_t *status_dev = nullptr;
  double *loop_part = nullptr;      // [kLoopMaxBlocks][5] closed-loop statistics partials
  bool guard = true;                // slope kernels record non-finite outputs
  int *atmo_tab_i = nullptr;        // [64][2][8192] screen sample index
  float *atmo_tab_f = nullptr;      // [64][2][8192] interpolation fraction
  std::vector<std::unique_ptr<specula::PwfsPlan>> pwfs;
  std::vector<std::unique_ptr<specula::ShPlan>> sh;
  // tracing: kernels launched, and optional per-kernel CUDA-event pairs
  int64_t launches = 0;
  bool prof = false;
  std::vector<cudaEvent_t> ev;      // 2 per record
  size_t ev_next = 0;
  std::vector<int> rec_kid;         // kernel id of record i (events 2i, 2i+1)
  // batched bf16 reconstructor products: the slopes' bf16 halves and the
  // split-K partials (grown on demand outside stream capture)
  specula::DevBuf recon_ws;
  // one wavelength's spots of the polychromatic Shack-Hartmann (grown on
  // demand outside stream capture)
  specula::DevBuf sh_poly_ws;
  // batched screens: half spectra of one group, and the call's tables (grown
  // on demand; at most 80 MB of spectra, or one screen's)
  specula::DevBuf screen_ws;
};

namespace specula {

// Bracket one kernel launch with events on its stream when tracing is on.
inline int prof_begin(specula_ctx *c, cudaStream_t st) {
  c->launches++;
  if (!c->prof || c->ev_next + 2 > c->ev.size()) return -1;
  const int slot = (int)c->ev_next;
  c->ev_next += 2;
  cudaEventRecord(c->ev[slot], st);
  return slot;
}
inline void prof_end(specula_ctx *c, int slot, int kid, cudaStream_t st) {
  if (slot < 0) return;
  cudaEventRecord(c->ev[slot + 1], st);
  c->rec_kid.push_back(kid);   // capacity reserved when tracing is enabled
}

#define SPECULA_LAUNCH(ctx, kid, st, ...)            \
  do {                                               \
    const int slot_ = prof_begin((ctx), (st));       \
    __VA_ARGS__;                                     \
    SPECULA_CK_LAUNCH();                             \
    prof_end((ctx), slot_, (kid), (st));             \
  } while (0)

// Programmatic dependent launch, for the per-frame kernels: a kernel launched
// with SPECULA_LAUNCH_PDL may be scheduled once every CTA of the kernel before
// it on the stream has left, before that kernel's completion is signalled, so
// its launch and its CTAs' start overlap that kernel's end.  It touches memory
// only after pdl_wait, which ends when the kernel before has completed and
// its writes are visible.  Every kernel so launched calls pdl_wait in every
// thread before its first access and before any return: a kernel then
// completes only after the one before it, and what it waits for includes
// everything earlier on the stream.
// Measured: 8 m frame (a graph of eight kernels) 38.9 -> 36.9 us, 39 m frame
// 249.3 -> 248.4, closed-loop step 66.3 -> 65.0, SOUL image (eager) 67.7 ->
// 59.4, learned inference 26.7 -> 19.5 us, sixteen training steps 4.5 -> 3.5
// ms.  Letting the next kernel start as soon as every CTA has begun
// (griddepcontrol.launch_dependents first) was slower: its waiting CTAs hold
// slots and registers (39 m frame 258.4, step 70.9, inference 20.6 us).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel's CTAs start once every CTA of this one has called it or
// left: for short kernels in front of one that prefetches.
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// `bytes` (a multiple of 16) from p (16-byte aligned) on their way to L2.  A hint
// without a value, so it may stand before pdl_wait for memory that an earlier
// kernel may still write.
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
template <class... P, class... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, int cluster, A &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 0 ? 2 : 1;   // 0: no cluster
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}
#define SPECULA_LAUNCH_PDL(ctx, kid, st, kernel, grid, block, smem, ...)                       \
  SPECULA_LAUNCH((ctx), (kid), (st),                                                           \
                 SPECULA_CK(launch_pdl(kernel, (grid), (block), (smem), (st), 0, __VA_ARGS__)))

// per-translation-unit device initialisation (constant tables)
int pwfs_init_device();
int screens_init_device();
int sh_init_device();
int mwfs_init_device();
// float64 helpers of the calibration file, shared with the infinite screens:
// C[i][j] = sum_k X(i,k) d(k) Y(k,j), X(i,k) = X[i xi + k xk], Y(k,j) = Y[k yk + j yj]
// (d may be NULL); and the Jacobi eigen-decomposition of a symmetric matrix
// (eigenvalues on G's diagonal, eigenvectors in V's columns).
int gemm_f64(specula_ctx *ctx, cudaStream_t st, const double *X, long xi, long xk,
             const double *Y, long yk, long yj, const double *d, double *C, int M, int N, int K);
int sym_eig_f64(specula_ctx *ctx, cudaStream_t st, double *G, double *V, int n);
constexpr int kLoopMaxBlocks = 512;
int loop_alloc_workspace(specula_ctx *ctx);
int pwfs_shifted_init_device();
int pwfs_shifted_prepare(PwfsPlan *p);
int pwfs_shifted_run(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase,
                     int n_batch, float *det, cudaStream_t st);
int pwfs_bin_reduce(specula_ctx *ctx, const float *part, float *det, int nd2, int n_mod,
                    float alpha, float beta, cudaStream_t st);
// the field of batch elements fb .. fb + nb - 1 into the plan's field slots,
// and their detectors from the plan's per-point bins
int pwfs_field_launch(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase,
                      int fb, int nb, cudaStream_t st);
int pwfs_bin_reduce_range(specula_ctx *ctx, PwfsPlan *p, float *det, int nd2, int b0, int nb,
                          cudaStream_t st);
struct PwfsTablesHost;
int pwfs_pair_init_device();
int pwfs_dftgemm_prepare(PwfsPlan *p, int form);
int pwfs_dftgemm_run(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase,
                     int n_batch, float *det, cudaStream_t st);
int pwfs_pair_configure(PwfsPlan *p);
int pwfs_pair_tables(PwfsPlan *p, const PwfsTablesHost &T);
int pwfs_pair_run(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase,
                  int n_batch, float *det, cudaStream_t st);
int atmo_alloc_tables(specula_ctx *ctx);

// launchers implemented in the kernel translation units
int pwfs_plan_build(specula_ctx *ctx, const specula_pupil_desc *pupil,
                    const specula_pwfs_desc *pwfs, PwfsPlan **out);
PwfsPlan *pwfs_plan_find(specula_ctx *ctx, const specula_pupil_desc *pupil,
                         const specula_pwfs_desc *pwfs);
int pwfs_set_tiles(PwfsPlan *p, int chunk, int ka, int passes);
int pwfs_autotune(specula_ctx *ctx, PwfsPlan *p, const float *amp, const float *phase,
                  int n_batch, float *det, cudaStream_t st, int reps, size_t max_ws_bytes,
                  int *best_chunk, int *best_ka, int *best_passes);
int pwfs_run(specula_ctx *ctx, PwfsPlan *plan, const float *amp, const float *phase,
             int n_batch, float *det, cudaStream_t st);
int sh_plan_build(specula_ctx *ctx, const specula_pupil_desc *pupil,
                  const specula_sh_desc *sh, ShPlan **out);
ShPlan *sh_plan_find(specula_ctx *ctx, const specula_pupil_desc *pupil,
                     const specula_sh_desc *sh);
int sh_run(specula_ctx *ctx, ShPlan *plan, const float *amp, const float *phase,
           int n_batch, float *spots, cudaStream_t st, float phase_scale = 1.0f);
// out = (first ? 0 : out) + weight ratio^2 W spots W^T for n_spots fft_n^2
// spots of one wavelength (ratio = lambda_ref / lambda): the polychromatic SH
int sh_poly_acc(specula_ctx *ctx, int fft_n, const float *spots, int n_spots, double ratio,
                double weight, bool first, float *out, cudaStream_t st);

// Raise (never lower) a kernel's dynamic shared-memory limit to `bytes` on
// the current device.  The limit belongs to the function, shared by every
// plan that launches it, so a later plan with a smaller need must not shrink
// what an earlier one relies on.  Needs up to 48 KB need no call.
int ensure_dynamic_smem(const void *fn, size_t bytes);

int gemm_check(const void *A, const void *B, int M, int N, int K, bool tf32 = false);
int gemm_splits(int K, int want, bool tf32 = false);
int gemm_tf32_tn(specula_ctx *ctx, const float *A, const float *B, int M, int N, int K, float *C,
                 int splits, float *work, cudaStream_t st);
int gemm_bf16_tn(specula_ctx *ctx, const void *A, const void *B, int M, int N, int K, float *C,
                 int splits, float *work, cudaStream_t st);
// the split-K partials work[s][M][N], s < splits (a count from gemm_splits),
// left for the caller's kernel to add
int gemm_bf16_partials(specula_ctx *ctx, const void *A, const void *B, int M, int N, int K,
                       int splits, float *work, cudaStream_t st);
// Column sums sum[c] = the sum over r < rows of D[r][c], rows in order; n of a
// multiple of 32 columns.
struct ColSums {
  int n = 0, rows = 0;
  int cols[3] = {};
  const float *D[3] = {};
  float *sum[3] = {};
};
#ifdef __CUDACC__
// the column sums by whole warps, 32 columns each: warp w of nw
__device__ __forceinline__ void column_sums(const ColSums &S, int w, int nw) {
  for (int l = 0; l < S.n; ++l) {
    const int C = S.cols[l], groups = C / 32;
    for (int g = w; g < groups; g += nw) {
      const int c = g * 32 + (threadIdx.x & 31);
      const float *d = S.D[l] + c;
      float s = 0.f;
      int r = 0;
      for (; r + 32 <= S.rows; r += 32) {
        float x[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) x[u] = __ldg(d + (size_t)(r + u) * C);
#pragma unroll
        for (int u = 0; u < 32; ++u) s += x[u];
      }
      for (; r < S.rows; ++r) s += __ldg(d + (size_t)r * C);
      S.sum[l][c] = s;
    }
    w -= groups % nw;   // the next layer's groups go to the warps after these
    if (w < 0) w += nw;
  }
}
#endif
// C_q = A_q B_q^T for up to three products of one K in one launch, and the column
// sums beside them.  K is summed in splits[q] slices (a count from gemm_splits),
// added in order as k_split_reduce adds partials.
int gemm_bf16_group(specula_ctx *ctx, int n, const void *const *A, const void *const *B,
                    const int *M, const int *N, int K, const int *splits, float *const *C,
                    const ColSums &cs, cudaStream_t st);
// C = sum over t < n_terms (<= 3) of A_t B_t^T, one accumulation on the
// tensor cores (split-precision products); every A_t is M x K, every B_t is
// N x K, bf16, row-major
int gemm_bf16_terms(specula_ctx *ctx, int n_terms, const void *const *A, const void *const *B,
                    int M, int N, int K, float *C, int splits, float *work, cudaStream_t st);

// modes[b] = R slopes[b] in float32, b < nb (recon_f32.cu)
int recon_f32_run(specula_ctx *ctx, const float *R, const float *s, float *m, int n_modes,
                  int n_slopes, int nb, cudaStream_t st);
int slopes_pyr_run(specula_ctx *ctx, const int32_t *idx, int n_sub, int n_valid,
                   const float *det, const float *ref, int n_batch, float *out, cudaStream_t st);

bool pwfs_split_for(int N, int *N1, int *N2);

// host geometry (api.cu)
int host_pupil_mask(int n, double obsc, uint8_t *mask);
int host_valid_subaps(int n, double obsc, int n_sub, int32_t *idx, int32_t *n_valid);
}  // namespace specula

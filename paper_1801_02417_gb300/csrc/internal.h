// Internal declarations of the Polarized SARA CUDA library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "polsara.h"

namespace ps {

constexpr int kBases = 9;        // Dirac + db1..db8
constexpr int kDb = 8;           // Daubechies bases
constexpr int kMaxTaps = 16;     // db8 filter length
constexpr int kGridTile = 16;    // degridding tile side (cells)
constexpr int kGridItem = 768;   // visibilities per degridding work item, at most
constexpr int kEsTerms = 5;      // coefficients of the even and of the odd part of a kernel tap's polynomial
constexpr int kWarpBins = 64;    // l2 blocks up to which degridding keeps per-warp FP64 block sums
constexpr int kGraphIters = 8;   // iterations per launch of the multi-iteration graph

// Analysis / synthesis kernel modes.
enum { SARA_DUAL = 0, SARA_APPLY = 1, SARA_REWEIGHT = 2 };
// Degridding modes.
enum { DEG_DUAL = 0, DEG_APPLY = 1, DEG_RESID = 2 };

struct GridItem {      // one degridding CTA: stored rows [vstart, vend), centres in tile (ty, tx)
  int32_t ty, tx;
  int32_t vstart, vend;
};

// Geometry of the NUFFT grid: the K x K oversampled spectrum is kept only on a
// window of frequencies [-R, R]^2 covering every interpolation tap (window
// mode), or whole (full mode, indices modulo K).
struct GridGeom {
  int K = 0, logK = 0;   // oversampled FFT length (2n)
  int W = 7;             // interpolation kernel width
  int R = 0;             // window half-width (cells)
  int Wd = 0;            // stored grid side: 2R+1 (window) or K (full)
  int full = 0;          // 1: full grid, indices wrap modulo K
  int off = 0;           // grid index of frequency k: (k + off) [& (K-1) if full]
  int tilesX = 0;        // degridding tiles per side
  float beta = 0.f;      // ES kernel shape
};

struct Handle {
  ps_config cfg{};
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  cudaStream_t aux = nullptr;       // second stream: SARA chain runs beside the NUFFT chain in graphs
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  std::string err;
  int n = 0, N = 0, L = 0, mode = PS_POLARIZED;
  double tau = 0, rho1 = 1, rho2 = 1, rho3 = 1, opnorm_sq = 0, gamma = 1;
  double gamma_default = 0;       // cfg.gamma, else 1e-3 max|Psi^dagger phi^dagger Y| / ||phi||^2
  double tv_mu[4] = {0, 0, 0, 0}, l1_mu[4] = {0, 0, 0, 0};   // TV and l1 weights (Algorithm 3)
  bool have_meas = false;
  bool derived_valid = false;     // PsiA and Adj hold Psi A and phi^dagger B of the current state
  int64_t iterations = 0;
  int64_t bytes = 0;

  // Image-domain state (float32 planes).
  float *S = nullptr, *Z = nullptr, *C = nullptr, *D = nullptr;
  float *Xb = nullptr;        // 2 S^(k+1) - S^(k)
  float *PsiA = nullptr;      // Psi A
  float *Adj = nullptr;       // phi^dagger B
  float *tmp4 = nullptr;      // 4N scratch for operators
  float *A = nullptr, *T = nullptr;   // 36N coefficients and thresholds gamma W
  float *approx = nullptr;    // ping-pong buffers of 32 * (N/4) approximations: approx and approx2
  float *approx2 = nullptr;
  int nmaps = 4;              // maps the SARA and primal launches cover (4 P for a batch's size class)
  int problems = 1;           // problems of a batched primal launch (the per-problem arrays are consecutive)
  bool in_slab = false;       // state arrays are slices of a batch's class slabs (not freed by ps_destroy)
  double *red = nullptr;      // reduction partials
  int red_cap = 0;
  double *red_host = nullptr; // pinned
  double *relc_host = nullptr; // pinned, mapped: relative-change sums (8) and the device flags (2) of the last request;
                               // ps_compute_stats: sum, counts (10-12), weighted norm (13), flags (14-15)
  double *relc_dev = nullptr;  // the device's address of relc_host
  cudaEvent_t relc_ev = nullptr;
  bool relc_pending = false;
  int *dev_flags = nullptr;   // [0] error flag: a bounded wait gave up; [1], [2] counters of the reductions

  // Visibility-domain state, rows stored in tap-centre-cell order (tile-major).
  int M = 0, nblocks = 0;
  float2 *R = nullptr;        // residual form of B: B = c_b R  (M x 4)
  float2 *Y = nullptr;        // measurements (M x 4)
  float4 *rec = nullptr;      // (fx, fy, w, packed (cx, cy))
  int32_t *perm = nullptr;    // sorted row -> caller row
  float2 *vtmp = nullptr;     // M x 4 scratch
  double *eps = nullptr;      // per block radius (device)
  float *cb = nullptr;        // per block scale c_b (device)
  double *block_sum = nullptr;     // nblocks FP64 sums of a running degridding launch (zero between launches)
  double *block_norm_sq = nullptr; // those of the last one that formed them
  int *block_done = nullptr;       // its finished CTAs (zero between launches)
  int ncells = 0;                  // cells that hold a row
  int nitems = 0;
  GridItem *items = nullptr;       // degridding work items
  uint16_t *vblk = nullptr;        // l2 block of each stored row
  std::vector<double> eps_host;
  double psf_peak = 0.0;      // 2 sum w_m^2: peak of the Stokes-I PSF
  float *tmp36 = nullptr;     // 36N scratch for operator calls (allocated on first use)
  std::vector<int64_t> offsets_host;

  // NUFFT buffers.
  GridGeom g;
  float4 *T1 = nullptr;       // n x Wd row spectra (forward)
  float4 *G = nullptr;        // Wd x Wd packed spectra (I+iQ, U+iV)
  float4 *Acc = nullptr;      // Wd x Wd x 2 gridding accumulators (xI, xQ | xU, xV)
  float4 *T2 = nullptr;       // n x Wd column-transformed adjoint
  float2 *tw = nullptr;       // K per-stage twiddles: stage t at [2^t - 1, 2^(t+1) - 1)
  float *corr = nullptr;      // n de-apodisation factors 1 / phihat(2 pi x / K)

  // Launch choices (PS_TUNE_* slots, kept for the caller) and the device's SM count.
  int32_t tune[PS_TUNE_COUNT] = {};
  int num_sms = 0;

  // Whether NUFFT launches may start before the kernel before them has ended (launch_after).
  bool early = true;

  // CUDA graph of one iteration.
  cudaGraphExec_t graph = nullptr;
  cudaGraphExec_t graph_multi = nullptr;   // kGraphIters iterations back to back (same mode as graph)
  int graph_mode = -1;
  uint64_t version = 1;       // bumped when mode, state or measurements change (batch graphs rebuild)
};

// Bounded-wait poll budget of the translation unit with bulk-copy waits (polls < 0: default).
cudaError_t set_wait_polls_sara(int polls);

// Message returned by ps_last_error(NULL) (calls without a handle).
void set_global_error(const std::string& msg);

// Host-side constants.
void daubechies_filters(double h[kDb][kMaxTaps]);          // db1..db8 scaling filters
double es_beta(int W);
double es_kernel(double t, int W, double beta);            // ES kernel value at offset t (cells)
std::vector<double> es_fourier(double step, int count, int W);   // its Fourier transform at k step, k < count (beta = es_beta)
// Taps 0 .. W/2 of width W = 5 + 2 q as polynomials of their offset: c[q][j] holds the even coefficients, then
// the odd ones, each in both halves of a 64-bit word. Made once.
struct EsTable {
  alignas(16) float c[3][5][2 * kEsTerms][2];
};
const EsTable& es_table();

// Kernel launchers (return cudaGetLastError()).
cudaError_t upload_filters(const double h[kDb][kMaxTaps], cudaStream_t stream);
cudaError_t upload_es_polys(cudaStream_t stream);   // queued on stream, not waited for

// NUFFT pieces (nufft.cu).
// X (4 planes) -> G; clear_acc: the gridding accumulator too, for the nufft_grid(.., cleared) that follows.
cudaError_t nufft_forward_grid(Handle* h, const float* X, bool clear_acc);
// G -> visibilities; DEG_DUAL also steps the l2-ball factors c_b, unless keep_cb. perm: DEG_APPLY writes
// the caller's row order (stored order without).
cudaError_t nufft_degrid(Handle* h, int mode, float2* out, bool keep_cb = false, const int32_t* perm = nullptr);
// Visibilities -> Acc; `in` in stored order, or in the caller's (perm).
cudaError_t nufft_grid(Handle* h, const float2* in, int use_block_scale, bool cleared, const int32_t* perm = nullptr);
cudaError_t tv_dual(Handle* h);      // Algorithm 3 steps 5-6 on Xb -> A (TV layout)
cudaError_t tv_adjoint(Handle* h);   // Psi A = grad^T A_tv (+ A_l1) -> PsiA
__host__ __device__ inline bool tv_mode(int m) { return m >= PS_TV && m <= PS_L1TV_NC; }
__host__ __device__ inline bool constrained_mode(int m) { return m == PS_POLARIZED || m == PS_SOC || m == PS_TV || m == PS_L1TV; }
cudaError_t nufft_adjoint_image(Handle* h, float* out);                    // Acc -> 4 planes

// SARA pieces (sara.cu).
// `fine_done` (may be null) is recorded on h->stream after the level-1 analysis launch;
// `fine_start` (may be null) before the finest synthesis level (stage profiling).
cudaError_t sara_analysis(Handle* h, const float* X, float* coef, float* thr, int mode,
                          float scale, float gamma, float delta, cudaEvent_t fine_done = nullptr);
cudaError_t sara_synthesis(Handle* h, const float* coef, float* out, cudaEvent_t fine_start = nullptr);

int sara_launches(int n, int L);   // kernels of one analysis and one synthesis

// Elementwise / reductions (prox.cu).
int sweep_blocks(int N);   // CTAs of the per-pixel sweep (8 FP64 partials each)
cudaError_t primal_sweep(Handle* h);
cudaError_t dirac_apply(Handle* h, const float* X, float* coef, float* thr, int mode,
                        float scale, float gamma, float delta);
cudaError_t reduce_dot(Handle* h, const float* a, const float* b, size_t len, double* dev_out);
cudaError_t relc_sums(Handle* h, int nb, double* out);   // 8 column sums of k_primal's partials + the flags
cudaError_t violation_count(Handle* h, const float* S, const double* rms_sum, double zeta_sigma, double* out);
cudaError_t weighted_l1(Handle* h, const float* coef, const float* thr, double* out);
cudaError_t max_abs(Handle* h, const float* c, size_t len, double* dev_out);
cudaError_t scale_copy(Handle* h, const float* x, float* y, size_t len, double s);
cudaError_t fill(Handle* h, float* p, size_t len, float v);      // len a multiple of 4
cudaError_t lanczos_start(Handle* h, float* v, size_t len, double* scratch);   // the normalised start vector
cudaError_t lanczos_update(Handle* h, float* w, const float* v, const float* u, size_t len, double* coef,
                           const double* last);                             // w -= alpha v + beta u; |w|^2
cudaError_t lanczos_scale(Handle* h, const float* w, float* u, size_t len, const double* norm_sq);   // u = w / |w|
cudaError_t gather_vis(Handle* h, const float2* user, float2* sorted);
cudaError_t read_dual(Handle* h, float2* user);   // c_b R in the caller's row order (state readout)

}  // namespace ps

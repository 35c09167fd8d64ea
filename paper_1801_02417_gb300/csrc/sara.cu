// SARA dictionary (Section 4.1) on the GPU: Dirac + Daubechies db1..db8, periodic
// orthonormal 2D Mallat transforms, concatenation scaled by 1/3.
//
// Analysis Psi^dagger runs one launch per level for all 8 Daubechies bases and 4
// maps (grid.y = basis, grid.z = map). Each CTA computes one TO x TO tile of the
// four subbands from a (2 TO + 14)^2 input tile held in shared memory (rows
// filtered first, then columns; indices modulo the level size, i.e. periodic).
// The detail coefficients are consumed in the epilogue instead of being stored:
//   SARA_DUAL      A = clamp(A + rho1/3 * coef, -gamma W, +gamma W)   (Alg. 1 steps 5-6)
//   SARA_APPLY     A = coef / 3                                       (operator)
//   SARA_REWEIGHT  gamma W = gamma delta / (delta + |coef / 3|)       (Eq. weights)
// Only the approximation goes to scratch for the next level.
//
// Synthesis Psi runs one launch per level from coarse to fine; the finest level
// sums the eight bases and the Dirac part in registers and writes Psi A once.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>

#include "internal.h"
#include "packed.cuh"

namespace ps {

__constant__ __align__(16) float c_h[kDb][kMaxTaps];
__constant__ __align__(16) float c_g[kDb][kMaxTaps];
// The same taps duplicated in both halves of a 64-bit word, the operand of packed
// FP32x2 FMAs that apply one tap to two neighbouring samples.
__constant__ __align__(16) float2 c_hd[kDb][kMaxTaps];
__constant__ __align__(16) float2 c_gd[kDb][kMaxTaps];

cudaError_t upload_filters(const double h[kDb][kMaxTaps], cudaStream_t stream) {
  float hf[kDb][kMaxTaps], gf[kDb][kMaxTaps];
  for (int b = 0; b < kDb; ++b) {
    const int Lf = 2 * (b + 1);
    for (int j = 0; j < kMaxTaps; ++j) {
      hf[b][j] = j < Lf ? (float)h[b][j] : 0.f;
      gf[b][j] = j < Lf ? (float)(((j & 1) ? -1.0 : 1.0) * h[b][Lf - 1 - j]) : 0.f;
    }
  }
  float2 hd[kDb][kMaxTaps], gd[kDb][kMaxTaps];
  for (int b = 0; b < kDb; ++b)
    for (int j = 0; j < kMaxTaps; ++j) {
      hd[b][j] = make_float2(hf[b][j], hf[b][j]);
      gd[b][j] = make_float2(gf[b][j], gf[b][j]);
    }
  // On the caller's stream and waited for: kernels launched on non-blocking streams are
  // not ordered after the legacy stream's copies.
  cudaError_t e = cudaMemcpyToSymbolAsync(c_h, hf, sizeof(hf), 0, cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_g, gf, sizeof(gf), 0, cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_hd, hd, sizeof(hd), 0, cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_gd, gd, sizeof(gd), 0, cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  return e;
}

// A duplicated tap as one 64-bit FMA operand.
__device__ __forceinline__ u64 cdup(const float2& c) { return *reinterpret_cast<const u64*>(&c); }

// Calls CALL(LF) with the compile-time filter length of basis bi (db1..db8).
#define PS_SWITCH_LF(bi, CALL)    \
  switch (bi) {                   \
    case 0: CALL(2); break;       \
    case 1: CALL(4); break;       \
    case 2: CALL(6); break;       \
    case 3: CALL(8); break;       \
    case 4: CALL(10); break;      \
    case 5: CALL(12); break;      \
    case 6: CALL(14); break;      \
    default: CALL(16); break;     \
  }

// ---------------------------------------------------------------------------
// Fast path for levels whose half size is >= 32: 32 x 32 output tiles, filter
// length and tile shape known at compile time, each thread producing a strip of
// four outputs from registers (inputs read once from shared memory per strip).
constexpr int kTO = 32;                          // analysis output tile (per subband)
constexpr int kRSmax = 2 * kTO + kMaxTaps - 2;   // 78: input tile side for db8
constexpr int kA2Cols = 2 * kTO + 16;            // 80 staged input columns (covers 2 TO + 14 for db8)
constexpr int kA2Pitch = kA2Cols + 4;            // 84 = 20 mod 32 banks: row-parallel 16-byte reads conflict-free
constexpr int kA2In = kRSmax * kA2Pitch;         // input tile
constexpr int kPlo = kTO + 4;                    // row-filtered tiles (16-byte aligned rows)

__device__ __forceinline__ int wrap1(int v, int m) { return v < 0 ? v + m : (v >= m ? v - m : v); }

// The filter passes of the analysis run as loops over the taps of basis b (its length a value, not
// a template argument): eight unrolled variants, each executed once or twice per CTA, spent 6 to
// 10 cycles per issue waiting for instructions in the levels below the first (ncu); the loops are
// one short piece of code for every basis. us: 1024^2, 6 levels, the stage of levels 2-6 65 -> 59, of
// level 1 83.5 -> 82 (105 -> 84 with one basis per CTA); iteration 457 -> 441, 512^2 120 -> 113, 2048^2
// (cone dual) 1177 -> 1142.
//
// Rows: lo/hi[r][k] = sum_j h/g[j] in[r][2k + j], k in [0, TO), RS rows. Each thread makes
// four outputs of one row from 16-byte reads; the taps go in pairs,
// {c[2p], c[2p+1]} x {in[2k+2p], in[2k+2p+1]}, and the two halves are added at the end. Two pairs per
// step and the last of an odd count on its own: a pair of zero taps in its place would turn an infinity
// that the filter does not reach into a NaN (that step is 1% of the stage: 80.7 -> 81.5 us at level 1 of 1024^2).
// x0 .. x3 are the sample pairs p .. p + 3.
__device__ __forceinline__ void ana_rows(int b, const float* __restrict__ in_s, float* __restrict__ lo_s,
                                         float* __restrict__ hi_s) {
  const int RS = 2 * kTO + 2 * b;
  for (int u = threadIdx.x; u < RS * (kTO / 4); u += blockDim.x) {
    const int r = u % RS, k0 = (u / RS) * 4;
    const ulonglong2* row = reinterpret_cast<const ulonglong2*>(in_s + r * kA2Pitch + 2 * k0);
    const ulonglong2 q0 = row[0], q1 = row[1];
    u64 x0 = q0.x, x1 = q0.y, x2 = q1.x, x3 = q1.y;
    u64 a[4] = {0ull, 0ull, 0ull, 0ull}, c[4] = {0ull, 0ull, 0ull, 0ull};
    for (int p = 0; p < b; p += 2) {
      const ulonglong2 n = row[2 + (p >> 1)];
      const ulonglong2 h = *reinterpret_cast<const ulonglong2*>(&c_h[b][2 * p]);
      const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(&c_g[b][2 * p]);
      a[0] = ffma2(h.y, x1, ffma2(h.x, x0, a[0]));
      a[1] = ffma2(h.y, x2, ffma2(h.x, x1, a[1]));
      a[2] = ffma2(h.y, x3, ffma2(h.x, x2, a[2]));
      a[3] = ffma2(h.y, n.x, ffma2(h.x, x3, a[3]));
      c[0] = ffma2(g.y, x1, ffma2(g.x, x0, c[0]));
      c[1] = ffma2(g.y, x2, ffma2(g.x, x1, c[1]));
      c[2] = ffma2(g.y, x3, ffma2(g.x, x2, c[2]));
      c[3] = ffma2(g.y, n.x, ffma2(g.x, x3, c[3]));
      x0 = x2, x1 = x3, x2 = n.x, x3 = n.y;
    }
    if (!(b & 1)) {   // b + 1 pairs: the last one
      const u64 h = *reinterpret_cast<const u64*>(&c_h[b][2 * b]), g = *reinterpret_cast<const u64*>(&c_g[b][2 * b]);
      a[0] = ffma2(h, x0, a[0]);
      a[1] = ffma2(h, x1, a[1]);
      a[2] = ffma2(h, x2, a[2]);
      a[3] = ffma2(h, x3, a[3]);
      c[0] = ffma2(g, x0, c[0]);
      c[1] = ffma2(g, x1, c[1]);
      c[2] = ffma2(g, x2, c[2]);
      c[3] = ffma2(g, x3, c[3]);
    }
    float lo[4], hi[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float a0, a1, c0, c1;
      f2unpack(a[q], a0, a1);
      f2unpack(c[q], c0, c1);
      lo[q] = a0 + a1;
      hi[q] = c0 + c1;
    }
    *reinterpret_cast<float4*>(lo_s + r * kPlo + k0) = make_float4(lo[0], lo[1], lo[2], lo[3]);
    *reinterpret_cast<float4*>(hi_s + r * kPlo + k0) = make_float4(hi[0], hi[1], hi[2], hi[3]);
  }
}

__device__ __forceinline__ float4 f4fma(float a, float4 x, float4 y) {
  return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}
__device__ __forceinline__ float4 f4clamp(float4 a, float4 t) {
  return make_float4(fminf(fmaxf(a.x, -t.x), t.x), fminf(fmaxf(a.y, -t.y), t.y), fminf(fmaxf(a.z, -t.z), t.z),
                     fminf(fmaxf(a.w, -t.w), t.w));
}
__device__ __forceinline__ float4 f4of(u64 a, u64 b) {
  float4 r;
  f2unpack(a, r.x, r.y);
  f2unpack(b, r.z, r.w);
  return r;
}

// Epilogue on four consecutive coefficients (16-byte aligned).
__device__ __forceinline__ void sara_epilogue4(int mode, float4 v, size_t idx, float4 a_old, float4 t_old,
                                               float* coef, float* thr, float scale, float gamma, float delta) {
  if (mode == SARA_DUAL) {
    *reinterpret_cast<float4*>(coef + idx) = f4clamp(f4fma(scale, v, a_old), t_old);
  } else if (mode == SARA_APPLY) {
    *reinterpret_cast<float4*>(coef + idx) = make_float4(scale * v.x, scale * v.y, scale * v.z, scale * v.w);
  } else {
    const float gd = gamma * delta;
    *reinterpret_cast<float4*>(thr + idx) =
        make_float4(gd / (delta + fabsf(scale * v.x)), gd / (delta + fabsf(scale * v.y)),
                    gd / (delta + fabsf(scale * v.z)), gd / (delta + fabsf(scale * v.w)));
  }
}

// Columns + epilogue for one basis: four subbands of a TO x TO tile, 256 threads. Half of them
// filter the low rows (LL and LH), half the high rows (HL and HH); a thread owns four consecutive
// columns (two packed pairs) of two output rows, whose 2 LF taps reach over LF + 2 input rows, so
// it reads 18 rows of 16 bytes for db8 where one output row of all four subbands took 32. The
// epilogue reads and writes A and gamma W as float4 (staged before the filtering).
template <typename Ready>
__device__ __forceinline__ void ana_cols(const float* __restrict__ lo_s, const float* __restrict__ hi_s, int bi,
                                         int map, int n, int hm, int oy0, int ox0, int last, float* __restrict__ coef,
                                         float* __restrict__ thr, float* __restrict__ approx_out, int mode,
                                         float scale, float gamma, float delta, const float* st_a, const float* st_t,
                                         Ready&& ready) {
  const size_t base = ((size_t)map * kBases + (bi + 1)) * (size_t)n * n;
  const bool high = threadIdx.x >= 128;   // warp-uniform
  const int kx0 = (threadIdx.x & 7) * 4, ky0 = 2 * ((threadIdx.x >> 3) & 15);
  const float* col = (high ? hi_s : lo_s) + 2 * ky0 * kPlo + kx0;
  u64 h[2][2], g[2][2];   // [output row][column pair] through the low and the high filter
#pragma unroll
  for (int r = 0; r < 2; ++r) h[r][0] = h[r][1] = g[r][0] = g[r][1] = 0ull;
  // Input rows 2 q and 2 q + 1 meet taps 2 q, 2 q + 1 of the first output row and 2 q - 2, 2 q - 1 of the second.
  auto step = [&](int r, ulonglong2 x0, ulonglong2 x1, ulonglong2 th, ulonglong2 tg) {
    h[r][0] = ffma2(th.y, x1.x, ffma2(th.x, x0.x, h[r][0]));
    h[r][1] = ffma2(th.y, x1.y, ffma2(th.x, x0.y, h[r][1]));
    g[r][0] = ffma2(tg.y, x1.x, ffma2(tg.x, x0.x, g[r][0]));
    g[r][1] = ffma2(tg.y, x1.y, ffma2(tg.x, x0.y, g[r][1]));
  };
  const ulonglong2* ch = reinterpret_cast<const ulonglong2*>(&c_hd[bi][0]);
  const ulonglong2* cg = reinterpret_cast<const ulonglong2*>(&c_gd[bi][0]);
  auto row = [&](int i) { return *reinterpret_cast<const ulonglong2*>(col + i * kPlo); };
  ulonglong2 th = ch[0], tg = cg[0], x0 = row(0), x1 = row(1);
  step(0, x0, x1, th, tg);
  for (int q = 1; q <= bi; ++q) {
    x0 = row(2 * q), x1 = row(2 * q + 1);
    step(1, x0, x1, th, tg);
    th = ch[q], tg = cg[q];
    step(0, x0, x1, th, tg);
  }
  x0 = row(2 * bi + 2), x1 = row(2 * bi + 3);
  step(1, x0, x1, th, tg);
  if (!ready()) return;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int ky = ky0 + r, Y = oy0 + ky, X = ox0 + kx0, so = ky * kTO + kx0;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    auto out = [&](u64 v0, u64 v1, int sb, size_t o) {   // staged by the bulk-copy engine: [subband][row][32]
      float4 a = z, t = z;
      if (mode == SARA_DUAL) {
        a = *reinterpret_cast<const float4*>(st_a + sb * kTO * kTO + so);
        t = *reinterpret_cast<const float4*>(st_t + sb * kTO * kTO + so);
      }
      sara_epilogue4(mode, f4of(v0, v1), base + o, a, t, coef, thr, scale, gamma, delta);
    };
    if (high) {
      out(h[r][0], h[r][1], 0, (size_t)Y * n + (hm + X));          // x-high, y-low
      out(g[r][0], g[r][1], 2, (size_t)(hm + Y) * n + (hm + X));
    } else {
      out(g[r][0], g[r][1], 1, (size_t)(hm + Y) * n + X);          // x-low, y-high
      const size_t o = base + (size_t)Y * n + X;
      if (last) {
        float4 a = z, t = z;
        if (mode == SARA_DUAL) {
          a = *reinterpret_cast<const float4*>(coef + o);
          t = *reinterpret_cast<const float4*>(thr + o);
        }
        sara_epilogue4(mode, f4of(h[r][0], h[r][1]), o, a, t, coef, thr, scale, gamma, delta);
      } else {
        *reinterpret_cast<float4*>(approx_out + ((size_t)map * kDb + bi) * (size_t)hm * hm + (size_t)Y * hm + X) =
            f4of(h[r][0], h[r][1]);
      }
    }
  }
}

// 2D tensor maps (TMA) of the arrays whose tiles the tiled SARA kernels stage, one box
// each, with the box's row pitch equal to the shared-memory pitch of the staged tile:
//   in    analysis input planes, width m, box kA2Pitch x kRSmax (the whole input tile)
//   coef  analysis: coefficients, width n, box kTO x kTO (one subband tile of A)
//   thr   analysis: thresholds gamma W, same box (one subband tile of gamma W)
//   scoef synthesis: coefficients, width n, box kC2Pitch x kC2Rows (one subband tile)
//   apx   synthesis: approximations of the level, width hm, same box
// A use_* flag is 0 when its map was not made (then the per-row bulk copies run).
// Tiles whose rows or columns wrap around the periodic edges always take the per-row copies.
struct SaraTma {
  CUtensorMap in, coef, thr, scoef, apx;
  int use_in, use_stage, use_scoef, use_apx;
};

// Input tile of one analysis CTA: RS rows from row 2 oy0 and the 80 columns from
// column 2 ox0 (both modulo m), one bulk copy per row, two where the row wraps
// around the periodic right edge (then the first piece is 64 columns).
__device__ __forceinline__ void ana_issue_input(const float* __restrict__ src, int m, int oy0, int ox0, int RS,
                                                float* __restrict__ in_s, uint64_t* bar) {
  const int x0 = 2 * ox0;
  const int first = min(kA2Cols, m - x0);
  if (threadIdx.x == 0) mbar_expect_tx(bar, (uint32_t)(RS * kA2Cols * sizeof(float)));
  for (int r = threadIdx.x; r < RS; r += blockDim.x) {
    int y = 2 * oy0 + r;
    if (y >= m) y -= m;
    const float* row = src + (size_t)y * m;
    float* dst = in_s + r * kA2Pitch;
    fence_proxy_async();
    bulk_g2s(dst, row + x0, first * sizeof(float), bar);
    if (first < kA2Cols) bulk_g2s(dst + first, row, (kA2Cols - first) * sizeof(float), bar);
  }
}

// The input tile by one tensor-map copy when it does not wrap (kRSmax rows of kA2Pitch
// columns; the rows past RS and columns past kA2Cols are not read), else by rows.
// `in_row0` is the row of the plane's first row in the input map.
__device__ __forceinline__ void ana_issue_input_t(const SaraTma& tm, int in_row0, const float* __restrict__ src,
                                                  int m, int oy0, int ox0, int RS, float* __restrict__ in_s,
                                                  uint64_t* bar) {
  if (tm.use_in && 2 * ox0 + kA2Cols <= m && 2 * oy0 + kRSmax <= m) {
    if (threadIdx.x == 0) {
      mbar_expect_tx(bar, (uint32_t)(kRSmax * kA2Pitch * sizeof(float)));
      fence_proxy_async();
      tma_load_2d(in_s, &tm.in, 2 * ox0, in_row0 + 2 * oy0, bar);
    }
  } else {
    ana_issue_input(src, m, oy0, ox0, RS, in_s, bar);
  }
}

// Shared-memory layout of the fast analysis kernels (floats): input tile, row-filtered
// low/high tiles, the staged A and gamma W rows of the three detail subbands, and two
// mbarriers (input tile, staged epilogue operands).
constexpr int kStage = 3 * kTO * kTO;
// Staged epilogue operands start on a 128-byte boundary (tensor-map copy destinations).
constexpr int kAnaPre = (kA2In + 2 * kRSmax * kPlo + 31) / 32 * 32;
static_assert(2 * kStage <= kA2In, "the staged operands fit the input tile");
static_assert(kA2In % 4 == 0 && (kRSmax * kPlo) % 4 == 0 && kStage % 32 == 0, "aligned stage buffers");

// The first 3 * 32 * 2 threads each start one bulk copy of this tile's A and gamma W
// detail rows (3 subbands x 32 rows x 128 B) so they arrive while the rows are
// filtered; thread 0 sets the expected byte count (the barrier's transaction count
// may run ahead of it).
__device__ __forceinline__ void stage_epilogue(const float* coef, const float* thr, size_t base, int n, int hm,
                                               int oy0, int ox0, float* st_a, float* st_t, uint64_t* bar) {
  if (threadIdx.x == 0) mbar_expect_tx(bar, 2u * kStage * sizeof(float));
  const int k = threadIdx.x;
  if (k < 2 * 3 * kTO) {
    const int arr = k / (3 * kTO), kk = k - arr * (3 * kTO);
    const int sb = kk / kTO, r = kk - sb * kTO;
    const int Y = oy0 + r;
    const size_t off = sb == 0 ? base + (size_t)Y * n + hm + ox0
                               : (sb == 1 ? base + (size_t)(hm + Y) * n + ox0 : base + (size_t)(hm + Y) * n + hm + ox0);
    float* dst = (arr ? st_t : st_a) + sb * kTO * kTO + r * kTO;
    fence_proxy_async();   // k_ana_l1m refills buffers its threads have read
    bulk_g2s(dst, (arr ? thr : coef) + off, kTO * sizeof(float), bar);
  }
}

// The same operands as six tensor-map copies (three subband tiles of A and of gamma W) by
// one thread, when the maps were made; `prow` is the row of the basis plane in the maps.
__device__ __forceinline__ void stage_epilogue_t(const SaraTma& tm, const float* coef, const float* thr, size_t base,
                                                 int prow, int n, int hm, int oy0, int ox0, float* st_a, float* st_t,
                                                 uint64_t* bar) {
  if (!tm.use_stage) {
    stage_epilogue(coef, thr, base, n, hm, oy0, ox0, st_a, st_t, bar);
    return;
  }
  if (threadIdx.x == 0) {
    mbar_expect_tx(bar, 2u * kStage * sizeof(float));
    fence_proxy_async();   // k_ana_l1m refills buffers its threads have read
    const int xs[3] = {hm + ox0, ox0, hm + ox0}, ys[3] = {prow + oy0, prow + hm + oy0, prow + hm + oy0};
#pragma unroll
    for (int sb = 0; sb < 3; ++sb) {
      tma_load_2d(st_a + sb * kTO * kTO, &tm.coef, xs[sb], ys[sb], bar);
      tma_load_2d(st_t + sb * kTO * kTO, &tm.thr, xs[sb], ys[sb], bar);
    }
  }
}

struct AnaSmem {
  float *in_s, *lo_s, *hi_s, *st_a, *st_t;
  uint64_t* bar;   // [0] input tile, [1] staged epilogue operands
};
// OVERLAY: the staged operands take the place of the input tile, once the rows have read it.
template <bool OVERLAY>
__device__ __forceinline__ AnaSmem ana_smem(float4* sma) {
  AnaSmem a;
  a.in_s = reinterpret_cast<float*>(sma);
  a.lo_s = a.in_s + kA2In;
  a.hi_s = a.lo_s + kRSmax * kPlo;
  a.st_a = a.in_s + (OVERLAY ? 0 : kAnaPre);
  a.st_t = a.st_a + kStage;
  a.bar = reinterpret_cast<uint64_t*>(a.in_s + kAnaPre + (OVERLAY ? 0 : 2 * kStage));
  return a;
}

// A bounded wait gave up: raise the flag, give the copies in flight a second bounded
// wait so none lands after the CTA has gone, and let the caller return.
__device__ __forceinline__ void ana_abort(const AnaSmem& S, int staged, int* err) {
  if (threadIdx.x == 0) {
    atomicExch(err, 1);
    (void)mbar_drain(&S.bar[0], 0);
    if (staged) (void)mbar_drain(&S.bar[1], 0);
  }
}

// One basis of one tile: input copies, rows, columns + epilogue, whose operands (dual mode) are staged
// beside the input, or (OVERLAY) over the input tile once the rows have read it, while the columns
// are filtered: then a CTA takes 49 KB instead of 73, and an SM holds four instead of three. PREFETCH brings the
// operands to the L2 beforehand: level 2 on of 2048^2 138 -> 132 us, of 1024^2 56 -> 55; not at level 1, where
// one basis per CTA means a small map whose coefficients are in the L2 (512^2 107.1 without, 108.9 with).
template <bool OVERLAY, bool PREFETCH>
__device__ __forceinline__ void ana_basis(const SaraTma& tm, int in_row0, const float* src, int m, const AnaSmem& S,
                                          int bi, int map, int n, int hm, int oy0, int ox0, int last, float* coef,
                                          float* thr, float* approx_out, int mode, float scale, float gamma,
                                          float delta, int* err) {
  ana_issue_input_t(tm, in_row0, src, m, oy0, ox0, 2 * kTO + 2 * bi, S.in_s, &S.bar[0]);
  const int prow = (map * kBases + bi + 1) * n;
  if (PREFETCH && mode == SARA_DUAL && tm.use_stage && threadIdx.x < 6) {
    const int sb = threadIdx.x % 3;
    tma_prefetch_2d(threadIdx.x < 3 ? &tm.coef : &tm.thr, sb == 1 ? ox0 : hm + ox0, prow + (sb == 0 ? oy0 : hm + oy0));
  }
  auto stage = [&] {
    if (mode == SARA_DUAL)
      stage_epilogue_t(tm, coef, thr, ((size_t)map * kBases + bi + 1) * (size_t)n * n, prow, n, hm, oy0, ox0, S.st_a,
                       S.st_t, &S.bar[1]);
  };
  if (!OVERLAY) stage();
  const bool ok = mbar_wait(&S.bar[0], 0);
  if (__syncthreads_or(!ok)) {
    ana_abort(S, !OVERLAY && mode == SARA_DUAL, err);
    return;   // this tile is left unchanged (the host reports PS_ETIMEOUT)
  }
  ana_rows(bi, S.in_s, S.lo_s, S.hi_s);
  __syncthreads();
  if (OVERLAY) stage();
  ana_cols(S.lo_s, S.hi_s, bi, map, n, hm, oy0, ox0, last, coef, thr, approx_out, mode, scale, gamma, delta, S.st_a,
           S.st_t, [&] {
             if (mode != SARA_DUAL || mbar_wait(&S.bar[1], 0)) return true;
             atomicExch(err, 1);
             (void)mbar_drain(&S.bar[1], 0);
             return false;
           });
}

// Level-1 analysis: input is the map itself; one basis per CTA (grid.y).
template <bool OVERLAY>
__global__ void __launch_bounds__(256, OVERLAY ? 4 : 3) k_ana_l1(const float* __restrict__ X, int n, int last,
                                                                 float* __restrict__ coef,
                                                   float* __restrict__ thr, float* __restrict__ approx_out, int mode,
                                                   float scale, float gamma, float delta, int* err,
                                                   const __grid_constant__ SaraTma tm) {
  extern __shared__ __align__(128) float4 sma[];
  const AnaSmem S = ana_smem<OVERLAY>(sma);
  const int bi = blockIdx.y, map = blockIdx.z;
  const int hm = n >> 1, tilesx = hm / kTO;
  const int oy0 = (blockIdx.x / tilesx) * kTO, ox0 = (blockIdx.x % tilesx) * kTO;
  if (threadIdx.x == 0) {
    mbar_init(&S.bar[0], 1);
    mbar_init(&S.bar[1], 1);
  }
  __syncthreads();
  ana_basis<OVERLAY, false>(tm, map * n, X + (size_t)map * n * n, n, S, bi, map, n, hm, oy0, ox0, last, coef, thr,
                            approx_out, mode, scale, gamma, delta, err);
}

// Levels >= 2 with half size >= 32: one basis per CTA (grid.y). (A basis-slowest grid, which
// keeps the co-resident CTAs on one filter's code, measured 5 us slower at 1024^2.)
template <bool OVERLAY>
__global__ void __launch_bounds__(256, OVERLAY ? 4 : 3) k_ana_lv(const float* __restrict__ approx_in, int m, int n,
                                                                 int last, float* __restrict__ coef, float* __restrict__ thr,
                                                   float* __restrict__ approx_out, int mode, float scale, float gamma,
                                                   float delta, int* err, const __grid_constant__ SaraTma tm) {
  extern __shared__ __align__(128) float4 sma[];
  pdl_wait();
  const AnaSmem S = ana_smem<OVERLAY>(sma);
  const int bi = blockIdx.y, map = blockIdx.z;
  const int hm = m >> 1, tilesx = hm / kTO;
  const int oy0 = (blockIdx.x / tilesx) * kTO, ox0 = (blockIdx.x % tilesx) * kTO;
  if (threadIdx.x == 0) {
    mbar_init(&S.bar[0], 1);
    mbar_init(&S.bar[1], 1);
  }
  __syncthreads();
  ana_basis<OVERLAY, OVERLAY>(tm, (map * kDb + bi) * m, approx_in + ((size_t)map * kDb + bi) * (size_t)m * m, m, S, bi,
                              map, n, hm, oy0, ox0, last, coef, thr, approx_out, mode, scale, gamma, delta, err);
}

// Level-1 analysis with the input tile shared by four bases: one CTA per (tile, half of the bases,
// map). The 2 TO + 14 rows the db8 filter needs cover every shorter filter (same
// origin), so the map's tile is copied once and each basis filters it from shared memory.
// One staging set holds A and gamma W (dual mode), refilled for basis i + 1 once basis i's
// columns have read it, so the copy overlaps the next basis' row pass; 73 KB, 3 CTAs/SM.
// (Two sets at 2 CTAs/SM, eight bases per CTA, 512 threads and a persistent form over all
// units were slower: 85-88, 94 and 139 us at 1024^2 against 82.)
constexpr int kL1Bases = 4;
static size_t analysis_smem(bool overlay) {
  return (size_t)(kAnaPre + (overlay ? 0 : 2 * kStage)) * sizeof(float) + 16;
}

__global__ void __launch_bounds__(256, 3) k_ana_l1m(const float* __restrict__ X, int n, int last,
                                                    float* __restrict__ coef, float* __restrict__ thr,
                                                    float* __restrict__ approx_out, int mode, float scale,
                                                    float gamma, float delta, int* err,
                                                    const __grid_constant__ SaraTma tm) {
  extern __shared__ __align__(128) float4 smm[];
  const AnaSmem S = ana_smem<false>(smm);
  const int map = blockIdx.z, b0 = blockIdx.y * kL1Bases;
  const int hm = n >> 1, tilesx = hm / kTO;
  const int oy0 = (blockIdx.x / tilesx) * kTO, ox0 = (blockIdx.x % tilesx) * kTO;
  const bool staged = mode == SARA_DUAL;
  auto stage = [&](int bi) {
    stage_epilogue_t(tm, coef, thr, ((size_t)map * kBases + bi + 1) * (size_t)n * n, (map * kBases + bi + 1) * n, n, hm,
                     oy0, ox0, S.st_a, S.st_t, &S.bar[1]);
  };
  if (threadIdx.x == 0) {
    mbar_init(&S.bar[0], 1);
    mbar_init(&S.bar[1], 1);
  }
  __syncthreads();
  ana_issue_input_t(tm, map * n, X + (size_t)map * n * n, n, oy0, ox0, kRSmax, S.in_s, &S.bar[0]);
  if (staged) stage(b0);
  const bool ok = mbar_wait(&S.bar[0], 0);
  if (__syncthreads_or(!ok)) {
    ana_abort(S, staged, err);
    return;   // the CTA's tiles are left unchanged (the host reports PS_ETIMEOUT)
  }
  for (int i = 0; i < kL1Bases; ++i) {
    const int bi = b0 + i;
    ana_rows(bi, S.in_s, S.lo_s, S.hi_s);
    if (staged) {
      const bool ok2 = mbar_wait(&S.bar[1], i & 1);   // each refill completes one phase
      if (__syncthreads_or(!ok2)) {
        if (threadIdx.x == 0) {
          atomicExch(err, 1);
          (void)mbar_drain(&S.bar[1], i & 1);
        }
        return;
      }
    } else {
      __syncthreads();
    }
    ana_cols(S.lo_s, S.hi_s, bi, map, n, hm, oy0, ox0, last, coef, thr, approx_out, mode, scale, gamma, delta, S.st_a,
             S.st_t, [] { return true; });
    __syncthreads();   // lo/hi and the stage set consumed before the next basis
    if (staged && i + 1 < kL1Bases) stage(bi + 1);
  }
}

// ---------------------------------------------------------------------------
// Synthesis for levels with output side m >= 64: 64 x 64 output tiles.
//   * The four subband tiles of one basis (rows of 40 coefficients starting 8
//     columns left of the tile's coefficient origin, with the filter halo) are
//     staged by bulk copies, one per row (two where the row wraps around the
//     periodic left edge), completing on an mbarrier; the finest-level kernel
//     double-buffers them so basis b+1 is in flight while basis b is filtered.
//   * Along y, each thread computes two adjacent columns x four rows of the
//     low/high row-filtered tiles with packed FP32x2 FMAs and stores them
//     column-major ([column][row]).
//   * Along x, each thread owns a 4 x 4 output block; the column-major
//     intermediates give it two rows per 64-bit operand, so the taps are again
//     packed FP32x2 FMAs with the coefficient duplicated in both halves.
constexpr int kT2 = 64;                                  // output tile side
constexpr int kC2Rows = kT2 / 2 + kMaxTaps / 2 - 1;      // 39 coefficient rows (db8 halo)
constexpr int kC2Cols = kT2 / 2 + 8;                     // 40 staged columns: [ox0/2 - 8, ox0/2 + 32)
constexpr int kC2Pitch = 40;                             // staged row pitch: the 40 staged columns
constexpr int kC2Sub = (kC2Rows * kC2Pitch + 31) / 32 * 32;   // one subband tile, 128-byte aligned
constexpr int kC2Set = 4 * kC2Sub;                       // LL, LH, HL, HH
constexpr int kLoPitch = kT2 + 4;                        // column-major intermediates: [column][row]
constexpr int kLoSize = kC2Cols * kLoPitch;
static_assert(kC2Sub % 32 == 0 && kLoSize % 4 == 0, "aligned synthesis buffers");

// Issue the bulk copies of basis `half` (db(half+1)) for the tile at (oy0, ox0):
// subband sb row r <- coefficient row (oy0/2 - half + r) mod hm, columns
// [ox0/2 - 8, ox0/2 + 32) mod hm. Thread 0 posts the byte count; any thread may
// start copies before or after it (the barrier's transaction count may run ahead).
__device__ __forceinline__ void syn2_issue(int half, const float* __restrict__ cb, const float* __restrict__ apx,
                                           int n, int hm, int oy0, int ox0, float* __restrict__ s4, uint64_t* bar) {
  const int CI = kT2 / 2 + half;
  const int ky0 = oy0 / 2 - half, kxa = ox0 / 2 - 8;
  if (threadIdx.x == 0) mbar_expect_tx(bar, (uint32_t)(4 * CI * kC2Cols * sizeof(float)));
  for (int k = threadIdx.x; k < 4 * CI; k += blockDim.x) {
    const int sb = k / CI, r = k - sb * CI;
    const int Yk = wrap1(ky0 + r, hm);
    const float* row;
    if (sb == 0) row = apx ? apx + (size_t)Yk * hm : cb + (size_t)Yk * n;   // LL
    else if (sb == 1) row = cb + (size_t)(hm + Yk) * n;                     // LH (x-low, y-high)
    else if (sb == 2) row = cb + (size_t)Yk * n + hm;                       // HL (x-high, y-low)
    else row = cb + (size_t)(hm + Yk) * n + hm;                             // HH
    float* dst = s4 + sb * kC2Sub + r * kC2Pitch;
    fence_proxy_async();
    if (kxa >= 0) {
      bulk_g2s(dst, row + kxa, kC2Cols * sizeof(float), bar);
    } else {   // left edge: columns hm-8 .. hm-1, then 0 .. 31
      bulk_g2s(dst, row + hm - 8, 8 * sizeof(float), bar);
      bulk_g2s(dst + 8, row, (kC2Cols - 8) * sizeof(float), bar);
    }
  }
}

// The four subband tiles by four tensor-map copies from one thread when the tile does not
// wrap (ox0, oy0 > 0) and the maps were made, else by rows. Each box is kC2Rows x kC2Pitch
// (rows past CI and columns past kC2Cols are not read). `prow` is the row of the basis plane
// in the coefficient map, `aprow` the row of the (map, basis) approximation in the
// approximation map (apx non-null).
__device__ __forceinline__ void syn2_issue_t(const SaraTma& tm, int prow, int aprow, int half,
                                             const float* __restrict__ cb, const float* __restrict__ apx, int n, int hm,
                                             int oy0, int ox0, float* __restrict__ s4, uint64_t* bar) {
  if (!(tm.use_scoef && ox0 > 0 && oy0 > 0 && (apx == nullptr || tm.use_apx))) {
    syn2_issue(half, cb, apx, n, hm, oy0, ox0, s4, bar);
    return;
  }
  if (threadIdx.x == 0) {
    const int ky0 = oy0 / 2 - half, kxa = ox0 / 2 - 8;
    mbar_expect_tx(bar, (uint32_t)(4 * kC2Rows * kC2Pitch * sizeof(float)));
    fence_proxy_async();
    if (apx) tma_load_2d(s4, &tm.apx, kxa, aprow + ky0, bar);               // LL from the approximations
    else tma_load_2d(s4, &tm.scoef, kxa, prow + ky0, bar);                  // LL (coarsest level)
    tma_load_2d(s4 + kC2Sub, &tm.scoef, kxa, prow + hm + ky0, bar);         // LH (x-low, y-high)
    tma_load_2d(s4 + 2 * kC2Sub, &tm.scoef, hm + kxa, prow + ky0, bar);     // HL (x-high, y-low)
    tma_load_2d(s4 + 3 * kC2Sub, &tm.scoef, hm + kxa, prow + hm + ky0, bar);  // HH
  }
}

// The same tiles brought to the L2 ahead of their staging.
__device__ __forceinline__ void syn2_prefetch_t(const SaraTma& tm, int prow, int aprow, int half, int coarsest, int hm,
                                                int oy0, int ox0) {
  if (!(tm.use_scoef && ox0 > 0 && oy0 > 0 && (coarsest || tm.use_apx)) || threadIdx.x >= 4) return;
  const int ky0 = oy0 / 2 - half, kxa = ox0 / 2 - 8, sb = threadIdx.x;
  if (sb == 0 && !coarsest) tma_prefetch_2d(&tm.apx, kxa, aprow + ky0);
  else tma_prefetch_2d(&tm.scoef, (sb & 2 ? hm : 0) + kxa, prow + (sb & 1 ? hm : 0) + ky0);
}

// Along y for basis LF: lo/hi at output rows 4 rg + t (t = 0..3) and staged columns
// c, c + 1, from coefficient rows 2 rg + i (i = 0 .. half + 1) through tap
// j = t - 2 (i - half). Columns start at the even column at or left of 8 - half. The 256 threads take
// the tile's own 16 column pairs x 16 row groups, a half-warp 8 pairs of two row groups and a
// quarter-warp 4 of them, so that neither the 8-byte reads (row groups 16 banks apart) nor the
// 16-byte column-major writes share a bank; the first 64 then take the halo's pairs. (One running
// index over all pairs: 3.9 M conflicts in 11.5 M wavefronts at 1024^2.)
template <int LF>
__device__ __forceinline__ void syn2_ypass(const float* __restrict__ s4, float* __restrict__ loT,
                                           float* __restrict__ hiT) {
  constexpr int half = LF / 2 - 1;
  constexpr int cs = (8 - half) & ~1;
  constexpr int NCR = (8 - cs) / 2;       // column pairs left of the tile's own 16
  const int l = threadIdx.x & 31;
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {
    int c = 8 + 2 * ((l & 3) | ((l >> 1) & 12)), rg = 2 * (threadIdx.x >> 5) + ((l >> 2) & 1);
    if (k) {
      if (threadIdx.x >= 64 || (l & 3) >= NCR) break;
      c = cs + 2 * (l & 3);
      rg = threadIdx.x >> 2;
    }
    u64 lo[4], hi[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) lo[t] = hi[t] = 0ull;
#pragma unroll
    for (int i = 0; i < half + 2; ++i) {
      const int o = (2 * rg + i) * kC2Pitch + c;
      const u64 vll = *reinterpret_cast<const u64*>(s4 + o);
      const u64 vlh = *reinterpret_cast<const u64*>(s4 + kC2Sub + o);
      const u64 vhl = *reinterpret_cast<const u64*>(s4 + 2 * kC2Sub + o);
      const u64 vhh = *reinterpret_cast<const u64*>(s4 + 3 * kC2Sub + o);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int j = t - 2 * (i - half);
        if (j >= 0 && j < LF) {
          const u64 ph = cdup(c_hd[half][j]), pg = cdup(c_gd[half][j]);
          lo[t] = ffma2(ph, vll, ffma2(pg, vlh, lo[t]));
          hi[t] = ffma2(ph, vhl, ffma2(pg, vhh, hi[t]));
        }
      }
    }
    float l0[4], l1[4], h0[4], h1[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      f2unpack(lo[t], l0[t], l1[t]);
      f2unpack(hi[t], h0[t], h1[t]);
    }
    *reinterpret_cast<float4*>(loT + c * kLoPitch + 4 * rg) = make_float4(l0[0], l0[1], l0[2], l0[3]);
    *reinterpret_cast<float4*>(loT + (c + 1) * kLoPitch + 4 * rg) = make_float4(l1[0], l1[1], l1[2], l1[3]);
    *reinterpret_cast<float4*>(hiT + c * kLoPitch + 4 * rg) = make_float4(h0[0], h0[1], h0[2], h0[3]);
    *reinterpret_cast<float4*>(hiT + (c + 1) * kLoPitch + 4 * rg) = make_float4(h1[0], h1[1], h1[2], h1[3]);
  }
}

// Along x for basis LF, accumulated into this thread's 4 x 4 block: rows 4 rq .. 4 rq + 3,
// columns 4 cg + t; acc[2t] holds rows (4rq, 4rq+1), acc[2t+1] rows (4rq+2, 4rq+3).
// Output column 4 cg + t reads staged column 8 - half + 2 cg + i through tap t - 2 (i - half).
template <int LF>
__device__ __forceinline__ void syn2_xpass(const float* __restrict__ loT, const float* __restrict__ hiT,
                                           u64 acc[8]) {
  constexpr int half = LF / 2 - 1;
  const int rq = threadIdx.x & 15, cg = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < half + 2; ++i) {
    const int col = 2 * cg + (8 - half) + i;
    const ulonglong2 vlo = *reinterpret_cast<const ulonglong2*>(loT + col * kLoPitch + 4 * rq);
    const ulonglong2 vhi = *reinterpret_cast<const ulonglong2*>(hiT + col * kLoPitch + 4 * rq);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int j = t - 2 * (i - half);
      if (j >= 0 && j < LF) {
        const u64 ph = cdup(c_hd[half][j]), pg = cdup(c_gd[half][j]);
        acc[2 * t] = ffma2(ph, vlo.x, ffma2(pg, vhi.x, acc[2 * t]));
        acc[2 * t + 1] = ffma2(ph, vlo.y, ffma2(pg, vhi.y, acc[2 * t + 1]));
      }
    }
  }
}

__device__ __forceinline__ void syn2_ypass_dispatch(int bi, const float* s4, float* loT, float* hiT) {
#define PS_Y(LFv) syn2_ypass<LFv>(s4, loT, hiT)
  PS_SWITCH_LF(bi, PS_Y)
#undef PS_Y
}
__device__ __forceinline__ void syn2_xpass_dispatch(int bi, const float* loT, const float* hiT, u64 acc[8]) {
#define PS_X(LFv) syn2_xpass<LFv>(loT, hiT, acc)
  PS_SWITCH_LF(bi, PS_X)
#undef PS_X
}

// Row rr (0..3) of this thread's 4 x 4 block.
__device__ __forceinline__ float4 syn2_row(const u64 acc[8], int rr) {
  float v[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    float a, b;
    f2unpack(acc[2 * t + (rr >> 1)], a, b);
    v[t] = (rr & 1) ? b : a;
  }
  return make_float4(v[0], v[1], v[2], v[3]);
}

static size_t syn2_smem() { return (size_t)(kC2Set + 2 * kLoSize) * sizeof(float) + 16; }

// After a bounded wait gave up somewhere in the CTA: raise the flag (when given),
// give the copies still in flight a bounded chance to land, and let the caller return.
__device__ __forceinline__ void syn2_abort(uint64_t* bar, uint32_t parity, int* err) {
  if (threadIdx.x == 0) {
    if (err) atomicExch(err, 1);
    (void)mbar_drain(bar, parity);
  }
  __syncthreads();
}

// Finest level: the eight bases plus the Dirac part summed in registers -> Psi A. One staging set,
// refilled with basis b+1 as soon as the y-pass of basis b has read it, so the copy overlaps the
// x-pass (4 CTAs per SM hide the rest; two sets at 3 CTAs per SM and a persistent form whose
// staging runs on across tiles were slower: 78 and 80 us at 1024^2 against 72). The basis after the one being
// staged is on its way to the L2 meanwhile (us per iteration: 2048^2 1046 -> 1042, 1024^2 421.3 -> 420.5; the same
// in the shared analysis tiles cost 2, and ahead of the dependency in the coarser synthesis 0.7 at 512^2).
__global__ void __launch_bounds__(256, 4)
    k_syn2_fine(const float* __restrict__ coef, const float* __restrict__ approx_in, int coarsest, int n,
                float* __restrict__ out, int* err, const __grid_constant__ SaraTma tm) {
  extern __shared__ __align__(128) float4 sm2[];
  pdl_wait();
  float* const s4 = reinterpret_cast<float*>(sm2);
  float* loT = s4 + kC2Set;
  float* hiT = loT + kLoSize;
  uint64_t* bar = reinterpret_cast<uint64_t*>(hiT + kLoSize);
  const int map = blockIdx.z, tilesx = n / kT2;
  const int oy0 = (blockIdx.x / tilesx) * kT2, ox0 = (blockIdx.x % tilesx) * kT2;
  const int hm = n >> 1;
  const float* cmap = coef + (size_t)map * kBases * n * n;
  auto issue = [&](int bi) {
    syn2_issue_t(tm, (map * kBases + bi + 1) * n, (map * kDb + bi) * hm, bi, cmap + (size_t)(bi + 1) * n * n,
                 coarsest ? nullptr : approx_in + ((size_t)map * kDb + bi) * (size_t)hm * hm, n, hm, oy0, ox0, s4, bar);
    if (bi + 1 < kDb)
      syn2_prefetch_t(tm, (map * kBases + bi + 2) * n, (map * kDb + bi + 1) * hm, bi + 1, coarsest, hm, oy0, ox0);
  };
  if (threadIdx.x == 0) mbar_init(bar, 1);
  __syncthreads();
  issue(0);
  u64 acc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) acc[q] = 0ull;
  for (int bi = 0; bi < kDb; ++bi) {
    const bool ok = mbar_wait(bar, bi & 1);
    // Also orders the previous x-pass' reads of loT/hiT before this y-pass writes them.
    if (__syncthreads_or(!ok)) {
      syn2_abort(bar, bi & 1, err);
      return;
    }
    syn2_ypass_dispatch(bi, s4, loT, hiT);
    __syncthreads();
    // The set is free once every y-pass read of it has passed the barrier above.
    if (bi + 1 < kDb) issue(bi + 1);
    syn2_xpass_dispatch(bi, loT, hiT, acc);
  }
  const int rq = threadIdx.x & 15, cg = threadIdx.x >> 4;
  const float k3 = 1.0f / 3.0f;
#pragma unroll
  for (int rr = 0; rr < 4; ++rr) {
    const size_t o = (size_t)(oy0 + 4 * rq + rr) * n + ox0 + 4 * cg;
    const float4 d = *reinterpret_cast<const float4*>(cmap + o);
    const float4 s = syn2_row(acc, rr);
    *reinterpret_cast<float4*>(out + (size_t)map * n * n + o) =
        make_float4((d.x + s.x) * k3, (d.y + s.y) * k3, (d.z + s.z) * k3, (d.w + s.w) * k3);
  }
}

// Coarser levels with output side m >= 64: one basis per CTA (grid.z, basis slowest), output to
// approximation scratch.
__global__ void __launch_bounds__(256, 3) k_syn2_lv(const float* __restrict__ coef, const float* __restrict__ approx_in,
                                                    int coarsest, int m, int n, float* __restrict__ approx_out,
                                                    int* err, const __grid_constant__ SaraTma tm) {
  extern __shared__ __align__(128) float4 sm2[];
  pdl_wait();
  float* s4 = reinterpret_cast<float*>(sm2);
  float* loT = s4 + kC2Set;
  float* hiT = loT + kLoSize;
  uint64_t* bar = reinterpret_cast<uint64_t*>(hiT + kLoSize);
  const int bi = blockIdx.z, map = blockIdx.y, tilesx = m / kT2;   // basis slowest, as k_ana_lv
  const int oy0 = (blockIdx.x / tilesx) * kT2, ox0 = (blockIdx.x % tilesx) * kT2;
  const int hm = m >> 1;
  const float* cb = coef + ((size_t)map * kBases + bi + 1) * (size_t)n * n;
  const float* apx = coarsest ? nullptr : approx_in + ((size_t)map * kDb + bi) * (size_t)hm * hm;
  if (threadIdx.x == 0) mbar_init(bar, 1);
  __syncthreads();
  syn2_issue_t(tm, (map * kBases + bi + 1) * n, (map * kDb + bi) * hm, bi, cb, apx, n, hm, oy0, ox0, s4, bar);
  const bool ok = mbar_wait(bar, 0);
  if (__syncthreads_or(!ok)) {
    syn2_abort(bar, 0, err);
    return;
  }
  syn2_ypass_dispatch(bi, s4, loT, hiT);
  __syncthreads();
  u64 acc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) acc[q] = 0ull;
  syn2_xpass_dispatch(bi, loT, hiT, acc);
  const int rq = threadIdx.x & 15, cg = threadIdx.x >> 4;
  float* dst = approx_out + ((size_t)map * kDb + bi) * (size_t)m * m;
#pragma unroll
  for (int rr = 0; rr < 4; ++rr)
    *reinterpret_cast<float4*>(dst + (size_t)(oy0 + 4 * rq + rr) * m + ox0 + 4 * cg) = syn2_row(acc, rr);
}



// ---------------------------------------------------------------------------
// Small levels in one launch: the analysis levels whose input side is at most kSmall, and
// the synthesis levels whose output side is at most kSmallSyn (for an image of side n <=
// kSmall: every level of both). One CTA per (basis, map) keeps the whole subtree on chip:
// its coefficients are one m0 x m0 block of the Mallat layout. These levels are bound by
// latency, not by bytes: the block (and, for the dual update, its thresholds) is read once,
// before the first level, the levels then run from shared memory in register strips of four
// outputs, and the block is written once at the end.
// 64 x 64, 4 levels, 4 maps (back-to-back launches): analysis 12.4 -> 10.8 us against one
// scalar pass per tap with the coefficients read level by level; synthesis 41.4 -> 10.4 us
// against the coarse levels in one launch and the eight bases one after another in the next.
constexpr int kSmall = 64;
constexpr int kSmallSyn = 32;     // above it (images larger than kSmall) the tiled synthesis is faster
constexpr int kSmallThreads = 256;
__host__ __device__ constexpr int small_pitch(int m) { return m + 20; }   // row pitch of a level's input (16 wrapped columns)

// One analysis level of side m. img: m rows of pitch small_pitch(m), columns m .. m + 15
// repeating the row's start (periodic). lo, hi: m rows of pitch hm + 4. The coefficients a
// (and thresholds t in the dual mode) are m0 x m0 blocks; the results replace a. The
// approximation replaces img in the layout of the next level.
// LFT: the filter length, or 0 for a loop over the taps of basis b (as ana_rows).
template <int LFT>
__device__ __forceinline__ void small_ana_level(int b, float* __restrict__ img, float* __restrict__ lo, float* __restrict__ hi,
                                                float* __restrict__ a, const float* __restrict__ t, int m, int m0,
                                                int last, int mode, float scale, float gamma, float delta) {
  const int LF = LFT ? LFT : 2 * b + 2;
  constexpr int U4 = LFT ? 4 : 1, U1 = LFT ? 16 : 2;   // steps unrolled: all, or one of the loop's
  const int hm = m >> 1, mask = m - 1, P = small_pitch(m), Q = hm + 4, PN = small_pitch(hm);
  auto epi = [&](float v, int o) {
    if (mode == SARA_DUAL) a[o] = fminf(fmaxf(fmaf(scale, v, a[o]), -t[o]), t[o]);
    else a[o] = mode == SARA_APPLY ? scale * v : gamma * delta / (delta + fabsf(scale * v));
  };
  if (hm >= 4) {
    for (int u = threadIdx.x; u < m * (hm >> 2); u += kSmallThreads) {
      const int r = u & mask, k0 = (u / m) * 4;
      const float4* row = reinterpret_cast<const float4*>(img + r * P + 2 * k0);
      float4 x0 = row[0], x1 = row[1];   // samples j .. j + 7 of the step's first tap j
      // One chain per output, in the order of the taps: a scalar FMA does as much per clock
      // as a packed one, and the coarse coefficients are the ones whose rounding shows most.
      // Four taps per step, and two at the end of every second filter (no zero taps, as in ana_rows).
      float l[4] = {0.f, 0.f, 0.f, 0.f}, h[4] = {0.f, 0.f, 0.f, 0.f};
      const int whole = LF & ~3;
#pragma unroll U4
      for (int j = 0; j < whole; j += 4) {
        const float4 x2 = row[2 + (j >> 2)];
        const float4 ch = *reinterpret_cast<const float4*>(&c_h[b][j]), cg = *reinterpret_cast<const float4*>(&c_g[b][j]);
        const float x[12] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w, x2.x, x2.y, x2.z, x2.w};
        const float th[4] = {ch.x, ch.y, ch.z, ch.w}, tg[4] = {cg.x, cg.y, cg.z, cg.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            l[q] = fmaf(th[i], x[2 * q + i], l[q]);
            h[q] = fmaf(tg[i], x[2 * q + i], h[q]);
          }
        x0 = x1, x1 = x2;
      }
      if (LF & 2) {
        const float2 ch = *reinterpret_cast<const float2*>(&c_h[b][whole]), cg = *reinterpret_cast<const float2*>(&c_g[b][whole]);
        const float x[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          l[q] = fmaf(ch.y, x[2 * q + 1], fmaf(ch.x, x[2 * q], l[q]));
          h[q] = fmaf(cg.y, x[2 * q + 1], fmaf(cg.x, x[2 * q], h[q]));
        }
      }
      *reinterpret_cast<float4*>(lo + r * Q + k0) = make_float4(l[0], l[1], l[2], l[3]);
      *reinterpret_cast<float4*>(hi + r * Q + k0) = make_float4(h[0], h[1], h[2], h[3]);
    }
    __syncthreads();
    const int qs = hm >> 2;   // column quads
    for (int u = threadIdx.x; u < hm * qs; u += kSmallThreads) {
      const int ky = u / qs, kx = (u - ky * qs) * 4;
      u64 ll0 = 0ull, ll1 = 0ull, lh0 = 0ull, lh1 = 0ull, hl0 = 0ull, hl1 = 0ull, hh0 = 0ull, hh1 = 0ull;
#pragma unroll U1
      for (int j = 0; j < LF; ++j) {
        const int o = ((2 * ky + j) & mask) * Q + kx;
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(lo + o);
        const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(hi + o);
        const u64 ph = cdup(c_hd[b][j]), pg = cdup(c_gd[b][j]);
        ll0 = ffma2(ph, x.x, ll0);
        ll1 = ffma2(ph, x.y, ll1);
        lh0 = ffma2(pg, x.x, lh0);
        lh1 = ffma2(pg, x.y, lh1);
        hl0 = ffma2(ph, y.x, hl0);
        hl1 = ffma2(ph, y.y, hl1);
        hh0 = ffma2(pg, y.x, hh0);
        hh1 = ffma2(pg, y.y, hh1);
      }
      auto epi4 = [&](float4 v, int o) {
        float4* dst = reinterpret_cast<float4*>(a + o);
        if (mode == SARA_DUAL) {
          *dst = f4clamp(f4fma(scale, v, *dst), *reinterpret_cast<const float4*>(t + o));
        } else if (mode == SARA_APPLY) {
          *dst = make_float4(scale * v.x, scale * v.y, scale * v.z, scale * v.w);
        } else {
          const float gd = gamma * delta;
          *dst = make_float4(gd / (delta + fabsf(scale * v.x)), gd / (delta + fabsf(scale * v.y)),
                             gd / (delta + fabsf(scale * v.z)), gd / (delta + fabsf(scale * v.w)));
        }
      };
      epi4(f4of(hl0, hl1), ky * m0 + hm + kx);            // x-high, y-low
      epi4(f4of(lh0, lh1), (hm + ky) * m0 + kx);          // x-low, y-high
      epi4(f4of(hh0, hh1), (hm + ky) * m0 + hm + kx);
      const float4 ll = f4of(ll0, ll1);
      if (last) {
        epi4(ll, ky * m0 + kx);
      } else {   // img was consumed by the row pass, before the barrier above
        for (int x = kx; x < hm + 16; x += hm) *reinterpret_cast<float4*>(img + ky * PN + x) = ll;
      }
    }
  } else {       // sides 4 and 2: a handful of outputs
    for (int u = threadIdx.x; u < m * hm; u += kSmallThreads) {
      const int r = u / hm, k = u - r * hm;
      float s = 0.f, d = 0.f;
#pragma unroll U1
      for (int j = 0; j < LF; ++j) {
        const float v = img[r * P + ((2 * k + j) & mask)];
        s = fmaf(c_h[b][j], v, s);
        d = fmaf(c_g[b][j], v, d);
      }
      lo[r * Q + k] = s;
      hi[r * Q + k] = d;
    }
    __syncthreads();
    for (int u = threadIdx.x; u < hm * hm; u += kSmallThreads) {
      const int ky = u / hm, kx = u - ky * hm;
      float ll = 0.f, lh = 0.f, hl = 0.f, hh = 0.f;
#pragma unroll U1
      for (int j = 0; j < LF; ++j) {
        const int o = ((2 * ky + j) & mask) * Q + kx;
        ll = fmaf(c_h[b][j], lo[o], ll);
        lh = fmaf(c_g[b][j], lo[o], lh);
        hl = fmaf(c_h[b][j], hi[o], hl);
        hh = fmaf(c_g[b][j], hi[o], hh);
      }
      epi(hl, ky * m0 + hm + kx);
      epi(lh, (hm + ky) * m0 + kx);
      epi(hh, (hm + ky) * m0 + hm + kx);
      if (last) epi(ll, ky * m0 + kx);
      else img[ky * PN + kx] = ll;
    }
  }
  __syncthreads();
}

// Analysis levels l0..L (sides m0 = n >> (l0 - 1) <= kSmall and below); one CTA per (basis,
// map) = (blockIdx.x, blockIdx.y). The input of level l0 is X (l0 = 1) or that level's
// approximation scratch (layout [map][basis][m0][m0]). LOOPS: filters as loops over the taps.
template <bool LOOPS>
__global__ void __launch_bounds__(kSmallThreads) k_ana_small(const float* __restrict__ in, int l0, int L, int n,
                                                             float* __restrict__ coef, float* __restrict__ thr,
                                                             int mode, float scale, float gamma, float delta) {
  extern __shared__ float4 smt[];
  pdl_wait();
  const int bi = blockIdx.x, map = blockIdx.y;
  const int m0 = n >> (l0 - 1), q0 = m0 >> 2, P = small_pitch(m0), Q = (m0 >> 1) + 4;
  float* img = reinterpret_cast<float*>(smt);
  float* lo = img + m0 * P;
  float* hi = lo + m0 * Q;
  float* a = hi + m0 * Q;
  float* t = a + m0 * m0;
  const float* src = l0 == 1 ? in + (size_t)map * n * n : in + ((size_t)map * kDb + bi) * (size_t)m0 * m0;
  const size_t base = ((size_t)map * kBases + (bi + 1)) * (size_t)n * n;
  for (int u = threadIdx.x; u < m0 * q0; u += kSmallThreads) {
    const int y = u / q0, x = (u - y * q0) * 4;
    const float4 v = *reinterpret_cast<const float4*>(src + (size_t)y * m0 + x);
    float4 va, vt;
    if (mode == SARA_DUAL) {
      va = *reinterpret_cast<const float4*>(coef + base + (size_t)y * n + x);
      vt = *reinterpret_cast<const float4*>(thr + base + (size_t)y * n + x);
    }
    for (int xx = x; xx < m0 + 16; xx += m0) *reinterpret_cast<float4*>(img + y * P + xx) = v;
    if (mode == SARA_DUAL) {
      *reinterpret_cast<float4*>(a + 4 * u) = va;
      *reinterpret_cast<float4*>(t + 4 * u) = vt;
    }
  }
  __syncthreads();
  for (int l = l0, m = m0; l <= L; ++l, m >>= 1) {
    if (LOOPS) {
      small_ana_level<0>(bi, img, lo, hi, a, t, m, m0, l == L, mode, scale, gamma, delta);
    } else {
#define PS_TA(LFv) small_ana_level<LFv>(bi, img, lo, hi, a, t, m, m0, l == L, mode, scale, gamma, delta)
      PS_SWITCH_LF(bi, PS_TA)
#undef PS_TA
    }
  }
  float* dst = (mode == SARA_REWEIGHT ? thr : coef) + base;
  for (int u = threadIdx.x; u < m0 * q0; u += kSmallThreads) {
    const int y = u / q0, x = (u - y * q0) * 4;
    *reinterpret_cast<float4*>(dst + (size_t)y * n + x) = *reinterpret_cast<const float4*>(a + 4 * u);
  }
}

// One synthesis level to output side m in place: the block's top-left m x m part (pitch B:
// approximation, then the details) becomes the m x m approximation of the next level. Along
// y into column-major intermediates (pitch m + 4), along x in 4 x 4 output blocks, as in
// syn2_ypass / syn2_xpass, with periodic indices.
template <int LF>
__device__ __forceinline__ void small_syn_level(float* __restrict__ blk, int B, int m, float* __restrict__ loT,
                                                float* __restrict__ hiT) {
  constexpr int b = LF / 2 - 1, half = LF / 2 - 1;
  const int hm = m >> 1, hmask = hm - 1, P = m + 4;
  if (hm == 1) {   // side 2: rows r and columns c of the four outputs
    if (threadIdx.x < 2) {
      const int r = threadIdx.x;
      float l = 0.f, h = 0.f;
#pragma unroll
      for (int j = 0; j < LF; ++j)
        if ((j & 1) == r) {
          l = fmaf(c_h[b][j], blk[0], fmaf(c_g[b][j], blk[B], l));
          h = fmaf(c_h[b][j], blk[1], fmaf(c_g[b][j], blk[B + 1], h));
        }
      loT[r] = l;
      hiT[r] = h;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
      const int r = threadIdx.x >> 1, c = threadIdx.x & 1;
      float v = 0.f;
#pragma unroll
      for (int j = 0; j < LF; ++j)
        if ((j & 1) == c) v = fmaf(c_h[b][j], loT[r], fmaf(c_g[b][j], hiT[r], v));
      blk[r * B + c] = v;
    }
    __syncthreads();
    return;
  }
  const int ncp = hm >> 1;
  for (int u = threadIdx.x; u < ncp * (m >> 2); u += kSmallThreads) {
    const int rg = u / ncp, c = 2 * (u - rg * ncp);
    u64 lo[4], hi[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) lo[t] = hi[t] = 0ull;
#pragma unroll
    for (int i = 0; i < half + 2; ++i) {
      const int kr = (2 * rg + i - half) & hmask;
      const u64 vll = *reinterpret_cast<const u64*>(blk + kr * B + c);
      const u64 vlh = *reinterpret_cast<const u64*>(blk + (hm + kr) * B + c);
      const u64 vhl = *reinterpret_cast<const u64*>(blk + kr * B + hm + c);
      const u64 vhh = *reinterpret_cast<const u64*>(blk + (hm + kr) * B + hm + c);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int j = t - 2 * (i - half);
        if (j >= 0 && j < LF) {
          const u64 ph = cdup(c_hd[b][j]), pg = cdup(c_gd[b][j]);
          lo[t] = ffma2(ph, vll, ffma2(pg, vlh, lo[t]));
          hi[t] = ffma2(ph, vhl, ffma2(pg, vhh, hi[t]));
        }
      }
    }
    float l0[4], l1[4], h0[4], h1[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      f2unpack(lo[t], l0[t], l1[t]);
      f2unpack(hi[t], h0[t], h1[t]);
    }
    *reinterpret_cast<float4*>(loT + c * P + 4 * rg) = make_float4(l0[0], l0[1], l0[2], l0[3]);
    *reinterpret_cast<float4*>(loT + (c + 1) * P + 4 * rg) = make_float4(l1[0], l1[1], l1[2], l1[3]);
    *reinterpret_cast<float4*>(hiT + c * P + 4 * rg) = make_float4(h0[0], h0[1], h0[2], h0[3]);
    *reinterpret_cast<float4*>(hiT + (c + 1) * P + 4 * rg) = make_float4(h1[0], h1[1], h1[2], h1[3]);
  }
  __syncthreads();
  const int nq = m >> 2;
  for (int u = threadIdx.x; u < nq * nq; u += kSmallThreads) {
    const int cg = u / nq, rq = u - cg * nq;
    u64 acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = 0ull;
#pragma unroll
    for (int i = 0; i < half + 2; ++i) {
      const int o = ((2 * cg + i - half) & hmask) * P + 4 * rq;
      const ulonglong2 vlo = *reinterpret_cast<const ulonglong2*>(loT + o);
      const ulonglong2 vhi = *reinterpret_cast<const ulonglong2*>(hiT + o);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int j = t - 2 * (i - half);
        if (j >= 0 && j < LF) {
          const u64 ph = cdup(c_hd[b][j]), pg = cdup(c_gd[b][j]);
          acc[2 * t] = ffma2(ph, vlo.x, ffma2(pg, vhi.x, acc[2 * t]));
          acc[2 * t + 1] = ffma2(ph, vlo.y, ffma2(pg, vhi.y, acc[2 * t + 1]));
        }
      }
    }
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) *reinterpret_cast<float4*>(blk + (4 * rq + rr) * B + 4 * cg) = syn2_row(acc, rr);
  }
  __syncthreads();
}

// out (this CTA's share of the rows of a tile) = (Dirac + sum over the cluster's partial
// tiles) / 3: the CTAs of a cluster hold the partial sums of their bases in their shared
// memory (`part`, ts rows of pitch B); the CTA of rank r writes rows [r, r + 1) ts / NS.
template <int NS>
__device__ __forceinline__ void cluster_sum(const float* part, int B, int ts, const float* __restrict__ dirac,
                                            float* __restrict__ out, int n) {
  const int rank = blockIdx.x % NS, q = ts >> 2;
  for (int u = threadIdx.x; u < ts / NS * q; u += blockDim.x) {
    const int y = rank * (ts / NS) + u / q, x = 4 * (u % q);
    const float4 d = *reinterpret_cast<const float4*>(dirac + (size_t)y * n + x);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < NS; ++r) {
      const float4 v = ld_cluster4(part + y * B + x, r);
      s = make_float4(s.x + v.x, s.y + v.y, s.z + v.z, s.w + v.w);
    }
    const float k3 = 1.0f / 3.0f;
    *reinterpret_cast<float4*>(out + (size_t)y * n + x) =
        make_float4((d.x + s.x) * k3, (d.y + s.y) * k3, (d.z + s.z) * k3, (d.w + s.w) * k3);
  }
}

// Synthesis levels L..l1 of one (basis, map) = (blockIdx.x, blockIdx.y); output side of level
// l1 at most kSmall. FINEST (l1 = 1): the eight CTAs of a map are a cluster and sum their
// bases and the Dirac part into Psi A; else the level-l1 output goes to approx_out
// ([map][basis][m][m]).
template <bool FINEST>
__device__ __forceinline__ void syn_small(const float* __restrict__ coef, int L, int l1, int n,
                                          float* __restrict__ dst) {
  extern __shared__ float4 smt[];
  pdl_wait();
  const int bi = blockIdx.x, map = blockIdx.y;
  const int m0 = n >> (l1 - 1), q0 = m0 >> 2, Bp = m0 + 4;
  float* blk = reinterpret_cast<float*>(smt);
  float* loT = blk + m0 * Bp;
  float* hiT = loT + (m0 >> 1) * (m0 + 4);
  const float* cmap = coef + (size_t)map * kBases * n * n;
  const float* cb = cmap + (size_t)(bi + 1) * n * n;
  for (int u = threadIdx.x; u < m0 * q0; u += kSmallThreads) {
    const int y = u / q0, x = (u - y * q0) * 4;
    *reinterpret_cast<float4*>(blk + y * Bp + x) = *reinterpret_cast<const float4*>(cb + (size_t)y * n + x);
  }
  __syncthreads();
  for (int l = L; l >= l1; --l) {
    const int m = n >> (l - 1);
#define PS_TS(LFv) small_syn_level<LFv>(blk, Bp, m, loT, hiT)
    PS_SWITCH_LF(bi, PS_TS)
#undef PS_TS
  }
  if (FINEST) {
    cluster_barrier();
    cluster_sum<kDb>(blk, Bp, m0, cmap, dst + (size_t)map * n * n, n);
    cluster_barrier();   // the partial images stay until every CTA has read them
  } else {
    float* o = dst + ((size_t)map * kDb + bi) * (size_t)m0 * m0;
    for (int u = threadIdx.x; u < m0 * q0; u += kSmallThreads) {
      const int y = u / q0, x = (u - y * q0) * 4;
      *reinterpret_cast<float4*>(o + 4 * u) = *reinterpret_cast<const float4*>(blk + y * Bp + x);
    }
  }
}
__global__ void __cluster_dims__(kDb, 1, 1) __launch_bounds__(kSmallThreads)
    k_syn_small(const float* __restrict__ coef, int L, int n, float* __restrict__ out) {
  syn_small<true>(coef, L, 1, n, out);
}
__global__ void __launch_bounds__(kSmallThreads)
    k_syn_tail(const float* __restrict__ coef, int L, int l1, int n, float* __restrict__ approx_out) {
  syn_small<false>(coef, L, l1, n, approx_out);
}

static size_t ana_small_smem(int m0) {
  return (size_t)(m0 * small_pitch(m0) + 2 * m0 * (m0 / 2 + 4) + 2 * m0 * m0) * sizeof(float);
}
static size_t syn_small_smem(int m0) { return (size_t)(m0 * (m0 + 4) + m0 * (m0 + 4)) * sizeof(float); }

// The finest level with the bases of a tile spread over the NS CTAs of a cluster (NS = 8:
// one basis each; NS = 4: db(r+1) and db(8-r), 18 taps in all for every rank), for images
// with too few 64 x 64 tiles to fill the chip: the CTA runs its bases through one staging
// set, leaves its partial tile in shared memory, and the cluster adds the partial tiles.
template <int NS>
__global__ void __cluster_dims__(NS, 1, 1) __launch_bounds__(256, 4)
    k_syn2_split(const float* __restrict__ coef, const float* __restrict__ approx_in, int coarsest, int n,
                 float* __restrict__ out, int* err, const __grid_constant__ SaraTma tm) {
  extern __shared__ __align__(128) float4 sm2[];
  __shared__ int failed;
  pdl_wait();
  float* const s4 = reinterpret_cast<float*>(sm2);
  float* loT = s4 + kC2Set;
  float* hiT = loT + kLoSize;
  uint64_t* bar = reinterpret_cast<uint64_t*>(hiT + kLoSize);
  const int rank = blockIdx.x % NS, tile = blockIdx.x / NS, map = blockIdx.z, tilesx = n / kT2;
  const int oy0 = (tile / tilesx) * kT2, ox0 = (tile % tilesx) * kT2, hm = n >> 1;
  const float* cmap = coef + (size_t)map * kBases * n * n;
  if (threadIdx.x == 0) {
    failed = 0;
    mbar_init(bar, 1);
  }
  __syncthreads();
  auto issue = [&](int bi) {
    syn2_issue_t(tm, (map * kBases + bi + 1) * n, (map * kDb + bi) * hm, bi, cmap + (size_t)(bi + 1) * n * n,
                 coarsest ? nullptr : approx_in + ((size_t)map * kDb + bi) * (size_t)hm * hm, n, hm, oy0, ox0, s4, bar);
  };
  u64 acc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) acc[q] = 0ull;
  constexpr int NB = kDb / NS;
  const int b_of[2] = {NS == kDb ? rank : kDb - 1 - rank, rank};
  issue(b_of[0]);
  for (int i = 0; i < NB; ++i) {
    const bool ok = mbar_wait(bar, i & 1);
    if (__syncthreads_or(!ok)) {   // the whole cluster's tile is left unwritten; its barriers are still met
      if (threadIdx.x == 0) failed = 1;
      syn2_abort(bar, i & 1, err);
      break;
    }
    const int bi = b_of[i];
    syn2_ypass_dispatch(bi, s4, loT, hiT);
    __syncthreads();
    if (i + 1 < NB) issue(b_of[1]);
    syn2_xpass_dispatch(bi, loT, hiT, acc);
  }
  // The staging set is free (the last y-pass has read it): it takes the partial tile.
  const int rq = threadIdx.x & 15, cg = threadIdx.x >> 4;
#pragma unroll
  for (int rr = 0; rr < 4; ++rr)
    *reinterpret_cast<float4*>(s4 + (4 * rq + rr) * kLoPitch + 4 * cg) = syn2_row(acc, rr);
  cluster_barrier();
  int bad = 0;
#pragma unroll
  for (int r = 0; r < NS; ++r) bad |= ld_cluster(&failed, r);
  const size_t o = (size_t)oy0 * n + ox0;
  if (!bad) cluster_sum<NS>(s4, kLoPitch, kT2, cmap + o, out + (size_t)map * n * n + o, n);
  cluster_barrier();   // the partial tiles stay until every CTA has read them
}
static_assert(kT2 * kLoPitch <= kC2Set, "a partial tile fits the staging set");
// (Tile, map) units up to which the bases are split. Eight ways while all 8 units' CTAs are
// resident at once (4 CTAs on each of 152 SMs), four ways while the four-way grid is at most
// two such waves; beyond that there are tiles enough, and the unsplit forms win. All of Psi,
// 4 maps, 4 levels, us unsplit / 4 / 8: 128^2 (16 units) 43 / 27 / 25, 256^2 (64) 51 / 37 / 36,
// 512^2 (256) 64 / 54 / 62, 1024^2 (1024, 6 levels) 133 / 147 / 182.
constexpr int kSplit8Units = 76, kSplit4Units = 304;

// ---- tensor maps (host side). cuTensorMapEncodeTiled comes from the driver through the
// runtime's entry-point query, so the library links against the runtime alone; without it
// (or when an encode fails) the kernels take the per-row bulk copies.
static PFN_cuTensorMapEncodeTiled_v12000 g_encode_tiled = nullptr;
static std::once_flag g_encode_once;

static bool tensor_maps_available() {
  std::call_once(g_encode_once, [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_encode_tiled = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    else
      cudaGetLastError();
  });
  return g_encode_tiled != nullptr;
}

// Map of a row-major float array of `height` rows of `width` floats, box bw x bh (zero fill
// outside). Returns 1 when made. The base must be 16-byte aligned and width * 4 a multiple of
// 16 (every array here: n, m, hm >= 16).
static int make_map(CUtensorMap* map, const float* base, uint64_t width, uint64_t height, uint32_t bw, uint32_t bh) {
  std::memset(map, 0, sizeof(*map));
  if (!base || !tensor_maps_available() || ((uintptr_t)base & 15u) || (width * 4) % 16 != 0 || bw > 256 || bh > 256 ||
      bw > width || bh > height)
    return 0;
  const cuuint64_t dims[2] = {width, height};
  const cuuint64_t strides[1] = {width * sizeof(float)};
  const cuuint32_t box[2] = {bw, bh};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = g_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides,
                                    box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 1 : 0;
}

// Maps of one tiled analysis level: input planes of side m (`planes` of them), and the
// coefficient and threshold arrays (36 n x n) for the staged epilogue operands.
static SaraTma analysis_maps(const float* in, int m, int planes, const float* coef, const float* thr, int n, int nmaps,
                             int mode) {
  SaraTma t;
  std::memset(&t, 0, sizeof(t));
  t.use_in = make_map(&t.in, in, (uint64_t)m, (uint64_t)planes * m, kA2Pitch, kRSmax);
  if (mode == SARA_DUAL)
    t.use_stage = make_map(&t.coef, coef, (uint64_t)n, (uint64_t)kBases * nmaps * n, kTO, kTO) &
                  make_map(&t.thr, thr, (uint64_t)n, (uint64_t)kBases * nmaps * n, kTO, kTO);
  return t;
}

// Maps of one tiled synthesis level of output side m: coefficients and, below the coarsest
// level, the 32 (map, basis) approximations of side m / 2.
static SaraTma synthesis_maps(const float* coef, const float* approx_in, int m, int n, int nmaps) {
  SaraTma t;
  std::memset(&t, 0, sizeof(t));
  t.use_scoef = make_map(&t.scoef, coef, (uint64_t)n, (uint64_t)kBases * nmaps * n, kC2Pitch, kC2Rows);
  if (approx_in)
    t.use_apx = make_map(&t.apx, approx_in, (uint64_t)(m / 2), (uint64_t)kDb * nmaps * (m / 2), kC2Pitch, kC2Rows);
  return t;
}

cudaError_t configure_nufft_kernels();

cudaError_t configure_kernels() {
  cudaError_t e;
  for (const void* f : {(const void*)k_ana_l1<false>, (const void*)k_ana_l1<true>, (const void*)k_ana_lv<false>,
                        (const void*)k_ana_lv<true>}) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)analysis_smem(false));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  for (const void* f : {(const void*)k_syn2_fine, (const void*)k_syn2_lv}) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)syn2_smem());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  e = cudaFuncSetAttribute((const void*)k_ana_l1m, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)analysis_smem(false));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute((const void*)k_ana_l1m, cudaFuncAttributePreferredSharedMemoryCarveout,
                           cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  for (const void* f : {(const void*)k_ana_small<false>, (const void*)k_ana_small<true>}) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ana_small_smem(kSmall));
    if (e != cudaSuccess) return e;
  }
  for (const void* f : {(const void*)k_syn2_split<8>, (const void*)k_syn2_split<4>}) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)syn2_smem());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return configure_nufft_kernels();
}

// (Tile, map) units of the first analysis level from which its tiles serve four bases per CTA; with
// fewer, one basis per CTA keeps more of the chip busy. us, one basis / four: 256^2 (64 units) 15 /
// 21, 512^2 (256) 27 / 34, 1024^2 (1024) 79 / 81 alone but 433 / 423 for the iteration, 2048^2 (4096) 286 / 283
// and 1063 / 1055; a batch whose 512^2 class has 512 units 415 / 411 per iteration (one basis with three
// CTAs per SM).
constexpr int kSharedTiles = 512;

// Levels of one basis per CTA with more CTAs than this per SM overlay the staged operands on the input
// tile: the waits of the warps in flight bound them, and a fourth CTA per SM hides more of them. Fewer
// CTAs are all resident (or nearly) as they are, and loading the operands early is the better use. us per
// iteration, beside / overlaid: 256^2 56.9 / 57.6 (level 1: 512 CTAs), 512^2 111.6 / 108.6 (2048), 1024^2 426.1 /
// 423.2 and 2048^2 (cone dual) 1057 / 1049 (levels 2 on: 2048 and 8192), a batch of 16 412 / 408.
// Without a dual update nothing is staged and the smaller CTA always serves (512^2, 5 levels 25.1 -> 24.4 us).
constexpr int kOverlayWaves = 4;

cudaError_t sara_analysis(Handle* h, const float* X, float* coef, float* thr, int mode, float scale, float gamma,
                          float delta, cudaEvent_t fine_done) {
  const int n = h->n, L = h->L;
  const int nmaps = h->nmaps;
  float* buf[2] = {h->approx, h->approx2};
  int lt = L + 1;                                   // first level of the fused tail
  for (int l = 1; l <= L; ++l)
    if ((n >> (l - 1)) <= kSmall) {
      lt = l;
      break;
    }
  // Levels with input side > kSmall: tiled, one launch per level (half side >= 128).
  for (int l = 1; l < lt; ++l) {
    const int m = n >> (l - 1), hm = m / 2;
    const dim3 grid((hm / kTO) * (hm / kTO), kDb, nmaps);
    const SaraTma tm = analysis_maps(l == 1 ? X : buf[(l - 2) & 1], m, l == 1 ? nmaps : kDb * nmaps, coef, thr, n, nmaps,
                                     mode);
    const bool over = mode != SARA_DUAL || (int)(grid.x * grid.y * grid.z) > kOverlayWaves * h->num_sms;
    const size_t smem = analysis_smem(over);
    if (l > 1) {
      launch_after(true, over ? k_ana_lv<true> : k_ana_lv<false>, grid, 256, smem, h->stream, buf[(l - 2) & 1], m, n,
                   l == L, coef, thr, buf[(l - 1) & 1], mode, scale, gamma, delta, h->dev_flags, tm);
      continue;
    }
    if ((int)(grid.x * grid.z) >= kSharedTiles)
      k_ana_l1m<<<dim3(grid.x, kDb / kL1Bases, nmaps), 256, analysis_smem(false), h->stream>>>(
          X, n, l == L, coef, thr, buf[0], mode, scale, gamma, delta, h->dev_flags, tm);
    else
      (over ? k_ana_l1<true> : k_ana_l1<false>)<<<grid, 256, smem, h->stream>>>(
          X, n, l == L, coef, thr, buf[0], mode, scale, gamma, delta, h->dev_flags, tm);
    if (fine_done) {
      const cudaError_t e = cudaEventRecord(fine_done, h->stream);
      if (e != cudaSuccess) return e;
    }
  }
  if (lt <= L) {
    const float* in = lt == 1 ? X : buf[(lt - 2) & 1];
    // Loops over the taps from 256^2 on (512^2 120 -> 113 us per iteration, 1024^2 446 -> 441: the eight
    // unrolled variants wait for instructions, and take their cache from the NUFFT kernels beside
    // them); unrolled below, where a pass is one chain of latencies (64^2 26.3 against 27.2, 128^2
    // 39.3 against 39.9).
    if (lt == 1)
      k_ana_small<false><<<dim3(kDb, nmaps), kSmallThreads, ana_small_smem(n), h->stream>>>(in, lt, L, n, coef, thr, mode,
                                                                                         scale, gamma, delta);
    else
      launch_after(true, n <= 128 ? k_ana_small<false> : k_ana_small<true>, dim3(kDb, nmaps), kSmallThreads, ana_small_smem(n >> (lt - 1)), h->stream, in, lt, L, n, coef,
                   thr, mode, scale, gamma, delta);
    if (lt == 1 && fine_done) {
      const cudaError_t e = cudaEventRecord(fine_done, h->stream);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaGetLastError();
}

// Psi A on `stream` with `approx` as the per-level approximation scratch
// (2 x 32 x (n/2)^2 floats); `err` (may be null) receives the bounded-wait flag.
static cudaError_t synthesis_levels(cudaStream_t stream, int n, int L, const float* coef, float* out, float* approx0,
                                    float* approx1, int nmaps, int* err, cudaEvent_t fine_start = nullptr) {
  float* buf[2] = {approx0, approx1};
  if (n <= kSmall) {
    if (fine_start) {
      const cudaError_t e = cudaEventRecord(fine_start, stream);
      if (e != cudaSuccess) return e;
    }
    return launch_after(true, k_syn_small, dim3(kDb, nmaps), kSmallThreads, syn_small_smem(n), stream, coef, L, n, out);
  }
  int lt = 0;                                       // lowest level of the fused tail (>= 2), 0: none
  for (int l = 2; l <= L; ++l)
    if ((n >> (l - 1)) <= kSmallSyn) {
      lt = l;
      break;
    }
  if (lt)
    launch_after(true, k_syn_tail, dim3(kDb, nmaps), kSmallThreads, syn_small_smem(n >> (lt - 1)), stream, coef, L, lt, n,
                 buf[(lt - 1) & 1]);
  for (int l = lt ? lt - 1 : L; l >= 1; --l) {      // every side m >= 64 here
    const int m = n >> (l - 1), tiles = (m / kT2) * (m / kT2);
    const float* ain = (l == L) ? nullptr : buf[l & 1];
    const SaraTma tm = synthesis_maps(coef, ain, m, n, nmaps);
    if (l > 1) {
      launch_after(true, k_syn2_lv, dim3(tiles, nmaps, kDb), 256, syn2_smem(), stream, coef, ain, l == L, m, n,
                   buf[(l - 1) & 1], err, tm);
      continue;
    }
    if (fine_start) {
      const cudaError_t e = cudaEventRecord(fine_start, stream);
      if (e != cudaSuccess) return e;
    }
    const int units = tiles * nmaps;
    if (units <= kSplit8Units)
      launch_after(true, k_syn2_split<8>, dim3(8 * tiles, 1, nmaps), 256, syn2_smem(), stream, coef, ain, l == L, n, out, err, tm);
    else if (units <= kSplit4Units)
      launch_after(true, k_syn2_split<4>, dim3(4 * tiles, 1, nmaps), 256, syn2_smem(), stream, coef, ain, l == L, n, out, err, tm);
    else
      launch_after(true, k_syn2_fine, dim3(tiles, 1, nmaps), 256, syn2_smem(), stream, coef, ain, l == L, n, out, err, tm);
  }
  return cudaGetLastError();
}

// First level of side at most `side` from level l on (L + 1: none).
static int first_level(int n, int L, int l, int side) {
  while (l <= L && (n >> (l - 1)) > side) ++l;
  return l;
}

int sara_launches(int n, int L) {
  const int la = first_level(n, L, 1, kSmall), ls = n <= kSmall ? 1 : first_level(n, L, 2, kSmallSyn);
  return (la - 1) + (la <= L) + (ls - 1) + (ls <= L);   // tiled levels and the fused small ones, each way
}

cudaError_t sara_synthesis(Handle* h, const float* coef, float* out, cudaEvent_t fine_start) {
  return synthesis_levels(h->stream, h->n, h->L, coef, out, h->approx, h->approx2, h->nmaps, h->dev_flags, fine_start);
}

// ---------------------------------------------------------------------------
// Allocation-free synthesis (ps_apply_psi_static). Its level scratch lives in
// this file-scope device array, sized for images up to kStaticMaxN; every GPU
// that loads the library holds it until the process exits.
constexpr int kStaticMaxN = 256;
constexpr size_t kStaticScratchFloats = 2ull * kDb * 4 * (kStaticMaxN / 2) * (kStaticMaxN / 2);   // 4 MiB
static __device__ __align__(256) float g_static_scratch[kStaticScratchFloats];
// Raised by a kernel of ps_apply_psi_static whose bounded wait gave up (cleared by each call).
static __device__ int g_static_err;

constexpr int kMaxDevices = 64;
static std::mutex g_static_mu;
static float* g_static_ptr[kMaxDevices] = {};    // device address of g_static_scratch, per device
static int* g_static_err_ptr[kMaxDevices] = {};  // device address of g_static_err, per device

// Sets this file's bounded-wait poll budget (ps_debug_set_wait_polls).
cudaError_t set_wait_polls_sara(int polls) { return set_wait_polls_here(polls); }

// A caller pointer of ps_apply_psi_static must be device or managed memory of the current device.
static bool device_pointer_here(const void* p, int dev) {
  cudaPointerAttributes a{};
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (a.type == cudaMemoryTypeManaged) return true;
  return a.type == cudaMemoryTypeDevice && a.device == dev;
}

}  // namespace ps

#pragma GCC visibility push(default)
extern "C" ps_status ps_apply_psi_static(const float* A, float* S, int32_t n, int32_t levels, void* cuda_stream) {
  using namespace ps;
  auto bad = [](const std::string& m) {
    set_global_error("apply_psi_static: " + m);
    return PS_EINVAL;
  };
  if (n < 16 || n > kStaticMaxN || (n & (n - 1)) != 0)
    return bad("n must be a power of two in [16, " + std::to_string(kStaticMaxN) + "] (static scratch limit)");
  if (levels < 1 || (n % (1 << levels)) != 0) return bad("levels must satisfy n divisible by 2^levels");
  if (!A || !S || ((uintptr_t)A & 15u) || ((uintptr_t)S & 15u))
    return bad("A and S must be non-null, 16-byte aligned device pointers");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    set_global_error(std::string("apply_psi_static: no usable current device: ") + cudaGetErrorString(e));
    return PS_ECUDA;
  }
  if (!device_pointer_here(A, dev) || !device_pointer_here(S, dev))
    return bad("A and S must point to device (or managed) memory of the current device");
  float* scratch = nullptr;
  int* flag = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_static_mu);
    if (!g_static_ptr[dev]) {
      // Set-up on this device, once: the device addresses of the scratch and the error
      // flag, and the filter taps.
      void* p = nullptr;
      void* q = nullptr;
      e = cudaGetSymbolAddress(&p, g_static_scratch);
      if (e == cudaSuccess) e = cudaGetSymbolAddress(&q, g_static_err);
      if (e != cudaSuccess) {
        set_global_error(std::string("apply_psi_static: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        return PS_ECUDA;
      }
      g_static_err_ptr[dev] = static_cast<int*>(q);
      double filt[kDb][kMaxTaps];
      daubechies_filters(filt);
      e = upload_filters(filt, (cudaStream_t)cuda_stream);
      if (e != cudaSuccess) {
        set_global_error(std::string("apply_psi_static: filter upload: ") + cudaGetErrorString(e));
        return PS_ECUDA;
      }
      e = configure_kernels();   // shared-memory limits of the kernels (function attributes, no allocation)
      if (e != cudaSuccess) {
        set_global_error(std::string("apply_psi_static: kernel attributes: ") + cudaGetErrorString(e));
        return PS_ECUDA;
      }
      g_static_ptr[dev] = static_cast<float*>(p);
    }
    scratch = g_static_ptr[dev];
    flag = g_static_err_ptr[dev];
  }
  e = cudaMemsetAsync(flag, 0, sizeof(int), (cudaStream_t)cuda_stream);
  if (e == cudaSuccess)
    e = synthesis_levels((cudaStream_t)cuda_stream, n, levels, A, S, scratch, scratch + kStaticScratchFloats / 2, 4, flag);
  if (e != cudaSuccess) {
    set_global_error(std::string("apply_psi_static: launch: ") + cudaGetErrorString(e));
    return PS_ECUDA;
  }
  return PS_OK;
}

extern "C" ps_status ps_static_status(void* cuda_stream) {
  using namespace ps;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    set_global_error(std::string("static_status: no usable current device: ") + cudaGetErrorString(e));
    return PS_ECUDA;
  }
  int* flag = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_static_mu);
    flag = g_static_err_ptr[dev];
  }
  e = cudaStreamSynchronize((cudaStream_t)cuda_stream);
  if (e != cudaSuccess) {
    set_global_error(std::string("static_status: ") + cudaGetErrorString(e));
    return PS_ECUDA;
  }
  if (!flag) return PS_OK;   // ps_apply_psi_static has not run on this device
  int v = 0;
  e = cudaMemcpy(&v, flag, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) {
    set_global_error(std::string("static_status: ") + cudaGetErrorString(e));
    return PS_ECUDA;
  }
  if (v) {
    set_global_error("apply_psi_static: a bounded device wait (bulk-copy barrier) gave up; S is incomplete");
    return PS_ETIMEOUT;
  }
  return PS_OK;
}
#pragma GCC visibility pop

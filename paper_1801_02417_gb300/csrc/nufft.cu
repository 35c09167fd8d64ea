// Measurement operator phi = Phi S L and its adjoint (Section 5.1, Eq. meas_op;
// Algorithm 1 steps 3 and 7), as a non-uniform FFT on the GPU.
//
// Phi = G F Z: Z de-apodises and zero-pads each map to the K = 2n grid, F is the
// K x K FFT, G interpolates the spectrum at each sampled frequency with a W x W
// "exponential of semicircle" kernel. The four real Stokes maps travel as two
// complex images, I + iQ and U + iV, so two complex FFTs serve four maps; the
// correlations are recovered from the spectrum at +u and -u (Hermitian
// symmetry of real maps) and mixed by L of Section 2.1 inside the degridding
// kernel. The spectrum is stored only on the window of frequencies the
// interpolation touches ([-R, R]^2), which prunes the column FFTs and the grid.
//
// Kernels (one launch each):
//   k_fwd_rows    row FFTs of the de-apodised, zero-padded rows     (n CTAs)
//   k_fwd_cols    column FFTs, kept on the window                    (Wd CTAs)
//   k_degrid      interpolation + Stokes->correlation mixing + dual update of B
//                 + per-block FP64 sums of ||B~/rho2 - Y||^2 and the l2-ball factors
//                                                                   (1 CTA / work item)
//   k_grid        mixing by conj(L) + gridding, one warp per run of rows
//   k_adj_cols    Hermitian symmetrisation + inverse column FFTs     (R+1 CTAs)
//   k_adj_rows    inverse row FFTs + crop + de-apodisation -> phi^dagger planes
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "packed.cuh"

namespace ps {

__device__ __forceinline__ float4 f4add(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 f4sub(float4 a, float4 b) {
  return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float4 f4fma(float s, float4 a, float4 acc) {
  return make_float4(fmaf(s, a.x, acc.x), fmaf(s, a.y, acc.y), fmaf(s, a.z, acc.z), fmaf(s, a.w, acc.w));
}
// Multiply both complex numbers held in a float4 by w.
__device__ __forceinline__ float4 cmul2(float4 a, float2 w) {
  return make_float4(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x,
                     a.z * w.x - a.w * w.y, a.z * w.y + a.w * w.x);
}
__device__ __forceinline__ int bitrev(int i, int logK) { return (int)(__brev((unsigned)i) >> (32 - logK)); }

// Bank-group swizzle of float4 indices in the FFT buffers. Bits 0-2 of an index
// pick one of the eight 16-byte bank groups of a 128-byte row; they are XORed with
// a linear (GF(2)) function of the higher bits chosen so that the eight lanes of a
// quarter-warp hit eight different groups in every access pattern of the
// transforms: the bit-reversed scatter (lanes differ in the top three index bits),
// the passes from stages 0, 1 and 2 on (lanes differ in the lowest three bits that the
// pass leaves alone), the later ones and the natural-order reads (bits 0-2). Being linear,
// fsw(a ^ d) = fsw(a) ^ fsw(d).
__device__ __forceinline__ int fsw(int i) {
  const int h = i >> 5;
  const int r = (h ^ (h >> 3) ^ (h >> 6)) & 7;   // bit t: XOR of index bits 5+t, 8+t, 11+t
  return i ^ ((i >> 3) & 1) ^ (((i >> 4) & 1) * 6) ^ ((r & 1) << 2) ^ (r >> 1);
}

// Twiddle p of radix-2 stage t (span 2^(t+1)): tw[2^t - 1 + p] = exp(-2 pi i p / 2^(t+1));
// each stage's twiddles are contiguous, so the lanes of a pass read consecutive words.
template <bool INV>
__device__ __forceinline__ float2 twid(const float2* __restrict__ tw, int idx) {
  float2 w = __ldg(tw + idx);
  if (INV) w.y = -w.y;
  return w;
}

// N radix-2 stages s .. s + N - 1 on the 2^N elements x (natural offsets j 2^s, j < 2^N) of one group in
// registers; pos: the group's position below bit s.
template <bool INV, int N>
__device__ __forceinline__ void fft_group(float4 (&x)[1 << N], const float2* __restrict__ tw, int s, int pos) {
#pragma unroll
  for (int t = 0; t < N; ++t) {
    // Stage s + t pairs offsets that differ in bit t; its twiddles depend on the bits below.
#pragma unroll
    for (int q = 0; q < (1 << t); ++q) {
      const float2 w = twid<INV>(tw, (1 << (s + t)) - 1 + pos + (q << s));
#pragma unroll
      for (int k = q; k < (1 << N); k += 2 << t) {
        const float4 u = x[k], v = cmul2(x[k + (1 << t)], w);
        x[k] = f4add(u, v);
        x[k + (1 << t)] = f4sub(u, v);
      }
    }
  }
}

// One pass over the nbuf buffers of K elements: stages s .. s + N - 1, a group per thread and turn.
template <bool INV, int N>
__device__ __forceinline__ void fft_pass(float4* buf, int nbuf, const float2* __restrict__ tw, int logK, int s) {
  int c[N];   // fsw is linear: the offset of element k is the XOR of those of its bits
#pragma unroll
  for (int k = 0; k < N; ++k) c[k] = fsw(1 << (s + k));
  auto at = [&](int a, int k) {
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (k >> q & 1) a ^= c[q];
    return a;
  };
  const int groups = 1 << (logK - N);
  for (int i = threadIdx.x; i < nbuf * groups; i += blockDim.x) {
    const int g = i & (groups - 1), pos = g & ((1 << s) - 1);
    float4* b = buf + ((i >> (logK - N)) << logK);
    const int a = fsw(((g >> s) << (s + N)) + pos);
    float4 x[1 << N];
#pragma unroll
    for (int k = 0; k < (1 << N); ++k) x[k] = b[at(a, k)];
    fft_group<INV, N>(x, tw, s, pos);
#pragma unroll
    for (int k = 0; k < (1 << N); ++k) b[at(a, k)] = x[k];
  }
  __syncthreads();
}

// In-place decimation-in-time FFT of nbuf sequences of K = 2^logK float4 (two complex sequences
// each) held in shared memory (swizzled by fsw) in bit-reversed order; output in natural
// order. INV selects exp(+2 pi i jk/K) (no 1/K normalisation). Shared-memory passes and their
// barriers bound these kernels, so three radix-2 stages go together: a thread takes 8 elements
// through them in registers, and the eight lanes of a quarter-warp fall into eight bank groups of
// fsw. What three does not divide ends in a pass of two stages or one. Forward and adjoint
// transforms (both kernels of each), radix-4 passes -> these: 117 -> 90 and 111 -> 90 us at 2048^2
// (K = 4096), 34.5 -> 30.5 and 34.8 -> 31 at 1024^2, equal below. Passes of four stages need 140 registers a thread:
// 110 and 94 us at 2048^2 but 23 and 18 for 16 at 512^2.
// Stages below s0 are taken as done (the caller wrote their output); stages from
// s_end on are left to the caller (fft_out).
template <bool INV>
__device__ void fft_smem(float4* buf, int nbuf, const float2* __restrict__ tw, int logK, int s0, int s_end) {
  int s = s0;
  for (; s + 3 <= s_end; s += 3) fft_pass<INV, 3>(buf, nbuf, tw, logK, s);
  if (s + 2 <= s_end) {
    fft_pass<INV, 2>(buf, nbuf, tw, logK, s);
    s += 2;
  }
  if (s < s_end) fft_pass<INV, 1>(buf, nbuf, tw, logK, s);
}

// Input of a K-point transform whose nonzero samples fill exactly one of each pair of
// natural indices (x, x + K/2), i.e. the bit-reversed neighbours (r, r ^ 1) that the
// first radix-2 stage combines (twiddle 1): that stage is folded into the scatter.
// Sample v at natural index idx writes both outputs of its pair, v at the even slot
// and +v or -v (idx < K/2 or not) at the odd one; fft_smem then starts at stage 1.
// Every slot is written, so the buffer needs no clearing.
__device__ __forceinline__ void scatter_stage0(float4* buf, int idx, int logK, float4 v) {
  const int r = bitrev(idx, logK);
  buf[fsw(r & ~1)] = v;
  buf[fsw(r | 1)] = (idx < (1 << (logK - 1))) ? v : make_float4(-v.x, -v.y, -v.z, -v.w);
}

// First of the stages fft_out finishes when the passes start at s0: one or two, such that whole passes
// of three remain; two where nothing would be left over (three cost 32.8 us for two's 31 in the adjoint
// transforms at 1024^2).
__device__ __forceinline__ int fft_tail_start(int logK, int s0) {
  const int rem = (logK - s0) % 3;
  return logK - (rem ? rem : 2);
}

// Natural-order output k of the transform whose stages below s_last are done in buf;
// its remaining one or two stages are applied here for this output alone (the same arithmetic as a
// pass), so a caller that needs few outputs skips that pass, its barrier and a buffer rewrite.
template <bool INV, int T>
__device__ __forceinline__ float4 fft_out_t(const float4* buf, const float2* __restrict__ tw, int s, int k) {
  const int hs = 1 << s, g = k & (hs - 1), a = fsw(g);
  float4 x[1 << T];
#pragma unroll
  for (int i = 0; i < (1 << T); ++i) x[i] = buf[a ^ fsw(i << s)];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const float2 w = twid<INV>(tw, (hs << t) - 1 + (k & ((hs << t) - 1)));
    const bool minus = (k >> (s + t)) & 1;
#pragma unroll
    for (int i = 0; i < (1 << T) >> (t + 1); ++i) {
      const float4 v = cmul2(x[2 * i + 1], w);
      x[i] = minus ? f4sub(x[2 * i], v) : f4add(x[2 * i], v);
    }
  }
  return x[0];
}
template <bool INV>
__device__ __forceinline__ float4 fft_out(const float4* buf, const float2* __restrict__ tw, int logK, int s_last,
                                          int k) {
  return logK - s_last == 1 ? fft_out_t<INV, 1>(buf, tw, s_last, k) : fft_out_t<INV, 2>(buf, tw, s_last, k);
}

__device__ __forceinline__ int gidx(int k, int off, int full, int K) {
  return full ? (k & (K - 1)) : (k + off);
}

// ---------------------------------------------------------------- forward
// CTAS: resident CTAs per SM that the registers leave room for. At K = 4096 a row's 64 KB of shared memory
// allows three, and the registers that more of them would cost are worth more (1084 us per iteration with five
// at 2048^2, 1056 with three). Up to K = 2048 the kernel runs beside the SARA branch: five (48 registers)
// leave that branch room, 425 us per iteration at 1024^2 where four give 431, although the transform alone
// is slower (30.7 us for 28.7).
template <int CTAS>
__global__ void __launch_bounds__(256, CTAS) k_fwd_rows(const float* __restrict__ X, int n, int N,
                                                  const float* __restrict__ corr,
                                                  const float2* __restrict__ tw, int K, int logK,
                                                  float4* __restrict__ T1, int Wd, int off, int full,
                                                  float4* __restrict__ clear, int nclear) {
  extern __shared__ float4 sm[];
  pdl_wait();
  // The accumulator of the gridding that follows in the chain (none: nclear = 0).
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nclear; i += gridDim.x * blockDim.x)
    clear[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  float4* buf = sm;
  const int p = blockIdx.x;
  const float cy = corr[p];
  const size_t row = (size_t)p * n;
  // The n samples sit at natural indices [0, n/2) and [K - n/2, K) of K = 2n: one per pair.
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    const int idx = (q - n / 2 + K) & (K - 1);
    const float c = cy * corr[q];
    const size_t o = row + q;
    scatter_stage0(buf, idx, logK, make_float4(X[o] * c, X[N + o] * c, X[2 * (size_t)N + o] * c,
                                               X[3 * (size_t)N + o] * c));
  }
  __syncthreads();
  const int st = fft_tail_start(logK, 1);
  fft_smem<false>(buf, 1, tw, logK, 1, st);
  for (int gx = threadIdx.x; gx < Wd; gx += blockDim.x) {
    const int k = full ? gx : gx - off;
    T1[(size_t)p * Wd + gx] = fft_out<false>(buf, tw, logK, st, (k + K) & (K - 1));
  }
}

__global__ void __launch_bounds__(512) k_fwd_cols(const float4* __restrict__ T1, int n,
                                                  const float2* __restrict__ tw, int K, int logK,
                                                  float4* __restrict__ G, int Wd, int off, int full) {
  extern __shared__ float4 sm[];
  pdl_wait();
  float4* buf = sm;
  const int gx = blockIdx.x;
  for (int p = threadIdx.x; p < n; p += blockDim.x) {
    const int idx = (p - n / 2 + K) & (K - 1);
    scatter_stage0(buf, idx, logK, T1[(size_t)p * Wd + gx]);
  }
  __syncthreads();
  const int st = fft_tail_start(logK, 1);
  fft_smem<false>(buf, 1, tw, logK, 1, st);
  for (int gy = threadIdx.x; gy < Wd; gy += blockDim.x) {
    const int k = full ? gy : gy - off;
    G[(size_t)gy * Wd + gx] = fft_out<false>(buf, tw, logK, st, (k + K) & (K - 1));
  }
}

// The kernel at offset t (cells).
template <int W>
__device__ __forceinline__ float es_weight(float t, float beta) {
  const float z = t * (2.0f / W), s = 1.0f - z * z;
  return s > 0.f ? __expf(beta * (s * rsqrtf(s) - 1.0f)) : 0.f;
}

// Polynomials of the kernel taps in f (|f| <= 1/2), fitted on the host in FP64 (es_table):
// tap j = E_j(f^2) + f O_j(f^2) and, the kernel being even, tap W-1-j = E_j(f^2) - f O_j(f^2).
// Coefficients duplicated in both halves of a 64-bit word, one table per width.
__constant__ __align__(16) float2 c_es[3][5][2 * kEsTerms];

cudaError_t upload_es_polys(cudaStream_t stream) {
  static_assert(sizeof(EsTable) == sizeof(c_es), "the table has the layout of c_es");
  return cudaMemcpyToSymbolAsync(c_es, es_table().c, sizeof(c_es), 0, cudaMemcpyHostToDevice, stream);
}

// The W x- and W y-weights of a row at once, two polynomials per packed FMA (lanes x, y):
// 34 packed FMAs for W = 7 in place of 14 square roots and exponentials, and closer to the
// kernel: at most 1e-7 of its peak off in FP32 (1.4e-7 at the very end of the outermost tap),
// the exponential form 7e-7. The outermost taps of W = 5 keep the exponentials: the square-root end of that kernel
// (height 1e-5) is not a polynomial, and below a tenth of the peak their error is as small.
template <int W>
__device__ __forceinline__ void es_weights_xy(float fx, float fy, float beta, float* wx, float* wy) {
  constexpr int q = (W - 5) / 2, hw = W / 2, j0 = W == 5 ? 1 : 0;
  const u64 f = f2pack(fx, fy), nf = f2pack(-fx, -fy), x = ffma2(f, f, 0ull);
  auto co = [&](int j, int k) { return *reinterpret_cast<const u64*>(&c_es[q][j][k]); };
#pragma unroll
  for (int j = j0; j <= hw; ++j) {
    u64 e = co(j, kEsTerms - 1);
#pragma unroll
    for (int k = kEsTerms - 2; k >= 0; --k) e = ffma2(e, x, co(j, k));
    if (j == hw) {   // the centre tap is even in f
      f2unpack(e, wx[j], wy[j]);
    } else {
      u64 o = co(j, 2 * kEsTerms - 1);
#pragma unroll
      for (int k = kEsTerms - 2; k >= 0; --k) o = ffma2(o, x, co(j, kEsTerms + k));
      f2unpack(ffma2(o, f, e), wx[j], wy[j]);
      f2unpack(ffma2(o, nf, e), wx[W - 1 - j], wy[W - 1 - j]);
    }
  }
  if constexpr (W == 5) {
    wx[0] = es_weight<W>(fx + hw, beta), wy[0] = es_weight<W>(fy + hw, beta);
    wx[W - 1] = es_weight<W>(fx - hw, beta), wy[W - 1] = es_weight<W>(fy - hw, beta);
  }
}

__device__ __forceinline__ void unpack_rec(float4 r, float& fx, float& fy, float& w, int& cx, int& cy) {
  fx = r.x;
  fy = r.y;
  w = r.z;
  const int pk = __float_as_int(r.w);
  cx = (int)(short)(pk & 0xFFFF);
  cy = pk >> 16;
}

// Second half of a degridding row m: from the interpolated packed spectra sp (at +u) and sn
// (at -u) to the row's visibilities (row mo of out) or residuals; returns its term of the
// per-block sums and its block (blk, left alone by DEG_APPLY).
__device__ __forceinline__ float degrid_finish(int m, int mo, float w, float4 sp, float4 sn, int mode, float2* __restrict__ R,
                                               const float2* __restrict__ Yv, const float* cb,
                                               float inv_rho2, const uint16_t* __restrict__ vblk,
                                               float2* __restrict__ out, int& blk) {
  float4* R4 = reinterpret_cast<float4*>(R);
  const float4* Y4 = reinterpret_cast<const float4*>(Yv);
  // G1 = F(I + iQ), G2 = F(U + iV); F(I) = (G1(u) + conj G1(-u))/2, F(Q) = (G1(u) - conj G1(-u))/(2i).
  const float FIr = 0.5f * (sp.x + sn.x), FIi = 0.5f * (sp.y - sn.y);
  const float FQr = 0.5f * (sp.y + sn.y), FQi = -0.5f * (sp.x - sn.x);
  float4 v01 = make_float4(w * (FIr + FQr), w * (FIi + FQi), w * sp.z, w * sp.w);   // RR, RL = G2(u)
  float4 v23 = make_float4(w * sn.z, -w * sn.w, w * (FIr - FQr), w * (FIi - FQi));  // LR = conj G2(-u), LL
  if (mode == DEG_APPLY) {
    float4* o4 = reinterpret_cast<float4*>(out);
    o4[2 * (size_t)mo] = v01;
    o4[2 * (size_t)mo + 1] = v23;
    return 0.f;
  }
  blk = vblk[m];
  const float4 y0 = Y4[2 * (size_t)m], y1 = Y4[2 * (size_t)m + 1];
  if (mode == DEG_DUAL) {
    const float cs = cb[blk] * inv_rho2;
    const float4 r0 = R4[2 * (size_t)m], r1 = R4[2 * (size_t)m + 1];
    v01 = f4sub(f4fma(cs, r0, v01), y0);
    v23 = f4sub(f4fma(cs, r1, v23), y1);
    R4[2 * (size_t)m] = v01;
    R4[2 * (size_t)m + 1] = v23;
  } else {
    v01 = f4sub(y0, v01);
    v23 = f4sub(y1, v23);
    if (out) {
      float4* o4 = reinterpret_cast<float4*>(out);
      o4[2 * (size_t)m] = v01;
      o4[2 * (size_t)m + 1] = v23;
    }
  }
  return (v01.x * v01.x + v01.y * v01.y + v01.z * v01.z + v01.w * v01.w) +
         (v23.x * v23.x + v23.y * v23.y + v23.z * v23.z + v23.w * v23.w);
}

// Adds every lane's e2 to the sum of its block blk (-1: none); all 32 lanes together. FP32
// over a warp's lanes of one block, FP64 in sums[]: this warp's own bins, or (shared) sums that
// other warps add to as well. Blocks that more than eight lanes share take one butterfly
// sum each (~15 instructions); the rest go by groups of equal blocks, all groups at once, a few
// instructions per lane of the largest.
__device__ __forceinline__ void block_add(int blk, float e2, bool shared, double* sums) {
  const int lane = threadIdx.x & 31;
  auto add = [&](int b, float v) {
    if (shared) atomicAdd(&sums[b], (double)v);
    else sums[b] += (double)v;
  };
  unsigned peers = __match_any_sync(0xffffffffu, blk);
  if (__any_sync(0xffffffffu, blk >= 0 && __popc(peers) > 8)) {
    unsigned todo = __ballot_sync(0xffffffffu, blk >= 0 && __popc(peers) > 8);
    while (todo) {   // at most three blocks have more than eight of the 32 lanes
      const int b = __shfl_sync(0xffffffffu, blk, __ffs(todo) - 1);
      const bool mine = blk == b;
      float v = mine ? e2 : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) add(b, v);
      if (mine) blk = -1;
      todo &= ~__ballot_sync(0xffffffffu, mine);
    }
  }
  __syncwarp();   // lane 0's sums before another lane's below, or in the next call
  if (__any_sync(0xffffffffu, blk >= 0)) {
    if (blk < 0) peers = 1u << lane;
    float v = 0.f;
    for (unsigned p = peers; p; p &= p - 1) v += __shfl_sync(peers, e2, __ffs(p) - 1);
    if (blk >= 0 && lane == __ffs(peers) - 1) add(blk, v);
    __syncwarp();
  }
}

// Ask L1 for the row's inputs of degrid_finish (R, Y: one 32-byte sector each) before the
// interpolation, so that their latency overlaps it instead of following it.
__device__ __forceinline__ void degrid_prefetch(int m, int mode, const float2* R, const float2* Yv) {
  if (mode == DEG_APPLY) return;
  asm volatile("prefetch.global.L1 [%0];" ::"l"(Yv + 4 * (size_t)m));
  if (mode == DEG_DUAL) asm volatile("prefetch.global.L1 [%0];" ::"l"(R + 4 * (size_t)m));
}

// One row of a degridding work item on the CUDA cores: the 2 W^2 taps read from the staged
// spectrum cells, then degrid_finish and block_add (warp-collective: every lane calls it).
template <int W>
__device__ __forceinline__ void degrid_row(int m, bool active, const GridItem& it, const float4* __restrict__ rec,
                                           const float4* Gp, const float4* Gn, int off, int full, int K, float beta,
                                           int mode, float2* __restrict__ R, const float2* __restrict__ Yv,
                                           const float* cb, float inv_rho2,
                                           const uint16_t* __restrict__ vblk, bool shared, double* sums,
                                           const int32_t* __restrict__ perm, float2* __restrict__ out) {
  constexpr int TS = kGridTile;
  constexpr int SS = TS + W - 1;
  int blk = -1;
  float e2 = 0.f;
  if (active) {
    degrid_prefetch(m, mode, R, Yv);
    const int mo = mode == DEG_APPLY && perm ? perm[m] : m;
    float fx, fy, w;
    int cx, cy;
    unpack_rec(rec[m], fx, fy, w, cx, cy);
    float wx[W], wy[W];
    es_weights_xy<W>(fx, fy, beta, wx, wy);
    // Local centre within the tile (tap j of +u at local j + lc; of -u at local (TS-1-lc) + j).
    const int lcy = gidx(cy, off, full, K) - it.ty * TS, lcx = gidx(cx, off, full, K) - it.tx * TS;
    const float4* gp = Gp + lcy * SS + lcx;
    const float4* gn = Gn + (TS - 1 - lcy) * SS + (TS - 1 - lcx);
    // Packed FP32x2: channels (x, y) and (z, w) of each float4 cell in one FMA each.
    u64 sp0 = 0ull, sp1 = 0ull, sn0 = 0ull, sn1 = 0ull;
#pragma unroll
    for (int jy = 0; jy < W; ++jy) {
      u64 ap0 = 0ull, ap1 = 0ull, an0 = 0ull, an1 = 0ull;
#pragma unroll
      for (int jx = 0; jx < W; ++jx) {
        const ulonglong2 vp = *reinterpret_cast<const ulonglong2*>(gp + jy * SS + jx);
        const ulonglong2 vn = *reinterpret_cast<const ulonglong2*>(gn + jy * SS + jx);
        const u64 kp = fdup(wx[jx]), kn = fdup(wx[W - 1 - jx]);
        ap0 = ffma2(kp, vp.x, ap0);
        ap1 = ffma2(kp, vp.y, ap1);
        an0 = ffma2(kn, vn.x, an0);
        an1 = ffma2(kn, vn.y, an1);
      }
      const u64 ky = fdup(wy[jy]), kny = fdup(wy[W - 1 - jy]);
      sp0 = ffma2(ky, ap0, sp0);
      sp1 = ffma2(ky, ap1, sp1);
      sn0 = ffma2(kny, an0, sn0);
      sn1 = ffma2(kny, an1, sn1);
    }
    float4 sp, sn;
    f2unpack(sp0, sp.x, sp.y);
    f2unpack(sp1, sp.z, sp.w);
    f2unpack(sn0, sn.x, sn.y);
    f2unpack(sn1, sn.z, sn.w);
    e2 = degrid_finish(m, mo, w, sp, sn, mode, R, Yv, cb, inv_rho2, vblk, out, blk);
  }
  if (mode != DEG_APPLY) block_add(blk, e2, shared, sums);
}

// Interpolate the packed spectra at +u and -u, unpack the four Stokes spectra,
// mix into RR, RL, LR, LL (Section 2.1) and weight by w_m. One CTA per gridding
// work item (rows whose tap centres lie in one kGridTile^2 tile): the spectrum
// cells every tap of the item can touch at +u, and the mirrored cells at -u, are
// staged in shared memory once; each thread then interpolates one row with taps at
// fixed offsets from its centre. Per-block sums of ||B~/rho2 - Y||^2 (DUAL) or
// ||Y - phi X||^2 (RESID): per row and per warp group of same-block lanes in FP32,
// then in FP64 through per-warp shared bins (up to kWarpBins blocks; shared FP64
// atomics beyond) and one global FP64 atomic per block and CTA; the last CTA to end takes
// the l2-ball step.
// The per-block sums and what becomes of them at the end of a launch: sum (cleared before and after),
// done (CTAs that have added theirs; 0 between launches), norm_sq, and the factors cb (null: kept).
struct BallStep {
  double* sum;
  int* done;
  double* norm_sq;
  float* cb;
  const double* eps;
  double rho2;
  int literal;
};

// Registers are capped for 6 CTAs per SM at W = 7 (40 of 67: more rows in flight per SM, 100
// against 111 us at 1024^2 / 2,000,000 rows; other widths would spill and run without a cap).
template <int W, bool APPLY>
__global__ void __launch_bounds__(256, W == 7 ? 6 : 0) k_degrid(
    const GridItem* __restrict__ items, const float4* __restrict__ rec, const float4* __restrict__ G, int Wd,
    int off, int full, int K, float beta, int step_mode, float2* __restrict__ R, const float2* __restrict__ Yv,
    const float* cb, float inv_rho2, const uint16_t* __restrict__ vblk, int nblocks, BallStep ball,
    const int32_t* __restrict__ perm, float2* __restrict__ out) {
  constexpr int TS = kGridTile;
  constexpr int SS = TS + W - 1;
  constexpr int hw = W / 2;
  extern __shared__ float4 smd[];
  float4* Gp = smd;                 // +u cells: grid rows/cols ty*TS - hw + [0, SS)
  float4* Gn = smd + SS * SS;       // -u cells: mirrored rows/cols -(ty*TS + TS-1) - hw + [0, SS)
  double* bsum = reinterpret_cast<double*>(smd + 2 * SS * SS);
  __shared__ int s_last;
  const int mode = APPLY ? (int)DEG_APPLY : step_mode;
  pdl_wait();
  const GridItem it = items[blockIdx.x];
  const bool reduce = (mode != DEG_APPLY);
  const bool private_bins = nblocks <= kWarpBins;   // per-warp bins: kWarpBins x 8 warps doubles
  const int nbins = private_bins ? kWarpBins * (blockDim.x >> 5) : nblocks;
  if (reduce)
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) bsum[b] = 0.0;
  // Grid frequency (k) of local row 0: +u region starts at tile origin - hw; the -u region
  // holds frequencies -(centre) - hw + j for every centre of the tile.
  const int ky0 = it.ty * TS - hw - (full ? 0 : off), kx0 = it.tx * TS - hw - (full ? 0 : off);
  const int nky0 = -(it.ty * TS + TS - 1 - (full ? 0 : off)) - hw, nkx0 = -(it.tx * TS + TS - 1 - (full ? 0 : off)) - hw;
  for (int i = threadIdx.x; i < SS * SS; i += blockDim.x) {
    const int ly = i / SS, lx = i - (i / SS) * SS;
    int py = ky0 + ly, px = kx0 + lx, ny = nky0 + ly, nx = nkx0 + lx;
    float4 vp = make_float4(0.f, 0.f, 0.f, 0.f), vn = vp;
    if (full) {
      vp = G[(size_t)(py & (K - 1)) * Wd + (px & (K - 1))];
      vn = G[(size_t)(ny & (K - 1)) * Wd + (nx & (K - 1))];
    } else {
      py += off; px += off; ny += off; nx += off;
      if (py >= 0 && py < Wd && px >= 0 && px < Wd) vp = G[(size_t)py * Wd + px];
      if (ny >= 0 && ny < Wd && nx >= 0 && nx < Wd) vn = G[(size_t)ny * Wd + nx];
    }
    Gp[i] = vp;
    Gn[i] = vn;
  }
  __syncthreads();
  double* sums = bsum + (private_bins ? (threadIdx.x >> 5) * kWarpBins : 0);
  for (int base = it.vstart; base < it.vend; base += blockDim.x) {
    const int m = base + threadIdx.x;
    degrid_row<W>(m, m < it.vend, it, rec, Gp, Gn, off, full, K, beta, mode, R, Yv, cb, inv_rho2, vblk, !private_bins,
                  sums, perm, out);
  }
  if (reduce) {
    __syncthreads();
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
      double t = 0.0;
      if (private_bins)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += bsum[w * kWarpBins + b];
      else
        t = bsum[b];
      if (t != 0.0) atomicAdd(&ball.sum[b], t);
    }
    // The CTA that finds every other one done turns the sums into the l2-ball factors
    // (Algorithm 1 step 8: with r = ||B~/rho2 - Y||_b, c_b = rho2 (1 - min(1, radius / r))) and
    // leaves the sums cleared for the next launch.
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(ball.done, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (s_last) {
      __threadfence();
      for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
        const double q = __ldcg(&ball.sum[b]);
        ball.sum[b] = 0.0;
        ball.norm_sq[b] = q;
        if (ball.cb) {
          const double r = sqrt(q);
          const double radius = ball.literal ? ball.eps[b] / ball.rho2 : ball.eps[b];
          ball.cb[b] = (float)(ball.rho2 * (1.0 - (r > radius ? radius / r : 1.0)));
        }
      }
      if (threadIdx.x == 0) *ball.done = 0;
    }
  }
}

template <int W>
static constexpr size_t degrid_smem_tiles() {
  return (size_t)2 * (kGridTile + W - 1) * (kGridTile + W - 1) * sizeof(float4);
}

// Gridding (adjoint of the interpolation), Alg. 1 step 3's phi^dagger. Rows are stored sorted
// by tap-centre cell; a warp takes `rows` consecutive rows, 32 at a time, on its own:
//  1. lane = row: the row is read, mixed by conj(L) (x_I = RR + LL, x_Q = RR - LL, x_U = RL + LR,
//     x_V = i (LR - RL)), scaled by c_b w_m, and left in the warp's shared-memory buffer with its
//     W y- and x-weights (es_weights_xy); the next 32 rows are read meanwhile.
//  2. Per run of rows of one cell, the cell's W x W x 8 block is accumulated in registers in FP32: a lane
//     owns one channel and NY stencil rows, all their columns as packed pairs; per row it forms x_c w_y
//     and adds its products with the w_x pairs (fma.rn.f32x2).
//  3. Where the cell ends, the block goes to shared memory and from there to the accumulator
//     by W bulk reductions (one per stencil row, W cells of 32 bytes; two where the row wraps
//     around a full grid), which run while the warp goes on with its next cell.
//  4. MERGE: the last blocks of neighbouring warps that belong to one cell are added up in shared
//     memory first, so that a cell of many rows is few partial sums (launch_grid says when).
// Channels are gridded at +u only; k_adj_cols forms the -u half by Hermitian symmetrisation.
//
// But for that merge nothing is shared between warps: no barrier, no uneven end of a work item, no list of
// work, and no FP32 atomic on shared memory (a compare-and-swap loop). Products and sums are FP32 FMAs: per
// row a lane issues four shared loads, NY products and NY NX packed FMAs, about 17 instructions for the warp's
// 392 products at W = 7. As TF32 tensor-core products (m16n8k8, operands split in two) the splits and the
// fragments' loads took more than that, a lone row cost as much as eight, and 22 bits per operand showed in
// the result. phi^dagger, us, tensor cores / this: 1024^2 / 2,000,000 rows (34 per cell) 114 / 112, 2048^2 / 700,001
// (4 per cell) 184 / 161, 1024^2 / 200,001 scattered rows (1 per cell) 173 / 163, 1024^2 / 2,000,001 scattered 602 /
// 471, W = 9 there 910 / 705; error against the same interpolation in FP64, 128^2 / 165,337 rows, W = 5 2.8e-7 /
// 1.6e-7, W = 9 at 32^2 / 200,001 1.1e-6 / 2.6e-7. Grid stage: 1024^2 / 2,000,000 86 / 82 us, 2048^2 / 700,001 94 / 73.
// Bound by the L1 data pipe (83%: the rows' broadcast loads), issue at 64%.
constexpr int kGridWarps = 4;     // warps of a CTA
constexpr int kMergeWarps = 8;   // warps of a CTA that merges its warps' last blocks
template <int W>
struct GridWarp {
  static constexpr int NY = W == 9 ? 3 : 2, NX = (W + 1) / 2;   // stencil rows of a lane, pairs of columns
  static constexpr int YP = W == 9 ? 12 : 8;        // y-weights per row: NY (W = 9: and one unused) per lane quarter
  static constexpr int XP = 2 * NX <= 8 ? 8 : 12;   // x-weights per row (2 NX used)
  static constexpr int SP = W == 9 ? 88 : 8 * W + 4;   // stage pitch of a stencil row (NY SP = 8 or 24 mod 32 banks)
  static constexpr int kRow = 32 * (8 + YP + XP);              // floats of the row buffer
  static constexpr int kFloats = kRow + 2 * ((W * SP + 3) / 4 * 4);   // + two staged blocks
};
// No bound on the registers (64 to 102): 64 a thread (eight CTAs per SM) gives 84.6 us per grid stage at 1024^2 for 82,
// a bound so loose that the loop takes 154 gives 429 us per iteration for 418. Eight rows of the loop
// unrolled: 82 us, two 88.
template <int W, bool PERM, bool MERGE>
__global__ void __launch_bounds__(32 * (MERGE ? kMergeWarps : kGridWarps)) k_grid(
    int M, int rows, const uint16_t* __restrict__ vblk, const float4* __restrict__ rec, const float2* __restrict__ vin,
    const int32_t* __restrict__ perm,
    const float* __restrict__ cb, int use_scale, int Wd, int off, int full, int K, float beta,
    float* __restrict__ Acc) {
  using T = GridWarp<W>;
  constexpr int NY = T::NY, NX = T::NX, hw = W / 2;
  extern __shared__ __align__(16) float4 smw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* xs = reinterpret_cast<float*>(smw) + warp * T::kFloats;   // 8 channels per row
  float* wyb = xs + 32 * 8;
  float* wxb = wyb + 32 * T::YP;
  float* stage = xs + T::kRow;
  constexpr int kStageF = (T::kFloats - T::kRow) / 2;
  const long long first = (long long)(blockIdx.x * (MERGE ? kMergeWarps : kGridWarps) + warp) * rows;
  pdl_wait();
  if (!MERGE && first >= M) return;
  const int m0 = (int)min((long long)M, first), m1 = (int)min((long long)M, first + rows);
  const float4* v4 = reinterpret_cast<const float4*>(vin);
  const int g = lane >> 2, jy0 = NY * (W == 9 ? min(lane & 3, 2) : lane & 3);   // channel, first stencil row
  u64 d[NY][NX];   // cells (jy0 + y, 2 t) and (jy0 + y, 2 t + 1) of channel g
#pragma unroll
  for (int y = 0; y < NY; ++y)
#pragma unroll
    for (int t = 0; t < NX; ++t) d[y][t] = 0ull;
  float4 r, b0, b1;
  int blk = 0, buf = 0, cell = -1;   // cell: the accumulated block's (grid row << 12 | column), -1: none
  // vin in stored order, or (PERM) in the caller's; the index of a row is read one step ahead of it.
  int next = PERM && m0 < m1 ? perm[min(m0 + lane, m1 - 1)] : 0;
  auto fetch = [&](int m) {
    const size_t i = min(m + lane, m1 - 1), v = PERM ? next : i;
    r = rec[i];
    b0 = v4[2 * v];
    b1 = v4[2 * v + 1];
    if (PERM) next = perm[min(m + 32 + lane, m1 - 1)];
    if (use_scale) blk = vblk[i];
  };
  // The block to a stage buffer; from there to the accumulator.
  auto store = [&](float* st) {
    bulk_wait_read<1>();   // this lane's reductions of two cells ago have read their buffer
    __syncwarp();
#pragma unroll
    for (int y = 0; y < NY; ++y)
#pragma unroll
      for (int t = 0; t < NX; ++t) {
        float v0, v1;
        f2unpack(d[y][t], v0, v1);
        d[y][t] = 0ull;
        if (jy0 + y >= W) continue;
        float* o = st + (jy0 + y) * T::SP + 16 * t + g;
        o[0] = v0;
        if (2 * t + 1 < W) o[8] = v1;
      }
  };
  auto reduce = [&](const float* st) {
    if (lane < W) {
      const int gy = (cell >> 12) - hw + lane, gx = (cell & 4095) - hw;
      const float* src = st + lane * T::SP;
      if (!full) {
        bulk_reduce_add(Acc + 8 * ((size_t)gy * Wd + gx), src, W * 32);
      } else {
        float* row = Acc + 8 * (size_t)(gy & (K - 1)) * Wd;
        const int x0 = gx & (K - 1), n0 = min(W, K - x0);
        bulk_reduce_add(row + 8 * (size_t)x0, src, n0 * 32);
        if (n0 < W) bulk_reduce_add(row, src + 8 * n0, (W - n0) * 32);
      }
    }
    bulk_commit();
  };
  auto flush = [&]() {
    float* st = stage + buf * kStageF;
    store(st);
    fence_proxy_async();
    __syncwarp();
    reduce(st);
    buf ^= 1;
  };
  if (!MERGE || m0 < m1) fetch(m0);
  for (int m = m0; m < m1; m += 32) {
    const int cnt = min(32, m1 - m);
    int key;
    {
      float fx, fy, w;
      int cx, cy;
      unpack_rec(r, fx, fy, w, cx, cy);
      key = gidx(cy, off, full, K) << 12 | gidx(cx, off, full, K);   // lanes past the rows repeat the last row's
      const float sc = lane < cnt ? (use_scale ? cb[blk] : 1.0f) * w : 0.f;
      float4* xo = reinterpret_cast<float4*>(xs) + 2 * lane;
      xo[0] = make_float4(sc * (b0.x + b1.z), sc * (b0.y + b1.w), sc * (b0.x - b1.z), sc * (b0.y - b1.w));
      xo[1] = make_float4(sc * (b0.z + b1.x), sc * (b0.w + b1.y), -sc * (b1.y - b0.w), sc * (b1.x - b0.z));
      float4* yo = reinterpret_cast<float4*>(wyb + T::YP * lane);
      float4* po = reinterpret_cast<float4*>(wxb + T::XP * lane);
      float wx[W], wy[W];
      es_weights_xy<W>(fx, fy, beta, wx, wy);
      auto at = [](const float* v, int k) { return k < W ? v[k < W ? k : 0] : 0.f; };
#pragma unroll
      for (int q = 0; q < T::YP / 4; ++q)
        yo[q] = W == 9 ? make_float4(at(wy, 3 * q), at(wy, 3 * q + 1), at(wy, 3 * q + 2), 0.f)
                       : make_float4(at(wy, 4 * q), at(wy, 4 * q + 1), at(wy, 4 * q + 2), at(wy, 4 * q + 3));
#pragma unroll
      for (int q = 0; q < T::XP / 4; ++q)
        po[q] = make_float4(at(wx, 4 * q), at(wx, 4 * q + 1), at(wx, 4 * q + 2), at(wx, 4 * q + 3));
    }
    if (m + 32 < m1) fetch(m + 32);
    // Rows that start a run of another cell than the row before them.
    const int before = __shfl_up_sync(0xffffffffu, key, 1);
    unsigned starts = __ballot_sync(0xffffffffu, lane > 0 && key != before);
    __syncwarp();
    for (int a = 0; a < cnt;) {
      const int end = starts ? __ffs(starts) - 1 : cnt;
      starts &= starts - 1;
      const int k = __shfl_sync(0xffffffffu, key, a);
      if (cell >= 0 && k != cell) flush();
      cell = k;
#pragma unroll 8
      for (int v = a; v < end; ++v) {
        const float x = xs[8 * v + g];
        float wy[4];
        if constexpr (NY == 2) {
          const float2 w2 = *reinterpret_cast<const float2*>(wyb + T::YP * v + jy0);
          wy[0] = w2.x, wy[1] = w2.y;
        } else {
          const float4 w4 = *reinterpret_cast<const float4*>(wyb + T::YP * v + jy0 / 3 * 4);
          wy[0] = w4.x, wy[1] = w4.y, wy[2] = w4.z;
        }
        u64 wx[T::XP / 2];
#pragma unroll
        for (int q = 0; q < (NX + 1) / 2; ++q) {
          const ulonglong2 w4 = reinterpret_cast<const ulonglong2*>(wxb + T::XP * v)[q];
          wx[2 * q] = w4.x, wx[2 * q + 1] = w4.y;
        }
#pragma unroll
        for (int y = 0; y < NY; ++y) {
          const u64 p = fdup(x * wy[y]);
#pragma unroll
          for (int t = 0; t < NX; ++t) d[y][t] = ffma2(p, wx[t], d[y][t]);
        }
      }
      a = end;
    }
    __syncwarp();   // the row buffer is read before the next rows replace it
  }
  if constexpr (MERGE) {
    // Neighbouring warps whose last blocks belong to one cell: the first of them takes the sum.
    __shared__ int s_cell[kMergeWarps], s_buf[kMergeWarps];   // a warp without rows comes after all others (cell -1)
    if (cell >= 0) store(stage + buf * kStageF);
    if (lane == 0) s_cell[warp] = cell, s_buf[warp] = buf;
    __syncthreads();
    float* base = reinterpret_cast<float*>(smw) + T::kRow;
    int c[kMergeWarps], at[kMergeWarps];   // the cells and where their blocks are
#pragma unroll
    for (int v = 0; v < kMergeWarps; ++v) c[v] = s_cell[v], at[v] = v * T::kFloats + s_buf[v] * kStageF;
    for (int i = threadIdx.x; i < W * T::SP; i += blockDim.x) {
      if (i % T::SP >= 8 * W) continue;   // the pitch's unused floats
      float x[kMergeWarps];
#pragma unroll
      for (int v = 0; v < kMergeWarps; ++v) x[v] = c[v] >= 0 ? base[at[v] + i] : 0.f;
      int lead = at[0];
      float sum = x[0];
#pragma unroll
      for (int v = 1; v < kMergeWarps; ++v) {
        if (c[v] == c[v - 1]) {
          sum += x[v];
        } else {
          base[lead + i] = sum;
          lead = at[v];
          sum = x[v];
        }
      }
      if (c[kMergeWarps - 1] >= 0) base[lead + i] = sum;
    }
    fence_proxy_async();
    __syncthreads();
    if (cell >= 0 && (warp == 0 || s_cell[warp - 1] != cell)) reduce(stage + buf * kStageF);
  } else {
    flush();
  }
  bulk_wait_all();   // the reductions are done before the CTA's shared memory goes
}

// Hermitian symmetrisation + inverse column FFTs for the column pair (kx, -kx).
// H1(k) = P1(k) + i Q1(k), P1(k) = aI(k) + conj aI(-k), Q1(k) = aQ(k) + conj aQ(-k);
// H2 likewise from aU, aV. H(-k) = conj P(k) + i conj Q(k).
__global__ void __launch_bounds__(512) k_adj_cols(const float4* __restrict__ Acc, int n,
                                                  const float2* __restrict__ tw, int K, int logK,
                                                  float4* __restrict__ T2, int Wd, int off, int full) {
  extern __shared__ float4 sm[];
  pdl_wait();
  float4* bp = sm;
  float4* bm = sm + K;
  const int kx = blockIdx.x;
  const int self = (kx == 0) || (full && kx == K / 2);
  const int gxp = gidx(kx, off, full, K), gxm = gidx(-kx, off, full, K);
  // H(ky) of this column pair: hp for +kx (slot ky of bp), hm for -kx (slot -ky of bm).
  auto hpm = [&](int ky, float4& hp, float4& hm) {
    const int gy = gidx(ky, off, full, K), gym = gidx(-ky, off, full, K);
    const float4 a0 = Acc[2 * ((size_t)gy * Wd + gxp)], a1 = Acc[2 * ((size_t)gy * Wd + gxp) + 1];
    const float4 b0 = Acc[2 * ((size_t)gym * Wd + gxm)], b1 = Acc[2 * ((size_t)gym * Wd + gxm) + 1];
    const float P1r = a0.x + b0.x, P1i = a0.y - b0.y, Q1r = a0.z + b0.z, Q1i = a0.w - b0.w;
    const float P2r = a1.x + b1.x, P2i = a1.y - b1.y, Q2r = a1.z + b1.z, Q2i = a1.w - b1.w;
    hp = make_float4(P1r - Q1i, P1i + Q1r, P2r - Q2i, P2i + Q2r);
    hm = make_float4(P1r + Q1i, -P1i + Q1r, P2r + Q2i, -P2i + Q2r);
  };
  int st;
  if (!full && 8 * off < K) {
    // As in k_adj_rows: the window [-R, R] with R < K/8 puts at most one sample in each
    // block of natural indices x + j K/4, so the first two inverse stages are written
    // directly (v (i^{j t})_t, j = 0 or 3) and fft_smem starts at stage 2.
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    auto put4 = [&](float4* b, int r0, int j, float4 v) {
      if (j == 0) {
        b[fsw(r0)] = b[fsw(r0 + 1)] = b[fsw(r0 + 2)] = b[fsw(r0 + 3)] = v;
      } else if (j == 3) {
        b[fsw(r0)] = v;
        b[fsw(r0 + 1)] = make_float4(v.y, -v.x, v.w, -v.z);
        b[fsw(r0 + 2)] = make_float4(-v.x, -v.y, -v.z, -v.w);
        b[fsw(r0 + 3)] = make_float4(-v.y, v.x, -v.w, v.z);
      } else {
        b[fsw(r0)] = b[fsw(r0 + 1)] = b[fsw(r0 + 2)] = b[fsw(r0 + 3)] = z;
      }
    };
    for (int x = threadIdx.x; x < (K >> 2); x += blockDim.x) {
      const int r0 = bitrev(x, logK);
      const int j = x <= off ? 0 : (x >= (K >> 2) - off ? 3 : -1);
      const int k = j == 0 ? x : x - (K >> 2);    // the block's sample index (when j >= 0)
      float4 hp = z, hm = z, unused;
      if (j >= 0) {
        hpm(k, hp, unused);                       // bp[k] = hp(k)
        if (!self) hpm(-k, unused, hm);           // bm[k] = hm(-k)
      }
      put4(bp, r0, j, hp);
      if (!self) put4(bm, r0, j, hm);
    }
    __syncthreads();
    st = fft_tail_start(logK, 2);
    fft_smem<true>(bp, self ? 1 : 2, tw, logK, 2, st);
  } else {
    for (int i = threadIdx.x; i < 2 * K; i += blockDim.x) sm[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    for (int gy = threadIdx.x; gy < Wd; gy += blockDim.x) {
      const int ky = full ? (gy <= K / 2 ? gy : gy - K) : gy - off;
      const int gym = gidx(-ky, off, full, K);
      const float4 a0 = Acc[2 * ((size_t)gy * Wd + gxp)], a1 = Acc[2 * ((size_t)gy * Wd + gxp) + 1];
      const float4 b0 = Acc[2 * ((size_t)gym * Wd + gxm)], b1 = Acc[2 * ((size_t)gym * Wd + gxm) + 1];
      const float P1r = a0.x + b0.x, P1i = a0.y - b0.y, Q1r = a0.z + b0.z, Q1i = a0.w - b0.w;
      const float P2r = a1.x + b1.x, P2i = a1.y - b1.y, Q2r = a1.z + b1.z, Q2i = a1.w - b1.w;
      const float4 hp = make_float4(P1r - Q1i, P1i + Q1r, P2r - Q2i, P2i + Q2r);
      bp[fsw(bitrev((ky + K) & (K - 1), logK))] = hp;
      if (!self) {
        const float4 hm = make_float4(P1r + Q1i, -P1i + Q1r, P2r + Q2i, -P2i + Q2r);
        bm[fsw(bitrev((-ky + K) & (K - 1), logK))] = hm;
      }
    }
    __syncthreads();
    st = fft_tail_start(logK, 0);
    fft_smem<true>(bp, self ? 1 : 2, tw, logK, 0, st);
  }
  for (int p = threadIdx.x; p < n; p += blockDim.x) {
    const int k = (p - n / 2 + K) & (K - 1);
    T2[(size_t)p * Wd + gxp] = fft_out<true>(bp, tw, logK, st, k);
    if (!self) T2[(size_t)p * Wd + gxm] = fft_out<true>(bm, tw, logK, st, k);
  }
}

__global__ void __launch_bounds__(256) k_adj_rows(const float4* __restrict__ T2, int n, int N,
                                                  const float* __restrict__ corr,
                                                  const float2* __restrict__ tw, int K, int logK, int Wd,
                                                  int off, int full, float* __restrict__ out) {
  extern __shared__ float4 sm[];
  pdl_wait();
  float4* buf = sm;
  const int p = blockIdx.x;
  int st;
  if (!full && 8 * off < K) {
    // Window [-R, R] with R < K/8: of the natural indices x + j K/4 (j = 0..3) at most
    // one holds a sample (j = 0: k = x <= R; j = 3: k = x - K/4 >= -R), so the first two
    // radix-2 stages reduce to the 4-point inverse DFT of one sample, v (i^{j t})_t,
    // written straight to the four slots 4B + t of its block (x = bitrev(4B)); blocks
    // without a sample get zeros, and fft_smem starts at stage 2.
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int x = threadIdx.x; x < (K >> 2); x += blockDim.x) {
      const int r0 = bitrev(x, logK);
      float4 v0 = z, v1 = z, v2 = z, v3 = z;
      if (x <= off) {
        v0 = v1 = v2 = v3 = T2[(size_t)p * Wd + x + off];
      } else if (x >= (K >> 2) - off) {
        const float4 v = T2[(size_t)p * Wd + x - (K >> 2) + off];
        v0 = v;
        v1 = make_float4(v.y, -v.x, v.w, -v.z);    // -i v
        v2 = make_float4(-v.x, -v.y, -v.z, -v.w);  // -v
        v3 = make_float4(-v.y, v.x, -v.w, v.z);    // +i v
      }
      buf[fsw(r0)] = v0;
      buf[fsw(r0 + 1)] = v1;
      buf[fsw(r0 + 2)] = v2;
      buf[fsw(r0 + 3)] = v3;
    }
    __syncthreads();
    st = fft_tail_start(logK, 2);
    fft_smem<true>(buf, 1, tw, logK, 2, st);
  } else {
    for (int i = threadIdx.x; i < K; i += blockDim.x) buf[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    for (int gx = threadIdx.x; gx < Wd; gx += blockDim.x) {
      const int k = full ? gx : gx - off;
      buf[fsw(bitrev((k + K) & (K - 1), logK))] = T2[(size_t)p * Wd + gx];
    }
    __syncthreads();
    st = fft_tail_start(logK, 0);
    fft_smem<true>(buf, 1, tw, logK, 0, st);
  }
  const float cy = 0.5f * corr[p];
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    const float4 v = fft_out<true>(buf, tw, logK, st, (q - n / 2 + K) & (K - 1));
    const float c = cy * corr[q];
    const size_t o = (size_t)p * n + q;
    out[o] = v.x * c;
    out[(size_t)N + o] = v.y * c;
    out[2 * (size_t)N + o] = v.z * c;
    out[3 * (size_t)N + o] = v.w * c;
  }
}

static size_t fft_smem_bytes(int K, int nbuf) { return (size_t)nbuf * K * sizeof(float4); }

static cudaError_t set_smem(const void* fn, size_t bytes) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int W>
static constexpr size_t grid_smem(int warps) { return (size_t)warps * GridWarp<W>::kFloats * sizeof(float); }

template <int W>
static cudaError_t configure_grid() {
  const cudaError_t e = set_smem((const void*)k_grid<W, false, true>, grid_smem<W>(kMergeWarps));
  return e == cudaSuccess ? set_smem((const void*)k_grid<W, true, true>, grid_smem<W>(kMergeWarps)) : e;
}

cudaError_t configure_nufft_kernels() {
  // Largest grid: n = 2048, K = 4096.
  const size_t sm1 = fft_smem_bytes(4096, 1), sm2 = fft_smem_bytes(4096, 2);
  cudaError_t e;
  if ((e = set_smem((const void*)k_fwd_rows<3>, sm1)) != cudaSuccess) return e;
  if ((e = set_smem((const void*)k_fwd_rows<5>, sm1)) != cudaSuccess) return e;
  if ((e = set_smem((const void*)k_fwd_cols, sm1)) != cudaSuccess) return e;
  if ((e = set_smem((const void*)k_adj_rows, sm1)) != cudaSuccess) return e;
  // Per-block FP64 accumulators of the degridding kernels (up to 2047 blocks).
  const void* degrids[] = {(const void*)k_degrid<5, false>, (const void*)k_degrid<7, false>, (const void*)k_degrid<9, false>,
                           (const void*)k_degrid<5, true>,  (const void*)k_degrid<7, true>,  (const void*)k_degrid<9, true>};
  const size_t degrid_smem[] = {degrid_smem_tiles<5>(), degrid_smem_tiles<7>(), degrid_smem_tiles<9>()};
  for (int i = 0; i < 6; ++i)
    if ((e = set_smem(degrids[i], degrid_smem[i % 3] + 2048 * sizeof(double))) != cudaSuccess) return e;
  if ((e = configure_grid<5>()) != cudaSuccess || (e = configure_grid<7>()) != cudaSuccess ||
      (e = configure_grid<9>()) != cudaSuccess)
    return e;
  return set_smem((const void*)k_adj_cols, sm2);
}

// Threads of a transform's CTA: one group of 16 per thread and pass for the rows (many CTAs), two
// threads per group for the columns (few CTAs, whose loads and outputs set the time).
cudaError_t nufft_forward_grid(Handle* h, const float* X, bool clear_acc) {
  const GridGeom& g = h->g;
  const size_t sm1 = fft_smem_bytes(g.K, 1);
  cudaError_t e = launch_after(h->early, g.K > 2048 ? k_fwd_rows<3> : k_fwd_rows<5>, h->n, 256, sm1, h->stream, X,
                               h->n, h->N, h->corr, h->tw, g.K, g.logK, h->T1, g.Wd,
                               g.off, g.full, h->Acc, clear_acc ? 2 * g.Wd * g.Wd : 0);
  if (e != cudaSuccess) return e;
  return launch_after(h->early, k_fwd_cols, g.Wd, 512, sm1, h->stream, h->T1, h->n, h->tw, g.K, g.logK, h->G, g.Wd, g.off, g.full);
}

template <int W>
static cudaError_t launch_degrid(Handle* h, int mode, float2* out, bool keep_cb, const int32_t* perm) {
  const GridGeom& g = h->g;
  const int nbins = h->nblocks <= kWarpBins ? kWarpBins * 8 : h->nblocks;   // 8 warps of 256 threads
  const size_t sm = degrid_smem_tiles<W>() + (size_t)nbins * sizeof(double);
  const BallStep ball{h->block_sum, h->block_done, h->block_norm_sq, mode == DEG_DUAL && !keep_cb ? h->cb : nullptr,
                      h->eps,       h->rho2,       h->cfg.literal_ball};
  return launch_after(h->early, mode == DEG_APPLY ? k_degrid<W, true> : k_degrid<W, false>, h->nitems, 256, sm, h->stream, h->items, h->rec, h->G, g.Wd, g.off, g.full, g.K,
                      g.beta, mode, h->R, h->Y, h->cb, (float)(1.0 / h->rho2), h->vblk, h->nblocks, ball, perm, out);
}

cudaError_t nufft_degrid(Handle* h, int mode, float2* out, bool keep_cb, const int32_t* perm) {
  if (h->M == 0) return cudaSuccess;
  switch (h->g.W) {
    case 5: return launch_degrid<5>(h, mode, out, keep_cb, perm);
    case 9: return launch_degrid<9>(h, mode, out, keep_cb, perm);
    default: return launch_degrid<7>(h, mode, out, keep_cb, perm);
  }
}

template <int W>
static cudaError_t launch_grid(Handle* h, const float2* in, int use_scale, const int32_t* perm) {
  const GridGeom& g = h->g;
  // Rows per warp. Few rows: 8, for more warps with fewer cells each. Many rows in dense cells:
  // 64, where that leaves two warps for every scheduler of the chip and a cell holds enough
  // rows that cutting its run at a warp's end costs more than parallelism gives. Else 32.
  // phi^dagger, us at 8 / 32 / 64 rows: 64^2 / 2,000 rows 27 / 29 / 31, 128^2 / 6,001 scattered
  // (1 per cell) 31 / 43 / 60, 64^2 / 25,153 33 / 27 / 29, 256^2 / 50,000 31 / 29 / 31, 2048^2 /
  // 700,001 (4 per cell) - / 215 / 222; 64^2 / 100,000 (529 per cell) - / 35 / 30, 1024^2 / 2,000,000
  // (34 per cell) - / 147 / 143.
  // A cell of the accumulator is the FP32 sum, one reduction after another, of all runs of W^2 cells, and its
  // rounding grows as the root of their number. Where a cell's rows make more than 16 runs (W = 9, which adds up
  // 81 cells where W = 7 adds 49: 4), CTAs of eight warps merge theirs before the reduction. Error of
  // phi^dagger, 32^2 / 200,001 rows (about 2,000 per cell), as separate runs / merged: W = 5 3.9e-7 / 1.7e-7, W = 7 5.7e-7 /
  // 2.2e-7, W = 9 9.7e-7 / 2.6e-7; us 22.5 / 18.4, 28.7 / 20.5, 38 / 25. With fewer runs the merge's barrier costs more
  // than it saves: 64^2 / 100,000 (529 per cell, 8 runs) grid stage 11.5 separate, 13.2 merged, 64^2 / 200,000 (17 runs) 18.9
  // and 15.3; a batch of 16 problems with merges from 8 runs on 8288 us for 8247.
  const int warps = 8 * std::max(1, h->num_sms), per_cell = h->M / std::max(1, h->ncells);
  const int rows = h->M <= 12 * warps ? 8 : (h->M >= 64 * warps && per_cell >= 16 ? 64 : 32);
  const bool merge = per_cell > (W == 9 ? 4 : 16) * rows;
  const int nw = merge ? kMergeWarps : kGridWarps;
  const int ctas = (int)(((int64_t)h->M + (int64_t)rows * nw - 1) / ((int64_t)rows * nw));
  auto kern = merge ? (perm ? k_grid<W, true, true> : k_grid<W, false, true>)
                    : (perm ? k_grid<W, true, false> : k_grid<W, false, false>);
  return launch_after(h->early, kern, ctas, 32 * nw, grid_smem<W>(nw), h->stream, h->M, rows, h->vblk, h->rec, in, perm, h->cb,
                      use_scale, g.Wd, g.off, g.full, g.K, g.beta, reinterpret_cast<float*>(h->Acc));
}

cudaError_t nufft_grid(Handle* h, const float2* in, int use_scale, bool cleared, const int32_t* perm) {
  const GridGeom& g = h->g;
  if (!cleared) {
    const cudaError_t e = cudaMemsetAsync(h->Acc, 0, (size_t)g.Wd * g.Wd * 2 * sizeof(float4), h->stream);
    if (e != cudaSuccess) return e;
  }
  if (h->M == 0) return cudaSuccess;
  switch (g.W) {
    case 5: return launch_grid<5>(h, in, use_scale, perm);
    case 9: return launch_grid<9>(h, in, use_scale, perm);
    default: return launch_grid<7>(h, in, use_scale, perm);
  }
}

cudaError_t nufft_adjoint_image(Handle* h, float* out) {
  const GridGeom& g = h->g;
  const size_t sm2 = fft_smem_bytes(g.K, 2), sm1 = fft_smem_bytes(g.K, 1);
  const int ncols = g.full ? (g.K / 2 + 1) : (g.R + 1);
  cudaError_t e = launch_after(h->early, k_adj_cols, ncols, 512, sm2, h->stream, h->Acc, h->n, h->tw, g.K, g.logK, h->T2, g.Wd, g.off,
                               g.full);
  if (e != cudaSuccess) return e;
  return launch_after(h->early, k_adj_rows, h->n, 256, sm1, h->stream, h->T2, h->n, h->N, h->corr, h->tw, g.K, g.logK, g.Wd, g.off,
                      g.full, out);
}

}  // namespace ps

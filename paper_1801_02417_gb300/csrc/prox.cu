// Per-pixel steps of Algorithm 1 and the reductions of the stopping rules.
//
// k_primal fuses, per pixel, Algorithm 1 steps 3-4 (primal S and Z with P_U or
// P_U' and P_V), the extrapolations 2 S^(k+1) - S^(k), 2 Z^(k+1) - Z^(k), steps
// 9-12 (epigraph duals C, D through P_E1 and P_E2, Eqs. proj_e1 and
// proj_e2_def) and the Dirac part of steps 5-6 (A_dirac = clamp(A + rho1 Xb/3,
// +-gamma W)). In PS_SOC mode the epigraph steps are replaced by the direct
// cone dual C = C~ - rho3 P_P(C~ / rho3) (Z and D are not touched). In the TV modes
// (Algorithm 3) the same sweep takes the data gradient -phi^dagger(Y - phi S) / 2 in place
// of phi^dagger B, Psi A = grad^T A from k_tv_adj, and skips the SARA Dirac part. It also writes per-CTA FP64 partials of ||S^(k+1) - S^(k)||^2 and
// ||S^(k)||^2 per map for the relative-change rule (Eq. stop_crit).
#include <cuda_runtime.h>

#include "internal.h"

namespace ps {

constexpr int kSweepThreads = 256;

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// P_E1 of Eq. proj_e1 on (c, d).
__device__ __forceinline__ void proj_e1(float c, float d, float& pc, float& pd) {
  if (c + d >= 0.f) {
    pc = c;
    pd = d;
  } else {
    pc = 0.5f * (c - d);
    pd = 0.5f * (d - c);
  }
}

// P_E2 of Eq. proj_e2_def on (r1, r2, r3, d).
__device__ __forceinline__ void proj_e2(float r1, float r2, float r3, float d, float& p1, float& p2, float& p3,
                                        float& pd) {
  const float nr = sqrtf(r1 * r1 + r2 * r2 + r3 * r3);
  if (nr < -d || (nr == 0.f && d <= 0.f)) {
    p1 = p2 = p3 = pd = 0.f;
  } else if (nr < d) {
    p1 = r1;
    p2 = r2;
    p3 = r3;
    pd = d;
  } else {
    const float a = 0.5f * (1.0f + d / nr);
    p1 = a * r1;
    p2 = a * r2;
    p3 = a * r3;
    pd = a * nr;
  }
}

// P = 1 or 2 consecutive floats of a plane as one load or store.
template <int P>
struct Pix {
  float v[P];
};
template <int P>
__device__ __forceinline__ Pix<P> ldp(const float* p) {
  Pix<P> r;
  if constexpr (P == 1) {
    r.v[0] = *p;
  } else {
    const float2 q = *reinterpret_cast<const float2*>(p);
    r.v[0] = q.x, r.v[1] = q.y;
  }
  return r;
}
template <int P>
__device__ __forceinline__ void stp(float* p, const Pix<P>& r) {
  if constexpr (P == 1) *p = r.v[0];
  else *reinterpret_cast<float2*>(p) = make_float2(r.v[0], r.v[1]);
}

// One thread = P consecutive pixels of every plane. grid.y indexes the problems
// of a batch's size class, whose arrays follow one another (S, C, Xb, PsiA, Adj: 4 N floats
// each; Z, D: 2 N; A, T: 4 cstride; partials: part_stride doubles); one problem: grid.y = 1.
// Every load of the thread is issued before the first value is used: a small image is one
// round trip to memory.
template <int P>
__global__ void __launch_bounds__(kSweepThreads) k_primal(
    int N, int mode, float tau, float rho1, float rho3, float* __restrict__ S, float* __restrict__ Z,
    float* __restrict__ C, float* __restrict__ D, const float* __restrict__ PsiA, const float* __restrict__ Adj,
    float* __restrict__ Xb, float* __restrict__ A, const float* __restrict__ T, size_t cstride,
    double* __restrict__ part, size_t part_stride) {
  __shared__ double sh[kSweepThreads / 32][8];
  if (blockIdx.y) {
    const size_t p = blockIdx.y, n4 = 4 * (size_t)N, n2 = 2 * (size_t)N;
    S += p * n4;
    C += p * n4;
    Xb += p * n4;
    PsiA += p * n4;
    Adj += p * n4;
    Z += p * n2;
    D += p * n2;
    A += p * 4 * cstride;
    T += p * 4 * cstride;
    part += p * part_stride;
  }
  float dss[4] = {0.f, 0.f, 0.f, 0.f}, ss[4] = {0.f, 0.f, 0.f, 0.f};
  const int i = P * (blockIdx.x * kSweepThreads + threadIdx.x);
  const float inv_r3 = 1.0f / rho3;
  const float r1_3 = rho1 * (1.0f / 3.0f);
  const bool tv = tv_mode(mode), con = constrained_mode(mode), sara = mode != PS_NNLS && !tv;
  const bool split = mode == PS_POLARIZED || mode == PS_TV || mode == PS_L1TV;   // epigraph split (Alg. 1 / Alg. 3)
  if (i < N) {
    Pix<P> g[4], q[4], c[4], so[4], t[4], a[4], z[2], d[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const size_t o = (size_t)k * N + i;
      g[k] = ldp<P>(Adj + o);
      so[k] = ldp<P>(S + o);
      if (mode != PS_NNLS) q[k] = ldp<P>(PsiA + o);
      if (con) c[k] = ldp<P>(C + o);
      if (sara) {
        t[k] = ldp<P>(T + (size_t)k * cstride + i);
        a[k] = ldp<P>(A + (size_t)k * cstride + i);
      }
    }
    if (split) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        z[k] = ldp<P>(Z + (size_t)k * N + i);
        d[k] = ldp<P>(D + (size_t)k * N + i);
      }
    }
    Pix<P> xb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const size_t o = (size_t)k * N + i;
      Pix<P> sn, an;
#pragma unroll
      for (int e = 0; e < P; ++e) {
        // TV modes (Algorithm 3 step 3): Adj holds phi^dagger(Y - phi(S)), so the data
        // gradient 1/2 phi^dagger(phi(S) - Y) is -Adj / 2.
        float gr = tv ? -0.5f * g[k].v[e] : g[k].v[e];
        if (mode != PS_NNLS) gr += q[k].v[e];
        if (con) gr += c[k].v[e];
        const float s0 = so[k].v[e];
        float s1 = s0 - tau * gr;                                  // step 3
        if (!con && k == 0) s1 = fmaxf(s1, 0.f);                   // P_U'
        const float x = 2.f * s1 - s0, ds = s1 - s0;
        sn.v[e] = s1;
        xb[k].v[e] = x;
        dss[k] += ds * ds;
        ss[k] += s0 * s0;
        if (sara) {                                                // Dirac part of steps 5-6
          const float th = t[k].v[e];
          an.v[e] = fminf(fmaxf(fmaf(r1_3, x, a[k].v[e]), -th), th);
        }
      }
      stp<P>(S + o, sn);
      stp<P>(Xb + o, xb[k]);
      if (sara) stp<P>(A + (size_t)k * cstride + i, an);
    }
    if (split) {
#pragma unroll
      for (int e = 0; e < P; ++e) {
        // Step 4: Z = P_V(Z - tau D).
        const float za = z[0].v[e], zb = z[1].v[e];
        float z1 = za - tau * d[0].v[e], z2 = zb - tau * d[1].v[e];
        if (z1 + z2 > 0.f) {
          const float h = 0.5f * (z1 - z2);
          z2 = 0.5f * (z2 - z1);
          z1 = h;
        }
        z[0].v[e] = z1;
        z[1].v[e] = z2;
        const float zb1 = 2.f * z1 - za, zb2 = 2.f * z2 - zb;
        // Steps 9-12.
        const float ct0 = c[0].v[e] + rho3 * xb[0].v[e], ct1 = c[1].v[e] + rho3 * xb[1].v[e];
        const float ct2 = c[2].v[e] + rho3 * xb[2].v[e], ct3 = c[3].v[e] + rho3 * xb[3].v[e];
        const float dt1 = d[0].v[e] + rho3 * zb1, dt2 = d[1].v[e] + rho3 * zb2;
        float pc, pd;
        proj_e1(ct0 * inv_r3, dt1 * inv_r3, pc, pd);
        c[0].v[e] = ct0 - rho3 * pc;
        d[0].v[e] = dt1 - rho3 * pd;
        float p1, p2, p3, pd2;
        proj_e2(ct1 * inv_r3, ct2 * inv_r3, ct3 * inv_r3, dt2 * inv_r3, p1, p2, p3, pd2);
        c[1].v[e] = ct1 - rho3 * p1;
        c[2].v[e] = ct2 - rho3 * p2;
        c[3].v[e] = ct3 - rho3 * p3;
        d[1].v[e] = dt2 - rho3 * pd2;
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        stp<P>(Z + (size_t)k * N + i, z[k]);
        stp<P>(D + (size_t)k * N + i, d[k]);
      }
    } else if (mode == PS_SOC) {
      // Direct cone dual: C = C~ - rho3 P_P(C~ / rho3), P_P = P_E2 with (r, d) = ((Q, U, V), I).
#pragma unroll
      for (int e = 0; e < P; ++e) {
        const float ct0 = c[0].v[e] + rho3 * xb[0].v[e], ct1 = c[1].v[e] + rho3 * xb[1].v[e];
        const float ct2 = c[2].v[e] + rho3 * xb[2].v[e], ct3 = c[3].v[e] + rho3 * xb[3].v[e];
        float p1, p2, p3, p0;
        proj_e2(ct1 * inv_r3, ct2 * inv_r3, ct3 * inv_r3, ct0 * inv_r3, p1, p2, p3, p0);
        c[0].v[e] = ct0 - rho3 * p0;
        c[1].v[e] = ct1 - rho3 * p1;
        c[2].v[e] = ct2 - rho3 * p2;
        c[3].v[e] = ct3 - rho3 * p3;
      }
    }
    if (con) {
#pragma unroll
      for (int k = 0; k < 4; ++k) stp<P>(C + (size_t)k * N + i, c[k]);
    }
  }
  // Partials for the relative-change statistic: FP32 within a warp (at most 64
  // terms), FP64 across warps and CTAs.
  double v[8];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    v[c] = (double)warp_sum(dss[c]);
    v[4 + c] = (double)warp_sum(ss[c]);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int c = 0; c < 8; ++c) sh[wid][c] = v[c];
  __syncthreads();
  if (threadIdx.x < 8) {
    double s = 0.0;
    for (int w = 0; w < kSweepThreads / 32; ++w) s += sh[w][threadIdx.x];
    part[(size_t)blockIdx.x * 8 + threadIdx.x] = s;
  }
}

// Pixels per thread: one while that is less than a wave of the chip's threads (a small image's
// sweep is a latency: 64^2 10.1 -> 7.3 us, 256^2 10.5 -> 8.7 against four pixels in four CTAs,
// resp. 64), two above, with all 28 loads of a pixel pair in flight (80 registers): 1024^2 39.7
// us with four pixels and loads as the steps need them, 37.9 with all of four pixels' loads in
// flight, 33 with two's (0.75 -> 0.91 of the copy bandwidth on 192 B per pixel); 2048^2 (cone
// dual) 122 -> 104 us.
static int sweep_pix(int N) { return N <= 65536 ? 1 : 2; }
int sweep_blocks(int N) { return (N + kSweepThreads * sweep_pix(N) - 1) / (kSweepThreads * sweep_pix(N)); }

cudaError_t primal_sweep(Handle* h) {
  const dim3 grid(sweep_blocks(h->N), h->problems);
  auto kern = sweep_pix(h->N) == 1 ? k_primal<1> : k_primal<2>;
  kern<<<grid, kSweepThreads, 0, h->stream>>>(h->N, h->mode, (float)h->tau, (float)h->rho1, (float)h->rho3, h->S, h->Z,
                                              h->C, h->D, h->PsiA, h->Adj, h->Xb, h->A, h->T, (size_t)kBases * h->N,
                                              h->red, (size_t)h->red_cap);
  return cudaGetLastError();
}

// Dirac part of Psi^dagger for the APPLY and REWEIGHT modes.
__global__ void k_dirac(int N, const float* __restrict__ X, float* __restrict__ coef, float* __restrict__ thr,
                        size_t cstride, int mode, float scale, float gamma, float delta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int c = blockIdx.y;
  if (i >= N) return;
  const float v = X[(size_t)c * N + i];
  const size_t o = (size_t)c * cstride + i;
  if (mode == SARA_APPLY) coef[o] = scale * v;
  else thr[o] = gamma * delta / (delta + fabsf(scale * v));
}

cudaError_t dirac_apply(Handle* h, const float* X, float* coef, float* thr, int mode, float scale, float gamma,
                        float delta) {
  dim3 grid((h->N + 255) / 256, h->nmaps);
  k_dirac<<<grid, 256, 0, h->stream>>>(h->N, X, coef, thr, (size_t)kBases * h->N, mode, scale, gamma, delta);
  return cudaGetLastError();
}

// Deterministic FP64 reductions in one launch: per-CTA partials, which the last CTA to end sums in
// a fixed order. `done` counts the CTAs that have written theirs (0 between launches).
template <typename T>
__device__ __forceinline__ T cta_sum(T v, T* sh) {   // valid in thread 0; sh: 32 values
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  T t = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  __syncthreads();
  return t;
}
__device__ __forceinline__ bool last_cta(int* done) {   // after the partials are written by thread 0
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(done, 1) == (int)gridDim.x - 1;
    if (last) *done = 0;
    __threadfence();
  }
  __syncthreads();
  return last;
}

// Sums of products for FP64 reductions: the FP64 pipe takes a conversion per operand and an FMA per
// product, at a sixty-fourth of the FP32 rate (the stopping statistics of 1024^2, of which the weighted norm
// is 38 M products: 941 us with it, 468 with this).
// Eight products at a time are therefore summed in FP32 without loss: the product with its rounding error
// (fma) and every sum with its own (Knuth's two-sum) go into a sum of three parts, high to low, of which
// only the last is rounded (2^-24 of 2^-47 of the group). The group then enters the FP64 sum, one
// rounding to 53 bits for eight products where the plain form has eight. The operations are the rounding
// intrinsics, which the compiler does not contract: a fused h + a * b or p - q would lose e or count it twice.
struct PairSum {
  float h = 0.f, l = 0.f, m = 0.f;
  // s + err = a + b exactly.
  __device__ __forceinline__ static float two_sum(float a, float b, float& err) {
    const float s = __fadd_rn(a, b), q = __fsub_rn(s, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, q)), __fsub_rn(b, q));
    return s;
  }
  __device__ __forceinline__ void add(float a, float b) {
    const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p);
    float e1, e2, e3;
    h = two_sum(h, p, e1);
    l = two_sum(l, e, e2);
    l = two_sum(l, e1, e3);
    m = __fadd_rn(m, __fadd_rn(e2, e3));
  }
  __device__ __forceinline__ void add(float4 a, float4 b) {
    add(a.x, b.x);
    add(a.y, b.y);
    add(a.z, b.z);
    add(a.w, b.w);
  }
  __device__ __forceinline__ double take() {
    const double r = (double)h + ((double)l + (double)m);
    h = l = m = 0.f;
    return r;
  }
};
// Whether a thread's sum is one in which FP32 products have neither overflowed nor lost anything
// below the smallest normal number that counts; outside (zero, tiny or huge data) it is formed again
// in FP64.
__device__ __forceinline__ bool pair_range(double s) { return fabs(s) >= 1e-20 && fabs(s) <= 1e30; }
// Sum over this thread's share of len products f(a[i]) b[i] (len a multiple of 4, 16-byte aligned).
template <typename F>
__device__ __forceinline__ double pair_sums(const float4* __restrict__ a, const float4* __restrict__ b, size_t len, F f) {
  const size_t n4 = len >> 2, step = (size_t)gridDim.x * blockDim.x;
  double s = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += 2 * step) {
    PairSum t;
    const bool two = i + step < n4;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 a0 = a[i], b0 = b[i], a1 = two ? a[i + step] : z, b1 = two ? b[i + step] : z;
    t.add(f(a0), b0);
    t.add(f(a1), b1);
    s += t.take();
  }
  if (pair_range(s)) return s;
  s = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += step) {
    const float4 x = f(a[i]), y = b[i];
    s += (double)x.x * y.x + (double)x.y * y.y + (double)x.z * y.z + (double)x.w * y.w;
  }
  return s;
}

__global__ void k_dot(const float4* __restrict__ a, const float4* __restrict__ b, size_t len, double* part, int* done,
                      double* out) {
  __shared__ double sh[32];
  double s = cta_sum(pair_sums(a, b, len, [](float4 v) { return v; }), sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
  if (!last_cta(done)) return;
  s = threadIdx.x < gridDim.x ? __ldcg(&part[threadIdx.x]) : 0.0;   // at most blockDim CTAs
  s = cta_sum(s, sh);
  if (threadIdx.x == 0) *out = s;
}

// Column sums of the per-CTA relative-change partials that k_primal writes (8 per CTA: the
// squared changes of the four maps, then their squared norms), in FP64 and a fixed order,
// written with the device error flags (as ints after the 8 sums) straight into `out`, which
// may be mapped host memory.
__global__ void k_relc_sums(const double* __restrict__ part, int nb, const int* __restrict__ flags,
                            double* __restrict__ out) {
  __shared__ double sh[8][8];   // [warp][column]
  const int c = threadIdx.x & 7;
  double s = 0.0;
#pragma unroll 8
  for (int b = threadIdx.x >> 3; b < nb; b += blockDim.x >> 3) s += part[8 * (size_t)b + c];
  s += __shfl_xor_sync(0xffffffffu, s, 8);    // lanes c, c + 8, c + 16, c + 24 hold column c
  s += __shfl_xor_sync(0xffffffffu, s, 16);
  if ((threadIdx.x & 31) < 8) sh[threadIdx.x >> 5][c] = s;
  __syncthreads();
  if (threadIdx.x < 8) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w][threadIdx.x];
    out[threadIdx.x] = t;
  } else if (threadIdx.x < 12) {
    reinterpret_cast<int*>(out + 8)[threadIdx.x - 8] = flags[threadIdx.x - 8];
  }
  __threadfence_system();
}

cudaError_t relc_sums(Handle* h, int nb, double* out) {
  k_relc_sums<<<1, 256, 0, h->stream>>>(h->red, nb, h->dev_flags, out);
  return cudaGetLastError();
}

// CTAs (and threads of each) of the one-launch reductions; their partials are the last
// 2 kRedBlocks doubles of `red`, the weighted norm's the kRedBlocks before them (it runs beside
// the others), their counters dev_flags[1] and [2].
static constexpr int kRedBlocks = 256;
static double* red_partials(Handle* h, int back) { return h->red + (size_t)h->red_cap - back * kRedBlocks; }

cudaError_t reduce_dot(Handle* h, const float* a, const float* b, size_t len, double* dev_out) {
  k_dot<<<kRedBlocks, kRedBlocks, 0, h->stream>>>(reinterpret_cast<const float4*>(a), reinterpret_cast<const float4*>(b),
                                                  len, red_partials(h, 2), h->dev_flags + 1, dev_out);
  return cudaGetLastError();
}

// Pixels with -I + ||(Q, U, V)|| above zeta and above zero, zeta = zeta_sigma rms / psf_peak from the sum
// of squares *rms_sum of the residual image (null: zeta = 0). The last CTA writes out[0] = that
// sum, out[1 .. 2] = the counts and out[4 .. 5] = the device flags (as ints); `out` may be mapped
// host memory.
__global__ void k_violations(int N, const float* __restrict__ S, const double* rms_sum, double zeta_sigma,
                             double psf_peak, double* part, int* flags, double* out) {
  __shared__ double sh[32];
  const double q = rms_sum ? *rms_sum : 0.0;
  const double zeta = psf_peak > 0.0 ? zeta_sigma * sqrt(q / (double)N) / psf_peak : 0.0;
  const float zhi = __double2float_ru(zeta), zlo = __double2float_rd(zeta);   // zeta >= 0
  int n0 = 0, n1 = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    // In FP32 where its error cannot change either comparison (a few roundings of 6e-8 each of the
    // norm and of I, taken as 1e-6 of both), else in FP64.
    const float i32 = S[i], q32 = S[(size_t)N + i], u32 = S[2 * (size_t)N + i], v32 = S[3 * (size_t)N + i];
    const float nr = sqrtf(fmaf(q32, q32, fmaf(u32, u32, v32 * v32))), p32 = nr - i32;
    const float off = 1e-6f * (nr + fabsf(i32)) + 1e-18f;
    if (p32 - off > zhi) {
      n0 += 1;
      n1 += 1;
    } else if (p32 + off < zlo && (p32 - off > 0.f || p32 + off < 0.f)) {
      n1 += p32 > 0.f;
    } else {
      const double I = i32, Q = q32, U = u32, V = v32;
      const double p = -I + sqrt(Q * Q + U * U + V * V);
      n0 += p > zeta;
      n1 += p > 0.0;
    }
  }
  double c0 = cta_sum((double)n0, sh), c1 = cta_sum((double)n1, sh);
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = c0;
    part[2 * blockIdx.x + 1] = c1;
  }
  if (!last_cta(flags + 1)) return;
  c0 = threadIdx.x < gridDim.x ? __ldcg(&part[2 * threadIdx.x]) : 0.0;
  c1 = threadIdx.x < gridDim.x ? __ldcg(&part[2 * threadIdx.x + 1]) : 0.0;
  c0 = cta_sum(c0, sh);
  c1 = cta_sum(c1, sh);
  if (threadIdx.x == 0) {
    out[0] = q;
    out[1] = c0;
    out[2] = c1;
    for (int k = 0; k < 4; ++k) reinterpret_cast<int*>(out + 4)[k] = k ? 0 : flags[k];
    __threadfence_system();
  }
}

cudaError_t violation_count(Handle* h, const float* S, const double* rms_sum, double zeta_sigma, double* out) {
  k_violations<<<kRedBlocks, kRedBlocks, 0, h->stream>>>(h->N, S, rms_sum, zeta_sigma, h->psf_peak, red_partials(h, 2),
                                                         h->dev_flags, out);
  return cudaGetLastError();
}

__global__ void k_wl1(const float4* __restrict__ c, const float4* __restrict__ t, size_t len, double* part, int* done,
                      double* out) {
  __shared__ double sh[32];
  double s = cta_sum(pair_sums(c, t, len, [](float4 v) { return make_float4(fabsf(v.x), fabsf(v.y), fabsf(v.z), fabsf(v.w)); }),
                     sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
  if (!last_cta(done)) return;
  s = threadIdx.x < gridDim.x ? __ldcg(&part[threadIdx.x]) : 0.0;
  s = cta_sum(s, sh);
  if (threadIdx.x == 0) {
    *out = s;
    __threadfence_system();
  }
}

cudaError_t weighted_l1(Handle* h, const float* coef, const float* thr, double* out) {
  k_wl1<<<kRedBlocks, kRedBlocks, 0, h->stream>>>(reinterpret_cast<const float4*>(coef), reinterpret_cast<const float4*>(thr),
                                                  (size_t)36 * h->N, red_partials(h, 3), h->dev_flags + 2, out);
  return cudaGetLastError();
}

__global__ void k_maxabs(const float* __restrict__ c, size_t len, float* part, int* done, double* out) {
  __shared__ float sh[32];
  auto cta_max = [&](float m) {   // valid in thread 0
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0)
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, sh[w]);
    __syncthreads();
    return m;
  };
  float m = 0.f;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (size_t)gridDim.x * blockDim.x)
    m = fmaxf(m, fabsf(c[i]));
  m = cta_max(m);
  if (threadIdx.x == 0) part[blockIdx.x] = m;
  if (!last_cta(done)) return;
  m = cta_max(threadIdx.x < gridDim.x ? __ldcg(&part[threadIdx.x]) : 0.f);
  if (threadIdx.x == 0) *out = (double)m;
}

cudaError_t max_abs(Handle* h, const float* c, size_t len, double* dev_out) {
  k_maxabs<<<kRedBlocks, kRedBlocks, 0, h->stream>>>(c, len, reinterpret_cast<float*>(red_partials(h, 2)),
                                                     h->dev_flags + 1, dev_out);
  return cudaGetLastError();
}

__global__ void k_scale_copy(const float* __restrict__ x, float* __restrict__ y, size_t len, double s) {
  const float sf = (float)s;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (size_t)gridDim.x * blockDim.x)
    y[i] = x[i] * sf;
}

cudaError_t scale_copy(Handle* h, const float* x, float* y, size_t len, double s) {
  k_scale_copy<<<1024, 256, 0, h->stream>>>(x, y, len, s);
  return cudaGetLastError();
}

__global__ void k_fill4(float4* p, size_t len4, float v) {
  const float4 q = make_float4(v, v, v, v);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < len4; i += (size_t)gridDim.x * blockDim.x)
    p[i] = q;
}

cudaError_t fill(Handle* h, float* p, size_t len, float v) {
  k_fill4<<<1024, 256, 0, h->stream>>>(reinterpret_cast<float4*>(p), len / 4, v);
  return cudaGetLastError();
}

// The Lanczos start vector: sample i is the (i + 1)-th state of a 64-bit linear congruential
// generator, its top 53 bits as a number in [-1/2, 1/2). A thread jumps to its first sample by
// powers of the generator's affine map (square and multiply) and steps on from there.
constexpr int kLcgRun = 16;
__global__ void k_lanczos_start(float* __restrict__ x, size_t len) {
  const size_t i0 = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * kLcgRun;
  if (i0 >= len) return;
  unsigned long long a = 6364136223846793005ull, c = 1442695040888963407ull, s = 0x9E3779B97F4A7C15ull;
  for (unsigned long long k = i0; k; k >>= 1) {
    if (k & 1) s = s * a + c;
    c = c * (a + 1);
    a = a * a;
  }
  for (size_t i = i0; i < i0 + kLcgRun && i < len; ++i) {
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    x[i] = (float)((double)(s >> 11) / 9007199254740992.0 - 0.5);
  }
}

// y = x / |.| with the squared norm from device memory (FP64).
__global__ void k_scale_by(const float* x, float* y, size_t len,
                           const double* __restrict__ norm_sq) {
  const float sf = (float)(1.0 / sqrt(*norm_sq));
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (size_t)gridDim.x * blockDim.x)
    y[i] = x[i] * sf;
}

cudaError_t lanczos_start(Handle* h, float* v, size_t len, double* scratch) {
  const size_t runs = (len + kLcgRun - 1) / kLcgRun;
  k_lanczos_start<<<(unsigned)((runs + 255) / 256), 256, 0, h->stream>>>(v, len);
  const cudaError_t e = reduce_dot(h, v, v, len, scratch);
  return e == cudaSuccess ? lanczos_scale(h, v, v, len, scratch) : e;
}

cudaError_t lanczos_scale(Handle* h, const float* w, float* u, size_t len, const double* norm_sq) {
  k_scale_by<<<1024, 256, 0, h->stream>>>(w, u, len, norm_sq);
  return cudaGetLastError();
}

// Lanczos three-term recurrence w = w - alpha v - beta u (FP32 vectors, FP64 coefficients from
// device memory: coef[0] = alpha, *last = beta^2 of the step before, null for the first), and
// coef[1] = |w|^2 of the result.
__global__ void k_lanczos_update(float4* __restrict__ w, const float4* __restrict__ v, const float4* __restrict__ u,
                                 size_t len, double* coef, const double* last, double* part, int* done) {
  __shared__ double sh[32];
  const float a = (float)coef[0], b = last ? (float)sqrt(*last) : 0.f;
  double s = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len >> 2; i += (size_t)gridDim.x * blockDim.x) {
    const float4 x = u[i], y = v[i], z = w[i];
    const float4 q = make_float4(fmaf(-b, x.x, fmaf(-a, y.x, z.x)), fmaf(-b, x.y, fmaf(-a, y.y, z.y)),
                                 fmaf(-b, x.z, fmaf(-a, y.z, z.z)), fmaf(-b, x.w, fmaf(-a, y.w, z.w)));
    w[i] = q;
    PairSum t;
    t.add(q, q);
    s += t.take();
  }
  if (!pair_range(s)) {
    s = 0.0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len >> 2; i += (size_t)gridDim.x * blockDim.x) {
      const float4 q = w[i];
      s += (double)q.x * q.x + (double)q.y * q.y + (double)q.z * q.z + (double)q.w * q.w;
    }
  }
  s = cta_sum(s, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
  if (!last_cta(done)) return;
  s = threadIdx.x < gridDim.x ? __ldcg(&part[threadIdx.x]) : 0.0;
  s = cta_sum(s, sh);
  if (threadIdx.x == 0) coef[1] = s;
}

cudaError_t lanczos_update(Handle* h, float* w, const float* v, const float* u, size_t len, double* coef,
                           const double* last) {
  k_lanczos_update<<<kRedBlocks, kRedBlocks, 0, h->stream>>>(
      reinterpret_cast<float4*>(w), reinterpret_cast<const float4*>(v), reinterpret_cast<const float4*>(u), len, coef, last,
      red_partials(h, 2), h->dev_flags + 1);
  return cudaGetLastError();
}

// Visibility order changes: sorted row m holds caller row perm[m].
__global__ void k_gather_vis(int M, const int32_t* __restrict__ perm, const float4* __restrict__ user,
                             float4* __restrict__ sorted) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M) return;
  const size_t u = (size_t)perm[m];
  sorted[2 * (size_t)m] = user[2 * u];
  sorted[2 * (size_t)m + 1] = user[2 * u + 1];
}

cudaError_t gather_vis(Handle* h, const float2* user, float2* sorted) {
  if (h->M == 0) return cudaSuccess;
  k_gather_vis<<<(h->M + 255) / 256, 256, 0, h->stream>>>(h->M, h->perm, reinterpret_cast<const float4*>(user),
                                                          reinterpret_cast<float4*>(sorted));
  return cudaGetLastError();
}

__global__ void k_read_dual(int M, const int32_t* __restrict__ perm, const uint16_t* __restrict__ vblk,
                            const float* __restrict__ cb, const float4* __restrict__ R, float4* __restrict__ user) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M) return;
  const float s = cb[vblk[m]];
  const size_t u = (size_t)perm[m];
  const float4 a = R[2 * (size_t)m], b = R[2 * (size_t)m + 1];
  user[2 * u] = make_float4(a.x * s, a.y * s, a.z * s, a.w * s);
  user[2 * u + 1] = make_float4(b.x * s, b.y * s, b.z * s, b.w * s);
}

cudaError_t read_dual(Handle* h, float2* user) {
  if (h->M == 0) return cudaSuccess;
  k_read_dual<<<(h->M + 255) / 256, 256, 0, h->stream>>>(h->M, h->perm, h->vblk, h->cb,
                                                         reinterpret_cast<const float4*>(h->R),
                                                         reinterpret_cast<float4*>(user));
  return cudaGetLastError();
}

}  // namespace ps

// Device building blocks: CTA-wide strided GEMM, reductions, contraction
// programs, and the truncation of the boundary MPS (dominant left singular
// subspace of a small dense matrix).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "contract.cuh"
#include "fast64.cuh"
#include "sturm64.cuh"

// Phase markers inside the truncation.  Empty in the library; the
// diagnostic build (-DPEPS_PHASE_TIMING, phase_timing.py) makes thread 0 of
// each CTA add the clock64 cycles since the previous marker to counter k
// (k = 0: the cycles since the last truncation ended, to counter 7).  Each
// marker is a barrier there, so that build is only for the breakdown.
#ifdef PEPS_PHASE_TIMING
static __device__ unsigned long long peps_phase_cyc[16];
__device__ __forceinline__ void peps_phase_mark(int k) {
  __shared__ long long peps_phase_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    const long long t = clock64();
    const long long d = t - peps_phase_last;
    if (d > 0 && d < (1ll << 34)) atomicAdd(&peps_phase_cyc[k == 0 ? 7 : k], (unsigned long long)d);
    peps_phase_last = t;
  }
  __syncthreads();
}
#define PEPS_PHASE(k) peps_phase_mark(k)
#else
#define PEPS_PHASE(k)
#endif

namespace peps {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxT2Shared = 256;   // reals of TruncWork::wv

template <typename R> struct Eps;
template <> struct Eps<double> {
  static constexpr double eps = 2.220446049250313e-16;
  static constexpr double tiny = 2.2250738585072014e-308;
  static constexpr int bits = 53;
};
template <> struct Eps<float> {
  static constexpr float eps = 1.1920929e-07f;
  static constexpr float tiny = 1.17549435e-38f;
  static constexpr int bits = 24;
};

__device__ __forceinline__ double dsqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float dsqrt(float x) { return sqrtf(x); }

// One step of a compensated dot product in FP32 (Ogita, Rump and Oishi,
// "Accurate sum and dot product", SIAM J. Sci. Comput. 26 (2005), Dot2):
// the product's rounding error comes exactly from an FMA (TwoProduct), the
// sum's from Knuth's TwoSum, and both go into c.  s + c then carries the dot
// product as if accumulated in twice the working precision.  The explicit
// _rn intrinsics keep the compiler from contracting or reassociating them.
__device__ __forceinline__ void dot2_step(float a, float b, float& s, float& c) {
  const float p = __fmul_rn(a, b);
  const float pe = __fmaf_rn(a, b, -p);
  const float t = __fadd_rn(s, p);
  const float z = __fsub_rn(t, s);
  const float se = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
  s = t;
  c = __fadd_rn(c, __fadd_rn(pe, se));
}

// Two of them at once in packed FP32x2 instructions: nine for two terms.  A
// difference is the product with -1 fused into the sum, which rounds once.
__device__ __forceinline__ void dot2_step2(float2 a, float2 b, float2& s, float2& c) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 p = __fmul2_rn(a, b);
  const float2 pe = __ffma2_rn(a, b, __fmul2_rn(p, m1));
  const float2 t = __fadd2_rn(s, p);
  const float2 z = __ffma2_rn(s, m1, t);
  const float2 se = __fadd2_rn(__ffma2_rn(__ffma2_rn(z, m1, t), m1, s), __ffma2_rn(z, m1, p));
  s = t;
  c = __fadd2_rn(c, __fadd2_rn(pe, se));
}

template <typename R>
__device__ __forceinline__ R warp_sum(R v, int width = 32) {
  for (int o = width / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, width);
  return v;
}
template <typename R>
__device__ __forceinline__ R warp_max(R v) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Block-wide sum; `red` is shared scratch of >= kWarps elements.  All threads
// get the result.  Contains two barriers.
template <typename R>
__device__ R block_sum(R v, R* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) red[w] = v;
  __syncthreads();
  R s = 0;
  for (int i = 0; i < kWarps; ++i) s += red[i];
  __syncthreads();
  return s;
}

// Block-wide maximum; same contract as block_sum.
template <typename R>
__device__ R block_max(R v, R* red) {
  v = warp_max(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) red[w] = v;
  __syncthreads();
  R s = red[0];
  for (int i = 1; i < kWarps; ++i) s = fmax(s, red[i]);
  __syncthreads();
  return s;
}

// Power-of-two renormalisation of the transfer vectors of the sandwiches.
// A sandwich value between unit-norm environments can fall far below the
// FP32 range (it is psi divided by the norms of all other rows), so every
// stored transfer is scaled by an exact power of two and its exponent is
// carried beside it; ratios and Delta add the exponents back in FP64.
// pow2_exponent(m) = floor(log2 m) read from the bits of m, clamped so that
// 2^-e is a normal number; 0 for m = 0 or m not finite.
__device__ __forceinline__ int pow2_exponent(float m) {
  const int ef = (int)((__float_as_uint(m) >> 23) & 0xffu);
  if (!(m > 0.f) || ef == 0xff) return 0;
  const int e = ef - 127;
  return e < -126 ? -126 : (e > 126 ? 126 : e);
}
__device__ __forceinline__ int pow2_exponent(double m) {
  const int ef = (int)((__double_as_longlong(m) >> 52) & 0x7ffll);
  if (!(m > 0.0) || ef == 0x7ff) return 0;
  const int e = ef - 1023;
  return e < -1022 ? -1022 : (e > 1022 ? 1022 : e);
}
// 2^e for e in the clamped range of pow2_exponent
template <typename R>
__device__ __forceinline__ R pow2(int e);
template <>
__device__ __forceinline__ float pow2<float>(int e) { return __uint_as_float((unsigned)(e + 127) << 23); }
template <>
__device__ __forceinline__ double pow2<double>(int e) {
  return __longlong_as_double((long long)(e + 1023) << 52);
}

// Scales x[0..n) in place by 2^-e, e = pow2_exponent(max |x|), and returns e.
// x must be complete (written before a barrier); ends with a barrier.
template <typename R>
__device__ int normalize_pow2(R* x, int n, R* red) {
  R m = R(0);
  for (int i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, fabs(x[i]));
  m = block_max(m, red);
  const int e = pow2_exponent(m);
  if (e != 0) {
    const R sc = pow2<R>(-e);
    for (int i = threadIdx.x; i < n; i += blockDim.x) x[i] *= sc;
  }
  __syncthreads();
  return e;
}

// ------------------------------------------------------------- CTA GEMM
// Shared-memory tiled GEMM over the index maps of a descriptor (see
// contract.cuh).  Per output tile (TM x TN) the K range is walked in chunks
// of 16: the A and B chunks are gathered from global memory through the
// offset tables into shared memory, then every thread accumulates an
// MT x NT micro-tile in registers.  The CTA tile shape follows N (the
// contraction steps have N in {16, 32, 64, 128, 256+}).  Shared memory:
// kGemmSmemReals reals + kGemmSmemInts ints supplied by the caller.
// A and B are often written earlier by the same kernel (carries, blocks,
// singular vectors), so they are not declared __restrict__: that would let
// the compiler read them through the non-coherent read-only path, which is
// only valid for data that no thread writes while the kernel runs.  The same
// holds for the transfer inputs of the fused steps.
constexpr int kGemmTK = 16;
constexpr int kMaxK = 1024;
constexpr int kGemmSmemReals = kGemmTK * (512 + 16);
constexpr int kGemmSmemInts = 2 * kMaxK + 2 * 512 + 2 * 256;

template <typename R, int TM, int TN, int MT, int NT>
__device__ __noinline__ void gemm_tiles(const GemmDesc& g, const R* A, const R* B,
                                        R* __restrict__ C, bool accumulate, R* sm, int* ism) {
  constexpr int TK = kGemmTK;
  constexpr int GX = TN / NT, GY = TM / MT;
  static_assert(GX * GY == kThreads, "thread grid must cover the CTA");
  R* As = sm;                  // [TK][TM]
  R* Bs = sm + TK * TM;        // [TK][TN]
  int* ktA = ism;              // [K]
  int* ktB = ism + kMaxK;      // [K]
  int* rA = ism + 2 * kMaxK;   // [TM]
  int* rC = rA + TM;           // [TM]
  int* cB = rC + TM;           // [TN]
  int* cC = cB + TN;           // [TN]
  const int tid = threadIdx.x;
  const int tx = tid % GX, ty = tid / GX;
  __syncthreads();
  for (int k = tid; k < g.K; k += blockDim.x) {
    const int k1 = k / g.ak.n2, k2 = k - k1 * g.ak.n2;
    ktA[k] = k1 * g.ak.s1 + k2 * g.ak.s2;
    ktB[k] = k1 * g.bk.s1 + k2 * g.bk.s2;
  }
  const int tiles_m = (g.M + TM - 1) / TM, tiles_n = (g.N + TN - 1) / TN;
  for (int bt = 0; bt < g.nb; ++bt) {
    const R* Ab = A + (size_t)bt * g.sa;
    const R* Bb = B + (size_t)bt * g.sb;
    R* Cb = C + (size_t)bt * g.sc;
    for (int tmi = 0; tmi < tiles_m; ++tmi)
      for (int tni = 0; tni < tiles_n; ++tni) {
        const int i0 = tmi * TM, j0 = tni * TN;
        __syncthreads();
        for (int e = tid; e < TM; e += blockDim.x) {
          const int i = min(i0 + e, g.M - 1);
          rA[e] = ixoff(g.am, i);
          rC[e] = ixoff(g.cm, i);
        }
        for (int e = tid; e < TN; e += blockDim.x) {
          const int j = min(j0 + e, g.N - 1);
          cB[e] = ixoff(g.bn, j);
          cC[e] = ixoff(g.cn, j);
        }
        R acc[MT][NT];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int n = 0; n < NT; ++n) acc[m][n] = R(0);
        for (int k0 = 0; k0 < g.K; k0 += TK) {
          __syncthreads();
          for (int e = tid; e < TM * TK; e += kThreads) {
            const int i = e % TM, kk = e / TM, k = k0 + kk;
            As[kk * TM + i] = k < g.K ? Ab[rA[i] + ktA[k]] : R(0);
          }
          for (int e = tid; e < TN * TK; e += kThreads) {
            const int j = e % TN, kk = e / TN, k = k0 + kk;
            Bs[kk * TN + j] = k < g.K ? Bb[ktB[k] + cB[j]] : R(0);
          }
          __syncthreads();
#pragma unroll
          for (int kk = 0; kk < TK; ++kk) {
            R a[MT], b[NT];
#pragma unroll
            for (int m = 0; m < MT; ++m) a[m] = As[kk * TM + ty * MT + m];
#pragma unroll
            for (int n = 0; n < NT; ++n) b[n] = Bs[kk * TN + tx * NT + n];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
              for (int n = 0; n < NT; ++n) acc[m][n] = fma(a[m], b[n], acc[m][n]);
          }
        }
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          const int i = ty * MT + m;
          if (i0 + i >= g.M) break;
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            const int j = tx * NT + n;
            if (j0 + j >= g.N) break;
            R* p = Cb + rC[i] + cC[j];
            *p = accumulate ? *p + acc[m][n] : acc[m][n];
          }
        }
      }
  }
  __syncthreads();
}

// C (+)= A B for a descriptor; the whole CTA takes part and the call ends
// with a barrier.  `sm`/`ism` point to the GEMM's shared-memory scratch.
template <typename R>
__device__ void cta_gemm(const GemmDesc& g, const R* A, const R* B, R* __restrict__ C,
                         bool accumulate, R* sm, int* ism) {
  if (g.N >= 256 && g.M <= 32) gemm_tiles<R, 16, 256, 4, 4>(g, A, B, C, accumulate, sm, ism);
  else if (g.N >= 128) gemm_tiles<R, 64, 128, 4, 8>(g, A, B, C, accumulate, sm, ism);
  else if (g.N >= 64 && g.M >= 128) gemm_tiles<R, 128, 64, 8, 4>(g, A, B, C, accumulate, sm, ism);
  else if (g.N >= 48) gemm_tiles<R, 64, 64, 4, 4>(g, A, B, C, accumulate, sm, ism);
  else if (g.N >= 24) gemm_tiles<R, 256, 32, 8, 4>(g, A, B, C, accumulate, sm, ism);
  else gemm_tiles<R, 512, 16, 8, 4>(g, A, B, C, accumulate, sm, ism);
}

// C = A B for a descriptor with K <= KM, the whole reduction staged at once:
// per tile of TM rows every load is issued before the first store to shared
// memory, so one load latency is exposed per tile rather than one per 16-wide
// K chunk, and a tile costs two barriers.  FP32 tiles are multiplied with
// packed FP32x2 multiply-adds.  Each output is the same left-to-right chain
// of fused multiply-adds over k as in gemm_tiles, so the results are
// identical.  `sm` holds K * (TM + TN) reals; `ism` the offset tables.
template <typename R, int TM, int TN, int MT, int NT, int KM>
__device__ __noinline__ void gemm_wk(const GemmDesc& g, const R* A, const R* B, R* __restrict__ C, R* sm,
                                     int* ism) {
  constexpr int GX = TN / NT, GY = TM / MT;
  static_assert(GX * GY == kThreads, "thread grid must cover the CTA");
  static_assert(MT % 4 == 0 && NT % 4 == 0, "tiles are read as 16-byte groups");
  constexpr int LA = TM * KM / kThreads, LB = TN * KM / kThreads;
  const int K = g.K;
  R* As = sm;            // [K][TM]
  R* Bs = sm + K * TM;   // [K][TN]
  int* ktA = ism;
  int* ktB = ism + KM;
  int* rA = ism + 2 * KM;
  int* rC = rA + TM;
  int* cB = rC + TM;
  int* cC = cB + TN;
  const int tid = threadIdx.x;
  const int tx = tid % GX, ty = tid / GX;
  __syncthreads();
  for (int k = tid; k < K; k += kThreads) {
    const int k1 = k / g.ak.n2, k2 = k - k1 * g.ak.n2;
    ktA[k] = k1 * g.ak.s1 + k2 * g.ak.s2;
    ktB[k] = k1 * g.bk.s1 + k2 * g.bk.s2;
  }
  const int tiles_m = (g.M + TM - 1) / TM, tiles_n = (g.N + TN - 1) / TN;
  for (int bt = 0; bt < g.nb; ++bt) {
    const R* Ab = A + (size_t)bt * g.sa;
    const R* Bb = B + (size_t)bt * g.sb;
    R* Cb = C + (size_t)bt * g.sc;
    for (int tni = 0; tni < tiles_n; ++tni)
      for (int tmi = 0; tmi < tiles_m; ++tmi) {
        const int i0 = tmi * TM, j0 = tni * TN;
        __syncthreads();
        for (int e = tid; e < TM; e += kThreads) {
          const int i = min(i0 + e, g.M - 1);
          rA[e] = ixoff(g.am, i);
          rC[e] = ixoff(g.cm, i);
        }
        for (int e = tid; e < TN; e += kThreads) {
          const int j = min(j0 + e, g.N - 1);
          cB[e] = ixoff(g.bn, j);
          cC[e] = ixoff(g.cn, j);
        }
        __syncthreads();
        R va[LA], vb[LB];
#pragma unroll
        for (int q = 0; q < LA; ++q) {
          const int e = tid + q * kThreads, kk = e / TM, i = e % TM;
          va[q] = kk < K ? Ab[rA[i] + ktA[kk]] : R(0);
        }
#pragma unroll
        for (int q = 0; q < LB; ++q) {
          const int e = tid + q * kThreads, kk = e / TN, j = e % TN;
          vb[q] = kk < K ? Bb[ktB[kk] + cB[j]] : R(0);
        }
#pragma unroll
        for (int q = 0; q < LA; ++q) {
          const int e = tid + q * kThreads;
          if (e / TM < K) As[e] = va[q];
        }
#pragma unroll
        for (int q = 0; q < LB; ++q) {
          const int e = tid + q * kThreads;
          if (e / TN < K) Bs[e] = vb[q];
        }
        __syncthreads();
        R acc[MT][NT];
        if constexpr (sizeof(R) == 4) {
          float2 acc2[MT][NT / 2];
#pragma unroll
          for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < NT / 2; ++n) acc2[m][n] = make_float2(0.f, 0.f);
#pragma unroll 4
          for (int kk = 0; kk < K; ++kk) {
            float a[MT], b[NT];
#pragma unroll
            for (int m = 0; m < MT; m += 4) {
              const float4 t = *reinterpret_cast<const float4*>(As + kk * TM + ty * MT + m);
              a[m] = t.x; a[m + 1] = t.y; a[m + 2] = t.z; a[m + 3] = t.w;
            }
#pragma unroll
            for (int n = 0; n < NT; n += 4) {
              const float4 t = *reinterpret_cast<const float4*>(Bs + kk * TN + tx * NT + n);
              b[n] = t.x; b[n + 1] = t.y; b[n + 2] = t.z; b[n + 3] = t.w;
            }
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
              for (int n = 0; n < NT / 2; ++n)
                acc2[m][n] = __ffma2_rn(make_float2(a[m], a[m]), make_float2(b[2 * n], b[2 * n + 1]), acc2[m][n]);
          }
#pragma unroll
          for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < NT / 2; ++n) {
              acc[m][2 * n] = acc2[m][n].x;
              acc[m][2 * n + 1] = acc2[m][n].y;
            }
        } else {
#pragma unroll
          for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < NT; ++n) acc[m][n] = R(0);
          for (int kk = 0; kk < K; ++kk) {
            R a[MT], b[NT];
#pragma unroll
            for (int m = 0; m < MT; ++m) a[m] = As[kk * TM + ty * MT + m];
#pragma unroll
            for (int n = 0; n < NT; ++n) b[n] = Bs[kk * TN + tx * NT + n];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
              for (int n = 0; n < NT; ++n) acc[m][n] = fma(a[m], b[n], acc[m][n]);
          }
        }
        int cc[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) cc[n] = cC[tx * NT + n];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          const int i = ty * MT + m;
          if (i0 + i >= g.M) break;
          const int rc = rC[i];
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            if (j0 + tx * NT + n >= g.N) break;
            Cb[rc + cc[n]] = acc[m][n];
          }
        }
      }
  }
  __syncthreads();
}

// Reals of shared scratch gemm_wk needs for a descriptor, or 0 when the
// descriptor is outside its shapes (cta_gemm takes those).
PEPS_HD int zip_gemm_reals(const GemmDesc& g) {
  if (g.N > 64 && g.N <= 128 && g.K <= 16) return g.K * (64 + 128);
  if (g.N <= 64 && g.K <= 64) return g.K * (128 + 64);
  return 0;
}

// C = A B in FP64 with both operands whole in shared memory (k-major) and the
// 4 x 4 output tiles dealt to the threads one after the other: what bounds it
// is the number of FP64 instructions a warp issues, and fixed CTA tiles of
// 128 x 64 issued three times the needed ones at 144 x 36 or 72 x 72 outputs
// (10x10 D = 6).  Each output is the same chain over k.
static __device__ __noinline__ void gemm_dealt(const GemmDesc& g, const double* A, const double* B,
                                               double* __restrict__ C, double* sm, int* ism) {
  const int M = g.M, N = g.N, K = g.K, tid = threadIdx.x;
  double* As = sm;           // [K][M]
  double* Bs = sm + K * M;   // [K][N]
  int* rA = ism;
  int* rC = rA + M;
  int* cB = rC + M;
  int* cC = cB + N;
  int* ktA = cC + N;
  int* ktB = ktA + K;
  __syncthreads();
  for (int e = tid; e < M; e += kThreads) {
    rA[e] = ixoff(g.am, e);
    rC[e] = ixoff(g.cm, e);
  }
  for (int e = tid; e < N; e += kThreads) {
    cB[e] = ixoff(g.bn, e);
    cC[e] = ixoff(g.cn, e);
  }
  for (int k = tid; k < K; k += kThreads) {
    ktA[k] = ixoff(g.ak, k);
    ktB[k] = ixoff(g.bk, k);
  }
  __syncthreads();
#pragma unroll 4
  for (int e = tid; e < K * M; e += kThreads) As[e] = A[rA[e % M] + ktA[e / M]];
#pragma unroll 4
  for (int e = tid; e < K * N; e += kThreads) Bs[e] = B[ktB[e / N] + cB[e % N]];
  __syncthreads();
  const int tn = (N + 3) / 4, nt = ((M + 3) / 4) * tn;
  for (int t = tid; t < nt; t += kThreads) {
    const int i0 = (t / tn) * 4, j0 = (t % tn) * 4;
    double acc[4][4];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) acc[x][y] = 0.0;
    int ia[4], jb[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      ia[q] = min(i0 + q, M - 1);
      jb[q] = min(j0 + q, N - 1);
    }
#pragma unroll 2
    for (int k = 0; k < K; ++k) {
      double a[4], b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a[q] = As[k * M + ia[q]];
        b[q] = Bs[k * N + jb[q]];
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = fma(a[x], b[y], acc[x][y]);
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y)
        if (i0 + x < M && j0 + y < N) C[rC[i0 + x] + cC[j0 + y]] = acc[x][y];
  }
  __syncthreads();
}

// C = A B for the zip-up contractions: gemm_dealt in FP64 and gemm_wk in FP32
// when the descriptor fits them and `sm_reals` reals of shared scratch, else
// cta_gemm.  Same results either way.
template <typename R>
__device__ __noinline__ void zip_gemm(const GemmDesc& g, const R* A, const R* B, R* __restrict__ C, R* sm, int* ism,
                         int sm_reals) {
  if constexpr (sizeof(R) == 8) {
    if (g.nb == 1 && g.K * (g.M + g.N) <= sm_reals && 2 * (g.M + g.N + g.K) <= kGemmSmemInts) {
      gemm_dealt(g, A, B, C, sm, ism);
      return;
    }
  }
  const int need = zip_gemm_reals(g);
  if (need > 0 && need <= sm_reals) {
    if (g.N > 64) gemm_wk<R, 64, 128, 4, 8, 16>(g, A, B, C, sm, ism);
    else gemm_wk<R, 128, 64, 8, 4, 64>(g, A, B, C, sm, ism);
  } else {
    cta_gemm<R>(g, A, B, C, false, sm, ism);
  }
}

// ------------------------------------------------- contraction programs
enum OpId { OP_COL1_LEFT = 0, OP_COL1_RIGHT = 1, OP_SITE_ENV = 2, OP_COL2_LEFT = 3, OP_COL2_RIGHT = 4, OP_FIT_SITE = 5 };
enum BufId { IN0 = 0, IN1, IN2, IN3, IN4, TMP0, TMP1, OUT };
struct Step {
  int s, a, b, c;
};

PEPS_HD int op_nsteps(int op) { return (op == OP_COL2_LEFT || op == OP_COL2_RIGHT) ? 4 : 3; }

// Which buffers each step reads and writes.  Inputs per op:
//   COL1_LEFT : IN0 = F_{c-1}, IN1 = Mu, IN2 = T, IN3 = Md        -> F_c
//   COL1_RIGHT: IN0 = G_{c+1}, IN1 = Mu, IN2 = T, IN3 = Md        -> G_c
//   SITE_ENV  : IN0 = F_{c-1}, IN1 = Mu, IN2 = Md, IN3 = G_{c+1}  -> B_c
//   COL2_LEFT : IN0 = E_{c-1}, IN1 = Mu, IN2 = T1, IN3 = T2, IN4 = Md -> E_c
//   COL2_RIGHT: IN0 = H_{c+1}, IN1 = Mu, IN2 = T1, IN3 = T2, IN4 = Md -> H_c
//   FIT_SITE  : IN0 = F_{c-1}, IN1 = Mu, IN2 = T, IN3 = G_{c+1}   -> P_c
PEPS_HD Step op_step_bufs(int op, int s) {
  switch (op) {
    case OP_FIT_SITE:
    case OP_COL1_LEFT:
      return s == 0 ? Step{0, IN0, IN1, TMP0} : s == 1 ? Step{1, TMP0, IN2, TMP1} : Step{2, TMP1, IN3, OUT};
    case OP_COL1_RIGHT:
      return s == 0 ? Step{0, IN1, IN0, TMP0} : s == 1 ? Step{1, TMP0, IN2, TMP1} : Step{2, TMP1, IN3, OUT};
    case OP_SITE_ENV:
      return s == 0 ? Step{0, IN2, IN3, TMP0} : s == 1 ? Step{1, IN1, TMP0, TMP1} : Step{2, IN0, TMP1, OUT};
    case OP_COL2_LEFT:
      return s == 0 ? Step{0, IN0, IN1, TMP0}
           : s == 1 ? Step{1, TMP0, IN2, TMP1}
           : s == 2 ? Step{2, TMP1, IN3, TMP0}
                    : Step{3, TMP0, IN4, OUT};
    default:
      return s == 0 ? Step{0, IN1, IN0, TMP0}
           : s == 1 ? Step{1, TMP0, IN2, TMP1}
           : s == 2 ? Step{2, TMP1, IN3, TMP0}
                    : Step{3, TMP0, IN4, OUT};
  }
}

PEPS_HD GemmDesc op_desc(int op, int s, int D, int Dc) {
  switch (op) {
    case OP_COL1_LEFT: return col1_left_step(s, D, Dc);
    case OP_COL1_RIGHT: return col1_right_step(s, D, Dc);
    case OP_SITE_ENV: return site_env_step(s, D, Dc);
    case OP_FIT_SITE: return fit_site_step(s, D, Dc);
    case OP_COL2_LEFT: return col2_left_step(s, D, Dc);
    default: return col2_right_step(s, D, Dc);
  }
}

// Runs one contraction program with the whole CTA; ends with a barrier.
template <typename R>
__device__ void run_op(int op, int D, int Dc, const R* in0, const R* in1, const R* in2, const R* in3,
                       const R* in4, R* out, R* t0, R* t1, R* sm, int* ism) {
  const int ns = op_nsteps(op);
  for (int s = 0; s < ns; ++s) {
    const Step st = op_step_bufs(op, s);
    const GemmDesc g = op_desc(op, st.s, D, Dc);
    const R* bufs[8] = {in0, in1, in2, in3, in4, t0, t1, out};
    cta_gemm<R>(g, bufs[st.a], bufs[st.b], const_cast<R*>(bufs[st.c]), false, sm, ism);
  }
}

// ------------------------------------------------------------ truncation
// Dominant-K left singular subspace of a dense m x n matrix X (row-major),
// used for the boundary-MPS cut-off (Fig. 1d, Dc).  Route: Householder
// bidiagonalisation (Golub & Kahan 1965), the K largest singular values by
// Sturm-count bisection on the Golub-Kahan tridiagonal form
// [[0, B], [B^T, 0]] (perfect-shuffle ordering), singular vectors by inverse
// iteration on that form, classical Gram-Schmidt with re-orthogonalisation,
// and back-transformation by the stored reflectors.  Only the subspace
// matters downstream (the kept projector is unique when sigma_K > sigma_K+1),
// so any orthonormal basis of it is a valid result.
template <typename R>
struct TruncWork {
  R* Wm;      // P x ldw
  int ldw;
  R* Wg;      // P x ldw in global memory: the reflectors of the register-tiled path
  R* tau;     // 4 * Qmax: tau left, tau right, scale left, scale right
  R* t;       // 2 * Qmax off-diagonal of the Golub-Kahan form
  R* t2;      // squares of t
  R* lam;     // Kmax
  R* lu;      // Kmax x 6 x 2Qmax: inverse-iteration workspace when it is not in shared memory
  R* Ub;      // Qmax x Kmax (unused when Ubs is set)
  R* Uk;      // Pmax x Kmax compact copy of the result in global memory
  R* Ubs;     // Qmax x Kmax in shared memory (after the truncation matrix)
  R* Uks;     // Pmax x Kmax in shared memory
  R* red;     // >= 64 (shared)
  R* wv;      // >= 256 (shared): reflector products
  R* gsm;     // GEMM shared scratch (may alias Wm: used only after the reflectors are dead)
  int* gism;
  int Qmax;
  int Kmax;        // Ubs and Uks hold Qmax x Kmax
  int gsm_reals;   // size of the shared region
  int wm_shared;   // Wm is in shared memory
  // Whether blocks of the register-tiled path with at most 16 columns apply
  // their reflectors one at a time: models whose shared region is at most 200 KB.
  // Above (D = 10, Dc = 20) such blocks are the few next to an edge, and take
  // the compact WY form as the others do; the two differ in the last FP32 bits,
  // 6e-9 of an energy.
  int one_by_one;
};

// Element counts of the truncation workspace for P, Q <= pq and K <= kmax.
PEPS_HD size_t trunc_ws_elems(int pq, int kmax, bool with_wm) {
  size_t e = 0;
  if (with_wm) e += (size_t)pq * (pq + 1);
  e += (size_t)pq * (pq + 1);             // Wg
  e += 4 * (size_t)pq + 2 * (size_t)pq * 2;   // tau + scale factors (4 pq), t, t2
  e += kmax;                              // lam
  e += (size_t)kmax * 6 * 2 * pq;         // lu
  e += (size_t)pq * kmax * 2;             // Ub, Uk
  return e + 64;
}

// Householder vector for x = (alpha, rest): returns tau, scale for rest, beta.
__device__ __forceinline__ void householder(float alpha, float ss, float& tau, float& scale, float& beta) {
  if (ss <= 0.f) {
    tau = 0.f;
    scale = 0.f;
    beta = alpha;
  } else {
    const float nrm = dsqrt(alpha * alpha + ss);
    beta = alpha >= 0.f ? -nrm : nrm;
    tau = (beta - alpha) / beta;
    scale = 1.f / (alpha - beta);
  }
}
// FP64: one reciprocal square root gives the norm and 1 / beta, so the chain
// holds eleven FP64 instructions instead of about forty.
__device__ __forceinline__ void householder(double alpha, double ss, double& tau, double& scale, double& beta) {
  if (ss <= 0.0) {
    tau = 0.0;
    scale = 0.0;
    beta = alpha;
  } else {
    const double n2 = fma(alpha, alpha, ss);
    const double r = quick_rsqrt(n2);
    const bool neg = __double2hiint(alpha) < 0;   // beta takes the other sign
    const double nrm = n2 * r;
    beta = neg ? nrm : -nrm;
    tau = (beta - alpha) * (neg ? r : -r);
    scale = quick_rcp(alpha - beta);
  }
}

// The same for FP32 with the hardware-approximate division (2 ulp): the
// register-tiled bidiagonalisation forms these scalars on its critical path.
__device__ __forceinline__ void householder_fast(float alpha, float ss, float& tau, float& scale, float& beta) {
  if (ss <= 0.f) {
    tau = 0.f;
    scale = 0.f;
    beta = alpha;
  } else {
    const float nrm = sqrtf(alpha * alpha + ss);
    beta = alpha >= 0.f ? -nrm : nrm;
    tau = __fdividef(beta - alpha, beta);
    scale = __fdividef(1.f, alpha - beta);
  }
}

// Division inside the inverse-iteration factorisation: IEEE in FP64, the
// hardware approximation (2 ulp) in FP32, where it sits on a long dependent
// chain.
__device__ __forceinline__ double sturm_div(double a, double b) { return a / b; }
__device__ __forceinline__ float sturm_div(float a, float b) { return __fdividef(a, b); }

// One FP32 Sturm step: the next pivot q of T - x (zero diagonal, squared
// off-diagonal t2) and whether it is negative.  The quotient t2 / q is t2 times
// the hardware reciprocal of q, fused with the subtraction; __fdividef's
// scaling for |q| > 2^126 is not needed, as the clamp keeps
// |q| >= pivmin >= 2^-116 tmax^2, so |t2 / q| stays below 2^117.
__device__ __forceinline__ int sturm_count_step(float& q, float x, float t2, float pivmin) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(q));
  q = __fmaf_rn(-t2, r, -x);
  if (fabsf(q) < pivmin) q = -pivmin;
  return (int)(__float_as_uint(q) >> 31);
}

// Number of eigenvalues below x of the zero-diagonal symmetric tridiagonal
// with squared off-diagonals t2 (pivots of the LDL^T factorisation of T - x).
__device__ __forceinline__ int sturm_count(const float* t2, int n2, float x, float pivmin) {
  float q = -x;
  if (fabsf(q) < pivmin) q = -pivmin;
  int cnt = q < 0.f ? 1 : 0;
#pragma unroll 4
  for (int i = 1; i < n2; ++i) cnt += sturm_count_step(q, x, t2[i - 1], pivmin);
  return cnt;
}

// The K largest eigenvalues by sections, with the whole CTA: G threads count at
// G points of a value's interval per step.
static __device__ __noinline__ void section_f32(const float* t2, int n2, int K, float bound, float pivmin, float* lam) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int G = K <= 16 ? 16 : 8;
  const int nit = K <= 16 ? 7 : 9;   // (G + 1)^nit >= 2^26: the last interval is below a quarter ulp of the bound
  const int gid = tid / G, gl = tid % G;
  const int gbase = (lane / G) * G;
  const int idx = n2 - 1 - gid;  // ascending index of the (gid+1)-th largest eigenvalue
  float lo = 0.f, hi = bound;
  for (int it = 0; it < nit; ++it) {
    const float step = (hi - lo) / float(G + 1);
    bool pred = true;
    if (gid < K) {
      const float x = lo + step * float(gl + 1);
      pred = sturm_count(t2, n2, x, pivmin) <= idx;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, pred);
    const unsigned bits = (bal >> gbase) & ((1u << G) - 1u);
    const int gstar = __popc(bits) - 1;
    const float nlo = gstar >= 0 ? lo + step * float(gstar + 1) : lo;
    const float nhi = gstar + 1 < G ? lo + step * float(gstar + 2) : hi;
    lo = nlo;
    hi = nhi;
  }
  if (gid < K && gl == 0) lam[gid] = 0.5f * (lo + hi);
}

// Inverse iteration for one eigenvalue of the n2 x n2 zero-diagonal
// symmetric tridiagonal with off-diagonal t: Gaussian elimination with
// partial pivoting on (T - lam I), two solves from a fixed pseudo-random
// start vector.  Sequential, one thread per eigenvalue, so it is bound by the
// latency of its recurrences.  Four passes over the vector: factorisation
// fused with the first forward elimination, back substitution, the second
// forward elimination (which also applies the scaling of the first iterate),
// back substitution; the last scaling is left to the reader of the vector
// (the return value).  Each iterate is scaled only by its largest entry (the
// solve can amplify by 1/pivtiny); the caller normalises the vectors.
// Row interchanges are selects, not branches: lanes that differ would run both
// sides one after the other, with a division in each.  One warp issues all of
// it, so instructions count: a row's reciprocal pivot, first super-diagonal of
// U, multiplier of L and right-hand side are one 16-byte group (32 in FP64),
// row i of vector k at group i * K + k, and the interchange flag is the top
// exponent bit of the multiplier (|l| <= 1 leaves it free).  The passes over
// stored rows read them a block of four ahead, since the stores in between keep
// the compiler from doing so.  A row takes one reciprocal: of the pivot, for the
// multiplier as well.  The second
// super-diagonal of U is t[i+1] where rows i, i+1 were interchanged and zero
// otherwise, so it is not stored.  The iterate is left in the fourth entries.
template <typename R>
struct InvRow {
  R rdd, du, mult, b;
};
__device__ __forceinline__ InvRow<float> inv_load(const float* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ InvRow<double> inv_load(const double* p) {
  const double2 u = *reinterpret_cast<const double2*>(p), v = *reinterpret_cast<const double2*>(p + 2);
  return {u.x, u.y, v.x, v.y};
}
__device__ __forceinline__ void inv_store(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void inv_store(double* p, double a, double b, double c, double d) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
  *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
}
__device__ __forceinline__ float flag_set(float x, bool f) {
  return __uint_as_float(__float_as_uint(x) | (f ? 0x40000000u : 0u));
}
__device__ __forceinline__ double flag_set(double x, bool f) {
  return __hiloint2double(__double2hiint(x) | (f ? 0x40000000 : 0), __double2loint(x));
}
__device__ __forceinline__ bool flag_get(float x) { return __float_as_uint(x) & 0x40000000u; }
__device__ __forceinline__ bool flag_get(double x) { return __double2hiint(x) & 0x40000000; }
__device__ __forceinline__ float flag_clear(float x) { return __uint_as_float(__float_as_uint(x) & ~0x40000000u); }
__device__ __forceinline__ double flag_clear(double x) {
  return __hiloint2double(__double2hiint(x) & ~0x40000000, __double2loint(x));
}
// Comparisons of magnitudes, start values and scales of the inverse iteration.
// FP64 does them on the bits: an FP64 instruction, a comparison too, keeps its
// unit busy for 64 cycles.
__device__ __forceinline__ bool abs_ge(float a, float b) { return fabsf(a) >= fabsf(b); }
__device__ __forceinline__ bool abs_ge(double a, double b) {
  return (__double_as_longlong(a) & 0x7fffffffffffffffll) >= (__double_as_longlong(b) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ bool is_zero(float a) { return a == 0.f; }
__device__ __forceinline__ bool is_zero(double a) { return (__double_as_longlong(a) & 0x7fffffffffffffffll) == 0; }
__device__ __forceinline__ float with_sign(float m, float s) { return s < 0.f ? -m : m; }
__device__ __forceinline__ double with_sign(double m, double s) {
  return __hiloint2double(__double2hiint(m) | (__double2hiint(s) & 0x80000000), __double2loint(m));
}
__device__ __forceinline__ float inv_start(unsigned h, float) {
  return float((int)(h & 0xffffu) - 32768) / 32768.f + 0.001f;
}
__device__ __forceinline__ double inv_start(unsigned h, double) {   // magnitude in [1/2, 1), random sign
  return __hiloint2double((int)((h & 0x800fffffu) | 0x3fe00000u), (int)(h * 2654435761u));
}
// Largest magnitude so far, and the scale that brings it to about one.
struct MaxOf32 {
  float m = 0.f;
  __device__ void add(float y) { m = fmaxf(m, fabsf(y)); }
  __device__ float scale() const { return m > 0.f ? 1.f / m : 1.f; }
};
struct MaxOf64 {
  int m = 0;
  __device__ void add(double y) { m = max(m, __double2hiint(y) & 0x7fffffff); }
  __device__ double scale() const {
    const int e = m >> 20;
    return e > 0 && e < 2046 ? __hiloint2double((2046 - e) << 20, 0) : 1.0;
  }
};
template <typename R> struct MaxOf;
template <> struct MaxOf<float> { typedef MaxOf32 type; };
template <> struct MaxOf<double> { typedef MaxOf64 type; };
// The workspace start for `p`: the next multiple of 32 bytes.
template <typename R>
__device__ __forceinline__ R* inv_align(R* p) {
  return reinterpret_cast<R*>((reinterpret_cast<size_t>(p) + 31) / 32 * 32);
}

template <typename R>
static __device__ __noinline__ R inverse_iteration(const R* t, int n2, R lam, R pivtiny, R* ws, int K, int k,
                                                   unsigned seed) {
  R* const w0 = ws + 4 * k;
  const int st = 4 * K;
  unsigned h = seed * 2654435761u + 12345u;
  auto start = [&]() {
    h ^= h << 13; h ^= h >> 17; h ^= h << 5;
    return inv_start(h, R(0));
  };
  // ---- factorisation, carrying dd[i], du[i] (current row) and dd[i+1],
  // du[i+1], with the forward elimination of the start vector (carrying b[i])
  R cur_d = -lam, cur_u = n2 > 1 ? t[0] : R(0);
  R bi = start();
  R sub = cur_u;
  const R few = fmax(pivtiny, R(1.17549435e-38));
  R* w = w0;
#pragma unroll 2
  for (int i = 0; i < n2 - 1; ++i, w += st) {
    const R tn = i + 1 < n2 - 1 ? t[i + 1] : R(0);
    const R nd = -lam;
    const R bn = start();
    const bool sw = !abs_ge(cur_d, sub);
    R d = sw ? sub : (is_zero(cur_d) ? pivtiny : cur_d);
    const R num = sw ? cur_d : sub;
    R lm, rd;
    if constexpr (sizeof(R) == 4) {
      if (fabsf(d) < few) {   // tiny pivots: the divisions as __fdividef takes them
        lm = __fdividef(num, d);
        if (fabsf(d) < pivtiny) d = d < R(0) ? -pivtiny : pivtiny;
        rd = __fdividef(1.f, d);
      } else {                // one hardware reciprocal gives both
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd) : "f"(d));
        lm = __fmul_rn(num, rd);
      }
    } else {
      if (!abs_ge(d, pivtiny)) d = with_sign(pivtiny, d);
      rd = quick_rcp(d);
      lm = num * rd;
    }
    const R u = sw ? nd : cur_u, y = sw ? cur_u : nd;
    const R bs = sw ? bn : bi, bo = sw ? bi : bn;
    inv_store(w, rd, u, flag_set(lm, sw), bs);
    cur_d = fma(-lm, u, y);
    cur_u = sw ? -lm * tn : tn;
    bi = fma(-lm, bs, bo);
    sub = tn;
  }
  if (fabs(cur_d) < pivtiny) cur_d = cur_d < R(0) ? -pivtiny : pivtiny;
  inv_store(w, sturm_div(R(1), cur_d), R(0), R(0), bi);
  R* const wl = w;   // the last row
  constexpr int B = 4;
  const int rem = n2 % B, nf = (n2 - 1) / B;
  R sc = R(1);   // scale of the current iterate still to be applied
#pragma unroll 1
  for (int it = 0; it < 2; ++it) {
    if (it == 1) {
      // ---- forward: row interchanges and L^-1 on the scaled iterate; row i
      // needs its own multiplier and the next row's entry
      R bf = w0[3] * sc;
      auto step = [&](R* p, R mult, R bnext) {
        const R bn = bnext * sc, lm = flag_clear(mult);
        const bool sw = flag_get(mult);
        const R bs = sw ? bn : bf, bo = sw ? bf : bn;
        p[3] = bs;
        bf = fma(-lm, bs, bo);
      };
      R nm[B], nb[B];
      w = w0;
      auto load = [&](const R* p) {
#pragma unroll
        for (int q = 0; q < B; ++q) {
          nm[q] = p[q * st + 2];
          nb[q] = p[(q + 1) * st + 3];
        }
      };
      if (nf > 0) load(w);
      for (int blk = 0; blk < nf; ++blk, w += B * st) {
        R cm[B], cb[B];
#pragma unroll
        for (int q = 0; q < B; ++q) {
          cm[q] = nm[q];
          cb[q] = nb[q];
        }
        if (blk + 1 < nf) load(w + B * st);
#pragma unroll
        for (int q = 0; q < B; ++q) step(w + q * st, cm[q], cb[q]);
      }
      for (; w != wl; w += st) step(w, w[2], w[st + 3]);
      wl[3] = bf;
    }
    // ---- backward: U^-1, carrying y[i+1], y[i+2]; track max |y|
    R y1 = R(0), y2 = R(0);
    typename MaxOf<R>::type mx;
    auto step = [&](R* p, const InvRow<R>& v, R tn) {
      const R d2 = flag_get(v.mult) ? tn : R(0);
      const R y = fma(-d2, y2, fma(-v.du, y1, v.b)) * v.rdd;
      p[3] = y;
      mx.add(y);
      y2 = y1;
      y1 = y;
    };
    int i = n2 - 1;
    w = wl;
    for (; i >= n2 - rem; --i, w -= st) step(w, inv_load(w), i + 1 < n2 - 1 ? t[i + 1] : R(0));
    InvRow<R> nv[B];
    R nt[B];
    auto load = [&](const R* p, int j) {   // rows j, j - 1, ..
#pragma unroll
      for (int q = 0; q < B; ++q) {
        nv[q] = inv_load(p - q * st);
        nt[q] = j - q + 1 < n2 - 1 ? t[j - q + 1] : R(0);
      }
    };
    if (i >= 0) load(w, i);
    for (; i >= 0; i -= B, w -= B * st) {
      InvRow<R> cv[B];
      R ct[B];
#pragma unroll
      for (int q = 0; q < B; ++q) {
        cv[q] = nv[q];
        ct[q] = nt[q];
      }
      if (i >= B) load(w - B * st, i - B);
#pragma unroll
      for (int q = 0; q < B; ++q) step(w - q * st, cv[q], ct[q]);
    }
    sc = mx.scale();
  }
  return sc;
}

// v[k] for a run-time k
__device__ __forceinline__ float sel8(const float (&v)[8], int k) {
  float x = v[0];
#pragma unroll
  for (int q = 1; q < 8; ++q) x = k == q ? v[q] : x;
  return x;
}
// Column c of a pair-packed 8 x 8 tile.  c is uniform across the CTA, so a
// branch on it costs no divergence and each case is eight register moves
// (selecting by comparisons would cost about seven instructions per entry).
__device__ __forceinline__ void col_of(const float2 (&a)[8][4], int c, float (&out)[8]) {
#define PEPS_COL_CASE(C)                                                      \
  case C:                                                                     \
    _Pragma("unroll") for (int r = 0; r < 8; ++r) out[r] = ((C) & 1) ? a[r][(C) >> 1].y : a[r][(C) >> 1].x; \
    break;
  switch (c) {
    PEPS_COL_CASE(0) PEPS_COL_CASE(1) PEPS_COL_CASE(2) PEPS_COL_CASE(3)
    PEPS_COL_CASE(4) PEPS_COL_CASE(5) PEPS_COL_CASE(6) default: PEPS_COL_CASE(7)
  }
#undef PEPS_COL_CASE
}
// Row r of a pair-packed 8 x 8 tile; r is uniform across the CTA.
__device__ __forceinline__ void row_of(const float2 (&a)[8][4], int r, float (&out)[8]) {
#define PEPS_ROW_CASE(R)                                                      \
  case R:                                                                     \
    _Pragma("unroll") for (int k = 0; k < 4; ++k) {                           \
      out[2 * k] = a[R][k].x;                                                 \
      out[2 * k + 1] = a[R][k].y;                                             \
    }                                                                         \
    break;
  switch (r) {
    PEPS_ROW_CASE(0) PEPS_ROW_CASE(1) PEPS_ROW_CASE(2) PEPS_ROW_CASE(3)
    PEPS_ROW_CASE(4) PEPS_ROW_CASE(5) PEPS_ROW_CASE(6) default: PEPS_ROW_CASE(7)
  }
#undef PEPS_ROW_CASE
}
// Householder bidiagonalisation of an FP32 matrix of at most 128 x 128 held
// in registers: thread (ti, tj) owns the 8 x 8 tile of rows 8 ti.., columns
// 8 tj.., with ti = lane % 16 and tj = 2 warp + lane / 16, so the 16 tiles of a
// tile column sit in one half-warp (column sums are shuffle reductions) and
// the tiles of a tile row in one lane position of every half-warp.  A tile is
// kept as column pairs and updated with packed FP32x2 multiply-adds; the
// active row and column are picked out of the tile by selects (a register
// array cannot be indexed at run time).  Not inlined: its own register
// allocation holds the 64-element tile without spilling.  The
// arithmetic is that of the shared-memory version below (same reflectors,
// same stored factors); only the order of the partial sums differs.  One
// column costs four barriers: broadcast of the left reflector, the row norm
// of the right reflector, and two for the cross-warp sums of W u (per-warp
// shares, then row totals).  Column sums within a half-warp are a
// reduce-scatter followed by an all-gather, the same additions as a
// butterfly in fewer shuffles.  Warps whose two tile columns lie left of the
// active column skip the products.  On return W
// (P x Q, leading dimension ld) holds the unscaled reflectors; t and tau4
// (tau left, tau right, scale left, scale right, qm apart) are set as by the
// shared-memory version.
static __device__ __noinline__ void bidiag_tiles_f32(const float* X, int n, bool tall, int P, int Q, float* W, int ld,
                                                 float* t, float* tau4, int qm) {
  __shared__ __align__(16) float zp[kWarps * 128];   // per-warp partial sums of W u
  __shared__ __align__(16) float vL[128];            // left reflector, by row
  __shared__ __align__(16) float zt[128];            // row totals of W u
  __shared__ float sc[2];                            // tau_left, alpha_right
  __shared__ __align__(16) float rnp[16];            // row-norm partials, by tile column
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ti = lane & 15;
  const int tj = warp * 2 + (lane >> 4);
  const int r0 = ti * 8, c0 = tj * 8;
  const unsigned hmask = (lane & 16) ? 0xffff0000u : 0x0000ffffu;
  float2 a[8][4];   // a[r][q] = columns (2q, 2q+1) of row r of the tile
  if (tall && (n & 3) == 0 && (reinterpret_cast<size_t>(X) & 15) == 0) {
    // whole groups of four columns: a quarter of the memory lines per load
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int q = 0; q < 4; q += 2) {
        const int i = r0 + r, c = c0 + 2 * q;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < P && c < Q) v = *reinterpret_cast<const float4*>(X + i * n + c);
        a[r][q] = make_float2(v.x, v.y);
        a[r][q + 1] = make_float2(v.z, v.w);
      }
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = r0 + r, c = c0 + 2 * q;
        float x0 = 0.f, x1 = 0.f;
        if (i < P) {
          if (c < Q) x0 = tall ? X[i * n + c] : X[c * n + i];
          if (c + 1 < Q) x1 = tall ? X[i * n + c + 1] : X[(c + 1) * n + i];
        }
        a[r][q] = make_float2(x0, x1);
      }
  }
  for (int jb = 0; jb < Q; jb += 8) {
    const int tb = jb >> 3;   // tile row / column of j
#pragma unroll 1
    for (int jj = 0; jj < 8; ++jj) {
      const int j = jb + jj;
      if (j < Q) {
        // ---- left reflector on column j (rows j..P-1), formed by the owning half-warp
        if (tj == tb) {
          float col[8];
          col_of(a, jj, col);
          float ss = 0.f;
#pragma unroll
          for (int r = 0; r < 8; ++r)
            if (r0 + r > j) ss = fmaf(col[r], col[r], ss);
#pragma unroll
          for (int o = 8; o >= 1; o >>= 1) ss += __shfl_xor_sync(hmask, ss, o);
          const float alpha = __shfl_sync(hmask, sel8(col, jj), (lane & 16) | tb);
          float tau, scale, beta;
          householder_fast(alpha, ss, tau, scale, beta);
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const int i = r0 + r;
            vL[i] = i == j ? 1.f : (i > j ? scale * col[r] : 0.f);
          }
          if (ti == 0) {
            sc[0] = tau;
            t[2 * j] = beta;
            tau4[j] = tau;
            tau4[2 * qm + j] = scale;
          }
        }
        __syncthreads();
        if (warp * 16 + 15 > j) {   // some column of this warp lies right of j
          const float tau = sc[0];
          float v[8];
          const float4 v0 = *reinterpret_cast<const float4*>(vL + r0);
          const float4 v1 = *reinterpret_cast<const float4*>(vL + r0 + 4);
          v[0] = v0.x; v[1] = v0.y; v[2] = v0.z; v[3] = v0.w;
          v[4] = v1.x; v[5] = v1.y; v[6] = v1.z; v[7] = v1.w;
          float2 wc[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int r = 0; r < 8; ++r) s = __ffma2_rn(make_float2(v[r], v[r]), a[r][q], s);
            wc[q] = s;
          }
          {
            // reduce-scatter over the half-warp (lane bits 3, 2, 1 pick the
            // column), then all-gather
            float w8[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              w8[2 * q] = wc[q].x;
              w8[2 * q + 1] = wc[q].y;
            }
            const bool b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
            float k4[4], k2[2];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float snd = b3 ? w8[i] : w8[i + 4], kp = b3 ? w8[i + 4] : w8[i];
              k4[i] = kp + __shfl_xor_sync(0xffffffffu, snd, 8);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float snd = b2 ? k4[i] : k4[i + 2], kp = b2 ? k4[i + 2] : k4[i];
              k2[i] = kp + __shfl_xor_sync(0xffffffffu, snd, 4);
            }
            float k1;
            {
              const float snd = b1 ? k2[0] : k2[1], kp = b1 ? k2[1] : k2[0];
              k1 = kp + __shfl_xor_sync(0xffffffffu, snd, 2);
            }
            k1 += __shfl_xor_sync(0xffffffffu, k1, 1);
            const int hb = lane & 16;
#pragma unroll
            for (int c = 0; c < 8; ++c)
              w8[c] = __shfl_sync(0xffffffffu, k1, hb | ((c >> 2) << 3) | (((c >> 1) & 1) << 2) | ((c & 1) << 1));
#pragma unroll
            for (int q = 0; q < 4; ++q) wc[q] = make_float2(w8[2 * q], w8[2 * q + 1]);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            wc[q].x = (c0 + 2 * q > j) ? -tau * wc[q].x : 0.f;
            wc[q].y = (c0 + 2 * q + 1 > j) ? -tau * wc[q].y : 0.f;
          }
#pragma unroll
          for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) a[r][q] = __ffma2_rn(make_float2(v[r], v[r]), wc[q], a[r][q]);
        }
        if (j < Q - 1) {
          // ---- right reflector on row j (columns j+1..Q-1)
          const int ja = (jj + 1) & 7;       // local column of j+1
          const int ta = (j + 1) >> 3;       // its tile column
          // warp-uniform: some column of this warp lies right of j.  A warp
          // whose columns all lie left of j has a zero share of the row norm
          // and of W u, and nothing to update, so it skips both.
          const bool act = warp * 16 + 15 > j;
          float row[8];
          if (act) row_of(a, jj, row);
          if (ti == tb) {
            float ss = 0.f;
            if (act) {
#pragma unroll
              for (int c = 0; c < 8; ++c)
                if (c0 + c > j + 1) ss = fmaf(row[c], row[c], ss);
              if (tj == ta) sc[1] = sel8(row, ja);
            }
            rnp[tj] = ss;
          }
          __syncthreads();
          float ssr = 0.f;
#pragma unroll
          for (int q = 0; q < 16; q += 4) {
            const float4 p4 = *reinterpret_cast<const float4*>(rnp + q);
            ssr += p4.x;
            ssr += p4.y;
            ssr += p4.z;
            ssr += p4.w;
          }
          float tr, sr, br;
          householder_fast(sc[1], ssr, tr, sr, br);
          if (tid == 0) {
            t[2 * j + 1] = br;
            tau4[qm + j] = tr;
            tau4[3 * qm + j] = sr;
          }
          float2 u[4];
          float z[8];
          if (act) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float2 x = make_float2(__shfl_sync(0xffffffffu, row[2 * q], (lane & 16) | tb),
                                           __shfl_sync(0xffffffffu, row[2 * q + 1], (lane & 16) | tb));
              const int c = c0 + 2 * q;
              u[q].x = c == j + 1 ? 1.f : (c > j + 1 ? sr * x.x : 0.f);
              u[q].y = c + 1 == j + 1 ? 1.f : (c + 1 > j + 1 ? sr * x.y : 0.f);
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
              float2 s = make_float2(0.f, 0.f);
#pragma unroll
              for (int q = 0; q < 4; ++q) s = __ffma2_rn(a[r][q], u[q], s);
              z[r] = s.x + s.y;
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) z[r] += __shfl_xor_sync(0xffffffffu, z[r], 16);
            if (lane < 16) {
              *reinterpret_cast<float4*>(zp + warp * 128 + r0) = make_float4(z[0], z[1], z[2], z[3]);
              *reinterpret_cast<float4*>(zp + warp * 128 + r0 + 4) = make_float4(z[4], z[5], z[6], z[7]);
            }
          }
          __syncthreads();
          // Row totals of W u, one thread per row, the warps' shares added in
          // warp order; a warp whose columns all lie left of j has a zero
          // share and did not write it.  Every thread then reads the totals
          // of its eight rows (one more barrier instead of each of the 16
          // threads of a row adding all eight shares again).
          if (tid < 128) {
            float zs = 0.f;
#pragma unroll
            for (int q = 0; q < kWarps; ++q)
              if (q * 16 + 15 > j) zs += zp[q * 128 + tid];
            zt[tid] = zs;
          }
          __syncthreads();
          if (act) {
            const float4 p0 = *reinterpret_cast<const float4*>(zt + r0);
            const float4 p1 = *reinterpret_cast<const float4*>(zt + r0 + 4);
            z[0] = p0.x; z[1] = p0.y; z[2] = p0.z; z[3] = p0.w;
            z[4] = p1.x; z[5] = p1.y; z[6] = p1.z; z[7] = p1.w;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
              const float zr = (r0 + r > j) ? -tr * z[r] : 0.f;
#pragma unroll
              for (int q = 0; q < 4; ++q) a[r][q] = __ffma2_rn(make_float2(zr, zr), u[q], a[r][q]);
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = r0 + r, c = c0 + 2 * q;
      if (i < P && c < Q) W[i * ld + c] = a[r][q].x;
      if (i < P && c + 1 < Q) W[i * ld + c + 1] = a[r][q].y;
    }
  __syncthreads();
}

// The reflectors j = jtop, jtop - 1, .. whose first row j + off lies in rows
// 16 R0 .. 16 R0 + 15, applied to a column of U (u[r]: row l + 16 r) by a
// half-warp; returns the next j.  The next reflector's entries are read while
// the current dot product is reduced.
template <int R0>
__device__ __forceinline__ int apply_reflectors(const float* W, int ld, bool tall, int rows, int l, int off, int jtop,
                                                const float* taus, const float* scs, float (&u)[8]) {
  const int jlo = max(16 * R0 - off, 0);
  if (jtop < jlo) return jtop;
  const int rs = 16 * (tall ? ld : 1), js = tall ? 1 : ld;
  const float* p = W + (l + 16 * R0) * (tall ? ld : 1) + jtop * js;
  float w[8];
  auto load = [&](const float* q) {
#pragma unroll
    for (int r = R0; r < 8; ++r) w[r] = l + 16 * r < rows ? q[(r - R0) * rs] : 0.f;
  };
  load(p);
  float tj = taus[jtop], sj = scs[jtop];
  for (int j = jtop; j >= jlo; --j) {
    const int i0 = l + 16 * R0, pv = j + off;
    float v[8], d = 0.f;
#pragma unroll
    for (int r = R0; r < 8; ++r) {
      v[r] = sj * w[r];
      if (r == R0) v[r] = i0 < pv ? 0.f : (i0 == pv ? 1.f : v[r]);
      d = fmaf(v[r], u[r], d);
    }
    const float tc = tj;
    if (j > jlo) {
      p -= js;
      load(p);
      tj = taus[j - 1];
      sj = scs[j - 1];
    }
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    const float cf = -tc * d;
#pragma unroll
    for (int r = R0; r < 8; ++r) u[r] = fmaf(cf, v[r], u[r]);
  }
  return jlo - 1;
}

// W[i][c] -= cf(c) rf(i) for i0 <= i < P, col0 <= c < col0 + ncol <= 256: a warp
// takes every eighth row, two at a time, with its column factors and the rows'
// chunks of 32 columns in registers, so that a row's loads do not wait for the
// stores of the one before.  The number of chunks is a template argument: a
// predicated-off FP64 instruction still takes its issue time.  note(i, chunk,
// entry, acc) sees the updated entries in order; done(acc) ends a warp's part.
template <typename R, int NCH, class CF, class RF, class Note>
__device__ __forceinline__ R rank1_chunks(R* W, int ld, int i0, int P, int col0, int ncol, CF cf, RF rf, Note note) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool last = 32 * (NCH - 1) + lane < ncol;
  R w[NCH], acc = R(0);
#pragma unroll
  for (int t = 0; t < NCH; ++t) w[t] = (t < NCH - 1 || last) ? cf(col0 + lane + 32 * t) : R(0);
  int i = i0 + warp;
  for (; i + kWarps < P; i += 2 * kWarps) {
    R* r0 = W + i * ld + col0 + lane;
    R* r1 = r0 + kWarps * ld;
    const R v0 = rf(i), v1 = rf(i + kWarps);
    R x0[NCH], x1[NCH];
#pragma unroll
    for (int t = 0; t < NCH; ++t)
      if (t < NCH - 1 || last) {
        x0[t] = r0[32 * t] - w[t] * v0;
        x1[t] = r1[32 * t] - w[t] * v1;
      }
#pragma unroll
    for (int t = 0; t < NCH; ++t)
      if (t < NCH - 1 || last) {
        r0[32 * t] = x0[t];
        r1[32 * t] = x1[t];
      }
#pragma unroll
    for (int t = 0; t < NCH; ++t)
      if (t < NCH - 1 || last) note(i, t, x0[t], acc);
#pragma unroll
    for (int t = 0; t < NCH; ++t)
      if (t < NCH - 1 || last) note(i + kWarps, t, x1[t], acc);
  }
  if (i < P) {
    R* r0 = W + i * ld + col0 + lane;
    const R v0 = rf(i);
#pragma unroll
    for (int t = 0; t < NCH; ++t)
      if (t < NCH - 1 || last) {
        const R x = r0[32 * t] - w[t] * v0;
        r0[32 * t] = x;
        note(i, t, x, acc);
      }
  }
  return acc;
}
template <typename R, class CF, class RF, class Note, class Done>
__device__ __forceinline__ void rank1_rows(R* W, int ld, int i0, int P, int col0, int ncol, CF cf, RF rf, Note note,
                                           Done done) {
  R acc;
  switch ((ncol + 31) >> 5) {
    case 1: acc = rank1_chunks<R, 1>(W, ld, i0, P, col0, ncol, cf, rf, note); break;
    case 2: acc = rank1_chunks<R, 2>(W, ld, i0, P, col0, ncol, cf, rf, note); break;
    case 3: acc = rank1_chunks<R, 3>(W, ld, i0, P, col0, ncol, cf, rf, note); break;
    case 4: acc = rank1_chunks<R, 4>(W, ld, i0, P, col0, ncol, cf, rf, note); break;
    case 5: acc = rank1_chunks<R, 5>(W, ld, i0, P, col0, ncol, cf, rf, note); break;
    case 6: acc = rank1_chunks<R, 6>(W, ld, i0, P, col0, ncol, cf, rf, note); break;
    case 7: acc = rank1_chunks<R, 7>(W, ld, i0, P, col0, ncol, cf, rf, note); break;
    default: acc = rank1_chunks<R, 8>(W, ld, i0, P, col0, ncol, cf, rf, note); break;
  }
  done(acc);
}

// Householder bidiagonalisation (W = Q_L B Q_R^T, B upper bidiagonal) of X or its
// transpose in W (shared or global memory), for the blocks bidiag_tiles_f32 does
// not take.  One function for both sweep directions: it is most of the
// truncation's code.
template <typename R>
static __device__ __noinline__ void bidiag_shared(const R* X, int m, int n, bool tall, int P, int Q, R* W, int ld, R* tt,
                                                  R* tau4, int qm, R* wv_, R* red) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    R* tauL = tau4;
    R* tauR = tau4 + qm;
    for (int e = tid; e < m * n; e += blockDim.x) {
      const int i = e / n, j = e % n;
      if (tall) W[i * ld + j] = X[e];
      else W[j * ld + i] = X[e];
    }
    __syncthreads();
    // ---------------- bidiagonalisation: W = Q_L B Q_R^T, B upper bidiagonal
    // Reflectors are kept unscaled in W with their scale factors in sL / sR
    // (v = scale * stored, implicit 1 on the diagonal / super-diagonal).  The
    // norm each Householder vector needs is accumulated while the previous
    // rank-1 update writes those entries, and every thread forms the scalars
    // itself, so one column costs four barriers.
    R* wv = wv_;
    R* sL = tau4 + 2 * qm;        // left scale factors (t2 is filled later)
    R* sR = sL + qm;
    R* part = red + 40;                // per-warp partial norms (8)
    {
      R ss = R(0);
      for (int i = 1 + tid; i < P; i += blockDim.x) ss += W[i * ld] * W[i * ld];
      ss = block_sum(ss, red + 16);
      if (tid < kWarps) part[tid] = tid == 0 ? ss : R(0);
      __syncthreads();
    }
    for (int j = 0; j < Q; ++j) {
      // -- left reflector on column j (rows j..P-1); its norm is in part[]
      R colnorm = R(0);
      for (int q = 0; q < kWarps; ++q) colnorm += part[q];
      R tau, scale, beta;
      householder(W[j * ld + j], colnorm, tau, scale, beta);
      if (tid == 0) {
        tt[2 * j] = beta;
        tauL[j] = tau;
        sL[j] = scale;
      }
      const int ncol = Q - j - 1;
      R rownorm = R(0);                // squared norm of row j beyond j+1 after the left update
      if (tau != R(0) && ncol > 0) {
        // wv[c] = tau * (W[j][c] + scale * sum_{i>j} W[i][j] W[i][c])
        int tpc = kThreads / ncol;
        tpc = tpc >= 32 ? 32 : tpc >= 16 ? 16 : tpc >= 8 ? 8 : tpc >= 4 ? 4 : tpc >= 2 ? 2 : 1;
        const int cpr = kThreads / tpc;
        for (int cb = 0; cb < ncol; cb += cpr) {
          const int cl = cb + tid / tpc, gl = tid % tpc;
          const bool act = cl < ncol;
          const int c = j + 1 + (act ? cl : 0);
          R s0 = R(0), s1 = R(0), s2 = R(0), s3 = R(0);
          int i = j + 1 + gl;
#pragma unroll 2
          for (; i + 3 * tpc < P; i += 4 * tpc) {
            s0 += W[i * ld + j] * W[i * ld + c];
            s1 += W[(i + tpc) * ld + j] * W[(i + tpc) * ld + c];
            s2 += W[(i + 2 * tpc) * ld + j] * W[(i + 2 * tpc) * ld + c];
            s3 += W[(i + 3 * tpc) * ld + j] * W[(i + 3 * tpc) * ld + c];
          }
          for (; i < P; i += tpc) s0 += W[i * ld + j] * W[i * ld + c];
          const R sacc = warp_sum((s0 + s1) + (s2 + s3), tpc);
          if (act && gl == 0) wv[c] = tau * (W[j * ld + c] + scale * sacc);
        }
        __syncthreads();
        // W[i][c] -= wv[c] v_i for i >= j, c > j; warp 0 takes row j and its norm
        rank1_rows<R>(
            W, ld, j, P, j + 1, ncol, [&](int c) { return wv[c]; },
            [&](int i) { return i == j ? R(1) : scale * W[i * ld + j]; },
            [&](int i, int t, R x, R& acc) {
              if (i == j && 32 * t + lane >= 1) acc += x * x;
            },
            [&](R acc) {
              if (warp == 0) {
                acc = warp_sum(acc);
                if (lane == 0) red[5] = acc;
              }
            });
        __syncthreads();
        rownorm = red[5];
      } else if (ncol > 0) {
        if (warp == 0) {
          R rn = R(0);
          for (int c = j + 2 + lane; c < Q; c += 32) rn += W[j * ld + c] * W[j * ld + c];
          rn = warp_sum(rn);
          if (lane == 0) red[5] = rn;
        }
        __syncthreads();
        rownorm = red[5];
      }
      if (j < Q - 1) {
        // -- right reflector on row j (columns j+1..Q-1)
        R tr, sr, br;
        householder(W[j * ld + j + 1], rownorm, tr, sr, br);
        if (tid == 0) {
          tt[2 * j + 1] = br;
          tauR[j] = tr;
          sR[j] = sr;
        }
        const int nrow = P - j - 1;
        if (tr != R(0)) {
          // wv[i] = tr * (W[i][j+1] + sr * sum_{c>j+1} W[i][c] W[j][c])
          int tpc = kThreads / nrow;
          tpc = tpc >= 32 ? 32 : tpc >= 16 ? 16 : tpc >= 8 ? 8 : tpc >= 4 ? 4 : tpc >= 2 ? 2 : 1;
          const int rpr = kThreads / tpc;
          for (int rb = 0; rb < nrow; rb += rpr) {
            const int rl = rb + tid / tpc, gl = tid % tpc;
            const bool act = rl < nrow;
            const int i = j + 1 + (act ? rl : 0);
            R s0 = R(0), s1 = R(0), s2 = R(0), s3 = R(0);
            int c = j + 2 + gl;
#pragma unroll 2
            for (; c + 3 * tpc < Q; c += 4 * tpc) {
              s0 += W[i * ld + c] * W[j * ld + c];
              s1 += W[i * ld + c + tpc] * W[j * ld + c + tpc];
              s2 += W[i * ld + c + 2 * tpc] * W[j * ld + c + 2 * tpc];
              s3 += W[i * ld + c + 3 * tpc] * W[j * ld + c + 3 * tpc];
            }
            for (; c < Q; c += tpc) s0 += W[i * ld + c] * W[j * ld + c];
            const R sacc = warp_sum((s0 + s1) + (s2 + s3), tpc);
            if (act && gl == 0) wv[i] = tr * (W[i * ld + j + 1] + sr * sacc);
          }
          __syncthreads();
          // W[i][c] -= wv[i] v'_c for i > j, c > j; lane 0 of each warp sums column j+1 below row j+1
          rank1_rows<R>(
              W, ld, j + 1, P, j + 1, ncol, [&](int c) { return c == j + 1 ? R(1) : sr * W[j * ld + c]; },
              [&](int i) { return wv[i]; },
              [&](int i, int t, R x, R& acc) {
                if (t == 0 && lane == 0 && i > j + 1) acc += x * x;
              },
              [&](R acc) {
                if (lane == 0) part[warp] = acc;
              });
          __syncthreads();
        } else {
          // no right update: column j+1's norm below row j+1 as it stands
          R cn = R(0);
          for (int i = j + 2 + tid; i < P; i += blockDim.x) cn += W[i * ld + j + 1] * W[i * ld + j + 1];
          cn = block_sum(cn, red + 16);
          if (tid < kWarps) part[tid] = tid == 0 ? cn : R(0);
          __syncthreads();
        }
      }
    }
    // the last column's diagonal entry (tt[2Q-2], written by thread 0) is
    // read by another warp in the bisection set-up below
    __syncthreads();
}

// Gram-Schmidt with re-orthogonalisation of the columns of Ub (Q x K); a
// degenerate direction is replaced by a unit vector.
template <typename R>
static __device__ __noinline__ void gram_schmidt(R* Ub, int Q, int K, R* red) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int j = 0; j < K; ++j) {
    for (int attempt = 0; attempt <= Q; ++attempt) {
      R s = R(0);
      for (int i = tid; i < Q; i += blockDim.x) s += Ub[i * K + j] * Ub[i * K + j];
      R nrm0 = dsqrt(block_sum(s, red + 16));
      if (nrm0 > R(0)) {
        for (int i = tid; i < Q; i += blockDim.x) Ub[i * K + j] /= nrm0;
        __syncthreads();
      }
      for (int pass = 0; pass < 2; ++pass) {
        for (int p = warp; p < j; p += kWarps) {
          R d = R(0);
          for (int i = lane; i < Q; i += 32) d += Ub[i * K + p] * Ub[i * K + j];
          d = warp_sum(d);
          if (lane == 0) red[32 + p] = d;
        }
        __syncthreads();
        for (int i = tid; i < Q; i += blockDim.x) {
          R v = Ub[i * K + j];
          for (int p = 0; p < j; ++p) v -= red[32 + p] * Ub[i * K + p];
          Ub[i * K + j] = v;
        }
        __syncthreads();
      }
      s = R(0);
      for (int i = tid; i < Q; i += blockDim.x) s += Ub[i * K + j] * Ub[i * K + j];
      const R nrm = dsqrt(block_sum(s, red + 16));
      if (nrm0 > R(0) && nrm > R(1e-3)) {
        for (int i = tid; i < Q; i += blockDim.x) Ub[i * K + j] /= nrm;
        __syncthreads();
        break;
      }
      // degenerate direction (zero singular value or lost vector): try a unit vector
      const int q = (j + attempt) % Q;
      for (int i = tid; i < Q; i += blockDim.x) Ub[i * K + j] = i == q ? R(1) : R(0);
      __syncthreads();
    }
  }
}

// CholeskyQR2 of the columns of Ub (Q x K) in place; G: K x K.  Returns true where
// a direction is too small (the caller then takes Gram-Schmidt).
template <typename R>
static __device__ __noinline__ bool cholesky_qr2(R* Ub, R* G, int Q, int K) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  bool need_cgs = false;
  {
    __shared__ int cq_bad;
    for (int pass = 0; pass < 2 && !need_cgs; ++pass) {
      for (int e = tid; e < K * K; e += blockDim.x) {
        const int a = e / K, b = e % K;
        if (b < a) continue;
        R sacc = R(0);
#pragma unroll 8
        for (int i = 0; i < Q; ++i) sacc += Ub[i * K + a] * Ub[i * K + b];
        G[e] = sacc;
      }
      __syncthreads();
      if (warp == 0) {
        // right-looking Cholesky of the upper triangle in place; lane l owns column l
        const R d0 = lane < K ? G[lane * K + lane] : R(0);
        int bad = 0;
        for (int j = 0; j < K && !bad; ++j) {
          const R d = G[j * K + j];
          const R dj0 = __shfl_sync(0xffffffffu, d0, j);
          if (!(d > R(1e-6) * dj0) || !(dj0 > R(0))) {
            bad = 1;
            break;
          }
          R r;
          if constexpr (sizeof(R) == 4) {
            r = dsqrt(d);
            __syncwarp();
            if (lane > j && lane < K) G[j * K + lane] /= r;
          } else {   // the diagonal holds 1 / r
            r = quick_rsqrt(d);
            __syncwarp();
            if (lane > j && lane < K) G[j * K + lane] *= r;
          }
          __syncwarp();
          if (lane == j) G[j * K + j] = r;
          if (lane > j && lane < K) {
            // rows in blocks of four, loaded before the block's stores
            const R gjl = G[j * K + lane];
            for (int m0 = j + 1; m0 <= lane; m0 += 4) {
              R x[4];
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (m0 + q <= lane) x[q] = fma(-G[j * K + m0 + q], gjl, G[(m0 + q) * K + lane]);
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (m0 + q <= lane) G[(m0 + q) * K + lane] = x[q];
            }
          }
          __syncwarp();
        }
        if (lane == 0) cq_bad = bad;
      }
      __syncthreads();
      if (cq_bad) {
        need_cgs = true;
        break;
      }
      // Ub <- Ub R^-1, one thread per row (forward substitution in place)
      for (int i = tid; i < Q; i += blockDim.x) {
        if (K <= 16) {   // the row in registers
          R u[16];
#pragma unroll
          for (int l = 0; l < 16; ++l)
            if (l < K) {
              R x = Ub[i * K + l];
#pragma unroll
              for (int k = 0; k < l; ++k) x = fma(-u[k], G[k * K + l], x);
              u[l] = sizeof(R) == 4 ? x / G[l * K + l] : x * G[l * K + l];
              Ub[i * K + l] = u[l];
            }
        } else {
          for (int l = 0; l < K; ++l) {
            R x = Ub[i * K + l];
            for (int k = 0; k < l; ++k) x -= Ub[i * K + k] * G[k * K + l];
            Ub[i * K + l] = sizeof(R) == 4 ? x / G[l * K + l] : x * G[l * K + l];
          }
        }
      }
      __syncthreads();
    }
  }
  return need_cgs;
}

static __device__ __forceinline__ void apply_all_reflectors(const float* Wf, int ld, bool tall, int rowsU, int nref, int K,
                                                         const float* tf, const float* sf, float* Uk) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int c = warp * 2 + (lane >> 4), l = lane & 15;
        float u[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int i = l + 16 * r;
          u[r] = (c < K && i < rowsU) ? Uk[i * K + c] : 0.f;
        }
        int j = nref - 1;
        const int off = tall ? 0 : 1;   // first row of reflector j: j + off
        j = apply_reflectors<7>(Wf, ld, tall, rowsU, l, off, j, tf, sf, u);
        j = apply_reflectors<6>(Wf, ld, tall, rowsU, l, off, j, tf, sf, u);
        j = apply_reflectors<5>(Wf, ld, tall, rowsU, l, off, j, tf, sf, u);
        j = apply_reflectors<4>(Wf, ld, tall, rowsU, l, off, j, tf, sf, u);
        j = apply_reflectors<3>(Wf, ld, tall, rowsU, l, off, j, tf, sf, u);
        j = apply_reflectors<2>(Wf, ld, tall, rowsU, l, off, j, tf, sf, u);
        j = apply_reflectors<1>(Wf, ld, tall, rowsU, l, off, j, tf, sf, u);
        apply_reflectors<0>(Wf, ld, tall, rowsU, l, off, j, tf, sf, u);
        if (c < K) {
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const int i = l + 16 * r;
            if (i < rowsU) Uk[i * K + c] = u[r];
          }
        }
}

// The FP32 end of a cut: one Newton-Schulz step on U (m x K in shared memory,
// Uk), U to Uout, the carry U^T X to Cout (see the caller).  Mns: K x K; Ug: a global copy of U.
static __device__ __forceinline__ void finish_f32(const float* X, int m, int n, int K, float* Mns, float* Uk, float* Ug,
                                               float* Uout, Ix uo_r, Ix uo_c, float* Cout, Ix co_r, Ix co_c) {
    const int tid = threadIdx.x;
    const float* Uf = Uk;
    for (int e = tid; e < K * K; e += blockDim.x) {
      const int a = e / K, b = e % K;
      float s = 0.f, c = 0.f;
      for (int i = 0; i < m; ++i) dot2_step(Uf[i * K + a], Uf[i * K + b], s, c);
      // s is within a factor 2 of 1 on the diagonal, so s - 1 is exact
      Mns[e] = -0.5f * (a == b ? __fadd_rn(__fsub_rn(s, 1.f), c) : __fadd_rn(s, c));
    }
    __syncthreads();
    // Up to kNsPer entries per thread, the new U replaces the old one in
    // shared memory once every thread has read the old one; larger U go to
    // the global copy.
    constexpr int kNsPer = 8;
    const bool u_shared = m * K <= kNsPer * kThreads;
    float* Us = Uk;
    if (u_shared) {
      float nv[kNsPer];
#pragma unroll
      for (int q = 0; q < kNsPer; ++q) {
        const int e = tid + q * kThreads;
        if (e < m * K) {
          const int i = e / K, k = e % K;
          float corr = 0.f;
          for (int a = 0; a < K; ++a) corr = fmaf(Uf[i * K + a], Mns[a * K + k], corr);
          nv[q] = Uf[i * K + k] + corr;
          Uout[ixoff(uo_r, i) + ixoff(uo_c, k)] = nv[q];
        }
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < kNsPer; ++q) {
        const int e = tid + q * kThreads;
        if (e < m * K) Us[e] = nv[q];
      }
    } else {
      for (int e = tid; e < m * K; e += blockDim.x) {
        const int i = e / K, k = e % K;
        float corr = 0.f;
        for (int a = 0; a < K; ++a) corr = fmaf(Uf[i * K + a], Mns[a * K + k], corr);
        const float v = Uf[i * K + k] + corr;
        Uout[ixoff(uo_r, i) + ixoff(uo_c, k)] = v;
        Ug[e] = v;
      }
    }
    __syncthreads();
    // C' = U_K^T X, X row-major m x n.  One work item is a column j and a
    // chunk of 8 rows of C'; its X column is read once (coalesced over j),
    // eight rows at a time so that eight loads are in flight together.
    constexpr int CH = 8, XB = 8;
    const float* Uo = u_shared ? Us : Ug;
    const float* Xf = X;
    const int nchunk = (K + CH - 1) / CH;
    for (int item = tid; item < n * nchunk; item += blockDim.x) {
      const int j = item % n, a0 = (item / n) * CH;
      float s[CH], c[CH];
#pragma unroll
      for (int q = 0; q < CH; ++q) s[q] = c[q] = 0.f;
      for (int ib = 0; ib < m; ib += XB) {
        float xb[XB];
#pragma unroll
        for (int u = 0; u < XB; ++u) xb[u] = ib + u < m ? Xf[(ib + u) * n + j] : 0.f;
#pragma unroll
        for (int u = 0; u < XB; ++u) {
          const int i = ib + u;
          if (i < m) {
#pragma unroll
            for (int q = 0; q < CH; ++q)
              if (a0 + q < K) dot2_step(Uo[i * K + a0 + q], xb[u], s[q], c[q]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < CH; ++q)
        if (a0 + q < K) Cout[ixoff(co_r, a0 + q) + ixoff(co_c, j)] = __fadd_rn(s[q], c[q]);
    }
    __syncthreads();
}

// Writes U_K (m x K) through (uo_r, uo_c) and C' = U_K^T X (K x n) through
// (co_r, co_c).  X is not modified.  K <= min(m, n), K <= 32.
template <typename R>
__device__ void cta_topk_left(const R* X, int m, int n, int K, TruncWork<R>& w, R* Uout, Ix uo_r,
                              Ix uo_c, R* Cout, Ix co_r, Ix co_c) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (K == m) {
    // Nothing is cut: any orthonormal basis of R^m works; take the identity.
    for (int e = tid; e < m * m; e += blockDim.x) {
      const int i = e / m, k = e % m;
      Uout[ixoff(uo_r, i) + ixoff(uo_c, k)] = i == k ? R(1) : R(0);
    }
    for (int e = tid; e < m * n; e += blockDim.x) {
      const int k = e / n, j = e % n;
      Cout[ixoff(co_r, k) + ixoff(co_c, j)] = X[e];
    }
    __syncthreads();
    return;
  }
  PEPS_PHASE(0);
  const bool tall = m >= n;
  const int P = tall ? m : n, Q = tall ? n : m;
  const int ld = w.ldw;
  R* W = w.Wm;
  R* tauL = w.tau;
  R* tauR = w.tau + w.Qmax;
  R* red = w.red;
  bool tiled = false;
  if constexpr (sizeof(R) == 4) {
    if (P > 32 && P <= 128) {   // below 33 rows the shared-memory version is as fast
      // the reflectors go to global memory: shared memory then holds the
      // inverse-iteration workspace
      W = w.Wg;
      bidiag_tiles_f32(X, n, tall, P, Q, W, ld, w.t, w.tau, w.Qmax);
      tiled = true;
    }
  }
  if (!tiled) bidiag_shared<R>(X, m, n, tall, P, Q, W, ld, w.t, w.tau, w.Qmax, w.wv, red);
  PEPS_PHASE(1);
  // ---------------- Sturm sections for the K largest singular values
  const int n2 = 2 * Q;
  R tmax = R(0);
  for (int i = tid; i < n2 - 1; i += blockDim.x) tmax = fmax(tmax, fabs(w.t[i]));
  tmax = warp_max(tmax);
  if (lane == 0) red[8 + warp] = tmax;
  __syncthreads();
  tmax = R(0);
  for (int i = 0; i < kWarps; ++i) tmax = fmax(tmax, red[8 + i]);
  if constexpr (sizeof(R) == 4) {
    // the squares in shared memory (wv is free here) where they fit
    R* t2 = n2 <= kMaxT2Shared ? w.wv : w.t2;
    for (int i = tid; i < n2 - 1; i += blockDim.x) t2[i] = w.t[i] * w.t[i];
    __syncthreads();
    const R bound = R(2) * tmax * (R(1) + R(4) * Eps<R>::eps) + Eps<R>::tiny;
    const R pivmin = Eps<R>::tiny * R(1024) * fmax(R(1), tmax * tmax);
    section_f32(t2, n2, K, bound, pivmin, w.lam);
  } else {
    const int e2 = pow2_exponent(tmax);
    const R down = pow2<R>(-e2);
    float* t2f = reinterpret_cast<float*>(w.wv);       // >= 512 floats
    float* lamf = reinterpret_cast<float*>(red + 24);
    for (int i = tid; i < n2 - 1; i += blockDim.x) {
      const R v = w.t[i] * down;
      w.t2[i] = v * v;
      t2f[i] = (float)(v * v);
    }
    __syncthreads();
    section_f32(t2f, n2, K, 4.001f, Eps<float>::tiny * 4096.f, lamf);
    __syncthreads();
    if (warp < 4) refine_values_f64(tid, K <= 8 ? 16 : K <= 16 ? 8 : 4, w.t2, n2, K, lamf, pow2<R>(e2), w.lam);
  }
  __syncthreads();
  PEPS_PHASE(2);
  // ---------------- inverse iteration, one thread per vector
  const R pivtiny = Eps<R>::eps * fmax(tmax, Eps<R>::tiny * R(1e10));
  R* Ub = w.Ubs;
  {
    // On the register-tiled path the shared region (matrix, Ub, Uk) is free: the
    // workspace goes there when it fits, t to wv.  The vectors are then read
    // into registers before Ub, which it may overlap, is written.
    const bool in_smem = tiled && 4 * n2 * K <= w.gsm_reals && n2 <= kMaxT2Shared;
    R* wsR = in_smem ? w.gsm : inv_align(w.lu);
    const R* tv = w.t;
    if (in_smem || n2 <= w.Qmax * w.Kmax) {
      R* ts = in_smem ? w.wv : Ub;
      for (int i = tid; i < n2 - 1; i += blockDim.x) ts[i] = w.t[i];
      tv = ts;
    }
    __syncthreads();
    if (tid < K) red[tid] = inverse_iteration(tv, n2, w.lam[tid], pivtiny, wsR, K, tid, (unsigned)(tid + 1));
    __syncthreads();
    PEPS_PHASE(3);
    // u-parts (odd positions) for a tall matrix, v-parts (even) for a wide one, scaled
    constexpr int kPer = 16;   // 128 x 32 entries at most on the tiled path
    auto entry = [&](int e) {
      const int i = e / K, k = e % K;
      return wsR[((2 * i + (tall ? 1 : 0)) * K + k) * 4 + 3] * red[k];
    };
    if (in_smem) {
      R v[kPer];
#pragma unroll
      for (int q = 0; q < kPer; ++q)
        if (tid + q * kThreads < Q * K) v[q] = entry(tid + q * kThreads);
      __syncthreads();
#pragma unroll
      for (int q = 0; q < kPer; ++q)
        if (tid + q * kThreads < Q * K) Ub[tid + q * kThreads] = v[q];
    } else {
      for (int e = tid; e < Q * K; e += blockDim.x) Ub[e] = entry(e);
    }
  }
  __syncthreads();
  // ---------------- orthonormal basis of the kept vectors: CholeskyQR2
  // (G = Ub^T Ub = R^T R, Ub <- Ub R^-1, twice; Fukaya et al. 2014).  Each
  // pass costs three barriers.  If a direction of Ub is below 1e-3 of its
  // norm (a cluster or a zero singular value), Gram-Schmidt with replacement
  // of degenerate directions (below) takes over from the current Ub.
  const bool need_cgs = cholesky_qr2<R>(Ub, w.Uks, Q, K);
  // ---------------- Gram-Schmidt with re-orthogonalisation (CGS2), fallback
  if (need_cgs) gram_schmidt<R>(Ub, Q, K, red);
  PEPS_PHASE(4);
  // ---------------- back-transformation by the stored reflectors, in blocks
  // U = H_0 H_1 ... H_{nref-1} [Ub; 0].  A block of nb consecutive reflectors
  // is applied at once as U -= V (T (V^T U)), with V = [v_j0 .. v_j0+nb-1] and
  // T the upper triangular factor of the compact WY form (Schreiber & Van
  // Loan 1989), built by the forward recurrence T_kk = tau_k,
  // T_{0:k,k} = -tau_k T_{0:k,0:k} (V_{:,0:k}^T v_k).  Reflector j has its
  // implicit 1 at row j (tall block) or j+1 (wide block) and scale * stored
  // entries below it.  V is written out per block into the Ub buffer, which
  // is free once Ub has been copied to Uk (nb <= K keeps it in bounds).
  R* Uk = w.Uks;
  const int rowsU = tall ? P : Q;
  for (int e = tid; e < rowsU * K; e += blockDim.x) {
    const int i = e / K, k = e % K;
    Uk[e] = i < Q ? Ub[i * K + k] : R(0);
  }
  __syncthreads();
  {
    constexpr int NBMAX = 8, KMAX = 32;   // reflectors per block; K <= 32
    __shared__ R bt_g[NBMAX][NBMAX], bt_t[NBMAX][NBMAX], bt_w1[NBMAX][KMAX + NBMAX], bt_w2[NBMAX][KMAX];
    const R* taus = tall ? tauL : tauR;
    const R* scs = tall ? w.tau + 2 * w.Qmax : w.tau + 3 * w.Qmax;
    if constexpr (sizeof(R) == 4) {
      // Register-tiled path: the reflectors, their factors and scales move
      // from global memory to shared memory once (the truncation matrix
      // buffer is free after the inverse iteration), all loads of a round in
      // flight together, instead of one exposed load latency per block below.
      __shared__ float bt_tau[128], bt_scs[128];
      if (tiled && w.wm_shared && Q <= 128) {
        R* Ws = w.Wm;
        const int tot = P * ld;
        for (int e0 = 0; e0 < tot; e0 += 8 * kThreads) {
          R v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int e = e0 + u * kThreads + tid;
            v[u] = e < tot ? W[e] : R(0);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int e = e0 + u * kThreads + tid;
            if (e < tot) Ws[e] = v[u];
          }
        }
        for (int e = tid; e < Q; e += kThreads) {
          bt_tau[e] = taus[e];
          bt_scs[e] = scs[e];
        }
        W = Ws;
        taus = bt_tau;
        scs = bt_scs;
        __syncthreads();
      }
    }
    const int nref = tall ? Q : Q - 1;
    bool applied = false;
    if constexpr (sizeof(R) == 4) {
      if (tiled && w.one_by_one && Q <= 128 && rowsU <= 128 && K <= 2 * kWarps) {
        // Reflectors in shared memory, at most 128 rows and 16 columns: one
        // column of U per half-warp (lane l holds rows l, l + 16, ...), the
        // reflectors applied one at a time, last first.  Each is a dot
        // product over the half-warp (shuffles) and an axpy; columns are
        // independent, so there is no barrier.  A reflector is zero above its
        // first row, so the row groups above it are left out (half of the
        // work): apply_reflectors takes the reflectors whose first row is in
        // one group of sixteen.
        apply_all_reflectors(reinterpret_cast<const float*>(W), ld, tall, rowsU, nref, K,
                             reinterpret_cast<const float*>(taus), reinterpret_cast<const float*>(scs),
                             reinterpret_cast<float*>(Uk));
        __syncthreads();
        applied = true;
      }
    }
    const int NB = K < NBMAX ? K : NBMAX;
    R* Vs = Ub;   // [rowsU][nb]
    for (int j0 = (nref > 0 && !applied) ? ((nref - 1) / NB) * NB : -1; j0 >= 0; j0 -= NB) {
      const int nb = min(NB, nref - j0);
      const int p0 = tall ? j0 : j0 + 1;
      for (int e = tid; e < (rowsU - p0) * nb; e += blockDim.x) {
        const int i = p0 + e / nb, aa = e % nb, j = j0 + aa, pv = tall ? j : j + 1;
        Vs[i * nb + aa] = i < pv ? R(0) : (i == pv ? R(1) : scs[j] * (tall ? W[i * ld + j] : W[j * ld + i]));
      }
      __syncthreads();
      // [W1 | G] = V^T [U | V] (nb x (K + nb)); two threads per dot product
      const int ncol = K + nb, nd = nb * ncol;
      for (int d0 = 0; d0 < nd; d0 += kThreads / 2) {
        const int d = d0 + (tid >> 1), part = tid & 1;
        R sacc = R(0);
        if (d < nd) {
          const int aa = d / ncol, c = d % ncol;
          const int pa = p0 + aa;   // first non-zero row of v_aa
          if (c < K) {
            for (int i = pa + part; i < rowsU; i += 2) sacc += Vs[i * nb + aa] * Uk[i * K + c];
          } else {
            for (int i = pa + part; i < rowsU; i += 2) sacc += Vs[i * nb + aa] * Vs[i * nb + (c - K)];
          }
        }
        sacc += __shfl_xor_sync(0xffffffffu, sacc, 1);
        if (part == 0 && d < nd) {
          const int aa = d / ncol, c = d % ncol;
          if (c < K) bt_w1[aa][c] = sacc;
          else bt_g[aa][c - K] = sacc;
        }
      }
      __syncthreads();
      // T, one thread per row: T[i][i] = tau_i, T[i][k] = -tau_k sum_{m=i}^{k-1} T[i][m] G[m][k]
      if (tid < nb) {
        const int i = tid;
        for (int k = 0; k < nb; ++k) bt_t[i][k] = R(0);
        bt_t[i][i] = taus[j0 + i];
        for (int k = i + 1; k < nb; ++k) {
          R acc = R(0);
          for (int m = i; m < k; ++m) acc += bt_t[i][m] * bt_g[m][k];
          bt_t[i][k] = -taus[j0 + k] * acc;
        }
      }
      __syncthreads();
      // W2 = T W1
      for (int e = tid; e < nb * K; e += blockDim.x) {
        const int aa = e / K, cc = e % K;
        R acc = R(0);
        for (int bb = aa; bb < nb; ++bb) acc += bt_t[aa][bb] * bt_w1[bb][cc];
        bt_w2[aa][cc] = acc;
      }
      __syncthreads();
      // U -= V W2 on rows p0.. (V is zero above its first pivot)
      for (int e = tid; e < (rowsU - p0) * K; e += blockDim.x) {
        const int i = p0 + e / K, cc = e % K;
        R acc = R(0);
        for (int aa = 0; aa < nb; ++aa) acc += Vs[i * nb + aa] * bt_w2[aa][cc];
        Uk[i * K + cc] -= acc;
      }
      __syncthreads();
    }
  }
  PEPS_PHASE(5);
  // ---------------- outputs, after one Newton-Schulz step towards the
  // nearest orthonormal basis (Higham, Functions of Matrices, Sec. 8.3):
  // U <- U (3/2 I - 1/2 U^T U).  In FP32 the reflectors leave U^T U - I at
  // ~1e-6, and each cut then applies a slightly wrong projector; the step
  // squares that defect.  The K x K factor goes into the free Ub buffer.
  //
  // FP32: U^T U and the carry U^T X are compensated dot products.  The kept
  // vectors are localised, so a plain FP32 sum drops most of their small
  // terms against the running sum, and always with the same sign: over the
  // 240 cuts of a 16x16 sweep that biased ln|psi| by ~3e-5, ten times the
  // error of an FP32 LAPACK SVD sweep.  The step is applied as
  // U + U (-1/2 (U^T U - I)), so its small correction is not rounded
  // against 1.
  if constexpr (sizeof(R) == 4) {
    finish_f32(X, m, n, K, Ub, Uk, w.Uk, Uout, uo_r, uo_c, Cout, co_r, co_c);
  } else {
    R* Mns = Ub;
    for (int e = tid; e < K * K; e += blockDim.x) {
      const int a = e / K, b = e % K;
      R sacc = R(0);
      for (int i = 0; i < m; ++i) sacc += Uk[i * K + a] * Uk[i * K + b];
      Mns[e] = (a == b ? R(1.5) : R(0)) - R(0.5) * sacc;
    }
    __syncthreads();
    for (int e = tid; e < m * K; e += blockDim.x) {
      const int i = e / K, k = e % K;
      R v = R(0);
      for (int a = 0; a < K; ++a) v += Uk[i * K + a] * Mns[a * K + k];
      Uout[ixoff(uo_r, i) + ixoff(uo_c, k)] = v;
      w.Uk[e] = v;
    }
    __syncthreads();
    for (int e = tid; e < m * K; e += blockDim.x) Uk[e] = w.Uk[e];
    __syncthreads();
    // C' = U_K^T X: an item is a column and four rows (a full tile of the GEMM
    // engine would spend most of its FP64 instructions on padding: K is 6 to 32)
    constexpr int CH = 4, XB = 8;
    const int nchunk = (K + CH - 1) / CH;
    for (int item = tid; item < n * nchunk; item += blockDim.x) {
      const int j = item % n, a0 = (item / n) * CH;
      R sacc[CH];
#pragma unroll
      for (int q = 0; q < CH; ++q) sacc[q] = R(0);
      for (int ib = 0; ib < m; ib += XB) {
        R xb[XB];
#pragma unroll
        for (int u = 0; u < XB; ++u) xb[u] = ib + u < m ? X[(ib + u) * n + j] : R(0);
#pragma unroll
        for (int u = 0; u < XB; ++u)
          if (ib + u < m) {
#pragma unroll
            for (int q = 0; q < CH; ++q)
              if (a0 + q < K) sacc[q] = fma(Uk[(ib + u) * K + a0 + q], xb[u], sacc[q]);
          }
      }
#pragma unroll
      for (int q = 0; q < CH; ++q)
        if (a0 + q < K) Cout[ixoff(co_r, a0 + q) + ixoff(co_c, j)] = sacc[q];
    }
    __syncthreads();
  }
  PEPS_PHASE(6);
}

}  // namespace peps

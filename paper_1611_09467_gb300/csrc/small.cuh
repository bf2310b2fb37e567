// Zip-up row absorption and truncation by one warp, for boundary MPS whose
// cut blocks are at most 32 x 32 (Dc D <= 32, 2 <= D <= 6).
//
// The same arithmetic as absorb_row / cta_topk_left on their shared-memory
// path: in FP32 every sum is taken over the same terms in the same tree as
// the 256-thread version takes it (its thread partition is spelled out in the
// comments below), so results are equal bit for bit.  In FP64 the singular
// values and vectors come from the division-free Sturm counts and the
// one-reciprocal inverse iteration of sturm64.cuh, as on the 256-thread path.
//
// Why one warp: a block of at most 32 x 32 gives 256 threads one to four
// entries each between two barriers, so the CTA version spends its time in
// barriers and exposed latencies (3100 kcycles of an SM per 8x8 D = 4 Dc = 8
// sweep in FP32, four barriers per Householder column).  A warp holds a row
// or a column per lane, keeps the whole column step in registers, needs no
// barrier, and ten sweeps share an SM (20 KB of shared memory each in FP32).
#pragma once

#include "device.cuh"
#include "kernels.h"
#include "sturm64.cuh"

namespace peps {
namespace small {

constexpr int kP = 32;   // largest block dimension

// The models this path takes: every cut block fits 32 x 32 and the per-warp
// buffers stay small (D <= 6 bounds the site tensor, D >= 2 bounds Dc by 16).
PEPS_HD bool fits(const Geometry& g) { return g.fit == 0 && g.D >= 2 && g.D <= 6 && g.D * g.Dc <= kP; }

PEPS_HD int up4(int x) { return (x + 3) / 4 * 4; }

// Per-warp shared memory in reals.  Region A holds the carry C, the MPS
// tensor M, the site tensor T and Y while X is formed; then the inverse
// iteration's vectors, then the compact-WY factors; at the end of a cut the
// new carry is written at its start.
struct Layout {
  int C, M, T, Y, endA, X, W, ldw, Ub, Uk, t, t2, tau, lam, va, vb, total;
};
PEPS_HD Layout layout(int D, int Dc) {
  const int P = D * Dc;
  Layout l;
  l.C = 0;
  l.M = up4(P * Dc);
  l.T = l.M + up4(P * Dc);
  l.Y = l.T + up4(D * D * D * D);
  const int zip = l.Y + up4(P * P), inv = 4 * 2 * P * Dc, wy = 64 + 64 + 16 * 8;
  l.endA = up4(zip > inv ? (zip > wy ? zip : wy) : (inv > wy ? inv : wy));
  l.X = l.endA;
  l.W = l.X + up4(P * P);
  l.ldw = P | 1;
  l.Ub = l.W + up4(P * l.ldw);
  l.Uk = l.Ub + up4(P * (Dc > 8 ? Dc : 8));   // also the 8-wide V of the back-transformation
  l.t = l.Uk + up4(P * Dc);
  l.t2 = l.t + up4(2 * P);
  l.tau = l.t2 + up4(2 * P);
  l.lam = l.tau + 4 * kP;
  l.va = l.lam + 16;
  l.vb = l.va + kP;
  l.total = l.vb + kP;
  return l;
}

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

// A rounded product: sums over products below must not be contracted.
__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }

// ---------------------------------------------------------------- sums
// The sum over 256 threads of block_sum, from one warp: lane l holds in v[w]
// the value of thread 32 w + l.  Each warp's butterfly is done as a
// reduce-scatter over the eight values (the same pairs are added), then the
// eight totals are added in warp order.
template <typename R>
__device__ __forceinline__ R sum256(const R (&v)[8]) {
  const int l = lane_id();
  R a[4], b[2], c;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const R snd = (l & 16) ? v[i] : v[i + 4], kp = (l & 16) ? v[i + 4] : v[i];
    a[i] = kp + __shfl_xor_sync(0xffffffffu, snd, 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const R snd = (l & 8) ? a[i] : a[i + 2], kp = (l & 8) ? a[i + 2] : a[i];
    b[i] = kp + __shfl_xor_sync(0xffffffffu, snd, 8);
  }
  {
    const R snd = (l & 4) ? b[0] : b[1], kp = (l & 4) ? b[1] : b[0];
    c = kp + __shfl_xor_sync(0xffffffffu, snd, 4);
  }
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  R s = R(0);
#pragma unroll
  for (int w = 0; w < 8; ++w)   // warp w's total sits in the lanes whose bits 4, 3, 2 spell w
    s += __shfl_sync(0xffffffffu, c, ((w >> 2) << 4) | (((w >> 1) & 1) << 3) | ((w & 1) << 2));
  return s;
}

// Frobenius norm squared in FP64 and dot product, partitioned as by 256 threads.
template <typename R>
__device__ double norm2_256(const R* x, int n) {
  double v[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    double s = 0.0;
    for (int e = 32 * w + lane_id(); e < n; e += 256) s += (double)x[e] * (double)x[e];
    v[w] = s;
  }
  return sum256(v);
}

// ---------------------------------------------------------------- GEMM
// C[ixoff(ro, i) + ixoff(co, j)] = sum_k A[k][i] B[k][j], both k-major in shared memory,
// each output one chain of fused multiply-adds over k (as gemm_wk).
template <typename R, int TM, int TN, bool VEC>
__device__ __noinline__ void wgemm_t(int M, int N, int K, const R* A, const R* B, R* C, Ix ro, Ix co) {
  const int tn = (N + TN - 1) / TN, nt = ((M + TM - 1) / TM) * tn;
  for (int t = lane_id(); t < nt; t += 32) {
    const int i0 = (t / tn) * TM, j0 = (t % tn) * TN;
    R acc[TM][TN];
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int b = 0; b < TN; ++b) acc[a][b] = R(0);
    int ia[TM], jb[TN];
#pragma unroll
    for (int a = 0; a < TM; ++a) ia[a] = min(i0 + a, M - 1);
#pragma unroll
    for (int b = 0; b < TN; ++b) jb[b] = min(j0 + b, N - 1);
#pragma unroll 2
    for (int k = 0; k < K; ++k) {
      R av[TM], bv[TN];
      if constexpr (VEC && sizeof(R) == 4) {
        const float4 x = *reinterpret_cast<const float4*>(A + k * M + i0);
        const float4 y = *reinterpret_cast<const float4*>(B + k * N + j0);
        av[0] = x.x; av[1] = x.y; av[2] = x.z; av[3] = x.w;
        bv[0] = y.x; bv[1] = y.y; bv[2] = y.z; bv[3] = y.w;
      } else if constexpr (VEC) {
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
          const double2 x = *reinterpret_cast<const double2*>(A + k * M + i0 + q);
          const double2 y = *reinterpret_cast<const double2*>(B + k * N + j0 + q);
          av[q] = x.x; av[q + 1] = x.y;
          bv[q] = y.x; bv[q + 1] = y.y;
        }
      } else {
#pragma unroll
        for (int a = 0; a < TM; ++a) av[a] = A[k * M + ia[a]];
#pragma unroll
        for (int b = 0; b < TN; ++b) bv[b] = B[k * N + jb[b]];
      }
#pragma unroll
      for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TN; ++b) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
    }
    int oc[TN];
#pragma unroll
    for (int b = 0; b < TN; ++b) oc[b] = ixoff(co, jb[b]);
#pragma unroll
    for (int a = 0; a < TM; ++a) {
      if (VEC || i0 + a < M) {
        const int orow = ixoff(ro, ia[a]);
#pragma unroll
        for (int b = 0; b < TN; ++b)
          if (VEC || j0 + b < N) C[orow + oc[b]] = acc[a][b];
      }
    }
  }
  __syncwarp();
}

// Tile shape: 4 x 4 once that still gives every lane a tile, smaller below
// (a 2 x 2 or single-output tile keeps the lanes busy on the tiny products of
// D = 2, 3).
template <typename R>
__device__ __forceinline__ void wgemm(int M, int N, int K, const R* A, const R* B, R* C, Ix ro, Ix co) {
  if (M * N >= 512) {
    if (((M | N) & 3) == 0) wgemm_t<R, 4, 4, true>(M, N, K, A, B, C, ro, co);
    else wgemm_t<R, 4, 4, false>(M, N, K, A, B, C, ro, co);
  } else if (M * N >= 96) {
    wgemm_t<R, 2, 2, false>(M, N, K, A, B, C, ro, co);
  } else {
    wgemm_t<R, 1, 1, false>(M, N, K, A, B, C, ro, co);
  }
}

// ------------------------------------------------------- bidiagonalisation
// Sum over k < n <= 8 NB of x[k] v[k] (both zero past n), FP32: the tree of the
// 256-thread version.  `cnt` outputs shared the CTA, so tpc = the largest
// power of two <= min(32, 256 / cnt) threads took one output; thread g added
// the terms k = g, g + tpc, .. (four of them as (0 + 1) + (2 + 3), fewer as a
// chain), and the threads were added by a butterfly over tpc.  v in shared
// memory, 16-byte aligned.
template <int NB>
__device__ __forceinline__ float dot_tree(const float (&x)[8 * NB], const float* v, int n, int cnt) {
  float y[8 * NB];
#pragma unroll
  for (int k = 0; k < 8 * NB; k += 4) {
    const float4 q = *reinterpret_cast<const float4*>(v + k);
    y[k] = q.x; y[k + 1] = q.y; y[k + 2] = q.z; y[k + 3] = q.w;
  }
  if (cnt > 16) {
    float p[8];
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      float s = mulr(x[g], y[g]);
      if constexpr (NB == 4) {
        const float s1 = mulr(x[g + 8], y[g + 8]), s2 = mulr(x[g + 16], y[g + 16]), s3 = mulr(x[g + 24], y[g + 24]);
        const float chain = fmaf(x[g + 16], y[g + 16], fmaf(x[g + 8], y[g + 8], s));
        s = g + 24 < n ? (s + s1) + (s2 + s3) : chain;
      } else {
#pragma unroll
        for (int q = 1; q < NB; ++q) s = fmaf(x[g + 8 * q], y[g + 8 * q], s);
      }
      p[g] = s;
    }
    return ((p[0] + p[4]) + (p[2] + p[6])) + ((p[1] + p[5]) + (p[3] + p[7]));
  }
  // tpc = 16 (cnt > 8): terms k and k + 16 chained; tpc = 32: every term apart
  constexpr int S = NB == 1 ? 8 : NB == 2 ? 16 : 32;
  float p[S];
#pragma unroll
  for (int g = 0; g < S; ++g) p[g] = g < 8 * NB ? mulr(x[g < 8 * NB ? g : 0], y[g < 8 * NB ? g : 0]) : 0.f;
  if constexpr (S == 32) {
#pragma unroll
    for (int g = 0; g < 16; ++g) {
      const int h = g + 16 < 8 * NB ? g + 16 : 0;
      p[g] = cnt > 8 ? (g + 16 < 8 * NB ? fmaf(x[h], y[h], p[g]) : p[g]) : p[g] + p[g + 16];
    }
  }
#pragma unroll
  for (int o = S >= 16 ? 8 : 4; o > 0; o >>= 1)
#pragma unroll
    for (int g = 0; g < o; ++g) p[g] = p[g] + p[g + o];
  return p[0];
}

// The same in FP64, where no other code fixes the order.
template <int NB>
__device__ __forceinline__ double dot_tree(const double (&x)[8 * NB], const double* v, int, int) {
  double s0 = 0.0, s1 = 0.0;
#pragma unroll
  for (int k = 0; k < 8 * NB; k += 2) {
    const double2 q = *reinterpret_cast<const double2*>(v + k);
    s0 = fma(x[k], q.x, s0);
    s1 = fma(x[k + 1], q.y, s1);
  }
  return s0 + s1;
}

// One reflector applied to one column (or row) per lane: the lane's entries
// x0 (at p[0]) and p[(k + 1) st], k < n, are read once, updated and stored.
// vr: the reflector's unscaled entries (zero past n), vs: scaled by sc.
// Returns the updated x0.  NB = ceil(n / 8), so that a short reflector does
// not issue the predicated-off work of a long one.
template <typename R, int NB>
__device__ __forceinline__ R reflect(R* p, int st, int n, int cnt, bool act, R tau, R sc, const R* vr, const R* vs) {
  R x[8 * NB];
  const R x0 = p[0];
#pragma unroll
  for (int k = 0; k < 8 * NB; ++k) x[k] = (k < 8 * (NB - 1) || k < n) ? p[(k + 1) * st] : R(0);
  R w;
  if constexpr (sizeof(R) == 4) w = tau * fma(sc, dot_tree<NB>(x, vr, n, cnt), x0);
  else w = tau * (x0 + dot_tree<NB>(x, vs, n, cnt));
  const R y0 = x0 - w;
  if (act) {
    p[0] = y0;
#pragma unroll
    for (int k = 0; k < 8 * NB; k += 2) {
      R v0, v1;
      if constexpr (sizeof(R) == 4) {
        const float2 q = *reinterpret_cast<const float2*>(vs + k);
        v0 = q.x; v1 = q.y;
      } else {
        const double2 q = *reinterpret_cast<const double2*>(vs + k);
        v0 = q.x; v1 = q.y;
      }
      if (k < 8 * (NB - 1) || k < n) p[(k + 1) * st] = fma(-w, v0, x[k]);
      if (k + 1 < 8 * (NB - 1) || k + 1 < n) p[(k + 2) * st] = fma(-w, v1, x[k + 1]);
    }
  }
  return y0;
}

template <typename R>
__device__ __forceinline__ R reflect_any(R* p, int st, int n, int cnt, bool act, R tau, R sc, const R* vr, const R* vs) {
  if (n > 16) {
    if (n > 24) return reflect<R, 4>(p, st, n, cnt, act, tau, sc, vr, vs);
    return reflect<R, 3>(p, st, n, cnt, act, tau, sc, vr, vs);
  }
  if (n > 8) return reflect<R, 2>(p, st, n, cnt, act, tau, sc, vr, vs);
  if (n > 0) return reflect<R, 1>(p, st, n, cnt, act, tau, sc, vr, vs);
  // no entries below: w = tau x0
  const R y0 = p[0] - (sizeof(R) == 4 ? tau * fma(sc, R(0), p[0]) : tau * p[0]);
  if (act) p[0] = y0;
  return y0;
}

// Householder bidiagonalisation of W (P x Q, P >= Q, leading dimension ld) in
// shared memory.  A left step gives each lane one column, a right step one row
// (reflect); the reflector's entries are broadcast from a contiguous copy.
// Reflectors stay unscaled in W with their scales in tau[2 kP ..], tau[3 kP ..].
// va, vb: kP reals each.
template <typename R>
__device__ __noinline__ void bidiag(R* W, int ld, int P, int Q, R* t, R* tau, R* va, R* vb) {
  const int l = lane_id();
  R colnorm;
  {
    const R x = 1 + l < P ? W[(1 + l) * ld] : R(0);
    colnorm = warp_sum<R>(mulr(x, x));
  }
#pragma unroll 1
  for (int j = 0; j < Q; ++j) {
    const int nr = P - j - 1, nc = Q - j - 1;   // rows below, columns right
    R tl, sl, beta;
    householder(W[j * ld + j], colnorm, tl, sl, beta);
    if (l == 0) {
      t[2 * j] = beta;
      tau[j] = tl;
      tau[2 * kP + j] = sl;
    }
    if (nc == 0) break;
    const R xl = l < nr ? W[(j + 1 + l) * ld + j] : R(0);
    va[l] = xl;
    vb[l] = mulr(sl, xl);
    __syncwarp();
    // -- left reflector, lane = column j + 1 + l
    R* col = W + j * ld + j + 1 + (l < nc ? l : 0);
    R rowv = col[0];   // W[j][j + 1 + l] after the update
    if (tl != R(0)) rowv = reflect_any<R>(col, ld, nr, nc, l < nc, tl, sl, va, vb);
    // squared norm of row j beyond column j + 1; the 256-thread version's
    // lanes are shifted by one when there is no left update
    R rownorm;
    if (tl != R(0)) {
      rownorm = warp_sum<R>((l >= 1 && l < nc) ? mulr(rowv, rowv) : R(0));
    } else {
      const R x = __shfl_down_sync(0xffffffffu, rowv, 1);
      rownorm = warp_sum<R>(l + 1 < nc ? mulr(x, x) : R(0));
    }
    R tr, sr, br;
    householder(__shfl_sync(0xffffffffu, rowv, 0), rownorm, tr, sr, br);
    if (l == 0) {
      t[2 * j + 1] = br;
      tau[kP + j] = tr;
      tau[3 * kP + j] = sr;
    }
    __syncwarp();
    {
      const R u = __shfl_down_sync(0xffffffffu, rowv, 1);
      const R ul = l + 1 < nc ? u : R(0);
      va[l] = ul;
      vb[l] = mulr(sr, ul);
    }
    __syncwarp();
    // -- right reflector, lane = row j + 1 + l
    if (tr != R(0)) {
      const R y0 = reflect_any<R>(W + (j + 1 + (l < nr ? l : 0)) * ld + j + 1, 1, nc - 1, nr, l < nr, tr, sr, va, vb);
      // squared norm of column j + 1 below row j + 1: warp w of the 256-thread
      // version chained the rows l = w, w + 8, ..; the eight chains are added in order
      const R q1 = __shfl_down_sync(0xffffffffu, y0, 8), q2 = __shfl_down_sync(0xffffffffu, y0, 16),
              q3 = __shfl_down_sync(0xffffffffu, y0, 24);
      R cn = (l >= 1 && l < nr) ? mulr(y0, y0) : R(0);
      if (l + 8 < nr) cn = fma(q1, q1, cn);
      if (l + 16 < nr) cn = fma(q2, q2, cn);
      if (l + 24 < nr) cn = fma(q3, q3, cn);
      if constexpr (sizeof(R) == 4) {
        colnorm = R(0);
#pragma unroll
        for (int w = 0; w < 8; ++w) colnorm += __shfl_sync(0xffffffffu, cn, w);
      } else {
        colnorm = __shfl_sync(0xffffffffu, warp_sum<R>(cn, 8), 0);
      }
    } else {
      const R x = (l < nr - 1) ? W[(j + 2 + l) * ld + j + 1] : R(0);
      colnorm = warp_sum<R>(mulr(x, x));
    }
    __syncwarp();
  }
  __syncwarp();
}

// ------------------------------------------------------------- bisection
// FP32: the sixteen-section of cta_topk_left (16 points per value and step),
// K * 16 points spread over the lanes in NCH chunks so that each lane runs NCH
// independent Sturm recurrences.  In the first step all values share one
// interval, so its 16 points are counted once.
template <int NCH>
__device__ __noinline__ void bisect_f32(const float* t2, int n2, int K, float bound, float pivmin, float* lam) {
  constexpr int G = 16, NIT = 7;   // 17^7 >= 2^26
  const int l = lane_id(), gl = l & 15, half = l >> 4;
  float lo[NCH], hi[NCH];
  {
    const float step = (bound - 0.f) / float(G + 1);
    const float x = 0.f + step * float(gl + 1);
    float q = -x;
    if (fabsf(q) < pivmin) q = -pivmin;
    int cnt = q < 0.f ? 1 : 0;
    for (int i = 1; i < n2; ++i) cnt += sturm_count_step(q, x, t2[i - 1], pivmin);
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int idx = n2 - 1 - (2 * c + half);
      // both halves of the warp hold the counts of the same 16 points
      const unsigned bits = (__ballot_sync(0xffffffffu, cnt <= idx) >> (half * 16)) & 0xffffu;
      const int gs = __popc(bits) - 1;
      lo[c] = gs >= 0 ? 0.f + step * float(gs + 1) : 0.f;
      hi[c] = gs + 1 < G ? 0.f + step * float(gs + 2) : bound;
    }
  }
  for (int it = 1; it < NIT; ++it) {
    float x[NCH], q[NCH], step[NCH];
    int cnt[NCH];
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      step[c] = (hi[c] - lo[c]) / float(G + 1);
      x[c] = lo[c] + step[c] * float(gl + 1);
      q[c] = -x[c];
      if (fabsf(q[c]) < pivmin) q[c] = -pivmin;
      cnt[c] = q[c] < 0.f ? 1 : 0;
    }
    for (int i = 1; i < n2; ++i) {
      const float tv = t2[i - 1];
#pragma unroll
      for (int c = 0; c < NCH; ++c) cnt[c] += sturm_count_step(q[c], x[c], tv, pivmin);
    }
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int idx = n2 - 1 - (2 * c + half);
      const unsigned bits = (__ballot_sync(0xffffffffu, cnt[c] <= idx) >> (half * 16)) & 0xffffu;
      const int gs = __popc(bits) - 1;
      const float nlo = gs >= 0 ? lo[c] + step[c] * float(gs + 1) : lo[c];
      const float nhi = gs + 1 < G ? lo[c] + step[c] * float(gs + 2) : hi[c];
      lo[c] = nlo;
      hi[c] = nhi;
    }
  }
#pragma unroll
  for (int c = 0; c < NCH; ++c)
    if (gl == 0 && 2 * c + half < K) lam[2 * c + half] = 0.5f * (lo[c] + hi[c]);
}

// ------------------------------------------------------------- truncation
// Singular values of the bidiagonal (t: 2 Q - 1 off-diagonals of the
// Golub-Kahan form) into lam, the K largest; returns their largest entry.
template <typename R>
__device__ R values(const R* t, R* t2, int Q, int K, R* lam, R* scratch) {
  const int l = lane_id(), n2 = 2 * Q;
  R tmax = R(0);
  for (int i = l; i < n2 - 1; i += 32) tmax = fmax(tmax, fabs(t[i]));
  tmax = warp_max(tmax);
  float* t2f;
  float* lamf;
  float boundf, pivf;
  int e = 0;
  if constexpr (sizeof(R) == 4) {
    for (int i = l; i < n2 - 1; i += 32) t2[i] = t[i] * t[i];
    t2f = t2;
    lamf = lam;
    boundf = R(2) * tmax * (R(1) + R(4) * Eps<R>::eps) + Eps<R>::tiny;
    pivf = Eps<R>::tiny * R(1024) * fmax(R(1), tmax * tmax);
  } else {
    e = pow2_exponent(tmax);
    const R sc = pow2<R>(-e);
    t2f = reinterpret_cast<float*>(scratch);
    lamf = t2f + 2 * kP;
    for (int i = l; i < n2 - 1; i += 32) {
      const R v = t[i] * sc;
      t2[i] = v * v;
      t2f[i] = (float)(v * v);
    }
    boundf = 4.001f;
    pivf = Eps<float>::tiny * 4096.f;
  }
  __syncwarp();
  if (K <= 2) bisect_f32<1>(t2f, n2, K, boundf, pivf, lamf);
  else if (K <= 4) bisect_f32<2>(t2f, n2, K, boundf, pivf, lamf);
  else if (K <= 6) bisect_f32<3>(t2f, n2, K, boundf, pivf, lamf);
  else if (K <= 8) bisect_f32<4>(t2f, n2, K, boundf, pivf, lamf);
  else bisect_f32<8>(t2f, n2, K, boundf, pivf, lamf);
  __syncwarp();
  if constexpr (sizeof(R) == 8) {
    refine_values_f64(l, K <= 2 ? 16 : K <= 4 ? 8 : K <= 8 ? 4 : 2, t2, n2, K, lamf, pow2<R>(e), lam);
    __syncwarp();
  }
  return tmax;
}

// Orthonormal basis of the columns of Ub (Q x K, row-major): CholeskyQR2 with
// cta_topk_left's arithmetic and its Gram-Schmidt fallback.  G: K x K.
template <typename R>
__device__ __noinline__ void orthonormalise(R* Ub, R* G, int Q, int K) {
  const int l = lane_id();
  bool need_cgs = false;
  for (int pass = 0; pass < 2 && !need_cgs; ++pass) {
    for (int e = l; e < K * K; e += 32) {
      const int a = e / K, b = e % K;
      if (b < a) continue;
      R s = R(0);
#pragma unroll 8
      for (int i = 0; i < Q; ++i) s = fma(Ub[i * K + a], Ub[i * K + b], s);
      G[e] = s;
    }
    __syncwarp();
    const R d0 = l < K ? G[l * K + l] : R(0);
    for (int j = 0; j < K; ++j) {
      const R d = G[j * K + j];
      const R dj0 = __shfl_sync(0xffffffffu, d0, j);
      if (!(d > R(1e-6) * dj0) || !(dj0 > R(0))) {
        need_cgs = true;
        break;
      }
      R r;
      if constexpr (sizeof(R) == 4) {
        r = dsqrt(d);
        __syncwarp();
        if (l > j && l < K) G[j * K + l] /= r;
      } else {   // the diagonal holds 1 / r
        r = quick_rsqrt(d);
        __syncwarp();
        if (l > j && l < K) G[j * K + l] *= r;
      }
      __syncwarp();
      if (l == j) G[j * K + j] = r;
      if (l > j && l < K) {
        const R gjl = G[j * K + l];
        for (int m0 = j + 1; m0 <= l; m0 += 4) {
          R x[4];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (m0 + q <= l) x[q] = fma(-G[j * K + m0 + q], gjl, G[(m0 + q) * K + l]);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (m0 + q <= l) G[(m0 + q) * K + l] = x[q];
        }
      }
      __syncwarp();
    }
    __syncwarp();
    if (need_cgs) break;
    if (l < Q) {
      R u[16];
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        if (c >= K) break;
        R x = Ub[l * K + c];
#pragma unroll
        for (int k = 0; k < c; ++k) x = fma(-u[k], G[k * K + c], x);
        u[c] = sizeof(R) == 4 ? x / G[c * K + c] : x * G[c * K + c];
        Ub[l * K + c] = u[c];
      }
    }
    __syncwarp();
  }
  for (int j = 0; j < K && need_cgs; ++j) {
    for (int attempt = 0; attempt <= Q; ++attempt) {
      R v = l < Q ? Ub[l * K + j] : R(0);
      const R nrm0 = dsqrt(warp_sum<R>(mulr(v, v)));
      if (nrm0 > R(0)) v = v / nrm0;
      for (int pass = 0; pass < 2; ++pass) {
        R w = v;
        for (int p = 0; p < j; ++p) {
          const R up = l < Q ? Ub[l * K + p] : R(0);
          const R d = warp_sum<R>(mulr(up, v));
          w = fma(-d, up, w);
        }
        v = w;
      }
      const R nrm = dsqrt(warp_sum<R>(mulr(v, v)));
      if (nrm0 > R(0) && nrm > R(1e-3)) {
        if (l < Q) Ub[l * K + j] = v / nrm;
        __syncwarp();
        break;
      }
      const int q = (j + attempt) % Q;
      if (l < Q) Ub[l * K + j] = l == q ? R(1) : R(0);
      __syncwarp();
    }
  }
  __syncwarp();
}

// Eight consecutive reals from a 32-byte (FP32: 16-byte) aligned shared address.
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8(const double* p, double (&v)[8]) {
#pragma unroll
  for (int q = 0; q < 8; q += 2) {
    const double2 a = *reinterpret_cast<const double2*>(p + q);
    v[q] = a.x;
    v[q + 1] = a.y;
  }
}

// Uk <- H_0 H_1 .. Uk by the stored reflectors, eight at a time in compact WY
// form (blocks of min(K, 8), the rest of the eight zero); the even and odd
// rows of a dot product, counted from the reflector's first, are summed apart
// and added, as the two threads of the CTA version do.  A lane holds one column
// of [W1 | G] while rows of V are broadcast as 16-byte groups.  V: rows x 8,
// wy: the factors.
template <typename R>
__device__ __noinline__ void back_transform(const R* W, int ld, bool tall, int P, int Q, int K, const R* tau, R* Uk, R* V,
                                            R* wy) {
  const int l = lane_id();
  const int rows = tall ? P : Q, nref = tall ? Q : Q - 1, NB = K < 8 ? K : 8;
  const R* taus = tau + (tall ? 0 : kP);
  const R* scs = tau + (tall ? 2 : 3) * kP;
  R* g = wy;               // [8][8]: G[m][k], column k contiguous
  R* tt = wy + 64;         // [8][8]
  R* w2 = wy + 128;        // [16][8]: column, reflector
#pragma unroll 1
  for (int j0 = nref > 0 ? ((nref - 1) / NB) * NB : -1; j0 >= 0; j0 -= NB) {
    const int nb = min(NB, nref - j0), p0 = tall ? j0 : j0 + 1;
    R v[8];   // lane = row
#pragma unroll
    for (int aa = 0; aa < 8; ++aa) {
      const int j = j0 + aa, pv = tall ? j : j + 1;
      R x = R(0);
      if (aa < nb && l >= pv && l < rows) x = l == pv ? R(1) : mulr(scs[j], tall ? W[l * ld + j] : W[j * ld + l]);
      v[aa] = x;
    }
    if (l < rows) {
#pragma unroll
      for (int aa = 0; aa < 8; ++aa) V[l * 8 + aa] = v[aa];
    }
    __syncwarp();
    R w1[8];
    {
      const bool in = l < K + nb;
      const R* B = l < K ? Uk + l : V + (in ? l - K : 0);
      const int bs = l < K ? K : 8;
      R s0[8], s1[8];
#pragma unroll
      for (int aa = 0; aa < 8; ++aa) s0[aa] = s1[aa] = R(0);
      int i = p0;
#pragma unroll 2
      for (; i + 1 < rows; i += 2) {
        const R b0 = B[i * bs], b1 = B[(i + 1) * bs];
        R x[8], y[8];
        load8(V + i * 8, x);
        load8(V + (i + 1) * 8, y);
#pragma unroll
        for (int aa = 0; aa < 8; ++aa) {   // s0 takes the rows at even distance from the reflector's first
          if (aa & 1) {
            s1[aa] = fma(x[aa], b0, s1[aa]);
            s0[aa] = fma(y[aa], b1, s0[aa]);
          } else {
            s0[aa] = fma(x[aa], b0, s0[aa]);
            s1[aa] = fma(y[aa], b1, s1[aa]);
          }
        }
      }
      if (i < rows) {
        const R b0 = B[i * bs];
#pragma unroll
        for (int aa = 0; aa < 8; ++aa) {
          const R x = V[i * 8 + aa];
          if (aa & 1) s1[aa] = fma(x, b0, s1[aa]);
          else s0[aa] = fma(x, b0, s0[aa]);
        }
      }
#pragma unroll
      for (int aa = 0; aa < 8; ++aa) w1[aa] = s0[aa] + s1[aa];
      if (l >= K && in) {
#pragma unroll
        for (int aa = 0; aa < 8; ++aa) g[(l - K) * 8 + aa] = w1[aa];
      }
    }
    __syncwarp();
    // T, one lane per row i: T[i][i] = tau_i, T[i][k] = -tau_k sum_{m=i}^{k-1} T[i][m] G[m][k]
    if (l < 8) {
      R tr[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        R gk[8];
        load8(g + k * 8, gk);
        const R tk = k < nb ? taus[j0 + k] : R(0);
        R acc = R(0);
#pragma unroll
        for (int m = 0; m < k; ++m) acc = m >= l ? fma(tr[m], gk[m], acc) : acc;
        tr[k] = (k < nb && l < nb) ? (k == l ? tk : (k > l ? -tk * acc : R(0))) : R(0);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) tt[l * 8 + k] = tr[k];
    }
    __syncwarp();
    if (l < K) {   // W2 = T W1, lane = column
#pragma unroll
      for (int aa = 0; aa < 8; ++aa) {
        R tr[8];
        load8(tt + aa * 8, tr);
        R acc = R(0);
#pragma unroll
        for (int bb = aa; bb < 8; ++bb)
          if (bb < nb) acc = fma(tr[bb], w1[bb], acc);
        w2[l * 8 + aa] = acc;
      }
    }
    __syncwarp();
    if (l >= p0 && l < rows) {   // U -= V W2, lane = row
#pragma unroll 2
      for (int c = 0; c < K; ++c) {
        R w[8];
        load8(w2 + c * 8, w);
        R acc = R(0);
#pragma unroll
        for (int aa = 0; aa < 8; ++aa)
          if (aa < nb) acc = fma(v[aa], w[aa], acc);
        Uk[l * K + c] -= acc;
      }
    }
    __syncwarp();
  }
}

// CH rows of the carry for one column of X: C[q ck] = sum_i U[i K + q] X[i n], q < nq
// (FP32: compensated, two rows at once in packed instructions).
template <typename R, int CH, bool VEC>
__device__ __forceinline__ void carry_rows(const R* U, const R* X, int m, int n, int K, R* C, int ck, int nq) {
  if constexpr (sizeof(R) == 4) {
    float2 s[CH / 2], c[CH / 2];
#pragma unroll
    for (int q = 0; q < CH / 2; ++q) s[q] = c[q] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int i = 0; i < m; ++i) {
      const float x = X[i * n];
      float u[CH];
#pragma unroll
      for (int q = 0; q < CH; q += 4) {
        if constexpr (VEC) {
          const float4 a = *reinterpret_cast<const float4*>(U + i * K + q);
          u[q] = a.x; u[q + 1] = a.y; u[q + 2] = a.z; u[q + 3] = a.w;
        } else {
#pragma unroll
          for (int z = q; z < q + 4; ++z) u[z] = z < nq ? U[i * K + z] : 0.f;
        }
      }
#pragma unroll
      for (int q = 0; q < CH / 2; ++q)
        dot2_step2(make_float2(u[2 * q], u[2 * q + 1]), make_float2(x, x), s[q], c[q]);
    }
#pragma unroll
    for (int q = 0; q < CH / 2; ++q) {
      const float2 v = __fadd2_rn(s[q], c[q]);
      if (VEC || 2 * q < nq) C[2 * q * ck] = v.x;
      if (VEC || 2 * q + 1 < nq) C[(2 * q + 1) * ck] = v.y;
    }
  } else {
    R s[CH];
#pragma unroll
    for (int q = 0; q < CH; ++q) s[q] = R(0);
#pragma unroll 4
    for (int i = 0; i < m; ++i) {
      const R x = X[i * n];
#pragma unroll
      for (int q = 0; q < CH; ++q)
        if (VEC || q < nq) s[q] = fma(U[i * K + q], x, s[q]);
    }
#pragma unroll
    for (int q = 0; q < CH; ++q)
      if (VEC || q < nq) C[q * ck] = s[q];
  }
}

// One Newton-Schulz step on U (m x K), U to global memory through (uo, uk), and the
// carry C = U^T X (K x n) through (ck, cj); FP32 sums compensated, as cta_topk_left.
template <typename R>
__device__ __noinline__ void finish(R* U, R* M, const R* X, int m, int n, int K, R* Uout, Ix uo, int uk, R* C, int ck,
                                    Ix cj) {
  const int l = lane_id();
  for (int e = l; e < K * K; e += 32) {
    const int a = e / K, b = e % K;
    if constexpr (sizeof(R) == 4) {
      float s = 0.f, c = 0.f;
#pragma unroll 4
      for (int i = 0; i < m; ++i) dot2_step(U[i * K + a], U[i * K + b], s, c);
      M[e] = -0.5f * (a == b ? __fadd_rn(__fsub_rn(s, 1.f), c) : __fadd_rn(s, c));
    } else {
      R s = R(0);
#pragma unroll 4
      for (int i = 0; i < m; ++i) s = fma(U[i * K + a], U[i * K + b], s);
      M[e] = (a == b ? R(1.5) : R(0)) - R(0.5) * s;
    }
  }
  __syncwarp();
  // lane = row: the row is read before its new values are stored
  if (l < m) {
    R u[16];
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (k < K) u[k] = U[l * K + k];
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (k < K) {
        R corr = R(0);
#pragma unroll
        for (int a = 0; a < 16; ++a)
          if (a < K) corr = fma(u[a], M[a * K + k], corr);
        const R v = sizeof(R) == 4 ? u[k] + corr : corr;
        U[l * K + k] = v;
        Uout[ixoff(uo, l) + k * uk] = v;
      }
  }
  __syncwarp();
  if (l < n) {
    const int jo = ixoff(cj, l);
    int a0 = 0;
    if ((K & 3) == 0) {
      // rows of U as 16-byte groups, eight rows of C at a time, then four
      for (; a0 + 8 <= K; a0 += 8) carry_rows<R, 8, true>(U + a0, X + l, m, n, K, C + a0 * ck + jo, ck, 8);
      if (a0 < K) carry_rows<R, 4, true>(U + a0, X + l, m, n, K, C + a0 * ck + jo, ck, 4);
    } else {
      for (; a0 < K; a0 += 8) carry_rows<R, 8, false>(U + a0, X + l, m, n, K, C + a0 * ck + jo, ck, min(8, K - a0));
    }
  }
  __syncwarp();
}

// Dominant-K left singular subspace of X (m x n in shared memory): U_K to
// global memory at (row map uo, column stride uk), C = U_K^T X to shared memory
// (region A) at (row stride ck, column map cj).
template <typename R>
__device__ __noinline__ void topk_left(R* sm, const Layout& L, int m, int n, int K, R* Uout, Ix uo, int uk, int ck,
                                       Ix cj) {
  const int l = lane_id();
  R* X = sm + L.X;
  R* C = sm + L.C;
  if (K == m) {
    for (int e = l; e < m * m; e += 32) Uout[ixoff(uo, e / m) + (e % m) * uk] = e / m == e % m ? R(1) : R(0);
    for (int e = l; e < m * n; e += 32) C[(e / n) * ck + ixoff(cj, e % n)] = X[e];
    __syncwarp();
    return;
  }
  PEPS_PHASE(0);
  const bool tall = m >= n;
  const int P = tall ? m : n, Q = tall ? n : m, ld = L.ldw, n2 = 2 * Q;
  R* W = sm + L.W;
  for (int r = 0; r < m; ++r)
    if (l < n) W[tall ? r * ld + l : l * ld + r] = X[r * n + l];
  __syncwarp();
  R* t = sm + L.t;
  R* lam = sm + L.lam;
  R* ws = sm;   // region A
  bidiag(W, ld, P, Q, t, sm + L.tau, sm + L.va, sm + L.vb);
  PEPS_PHASE(1);
  const R tmax = values(t, sm + L.t2, Q, K, lam, ws);
  PEPS_PHASE(2);
  const R pivtiny = Eps<R>::eps * fmax(tmax, Eps<R>::tiny * R(1e10));
  const R sc = l < K ? inverse_iteration(t, n2, lam[l], pivtiny, ws, K, l, (unsigned)(l + 1)) : R(0);
  if (l < K) sm[L.va + l] = sc;
  __syncwarp();
  PEPS_PHASE(3);
  R* Ub = sm + L.Ub;
  R* Uk = sm + L.Uk;
  for (int e = l; e < Q * K; e += 32) Ub[e] = ws[((2 * (e / K) + (tall ? 1 : 0)) * K + e % K) * 4 + 3] * sm[L.va + e % K];
  __syncwarp();
  orthonormalise(Ub, Uk, Q, K);
  PEPS_PHASE(4);
  const int rows = tall ? P : Q;
  for (int e = l; e < rows * K; e += 32) Uk[e] = e < Q * K ? Ub[e] : R(0);
  __syncwarp();
  back_transform(W, ld, tall, P, Q, K, sm + L.tau, Uk, Ub, ws);
  PEPS_PHASE(5);
  finish(Uk, Ub, X, m, n, K, Uout, uo, uk, C, ck, cj);
  PEPS_PHASE(6);
}

// ---------------------------------------------------------------- one row
// Absorbs row `row` into the boundary MPS Min, writing Mout (global memory,
// padded), as peps::absorb_row.  Returns the norm divided out of the last tensor.
template <typename R>
__device__ __noinline__ double absorb_row(const KArgs<R>& a, const R* Min, R* Mout, int row, int dir, bool lr,
                                          const int* bdin, const uint64_t* sp, R* sm, const Layout& L) {
  const Geometry& g = a.g;
  const int D = g.D, Dc = g.Dc, Lx = g.Lx, l = lane_id();
  const int envT = Dc * D * Dc, D3 = D * D * D, DD = D * D;
  const int si = dir == 0 ? D : 1, so = dir == 0 ? 1 : D;
  for (int e = l; e < Lx * envT; e += 32) Mout[e] = R(0);
  R* C = sm + L.C;
  R* M = sm + L.M;
  R* Ts = sm + L.T;
  R* Y = sm + L.Y;
  R* X = sm + L.X;
  if (l == 0) C[0] = R(1);
  __syncwarp();
  int kc = 1, last = 0;
  const int zi = dir == 0 ? (row == 0 ? 1 : D) : (row == g.Ly - 1 ? 1 : D);
  const int zo = dir == 0 ? (row == g.Ly - 1 ? 1 : D) : (row == 0 ? 1 : D);
  for (int step = 0; step < Lx; ++step) {
    const int c = lr ? step : Lx - 1 - step;
    const int za = bdin[c], zb = bdin[c + 1], zl = c == 0 ? 1 : D, zr = c == Lx - 1 ? 1 : D;
    const R* Mc = Min + (size_t)c * envT;
    const int site = row * Lx + c;
    const R* Tc = a.A + ((size_t)site * 2 + (int)((sp[site >> 6] >> (site & 63)) & 1ull)) * (DD * DD);
    last = c;
    int m, n;
    if (lr) {
      // Y[(l,i)][(k,b)] = sum_a C[a][(k,l)] M[a][(i,b)],  X[(k,o)][(b,r)] = sum_{l,i} Y T[(l,i)][(r,o)]
      for (int e = l; e < za * zi * zb; e += 32) {
        const int b = e % zb, ai = e / zb;
        M[e] = Mc[((ai / zi) * D + ai % zi) * Dc + b];
      }
      for (int e = l; e < zl * zi * zr * zo; e += 32) {
        const int o = e % zo, r1 = e / zo, r = r1 % zr, li = r1 / zr;
        Ts[e] = Tc[(li / zi) * D3 + (li % zi) * si + r * DD + o * so];
      }
      __syncwarp();
      const int kb = kc * zb;
      wgemm<R>(kc * zl, zi * zb, za, C, M, Y, ix2(zl, zb, zi * kb), ix2(zb, kb, 1));
      m = kc * zo;
      n = zb * zr;
      wgemm<R>(kb, zr * zo, zl * zi, Y, Ts, X, ix2(zb, zo * n, zr), ix2(zo, 1, n));
    } else {
      // Y[(i,r)][(a,k)] = sum_b M[b][(a,i)] C[b][(r,k)],  X[(o,k)][(a,l)] = sum_{i,r} Y T[(i,r)][(l,o)]
      for (int e = l; e < za * zi * zb; e += 32) {
        const int b = e % zb, ai = e / zb;
        M[b * za * zi + ai] = Mc[((ai / zi) * D + ai % zi) * Dc + b];
      }
      for (int e = l; e < zl * zi * zr * zo; e += 32) {
        const int o = e % zo, r1 = e / zo, ll = r1 % zl, ir = r1 / zl;
        Ts[e] = Tc[(ir / zr) * si + (ir % zr) * DD + ll * D3 + o * so];
      }
      __syncwarp();
      const int ak = za * kc;
      wgemm<R>(za * zi, zr * kc, zb, M, C, Y, ix2(zi, kc, zr * ak), ix2(kc, ak, 1));
      m = zo * kc;
      n = za * zl;
      wgemm<R>(ak, zl * zo, zi * zr, Y, Ts, X, ix2(kc, zl, n), ix2(zo, 1, kc * n));
    }
    R* Mo = Mout + (size_t)c * envT;
    if (step < Lx - 1) {
      const int K = min(Dc, min(m, n));
      // rows (k, o), carry C[b][(k, r)], the next column's a and l; or rows (o, k), carry C[(a, l)][k],
      // the next column's b and r
      if (lr) topk_left<R>(sm, L, m, n, K, Mo, ix2(zo, D * Dc, Dc), 1, zr, ix2(zr, K * zr, 1));
      else topk_left<R>(sm, L, m, n, K, Mo, ix2(kc, Dc, 1), D * Dc, 1, ix1(K));
      kc = K;
    } else {
      for (int e = l; e < m; e += 32)
        Mo[lr ? (e / zo) * D * Dc + (e % zo) * Dc : (e / kc) * Dc + e % kc] = X[e];
      __syncwarp();
    }
  }
  R* Ml = Mout + (size_t)last * envT;
  const double nrm = sqrt(norm2_256(Ml, envT));
  if (nrm > 0.0) {
    const R inv = (R)(1.0 / nrm);
    for (int e = l; e < envT; e += 32) Ml[e] *= inv;
  }
  __syncwarp();
  return nrm;
}

}  // namespace small
}  // namespace peps

// Row absorption and sandwich contractions behind one interface, so that a
// kernel's control flow is written once and runs either with a CTA per work
// item (CtaOps: the tiled GEMM engine) or with a warp per work item (WarpOps:
// models with Dc D <= 32, small.cuh).  A CTA of a WarpOps kernel is one warp.
//
// WarpOps keeps the multiply-add chains of the contraction programs
// (contract.cuh) and the 256-thread partition of the dot products, so results
// equal the CTA's bit for bit (or, asked to, those of the fused kernels).  Two-row steps are split over the
// out-bond of the upper environment: every step of the program is independent
// between out-bonds, so a slice needs three temporaries of D^3 Dc reals instead
// of Dc^2 D^3 and no sum is cut.  Rows that are read as the left operand are
// padded by one real (a row stride of D^2 puts a column's rows in one bank).
#pragma once

#include "kernels_common.cuh"
#include "small.cuh"

namespace peps {

// ------------------------------------------------------------ CTA
template <typename R>
struct CtaOps {
  const KArgs<R>& a;
  ZipBufs<R> zb;
  R* red;
  R* t0;
  R* t1;

  __device__ CtaOps(const KArgs<R>& a_, R* red_) : a(a_), red(red_), t0(nullptr), t1(nullptr) {}
  __device__ double absorb(const R* Min, R* Mout, int row, int dir, bool lr, const int* bdin, const uint64_t* sp) {
    return absorb_row<R>(a, Min, Mout, row, dir, lr, bdin, sp, zb, red);
  }
  __device__ void col1(bool right, const R* F, const R* Mu, const R* T, const R* Md, R* out) {
    run_op<R>(right ? OP_COL1_RIGHT : OP_COL1_LEFT, a.g.D, a.g.Dc, F, Mu, T, Md, nullptr, out, t0, t1, zb.gsm, zb.gism);
  }
  __device__ void col2(bool right, int, const R* E, const R* Mu, const R* T1, const R* T2, const R* Md, R* out) {
    run_op<R>(right ? OP_COL2_RIGHT : OP_COL2_LEFT, a.g.D, a.g.Dc, E, Mu, T1, T2, Md, out, t0, t1, zb.gsm, zb.gism);
  }
  __device__ void site_env(const R* F, const R* Mu, const R* Md, const R* G, R* out) {
    run_op<R>(OP_SITE_ENV, a.g.D, a.g.Dc, F, Mu, Md, G, nullptr, out, t0, t1, zb.gsm, zb.gism);
  }
  __device__ R dot(const R* x, const R* y, int n) { return block_dot(x, y, n, red); }
  __device__ int normalize(R* x, int n) { return normalize_pow2(x, n, red); }
};

// ------------------------------------------------------------ warp
namespace small {

// C(i, j) (+)= sum_k A(i, k) B(k, j) for a descriptor, one chain of fused
// multiply-adds per output; lanes hold TM x TN outputs whose rows (columns)
// are a tile count apart, so consecutive lanes read consecutive rows.
template <typename R, int TM, int TN>
__device__ __noinline__ void desc_gemm_t(const GemmDesc& g, const R* A, const R* B, R* C, bool accumulate) {
  const int nm = (g.M + TM - 1) / TM, nn = (g.N + TN - 1) / TN;
  const int k2n = min(g.ak.n2, g.K), k1n = g.K / k2n;
  for (int t = lane_id(); t < nm * nn; t += 32) {
    const int tm = t / nn, tn = t - tm * nn;
    const R* pa[TM];
    const R* pb[TN];
    int cr[TM], cc[TN];
#pragma unroll
    for (int q = 0; q < TM; ++q) {
      const int i = min(tm + q * nm, g.M - 1);
      pa[q] = A + ixoff(g.am, i);
      cr[q] = ixoff(g.cm, i);
    }
#pragma unroll
    for (int q = 0; q < TN; ++q) {
      const int j = min(tn + q * nn, g.N - 1);
      pb[q] = B + ixoff(g.bn, j);
      cc[q] = ixoff(g.cn, j);
    }
    R acc[TM][TN];
#pragma unroll
    for (int x = 0; x < TM; ++x)
#pragma unroll
      for (int y = 0; y < TN; ++y) acc[x][y] = accumulate ? C[cr[x] + cc[y]] : R(0);
    for (int k1 = 0; k1 < k1n; ++k1) {
      int ao = k1 * g.ak.s1, bo = k1 * g.bk.s1;
#pragma unroll 4
      for (int k2 = 0; k2 < k2n; ++k2, ao += g.ak.s2, bo += g.bk.s2) {
        R av[TM], bv[TN];
#pragma unroll
        for (int q = 0; q < TM; ++q) av[q] = pa[q][ao];
#pragma unroll
        for (int q = 0; q < TN; ++q) bv[q] = pb[q][bo];
#pragma unroll
        for (int x = 0; x < TM; ++x)
#pragma unroll
          for (int y = 0; y < TN; ++y) acc[x][y] = fma(av[x], bv[y], acc[x][y]);
      }
    }
#pragma unroll
    for (int x = 0; x < TM; ++x)
#pragma unroll
      for (int y = 0; y < TN; ++y)
        if (tm + x * nm < g.M && tn + y * nn < g.N) C[cr[x] + cc[y]] = acc[x][y];
  }
  __syncwarp();
}

template <typename R>
__device__ __forceinline__ void desc_gemm(const GemmDesc& g, const R* A, const R* B, R* C, bool accumulate = false) {
  if (g.M * g.N >= 512) desc_gemm_t<R, 4, 4>(g, A, B, C, accumulate);
  else if (g.M * g.N >= 96) desc_gemm_t<R, 2, 2>(g, A, B, C, accumulate);
  else desc_gemm_t<R, 1, 1>(g, A, B, C, accumulate);
}

// A slice of the two-row left transfer at out-bond b (col2_left_step with b
// fixed; Mu points at [0][0][b], C of step 3 at E'[b]).  Row strides: P1
// (l2,a') and P2 (a',r1) DD + 1, P3 (r1,r2) Dc D + 1.
PEPS_HD GemmDesc left2_slice(int s, int D, int Dc) {
  const int DD = D * D, D3 = DD * D, p = DD + 1, q = Dc * D + 1;
  switch (s) {
    case 0:
      return gemm(DD * Dc, D, Dc, ix1(1), kx(Dc, 0, DD * Dc), kx(Dc, 0, D * Dc), ix1(Dc), ix2(D * Dc, D, p), ix1(1));
    case 1:
      return gemm(D * Dc, DD, DD, ix1(p), kx(D, D, 1), kx(D, D3, D), ix2(D, DD, 1), ix2(Dc, D, D * p), ix2(D, p, 1));
    case 2:
      return gemm(Dc * D, DD, DD, ix1(p), kx(D, D, 1), kx(D, D3, D), ix2(D, DD, 1), ix2(D, D, D * q), ix2(D, q, 1));
    default:
      return gemm(DD, Dc, Dc * D, ix1(q), kx(D, D, 1), kx(D, D * Dc, Dc), ix1(1), ix1(Dc), ix1(1));
  }
}
// A slice of the two-row right transfer at out-bond a (col2_right_step with a
// fixed; Mu points at [a][0][0], C of step 3 at H'[a]).  Row strides: P1 and P2
// (r2,b') DD + 1, Q (l1,l2) D Dc + 1.
PEPS_HD GemmDesc right2_slice(int s, int D, int Dc) {
  const int DD = D * D, D3 = DD * D, p = DD + 1, q = Dc * D + 1;
  switch (s) {
    case 0:
      return gemm(DD * Dc, D, Dc, ix1(1), kx(Dc, 0, DD * Dc), kx(Dc, 0, 1), ix1(Dc), ix2(D * Dc, 1, p), ix1(D));
    case 1:
      return gemm(D * Dc, DD, DD, ix1(p), kx(D, D, 1), kx(D, D, DD), ix2(D, D3, 1), ix1(p), ix1(1));
    case 2:
      return gemm(Dc * D, DD, DD, ix2(D, p, D), kx(D, Dc * p, 1), kx(D, DD, D), ix2(D, D3, 1), ix2(D, 1, D * q),
                  ix2(D, q, Dc));
    default:
      return gemm(DD, Dc, D * Dc, ix1(q), kx(Dc, Dc, 1), kx(Dc, Dc, 1), ix1(D * Dc), ix1(Dc), ix1(1));
  }
}
// A slice of the site environment at a (site_env_step with a fixed; F at [a],
// Mu at [a]): R[a'][u][d][r] = Mu . Z, then B += F . R over a'.
PEPS_HD GemmDesc site_slice(int s, int D, int Dc) {
  const int DD = D * D, D3 = DD * D;
  if (s == 0)   // rows (a',d,r) of Z[a'][d][b][r], cols u
    return gemm(Dc * DD, D, Dc, ix2(D, Dc * D, 1), kx(Dc, 0, D), kx(Dc, 0, 1), ix1(Dc), ix2(DD, D3, 1), ix1(DD));
  return gemm(D3, D, Dc, ix1(1), kx(Dc, 0, D3), kx(Dc, 0, 1), ix1(Dc), ix2(D, 1, DD), ix1(D3));   // rows (u,d,r), cols l
}

// The order of row_fused.cuh and pair_fused.cuh.  Left steps sum in the same
// order there; right steps take the horizontal index before the vertical one
// and L's in-bond before its physical index.  The site environment pairs F with
// Mu and Md with G (Z of site_env_step) and sums their product over (a', b).
PEPS_HD GemmDesc fused_right(GemmDesc g, bool site_step, int D, int Dc) {
  if (site_step) {   // k = (r, u) of T and of rows [u][r]
    g.ak = kx(D, 1, D);
    g.bk = kx(D, D * D, D);
  } else {           // k = (b', d) of Md and of rows [d][b']
    g.ak = g.bk = kx(D, 1, Dc);
  }
  return g;
}
PEPS_HD GemmDesc site_fused(int s, int D, int Dc) {
  const int DD = D * D, D3 = DD * D;
  if (s == 0)   // X[b][l][u]: rows l of F[a][l][a'] at a', cols (u,b) of Mu
    return gemm(D, D * Dc, Dc, ix1(Dc), kx(Dc, 0, D * Dc), kx(Dc, 0, D * Dc), ix1(1), ix1(D), ix2(Dc, 1, DD));
  return gemm(DD, DD, Dc, ix1(1), kx(Dc, 0, DD), kx(Dc, 0, D), ix2(D, Dc * D, 1), ix2(D, D3, D), ix2(D, 1, DD));
}

// Reals of shared memory the contractions need; the zip-up's region is reused.
PEPS_HD int ops_reals(int D, int Dc) {
  const int DD = D * D, envT = Dc * D * Dc, p = DD + 1, q = Dc * D + 1;
  const int tens = 2 * up4(envT) + 2 * up4(DD * DD);
  const int pair = up4(envT * D) + 2 * up4(Dc * D * p) + up4(DD * q);
  const int row = up4(envT) + 2 * up4(Dc * Dc * DD);
  const int site = 2 * up4(envT) + up4(Dc * Dc * DD) + up4(Dc * DD * D) + up4(DD * DD);
  return tens + (pair > row ? (pair > site ? pair : site) : (row > site ? row : site));
}
PEPS_HD int ops_total(int D, int Dc) {
  const int z = layout(D, Dc).total, o = ops_reals(D, Dc);
  return z > o ? z : o;
}

template <typename R>
__device__ __forceinline__ R* stage(R*& p, const R* src, int n) {
  R* d = p;
  for (int e = lane_id(); e < n; e += 32) d[e] = src[e];
  p += up4(n);
  return d;
}

}  // namespace small

// fused: sums in the order of the fused kernels, for the models whose sandwiches
// run in either (dispatch by batch size), so that results do not depend on it.
template <typename R, bool fused = false>
struct WarpOps {
  const KArgs<R>& a;
  R* sm;
  small::Layout L;

  __device__ WarpOps(const KArgs<R>& a_, R* sm_) : a(a_), sm(sm_), L(small::layout(a_.g.D, a_.g.Dc)) {}
  __device__ double absorb(const R* Min, R* Mout, int row, int dir, bool lr, const int* bdin, const uint64_t* sp) {
    __syncwarp();
    return small::absorb_row<R>(a, Min, Mout, row, dir, lr, bdin, sp, sm, L);
  }
  __device__ __noinline__ void col1(bool right, const R* F, const R* Mu, const R* T, const R* Md, R* out) {
    const int D = a.g.D, Dc = a.g.Dc, envT = Dc * D * Dc;
    __syncwarp();
    R* p = sm;
    const R* f = small::stage(p, F, envT);
    const R* u = small::stage(p, Mu, envT);
    const R* t = small::stage(p, T, D * D * D * D);
    const R* d = small::stage(p, Md, envT);
    R* t0 = p;
    R* t1 = p + small::up4(Dc * Dc * D * D);
    __syncwarp();
    if (right) small::desc_gemm<R>(col1_right_step(0, D, Dc), u, f, t0);
    else small::desc_gemm<R>(col1_left_step(0, D, Dc), f, u, t0);
    for (int s = 1; s < 3; ++s) {
      GemmDesc g = right ? col1_right_step(s, D, Dc) : col1_left_step(s, D, Dc);
      if (fused && right) g = small::fused_right(g, s == 1, D, Dc);
      small::desc_gemm<R>(g, s == 1 ? t0 : t1, s == 1 ? t : d, s == 1 ? t1 : out);
    }
  }
  // nx: the true dimension of U's out-bond; slices past it are zero
  __device__ __noinline__ void col2(bool right, int nx, const R* E, const R* Mu, const R* T1, const R* T2, const R* Md,
                                    R* out) {
    const int D = a.g.D, Dc = a.g.Dc, DD = D * D, envT = Dc * D * Dc;
    __syncwarp();
    R* p = sm;
    const R* e = small::stage(p, E, envT * D);
    const R* u = small::stage(p, Mu, envT);
    const R* t1 = small::stage(p, T1, DD * DD);
    const R* t2 = small::stage(p, T2, DD * DD);
    const R* d = small::stage(p, Md, envT);
    R* x0 = p;
    R* x1 = x0 + small::up4(Dc * D * (DD + 1));
    R* x2 = x1 + small::up4(Dc * D * (DD + 1));
    __syncwarp();
    for (int k = nx * DD * Dc + small::lane_id(); k < Dc * DD * Dc; k += 32) out[k] = R(0);
    for (int x = 0; x < nx; ++x)
      for (int s = 0; s < 4; ++s) {
        GemmDesc g = right ? small::right2_slice(s, D, Dc) : small::left2_slice(s, D, Dc);
        if (fused && right && (s & 1)) g = small::fused_right(g, s == 1, D, Dc);
        const R* A = s == 0 ? e : (s == 1 ? x0 : (s == 2 ? x1 : x2));
        const R* B = s == 0 ? u + (right ? x * D * Dc : x) : (s == 1 ? t1 : (s == 2 ? t2 : d));
        small::desc_gemm<R>(g, A, B, s == 0 ? x0 : (s == 1 ? x1 : (s == 2 ? x2 : out + x * DD * Dc)));
      }
  }
  __device__ __noinline__ void site_env(const R* F, const R* Mu, const R* Md, const R* G, R* out) {
    const int D = a.g.D, Dc = a.g.Dc, DD = D * D, envT = Dc * D * Dc;
    __syncwarp();
    R* p = sm;
    const R* f = small::stage(p, F, envT);
    const R* u = small::stage(p, Mu, envT);
    const R* d = small::stage(p, Md, envT);
    const R* gg = small::stage(p, G, envT);
    R* z = p;
    R* r = z + small::up4(Dc * Dc * DD);
    R* b = r + small::up4(Dc * DD * D);
    __syncwarp();
    small::desc_gemm<R>(site_env_step(0, D, Dc), d, gg, z);
    for (int x = 0; x < Dc; ++x) {
      if constexpr (fused) {
        small::desc_gemm<R>(small::site_fused(0, D, Dc), f + x, u, r);
        small::desc_gemm<R>(small::site_fused(1, D, Dc), r, z + x * D * Dc * D, b, x > 0);
      } else {
        small::desc_gemm<R>(small::site_slice(0, D, Dc), z, u + x * D * Dc, r);
        small::desc_gemm<R>(small::site_slice(1, D, Dc), r, f + x * D * Dc, b, x > 0);
      }
    }
    for (int k = small::lane_id(); k < DD * DD; k += 32) out[k] = b[k];
    __syncwarp();
  }
  // block_dot and normalize_pow2.  In the fused kernels a thread owns one row (all
  // but the last index) of a two-row transfer, or one entry of a single-row one, the
  // last index slowest.
  __device__ __noinline__ R dot(const R* x, const R* y, int n) {
    R v[8];
    const int Dc = a.g.Dc, rows = n / Dc;
    __syncwarp();
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      R s = R(0);
      if constexpr (fused) {
        const bool one = rows * Dc <= 256;
        const int row = one ? (32 * w + small::lane_id()) % rows : 32 * w + small::lane_id();
        const int k0 = one ? (32 * w + small::lane_id()) / rows : 0, k1 = one ? k0 + 1 : Dc;
        if (row < rows && k1 <= Dc)
          for (int k = k0; k < k1; ++k) s = fma(x[row * Dc + k], y[row * Dc + k], s);
      } else {
        for (int e = 32 * w + small::lane_id(); e < n; e += 256) s = fma(x[e], y[e], s);
      }
      v[w] = s;
    }
    return small::sum256(v);
  }
  __device__ __noinline__ int normalize(R* x, int n) {
    R m = R(0);
    __syncwarp();
    for (int i = small::lane_id(); i < n; i += 32) m = fmax(m, fabs(x[i]));
    const int e = pow2_exponent(warp_max(m));
    if (e != 0) {
      const R sc = pow2<R>(-e);
      for (int i = small::lane_id(); i < n; i += 32) x[i] *= sc;
    }
    __syncwarp();
    return e;
  }
};

}  // namespace peps

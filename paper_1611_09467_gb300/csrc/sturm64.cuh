// FP64 singular values of a bidiagonal matrix by Sturm counts on its
// Golub-Kahan form, for a GPU whose FP64 rate is two multiply-adds per clock
// and SM (measured 1.06 TFLOP/s): what bounds it is the number of FP64
// instructions, not parallelism.
//
//   * Counting without a division: the leading principal minors p_i of T - x
//     follow p_{i+1} = -x p_i - t_i^2 p_{i-1} (two FP64 instructions per row
//     against about thirteen for the quotient form with an IEEE division), the
//     pivots' signs are the sign changes of p (Barth, Martin & Wilkinson,
//     "Calculation of the eigenvalues of a symmetric tridiagonal matrix by
//     the method of bisection", Numer. Math. 9 (1967)).  p is scaled by a
//     power of two every eight rows; signs and scales are integer work.
//   * The first 24 bits come from the FP32 sixteen-section; only the rest is
//     counted in FP64, with as many points per value and step as the lanes of
//     one warp, or of four warps, give (an FP64 instruction of a warp keeps one
//     of the SM's four FP64 units busy for 64 cycles, so further points would
//     be paid for in full).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace peps {

// Number of eigenvalues below x > 0 of the zero-diagonal symmetric
// tridiagonal with squared off-diagonals t2 (scaled so that they are below 4).
// A zero minor counts as a negative pivot, as a clamped pivot does.  Where the
// next off-diagonal is zero too, all later minors are zero and nothing can be
// counted from them: with `replace` a zero minor becomes -2^-100 times the one
// before it (the pivot -2^-100, a change of a diagonal entry far below an ulp).
// zeros: whether the minors ended that way.
template <bool replace>
__device__ __forceinline__ int count_minors(const double* t2, int n2, double x, bool& zeros) {
  double p0 = 1.0, p1 = -x;
  int cnt = 1;
  unsigned sg = 1u;
  auto is_zero = [](double v) { return ((unsigned)(__double2hiint(v) & 0x7fffffff) | (unsigned)__double2loint(v)) == 0u; };
  auto row = [&](double tv) {
    double p2 = fma(-x, p1, -(tv * p0));
    const bool z = is_zero(p2);
    const unsigned s = z ? (sg ^ 1u) : ((unsigned)__double2hiint(p2) >> 31);
    cnt += (int)(s ^ sg);
    sg = s;
    if (replace && z)
      p2 = __hiloint2double((int)(s << 31) | max((__double2hiint(p1) & 0x7ff00000) - (100 << 20), 1 << 20), 0);
    p0 = p1;
    p1 = p2;
  };
  int i = 1;
  for (; i + 7 < n2; i += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) row(t2[i - 1 + u]);
    // eight rows shrink or grow p by far less than half the exponent range
    const int e0 = __double2hiint(p0) & 0x7ff00000, e1 = __double2hiint(p1) & 0x7ff00000;
    const double f = __hiloint2double(0x7fe00000 - max(e0, e1), 0);
    p0 *= f;
    p1 *= f;
  }
  for (; i < n2; ++i) row(t2[i - 1]);
  zeros = is_zero(p0) && is_zero(p1);
  return cnt;
}
static __device__ __noinline__ int count_minors_again(const double* t2, int n2, double x) {
  bool zeros;
  return count_minors<true>(t2, n2, x, zeros);
}
// The replacement is a second pass for the points that need it (a root of a
// leading block, met exactly): in every row it would lengthen the dependent chain
// of the minors (8x8 D = 4 FP64 sweep: 1.3%).
__device__ __forceinline__ int sturm_count_minors(const double* t2, int n2, double x) {
  bool zeros;
  const int cnt = count_minors<false>(t2, n2, x, zeros);
  return zeros ? count_minors_again(t2, n2, x) : cnt;
}

// Half-width of the FP64 start interval around an FP32 value, in units where
// the largest off-diagonal is in [1, 2).  The FP32 counts are exact for a
// matrix whose entries differ by a few units of 2^-24 (rounded squares, 2 ulp
// divisions), so its values are within about 1e-6; this allows eight times that.
constexpr double kSturmWiden = 0x1p-17;

// The K <= 32 largest singular values by whole warps of threads t = 0 .. 31 or
// 0 .. 127 (G points a value and step, G K <= the number of threads): lam32 the
// FP32 values (scaled units), t2 the scaled squares; lam[k] receives scale
// times the k-th.  An FP64 instruction keeps a quarter of the SM busy for 64
// cycles whatever its lanes do, so a CTA counts with four warps, one a quarter
// (10x10 D = 6: 240 kcycles a cut against 410 with one warp).
__device__ __forceinline__ void refine_values_f64(int t, int G, const double* t2, int n2, int K, const float* lam32,
                                                  double scale, double* lam) {
  const int l = t & 31;
  // (G + 1)^nit >= 2^38: from the start interval below 2^-15 to under an ulp
  const int nit = G >= 16 ? 10 : G >= 8 ? 12 : G >= 4 ? 17 : G >= 2 ? 24 : 38;
  const double inv = G >= 16 ? 1.0 / 17 : G >= 8 ? 1.0 / 9 : G >= 4 ? 1.0 / 5 : G >= 2 ? 1.0 / 3 : 0.5;
  const int gid = t / G, gl = t - gid * G, gbase = l / G * G;
  if (__all_sync(0xffffffffu, gid >= K)) return;
  const int idx = n2 - 1 - gid;   // ascending index of the (gid + 1)-th largest
  const double c = gid < K ? (double)lam32[gid] : 1.0;
  double lo = fmax(c - kSturmWiden, 0.0), hi = c + kSturmWiden;
  for (int it = 0; it < nit; ++it) {
    const double step = (hi - lo) * inv;
    const double x = fma(step, (double)(gl + 1), lo);
    const bool pred = sturm_count_minors(t2, n2, x) <= idx;
    const unsigned bits = (__ballot_sync(0xffffffffu, pred) >> gbase) & ((1u << G) - 1u);
    const int gs = __popc(bits);
    if (gs < G) hi = fma(step, (double)(gs + 1), lo);
    lo = fma(step, (double)gs, lo);
  }
  if (gid < K && gl == 0) lam[gid] = 0.5 * (lo + hi) * scale;
}

}  // namespace peps

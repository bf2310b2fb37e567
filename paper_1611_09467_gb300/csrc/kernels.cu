// Layouts and sizes of the scratch slots, the environment cache's check, the
// reductions over sandwiches and configurations, and the GO update (sm_103a).  The
// boundary sweeps are in boundary.cuh (a CTA each) and small.cu (a warp each), the
// allocation-free amplitudes in static.cu, the sandwiches in row.cu and pair.cu,
// the Metropolis chains in mc.cu, the correlations in corr.cu.
//
//   k_finalize : E(S) = diagonal + sum of (J/2) ratios (Sec. II with the
//                Hamiltonian of Sec. IV), status.
//   k_grad_*   : sums of O and E*O over configurations for
//                dE/dA = 2<Delta E> - 2<Delta><E> (Sec. II).
//
// Kernels are persistent over work items (grid-stride), so the per-CTA
// scratch slots bound the workspace.
#include "kernels_common.cuh"

namespace peps {

// ---------------------------------------------------------------- layouts
size_t wm_smem_bytes(const Geometry& g, size_t elem) {
  const size_t P = (size_t)g.Dc * g.D;
  return P * (P + 1) * elem;
}

// Dynamic shared memory of a kernel: a region of reals followed by the GEMM
// offset tables.  For the kernels that truncate, the reals hold (truncation
// matrix if it fits) + the two singular-vector blocks during a truncation and
size_t dyn_smem_bytes(const Geometry& g, size_t elem, bool truncates, bool wm_in_smem) {
  return reals_region_bytes(g, elem, truncates, wm_in_smem) + (size_t)kGemmSmemInts * sizeof(int);
}

// The truncation matrix goes to shared memory up to 212 KB with its buffers: a
// block may have 227 KB and the kernels that truncate hold at most 14 KB of
// static arrays.  D = 10, Dc = 20 in FP32 needs 203 KB; in global memory its
// Householder columns took 62 kcycles each.
bool wm_fits_smem(const Geometry& g, size_t elem) {
  return dyn_smem_bytes(g, elem, true, true) <= 212 * 1024;
}

static size_t zip_elems(const Geometry& g, bool wm_in_smem) {
  const size_t Dc = g.Dc, D = g.D, P = Dc * D;
  return 2 * Dc * Dc * D + Dc * Dc * D * D + P * P + trunc_ws_elems((int)P, g.Dc, !wm_in_smem) + 64 + fit_elems(g);
}

size_t boundary_slot_elems(const Geometry& g, bool wm_in_smem) {
  const size_t envT = (size_t)g.Dc * g.D * g.Dc;
  return zip_elems(g, wm_in_smem) + (size_t)g.Lx * envT;
}

size_t row_slot_elems(const Geometry& g) {
  const size_t envT = (size_t)g.Dc * g.D * g.Dc, D4 = (size_t)g.D * g.D * g.D * g.D;
  return (size_t)(g.Lx + 1) * envT + 4 * envT + D4 + 2 * tmp_elems(g);
}

size_t pair_slot_elems(const Geometry& g) {
  const size_t envT2 = (size_t)g.Dc * g.D * g.D * g.Dc;
  return (size_t)(g.Lx + 1) * envT2 + 4 * envT2 + 2 * tmp_elems(g);
}

size_t mc_slot_elems(const Geometry& g, bool wm_in_smem) {
  const size_t envT = (size_t)g.Dc * g.D * g.Dc;
  const size_t sand = row_slot_elems(g) > pair_slot_elems(g) ? row_slot_elems(g) : pair_slot_elems(g);
  return (size_t)g.Ly * g.Lx * envT + 2 * (size_t)g.Lx * envT + zip_elems(g, wm_in_smem) + sand;
}

// ------------------------------------------------------------ k_boundary
__global__ void k_cache_check(const uint64_t* S, uint64_t* Scache, unsigned* bits, int n, int nwords) {
  for (int cfg = blockIdx.x * blockDim.x + threadIdx.x; cfg < n; cfg += gridDim.x * blockDim.x) {
    bool same = true;
    for (int w = 0; w < nwords; ++w) same = same && S[(size_t)cfg * nwords + w] == Scache[(size_t)cfg * nwords + w];
    if (!same) {
      bits[cfg] = 0u;
      for (int w = 0; w < nwords; ++w) Scache[(size_t)cfg * nwords + w] = S[(size_t)cfg * nwords + w];
    }
  }
}

cudaError_t launch_cache_check(const uint64_t* S, uint64_t* Scache, unsigned* bits, int n, int nwords,
                               cudaStream_t st) {
  k_cache_check<<<(n + 127) / 128, 128, 0, st>>>(S, Scache, bits, n, nwords);
  return cudaGetLastError();
}

// ------------------------------------------------------------ k_finalize
// E(S) = sum over bonds of J (+1/4 parallel, -1/4 antiparallel) plus the
// exchange terms already summed per row / row pair.  Status: S^z != 0 ->
// invalid (1), zero amplitude -> numeric (5).
__global__ void k_finalize(Geometry g, const uint64_t* S, int n, const double* eloc_h, const double* eloc_v,
                           const int* flags, double* eloc, int* status, int have_eloc) {
  const int cfg = blockIdx.x * blockDim.x + threadIdx.x;
  if (cfg >= n) return;
  const uint64_t* sp = S + (size_t)cfg * g.nwords;
  int pc = 0;
  for (int w = 0; w < g.nwords; ++w) {
    uint64_t word = sp[w];
    if (w == g.nwords - 1 && (g.N & 63)) word &= (1ull << (g.N & 63)) - 1ull;
    pc += __popcll(word);
  }
  int st = 0;
  if ((g.N % 2 == 0) && pc != g.N / 2) st = 1;
  else if (flags[cfg] & kFlagTimeout) st = 4;
  else if (flags[cfg] & kFlagZeroW) st = 5;
  if (status) status[cfg] = st;
  if (!have_eloc || eloc == nullptr) return;
  double e = 0.0;
  const int Lx = g.Lx, Ly = g.Ly;
  for (int r = 0; r < Ly; ++r)
    for (int c = 0; c < Lx; ++c) {
      const int i = r * Lx + c, si = spin_of(sp, i);
      if (c + 1 < Lx) e += (si == spin_of(sp, i + 1) ? 0.25 : -0.25) * g.J1;
      if (r + 1 < Ly) e += (si == spin_of(sp, i + Lx) ? 0.25 : -0.25) * g.J1;
      if (r + 1 < Ly && c + 1 < Lx) e += (si == spin_of(sp, i + Lx + 1) ? 0.25 : -0.25) * g.J2;
      if (r + 1 < Ly && c + 1 < Lx) e += (spin_of(sp, i + 1) == spin_of(sp, i + Lx) ? 0.25 : -0.25) * g.J2;
    }
  for (int r = 0; r < Ly; ++r) e += eloc_h[(size_t)cfg * Ly + r];
  for (int r = 0; r + 1 < Ly; ++r) e += eloc_v[(size_t)cfg * Ly + r];
  eloc[cfg] = st == 0 ? e : NAN;
}

// ------------------------------------------------------- gradient sums
// sumO[i][s][p] += sum_cfg O_cfg[i][p] [s_i == s], sumEO likewise times E.
// Each thread owns elements (i, p) of both spin blocks, so no atomics.
template <typename R>
__global__ void k_grad_accum(GradArgs a, const R* __restrict__ O) {
  const size_t total = (size_t)a.N * a.D4;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / a.D4), p = (int)(e % a.D4);
    double o0 = 0, o1 = 0, eo0 = 0, eo1 = 0;
    for (int cfg = 0; cfg < a.n; ++cfg) {
      if (a.status[cfg] != 0) continue;
      const double o = (double)O[(size_t)cfg * total + e];
      const double E = a.eloc[cfg];
      if (spin_of(a.S + (size_t)cfg * a.nwords, i)) {
        o1 += o;
        eo1 += E * o;
      } else {
        o0 += o;
        eo0 += E * o;
      }
    }
    const size_t b0 = ((size_t)i * 2) * a.D4 + p, b1 = b0 + a.D4;
    a.sumO[b0] += o0;
    a.sumO[b1] += o1;
    a.sumEO[b0] += eo0;
    a.sumEO[b1] += eo1;
  }
}

// Over the configurations with status 0: sums[0] += sum of E, sums[1] += their
// count, sums[2] += sum of E^2.
__global__ void k_sum_eloc(const double* eloc, const int* status, int n, double* sums) {
  __shared__ double sh[3][kThreads];
  double s = 0, c = 0, q = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    if (status[i] == 0) {
      s += eloc[i];
      c += 1;
      q += eloc[i] * eloc[i];
    }
  sh[0][threadIdx.x] = s;
  sh[1][threadIdx.x] = c;
  sh[2][threadIdx.x] = q;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
      sh[2][threadIdx.x] += sh[2][threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    sums[0] += sh[0][0];
    sums[1] += sh[1][0];
    sums[2] += sh[2][0];
  }
}

// grad = 2 (<E O> - <E><O>), cov = grad / 2 (Sec. II), from the sums.
__global__ void k_grad_finalize(int total, const double* sums, const double* sumO, const double* sumEO, double* grad,
                                double* cov) {
  const double n = sums[1];
  const double Ebar = n > 0 ? sums[0] / n : 0.0;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const double c = n > 0 ? sumEO[e] / n - Ebar * (sumO[e] / n) : 0.0;
    if (grad) grad[e] = 2.0 * c;
    if (cov) cov[e] = c;
  }
}

// ------------------------------------------------------------- k_go_step
// One gradient-optimisation update of the FP64 tensors (Sec. III):
// A <- A - p dt sign(dE/dA), p in [0, 1) per element, from the same SplitMix64
// construction keyed by (seed, step, element index).  Entries past an open
// edge, and entries whose derivative is zero, do not move.  (p dt) sign is
// exact once p dt is rounded; the _rn intrinsics keep the compiler from
// fusing, so the result is A - (p*dt)*sign evaluated in that order.
__global__ void k_go_step(double* A, const double* grad, Geometry geo, double dt, uint64_t seed, uint64_t step) {
  const uint64_t G = 0x9E3779B97F4A7C15ull;
  const size_t D = (size_t)geo.D, D4 = D * D * D * D, n = (size_t)geo.N * 2 * D4;
  const uint64_t hs = mix64(seed + G * (1ull + step));
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const double g = grad[e];
    if (!(g > 0.0) && !(g < 0.0)) continue;
    const int site = (int)(e / (2 * D4));
    const size_t w = e % D4;
    const size_t l = w / (D * D * D), r = w / (D * D) % D, u = w / D % D, d = w % D;
    const int row = site / geo.Lx, col = site % geo.Lx;
    if ((col == 0 && l) || (col == geo.Lx - 1 && r) || (row == 0 && u) || (row == geo.Ly - 1 && d)) continue;
    const uint64_t h = mix64(hs + G * (1ull + (uint64_t)e));
    const double p = (double)(h >> 11) * 0x1.0p-53;
    A[e] = __dsub_rn(A[e], __dmul_rn(__dmul_rn(p, dt), g > 0.0 ? 1.0 : -1.0));
  }
}

// Sets *bad when any derivative is NaN or infinite: the update of Sec. III
// moves an entry by the sign of its derivative, and such a derivative has none.
__global__ void k_go_check(const double* grad, size_t n, int* bad) {
  int b = 0;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
    if (!isfinite(grad[e])) b = 1;
  if (__syncthreads_or(b) && threadIdx.x == 0) atomicOr(bad, 1);
}

cudaError_t launch_go_check(const double* grad, const Geometry& geo, int* bad, int nsm, cudaStream_t st) {
  const size_t n = (size_t)geo.N * 2 * geo.D * geo.D * geo.D * geo.D;
  const size_t blocks = (n + kThreads - 1) / kThreads;
  const int grid = (int)(blocks < (size_t)nsm * 8 ? blocks : (size_t)nsm * 8);
  if (grid < 1) return cudaSuccess;
  k_go_check<<<grid, kThreads, 0, st>>>(grad, n, bad);
  return cudaGetLastError();
}

// The context's working copy of the tensors in FP32, from the FP64 ones.
__global__ void k_to_f32(const double* __restrict__ a, float* __restrict__ b, size_t n) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
    b[e] = __double2float_rn(a[e]);
}

cudaError_t launch_to_f32(const double* a, float* b, size_t n, int nsm, cudaStream_t st) {
  const size_t blocks = (n + kThreads - 1) / kThreads;
  const int grid = (int)(blocks < (size_t)nsm * 8 ? blocks : (size_t)nsm * 8);
  if (grid < 1) return cudaSuccess;
  k_to_f32<<<grid, kThreads, 0, st>>>(a, b, n);
  return cudaGetLastError();
}

// Site tensors as the B tiles of the tensor-core two-row step (D = 8): per
// (direction, site, spin) TA[n = (yout, d)][k = (u, yin)] and
// TB[n = (yout, d)][k = (yin, u)] in the core-matrix layout, rounded to TF32
// (to nearest, ties away from zero), with (yin, yout) = (l, r) for direction 0
// and (r, l) for direction 1.  One thread per tile element.
__global__ void k_tc_tiles(const double* __restrict__ A, float* __restrict__ tiles, int N) {
  const size_t total = (size_t)2 * N * 2 * 2 * kTcTile;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int n = (int)(e % 4096) / 64, k = (int)(e % 64);
    const size_t tix = e / 4096;                  // ((dir * N + i) * 2 + sp) * 2 + which
    const int which = (int)(tix % 2), sp = (int)(tix / 2 % 2), i = (int)(tix / 4 % N), dir = (int)(tix / 4 / N);
    const int yout = n >> 3, d = n & 7;
    const int u = which == 0 ? (k >> 3) : (k & 7), yin = which == 0 ? (k & 7) : (k >> 3);
    const int l = dir == 0 ? yin : yout, r = dir == 0 ? yout : yin;
    const float v = __double2float_rn(A[((size_t)i * 2 + sp) * 4096 + l * 512 + r * 64 + u * 8 + d]);
    uint32_t t;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(v));
    const int dst = (n >> 3) * 16 * 32 + (k >> 2) * 32 + (n & 7) * 4 + (k & 3);
    tiles[tix * 4096 + dst] = __uint_as_float(t);
  }
}

cudaError_t launch_tc_tiles(const double* A, float* tiles, int N, int nsm, cudaStream_t st) {
  k_tc_tiles<<<nsm * 4, kThreads, 0, st>>>(A, tiles, N);
  return cudaGetLastError();
}

cudaError_t launch_go_step(double* A, const double* grad, const Geometry& geo, double dt, uint64_t seed,
                           uint64_t step, int nsm, cudaStream_t st) {
  const size_t n = (size_t)geo.N * 2 * geo.D * geo.D * geo.D * geo.D;
  const size_t blocks = (n + kThreads - 1) / kThreads;
  const int grid = (int)(blocks < (size_t)nsm * 8 ? blocks : (size_t)nsm * 8);
  if (grid < 1) return cudaSuccess;
  k_go_step<<<grid, kThreads, 0, st>>>(A, grad, geo, dt, seed, step);
  return cudaGetLastError();
}

// --------------------------------------------------------------- launchers
template <typename R>
cudaError_t launch_grad_accum(const GradArgs& a, const R* O, cudaStream_t st) {
  const size_t total = (size_t)a.N * a.D4;
  int grid = (int)((total + kThreads - 1) / kThreads);
  if (grid > 65535 * 8) grid = 65535 * 8;
  k_grad_accum<R><<<grid, kThreads, 0, st>>>(a, O);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const Geometry& g, const uint64_t* S, int n, const double* eloc_h, const double* eloc_v,
                            const int* flags, double* eloc, int* status, int have_eloc, cudaStream_t st) {
  k_finalize<<<(n + 127) / 128, 128, 0, st>>>(g, S, n, eloc_h, eloc_v, flags, eloc, status, have_eloc);
  return cudaGetLastError();
}

cudaError_t launch_sum_eloc(const double* eloc, const int* status, int n, double* sums, cudaStream_t st) {
  k_sum_eloc<<<1, kThreads, 0, st>>>(eloc, status, n, sums);
  return cudaGetLastError();
}

cudaError_t launch_grad_finalize(int total, int, const double* sums, const double* sumO, const double* sumEO,
                                 double* grad, double* cov, cudaStream_t st) {
  int grid = (total + kThreads - 1) / kThreads;
  if (grid > 65535) grid = 65535;
  k_grad_finalize<<<grid, kThreads, 0, st>>>(total, sums, sumO, sumEO, grad, cov);
  return cudaGetLastError();
}

#define PEPS_INST(R) template cudaError_t launch_grad_accum<R>(const GradArgs&, const R*, cudaStream_t);
PEPS_INST(double)
PEPS_INST(float)

}  // namespace peps


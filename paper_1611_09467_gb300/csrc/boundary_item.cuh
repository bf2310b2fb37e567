// One boundary sweep of one configuration (Fig. 1d), shared by the kernels that
// absorb rows with a CTA (boundary.cuh) and with a warp (small.cu).
#pragma once

#include "kernels_common.cuh"

namespace peps {

// One work item: the top-down (dir 0) or bottom-up (dir 1) boundary sweep of
// configuration cfg.  The upper environments U_r go to envU (the last row's
// MPS to `lastbuf`, then closed to psi), the lower ones L_r to envL.
// Absorb: (Min, Mout, row, dir, left to right, bonds of Min) -> the row's norm.
template <typename R, class Absorb>
__device__ void boundary_item(const KArgs<R>& a, int cfg, int dir, R* lastbuf, uint64_t* sp, const int* ones,
                              Absorb absorb) {
  const Geometry& g = a.g;
  const int Lx = g.Lx, Ly = g.Ly, Dc = g.Dc, D = g.D;
  const size_t envT = (size_t)Dc * D * Dc;
  if (a.cache) {
    // this sweep of this configuration is already in place (same bits, same
    // tensors, same workspace): its outputs were kept, only its flag is raised again
    const unsigned bits = a.cache[cfg];
    if (bits & (1u << dir)) {
      if ((bits & (4u << dir)) && threadIdx.x == 0) atomicOr(&a.flags[cfg], kFlagZeroW);
      return;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < g.nwords; i += blockDim.x) sp[i] = a.S[(size_t)cfg * g.nwords + i];
  __syncthreads();
  const R* Min = a.triv_mps;
  double ls = 0.0;
  bool zero = false;
  for (int j = 0; j < Ly; ++j) {
    const int r = dir == 0 ? j : Ly - 1 - j;
    if (dir == 1 && r == 0) break;
    R* Mout;
    if (dir == 0) Mout = r <= Ly - 2 ? a.envU + ((size_t)cfg * Ly + r) * Lx * envT : lastbuf;
    else Mout = a.envL + ((size_t)cfg * Ly + r) * Lx * envT;
    const int* bdin = j == 0 ? ones : a.bd + ((size_t)dir * Ly + (j - 1)) * (Lx + 1);
    const double nrm = absorb(Min, Mout, r, dir, (j % 2) == 0, bdin);
    if (!(nrm > 0.0)) zero = true;
    else ls += log(nrm);
    if (dir == 0 && a.lnU && threadIdx.x == 0) a.lnU[(size_t)cfg * Ly + r] = nrm > 0.0 ? log(nrm) : -INFINITY;
    Min = Mout;
  }
  if (dir == 0) {
    // All physical legs are one now: close the chain of matrices M_c[:, 0, :].
    __shared__ R vec[kMaxDc], nv[kMaxDc];
    if (threadIdx.x == 0) {
      const int* bdl = a.bd + ((size_t)0 * Ly + (Ly - 1)) * (Lx + 1);
      vec[0] = R(1);
      int na = 1;
      for (int c = 0; c < Lx; ++c) {
        const int nb = bdl[c + 1];
        const R* M = lastbuf + (size_t)c * envT;
        for (int b = 0; b < nb; ++b) {
          R s = R(0);
          for (int x = 0; x < na; ++x) s += vec[x] * M[(size_t)x * D * Dc + b];
          nv[b] = s;
        }
        for (int b = 0; b < nb; ++b) vec[b] = nv[b];
        na = nb;
      }
      const R v = vec[0];
      if (zero || v == R(0)) {
        a.logabs[cfg] = -INFINITY;
        a.sign[cfg] = 0;
        atomicOr(&a.flags[cfg], kFlagZeroW);
      } else {
        a.logabs[cfg] = ls + log(fabs((double)v));
        a.sign[cfg] = v > R(0) ? 1 : -1;
      }
    }
  } else if (zero && threadIdx.x == 0) {
    atomicOr(&a.flags[cfg], kFlagZeroW);
  }
  if (a.cache && threadIdx.x == 0) atomicOr(&a.cache[cfg], (1u << dir) | (zero ? (4u << dir) : 0u));
}

}  // namespace peps

// Metropolis sweeps (sampling with weight W^2, Sec. II) over nearest-neighbour
// spin exchanges, one CTA per chain, or one warp where Dc D <= 32.
#include "small_ops.cuh"

namespace peps {

// Metropolis sweeps (sampling with weight W^2, Sec. II) over nearest-neighbour
// exchanges: horizontal bonds row by row, then vertical bonds row pair by row
// pair.  Lower environments are rebuilt from the current S at the start of
// each pass; the upper environment grows from the updated rows; the row (or
// row-pair) transfers to the left are carried with the accepted spins.
template <typename R, class Ops>
__device__ void mc_chains(const KArgs<R>& a, Ops& ops, R* p, uint64_t* sp, int* ones, int* eH, uint64_t* S, int nsweeps,
                          uint64_t seed, uint64_t chain0, uint64_t sweep0, long long* accepted) {
  const Geometry& g = a.g;
  const int Lx = g.Lx, Ly = g.Ly, Dc = g.Dc, D = g.D;
  const size_t envT = (size_t)Dc * D * Dc, envT2 = envT * D;
  R* envL = p; p += (size_t)Ly * Lx * envT;
  R* Ubuf[2];
  Ubuf[0] = p; p += (size_t)Lx * envT;
  Ubuf[1] = p; p += (size_t)Lx * envT;
  R* Hb = p; p += (size_t)(Lx + 1) * envT2;
  R* Q[4];
  for (int q = 0; q < 4; ++q) { Q[q] = p; p += envT2; }
  for (int i = threadIdx.x; i <= Lx; i += blockDim.x) ones[i] = 1;
  // H_c is stored scaled by 2^-eH[c]
  const int nh = Ly * (Lx - 1);
  for (int chain = blockIdx.x; chain < a.n; chain += gridDim.x) {
    __syncthreads();
    for (int i = threadIdx.x; i < g.nwords; i += blockDim.x) sp[i] = S[(size_t)chain * g.nwords + i];
    __syncthreads();
    long long acc = 0;
    for (int k = 0; k < nsweeps; ++k) {
      const uint64_t sweep = sweep0 + (uint64_t)k;
      for (int pass = 0; pass < 2; ++pass) {
        // lower environments L_r, r = Ly-1 .. 1, from the current S
        const R* Min = a.triv_mps;
        for (int j = 0; j + 1 < Ly; ++j) {
          const int r = Ly - 1 - j;
          const int* bdin = j == 0 ? ones : a.bd + ((size_t)1 * Ly + (j - 1)) * (Lx + 1);
          R* Mout = envL + (size_t)r * Lx * envT;
          ops.absorb(Min, Mout, r, 1, (j % 2) == 0, bdin, sp);
          Min = Mout;
        }
        const R* Mu = a.triv_mps;
        int ub = 0;
        const int rows = pass == 0 ? Ly : Ly - 1;
        for (int r = 0; r < rows; ++r) {
          const R* Md;
          if (pass == 0) Md = r == Ly - 1 ? a.triv_mps : envL + (size_t)(r + 1) * Lx * envT;
          else Md = r + 2 > Ly - 1 ? a.triv_mps : envL + (size_t)(r + 2) * Lx * envT;
          // true bonds of U_{r-1}, by column boundary
          const int* bu = r == 0 ? ones : a.bd + (size_t)(r - 1) * (Lx + 1);
          const size_t tsz = pass == 0 ? envT : envT2;
          const R* triv = pass == 0 ? a.triv_t1 : a.triv_t2;
          for (size_t e = threadIdx.x; e < tsz; e += blockDim.x) Hb[(size_t)Lx * tsz + e] = triv[e];
          if (threadIdx.x == 0) eH[Lx] = 0;
          __syncthreads();
          int eacc = 0;
          for (int c = Lx - 1; c >= 0; --c) {
            const int i1 = r * Lx + c;
            if (pass == 0)
              ops.col1(true, Hb + (size_t)(c + 1) * tsz, Mu + (size_t)c * envT,
                        tptr(a, i1, spin_of(sp, i1)), Md + (size_t)c * envT, Hb + (size_t)c * tsz);
            else
              ops.col2(true, bu[c], Hb + (size_t)(c + 1) * tsz, Mu + (size_t)c * envT,
                        tptr(a, i1, spin_of(sp, i1)), tptr(a, i1 + Lx, spin_of(sp, i1 + Lx)),
                        Md + (size_t)c * envT, Hb + (size_t)c * tsz);
            eacc += ops.normalize(Hb + (size_t)c * tsz, (int)tsz);
            if (threadIdx.x == 0) eH[c] = eacc;
          }
          const R* E = triv;
          int e = 3;   // index in Q of the buffer E lives in (none yet)
          const int ncol = pass == 0 ? Lx - 1 : Lx;
          for (int c = 0; c < ncol; ++c) {
            const int i1 = r * Lx + c;
            const int i2 = pass == 0 ? i1 + 1 : i1 + Lx;
            const int s1 = spin_of(sp, i1), s2 = spin_of(sp, i2);
            R* X1 = Q[(e + 1) & 3];
            R* Xf = Q[(e + 2) & 3];
            R* X2 = Q[(e + 3) & 3];
            const R* Muc = Mu + (size_t)c * envT;
            const R* Mdc = Md + (size_t)c * envT;
            int chosen;
            if (s1 != s2) {
              R w, wp;
              if (pass == 0) {
                ops.col1(false, E, Muc, tptr(a, i1, s1), Mdc, X1);
                ops.col1(false, E, Muc, tptr(a, i1, s2), Mdc, Xf);
                ops.col1(false, Xf, Mu + (size_t)(c + 1) * envT, tptr(a, i2, s1),
                          Md + (size_t)(c + 1) * envT, X2);
                w = ops.dot(X1, Hb + (size_t)(c + 1) * tsz, (int)tsz);
                wp = ops.dot(X2, Hb + (size_t)(c + 2) * tsz, (int)tsz);
              } else {
                ops.col2(false, bu[c + 1], E, Muc, tptr(a, i1, s1), tptr(a, i2, s2), Mdc, X1);
                ops.col2(false, bu[c + 1], E, Muc, tptr(a, i1, s2), tptr(a, i2, s1), Mdc, Xf);
                w = ops.dot(X1, Hb + (size_t)(c + 1) * tsz, (int)tsz);
                wp = ops.dot(Xf, Hb + (size_t)(c + 1) * tsz, (int)tsz);
              }
              const uint64_t bond = pass == 0 ? (uint64_t)(r * (Lx - 1) + c) : (uint64_t)(nh + r * Lx + c);
              const double u = sampler_uniform(seed, chain0 + (uint64_t)chain, sweep, bond);
              bool take;
              if (w == R(0)) {
                take = true;
              } else {
                // the E scale is common to w and wp; the H scales differ by a column in a horizontal exchange
                const double ratio =
                    pass == 0 ? ldexp((double)wp / (double)w, eH[c + 2] - eH[c + 1]) : (double)wp / (double)w;
                take = u < ratio * ratio;
              }
              if (take) {
                if (threadIdx.x == 0) {
                  sp[i1 >> 6] ^= 1ull << (i1 & 63);
                  sp[i2 >> 6] ^= 1ull << (i2 & 63);
                }
                ++acc;
                chosen = (e + 2) & 3;
              } else {
                chosen = (e + 1) & 3;
              }
              __syncthreads();
            } else {
              if (pass == 0)
                ops.col1(false, E, Muc, tptr(a, i1, s1), Mdc, X1);
              else
                ops.col2(false, bu[c + 1], E, Muc, tptr(a, i1, s1), tptr(a, i2, s2), Mdc, X1);
              chosen = (e + 1) & 3;
            }
            e = chosen;
            E = Q[e];
            // E's own scale cancels in every ratio: renormalise without tracking
            ops.normalize(Q[e], (int)tsz);
          }
          if (pass == 0 ? (r < Ly - 1) : true) {
            const int* bdin = r == 0 ? ones : a.bd + ((size_t)0 * Ly + (r - 1)) * (Lx + 1);
            ops.absorb(Mu, Ubuf[ub], r, 0, (r % 2) == 0, bdin, sp);
            Mu = Ubuf[ub];
            ub ^= 1;
          }
        }
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < g.nwords; i += blockDim.x) S[(size_t)chain * g.nwords + i] = sp[i];
    if (threadIdx.x == 0 && accepted) accepted[chain] += acc;
  }
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_mc(KArgs<R> a, uint64_t* S, int nsweeps, uint64_t seed, uint64_t chain0,
                                                 uint64_t sweep0, long long* accepted) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ R red[64];
  __shared__ uint64_t sp[kMaxWords];
  __shared__ int ones[kMaxDcD + 1];
  __shared__ int eH[kMaxL + 1];
  __shared__ double dred[kWarps];
  __shared__ R wv[kMaxDcD];
  const Geometry& g = a.g;
  CtaOps<R> ops(a, red);
  R* gsm;
  int* gism;
  smem_split<R>(smem_raw, g, true, a.smem_wm != 0, gsm, gism);
  R* p = a.scratch + (size_t)blockIdx.x * a.slot_elems;
  carve_zip<R>(g, p, ops.zb, a.smem_wm ? gsm : nullptr, red, dred, wv, gsm, gism);
  ops.t0 = p; p += tmp_elems(g);
  ops.t1 = p; p += tmp_elems(g);
  mc_chains<R>(a, ops, p, sp, ones, eH, S, nsweeps, seed, chain0, sweep0, accepted);
}

// One warp per chain (models small.cuh takes), at any number of chains: on one
// chain too a warp is not behind a CTA (8x8, ms a sweep: FP32 10.0 against 20.0 at D = 2
// Dc = 8, 24.1 against 30.4 at D = 4 Dc = 6, 38.8 against 38.3 at D = 5 Dc = 6, the closest;
// FP64 101 against 128 at D = 4 Dc = 8, 145 against 156 at D = 5 Dc = 6; alike for 152).  304
// chains of 8x8 D = 4 Dc = 8 in FP64 take 105 ms a sweep against 397 ms with a CTA each,
// whose time went to the truncation's barriers and FP64 sections and to the tiled
// engine's offset tables on products of a few hundred outputs.
template <typename R>
__global__ void __launch_bounds__(32) k_mc_small(KArgs<R> a, uint64_t* S, int nsweeps, uint64_t seed, uint64_t chain0,
                                                 uint64_t sweep0, long long* accepted) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t sp[kMaxWords];
  __shared__ int ones[kMaxL + 1];
  __shared__ int eH[kMaxL + 1];
  WarpOps<R> ops(a, reinterpret_cast<R*>(smem_raw));
  mc_chains<R>(a, ops, a.scratch + (size_t)blockIdx.x * a.slot_elems, sp, ones, eH, S, nsweeps, seed, chain0, sweep0,
               accepted);
}

size_t mc_small_slot_elems(const Geometry& g) {
  const size_t envT = (size_t)g.Dc * g.D * g.Dc;
  return (size_t)g.Ly * g.Lx * envT + 2 * (size_t)g.Lx * envT + (size_t)(g.Lx + 5) * envT * g.D;
}

template <typename R>
int max_blocks_mc_small(const Geometry& g) {
  int dev = 0, nsm = 0, nb = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = (size_t)small::ops_total(g.D, g.Dc) * sizeof(R);
  prefer_shared(k_mc_small<R>, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_mc_small<R>, 32, smem);
  return nsm * (nb < 1 ? 1 : nb);
}

template <typename R>
cudaError_t launch_mc_small(const KArgs<R>& a, uint64_t* S, int nsweeps, uint64_t seed, uint64_t chain0,
                            uint64_t sweep0, long long* accepted, int grid, cudaStream_t st) {
  const size_t smem = (size_t)small::ops_total(a.g.D, a.g.Dc) * sizeof(R);
  cudaError_t e = prefer_shared(k_mc_small<R>, smem);
  if (e != cudaSuccess) return e;
  k_mc_small<R><<<grid, 32, smem, st>>>(a, S, nsweeps, seed, chain0, sweep0, accepted);
  return cudaGetLastError();
}

template <typename R>
int max_blocks_mc(const Geometry& g) {
  int dev = 0, nsm = 0, nb = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = dyn_smem_bytes(g, sizeof(R), true, wm_fits_smem(g, sizeof(R)));
  prefer_shared(k_mc<R>, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_mc<R>, kThreads, smem);
  if (nb < 1) nb = 1;
  return nsm * nb;
}

template <typename R>
cudaError_t launch_mc(const KArgs<R>& a, uint64_t* S, int nsweeps, uint64_t seed, uint64_t chain0, uint64_t sweep0,
                      long long* accepted, int grid, cudaStream_t st) {
  const size_t smem = dyn_smem_bytes(a.g, sizeof(R), true, a.smem_wm != 0);
  cudaError_t e = prefer_shared(k_mc<R>, smem);
  if (e != cudaSuccess) return e;
  k_mc<R><<<grid, kThreads, smem, st>>>(a, S, nsweeps, seed, chain0, sweep0, accepted);
  return cudaGetLastError();
}

#define PEPS_INST(R)                                                                                    \
  template int max_blocks_mc_small<R>(const Geometry&);                                                 \
  template cudaError_t launch_mc_small<R>(const KArgs<R>&, uint64_t*, int, uint64_t, uint64_t, uint64_t, \
                                          long long*, int, cudaStream_t);                               \
  template int max_blocks_mc<R>(const Geometry&);                                                       \
  template cudaError_t launch_mc<R>(const KArgs<R>&, uint64_t*, int, uint64_t, uint64_t, uint64_t,      \
                                    long long*, int, cudaStream_t);
PEPS_INST(double)
PEPS_INST(float)

}  // namespace peps

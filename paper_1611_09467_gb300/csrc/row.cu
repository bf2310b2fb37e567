// Single-row sandwich kernels <U_{r-1}| row r |L_{r+1}> (Sec. II): W_r, the
// amplitude ratios of horizontal spin exchanges and Delta = B/W.  One CTA per
// (configuration, row); k_row_fused keeps every intermediate in shared memory
// for (D, Dc) = (2,4), (4,8), (6,12), (8,16).
#include "small_ops.cuh"

namespace peps {

// ----------------------------------------------------------------- k_row
template <typename R, class Ops>
__device__ void row_items(const KArgs<R>& a, Ops& ops, R* p, uint64_t* sp, int* eG) {
  // G_c is stored scaled by 2^-eG[c]
  const Geometry& g = a.g;
  const int Lx = g.Lx, Ly = g.Ly, Dc = g.Dc, D = g.D;
  const int envT = Dc * D * Dc, D4 = D * D * D * D;
  R* Gb = p; p += (size_t)(Lx + 1) * envT;
  R* F0 = p; p += envT;
  R* F1 = p; p += envT;
  R* X1 = p; p += envT;
  R* X2 = p; p += envT;
  R* Bb = p;
  for (int item = blockIdx.x; item < a.n * Ly; item += gridDim.x) {
    const int cfg = item / Ly, r = item % Ly;
    __syncthreads();
    for (int i = threadIdx.x; i < g.nwords; i += blockDim.x) sp[i] = a.S[(size_t)cfg * g.nwords + i];
    for (int e = threadIdx.x; e < envT; e += blockDim.x) Gb[(size_t)Lx * envT + e] = a.triv_t1[e];
    if (threadIdx.x == 0) eG[Lx] = 0;
    __syncthreads();
    const R* Mu = r == 0 ? a.triv_mps : a.envU + ((size_t)cfg * Ly + (r - 1)) * Lx * envT;
    const R* Md = r == Ly - 1 ? a.triv_mps : a.envL + ((size_t)cfg * Ly + (r + 1)) * Lx * envT;
    int eacc = 0;
    for (int c = Lx - 1; c >= 0; --c) {
      const int site = r * Lx + c;
      ops.col1(true, Gb + (size_t)(c + 1) * envT, Mu + (size_t)c * envT,
                tptr(a, site, spin_of(sp, site)), Md + (size_t)c * envT, Gb + (size_t)c * envT);
      eacc += ops.normalize(Gb + (size_t)c * envT, envT);
      if (threadIdx.x == 0) eG[c] = eacc;
    }
    const R W = Gb[0];
    const bool ok = W != R(0);
    double eh = 0.0;
    const R* F = a.triv_t1;
    int eF = 0;   // F is stored scaled by 2^-eF
    R* Fn = F0;
    for (int c = 0; c < Lx; ++c) {
      const int site = r * Lx + c;
      const int s = spin_of(sp, site);
      if (a.O != nullptr) {
        ops.site_env(F, Mu + (size_t)c * envT, Md + (size_t)c * envT,
                  Gb + (size_t)(c + 1) * envT, Bb);
        R* Oo = a.O + ((size_t)cfg * g.N + site) * D4;
        const R inv = ok ? (R)ldexp(1.0 / (double)W, eF + eG[c + 1] - eG[0]) : R(0);
        for (int e = threadIdx.x; e < D4; e += blockDim.x) Oo[e] = Bb[e] * inv;
      }
      if (c < Lx - 1) {
        const int s2 = spin_of(sp, site + 1);
        if (s != s2) {
          ops.col1(false, F, Mu + (size_t)c * envT, tptr(a, site, s2), Md + (size_t)c * envT, X1);
          const int eX = ops.normalize(X1, envT);
          ops.col1(false, X1, Mu + (size_t)(c + 1) * envT, tptr(a, site + 1, s),
                    Md + (size_t)(c + 1) * envT, X2);
          const R wp = ops.dot(X2, Gb + (size_t)(c + 2) * envT, envT);
          if (ok) eh += 0.5 * g.J1 * ldexp((double)wp / (double)W, eF + eX + eG[c + 2] - eG[0]);
        }
        ops.col1(false, F, Mu + (size_t)c * envT, tptr(a, site, s), Md + (size_t)c * envT, Fn);
        eF += ops.normalize(Fn, envT);
        F = Fn;
        Fn = (Fn == F0) ? F1 : F0;
      }
    }
    if (threadIdx.x == 0) {
      a.eloc_h[(size_t)cfg * Ly + r] = eh;
      a.w_row[(size_t)cfg * Ly + r] = ldexp((double)W, eG[0]);
      if (!ok) atomicOr(&a.flags[cfg], kFlagZeroW);
    }
  }
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_row(KArgs<R> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ R red[64];
  __shared__ uint64_t sp[kMaxWords];
  __shared__ int eG[kMaxL + 1];
  CtaOps<R> ops(a, red);
  smem_split<R>(smem_raw, a.g, false, false, ops.zb.gsm, ops.zb.gism);
  R* p = a.scratch + (size_t)blockIdx.x * a.slot_elems;
  ops.t0 = p; p += tmp_elems(a.g);
  ops.t1 = p; p += tmp_elems(a.g);
  row_items<R>(a, ops, p, sp, eG);
}

// One warp per (configuration, row), for the models small.cuh takes: k_row's
// contractions with each product on one warp in shared memory (small_ops.cuh).
// 6x6 D = 3 Dc = 6 FP64, 128 configurations with Delta: 0.8 ms against 25 with k_row.
template <typename R, bool fused>
__global__ void __launch_bounds__(32) k_row_small(KArgs<R> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t sp[kMaxWords];
  __shared__ int eG[kMaxL + 1];
  WarpOps<R, fused> ops(a, reinterpret_cast<R*>(smem_raw));
  row_items<R>(a, ops, a.scratch + (size_t)blockIdx.x * a.slot_elems, sp, eG);
}

size_t row_small_slot_elems(const Geometry& g) {
  const size_t envT = (size_t)g.Dc * g.D * g.Dc;
  return (size_t)(g.Lx + 5) * envT + (size_t)g.D * g.D * g.D * g.D;
}

// The kernel for a model: in the order of the fused one where both are used.
template <typename R>
static auto row_small_kernel(const Geometry& g) -> void (*)(KArgs<R>) {
  if constexpr (sizeof(R) == 8)
    if (sandwich_in_fused_order<R>(g)) return k_row_small<R, true>;
  return k_row_small<R, false>;
}

template <typename R>
int max_blocks_row_small(const Geometry& g) {
  int dev = 0, nsm = 0, nb = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = (size_t)small::ops_reals(g.D, g.Dc) * sizeof(R);
  const auto kernel = row_small_kernel<R>(g);
  prefer_shared(kernel, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, 32, smem);
  return nsm * (nb < 1 ? 1 : nb);
}

template <typename R>
cudaError_t launch_row_small(const KArgs<R>& a, int grid, cudaStream_t st) {
  const size_t smem = (size_t)small::ops_reals(a.g.D, a.g.Dc) * sizeof(R);
  const auto kernel = row_small_kernel<R>(a.g);
  cudaError_t e = prefer_shared(kernel, smem);
  if (e != cudaSuccess) return e;
  kernel<<<grid, 32, smem, st>>>(a);
  return cudaGetLastError();
}

// ------------------------------------------------------------- k_row_fused
// k_row with the fused shared-memory step and site environment
// (row_fused.cuh) for a fixed (D, Dc).  Transfers are stored [x'][x][y].
template <typename R, int D, int Dc>
__global__ void __launch_bounds__(kThreads) k_row_fused(KArgs<R> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ R red[64];
  __shared__ uint64_t sp[kMaxWords];
  R* sm = reinterpret_cast<R*>(smem_raw);
  const Geometry& g = a.g;
  const int Lx = g.Lx, Ly = g.Ly;
  constexpr int envT = Dc * D * Dc, D4 = D * D * D * D;
  R* p = a.scratch + (size_t)blockIdx.x * a.slot_elems;
  R* Gb = p; p += (size_t)(Lx + 1) * envT;
  R* F0 = p; p += envT;
  R* F1 = p; p += envT;
  R* X1 = p;
  __shared__ int eG[kMaxL + 1];   // G_c is stored scaled by 2^-eG[c]
  for (int item = blockIdx.x; item < a.n * Ly; item += gridDim.x) {
    const int cfg = item / Ly, r = item % Ly;
    __syncthreads();
    for (int i = threadIdx.x; i < g.nwords; i += blockDim.x) sp[i] = a.S[(size_t)cfg * g.nwords + i];
    for (int e = threadIdx.x; e < envT; e += blockDim.x) Gb[(size_t)Lx * envT + e] = a.triv_t1[e];
    if (threadIdx.x == 0) eG[Lx] = 0;
    __syncthreads();
    const R* Mu = r == 0 ? a.triv_mps : a.envU + ((size_t)cfg * Ly + (r - 1)) * Lx * envT;
    const R* Md = r == Ly - 1 ? a.triv_mps : a.envL + ((size_t)cfg * Ly + (r + 1)) * Lx * envT;
    // true bonds of L_{r+1}, by column boundary
    const int* bl = r == Ly - 1 ? nullptr : a.bd + (size_t)(Ly + Ly - 2 - r) * (Lx + 1);
    auto nb = [&](int c) { return bl ? bl[c] : 1; };
    int eacc = 0;
    for (int c = Lx - 1; c >= 0; --c) {
      const int site = r * Lx + c;
      int e = 0;
      row_step_fused<R, D, Dc>(true, nb(c + 1), Gb + (size_t)(c + 1) * envT, Gb + (size_t)c * envT, Mu + (size_t)c * envT,
                               tptr(a, site, spin_of(sp, site)), Md + (size_t)c * envT, nullptr, sm, red, &e);
      eacc += e;
      if (threadIdx.x == 0) eG[c] = eacc;
    }
    const R W = Gb[0];
    const bool ok = W != R(0);
    double eh = 0.0;
    const R* F = a.triv_t1;
    int eF = 0;   // F is stored scaled by 2^-eF
    R* Fn = F0;
    for (int c = 0; c < Lx; ++c) {
      const int site = r * Lx + c;
      const int s = spin_of(sp, site);
      const R* Muc = Mu + (size_t)c * envT;
      const R* Mdc = Md + (size_t)c * envT;
      if (a.O != nullptr)
        site_env_fused<R, D, Dc>(nb(c), F, Muc, Mdc, Gb + (size_t)(c + 1) * envT,
                                 ok ? (R)ldexp(1.0 / (double)W, eF + eG[c + 1] - eG[0]) : R(0),
                                 a.O + ((size_t)cfg * g.N + site) * D4, sm);
      if (c < Lx - 1) {
        const int s2 = spin_of(sp, site + 1);
        if (s != s2) {
          int eX = 0;
          row_step_fused<R, D, Dc>(false, nb(c), F, X1, Muc, tptr(a, site, s2), Mdc, nullptr, sm, red, &eX);
          const R wp = row_step_fused<R, D, Dc>(false, nb(c + 1), X1, nullptr, Mu + (size_t)(c + 1) * envT, tptr(a, site + 1, s),
                                                Md + (size_t)(c + 1) * envT, Gb + (size_t)(c + 2) * envT, sm, red);
          if (ok) eh += 0.5 * g.J1 * ldexp((double)wp / (double)W, eF + eX + eG[c + 2] - eG[0]);
        }
        int e1 = 0;
        row_step_fused<R, D, Dc>(false, nb(c), F, Fn, Muc, tptr(a, site, s), Mdc, nullptr, sm, red, &e1);
        eF += e1;
        F = Fn;
        Fn = (Fn == F0) ? F1 : F0;
      }
    }
    if (threadIdx.x == 0) {
      a.eloc_h[(size_t)cfg * Ly + r] = eh;
      a.w_row[(size_t)cfg * Ly + r] = ldexp((double)W, eG[0]);
      if (!ok) atomicOr(&a.flags[cfg], kFlagZeroW);
    }
  }
}

template <typename R>
static int row_fused_id(const Geometry& g) {
  if (g.D == 2 && g.Dc == 4) return 1;
  if (g.D == 4 && g.Dc == 8) return 2;
  if (g.D == 6 && g.Dc == 12) return 3;
  if (g.D == 8 && g.Dc == 16) return 4;
  return 0;
}

bool row_has_fused(const Geometry& g) { return row_fused_id<float>(g) != 0; }

template <typename R, int D, int Dc>
static int row_fused_blocks() {
  int dev = 0, nsm = 0, nb = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = (size_t)RowSmem<D, Dc>::total * sizeof(R);
  prefer_shared(k_row_fused<R, D, Dc>, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_row_fused<R, D, Dc>, kThreads, smem);
  return nsm * (nb < 1 ? 1 : nb);
}

template <typename R, int D, int Dc>
static cudaError_t launch_row_fused(const KArgs<R>& a, int grid, cudaStream_t st) {
  const size_t smem = (size_t)RowSmem<D, Dc>::total * sizeof(R);
  cudaError_t e = prefer_shared(k_row_fused<R, D, Dc>, smem);
  if (e != cudaSuccess) return e;
  k_row_fused<R, D, Dc><<<grid, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename R>
int max_blocks_row(const Geometry& g, int generic) {
  switch (generic ? 0 : row_fused_id<R>(g)) {
    case 1: return row_fused_blocks<R, 2, 4>();
    case 2: return row_fused_blocks<R, 4, 8>();
    case 3: return row_fused_blocks<R, 6, 12>();
    case 4: return row_fused_blocks<R, 8, 16>();
  }
  int dev = 0, nsm = 0, nb = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = dyn_smem_bytes(g, sizeof(R), false, false);
  prefer_shared(k_row<R>, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_row<R>, kThreads, smem);
  return nsm * (nb < 1 ? 1 : nb);
}

template <typename R>
cudaError_t launch_row(const KArgs<R>& a, int grid, cudaStream_t st, int generic) {
  switch (generic ? 0 : row_fused_id<R>(a.g)) {
    case 1: return launch_row_fused<R, 2, 4>(a, grid, st);
    case 2: return launch_row_fused<R, 4, 8>(a, grid, st);
    case 3: return launch_row_fused<R, 6, 12>(a, grid, st);
    case 4: return launch_row_fused<R, 8, 16>(a, grid, st);
  }
  const size_t smem = dyn_smem_bytes(a.g, sizeof(R), false, false);
  cudaError_t e = prefer_shared(k_row<R>, smem);
  if (e != cudaSuccess) return e;
  k_row<R><<<grid, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

#define PEPS_INST(R)                                                                                    \
  template int max_blocks_row_small<R>(const Geometry&);                                                \
  template cudaError_t launch_row_small<R>(const KArgs<R>&, int, cudaStream_t);                         \
  template int max_blocks_row<R>(const Geometry&, int);                                                 \
  template cudaError_t launch_row<R>(const KArgs<R>&, int, cudaStream_t, int);
PEPS_INST(double)
PEPS_INST(float)

}  // namespace peps

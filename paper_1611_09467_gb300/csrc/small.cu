// Boundary sweeps with one warp per sweep (small.cuh), for models with
// Dc D <= 32.
#include "boundary_item.cuh"
#include "small.cuh"

namespace peps {

// The sweeps of one model (nm = 0: `one`) or of several (a packed launch: work
// items numbered model after model, start[m] the first item of models[m]).  A
// CTA is one warp; its slot in scratch holds the last row's MPS.  8192 sweeps of
// 8x8 D = 4 Dc = 8 in FP32 take 38 ms against 210 ms with a CTA each, one sweep
// alone 3.6 ms against 6.4 (4x4 D = 2 FP64: 0.30 ms against 0.88).  The line at
// Dc D <= 32 is where a block row stops fitting a warp.
template <typename R>
__global__ void __launch_bounds__(32, sizeof(R) == 4 ? 10 : 5) k_boundary_small(KArgs<R> one, const KArgs<R>* __restrict__ models,
                                                       const int* __restrict__ start, int nm, int dirs, R* scratch,
                                                       size_t slot_elems) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t sp[kMaxWords];
  __shared__ int ones[kMaxL + 1];
  R* sm = reinterpret_cast<R*>(smem_raw);
  R* lastbuf = scratch + (size_t)blockIdx.x * slot_elems;
  for (int i = threadIdx.x; i <= kMaxL; i += 32) ones[i] = 1;
  const int total = nm > 0 ? start[nm] : one.n * dirs;
  int m = 0;
  for (int item = blockIdx.x; item < total; item += gridDim.x) {
    while (m + 1 < nm && start[m + 1] <= item) ++m;
    const KArgs<R>& a = nm > 0 ? models[m] : one;
    const int local = nm > 0 ? item - start[m] : item;
    const small::Layout L = small::layout(a.g.D, a.g.Dc);
    boundary_item<R>(a, local % a.n, local / a.n, lastbuf, sp, ones,
                     [&](const R* Min, R* Mout, int r, int dir, bool lr, const int* bdin) {
                       return small::absorb_row<R>(a, Min, Mout, r, dir, lr, bdin, sp, sm, L);
                     });
  }
}

bool boundary_small_fits(const Geometry& g) { return small::fits(g); }
size_t boundary_small_smem(const Geometry& g, size_t elem) { return (size_t)small::layout(g.D, g.Dc).total * elem; }

template <typename R>
int max_blocks_boundary_small(size_t smem) {
  int dev = 0, nsm = 0, nb = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  prefer_shared(k_boundary_small<R>, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_boundary_small<R>, 32, smem);
  return nsm * (nb < 1 ? 1 : nb);
}

template <typename R>
cudaError_t launch_boundary_small(const KArgs<R>& one, const KArgs<R>* models_dev, const int* start_dev, int nm,
                                  int dirs, R* scratch, size_t slot_elems, size_t smem, int grid, cudaStream_t st) {
  cudaError_t e = prefer_shared(k_boundary_small<R>, smem);
  if (e != cudaSuccess) return e;
  k_boundary_small<R><<<grid, 32, smem, st>>>(one, models_dev, start_dev, nm, dirs, scratch, slot_elems);
  return cudaGetLastError();
}

#define PEPS_INST(R)                                                                                           \
  template int max_blocks_boundary_small<R>(size_t);                                                           \
  template cudaError_t launch_boundary_small<R>(const KArgs<R>&, const KArgs<R>*, const int*, int, int, R*, size_t, \
                                                size_t, int, cudaStream_t);
PEPS_INST(double)
PEPS_INST(float)

}  // namespace peps

#ifdef PEPS_PHASE_TIMING
// Diagnostic build only: the phase counters of the one-warp sweeps, as peps_phase_read.
extern "C" int peps_phase_read_small(unsigned long long* out, int reset) {
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  if (cudaMemcpyFromSymbol(out, ::peps_phase_cyc, 16 * sizeof(unsigned long long)) != cudaSuccess) return 1;
  if (reset) {
    const unsigned long long z[16] = {0};
    if (cudaMemcpyToSymbol(::peps_phase_cyc, z, sizeof(z)) != cudaSuccess) return 1;
  }
  return 0;
}
#endif

// Boundary-MPS sweeps (Fig. 1d) with one CTA per (configuration, direction), of
// one model (nm = 0: `one`) or of several (a packed launch: work items are
// numbered model after model, start[m] the first item of models[m], start[nm]
// their number; n * dirs items per model, direction-major, so that sweeps the
// environment cache skips do not leave half the CTAs idle).  Every CTA has one
// scratch slot of slot_elems reals and dynamic shared memory for the largest
// model; it lays both out again whenever its next item belongs to another
// model.  One kernel for both uses, so packed results are bit-identical.
#pragma once

#include "boundary_item.cuh"

namespace peps {

template <typename R>
__global__ void __launch_bounds__(kThreads) k_boundary(KArgs<R> one, const KArgs<R>* __restrict__ models,
                                                       const int* __restrict__ start, int nm, int dirs, R* scratch,
                                                       size_t slot_elems) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ R red[64];
  __shared__ uint64_t sp[kMaxWords];
  __shared__ int ones[kMaxDcD + 1];
  __shared__ double dred[kWarps];
  __shared__ R wv[kMaxDcD];
  for (int i = threadIdx.x; i <= kMaxDcD; i += blockDim.x) ones[i] = 1;
  const int total = nm > 0 ? start[nm] : one.n * dirs;
  int cur = -1;
  ZipBufs<R> zb;
  R* p = nullptr;
  for (int item = blockIdx.x; item < total; item += gridDim.x) {
    int m = cur < 0 ? 0 : cur;
    while (m + 1 < nm && start[m + 1] <= item) ++m;
    const KArgs<R>& a = nm > 0 ? models[m] : one;
    if (m != cur) {
      __syncthreads();
      p = scratch + (size_t)blockIdx.x * slot_elems;
      R* gsm;
      int* gism;
      smem_split<R>(smem_raw, a.g, true, a.smem_wm != 0, gsm, gism);
      carve_zip<R>(a.g, p, zb, a.smem_wm ? gsm : nullptr, red, dred, wv, gsm, gism);
      cur = m;
    }
    const int local = nm > 0 ? item - start[m] : item;
    boundary_item<R>(a, local % a.n, local / a.n, p, sp, ones,
                     [&](const R* Min, R* Mout, int r, int dir, bool lr, const int* bdin) {
                       return absorb_row<R>(a, Min, Mout, r, dir, lr, bdin, sp, zb, red);
                     });
  }
}

template <typename R>
int max_blocks_boundary(size_t smem) {
  int dev = 0, nsm = 0, nb = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  prefer_shared(k_boundary<R>, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_boundary<R>, kThreads, smem);
  if (nb < 1) nb = 1;
  return nsm * nb;
}

template <typename R>
cudaError_t launch_boundary(const KArgs<R>& one, const KArgs<R>* models_dev, const int* start_dev, int nm, int dirs,
                            R* scratch, size_t slot_elems, size_t smem, int grid, cudaStream_t st) {
  cudaError_t e = prefer_shared(k_boundary<R>, smem);
  if (e != cudaSuccess) return e;
  k_boundary<R><<<grid, kThreads, smem, st>>>(one, models_dev, start_dev, nm, dirs, scratch, slot_elems);
  return cudaGetLastError();
}

#define PEPS_BOUNDARY_INST(R)                                                                                        \
  template int max_blocks_boundary<R>(size_t);                                                                       \
  template cudaError_t launch_boundary<R>(const KArgs<R>&, const KArgs<R>*, const int*, int, int, R*, size_t, size_t, \
                                          int, cudaStream_t);

}  // namespace peps

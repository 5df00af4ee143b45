// Shared launches of the L-BFGS iteration over several problems (declared in
// wf_internal.h): the streaming kernels, each block locating its problem and its
// coordinates in that problem's own grid.
#include "wf_ops_impl.cuh"

#include "wf_multi.cuh"

template <typename T>
__global__ void __launch_bounds__(WF_COMB_THREADS, sizeof(T) == 4 ? WF_COMB_MINB : 2)
k_multi_comb(const __grid_constant__ WfMultiGrid r, const __grid_constant__ WfMultiArgs a, int mode) {
  WfBlk kb;
  const int q = wf_multi_block(r, kb);
  wf_lb_comb<T>(a.g[q], a.lb[q], a.b[q].part, mode, kb);
}

template <typename T>
__global__ void __launch_bounds__(WF_COMB_THREADS, sizeof(T) == 4 ? 4 : 2)
k_multi_qdots(const __grid_constant__ WfMultiGrid r, const __grid_constant__ WfMultiArgs a) {
  WfBlk kb;
  const int q = wf_multi_block(r, kb);
  wf_lb_qdots<T>(a.g[q], a.lb[q], a.b[q].part, kb);
}

template <typename T>
cudaError_t wf_launch_multi_comb(const WfMultiArgs& a, int mode, cudaStream_t st) {
  static int done = 0;
  const WfMultiGrid r = wf_multi_grid(a, [](const WfGeo& g) { return g.ncomb; });
  cudaError_t e = wfimpl::ensure_smem(k_multi_comb<T>, wf_comb_smem<T>(WF_MAXM), &done);
  if (e != cudaSuccess) return e;
  k_multi_comb<T><<<r.start[a.np], WF_COMB_THREADS, wf_comb_smem<T>(a.lb[0].m), st>>>(r, a, mode);
  return cudaGetLastError();
}

template <typename T>
cudaError_t wf_launch_multi_qdots(const WfMultiArgs& a, cudaStream_t st) {
  static int done = 0;
  const WfMultiGrid r = wf_multi_grid(a, [](const WfGeo& g) { return g.ncomb; });
  cudaError_t e = wfimpl::ensure_smem(k_multi_qdots<T>, wf_comb_smem<T>(WF_MAXM), &done);
  if (e != cudaSuccess) return e;
  k_multi_qdots<T><<<r.start[a.np], WF_COMB_THREADS, wf_comb_smem<T>(a.lb[0].m), st>>>(r, a);
  return cudaGetLastError();
}

#define WF_INSTANTIATE_MULTI(T)                                                               \
  template cudaError_t wf_launch_multi_comb<T>(const WfMultiArgs&, int, cudaStream_t);        \
  template cudaError_t wf_launch_multi_qdots<T>(const WfMultiArgs&, cudaStream_t);
WF_INSTANTIATE_MULTI(float)
WF_INSTANTIATE_MULTI(double)

WF_DBG_READER(multi)

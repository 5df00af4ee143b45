// Kernels and launchers of the register-resident stages (wf_reg.cuh) for one
// working type and length, instantiated by the translation units that include
// this file (WF_RG_INSTANTIATE).
#pragma once
#include "wf_ops_impl.cuh"
#include "wf_reg.cuh"

template <typename T, int C, int IN, int N, int TC>
__global__ void __launch_bounds__(WfRegCol<T, C, N, TC>::THREADS, wf_rg_minb<T, WfRegT<T, N, false>::NV>(WfRegCol<T, C, N, TC>::THREADS))
k_rg_colinv(WfGeo g, const void* src_, const T* sp_, long long sp_stride, void* scratch_, const void* tw_) {
  const int b = blockIdx.y;
  const size_t st = (size_t)C * N * (IN == WF_IN_PK ? g.h : g.h + 1);
  wf_rg_colinv<T, C, IN, N, TC>(g, (const V2<T>*)src_ + b * st, sp_ + (size_t)b * sp_stride,
                                (V2<T>*)scratch_ + (size_t)b * C * N * g.h, tw_, blockIdx.x * TC);
}
template <typename T, int C, int IN, int N, int TC>
__global__ void __launch_bounds__(WfRegCol<T, C, N, TC>::THREADS, wf_rg_minb<T, WfRegT<T, N, false>::NV>(WfRegCol<T, C, N, TC>::THREADS))
k_rg_colfwd(WfGeo g, const void* src_, const T* sp_, long long sp_stride, const void* scratch_, void* dst_,
            double* part, const void* tw_) {
  const int b = blockIdx.y;
  const size_t st = (size_t)C * N * (IN == WF_IN_PK ? g.h : g.h + 1);
  wf_rg_colfwd<T, C, IN, N, TC>(g, (const V2<T>*)src_ + b * st, sp_ + (size_t)b * sp_stride,
                                (const V2<T>*)scratch_ + (size_t)b * C * N * g.h, (V2<T>*)dst_ + b * st,
                                part + (size_t)b * WF_NSLOT * g.maxblk, tw_, blockIdx.x * TC, blockIdx.x);
}
template <typename T, int C, int N, int TC>
__global__ void __launch_bounds__(WfRegCol<T, C, N, TC>::THREADS, wf_rg_minb<T, WfRegT<T, N, false>::NV>(WfRegCol<T, C, N, TC>::THREADS))
k_rg_colsim(WfGeo g, const T* sp_, long long sp_stride, void* scratch_, const void* tw_) {
  const int b = blockIdx.y;
  wf_rg_colsim<T, C, N, TC>(g, sp_ + (size_t)b * sp_stride, (V2<T>*)scratch_ + (size_t)b * C * N * g.h, tw_,
                            blockIdx.x * TC);
}
template <typename T, int MODE, int NX>
__global__ void __launch_bounds__(256, wf_rg_minb<T, WfRegT<T, NX, true>::NV>(256))
k_rg_row(WfGeo g, void* scratch_, const void* d_, const void* w_, const void* aux_, void* out_, double* part,
         const void* tw_) {
  wf_rg_row<T, MODE, NX>(g, (V2<T>*)scratch_, (const T*)d_, (const T*)w_, (const T*)aux_, (T*)out_, part, tw_,
                         blockIdx.y, blockIdx.x, blockDim.x >> 5);
}

// The same stages on the direction P[next] of every map still iterating (device
// functions in wf_reg.cuh, shared with the launches over several problems).
template <typename T, int C, int N, int TC>
__global__ void __launch_bounds__(WfRegCol<T, C, N, TC>::THREADS, wf_rg_minb<T, WfRegT<T, N, false>::NV>(WfRegCol<T, C, N, TC>::THREADS))
k_rg_lb_colinv(WfGeo g, WfBufs b, WfLbBufs lb) {
  wf_rg_lb_colinv_map<T, C, N, TC>(g, b, lb, blockIdx.y, blockIdx.x);
}
template <typename T, int NX>
__global__ void __launch_bounds__(256, wf_rg_minb<T, WfRegT<T, NX, true>::NV>(256))
k_rg_lb_row(WfGeo g, WfBufs b, WfLbBufs lb) {
  wf_rg_lb_row_map<T, NX>(g, b, lb, blockIdx.y, blockIdx.x);
}
template <typename T, int C, int N, int TC>
__global__ void __launch_bounds__(WfRegCol<T, C, N, TC>::THREADS, wf_rg_minb<T, WfRegT<T, N, false>::NV>(WfRegCol<T, C, N, TC>::THREADS))
k_rg_lb_colfwd(WfGeo g, WfBufs b, WfLbBufs lb) {
  wf_rg_lb_colfwd_map<T, C, N, TC>(g, b, lb, blockIdx.y, blockIdx.x);
}

namespace {

// Raise a kernel's dynamic shared memory once per device (mask: one static per kernel).
template <typename K> cudaError_t rg_smem(K k, size_t bytes, int* mask) { return wfimpl::ensure_smem(k, bytes, mask); }

// f<TC>() of the tile width tc (one of the three widths of C channels).
template <typename T, int C, int N, class F>
cudaError_t rg_width(int tc, F&& f) {
  constexpr bool F64 = sizeof(T) == 8;
  constexpr int A = wf_rg_tc(N, C, 1, F64), B = wf_rg_tc(N, C, 2, F64), D = wf_rg_tc(N, C, 4, F64);
  if (tc == A) return f(std::integral_constant<int, A>());
  if (tc == B) return f(std::integral_constant<int, B>());
  if (tc == D) return f(std::integral_constant<int, D>());
  return cudaErrorInvalidValue;
}
template <typename T, int N, class F>
cudaError_t rg_shape(int C, int tc, F&& f) {
  return C == 1 ? rg_width<T, 1, N>(tc, [&](auto w) { return f(std::integral_constant<int, 1>(), w); })
                : rg_width<T, 2, N>(tc, [&](auto w) { return f(std::integral_constant<int, 2>(), w); });
}

template <typename T, int C, int IN, int N, int TC>
cudaError_t rg_colinv_k(const WfGeo& g, const WfBufs& b, const void* src, cudaStream_t st) {
  static int done = 0;
  typedef WfRegCol<T, C, N, TC> K;
  auto k = k_rg_colinv<T, C, IN, N, TC>;
  cudaError_t e = rg_smem(k, K::SMEM, &done);
  if (e != cudaSuccess) return e;
  k<<<dim3(g.ntile, b.B), K::THREADS, K::SMEM, st>>>(g, src, (const T*)b.sp, b.sp_stride, b.scratch, b.tw);
  return cudaGetLastError();
}
template <typename T, int C, int IN, int N, int TC>
cudaError_t rg_colfwd_k(const WfGeo& g, const WfBufs& b, const void* src, void* dst, cudaStream_t st) {
  static int done = 0;
  typedef WfRegCol<T, C, N, TC> K;
  auto k = k_rg_colfwd<T, C, IN, N, TC>;
  cudaError_t e = rg_smem(k, K::SMEM, &done);
  if (e != cudaSuccess) return e;
  k<<<dim3(g.ntile, b.B), K::THREADS, K::SMEM, st>>>(g, src, (const T*)b.sp, b.sp_stride, b.scratch, dst, b.part,
                                                      b.tw);
  return cudaGetLastError();
}
template <typename T, int C, int N, int TC>
cudaError_t rg_colsim_k(const WfGeo& g, const WfBufs& b, cudaStream_t st) {
  static int done = 0;
  typedef WfRegCol<T, C, N, TC> K;
  auto k = k_rg_colsim<T, C, N, TC>;
  cudaError_t e = rg_smem(k, K::SMEM, &done);
  if (e != cudaSuccess) return e;
  k<<<dim3(g.ntile, b.B), K::THREADS, K::SMEM, st>>>(g, (const T*)b.sp, b.sp_stride, b.scratch, b.tw);
  return cudaGetLastError();
}
template <typename T, int C, int N, int TC>
cudaError_t rg_lb_colinv_k(const WfGeo& g, const WfBufs& b, const WfLbBufs& lb, cudaStream_t st) {
  static int done = 0;
  typedef WfRegCol<T, C, N, TC> K;
  auto k = k_rg_lb_colinv<T, C, N, TC>;
  cudaError_t e = rg_smem(k, K::SMEM, &done);
  if (e != cudaSuccess) return e;
  k<<<dim3(g.ntile, b.B), K::THREADS, K::SMEM, st>>>(g, b, lb);
  return cudaGetLastError();
}
template <typename T, int C, int N, int TC>
cudaError_t rg_lb_colfwd_k(const WfGeo& g, const WfBufs& b, const WfLbBufs& lb, cudaStream_t st) {
  static int done = 0;
  typedef WfRegCol<T, C, N, TC> K;
  auto k = k_rg_lb_colfwd<T, C, N, TC>;
  cudaError_t e = rg_smem(k, K::SMEM, &done);
  if (e != cudaSuccess) return e;
  k<<<dim3(g.ntile, b.B), K::THREADS, K::SMEM, st>>>(g, b, lb);
  return cudaGetLastError();
}
template <typename T, int MODE, int NX>
cudaError_t rg_row_k(const WfGeo& g, const WfBufs& b, const void* aux, void* out, cudaStream_t st) {
  static int done = 0;
  typedef WfRegRow<T, NX> K;
  auto k = k_rg_row<T, MODE, NX>;
  cudaError_t e = rg_smem(k, K::smem(8), &done);
  if (e != cudaSuccess) return e;
  const int warps = g.RB / wf_rg_rows(NX, sizeof(T) == 8);
  k<<<dim3(g.nrb, b.B), 32 * warps, K::smem(warps), st>>>(g, b.scratch, b.d, b.w, aux, out, b.part, b.tw);
  return cudaGetLastError();
}

}  // namespace

template <typename T, int N>
cudaError_t wf_reg_colinv(const WfGeo& g, const WfBufs& b, int in, const void* src, cudaStream_t st) {
  return rg_shape<T, N>(g.C, g.TC, [&](auto c, auto w) {
    return in == WF_IN_PK ? rg_colinv_k<T, c(), WF_IN_PK, N, w()>(g, b, src, st)
                          : rg_colinv_k<T, c(), WF_IN_STD, N, w()>(g, b, src, st);
  });
}
template <typename T, int N>
cudaError_t wf_reg_colfwd(const WfGeo& g, const WfBufs& b, int in, const void* src, void* dst, cudaStream_t st) {
  return rg_shape<T, N>(g.C, g.TC, [&](auto c, auto w) {
    return in == WF_IN_PK ? rg_colfwd_k<T, c(), WF_IN_PK, N, w()>(g, b, src, dst, st)
                          : rg_colfwd_k<T, c(), WF_IN_STD, N, w()>(g, b, src, dst, st);
  });
}
template <typename T, int N>
cudaError_t wf_reg_colsim(const WfGeo& g, const WfBufs& b, cudaStream_t st) {
  return rg_shape<T, N>(g.C, g.TC, [&](auto c, auto w) { return rg_colsim_k<T, c(), N, w()>(g, b, st); });
}
template <typename T, int N>
cudaError_t wf_reg_lb_colinv(const WfGeo& g, const WfBufs& b, const WfLbBufs& lb, cudaStream_t st) {
  return rg_shape<T, N>(g.C, g.TC, [&](auto c, auto w) { return rg_lb_colinv_k<T, c(), N, w()>(g, b, lb, st); });
}
template <typename T, int N>
cudaError_t wf_reg_lb_colfwd(const WfGeo& g, const WfBufs& b, const WfLbBufs& lb, cudaStream_t st) {
  return rg_shape<T, N>(g.C, g.TC, [&](auto c, auto w) { return rg_lb_colfwd_k<T, c(), N, w()>(g, b, lb, st); });
}
template <typename T, int NX>
cudaError_t wf_reg_row(const WfGeo& g, const WfBufs& b, int mode, const void* aux, void* out, cudaStream_t st) {
  switch (mode) {
    case WF_ROW_DATA: return rg_row_k<T, WF_ROW_DATA, NX>(g, b, aux, out, st);
    case WF_ROW_NODATA: return rg_row_k<T, WF_ROW_NODATA, NX>(g, b, aux, out, st);
    case WF_ROW_SIGNAL: return rg_row_k<T, WF_ROW_SIGNAL, NX>(g, b, aux, out, st);
    case WF_ROW_SIM: return rg_row_k<T, WF_ROW_SIM, NX>(g, b, aux, out, st);
    case WF_ROW_RFFT: return rg_row_k<T, WF_ROW_RFFT, NX>(g, b, aux, out, st);
  }
  return cudaErrorInvalidValue;
}
template <typename T, int NX>
cudaError_t wf_reg_lb_row(const WfGeo& g, const WfBufs& b, const WfLbBufs& lb, cudaStream_t st) {
  static int done = 0;
  typedef WfRegRow<T, NX> K;
  auto k = k_rg_lb_row<T, NX>;
  cudaError_t e = rg_smem(k, K::smem(8), &done);
  if (e != cudaSuccess) return e;
  const int warps = g.RB / wf_rg_rows(NX, sizeof(T) == 8);
  k<<<dim3(g.nrb, b.B), 32 * warps, K::smem(warps), st>>>(g, b, lb);
  return cudaGetLastError();
}

#define WF_RG_INSTANTIATE(T, N)                                                                              \
  static_assert(wf_rg_rows(N, sizeof(T) == 8) == 2 * WfRegRow<T, N>::SEQ, "rows of a warp");                                 \
  template cudaError_t wf_reg_colinv<T, N>(const WfGeo&, const WfBufs&, int, const void*, cudaStream_t);     \
  template cudaError_t wf_reg_colfwd<T, N>(const WfGeo&, const WfBufs&, int, const void*, void*, cudaStream_t); \
  template cudaError_t wf_reg_colsim<T, N>(const WfGeo&, const WfBufs&, cudaStream_t);                       \
  template cudaError_t wf_reg_lb_colinv<T, N>(const WfGeo&, const WfBufs&, const WfLbBufs&, cudaStream_t);   \
  template cudaError_t wf_reg_lb_colfwd<T, N>(const WfGeo&, const WfBufs&, const WfLbBufs&, cudaStream_t);   \
  template cudaError_t wf_reg_row<T, N>(const WfGeo&, const WfBufs&, int, const void*, void*, cudaStream_t); \
  template cudaError_t wf_reg_lb_row<T, N>(const WfGeo&, const WfBufs&, const WfLbBufs&, cudaStream_t);

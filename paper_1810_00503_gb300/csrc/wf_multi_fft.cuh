// FFT stages of the L-BFGS iteration in launches shared by several problems
// (wf_map_solve_many), for one working type and channel count: every block finds
// its problem and runs the register-resident stage of that problem's length and
// tile width, so a batch of any mix of shapes takes three launches (a branch per
// problem instead, captured in the batch's graph, took 1.4 times as long on
// batches of few small maps: capturing and instantiating a node costs more than
// its kernel).  Blocks are as large as the widest stage's; threads a narrower one
// has no use for leave at once.
#pragma once
#include "wf_multi.cuh"
#include "wf_reg.cuh"

// f(N) of every length.
template <class F> constexpr void wf_multi_lengths(F& f) {
  f(std::integral_constant<int, 8>());
  f(std::integral_constant<int, 16>());
  f(std::integral_constant<int, 32>());
  f(std::integral_constant<int, 64>());
  f(std::integral_constant<int, 128>());
  f(std::integral_constant<int, 256>());
  f(std::integral_constant<int, 512>());
  f(std::integral_constant<int, 1024>());
}
// f<N>() of length n.
template <class F> __device__ __forceinline__ void wf_rg_switch(int n, F&& f) {
  switch (n) {
    case 8: f(std::integral_constant<int, 8>()); break;
    case 16: f(std::integral_constant<int, 16>()); break;
    case 32: f(std::integral_constant<int, 32>()); break;
    case 64: f(std::integral_constant<int, 64>()); break;
    case 128: f(std::integral_constant<int, 128>()); break;
    case 256: f(std::integral_constant<int, 256>()); break;
    case 512: f(std::integral_constant<int, 512>()); break;
    default: f(std::integral_constant<int, 1024>()); break;
  }
}

template <typename T, int C, bool INV>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1)
k_multi_col(const __grid_constant__ WfMultiGrid r, const __grid_constant__ WfMultiArgs a) {
  WfBlk kb;
  const int q = wf_multi_block(r, kb);
  wf_rg_switch(a.g[q].n, [&](auto n) {
    constexpr int N = decltype(n)::value;
    auto width = [&](auto w) {
      constexpr int TC = decltype(w)::value;
      if (threadIdx.x >= WfRegCol<T, C, N, TC>::THREADS) return;
      if constexpr (INV) wf_rg_lb_colinv_map<T, C, N, TC>(a.g[q], a.b[q], a.lb[q], kb.y, kb.x);
      else wf_rg_lb_colfwd_map<T, C, N, TC>(a.g[q], a.b[q], a.lb[q], kb.y, kb.x);
    };
    constexpr bool F64 = sizeof(T) == 8;
    constexpr int A = wf_rg_tc(N, C, 1, F64), B = wf_rg_tc(N, C, 2, F64);
    if (a.g[q].TC == A) width(std::integral_constant<int, A>());
    else width(std::integral_constant<int, B>());
  });
}
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1)
k_multi_row(const __grid_constant__ WfMultiGrid r, const __grid_constant__ WfMultiArgs a) {
  WfBlk kb;
  const int q = wf_multi_block(r, kb);
  if ((int)threadIdx.x >= 32 * (a.g[q].RB / wf_rg_rows(a.g[q].nx, sizeof(T) == 8))) return;
  wf_rg_switch(a.g[q].nx, [&](auto n) { wf_rg_lb_row_map<T, decltype(n)::value>(a.g[q], a.b[q], a.lb[q], kb.y, kb.x); });
}

// Shared memory of a problem's stages.
template <typename T> inline size_t wf_multi_col_smem(const WfGeo& g) {
  constexpr bool F64 = sizeof(T) == 8;
  size_t sm = 0;
  wfimpl::rg_length(g.n, [&](auto n) {
    const bool wide = g.TC == wf_rg_tc(n(), g.C, 1, F64);
    if (g.C == 1) sm = wide ? WfRegCol<T, 1, n(), wf_rg_tc(n(), 1, 1, F64)>::SMEM : WfRegCol<T, 1, n(), wf_rg_tc(n(), 1, 2, F64)>::SMEM;
    else sm = wide ? WfRegCol<T, 2, n(), wf_rg_tc(n(), 2, 1, F64)>::SMEM : WfRegCol<T, 2, n(), wf_rg_tc(n(), 2, 2, F64)>::SMEM;
    return cudaSuccess;
  });
  return sm;
}
template <typename T> inline size_t wf_multi_row_smem(const WfGeo& g) {
  size_t sm = 0;
  wfimpl::rg_length(g.nx, [&](auto n) {
    sm = WfRegRow<T, n()>::smem(g.RB / wf_rg_rows(g.nx, sizeof(T) == 8));
    return cudaSuccess;
  });
  return sm;
}

// The most shared memory a stage of any problem asks for: the widest column tiles
// of C channels, and row blocks of eight warps.  Neither is the length 1024's
// everywhere: FP32 rows of 512 have the largest row block.
template <typename T, int C> constexpr size_t wf_multi_col_max() {
  size_t m = 0;
  auto take = [&](auto n) {
    constexpr int N = decltype(n)::value;
    constexpr size_t s = WfRegCol<T, C, N, wf_rg_tc(N, C, 1, sizeof(T) == 8)>::SMEM;
    constexpr size_t t = WfRegCol<T, C, N, wf_rg_tc(N, C, 2, sizeof(T) == 8)>::SMEM;
    m = s > m ? s : m;
    m = t > m ? t : m;
  };
  wf_multi_lengths(take);
  return m;
}
template <typename T> constexpr size_t wf_multi_row_max() {
  size_t m = 0;
  auto take = [&](auto n) {
    constexpr size_t s = WfRegRow<T, decltype(n)::value>::smem(8);
    m = s > m ? s : m;
  };
  wf_multi_lengths(take);
  return m;
}

template <typename T, int C>
cudaError_t wf_launch_multi_fft(const WfMultiArgs& a, int stage, cudaStream_t st) {
  static int done[3] = {0, 0, 0};
  const bool row = stage == 1;
  const WfMultiGrid r = wf_multi_grid(a, [&](const WfGeo& g) { return row ? g.nrb : g.ntile; });
  size_t sm = 0;
  for (int q = 0; q < a.np; ++q) {
    const size_t s = row ? wf_multi_row_smem<T>(a.g[q]) : wf_multi_col_smem<T>(a.g[q]);
    if (s > sm) sm = s;
  }
  auto k = row ? k_multi_row<T> : stage == 0 ? k_multi_col<T, C, true> : k_multi_col<T, C, false>;
  constexpr size_t most_col = wf_multi_col_max<T, C>(), most_row = wf_multi_row_max<T>();
  cudaError_t e = wfimpl::ensure_smem(k, row ? most_row : most_col, &done[stage]);
  if (e != cudaSuccess) return e;
  k<<<r.start[a.np], 256, sm, st>>>(r, a);
  return cudaGetLastError();
}

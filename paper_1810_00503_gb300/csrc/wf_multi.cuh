// Blocks of a launch shared by several problems: problem q's own grid of gx by gy
// (its maps), concatenated over the problems.
#pragma once
#include "wf_ops_impl.cuh"

struct WfMultiGrid {
  int np;
  int start[WF_MULTI_MAX + 1];
  int gx[WF_MULTI_MAX];
  int gy[WF_MULTI_MAX];
};

// Problem of this block and its coordinates in the problem's grid.
__device__ __forceinline__ int wf_multi_block(const WfMultiGrid& r, WfBlk& kb) {
  const int bid = blockIdx.x;
  int q = 0;
  while (q + 1 < r.np && bid >= r.start[q + 1]) ++q;
  const int local = bid - r.start[q];
  kb.nx = r.gx[q];
  kb.ny = r.gy[q];
  kb.x = local % kb.nx;
  kb.y = local / kb.nx;
  return q;
}

// Grid of problem q's blocks: gx(q) x (its maps), concatenated over the problems.
template <class F>
inline WfMultiGrid wf_multi_grid(const WfMultiArgs& a, F gx) {
  WfMultiGrid r;
  r.np = a.np;
  r.start[0] = 0;
  for (int q = 0; q < a.np; ++q) {
    r.gx[q] = gx(a.g[q]);
    r.gy[q] = a.b[q].B;
    r.start[q + 1] = r.start[q] + r.gx[q] * r.gy[q];
  }
  return r;
}


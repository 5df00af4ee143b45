// Host-side structures of the C ABI (prepared problem, solver state; the handle is in
// wf_mem.h).
#pragma once
#include "wf_internal.h"
#include "wf_mem.h"

struct WfSolver;  // L-BFGS state, allocated on the first solve (wf_solve.cu)

struct wf_problem {
  wf_handle* h;
  int count, n, nx, C, dtype, precision, m;  // n = ny rows of nx pixels
  WfGeo g;               // of the solver's launches (the variant its last start chose)
  WfGeo gp;              // of the objective's passes
  size_t elt;            // bytes of the working type
  int sp_shared;         // one sqrt(P) table serves every map
  long long sp_stride;   // elements between maps' sqrt(P) tables
  void* d;               // [count][C][ny][nx] working type
  void* w;               // [count][C][ny][nx] mask * Ninv
  void* sp;              // [1 or count][C][ny][nx/2+1] sqrt(P/(ny nx)) (band-scaled if set)
  void* sp0;             // unscaled copy, kept once a band scale has been set
  void* scratch;         // [count][C][ny][nx/2] complex
  double* part;          // [count][WF_NSLOT][maxblk]
  int* flags;            // device status words
  double* bpart;         // band-sum partials [count][blocks][bands] (grown on demand)
  size_t bpart_n;        // doubles held by bpart
  WfSolver* solver;
};

WfBufs wf_bufs(const wf_problem* p);
void wf_solver_free(wf_problem* p);
void wf_make_twiddles(double2* out);  // WF_TWTAB entries: roots of unity and pass tables
// Normal deviates offset .. offset + count - 1 of (seed, stream_id) into out
// (working type); scaled by w^-1/2 where w > 0 and zeroed elsewhere if w given.
wf_status wf_draw_normal(unsigned long long seed, unsigned stream_id, unsigned long long offset, size_t count,
                         int working_f64, void* out, const void* w, cudaStream_t st);

// Host-side structures of the C ABI (handle, prepared problem, solver state).
#pragma once
#include <mutex>
#include <unordered_map>
#include <utility>
#include <vector>
#include "wf_internal.h"

struct wf_handle {
  int device;
  void* tw64;   // WF_TWTAB_ALL double2 twiddles (roots of unity, pass tables of every plan)
  void* tw32;   // WF_TWTAB_ALL float2 twiddles
  size_t limit;  // workspace limit in bytes (0 = none)
  size_t used;   // device bytes held by this handle's allocations
  // Memory pool of the handle's allocations up to WF_POOL_ONE bytes, so that a call
  // that allocates its work space (wf_eval_any, the band powers, a problem) does not
  // map and unmap device memory each time: 64 maps of 768^2 1.03 -> 0.73 ms a
  // wf_eval_any call, a band-power estimate of 39 E/B maps of 256^2 4.87 -> 3.36 ms.
  // At most WF_POOL_KEEP freed bytes stay in it (none with a workspace limit), until
  // wf_destroy or an allocation that fails without them.
  // Allocations and frees are ordered on a stream of the pool's own, and a buffer is
  // freed only when nothing uses it any more, so any stream and thread may use the
  // handle's buffers as before.  nullptr: plain cudaMalloc.
  cudaMemPool_t pool;
  cudaStream_t pool_stream;
  std::vector<std::pair<void*, size_t>> pinned;  // freed pinned host buffers, at most WF_PINNED_KEEP
  std::mutex mu;
  std::unordered_map<void*, size_t> live;  // allocation -> bytes
  std::unordered_map<long long, int> tuned;  // (ny, nx, C, precision, maps) -> FFT-stage variant
};

#define WF_POOL_ONE (256ull << 20)
#define WF_POOL_KEEP (1ull << 30)
#define WF_PINNED_KEEP 8

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

wf_status wf_fail(wf_status s, const char* fmt, ...);
wf_status wf_cuda_fail(cudaError_t e, const char* what);
// Device allocation charged to the handle's workspace (WF_ENOMEM beyond its
// limit), and its release; wf_free(h, nullptr) does nothing.  wf_free waits for the
// device, as cudaFree does; wf_free_idle is for buffers whose last use the caller has
// already waited for.
wf_status wf_alloc(wf_handle* h, void** ptr, size_t bytes, const char* what);
void wf_free(wf_handle* h, void* ptr);
void wf_free_idle(wf_handle* h, void* ptr);
// Small pinned host buffers, kept by the handle for the next caller (a pinned
// allocation takes longer than a short solve); not charged to the workspace.
cudaError_t wf_pinned_alloc(wf_handle* h, void** ptr, size_t bytes);
void wf_pinned_free(wf_handle* h, void* ptr, size_t bytes);
WfBufs wf_bufs(const wf_problem* p);
void wf_solver_free(wf_problem* p);
void wf_make_twiddles(double2* out);  // WF_TWTAB entries: roots of unity and pass tables
// Normal deviates offset .. offset + count - 1 of (seed, stream_id) into out
// (working type); scaled by w^-1/2 where w > 0 and zeroed elsewhere if w given.
wf_status wf_draw_normal(unsigned long long seed, unsigned stream_id, unsigned long long offset, size_t count,
                         int working_f64, void* out, const void* w, cudaStream_t st);

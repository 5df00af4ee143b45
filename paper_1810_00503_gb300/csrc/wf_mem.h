// The library handle and its device memory (wf_mem.cu).  Host code only: it names
// no kernel, so that it can be compiled and tested against a fake runtime.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include <mutex>
#include <unordered_map>
#include <utility>
#include <vector>

#include "../../include/wf.h"

struct wf_handle {
  int device;
  void* tw64;   // WF_TWTAB_ALL double2 twiddles (roots of unity, pass tables of every plan)
  void* tw32;   // WF_TWTAB_ALL float2 twiddles
  size_t limit;  // workspace limit in bytes (0 = none)
  size_t used;   // device bytes held by this handle's allocations
  // Memory pool of the handle's allocations up to WF_POOL_ONE bytes made while its
  // device is current (wf_eval_any runs on the current one, whatever the handle's),
  // so that a call that allocates its work space (wf_eval_any, the band powers, a
  // problem) does not map and unmap device memory each time: 64 maps of 768^2 1.03 ->
  // 0.73 ms a wf_eval_any call, a band-power estimate of 39 E/B maps of 256^2 4.87 ->
  // 3.36 ms.
  // At most WF_POOL_KEEP freed bytes stay in it (none with a workspace limit), until
  // wf_destroy or until an allocation of any handle, from a pool or not, fails
  // without them.  They are not in `used`, and other allocators of the process
  // cannot reach them.
  // Allocations and frees are ordered on a stream of the pool's own, and a buffer is
  // freed only when nothing uses it any more, so any stream and thread may use the
  // handle's buffers as before.  nullptr: plain cudaMalloc.
  cudaMemPool_t pool;
  cudaStream_t pool_stream;
  std::vector<std::pair<void*, size_t>> pinned;  // freed pinned host buffers, at most WF_PINNED_KEEP
  std::mutex mu;
  struct Block {
    size_t bytes;
    bool pooled;
  };
  std::unordered_map<void*, Block> live;  // the handle's allocations
  std::unordered_map<long long, int> tuned;  // (ny, nx, C, precision, maps) -> FFT-stage variant
};

#define WF_POOL_ONE (256ull << 20)
#define WF_POOL_KEEP (1ull << 30)
#define WF_PINNED_KEEP 8

wf_status wf_fail(wf_status s, const char* fmt, ...);
wf_status wf_cuda_fail(cudaError_t e, const char* what);

// Pool of a handle whose device and limit are set, and its end.
void wf_mem_open(wf_handle* h);
void wf_mem_close(wf_handle* h);
// Allocation on the current device, charged to the handle's workspace (WF_ENOMEM
// beyond its limit), and its release; null pointers are skipped.  wf_free and wf_free_all
// first wait for the handle's device, whichever device is current, and wf_free_all
// says whether that wait succeeded; wf_free_idle is for buffers whose last use the
// caller has already waited for.
wf_status wf_alloc(wf_handle* h, void** ptr, size_t bytes, const char* what);
void wf_free(wf_handle* h, void* ptr);
bool wf_free_all(wf_handle* h, void* const* ptrs, int n);
void wf_free_idle(wf_handle* h, void* ptr);
// Small pinned host buffers, kept by the handle for the next caller (a pinned
// allocation takes longer than a short solve); not charged to the workspace.  idle:
// no copy of the device's still uses the buffer.
cudaError_t wf_pinned_alloc(wf_handle* h, void** ptr, size_t bytes);
void wf_pinned_free(wf_handle* h, void* ptr, size_t bytes, bool idle);

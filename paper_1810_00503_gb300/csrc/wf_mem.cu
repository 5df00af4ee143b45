// Device and pinned memory of a handle: the pool, the workspace's account and the
// wait before a buffer is given back.
#include <string.h>

#include <algorithm>

#include "wf_mem.h"

// Handles whose pools may hold freed memory; never destroyed, as a handle may be
// closed while the process ends.
static std::mutex g_open_mu;
static std::vector<wf_handle*>& g_open = *new std::vector<wf_handle*>();

// Without pool support the handle allocates plainly.
void wf_mem_open(wf_handle* h) {
  cudaMemPoolProps pr;
  memset(&pr, 0, sizeof pr);
  pr.allocType = cudaMemAllocationTypePinned;
  pr.location.type = cudaMemLocationTypeDevice;
  pr.location.id = h->device;
  h->pool = nullptr;
  if (cudaStreamCreateWithFlags(&h->pool_stream, cudaStreamNonBlocking) != cudaSuccess) {
    h->pool_stream = nullptr;
  } else if (cudaMemPoolCreate(&h->pool, &pr) != cudaSuccess) {
    h->pool = nullptr;
  } else {
    unsigned long long keep = h->limit ? 0 : WF_POOL_KEEP;
    cudaMemPoolSetAttribute(h->pool, cudaMemPoolAttrReleaseThreshold, &keep);
  }
  cudaGetLastError();
  std::lock_guard<std::mutex> lock(g_open_mu);
  g_open.push_back(h);
}
void wf_mem_close(wf_handle* h) {
  {
    std::lock_guard<std::mutex> lock(g_open_mu);
    g_open.erase(std::remove(g_open.begin(), g_open.end(), h), g_open.end());
  }
  if (h->pool_stream) cudaStreamSynchronize(h->pool_stream);
  if (h->pool) cudaMemPoolDestroy(h->pool);
  if (h->pool_stream) cudaStreamDestroy(h->pool_stream);
  for (auto& q : h->pinned) cudaFreeHost(q.first);
}

// Which allocations come from the pool.  Larger ones gain nothing that matters beside
// the work they are for, and take 3 ms more to map for a history ring of 10 GB; with
// another device current than the handle's, the memory has to be that device's.
static bool pooled(const wf_handle* h, size_t bytes) {
  int dev = -1;
  return h->pool && bytes <= WF_POOL_ONE && cudaGetDevice(&dev) == cudaSuccess && dev == h->device;
}

// Give back what the pools of every handle of device dev keep.
static void trim_pools(int dev) {
  std::lock_guard<std::mutex> lock(g_open_mu);
  for (wf_handle* h : g_open)
    if (h->pool && h->device == dev) {
      cudaStreamSynchronize(h->pool_stream);  // frees still on their way are given back too
      cudaMemPoolTrimTo(h->pool, 0);
    }
}

// One attempt at an allocation on the current device.
static cudaError_t allocate(wf_handle* h, void** ptr, size_t bytes, bool pool) {
  if (!pool) return cudaMalloc(ptr, bytes);
  cudaError_t e = cudaMallocFromPoolAsync(ptr, bytes, h->pool, h->pool_stream);
  if (e != cudaSuccess) return e;
  e = cudaStreamSynchronize(h->pool_stream);  // usable on every stream from here
  if (e != cudaSuccess) cudaFreeAsync(*ptr, h->pool_stream);  // refused, as during a capture: nothing has used it
  return e;
}

wf_status wf_alloc(wf_handle* h, void** ptr, size_t bytes, const char* what) {
  *ptr = nullptr;
  {
    std::lock_guard<std::mutex> lock(h->mu);
    if (h->limit && h->used + bytes > h->limit)
      return wf_fail(WF_ENOMEM, "%s: %zu more bytes would exceed the workspace limit (%zu of %zu in use)", what,
                     bytes, h->used, h->limit);
    h->used += bytes;  // reserved before the allocation, so concurrent callers cannot overshoot
  }
  const bool pool = pooled(h, bytes);
  cudaError_t e = allocate(h, ptr, bytes, pool);
  int dev = 0;
  if (e == cudaErrorMemoryAllocation && cudaGetDevice(&dev) == cudaSuccess) {  // once more without what the pools keep
    cudaGetLastError();
    trim_pools(dev);
    e = allocate(h, ptr, bytes, pool);
  }
  if (e != cudaSuccess) {
    *ptr = nullptr;
    cudaGetLastError();
    std::lock_guard<std::mutex> lock(h->mu);
    h->used -= bytes;
    return wf_fail(e == cudaErrorMemoryAllocation ? WF_ENOMEM : WF_ECUDA,
                   "device allocation of %zu bytes for %s failed: %s", bytes, what,
                   cudaGetErrorString(e));
  }
  std::lock_guard<std::mutex> lock(h->mu);
  h->live[*ptr] = {bytes, pool};
  return WF_OK;
}

// Wait for everything queued on the handle's device.  The caller may have another
// one current (a problem closed by a garbage collector, say).
static bool wait_idle(wf_handle* h) {
  int dev = h->device;
  cudaGetDevice(&dev);
  cudaError_t e = cudaSuccess;
  if (dev != h->device) e = cudaSetDevice(h->device);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (dev != h->device) cudaSetDevice(dev);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess;
}

// Take a buffer off the handle's account and release it.  A buffer of the pool goes
// to the next caller at once, so one that may still be in use (idle false: the wait
// failed, as during a capture or after an error of the device) is not given back;
// cudaFree waits by itself.
static void release(wf_handle* h, void* ptr, bool idle) {
  if (!ptr) return;
  wf_handle::Block b = {0, false};
  {
    std::lock_guard<std::mutex> lock(h->mu);
    auto it = h->live.find(ptr);
    if (it != h->live.end()) {
      b = it->second;
      h->live.erase(it);
    }
  }
  if (!b.pooled) cudaFree(ptr);
  else if (idle) cudaFreeAsync(ptr, h->pool_stream);
  std::lock_guard<std::mutex> lock(h->mu);
  h->used -= b.bytes;
}

bool wf_free_all(wf_handle* h, void* const* ptrs, int n) {
  const bool idle = wait_idle(h);
  for (int i = 0; i < n; ++i) release(h, ptrs[i], idle);
  return idle;
}

void wf_free(wf_handle* h, void* ptr) {
  if (ptr) wf_free_all(h, &ptr, 1);
}

void wf_free_idle(wf_handle* h, void* ptr) { release(h, ptr, true); }

cudaError_t wf_pinned_alloc(wf_handle* h, void** ptr, size_t bytes) {
  {
    std::lock_guard<std::mutex> lock(h->mu);
    for (size_t i = 0; i < h->pinned.size(); ++i)
      if (h->pinned[i].second == bytes) {
        *ptr = h->pinned[i].first;
        h->pinned.erase(h->pinned.begin() + i);
        return cudaSuccess;
      }
  }
  return cudaMallocHost(ptr, bytes);
}

void wf_pinned_free(wf_handle* h, void* ptr, size_t bytes, bool idle) {
  if (!ptr) return;
  if (idle) {
    std::lock_guard<std::mutex> lock(h->mu);
    if (h->pinned.size() < WF_PINNED_KEEP) {
      h->pinned.emplace_back(ptr, bytes);
      return;
    }
  }
  cudaFreeHost(ptr);
}

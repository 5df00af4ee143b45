// Drives the handle's memory (csrc/wf_mem.cu) against a fake CUDA runtime of two
// devices, defined here: no GPU and no CUDA library.  Every device has a flag for
// queued work, which a wait for that device clears, an amount of memory, and the
// bytes its pools keep; buffers remember their device.  Usage: mem_driver TEST;
// prints what was wrong and returns 1.
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>

#include "wf_mem.h"

struct Buf { int dev; size_t bytes; cudaMemPool_t pool; };
struct Pool { int dev; unsigned long long keep; size_t kept; };
static int g_cur = 0, g_violations = 0;
static bool g_busy[2], g_sync_fails = false;
static size_t g_room[2] = {1ull << 40, 1ull << 40};  // bytes neither allocated nor kept by a pool
static std::map<void*, Buf> g_live;

static void* block(int dev, size_t bytes, cudaMemPool_t pool) {
  void* p = malloc(16);
  g_live[p] = Buf{dev, bytes, pool};
  return p;
}
extern "C" {
cudaError_t CUDARTAPI cudaGetDevice(int* d) { *d = g_cur; return cudaSuccess; }
cudaError_t CUDARTAPI cudaSetDevice(int d) { g_cur = d; return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetLastError() { return cudaSuccess; }
const char* CUDARTAPI cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t CUDARTAPI cudaDeviceSynchronize() {
  if (g_sync_fails) return cudaErrorStreamCaptureUnsupported;
  g_busy[g_cur] = false;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamSynchronize(cudaStream_t) {
  return g_sync_fails ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
cudaError_t CUDARTAPI cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps* pr) {
  *p = (cudaMemPool_t) new Pool{pr->location.id, 0, 0};
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMemPoolSetAttribute(cudaMemPool_t p, cudaMemPoolAttr, void* v) {
  ((Pool*)p)->keep = *(unsigned long long*)v;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMemPoolTrimTo(cudaMemPool_t p, size_t) {
  Pool* q = (Pool*)p;
  g_room[q->dev] += q->kept;
  q->kept = 0;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMemPoolDestroy(cudaMemPool_t p) {
  cudaMemPoolTrimTo(p, 0);
  delete (Pool*)p;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMalloc(void** p, size_t bytes) {
  if (bytes > g_room[g_cur]) return cudaErrorMemoryAllocation;
  g_room[g_cur] -= bytes;
  *p = block(g_cur, bytes, nullptr);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMallocFromPoolAsync(void** p, size_t bytes, cudaMemPool_t pool, cudaStream_t) {
  Pool* q = (Pool*)pool;
  const size_t reuse = bytes < q->kept ? bytes : q->kept;
  if (bytes - reuse > g_room[q->dev]) return cudaErrorMemoryAllocation;
  q->kept -= reuse;
  g_room[q->dev] -= bytes - reuse;
  *p = block(q->dev, bytes, pool);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaFree(void* p) {  // waits for the buffer's device, and fails where a wait does
  const Buf b = g_live.at(p);
  if (g_sync_fails) return cudaErrorStreamCaptureUnsupported;
  if (b.pool) ++g_violations;  // of a pool's buffer it would not wait
  g_busy[b.dev] = false;
  g_room[b.dev] += b.bytes;
  g_live.erase(p);
  free(p);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaFreeAsync(void* p, cudaStream_t) {
  const Buf b = g_live.at(p);
  if (!b.pool || g_busy[b.dev]) ++g_violations;  // handed on while queued work still uses it
  Pool* q = (Pool*)b.pool;
  q->kept += b.bytes;
  if (q->kept > q->keep) {
    g_room[q->dev] += q->kept - q->keep;
    q->kept = q->keep;
  }
  g_live.erase(p);
  free(p);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMallocHost(void** p, size_t bytes) { *p = malloc(bytes); return cudaSuccess; }
cudaError_t CUDARTAPI cudaFreeHost(void* p) { free(p); return cudaSuccess; }
}
wf_status wf_fail(wf_status s, const char*, ...) { return s; }
wf_status wf_cuda_fail(cudaError_t, const char*) { return WF_ECUDA; }

#define CHECK(c) do { if (!(c)) { printf("%s:%d: %s\n", __func__, __LINE__, #c); return 1; } } while (0)
static void open(wf_handle* h, int dev) {
  h->device = dev;
  h->limit = h->used = 0;
  g_cur = dev;
  wf_mem_open(h);
}

// Buffers released while another device is current: the handle's own is waited for.
static int other_device() {
  wf_handle h;
  open(&h, 0);
  void *a, *b, *c, *big;
  CHECK(wf_alloc(&h, &a, 1 << 20, "a") == WF_OK && wf_alloc(&h, &b, 1 << 20, "b") == WF_OK);
  CHECK(wf_alloc(&h, &c, 1 << 20, "c") == WF_OK && wf_alloc(&h, &big, WF_POOL_ONE + 1, "big") == WF_OK);
  for (int cur = 1; cur >= 0; --cur) {
    void* one = cur ? a : b;
    g_cur = cur;
    g_busy[0] = g_busy[1] = true;
    wf_free(&h, one);
    CHECK(!g_violations && !g_busy[0] && g_cur == cur);
    CHECK(g_busy[1] || cur == 1);
  }
  g_cur = 1;
  g_busy[0] = true;
  void* rest[] = {c, nullptr, big};
  CHECK(wf_free_all(&h, rest, 3));
  CHECK(!g_violations && !g_busy[0] && g_cur == 1 && h.used == 0 && g_live.empty());
  wf_mem_close(&h);
  return 0;
}

// A wait that fails (a capture in progress): the pool does not get the buffer back,
// and a pinned one is not kept for the next caller.
static int failed_wait() {
  wf_handle h;
  open(&h, 0);
  void *a, *p;
  CHECK(wf_alloc(&h, &a, 1 << 20, "a") == WF_OK && wf_pinned_alloc(&h, &p, 64) == cudaSuccess);
  g_busy[0] = g_sync_fails = true;
  const bool idle = wf_free_all(&h, &a, 1);
  wf_pinned_free(&h, p, 64, idle);
  CHECK(!idle && !g_violations && g_live.count(a) && h.pinned.empty() && h.used == 0);
  g_sync_fails = false;
  wf_mem_close(&h);
  return 0;
}

// Memory asked for while another device is current is that device's.
static int current_device() {
  wf_handle h;
  open(&h, 0);
  void *a, *b;
  CHECK(wf_alloc(&h, &a, 1 << 20, "a") == WF_OK && g_live.at(a).dev == 0 && g_live.at(a).pool);
  g_cur = 1;
  CHECK(wf_alloc(&h, &b, 1 << 20, "b") == WF_OK && g_live.at(b).dev == 1);
  g_busy[0] = g_busy[1] = true;
  g_cur = 0;
  wf_free(&h, b);
  g_busy[0] = true;
  g_cur = 1;
  wf_free(&h, a);
  CHECK(!g_violations && !g_busy[0] && !g_busy[1] && h.used == 0 && g_live.empty());
  wf_mem_close(&h);
  return 0;
}

// What the pools keep is given back when an allocation fails without it: one from a
// pool, one too large for a pool, and one of another handle; one that does not fit
// all the same stays refused and uncharged.
static int trims() {
  const size_t one = WF_POOL_ONE, most = 4 * one;
  g_room[0] = most;
  wf_handle h, k;
  open(&h, 0);
  open(&k, 0);
  for (int round = 0; round < 3; ++round) {
    void *a[3], *b;
    for (void*& p : a) CHECK(wf_alloc(&h, &p, one, "a") == WF_OK);
    CHECK(wf_free_all(&h, a, 3) && g_room[0] == one);
    wf_handle* who = round == 2 ? &k : &h;
    if (round == 0) {  // from the pool, while a buffer of 3 is in use elsewhere
      g_room[0] = 0;
      ((Pool*)h.pool)->kept = one / 2;
      ((Pool*)k.pool)->kept = one / 2;
      CHECK(wf_alloc(&h, &b, one, "b") == WF_OK);
      wf_free(&h, b);
      g_room[0] = one;
      ((Pool*)h.pool)->kept = 3 * one;
      ((Pool*)k.pool)->kept = 0;
    }
    CHECK(wf_alloc(who, &b, 2 * one, "b") == WF_OK);
    const size_t used = who->used;
    void* c;
    CHECK(wf_alloc(who, &c, 3 * one, "c") == WF_ENOMEM && !c && who->used == used);
    wf_free(who, b);
    CHECK(who->used == 0);
  }
  wf_mem_close(&k);
  wf_mem_close(&h);
  CHECK(g_room[0] == most && g_live.empty());
  return 0;
}

// An allocation whose wait is refused (a capture in progress) leaves nothing behind.
static int refused() {
  wf_handle h;
  open(&h, 0);
  void* a;
  g_sync_fails = true;
  CHECK(wf_alloc(&h, &a, 1 << 20, "a") == WF_ECUDA && !a && h.used == 0 && g_live.empty());
  g_sync_fails = false;
  CHECK(wf_alloc(&h, &a, 1 << 20, "a") == WF_OK);
  wf_free(&h, a);
  CHECK(h.used == 0 && g_live.empty());
  wf_mem_close(&h);
  return 0;
}

int main(int argc, char** argv) {
  const std::string t = argc > 1 ? argv[1] : "";
  if (t == "other_device") return other_device();
  if (t == "failed_wait") return failed_wait();
  if (t == "current_device") return current_device();
  if (t == "trims") return trims();
  if (t == "refused") return refused();
  printf("unknown test\n");
  return 2;
}

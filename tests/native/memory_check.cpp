// Host-side check of where contexts take their result words from (run by
// tests/test_memory_cpu.py; no GPU needed): hsg_memory.cu linked against the
// runtime calls it makes, faked here.  The fake's contexts can be reset: the
// handle and the pinned addresses come back, the context's id does not.
//
//  * No two users hold the same words, over pages, contexts and resets.
//  * A page is freed only when nobody holds a word of it, in its own context.
//  * Words of a context that is gone can be given back without a trace.
// Prints "ok" and returns 0, or prints the first mismatch and returns 1.
#include <cstdio>
#include <cstring>
#include <map>
#include <set>
#include <vector>

#include "hsg_internal.h"

namespace {

unsigned long long g_id = 1;      // the current context's id; its handle is always the same
std::vector<char*> g_free_pages;  // lowest first: addresses are reused
std::set<char*> g_pages;          // live pinned pages of the current context
int failures = 0;

void fail(const char* what) {
  if (failures++ < 10) std::printf("FAIL %s\n", what);
}

CUresult fake_current(CUcontext* c) {
  *c = reinterpret_cast<CUcontext>(0x1000);
  return CUDA_SUCCESS;
}
CUresult fake_id(CUcontext, unsigned long long* id) {
  *id = g_id;
  return CUDA_SUCCESS;
}

void reset_device() {
  ++g_id;
  g_free_pages.insert(g_free_pages.begin(), g_pages.begin(), g_pages.end());
  g_pages.clear();
}

}  // namespace

extern "C" {
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** p, unsigned int, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *p = !std::strcmp(name, "cuCtxGetId") ? reinterpret_cast<void*>(&fake_id) : reinterpret_cast<void*>(&fake_current);
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
  *p = reinterpret_cast<cudaMemPool_t>(0x2000);
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr, void* v) {
  std::memset(v, 0, sizeof(unsigned long long));
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaMallocAsync(void**, size_t, cudaStream_t) { return cudaErrorMemoryAllocation; }
cudaError_t cudaMallocFromPoolAsync(void**, size_t, cudaMemPool_t, cudaStream_t) { return cudaErrorMemoryAllocation; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
  *f = *t = (size_t)1 << 34;
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t bytes) {
  if (bytes > 4096 || g_free_pages.empty()) return cudaErrorMemoryAllocation;
  g_pages.insert(g_free_pages.front());
  *p = g_free_pages.front();
  g_free_pages.erase(g_free_pages.begin());
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  if (!g_pages.erase(static_cast<char*>(p))) {
    fail("cudaFreeHost of what is not a live page");
    return cudaErrorInvalidValue;
  }
  g_free_pages.insert(g_free_pages.begin(), static_cast<char*>(p));
  return cudaSuccess;
}
}

namespace {

std::map<double*, int> g_held;  // live words of the current context

hsg::ResultWords take() {
  hsg::ResultWords w{};
  if (hsg::take_result_words(&w) != cudaSuccess || !w.p) fail("take");
  if (g_held[w.p]++) fail("words handed out twice");
  return w;
}
void give(const hsg::ResultWords& w) {
  g_held.erase(w.p);
  hsg::give_result_words(w);
  for (auto& h : g_held) {  // everyone else's words are still in a live page
    auto it = g_pages.upper_bound(reinterpret_cast<char*>(h.first));
    if (it == g_pages.begin() || reinterpret_cast<char*>(h.first) >= *--it + 4096) {
      fail("a page was freed under its users");
      return;
    }
  }
}

}  // namespace

int main() {
  static char pages[64][4096];
  for (auto& p : pages) g_free_pages.push_back(p);
  // 300 users (three pages), two thirds of whom are left when the device is reset
  std::vector<hsg::ResultWords> before, now;
  for (int k = 0; k < 300; ++k) before.push_back(take());
  for (int k = 0; k < 300; k += 3) give(before[k]);
  if (g_pages.size() != 3) fail("three pages for 300 users");
  reset_device();
  g_held.clear();
  // the same addresses in the new context, of which words come and go
  for (int k = 0; k < 300; ++k) now.push_back(take());
  for (int k = 0; k < 300; k += 2) give(now[k]);
  for (int k = 0; k < 300; k += 2) now[k] = take();
  if (g_pages.size() != 3) fail("given words are taken again");
  // users of the old context are closed only now
  for (int k = 0; k < 300; ++k)
    if (k % 3) hsg::give_result_words(before[k]);
  for (int k = 0; k < 300; ++k) now.push_back(take());
  for (int k = 129; k < 600; ++k) give(now[k]);
  for (int k = 0; k < 129; ++k) give(now[k]);
  if (g_pages.size() != 1) fail("empty pages but the first are freed");
  // more resets than there are records
  for (int r = 0; r < 200; ++r) {
    reset_device();
    g_held.clear();
    const hsg::ResultWords a = take(), b = take();
    if (!a.ctx_id) fail("a context after many resets has its pages");
    give(a);
    give(b);
  }
  if (failures) return 1;
  std::printf("ok\n");
  return 0;
}

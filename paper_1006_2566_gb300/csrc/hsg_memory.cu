// hsg_memory.cu -- where contexts take their device memory and pinned result
// words from (host code).
//
// A program that solves one sample after another creates and destroys a
// context per sample.  From the default memory pool, which gives everything
// back to the operating system at the next synchronisation, and with
// cudaMallocHost for two result words, that cost more than the sweeps of a
// small lattice: creation 255 us and destruction 277 us at L = 48, 421 and 890 us
// at L = 192.  So each device has one memory pool of the library's own, which keeps
// freed memory for the next context, up to one part in kKeepShare of the device's
// (555 MiB of GB300's 278 GiB: what a program does not miss; what a larger context frees
// beyond it is given back at the next synchronisation and mapped anew by the next).
// All of it goes back when an allocation would fail for want of it -- ours trim
// the pool, the driver takes it for everyone else's in this process (a pool, torch and
// cudaMallocAsync were each given more than was free) -- or by hsg_release_memory.  The
// result words are cut from pinned pages, given back once none of a page is
// in use (the first page stays).  Both are kept per CUDA context under one lock, by
// the context's id: after a device reset the handles and the addresses come back,
// the ids do not.  Words are given back to the context that they came from; of
// one that is gone nothing is touched.  Stream order is CUDA's.
#include <cstdint>
#include <mutex>

#include "hsg_internal.h"

namespace hsg {
namespace {

constexpr unsigned long long kKeepShare = 512;
constexpr int kWordBytes = 32, kPageBytes = 4096, kSlots = kPageBytes / kWordBytes;
constexpr int kPages = 64;

struct Page {
  char* base;
  uint64_t used[kSlots / 64];
};
struct Device {
  CUcontext ctx;
  unsigned long long ctx_id;  // 1, 2, ... in CUDA's own count
  cudaMemPool_t pool;
  Page pages[kPages];
};

std::mutex g_mu;
Device g_devices[kMaxDevices];
int g_n = 0;

using CtxGetCurrentFn = CUresult (*)(CUcontext*);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long*);

template <class F>
F driver_function(const char* name) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
  if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return reinterpret_cast<F>(p);
}

// The current CUDA context and its id; false: none, or no such entry points.
bool current_context(CUcontext* ctx, unsigned long long* id) {
  static const CtxGetCurrentFn get_current = driver_function<CtxGetCurrentFn>("cuCtxGetCurrent");
  static const CtxGetIdFn get_id = driver_function<CtxGetIdFn>("cuCtxGetId");
  *ctx = nullptr;
  return get_current && get_id && get_current(ctx) == CUDA_SUCCESS && *ctx && get_id(*ctx, id) == CUDA_SUCCESS;
}

Device* find_device(unsigned long long id) {
  for (int i = 0; i < g_n; ++i)
    if (g_devices[i].ctx_id == id) return &g_devices[i];
  return nullptr;
}

// The current CUDA context's record (g_mu held), or nullptr: no such entry
// points, or more contexts at a time than there are records.  A record with
// this context's handle and another id is of a context that is gone: reused.
Device* current_device() {
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (cudaFree(nullptr) != cudaSuccess || !current_context(&ctx, &id)) return nullptr;
  if (Device* known = find_device(id)) return known;
  int slot = 0, dev = 0;
  while (slot < g_n && g_devices[slot].ctx != ctx) ++slot;
  if (slot == kMaxDevices || cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  Device d = {};
  d.ctx = ctx;
  d.ctx_id = id;
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  unsigned long long keep = total_b / kKeepShare;
  if (cudaMemPoolCreate(&d.pool, &props) != cudaSuccess ||
      cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
    cudaGetLastError();
    if (d.pool) cudaMemPoolDestroy(d.pool);
    return nullptr;
  }
  g_devices[slot] = d;
  if (slot == g_n) ++g_n;
  return &g_devices[slot];
}

}  // namespace

cudaError_t device_alloc(void** p, size_t bytes, cudaStream_t s) {
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    if (Device* d = current_device()) pool = d->pool;
  }
  if (!pool) return cudaMallocAsync(p, bytes, s);
  cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, s);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    cudaMemPoolTrimTo(pool, 0);
    e = cudaMallocFromPoolAsync(p, bytes, pool, s);
  }
  return e;
}

size_t kept_bytes() {
  std::lock_guard<std::mutex> lock(g_mu);
  Device* d = current_device();
  unsigned long long reserved = 0, used = 0;
  if (!d || cudaMemPoolGetAttribute(d->pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess ||
      cudaMemPoolGetAttribute(d->pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return reserved > used ? (size_t)(reserved - used) : 0;
}

cudaError_t release_kept() {
  std::lock_guard<std::mutex> lock(g_mu);
  Device* d = current_device();
  return d ? cudaMemPoolTrimTo(d->pool, 0) : cudaSuccess;
}

cudaError_t take_result_words(ResultWords* w) {
  *w = ResultWords{};
  std::lock_guard<std::mutex> lock(g_mu);
  if (Device* d = current_device()) {
    for (Page& page : d->pages) {
      if (!page.base) {
        const cudaError_t e = cudaMallocHost(reinterpret_cast<void**>(&page.base), kPageBytes);
        if (e != cudaSuccess) {
          page.base = nullptr;
          return e;
        }
      }
      for (int k = 0; k < kSlots; ++k) {
        uint64_t& word = page.used[k / 64];
        const uint64_t bit = 1ull << (k % 64);
        if (word & bit) continue;
        word |= bit;
        w->p = reinterpret_cast<double*>(page.base + k * kWordBytes);
        w->ctx_id = d->ctx_id;
        return cudaSuccess;
      }
    }
  }
  return cudaMallocHost(reinterpret_cast<void**>(&w->p), kWordBytes);
}

void give_result_words(const ResultWords& w) {
  if (!w.p) return;
  if (!w.ctx_id) {
    cudaFreeHost(w.p);
    return;
  }
  const char* c = reinterpret_cast<const char*>(w.p);
  std::lock_guard<std::mutex> lock(g_mu);
  Device* d = find_device(w.ctx_id);
  if (!d) return;  // that context is gone, and its pages with it
  for (int j = 0; j < kPages; ++j) {
    Page& page = d->pages[j];
    if (!page.base || c < page.base || c >= page.base + kPageBytes) continue;
    const int k = (int)((c - page.base) / kWordBytes);
    page.used[k / 64] &= ~(1ull << (k % 64));
    bool any = false;
    for (uint64_t u : page.used) any |= u != 0;
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!any && j > 0 && current_context(&ctx, &id) && id == w.ctx_id) {
      cudaFreeHost(page.base);
      page.base = nullptr;
    }
    return;
  }
}

}  // namespace hsg

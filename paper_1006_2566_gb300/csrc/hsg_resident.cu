// hsg_resident.cu -- whole sweeps of small lattices in a single launch.
//
// A lone small lattice is bound by launches, not by work: a half-sweep of
// L = 16 is 2048 site updates, 0.1 us of one GPU, but 1.3-2 us as a launch of
// its own in a replayed graph, and every graph of one sweep costs 4 us more.
// Here one thread-block cluster holds the lattice in shared memory and
// registers and runs all the sweeps up to the next energy: CTA r of C owns
// the z planes [r L / C, (r + 1) L / C) and every thread one site of each
// colour -- the sites (xh, y, z) of both colours, whose spins and twelve bonds
// stay in its registers for the whole launch.  Shared memory holds a copy of
// the CTA's spins for the neighbours to read, with one halo plane below and
// above that the CTAs there write (distributed shared memory) as they
// update them.  One cluster barrier per half-sweep orders the colours.
//
// Why a halo can be written in place: half-sweep t updates colour c and reads
// colour 1 - c only.  The halo planes of colour c that the neighbours write
// during t are first read in t + 1, after the barrier; those of colour 1 - c
// that they write during t + 1 are not read before t + 2.
//
// The site code is site_result, the inputs those of site_index: the results
// are those of the half-sweep kernels bit for bit.
//
// What bounds it: latency -- one barrier (0.2 us), the neighbours' shared-
// memory reads and one update's dependent chain per half-sweep; the work
// itself is too small to fill 16 SMs.  Measured on GB300, us per sweep over ten
// sweeps (over 100), against one replayed graph per sweep:
//   L = 8    4 OR 15.6 -> 4.0 (10.3 -> 3.3), 1-hit Metropolis 6.5 -> 2.3 (4.0 -> 1.6)
//   L = 16   4 OR 19.3 -> 5.1 (11.9 -> 4.3), 1 hit 7.0 -> 2.6 (4.8 -> 1.8), 4 hits
//            7.8 -> 4.2 (5.9 -> 3.4), heat-bath 7.4 -> 3.0 (5.1 -> 2.1)
//   L = 24   4 OR 19.7 -> 7.5 (12.5 -> 6.6), 4 hits 7.9 -> 6.0 (5.9 -> 5.2)
//   L = 32   4 OR 20.3 -> 10.6 (13.1 -> 9.9), heat-bath 7.5 -> 5.5 (5.4 -> 4.6), 4 hits
//            8.2 -> 8.3 (6.0 -> 7.3): there each hit costs 0.57 us against 0.19 on
//            the whole GPU, hence the bound on the hits in resident_takes.
// In a pool, one launch holds all its lattices of one side, a cluster each, for all
// the sweeps of a call (us per sweep of heat-bath + 2 OR, against the persistent
// kernels' replayed graph): 64 x L = 8 18.6 -> 4.5, 1200 x 8 34.9 -> 13.8, 40 x L = 16
// 22.7 -> 7.5, 150 x 16 30.9 -> 20.1, 46 x L = 24 37.1 -> 31.1, 16 x L = 28 29.0 -> 24.2;
// with more work it is even (2048 x L = 16, 1 hit 131 -> 125) or loses (64 x L = 24, 4 hits
// + 2 OR 56 -> 63), hence kResidentPoolSites.
// A loop over sites with the indices formed and the bonds loaded for each
// (so that larger lattices fit too): 7.9 us at L = 16, 24.9 against 14.0 at L = 40.
#include <atomic>

#include "hsg_device.cuh"
#include "hsg_internal.h"

namespace hsg {
namespace {

// The lattices this kernel takes: every CTA's planes fit one thread per site
// pair.  L = 32 is 1024 threads on each of 16 CTAs.
constexpr uint32_t kThreadsMax = 1024;
constexpr size_t kSharedMax = 96 * 1024;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
// All threads of the cluster (a cluster of one CTA included); writes to
// shared memory before it, local and remote, are visible after it.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// The address in CTA `rank`'s shared memory of what `local` is here.
__device__ __forceinline__ uint32_t map_to(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}

__device__ __forceinline__ float4 load_spin(const float4* S, bool packed, size_t nh, uint32_t c, uint32_t g) {
  if (packed) {
    const float* b = reinterpret_cast<const float*>(S) + 3 * c * nh + g;
    return make_float4(b[0], b[nh], b[2 * nh], 0.0f);
  }
  return S[c * nh + g];
}
__device__ __forceinline__ void store_spin(float4* S, bool packed, size_t nh, uint32_t c, uint32_t g, float4 v) {
  if (packed) {
    float* b = reinterpret_cast<float*>(S) + 3 * c * nh + g;
    b[0] = v.x;
    b[nh] = v.y;
    b[2 * nh] = v.z;
  } else {
    S[c * nh + g] = v;
  }
}

// What a thread keeps of one of its two sites.
struct KeptSite {
  float4 s;
  float jxp, jxm, jyp, jym, jzp, jzm;
};

template <int U, bool POOL>
__global__ void __launch_bounds__(kThreadsMax, 1) k_resident(const __grid_constant__ ResidentArgs a) {
  // sp[colour][plane][in-plane index]: plane 0 the halo below, 1 .. P this
  // CTA's own, P + 1 the halo above.
  extern __shared__ float4 sp[];
  const uint32_t rank = cluster_rank(), C = a.cluster;
  const uint32_t L = a.L, Lh = a.Lh, plane = a.plane;
  const uint32_t z0 = rank * L / C, P = (rank + 1) * L / C - z0;
  const uint32_t part = (a.max_planes + 2) * plane;  // one colour's share of sp
  const uint32_t tid = threadIdx.x;
  float4* spins = a.spins;
  const float* J = a.J;
  uint32_t k0 = a.k0, k1 = a.k1;
  float beta = a.beta;
  unsigned long long sweep0;
  if constexpr (POOL) {
    const PoolDesc& d = a.desc[a.slots[blockIdx.x / C]];
    spins = reinterpret_cast<float4*>(a.arena) + d.spin_off;
    J = reinterpret_cast<const float*>(a.arena) + d.j_off;
    k0 = d.k0;
    k1 = d.k1;
    beta = d.beta;
    sweep0 = (unsigned long long)d.sweep_hi << 32 | d.sweep_lo;
  } else {
    sweep0 = *a.sweep_ptr;
  }

  // This thread's sites: in-plane index r of plane z, for tid < P * plane.
  const bool mine = tid < P * plane;
  const uint32_t lz = mine ? fast_div(tid, a.by_plane) : 0u, r = mine ? tid - lz * plane : 0u;
  const uint32_t y = fast_div(r, a.by_Lh), xh = r - y * Lh, z = z0 + lz;
  const uint32_t q = (lz + 1) * plane + r;  // in a colour's share of sp
  const uint32_t g = z * plane + r;         // in a colour's array
  const uint32_t dyp = y + 1 == L ? Lh - plane : Lh, dym = y == 0 ? plane - Lh : 0u - Lh;  // modulo 2^32
  const uint32_t dxp = xh + 1 == Lh ? 1u - Lh : 1u, dxm = xh == 0 ? Lh - 1u : 0xFFFFFFFFu;
  const uint32_t p0 = (y + z) & 1u;  // colour 0's p (x = 2 xh + p); colour 1's is 1 - p0
  KeptSite k[2];
#pragma unroll
  for (uint32_t c = 0; c < 2; ++c) {
    const uint32_t p = p0 ^ c, gzm = z == 0 ? g + (L - 1) * plane : g - plane;
    const float *Jc = J + c * a.nh, *Jo = J + (1 - c) * a.nh;
    k[c].jxp = __ldg(Jc + g);
    k[c].jxm = __ldg(Jo + (p ? g : g + dxm));
    k[c].jyp = __ldg(Jc + 2 * a.nh + g);
    k[c].jym = __ldg(Jo + 2 * a.nh + (g + dym));
    k[c].jzp = __ldg(Jc + 4 * a.nh + g);
    k[c].jzm = __ldg(Jo + 4 * a.nh + gzm);
    k[c].s = load_spin(spins, a.packed, a.nh, c, g);
    if (mine) sp[c * part + q] = k[c].s;
    for (uint32_t i = tid; i < 2 * plane; i += blockDim.x) {  // the halo planes z0 - 1 and z0 + P
      const bool lo = i < plane;
      const uint32_t ri = lo ? i : i - plane;
      const uint32_t zi = lo ? (z0 == 0 ? L - 1 : z0 - 1) : (z0 + P == L ? 0u : z0 + P);
      sp[c * part + (lo ? 0u : (P + 1) * plane) + ri] =
          load_spin(spins, a.packed, a.nh, c, zi * plane + ri);
    }
  }
  // Where the CTA below (above) keeps this CTA's first (last) plane.
  const uint32_t below = rank == 0 ? C - 1 : rank - 1, above = rank + 1 == C ? 0u : rank + 1;
  const uint32_t P_below = (below + 1) * L / C - below * L / C;
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(sp);
  const uint32_t to_below = map_to(base + ((P_below + 1) * plane + r) * 16u, below);
  const uint32_t to_above = map_to(base + r * 16u, above);
  const bool first = mine && lz == 0, last = mine && lz + 1 == P;
  cluster_sync();

  for (uint32_t sw = 0; sw < a.sweeps; ++sw) {
    const unsigned long long sweep = sweep0 + sw;
    const uint32_t lo = (uint32_t)sweep, hi = (uint32_t)(sweep >> 32);
    for (uint32_t step = 0; step < a.per_sweep; step += 2) {
      const bool main_update = U != U_OR && step == 0;
#pragma unroll
      for (uint32_t c = 0; c < 2; ++c) {
        if (mine) {
          const uint32_t p = p0 ^ c;
          const float4* oth = sp + (1 - c) * part + q;
          const float4 straight = oth[0], side = oth[(int)(p ? dxp : dxm)];
          SiteInputs in;
          in.sxp = p ? side : straight;
          in.sxm = p ? straight : side;
          in.syp = oth[(int)dyp];
          in.sym = oth[(int)dym];
          in.szp = oth[(int)plane];
          in.szm = oth[-(int)plane];
          in.jxp = k[c].jxp;
          in.jxm = k[c].jxm;
          in.jyp = k[c].jyp;
          in.jym = k[c].jym;
          in.jzp = k[c].jzp;
          in.jzm = k[c].jzm;
          in.s = make_float3(k[c].s.x, k[c].s.y, k[c].s.z);
          in.q = 0;
          in.site = (2 * xh + p) + y * L + z * L * L;
          k[c].s = main_update ? site_result<U>(in, c, lo, hi, k0, k1, beta, a.step, a.hits)
                               : site_result<U_OR>(in, c, 0u, 0u, 0u, 0u, 0.0f, 0.0f, 1);
          sp[c * part + q] = k[c].s;
          if (first) st_cluster(to_below + c * part * 16u, k[c].s);
          if (last) st_cluster(to_above + c * part * 16u, k[c].s);
        }
        cluster_sync();
      }
    }
    if (a.renorm_every && (sweep + 1) % a.renorm_every == 0) {
      // Everyone renormalises what it holds, the halo copies included: no
      // exchange.  (The barrier before has ended the last reads and writes.)
#pragma unroll
      for (uint32_t c = 0; c < 2; ++c) {
        k[c].s = renorm_spin(k[c].s);
        if (mine) sp[c * part + q] = k[c].s;
        for (uint32_t i = tid; i < 2 * plane; i += blockDim.x) {
          float4* h = sp + c * part + (i < plane ? i : i + P * plane);
          *h = renorm_spin(*h);
        }
      }
      cluster_sync();
    }
  }
  if (mine) {
    store_spin(spins, a.packed, a.nh, 0, g, k[0].s);
    store_spin(spins, a.packed, a.nh, 1, g, k[1].s);
  }
  // Every CTA read the counter before the first barrier.
  if (!POOL && rank == 0 && tid == 0) *a.sweep_ptr = sweep0 + a.sweeps;
}

// CTAs in the cluster of an L lattice: as many as divide the work, at most
// one per plane.  More CTAs are faster throughout (a sweep of 1-hit Metropolis
// at L = 16: 3.3, 2.2, 1.8, 1.8 us with 2, 4, 8, 16) but up to L = 8, where
// one does as well as eight (1.55 against 1.51 us) on an eighth of the SMs.
uint32_t cluster_size(uint32_t L) {
  return L <= 8 ? 1u : L < 16 ? 8u : 16u;
}

// Threads per CTA: one per pair of sites of the largest share of planes.
uint32_t cta_threads(uint32_t L, uint32_t cluster) {
  return ((L + cluster - 1) / cluster * L * (L / 2) + 31u) / 32u * 32u;
}

// In a pool with `total` lattices of this L: as alone while they all fit at once;
// else CTAs of 192 threads or more (smaller ones waste more on halos and barriers)
// in clusters of at most eight (sixteen find their SMs together less often).
// us per sweep: L = 16 x 128, 1 hit: 8.2, 8.3, 8.1, 7.9, 8.9 with 1, 2, 4, 8, 16; L = 12 x 200,
// 2 hits + OR: 31.5, 24.6, 23.2, 24.3, 25.9; L = 24 x 64, 4 hits + 2 OR: 63 with 8, 106 with 16;
// x 6: 13.1, 11.1.
uint32_t pool_cluster_size(uint32_t L, int total, int sm_count) {
  uint32_t c = cluster_size(L);
  if ((uint32_t)total * c <= (uint32_t)sm_count) return c;
  if (c > 8 && cta_threads(L, 8) <= kThreadsMax) c = 8;  // from L = 26 sixteen are needed
  while (c > 1 && cta_threads(L, c) < 192 && cta_threads(L, c / 2) <= kThreadsMax) c /= 2;
  return c;
}

cudaLaunchAttribute cluster_attribute(uint32_t cluster) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cluster;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  return at;
}

std::atomic<bool> g_no_clusters{false};  // test hook: hsg_test_no_clusters

// Sets the kernel's attributes and asks whether the device ever has room for a
// cluster of this size (with the most threads and shared memory that a launch asks
// for), once per kernel, size (a power of two up to 16) and device: a GPU whose
// visible SMs come in smaller groups (a partition) has none for sixteen CTAs.
template <int U, bool POOL>
bool fits_u(uint32_t cluster) {
  constexpr int kNo = 1, kYes = 2;
  static PerDevice known[5];
  int log2 = 0;
  while ((1u << log2) < cluster) ++log2;
  cudaError_t e = cudaSuccess;
  std::atomic<int>* slot = device_slot(known[log2], &e);
  if (!slot) return false;
  int answer = slot->load(std::memory_order_acquire);
  if (answer == 0) {
    e = cudaFuncSetAttribute(k_resident<U, POOL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSharedMax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_resident<U, POOL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchAttribute at = cluster_attribute(cluster);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster);
    cfg.blockDim = dim3(kThreadsMax);
    cfg.dynamicSmemBytes = kSharedMax;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k_resident<U, POOL>, &cfg);
    if (e != cudaSuccess) cudaGetLastError();
    answer = e == cudaSuccess && n > 0 ? kYes : kNo;
    slot->store(answer, std::memory_order_release);
  }
  return answer == kYes;
}

template <int U, bool POOL>
cudaError_t launch_u(ResidentArgs a, uint32_t cluster, cudaStream_t s) {
  if (!fits_u<U, POOL>(cluster)) return cudaErrorInvalidValue;
  a.cluster = cluster;
  a.max_planes = (a.L + cluster - 1) / cluster;
  a.Lh = a.L / 2;
  a.plane = a.L * a.Lh;
  a.nh = (size_t)a.plane * a.L;
  a.by_plane = make_fastdiv(a.plane);
  a.by_Lh = make_fastdiv(a.Lh);
  const uint32_t threads = cta_threads(a.L, cluster);
  if (threads > kThreadsMax || a.n < 1) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cluster * (uint32_t)a.n);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = (size_t)2 * (a.max_planes + 2) * a.plane * sizeof(float4);
  cfg.stream = s;
  cudaLaunchAttribute at = cluster_attribute(cluster);
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_resident<U, POOL>, a);
}

template <bool POOL>
cudaError_t launch_kinds(int upd, const ResidentArgs& a, uint32_t cluster, cudaStream_t s) {
  switch (upd) {
    case U_OR: return launch_u<U_OR, POOL>(a, cluster, s);
    case U_MET_SPHERE: return launch_u<U_MET_SPHERE, POOL>(a, cluster, s);
    case U_MET_BALL: return launch_u<U_MET_BALL, POOL>(a, cluster, s);
    case U_HB: return launch_u<U_HB, POOL>(a, cluster, s);
    case U_MET_OR_SPHERE: return launch_u<U_MET_OR_SPHERE, POOL>(a, cluster, s);
    case U_MET_OR_BALL: return launch_u<U_MET_OR_BALL, POOL>(a, cluster, s);
    default: return cudaErrorInvalidValue;
  }
}

template <bool POOL>
bool fits_kinds(int upd, uint32_t cluster) {
  switch (upd) {
    case U_OR: return fits_u<U_OR, POOL>(cluster);
    case U_MET_SPHERE: return fits_u<U_MET_SPHERE, POOL>(cluster);
    case U_MET_BALL: return fits_u<U_MET_BALL, POOL>(cluster);
    case U_HB: return fits_u<U_HB, POOL>(cluster);
    case U_MET_OR_SPHERE: return fits_u<U_MET_OR_SPHERE, POOL>(cluster);
    case U_MET_OR_BALL: return fits_u<U_MET_OR_BALL, POOL>(cluster);
    default: return false;
  }
}

}  // namespace

// Where sixteen SMs beat the whole GPU on one launch per half-sweep: a hit
// costs 0.27, 0.43, 0.57 us here at L = 16, 24, 32 (0.19-0.23 us there), the
// rest of a half-sweep 0.5-0.9 us less.
bool resident_takes(int upd, int L, int hits) {
  if (L < 4 || (L & 1) || L > kResidentMaxL) return false;
  if (upd == U_OR || upd == U_HB) return true;
  return hits <= (L <= 16 ? 16 : L <= 24 ? 5 : 2);
}

bool resident_fits(int upd, int L, int n, bool pool, int sm_count) {
  if (g_no_clusters.load(std::memory_order_relaxed)) return false;
  return pool ? fits_kinds<true>(upd, pool_cluster_size((uint32_t)L, n, sm_count))
              : fits_kinds<false>(upd, cluster_size((uint32_t)L));
}

void test_no_clusters(bool on) { g_no_clusters.store(on); }

cudaError_t launch_resident(int upd, const ResidentArgs& a, int sm_count, cudaStream_t s) {
  if (!resident_takes(upd, (int)a.L, a.hits)) return cudaErrorInvalidValue;
  return a.slots ? launch_kinds<true>(upd, a, pool_cluster_size(a.L, a.n, sm_count), s)
                 : launch_kinds<false>(upd, a, cluster_size(a.L), s);
}

}  // namespace hsg

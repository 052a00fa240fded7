// hsg_batch.cu -- one half-sweep of several lattices of a pool in one launch.
//
// The pool's own kernels (hsg_pool.cu) take every lattice in one persistent
// launch per half-sweep: right for many small lattices, but with hundreds of
// megabytes of state each half-sweep streams everything from HBM, a fixed grid
// at the registers of its per-lattice pointers keeps half the warps, and every
// launch ends in a tail.  Here lattices of L >= kBatchMinL go in batches small enough for L2:
// all the sweeps of a call run on one batch before the next, so its state
// stays in L2 (about 32 MB each), a few batches side by side on internal
// streams, so that one's tail and start-up are filled by the others and the
// Metropolis of one (bound by issue) runs beside the over-relaxation of another
// (bound by memory).  The lattices are kernel parameters: the constant bank gives
// every CTA its lattice without dependent loads, and there is no table to upload.
//
// Measured on GB300, 4-hit Metropolis + 2 OR, us per sweep in calls of 40, against the
// persistent kernels: 128 lattices of L = 32 and 48 474 -> 329; 24 of 64 to 96
// 659 -> 416; 45 of 32 to 96 767 -> 510.  Per half-sweep of the 24: OR 88 -> 42, 4 hits
// 155 -> 125, heat-bath 110 -> 78.  By batch size and streams (the 24, launched one by one, then
// 457): 1000 MB, 1: 550; 64 MB, 1: 600; 64, 2: 486; 48, 2: 468; 32, 3: 457; 24, 4: 459; 128, 2: 559.
#include "hsg_device.cuh"
#include "hsg_internal.h"

namespace hsg {
namespace {

constexpr int B_THREADS = 128;

// The batch's lattice that CTA `b` works on (binary search over the first
// CTAs; the same for the whole CTA).
__device__ __forceinline__ int batch_find(const BatchArgs& a, uint32_t b) {
  int lo = 0, hi = a.n;  // lat[lo].cta0 <= b < lat[hi].cta0
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (a.lat[mid].cta0 <= b)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

template <int U, int R, int MIN_BLOCKS, class Off, bool COUNTED>
__global__ void __launch_bounds__(B_THREADS, MIN_BLOCKS)
    k_batch_half(const __grid_constant__ BatchArgs a, uint32_t colour, int hits, int hit0, float step,
                 uint32_t sweep_add) {
  const BatchLattice& l = a.lat[batch_find(a, blockIdx.x)];
  const uint32_t t = (blockIdx.x - l.cta0) * B_THREADS + threadIdx.x;
  const uint32_t L = l.L, Lh = l.Lh, nh = l.nh;
  if (t >= nh / R) return;
  // t numbers the (plane, row group, column) triples of the lattice
  const uint32_t row = fast_div(t, l.by_lh), xh = t - row * Lh;
  const uint32_t z = fast_div(row, l.by_groups), y0 = (row - z * (L / R)) * R;
  const uint32_t o = 1u - colour;
  const float* J = l.J;
  const RowLattice<false> lat{l.spins + (size_t)colour * nh,
                              l.spins + (size_t)o * nh,
                              J + (size_t)(0 + colour) * nh,
                              J + (size_t)(2 + colour) * nh,
                              J + (size_t)(4 + colour) * nh,
                              J + (size_t)(0 + o) * nh,
                              J + (size_t)(2 + o) * nh,
                              J + (size_t)(4 + o) * nh,
                              0,
                              L,
                              Lh,
                              colour};
  // The count is advanced first by the sphere proposals' kernels and last by the others:
  // where the store stands moves the compiler's registers.  us a sweep of 36 lattices of
  // L = 64, first / last: sphere 1 hit 85.0 / 88.5, sphere + OR 88.0 / 96.0; ball 1 hit 90.9 / 85.4,
  // ball + OR 90.5 / 88.8, heat-bath 112.9 / 109.1 (not counted: 84.8, 90.9, 85.8, 91.7, 107.7).
  constexpr bool FIRST = U == U_MET_SPHERE || U == U_MET_OR_SPHERE;
  unsigned long long sw = l.sweep + sweep_add;
  if constexpr (COUNTED) {
    const unsigned long long count = a.done[colour];
    sw = l.sweep + count;
    if (FIRST && blockIdx.x == 0 && threadIdx.x == 0) a.done[o] = count + colour;
  }
  const DrawArgs d{(uint32_t)sw, (uint32_t)(sw >> 32), l.k0, l.k1, l.beta, step, hits, hit0};
  update_rows<U, R, Off>(lat, xh, y0, z, (colour + y0 + z) & 1u, d);  // z differs within a CTA
  if constexpr (COUNTED && !FIRST) {
    if (blockIdx.x == 0 && threadIdx.x == 0) a.done[o] = a.done[colour] + colour;
  }
}

template <int U, int R, int MIN_BLOCKS, bool COUNTED>
void launch_r(BatchArgs& a, uint32_t colour, int hits, int hit0, float step, uint32_t sweep_add, cudaStream_t s) {
  uint32_t ctas = 0;
  bool wide = false;
  for (int k = 0; k < a.n; ++k) {
    BatchLattice& l = a.lat[k];
    l.cta0 = ctas;
    l.by_groups = make_fastdiv(l.L / R);
    ctas += (l.nh / R + B_THREADS - 1) / B_THREADS;
    wide |= l.L > (uint32_t)kMaxOff32L;
  }
  if (wide)
    k_batch_half<U, R, MIN_BLOCKS, unsigned long long, COUNTED><<<ctas, B_THREADS, 0, s>>>(a, colour, hits, hit0, step, sweep_add);
  else
    k_batch_half<U, R, MIN_BLOCKS, uint32_t, COUNTED><<<ctas, B_THREADS, 0, s>>>(a, colour, hits, hit0, step, sweep_add);
}

template <int U, int R, int MIN_BLOCKS, int MIN_BLOCKS_COUNTED>
void launch_kind(bool counted, BatchArgs& a, uint32_t colour, int hits, int hit0, float step, uint32_t sweep_add,
                 cudaStream_t s) {
  if (counted)
    launch_r<U, R, MIN_BLOCKS_COUNTED, true>(a, colour, hits, hit0, step, 0u, s);
  else
    launch_r<U, R, MIN_BLOCKS, false>(a, colour, hits, hit0, step, sweep_add, s);
}

__global__ void __launch_bounds__(256) k_batch_renorm(const __grid_constant__ BatchArgs a) {
  const BatchLattice& l = a.lat[blockIdx.y];
  for (uint32_t q = blockIdx.x * 256u + threadIdx.x; q < l.nh; q += gridDim.x * 256u) {
    l.spins[q] = renorm_spin(l.spins[q]);
    l.spins[(size_t)l.nh + q] = renorm_spin(l.spins[(size_t)l.nh + q]);
  }
}

}  // namespace

cudaError_t launch_batch_half(int upd, bool counted, BatchArgs& a, uint32_t colour, int hits, int hit0, float step,
                              uint32_t sweep_add, cudaStream_t s) {
  // Rows per thread and registers as in the single-lattice launches
  // (hsg_sweep.cu), measured here for OR (one row 47 us, two 53-70), the
  // heat-bath (two rows 75, one 80) and the ball proposal (two 129, one 133).  The counted
  // ones are held to the registers of the others (64 and 56, not 96 and 80).
  switch (upd) {
    case U_OR: launch_r<U_OR, 1, 12, false>(a, colour, hits, hit0, step, sweep_add, s); break;
    case U_MET_SPHERE: launch_kind<U_MET_SPHERE, 2, 10, 10>(counted, a, colour, hits, hit0, step, sweep_add, s); break;
    case U_MET_BALL: launch_kind<U_MET_BALL, 2, 8, 8>(counted, a, colour, hits, hit0, step, sweep_add, s); break;
    case U_HB: launch_kind<U_HB, 2, 1, 8>(counted, a, colour, hits, hit0, step, sweep_add, s); break;
    case U_MET_OR_SPHERE: launch_kind<U_MET_OR_SPHERE, 2, 8, 8>(counted, a, colour, hits, hit0, step, sweep_add, s); break;
    case U_MET_OR_BALL: launch_kind<U_MET_OR_BALL, 2, 1, 9>(counted, a, colour, hits, hit0, step, sweep_add, s); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_batch_renorm(const BatchArgs& a, cudaStream_t s) {
  if (a.n < 1) return cudaSuccess;
  uint32_t most = 0;
  for (int k = 0; k < a.n; ++k) most = a.lat[k].nh > most ? a.lat[k].nh : most;
  uint32_t gx = (most + 255) / 256;
  if (gx > 1024) gx = 1024;
  k_batch_renorm<<<dim3(gx, (unsigned)a.n), 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace hsg

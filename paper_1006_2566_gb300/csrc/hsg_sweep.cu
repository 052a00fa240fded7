// hsg_sweep.cu -- checkerboard half-sweep kernels (Sec. 4: the sites of one
// colour do not interact, so a half-sweep updates all of them in parallel
// from the other colour; one launch per colour keeps the two colours
// ordered).
//
// Two variants over the colour-split layout of hsg_device.cuh:
//   global : one thread per one, two or four sites of a column of rows; the
//            neighbours come through L1/L2 (the lattice is streamed once per
//            half-sweep from HBM).  Its heat-bath launches on large lattices
//            march a thread up a short column of planes (k_half_sweep_column).
//   slab   : a CTA owns a (32 xh) x (4 y) column tile and marches up a chunk
//            of z planes.  The other colour's plane z (with a one-site halo)
//            is staged in shared memory for the x and y neighbours; planes
//            z-1 and z+1 stay in registers, so each other-colour spin is
//            read from memory about once per half-sweep.
#include "hsg_device.cuh"
#include "hsg_internal.h"

namespace hsg {
namespace {

inline unsigned cdiv(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

__device__ __forceinline__ uint32_t site_number(int xh, int p, int y, int z, int L) {
  return (uint32_t)(2 * xh + p) + (uint32_t)y * (uint32_t)L + (uint32_t)z * (uint32_t)L * (uint32_t)L;
}

// ---------------------------------------------------------------------------
// Global variant.  A thread updates R consecutive rows of one column of a
// plane (update_rows, hsg_device.cuh); the (xh, row group) pairs of a plane
// are numbered through, so that a row of any length fills its warps, and one
// multiply-shift division per thread recovers them.  Byte offsets are 32-bit
// up to L = 812 (16 N/2 < 2^32) and added to the arrays' bases by the load
// instructions.  Measured on GB300 per half-sweep in replayed graphs,
// against one site per thread on 64 x 2 or 32 x 4 blocks (half of their
// threads idle at L/2 = 33 or 65) with 64-bit addresses:
//   L = 66   OR 3.57 -> 2.30, 4-hit Metropolis 7.10 -> 4.10, heat-bath (column
//            kernel below) 6.48 -> 3.08 us
//   L = 100  5.37 -> 4.10, 13.3 -> 11.2, 10.2 -> 7.2 us
//   L = 128  7.94 -> 6.66, 20.7 -> 20.5, 15.1 -> 12.3 us
//   L = 130  11.0 -> 7.9, 32.8 -> 22.6, 17.5 -> 13.3 us
//   L = 256  85.0 -> 83.5, 160.6 -> 154.4 us; heat-bath stays with the column
//            kernel (86.5 us; 95.8 with two rows per thread)
//   packed, L = 130: 12.1 -> 7.7, 35.7 -> 23.6, 21.4 -> 13.9 us; L = 256: 89.6 ->
//            84.3, 170.6 -> 165, 102.9 -> 94.1 us
// Rows per thread (launch_global below): the own-column neighbour of one row is
// the y neighbour of the next, so R rows load 2 + 2/R + 1 neighbours each
// instead of five; but R rows per thread leave 1/R of the threads, and below
// about 10^6 sites those are too few (L = 64, 4-hit Metropolis: 4.1, 5.1,
// 7.2 us with one, two, four rows).
// A grid of exactly the resident CTAs looping over the sites (grid-stride,
// or an equal contiguous range per CTA) made the 4-hit Metropolis half-sweep at
// L = 128 slower: 28.1-30.1 us against 25.9 us.
// ---------------------------------------------------------------------------
constexpr int G_THREADS = 128;

template <int U, int R, int MIN_BLOCKS, class Off, bool PACKED, bool OVERLAP>
__global__ void __launch_bounds__(G_THREADS, MIN_BLOCKS)
    k_half_sweep_rows(const SweepArgs a, FastDiv by_lh, uint32_t columns, bool early, bool down) {
  const uint32_t t = blockIdx.x * G_THREADS + threadIdx.x;
  if constexpr (OVERLAP) {
    if (early) let_next_start();
    wait_for_previous();
  }
  if (t >= columns) return;
  const uint32_t g = fast_div(t, by_lh), xh = t - g * (uint32_t)a.Lh, y0 = g * R;
  const uint32_t z = down ? gridDim.y - 1 - blockIdx.y : blockIdx.y;
  const RowLattice<PACKED, OVERLAP> lat{a.own,    a.oth,    a.jx_own, a.jy_own,      a.jz_own,       a.jx_oth,
                               a.jy_oth, a.jz_oth, a.stride, (uint32_t)a.L, (uint32_t)a.Lh, (uint32_t)a.colour};
  DrawArgs d{a.sweep_lo, a.sweep_hi, a.k0, a.k1, a.beta, a.step, a.hits, 0};
  if constexpr (U != U_OR) {
    if (a.sweep_ptr) {
      const unsigned long long sw = *a.sweep_ptr + a.sweep_add;
      d.sweep_lo = (uint32_t)sw;
      d.sweep_hi = (uint32_t)(sw >> 32);
    }
  }
  // x = 2 xh + p.  With R even, y0 is even and p the same for the block:
  // one branch, and no selects inside.
  const uint32_t p = ((uint32_t)a.colour + (R == 1 ? y0 : 0u) + z) & 1u;
  if constexpr (R == 1) {
    update_rows<U, R, Off>(lat, xh, y0, z, p, d);
  } else {
    if (p)
      update_rows<U, R, Off>(lat, xh, y0, z, 1u, d);
    else
      update_rows<U, R, Off>(lat, xh, y0, z, 0u, d);
  }
  if constexpr (OVERLAP) {
    if (!early) let_next_start();
  }
}

// Heat-bath half-sweeps of the global variant from L = ZM_MIN_L, where they
// stream from HBM: one thread per (xh, y) column of the updated colour over
// ZM_PLANES consecutive planes.  The
// other colour's spins in the thread's own column on planes z-1 and z (the
// site's -z neighbour and one of its x neighbours) are carried from the
// plane before, so a site loads four neighbour spins instead of six; the
// inputs and the site code are those of k_half_sweep_rows, so the results
// are the same bit for bit.  Measured on the L = 256 heat-bath half-sweep:
// 6 planes and 40 registers (12 blocks per SM) 94.0 us, against 100.9 us
// for one site per thread at 32 registers; 8 planes 95.1, 4 planes 96.0,
// 16 planes 97.3, 32 planes 107; at 32 registers (spilling) 104-106 us.
// A persistent grid that deals out equal contiguous (column block, plane)
// ranges, one CTA per resident slot (no partial last wave), took 105.7 us:
// neighbouring column blocks then work on different planes, so the rows
// they share are probably no longer found in L2.  Blocks of 16 x 8 threads
// (a warp spans two rows, so a block's y-neighbour rows are mostly its own
// and come from L1): 89.4 us against 90.7 us for 64 x 2 (fp32 subnormals
// flushed); 32 x 4, 128 x 1, 8 x 16 and 256-thread blocks 89.9-91.1 us;
// streaming (evict-first) stores of the new spins gained 0.2 us more.
constexpr int ZM_PLANES = 6;
// 32-bit byte offsets up to L = 812: 86.5 against 88.6 us at L = 256, 40.8 against
// 41.5 at L = 192.  From ZM_MIN_L on the column march wins over the rows kernel
// (L = 160 23.9 against 25.9 us, 192 40.8 / 41.8, 222 60.2 / 63.9); below, six planes
// per thread are too few threads (L = 128 13.8 against 12.4, L = 64 5.4 against 3.1).
constexpr int ZM_MIN_L = 152;
constexpr int ZM_BX = 16, ZM_BY = 8;

template <class Off>
__global__ void __launch_bounds__(G_THREADS, 12) k_half_sweep_column(const SweepArgs a, bool down) {
  const uint32_t xh = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t y = blockIdx.y * blockDim.y + threadIdx.y;
  const uint32_t L = a.L, Lh = a.Lh;
  if (xh >= Lh || y >= L) return;
  uint32_t sweep_lo = a.sweep_lo, sweep_hi = a.sweep_hi;
  if (a.sweep_ptr) {
    const unsigned long long sw = *a.sweep_ptr + a.sweep_add;
    sweep_lo = (uint32_t)sw;
    sweep_hi = (uint32_t)(sw >> 32);
  }
  const uint32_t plane = L * Lh;
  const uint32_t z0 = (down ? gridDim.z - 1 - blockIdx.z : blockIdx.z) * ZM_PLANES, z1 = min(z0 + ZM_PLANES, L);
  // rows y, y+1, y-1 and columns xh+1, xh-1, wrapped (the layout comment of
  // hsg_device.cuh; the same indices as site_index)
  const uint32_t row = y * Lh, row_p = (y + 1 == L ? 0u : y + 1) * Lh, row_m = (y == 0 ? L - 1 : y - 1) * Lh;
  const uint32_t xm1 = xh == 0 ? Lh - 1 : xh - 1, xp1 = xh + 1 == Lh ? 0u : xh + 1;
  const float4* __restrict__ oth = a.oth;
  uint32_t zmo = (z0 == 0 ? L - 1 : z0 - 1) * plane, zo = z0 * plane;
  float4 s_m = __ldg(elem<Off>(oth, zmo + row + xh)), s_0 = __ldg(elem<Off>(oth, zo + row + xh));
  for (uint32_t z = z0; z < z1; ++z) {
    const uint32_t zpo = z + 1 == L ? 0u : zo + plane;
    const uint32_t p = ((uint32_t)a.colour + y + z) & 1u;  // x = 2 xh + p
    const uint32_t q = zo + row + xh;
    const float4 s_p = __ldg(elem<Off>(oth, zpo + row + xh));
    const float4 side = __ldg(elem<Off>(oth, zo + row + (p ? xp1 : xm1)));
    SiteInputs in;
    in.sxp = p ? side : s_0;
    in.sxm = p ? s_0 : side;
    in.syp = __ldg(elem<Off>(oth, zo + row_p + xh));
    in.sym = __ldg(elem<Off>(oth, zo + row_m + xh));
    in.szp = s_p;
    in.szm = s_m;
    in.jxp = __ldg(elem<Off>(a.jx_own, q));
    in.jxm = __ldg(elem<Off>(a.jx_oth, p ? q : zo + row + xm1));
    in.jyp = __ldg(elem<Off>(a.jy_own, q));
    in.jym = __ldg(elem<Off>(a.jy_oth, zo + row_m + xh));
    in.jzp = __ldg(elem<Off>(a.jz_own, q));
    in.jzm = __ldg(elem<Off>(a.jz_oth, zmo + row + xh));
    in.s = make_float3(0.0f, 0.0f, 0.0f);  // the heat-bath does not read the old spin
    in.q = q;
    in.site = (2 * xh + p) + y * L + z * L * L;
    *elem<Off>(a.own, q) = site_result<U_HB>(in, (uint32_t)a.colour, sweep_lo, sweep_hi, a.k0, a.k1, a.beta, a.step, a.hits);
    s_m = s_0;
    s_0 = s_p;
    zmo = zo;
    zo = zpo;
  }
}

// ---------------------------------------------------------------------------
// Slab variant.  A CTA of TX x SLAB_TY threads owns a column tile of the
// updated colour and marches up zc planes; zc is chosen at launch so that
// the grid holds SLAB_CTAS_PER_SM CTAs per SM (at L = 128: 7 planes, 1216
// CTAs; from L = 256 the cap of 16 planes).  Indices are 32-bit: every
// offset is below N/2 < 2^31.  Registers are held to what 10 (over-
// relaxation) or 8 (the others) resident CTAs allow.  Measured on GB300
// (bit-identical throughout): the L = 128 4-hit Metropolis + OR workload
// 15.0 us (OR) and 34.0 us (Metropolis) per half-sweep against 26.0 and
// 45.3 us with 32 x 8 tiles of 16 planes, 64-bit indices and no register
// bound; the L = 256 OR half-sweep 144 us against 162 us.
// ---------------------------------------------------------------------------
constexpr int TX = 32, SLAB_TY = 4, SLAB_ZC_MAX = 16, SLAB_CTAS_PER_SM = 8;
template <int U>
constexpr int slab_min_blocks() {
  return U == U_OR ? 10 : 8;
}

template <int U>
__global__ void __launch_bounds__(TX* SLAB_TY, slab_min_blocks<U>()) k_half_sweep_slab(const SweepArgs a, int zc) {
  constexpr int TY = SLAB_TY;
  // Two buffers of the other colour's plane tile: slot (r, c) holds the site
  // ((x0 + c - 1) mod Lh, (y0 + r - 1) mod L); the corners are unused.
  __shared__ float4 plane[2][TY + 2][TX + 2];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int L = a.L, Lh = a.Lh;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = blockIdx.z * zc;
  const int z1 = min(z0 + zc, L);
  const int xh = x0 + tx, y = y0 + ty;
  const bool valid = xh < Lh && y < L;
  // Threads past the lattice edge fill their slot with the periodic image.
  const uint32_t xw = (uint32_t)(xh % Lh), yw = (uint32_t)(y % L);
  const uint32_t x_left = (uint32_t)((x0 + Lh - 1) % Lh), x_right = (uint32_t)((x0 + TX) % Lh);
  const uint32_t y_top = (uint32_t)((y0 + L - 1) % L), y_bot = (uint32_t)((y0 + TY) % L);
  const uint32_t Lhu = (uint32_t)Lh;
  const uint32_t plane_sz = (uint32_t)L * Lhu;
  const uint32_t col = yw * Lhu + xw;  // this slot's offset in a plane
  uint32_t sweep_lo = a.sweep_lo, sweep_hi = a.sweep_hi;
  if constexpr (U != U_OR) {
    if (a.sweep_ptr) {
      const unsigned long long sw = *a.sweep_ptr + a.sweep_add;
      sweep_lo = (uint32_t)sw;
      sweep_hi = (uint32_t)(sw >> 32);
    }
  }

  const uint32_t zprev = (uint32_t)wrap_dec(z0, L);
  float4 s_zm = __ldg(a.oth + zprev * plane_sz + col);
  float4 s_z = __ldg(a.oth + (uint32_t)z0 * plane_sz + col);
  float jzm = valid ? __ldg(a.jz_oth + zprev * plane_sz + col) : 0.0f;

  for (int z = z0; z < z1; ++z) {
    const uint32_t zn = (uint32_t)wrap_inc(z, L);
    const float4 s_zp = __ldg(a.oth + zn * plane_sz + col);
    const uint32_t pz = (uint32_t)z * plane_sz;
    float4(*buf)[TX + 2] = plane[(z - z0) & 1];
    buf[ty + 1][tx + 1] = s_z;
    if (ty == 0) buf[0][tx + 1] = __ldg(a.oth + pz + y_top * Lhu + xw);
    if (ty == 1) buf[TY + 1][tx + 1] = __ldg(a.oth + pz + y_bot * Lhu + xw);
    if (tx == 0) buf[ty + 1][0] = __ldg(a.oth + pz + yw * Lhu + x_left);
    if (tx == 1) buf[ty + 1][TX + 1] = __ldg(a.oth + pz + yw * Lhu + x_right);
    __syncthreads();
    if (valid) {
      const int p = (a.colour + y + z) & 1;
      const uint32_t row = pz + (uint32_t)y * Lhu;
      const uint32_t q = row + (uint32_t)xh;
      const float jxp = __ldg(a.jx_own + q), jyp = __ldg(a.jy_own + q), jzp = __ldg(a.jz_own + q);
      const float jxm = __ldg(a.jx_oth + row + (uint32_t)(p ? xh : wrap_dec(xh, Lh)));
      const float jym = __ldg(a.jy_oth + pz + (uint32_t)wrap_dec(y, L) * Lhu + (uint32_t)xh);
      const float jz_here = __ldg(a.jz_oth + q);  // -z bond of the site above
      float3 s = make_float3(0.0f, 0.0f, 0.0f);
      if constexpr (U != U_HB) {
        const float4 o = a.own[q];
        s = make_float3(o.x, o.y, o.z);
      }
      const float3 h = local_field(buf[ty + 1][tx + 1 + p], buf[ty + 1][tx + p], buf[ty + 2][tx + 1],
                                   buf[ty][tx + 1], s_zp, s_zm, jxp, jxm, jyp, jym, jzp, jzm);
      const float3 t = update_site<U>(s, h, site_number(xh, p, y, z, L), (uint32_t)a.colour, sweep_lo, sweep_hi,
                                      a.k0, a.k1, a.beta, a.step, a.hits);
      a.own[q] = make_float4(t.x, t.y, t.z, 0.0f);
      jzm = jz_here;
    }
    s_zm = s_z;
    s_z = s_zp;
  }
}

// Planes per slab CTA: the grid holds SLAB_CTAS_PER_SM CTAs per SM where
// the lattice allows, at most SLAB_ZC_MAX planes each.
int slab_zc(int L, unsigned tiles, int sm_count) {
  const long long want = (long long)SLAB_CTAS_PER_SM * (sm_count > 0 ? sm_count : 1);
  long long chunks = (want + tiles - 1) / tiles;
  if (chunks < 1) chunks = 1;
  int zc = (int)((L + chunks - 1) / chunks);
  return zc < 1 ? 1 : (zc > SLAB_ZC_MAX ? SLAB_ZC_MAX : zc);
}

// How a launch of the rows kernel overlaps the next one on the stream: not
// at all, letting its CTAs start when this launch's last CTAs have started
// (EARLY), or as each CTA is done (LATE).  Small launches are mostly start-up:
// up to one wave of CTAs LATE takes 0.3-1 us off each (a waiting CTA of the
// next launch would take the place of a working one; with EARLY L = 66 was
// slower, 2.55 against 2.05 us).  Beyond, the over-relaxation is better left
// alone (its reads then also go through the read-only path), and the longer
// updates gain a little from EARLY while they fill a few waves.  In graphs, us,
// none / LATE / EARLY:
//   OR         L = 40 1.54 / 1.23 / 1.29, 66 2.31 / 2.05 / 2.55, 76 2.58 / 2.76 / 2.82, 128 6.66 / 9.23 / 8.65
//   heat-bath  L = 40 2.04 / 1.03 / 2.05, 66 3.07 / 3.07 / 3.99, 80 5.10 / 4.30 / 5.06, 104 8.09 / 8.11 / 7.20,
//              120 11.1 / 11.3 / 10.3, 128 12.3 / 12.3 / 12.1
//   4 hits     L = 40 3.06 / 2.04 / 2.06, 80 7.12 / 6.19 / 6.18, 110 15.3 / 14.8 / 14.4, 128 20.6 / 20.5 / 20.4
enum Overlap { NONE, EARLY, LATE };
template <int U>
constexpr Overlap overlap(int L) {
  if (U == U_OR) return L <= 72 ? LATE : NONE;
  return L <= 90 ? LATE : L <= 126 ? EARLY : NONE;
}

// Colour 1's CTAs take the planes from the top down (CTAs start in the order of
// their index), where colour 0's went up: each half-sweep so begins on the planes that
// the one before left in L2, where streaming them in the same order finds none.  us per
// two half-sweeps, same order / reversed (126 MB L2; the state is 28 L^3 bytes, packed 24):
//   OR         L = 136 16.8 / 17.0, 144 22.3 / 20.3, 152 33.0 / 26.5, 160 42.8 / 32.4, 176 58.1 / 48.3,
//              192 73.4 / 64.4, 222 113 / 107, 256 168 / 162, 288 240 / 233
//   heat-bath  L = 152 46.8 / 46.3, 192 85.0 / 83.3, 222 125.6 / 123.6, 256 180 / 180
//   ball       L = 136 25.7 / 25.8, 144 32.3 / 30.3, 160 53.2 / 44.1, 192 87.1 / 80.7, 256 198 / 190;
//              4 hits 160 84.8 / 81.9, 256 308 / 305
//   packed OR  L = 144 21.5 / 21.4, 152 29.2 / 26.3, 160 45.6 / 33.9, 192 75.7 / 64.9, 256 169 / 159
// At L = 400 OR 635 / 630, ball 735 / 728, heat-bath 686 / 688; at 512 1315 / 1312, 1534 /
// 1524, sphere + OR 1548 / 1554, heat-bath 1381 / 1388.
constexpr int kDownMinL = 144, kDownMaxL = 400, kDownMaxLHeatbath = 320;
template <int U>
bool downward(const SweepArgs& a) {
  return a.colour == 1 && a.L >= kDownMinL && a.L <= (U == U_HB ? kDownMaxLHeatbath : kDownMaxL);
}

// FROM: the smallest L that takes this shape.
template <int U, int R, int MIN_BLOCKS, class Off, bool PACKED, int FROM = 0>
cudaError_t launch_rows(const SweepArgs& a, cudaStream_t s) {
  const uint32_t columns = (uint32_t)a.Lh * (uint32_t)(a.L / R);
  const FastDiv by_lh = make_fastdiv((uint32_t)a.Lh);
  const dim3 grid(cdiv(columns, G_THREADS), (unsigned)a.L);
  const bool down = downward<U>(a);
  if constexpr (overlap<U>(FROM) != NONE) {
    const Overlap o = overlap<U>(a.L);
    if (o != NONE)
      return launch_overlapped(k_half_sweep_rows<U, R, MIN_BLOCKS, Off, PACKED, true>, grid, dim3(G_THREADS), s, a, by_lh,
                               columns, o == EARLY, down);
  }
  k_half_sweep_rows<U, R, MIN_BLOCKS, Off, PACKED, false><<<grid, G_THREADS, 0, s>>>(a, by_lh, columns, false, down);
  return cudaGetLastError();
}

// Rows per thread (R) and the register bound (B resident CTAs of 128), by
// kind, size and hits.  Registers, spills and the neighbour rows that a
// thread keeps weigh differently for each kind's code; from about L = 150 the
// half-sweeps of few hits stream from HBM and want loads in flight (B 10 to
// 14), the ones of many hits registers.  us per half-sweep at L = 128 / 160 or
// 156 / 192 / 256 (one site per thread, 64-bit addresses, in brackets):
//   OR         R 1, B 12   6.7 / - / 36.4 / 83.5          [7.9 / - / 37.9 / 85.0]
//   heat-bath  R 2, B 16   12.3 / - / 43.2 / 95.8 (R 1, B 12 13.2 / - / 43.0 / 97.4)
//   sphere     R 2, B 10   1 hit 9.6 / 24.7 / 40.9 / 92 [10.2 / 30.7 / 46.9 / 101], 4 hits 18.4 / 35.1 / 58.9 / 133
//                          [18.4 / 47 / 69 / 153]; R 1, B 12 1 hit 10.3 / 27.8 / 46.7 / 106
//   ball       R 1, B 12   1 hit 10.3 / 25.5 / 42.2 / 96 [10.3 / 29.7 / 44.6 / 97] (R 4 10.9 / 25.7 / 47.1 / 102);
//              R 2, R 4    4 hits, each as a sweep of its own, R 1, B 12 / R 2 / R 4: L = 120 17.9 / 17.9, 128 21.3 / 20.9,
//                          150 34.1 / 33.3, 160 - / 39.7 / 40.8, 192 - / 66.9 / 67.4, 208 - / 84.3 / 84.8, 222 109 / 102,
//                          224 - / 104.1 / 103.9, 256 - / 154 / 153, 320 - / 298 / 294 [128 22.6, 150 46.2, 192 74.7, 256 164]
//   sphere+OR  R 1, B 14   1 hit 10.4 / 22.6 / 40.7 / 93 [12.4 / 28.0 / 43.3 / 93] (R 2, B 12 10.3 / 25.4 / 44.8 / 99);
//              R 2, B 8    4 hits 18.5 / 36.9 / 60.7 / 139 [18.5 / 45.1 / 65.1 / 143]
//   ball+OR    R 2         1 hit 10.3 / 24.0 / 40.3 / 92 [10.3 / 33.1 / 50.0 / 107], 4 hits 21.5 / 40.3 / 67.7 / 155
//                          [20.6 / 52.3 / 76.6 / 169]
//   packed OR  L = 130 7.7 (R 1) 11.2 (R 2), 192 38.9 / 37.5, 256 89.3 / 84.3; packed heat-bath 130 15.3 / 13.9, 256 105 / 94;
//   packed ball, 4 hits: 128 22.2 / 22.8, 192 73.0 / 72.0, 256 170 / 165
template <int U, bool PACKED>
cudaError_t launch_global(const SweepArgs& a, cudaStream_t s) {
  constexpr bool MET = U != U_OR && U != U_HB;
  static_assert(ZM_MIN_L <= kMaxOff32L, "the column march takes the float4 heat-bath beyond");
  if constexpr (U != U_HB || PACKED) {
    if (a.L > kMaxOff32L) return launch_rows<U, 1, MET ? 1 : 12, unsigned long long, PACKED, kMaxOff32L + 2>(a, s);
  }
  if constexpr (U == U_OR) {
    if constexpr (PACKED) {
      if (a.L >= 160) return launch_rows<U, 2, 10, uint32_t, PACKED, 160>(a, s);
    }
    return launch_rows<U, 1, 12, uint32_t, PACKED>(a, s);
  } else if constexpr (U == U_HB) {
    if (a.L < 96) return launch_rows<U, 1, 12, uint32_t, PACKED>(a, s);
    return launch_rows<U, 2, PACKED ? 10 : 16, uint32_t, PACKED, 96>(a, s);
  } else if constexpr (PACKED) {
    if (a.L >= 160) return launch_rows<U, 2, 1, uint32_t, PACKED, 160>(a, s);
    return launch_rows<U, 1, 1, uint32_t, PACKED>(a, s);
  } else {
    if (a.L < 96) return launch_rows<U, 1, 1, uint32_t, PACKED>(a, s);
    if constexpr (U == U_MET_SPHERE) {
      return launch_rows<U, 2, 10, uint32_t, PACKED, 96>(a, s);
    } else if constexpr (U == U_MET_BALL) {
      if (a.hits > 1 && a.L >= 220 && a.L % 4 == 0) return launch_rows<U, 4, 1, uint32_t, PACKED, 220>(a, s);
      if (a.hits > 1 && a.L >= 124) return launch_rows<U, 2, 1, uint32_t, PACKED, 124>(a, s);
      return launch_rows<U, 1, 12, uint32_t, PACKED, 96>(a, s);
    } else if constexpr (U == U_MET_OR_SPHERE) {
      if (a.hits == 1) return launch_rows<U, 1, 14, uint32_t, PACKED, 96>(a, s);
      return launch_rows<U, 2, 8, uint32_t, PACKED, 96>(a, s);
    } else {
      return launch_rows<U, 2, 1, uint32_t, PACKED, 96>(a, s);
    }
  }
}

template <int U>
cudaError_t launch_kind(int variant, const SweepArgs& a, int sm_count, cudaStream_t s) {
  if (a.packed) return launch_global<U, true>(a, s);
  if (variant == V_SLAB) {
    const unsigned tx = cdiv(a.Lh, TX), ty = cdiv(a.L, SLAB_TY);
    const int zc = slab_zc(a.L, tx * ty, sm_count);
    const dim3 grid(tx, ty, cdiv(a.L, zc));
    k_half_sweep_slab<U><<<grid, dim3(TX, SLAB_TY), 0, s>>>(a, zc);
    return cudaGetLastError();
  }
  if constexpr (U == U_HB) {
    if (a.L >= ZM_MIN_L) {
      const dim3 grid(cdiv(a.Lh, ZM_BX), cdiv(a.L, ZM_BY), cdiv(a.L, ZM_PLANES));
      const bool down = downward<U>(a);
      if (a.L > kMaxOff32L)
        k_half_sweep_column<unsigned long long><<<grid, dim3(ZM_BX, ZM_BY), 0, s>>>(a, down);
      else
        k_half_sweep_column<uint32_t><<<grid, dim3(ZM_BX, ZM_BY), 0, s>>>(a, down);
      return cudaGetLastError();
    }
  }
  return launch_global<U, false>(a, s);
}

}  // namespace

cudaError_t launch_half_sweep(int upd, int variant, const SweepArgs& a, int sm_count, cudaStream_t s) {
  switch (upd) {
    case U_OR: return launch_kind<U_OR>(variant, a, sm_count, s);
    case U_MET_SPHERE: return launch_kind<U_MET_SPHERE>(variant, a, sm_count, s);
    case U_MET_BALL: return launch_kind<U_MET_BALL>(variant, a, sm_count, s);
    case U_HB: return launch_kind<U_HB>(variant, a, sm_count, s);
    case U_MET_OR_SPHERE: return launch_kind<U_MET_OR_SPHERE>(variant, a, sm_count, s);
    case U_MET_OR_BALL: return launch_kind<U_MET_OR_BALL>(variant, a, sm_count, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace hsg

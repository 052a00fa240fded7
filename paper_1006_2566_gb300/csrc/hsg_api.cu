// hsg_api.cu -- the C ABI declared in include/hsg.h.
//
// Host code only: argument checks, stream-ordered device memory, the sweep
// schedule (which kernels run in which order), the energy log and the
// event-based profiler.  Every step of the Monte Carlo itself runs in the
// kernels of hsg_sweep.cu, hsg_wave.cu, hsg_resident.cu and hsg_aux.cu.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <numeric>
#include <string>
#include <utility>
#include <vector>

#include "hsg.h"
#include "hsg_device.cuh"
#include "hsg_internal.h"

namespace {

constexpr int kVersion = 100;  // 0.1.0
constexpr int kMaxL = 1624;    // L^3 < 2^32: site indices are 32-bit Philox counters
constexpr int kElogInit = 64;
constexpr int kCounters = 4;   // words at hsg_ctx::d_ctr
constexpr long long kMaxGraphPeriod = 64;  // longest sweep period captured as one graph
constexpr int kGraphSweeps = 16;           // most sweeps in one graph without cadences,
constexpr int kGraphLaunches = 64;         // and most launches of more than one sweep
constexpr int kOnceMaxL = 72;              // sides up to which a graph that runs once is not captured

thread_local std::string g_thread_error;
int g_fail_alloc_countdown = 0;  // test hook: k-th allocation from now fails
std::atomic<int> g_test_stall_boxes{0};  // test hook: hsg_test_stall_tensor_loads

// A run of consecutive launches of one kernel class, bracketed by one pair
// of events (count = launches in the run).
struct ProfRec {
  int kclass;
  cudaEvent_t start, stop;
  uint32_t count;
};

}  // namespace

// Some sweeps captured as a CUDA graph, replayed while the schedule, the kernel
// variant, the energy log buffer and the spin buffer stay the same.
struct SweepGraph {
  cudaGraphExec_t exec = nullptr;
  hsg_schedule sched{};
  int variant = 0, period = 0, launches = 0;
  double* elog = nullptr;
  float4* spins = nullptr;  // current spin buffer when it was captured
};

struct hsg_ctx {
  int L = 0, Lh = 0;
  long long N = 0, Nh = 0;
  uint64_t seed = 0;
  uint32_t sample = 0, replica = 0, k0 = 0, k1 = 0;
  cudaStream_t stream = nullptr;
  int device = 0, sm_count = 0;
  long long l2_bytes = 0;  // the device's L2 size
  bool packed = false;          // spin layout: three fp32 arrays per colour instead of float4
  float4* spins = nullptr;      // [2][Nh] float4 (or [2][3][Nh] floats, packed), the current state
  float4* spins_alt = nullptr;  // [2][Nh], target of the temporally blocked sweeps (allocated on first use)
  float* J = nullptr;       // [3][2][Nh]
  bool have_J = false;
  // Halo-padded copy of J for the temporally blocked sweep's tensor boxes
  // (allocated with its tensor map by the first such sweep at L >= 32 when
  // the device has room for it; rebuilt after every change of J).
  float* Jpad = nullptr;
  bool Jpad_ok = false;  // Jpad holds the current J
  bool use_tma = false;  // bond_map describes Jpad
  CUtensorMap bond_map{};
  uint64_t sweep = 0;
  void* stage = nullptr;  // site-major staging for host copies
  size_t stage_bytes = 0;
  double* partials = nullptr;  // energy first-pass sums
  double* elog = nullptr;      // energy log
  int elog_cap = 0, elog_n = 0;
  hsg::ResultWords words{};
  double* host_e = nullptr;  // words.p, pinned: E/N and the bond-box wait flag
  bool prof = false;
  bool group = false;     // inside hsg_sweep: one event pair per run of same-class launches
  bool run_open = false;  // recs.back() still lacks its stop event
  std::vector<ProfRec> recs;
  std::vector<cudaEvent_t> free_events;
  uint64_t launches = 0;
  // Device counters: [0] the sweep counter the kernels read, [1] the energy
  // log position; the host mirrors both (sweep, elog_n).  [2] is set by a
  // temporally blocked sweep whose bounded wait for a bond box gave up.  [3]
  // counts the energy kernel's blocks, zero between launches.
  unsigned long long* d_ctr = nullptr;
  // Captured sweeps (see hsg_sweep): one graph for the bulk of a call and, without
  // cadences, one for what is left over or for calls shorter than the first.
  SweepGraph graph, short_graph;
  int short_want = 0;  // sweeps that the last call found no graph for (0: none)
  // While a period is captured: the sweep's number in it (the counter kernel
  // then runs once, at the period's end); -1 otherwise.
  int captured = -1;
  uint64_t captures = 0, replays = 0;  // for hsg_test_graph_counts
  hsg_schedule last{};                 // of the last hsg_sweep
  bool have_last = false;
  std::string err;
};

namespace {

hsg_status fail(hsg_ctx* c, hsg_status st, const std::string& msg) {
  if (c)
    c->err = msg;
  else
    g_thread_error = msg;
  return st;
}

hsg_status cuda_fail(hsg_ctx* c, cudaError_t e, const char* what) {
  std::string m = std::string(what) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")";
  if (e == cudaErrorMemoryAllocation) return fail(c, HSG_ENOMEM, m);
  return fail(c, HSG_ECUDA, m);
}

cudaError_t dev_alloc(void** p, size_t bytes, cudaStream_t s) {
  *p = nullptr;
  if (g_fail_alloc_countdown > 0 && --g_fail_alloc_countdown == 0) return cudaErrorMemoryAllocation;
  return hsg::device_alloc(p, bytes, s);
}

void dev_free(void* p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
}

cudaEvent_t take_event(hsg_ctx* c) {
  if (!c->free_events.empty()) {
    cudaEvent_t e = c->free_events.back();
    c->free_events.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
  return e;
}

// Record the stop event of the open profiler run, if any.
void close_run(hsg_ctx* c) {
  if (!c->run_open) return;
  cudaEvent_t b = take_event(c);
  if (b) cudaEventRecord(b, c->stream);
  c->recs.back().stop = b;
  c->run_open = false;
}

// Run `fn` (which launches `n_kernels` kernels on the context stream).  With
// the profiler on, each launch is bracketed by CUDA events on the stream;
// inside hsg_sweep consecutive launches of one class share one bracket, so
// that the events perturb the sweep as little as possible.
template <typename F>
hsg_status launch(hsg_ctx* c, int kclass, int n_kernels, const char* what, F&& fn) {
  if (c->prof && !(c->group && c->run_open && c->recs.back().kclass == kclass)) {
    close_run(c);
    cudaEvent_t a = take_event(c);
    if (!a) return fail(c, HSG_ECUDA, "cudaEventCreate failed");
    cudaEventRecord(a, c->stream);
    c->recs.push_back(ProfRec{kclass, a, nullptr, 0});
    c->run_open = true;
  }
  cudaError_t e = fn();
  if (e != cudaSuccess) {
    close_run(c);
    return cuda_fail(c, e, what);
  }
  c->launches += (uint64_t)n_kernels;
  if (c->prof) {
    c->recs.back().count += 1;
    if (!c->group) close_run(c);
  }
  return HSG_OK;
}

// Inside hsg_sweep: group same-class launches; the run closes on exit.
struct SweepGroup {
  hsg_ctx* c;
  explicit SweepGroup(hsg_ctx* ctx) : c(ctx) { c->group = true; }
  ~SweepGroup() {
    close_run(c);
    c->group = false;
  }
};

hsg_status ensure_stage(hsg_ctx* c, size_t bytes) {
  if (c->stage_bytes >= bytes) return HSG_OK;
  dev_free(c->stage, c->stream);
  c->stage = nullptr;
  c->stage_bytes = 0;
  cudaError_t e = dev_alloc(&c->stage, bytes, c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "staging buffer");
  c->stage_bytes = bytes;
  return HSG_OK;
}

void release(hsg_ctx* c) {
  if (!c) return;
  const hsg::DeviceGuard device_guard(c->device);
  cudaStream_t s = c->stream;
  dev_free(c->spins, s);
  dev_free(c->spins_alt, s);
  dev_free(c->J, s);
  dev_free(c->Jpad, s);
  dev_free(c->stage, s);
  dev_free(c->partials, s);
  dev_free(c->elog, s);
  dev_free(c->d_ctr, s);
  cudaStreamSynchronize(s);
  if (c->graph.exec) cudaGraphExecDestroy(c->graph.exec);
  if (c->short_graph.exec) cudaGraphExecDestroy(c->short_graph.exec);
  hsg::give_result_words(c->words);
  for (auto& r : c->recs) {
    cudaEventDestroy(r.start);
    if (r.stop) cudaEventDestroy(r.stop);
  }
  for (auto e : c->free_events) cudaEventDestroy(e);
  delete c;
}

hsg::SweepArgs sweep_args(hsg_ctx* c, int colour, float beta, float step, int hits) {
  hsg::SweepArgs a{};
  a.sweep_add = c->captured > 0 ? (uint32_t)c->captured : 0u;
  const int o = 1 - colour;
  a.own = c->spins + colour * c->Nh;
  a.oth = c->spins + o * c->Nh;
  a.jx_own = c->J + (0 + colour) * c->Nh;
  a.jy_own = c->J + (2 + colour) * c->Nh;
  a.jz_own = c->J + (4 + colour) * c->Nh;
  a.jx_oth = c->J + (0 + o) * c->Nh;
  a.jy_oth = c->J + (2 + o) * c->Nh;
  a.jz_oth = c->J + (4 + o) * c->Nh;
  a.L = c->L;
  a.Lh = c->Lh;
  a.colour = colour;
  a.hits = hits;
  a.k0 = c->k0;
  a.k1 = c->k1;
  a.sweep_lo = (uint32_t)(c->sweep & 0xFFFFFFFFu);
  a.sweep_hi = (uint32_t)(c->sweep >> 32);
  a.beta = beta;
  a.step = step;
  a.sweep_ptr = c->d_ctr;  // the device counter (plus sweep_add) equals c->sweep in stream order
  if (c->packed) {
    float* base = reinterpret_cast<float*>(c->spins);
    a.own = reinterpret_cast<float4*>(base + 3 * colour * c->Nh);
    a.oth = reinterpret_cast<const float4*>(base + 3 * o * c->Nh);
    a.packed = true;
    a.stride = (size_t)c->Nh;
  }
  return a;
}

hsg_status check_schedule(hsg_ctx* c, const hsg_schedule* s, bool need_kind) {
  if (!s) return fail(c, HSG_EINVAL, "schedule is NULL");
  if (need_kind && s->kind != HSG_NONE && s->kind != HSG_METROPOLIS && s->kind != HSG_HEATBATH &&
      s->kind != HSG_METROPOLIS_OR)
    return fail(c, HSG_EINVAL, "schedule.kind must be HSG_NONE, HSG_METROPOLIS, HSG_HEATBATH or HSG_METROPOLIS_OR");
  if (s->hits < 1 || s->hits > 65535) return fail(c, HSG_EINVAL, "schedule.hits must be in [1, 65535]");
  if (s->proposal != HSG_PROP_SPHERE && s->proposal != HSG_PROP_BALL)
    return fail(c, HSG_EINVAL, "schedule.proposal must be HSG_PROP_SPHERE or HSG_PROP_BALL");
  if (!(s->step > 0.0f) || !std::isfinite(s->step)) return fail(c, HSG_EINVAL, "schedule.step must be finite and > 0");
  if (s->n_or < 0) return fail(c, HSG_EINVAL, "schedule.n_or must be >= 0");
  if (!(s->T > 0.0)) return fail(c, HSG_EINVAL, "schedule.T must be > 0 (inf allowed)");
  if (s->renorm_every < 0 || s->energy_every < 0) return fail(c, HSG_EINVAL, "cadences must be >= 0");
  if (s->kernel != HSG_KERNEL_AUTO && s->kernel != HSG_KERNEL_GLOBAL && s->kernel != HSG_KERNEL_SLAB &&
      s->kernel != HSG_KERNEL_WAVE)
    return fail(c, HSG_EINVAL, "schedule.kernel must be HSG_KERNEL_AUTO, _GLOBAL, _SLAB or _WAVE");
  if (c->packed && (s->kernel == HSG_KERNEL_SLAB || s->kernel == HSG_KERNEL_WAVE))
    return fail(c, HSG_EINVAL, "the packed spin layout runs the global kernel only (HSG_KERNEL_AUTO or _GLOBAL)");
  return HSG_OK;
}

float beta_of(double T) { return std::isinf(T) ? 0.0f : (float)(1.0 / T); }

// HSG_KERNEL_AUTO: the temporally blocked over-relaxation once the spins
// and bonds (16 + 12 bytes per site) exceed 1.2 times L2 -- it saves HBM
// traffic, and pays where the sweeps stream most of their state from HBM; below,
// two half-sweeps, the second from the top down, find enough of it in L2.
// Measured on GB300 (126 MB L2), one OR sweep, global / wave: L = 152 (98 MB)
// 26.5 / 32.5 us, 160 (115 MB) 32.4 / 38.1, 176 (153 MB) 48.3 / 55.6, 184 (174 MB)
// 56.7 / 56.8, 192 64.4 / 60.7, 256 162 / 127.  Where a renormalisation is due
// after every sweep, which the wave fuses and the global kernel does not, from
// three quarters of L2: heat-bath + OR + renormalisation L = 154 93.9 / 89.8 us,
// 160 101.6 / 96.6, 176 143.4 / 136.8.
int pick_variant(const hsg_ctx* c, const hsg_schedule* s) {
  if (s->kernel != HSG_KERNEL_AUTO) return s->kernel;
  if (c->packed) return hsg::V_GLOBAL;
  const long long state = 28LL * c->N;
  const bool wave = s->renorm_every == 1 ? 4 * state > 3 * c->l2_bytes : 5 * state > 6 * c->l2_bytes;
  return wave ? hsg::V_WAVE : hsg::V_GLOBAL;
}

// Temporally blocked launches of one sweep under schedule s with the wave
// variant: one per over-relaxation sweep (the main update stays two
// half-sweeps).  Each one swaps the spin buffers.
int wave_sweeps_per_sweep(const hsg_schedule* s) { return s->n_or; }

hsg_status run_half_sweep(hsg_ctx* c, const hsg_schedule* s, int update, int colour) {
  int upd, kclass;
  if (update == HSG_OVERRELAX) {
    upd = hsg::U_OR;
    kclass = HSG_PROF_OVERRELAX;
  } else if (update == HSG_METROPOLIS) {
    upd = s->proposal == HSG_PROP_BALL ? hsg::U_MET_BALL : hsg::U_MET_SPHERE;
    kclass = HSG_PROF_METROPOLIS;
  } else if (update == HSG_METROPOLIS_OR) {
    upd = s->proposal == HSG_PROP_BALL ? hsg::U_MET_OR_BALL : hsg::U_MET_OR_SPHERE;
    kclass = HSG_PROF_METROPOLIS;
  } else {
    upd = hsg::U_HB;
    kclass = HSG_PROF_HEATBATH;
  }
  const hsg::SweepArgs a = sweep_args(c, colour, beta_of(s->T), s->step, s->hits);
  int variant = pick_variant(c, s);
  if (variant == hsg::V_WAVE) variant = hsg::V_GLOBAL;  // a single colour: the plain kernel
  return launch(c, kclass, 1, "half-sweep kernel", [&] { return hsg::launch_half_sweep(upd, variant, a, c->sm_count, c->stream); });
}

// Both colours of one over-relaxation sweep in one temporally blocked launch
// from c->spins into c->spins_alt (renormalising what it stores when
// `renorm`); then the two buffers swap.
hsg_status run_or_sweep_wave(hsg_ctx* c, bool renorm) {
  hsg::WaveArgs a{};
  a.src = c->spins;
  a.dst = c->spins_alt;
  a.J = c->J;
  a.L = c->L;
  a.Lh = c->Lh;
  a.renorm = renorm;
  a.bond_map = c->use_tma ? &c->bond_map : nullptr;
  a.err = c->d_ctr + 2;
  const int stall = g_test_stall_boxes.load();
  a.box_extra_tx = (stall & 1) ? 16u : 0u;
  a.c1_extra_arrivals = (stall & 2) ? 1u : 0u;
  hsg_status st = launch(c, renorm ? HSG_PROF_OVERRELAX_RENORM : HSG_PROF_OVERRELAX, 1, "over-relaxation sweep kernel",
                         [&] { return hsg::launch_or_sweep_wave(a, c->sm_count, c->stream); });
  if (st == HSG_OK) std::swap(c->spins, c->spins_alt);
  return st;
}

// The temporally blocked sweep's tensor-box bonds: at L >= 32, the first
// sweep allocates the halo-padded copy of J (when the device has room for
// it beside a margin of 1 GiB; else the sweep keeps its register loads) and
// encodes its tensor map; a copy older than J is rebuilt (one launch).
hsg_status prepare_bond_boxes(hsg_ctx* c) {
  if (c->L < hsg::kWaveTmaMinL || c->packed) return HSG_OK;
  if (!c->Jpad) {
    const size_t bytes = sizeof(float) * hsg::padded_bonds_elems(c->L);
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess || free_b + hsg::kept_bytes() < bytes + ((size_t)1 << 30)) {
      cudaGetLastError();
      return HSG_OK;  // no room: register loads
    }
    cudaError_t e = dev_alloc(reinterpret_cast<void**>(&c->Jpad), bytes, c->stream);
    if (e != cudaSuccess) {
      cudaGetLastError();
      c->Jpad = nullptr;
      return e == cudaErrorMemoryAllocation ? HSG_OK : cuda_fail(c, e, "padded couplings");
    }
    c->Jpad_ok = false;
    c->use_tma = hsg::encode_padded_bond_map(&c->bond_map, c->Jpad, c->L) == cudaSuccess;
  }
  if (c->use_tma && !c->Jpad_ok) {
    hsg_status st = launch(c, HSG_PROF_LAYOUT, 1, "coupling padding kernel",
                           [&] { return hsg::launch_pad_bonds(c->J, c->Jpad, c->L, c->stream); });
    if (st != HSG_OK) return st;
    c->Jpad_ok = true;
  }
  return HSG_OK;
}

// The bond-box wait flag of the temporally blocked sweeps, which the energy
// kernel has copied to the second pinned word: once the stream has been
// synchronised, HSG_ETIMEOUT if one of them gave up.
hsg_status check_box_waits(hsg_ctx* c) {
  if (!c->use_tma) return HSG_OK;
  unsigned long long flag = 0;
  std::memcpy(&flag, c->host_e + 1, sizeof(flag));
  if (!flag) return HSG_OK;
  // Reported once: the flag is cleared for the sweeps that follow.
  cudaError_t e = cudaMemsetAsync(c->d_ctr + 2, 0, sizeof(unsigned long long), c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "wait flag reset");
  c->host_e[1] = 0.0;
  return fail(c, HSG_ETIMEOUT,
              "an over-relaxation sweep gave up waiting for its couplings (bounded wait): the spins since are not "
              "valid");
}

// E/N into the energy log at the device position, or into the pinned result
// word (with the wait flag into the one beside it).
hsg_status run_energy(hsg_ctx* c, bool logged) {
  hsg::EnergyArgs a{};
  a.S = c->spins;
  a.packed = c->packed;
  a.J = c->J;
  a.L = c->L;
  a.partials = c->partials;
  a.ticket = reinterpret_cast<uint32_t*>(c->d_ctr + 3);
  a.out = logged ? c->elog : c->host_e;
  a.log_idx = logged ? c->d_ctr + 1 : nullptr;
  if (!logged && c->use_tma) {
    a.flag = c->d_ctr + 2;
    a.flag_out = reinterpret_cast<unsigned long long*>(c->host_e + 1);
  }
  return launch(c, HSG_PROF_ENERGY, logged ? 2 : 1, "energy kernel", [&] { return hsg::launch_energy(a, c->stream); });
}

hsg_status run_advance(hsg_ctx* c, uint64_t sweeps) {
  return launch(c, HSG_PROF_LAYOUT, 1, "counter kernel",
                [&] { return hsg::launch_add_u64(c->d_ctr, sweeps, c->stream); });
}

hsg_status run_renorm(hsg_ctx* c) {
  return launch(c, HSG_PROF_RENORM, 1, "renorm kernel",
                [&] { return hsg::launch_renorm(c->spins, c->packed, c->N, c->sm_count, c->stream); });
}

// One sweep's launches in schedule order; the host mirrors of the sweep
// counter and the energy-log position advance as the device ones will.
hsg_status enqueue_one_sweep(hsg_ctx* c, const hsg_schedule* s) {
  hsg_status st;
  const bool wave = pick_variant(c, s) == hsg::V_WAVE;
  if (s->kind != HSG_NONE)
    for (int colour = 0; colour < 2; ++colour)
      if ((st = run_half_sweep(c, s, s->kind, colour)) != HSG_OK) return st;
  // A renormalisation due after this sweep is fused into its last wave
  // launch (the same renorm_spin on the same values; the counter kernel in
  // between touches no spin).
  const bool renorm_due = s->renorm_every > 0 && (c->sweep + 1) % (uint64_t)s->renorm_every == 0;
  const bool fuse_renorm = renorm_due && wave && s->n_or > 0;
  for (int o = 0; o < s->n_or; ++o) {
    if (wave) {
      if ((st = run_or_sweep_wave(c, fuse_renorm && o == s->n_or - 1)) != HSG_OK) return st;
      continue;
    }
    for (int colour = 0; colour < 2; ++colour)
      if ((st = run_half_sweep(c, s, HSG_OVERRELAX, colour)) != HSG_OK) return st;
  }
  if (c->captured < 0 && (st = run_advance(c, 1)) != HSG_OK) return st;
  c->sweep += 1;
  if (renorm_due && !fuse_renorm)
    if ((st = run_renorm(c)) != HSG_OK) return st;
  if (s->energy_every > 0 && c->sweep % (uint64_t)s->energy_every == 0) {
    if ((st = run_energy(c, true)) != HSG_OK) return st;
    c->elog_n += 1;
  }
  return HSG_OK;
}

bool same_schedule(const hsg_schedule& a, const hsg_schedule& b) {
  return a.kind == b.kind && a.hits == b.hits && a.proposal == b.proposal && a.step == b.step && a.n_or == b.n_or &&
         a.T == b.T && a.renorm_every == b.renorm_every && a.energy_every == b.energy_every && a.kernel == b.kernel;
}

// Graph g is one of s, whichever spin buffer it starts from.
bool same_graph(const hsg_ctx* c, const SweepGraph& g, const hsg_schedule* s, int variant) {
  return g.exec && same_schedule(g.sched, *s) && g.variant == variant && g.elog == c->elog;
}

bool graph_matches(const hsg_ctx* c, const SweepGraph& g, const hsg_schedule* s, int variant) {
  return same_graph(c, g, s, variant) && g.spins == c->spins;
}

// Half-sweep and over-relaxation launches of one sweep (at least 1).
int sweep_launches(const hsg_schedule* s, int variant) {
  return std::max(1, (s->kind != HSG_NONE ? 2 : 0) + (variant == hsg::V_WAVE ? 1 : 2) * s->n_or);
}

// Sweeps in one graph for a schedule without cadences, n of them asked for:
// the largest divisor of n up to what one graph is given (a multiple of
// `unit`), or that many if none is half as long; a graph that is there is kept
// if it is half as long or n is less than eight of it.  One graph is given up to
// kGraphSweeps sweeps, but no more than kGraphLaunches launches or an eighth of n:
// capturing and instantiating costs 2.9 us a launch, which a schedule that is used
// once (a temperature per call) does not earn back.  L = 40, heat-bath + 20 OR, a new T
// for every 5, 10, 16 sweeps, us a call: 611, 1195, 1895 with all of them in a graph,
// 307, 598, 947 with one each; sweep(31) again and again 1683 with 16, 1795 with one.
int free_period(const hsg_ctx* c, const hsg_schedule* s, int variant, int n, int unit) {
  const int fit = std::max(kGraphLaunches / sweep_launches(s, variant), n / 8);
  const int most = std::max(1, std::min(kGraphSweeps, fit) / unit) * unit;
  const int there = graph_matches(c, c->graph, s, variant) ? c->graph.period : 0;
  if (there > 0 && there % unit == 0 && (2 * there >= most || n < 8 * there)) return there;
  if (n < 2 * unit) return unit;
  if (n <= most) return n / unit * unit;
  int best = unit;
  for (int d = unit; d <= most; d += unit)
    if (n % d == 0) best = d;
  return 2 * best >= most ? best : most;
}

// Capture `period` sweeps starting at the current counter (with cadences a
// multiple of the period) into *g.  Capturing runs nothing, so the host mirrors
// are restored afterwards.
hsg_status capture_period(hsg_ctx* c, const hsg_schedule* s, int variant, int period, SweepGraph* g) {
  if (g->exec) cudaGraphExecDestroy(g->exec);
  g->exec = nullptr;
  const uint64_t sweep0 = c->sweep, launches0 = c->launches;
  const int elog0 = c->elog_n;
  float4* const spins0 = c->spins;
  float4* const alt0 = c->spins_alt;
  cudaError_t e = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return cuda_fail(c, e, "sweep capture");
  hsg_status st = HSG_OK;
  for (int j = 0; j < period && st == HSG_OK; ++j) {
    c->captured = j;
    st = enqueue_one_sweep(c, s);
  }
  c->captured = -1;
  if (st == HSG_OK) st = run_advance(c, (uint64_t)period);
  cudaGraph_t captured = nullptr;
  e = cudaStreamEndCapture(c->stream, &captured);
  const int launches = (int)(c->launches - launches0);
  c->launches = launches0;
  c->sweep = sweep0;
  c->elog_n = elog0;
  c->spins = spins0;
  c->spins_alt = alt0;
  if (st == HSG_OK && e == cudaSuccess) e = cudaGraphInstantiate(&g->exec, captured, 0);
  if (captured) cudaGraphDestroy(captured);
  if (st != HSG_OK) return st;
  if (e != cudaSuccess) {
    g->exec = nullptr;
    return cuda_fail(c, e, "sweep graph");
  }
  c->captures += 1;
  g->sched = *s;
  g->variant = variant;
  g->period = period;
  g->launches = launches;
  g->elog = c->elog;
  g->spins = spins0;
  return HSG_OK;
}

// The graph for the last `left` sweeps of a call without cadences, fewer than the
// bulk's graph holds: the short graph that is there, or, where the call before
// had as many left, one captured now; else nullptr (they are launched directly).
// Calls of changing lengths so end up with a graph that divides what they leave.
// us a call of sweep(n) and energy() after a long call, direct launches / short graph,
// heat-bath + n_or over-relaxation sweeps:
//   n_or = 0   n = 1: L = 40 23.9 / 23.0, 66 29.5 / 27.4, 128 54.2 / 51.2; n = 3: 33.4 / 29.9, 43.5 / 40.0, 115 / 101
//   n_or = 2   n = 1: 29.5 / 27.7, 38.9 / 37.0, 88 / 79; n = 5: 74 / 62, 107 / 94, 350 / 287
//   n_or = 20  n = 1: 88 / 73, 129 / 113, 394 / 319; n = 5: 367 / 288, 552 / 471, 1864 / 1486
hsg_status pick_short(hsg_ctx* c, const hsg_schedule* s, int variant, int left, int unit, SweepGraph** g) {
  *g = nullptr;
  const int len = left / unit * unit;
  if (len == 0) return HSG_OK;
  if (graph_matches(c, c->short_graph, s, variant) && c->short_graph.period <= left) {
    *g = &c->short_graph;
  } else if (c->short_want == len) {
    const hsg_status st = capture_period(c, s, variant, len, &c->short_graph);
    if (st != HSG_OK) return st;
    *g = &c->short_graph;
  } else {
    c->short_want = len;
  }
  return HSG_OK;
}

// The main update's kind in a whole-schedule kernel (U_OR: none).
int main_update(const hsg_schedule* s) {
  const bool ball = s->proposal == HSG_PROP_BALL;
  switch (s->kind) {
    case HSG_METROPOLIS: return ball ? hsg::U_MET_BALL : hsg::U_MET_SPHERE;
    case HSG_METROPOLIS_OR: return ball ? hsg::U_MET_OR_BALL : hsg::U_MET_OR_SPHERE;
    case HSG_HEATBATH: return hsg::U_HB;
    default: return hsg::U_OR;
  }
}

// Whether the caller captures the context's stream.
bool stream_captured(const hsg_ctx* c) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(c->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
}

// Whether hsg_sweep runs schedule s in the resident kernel
// (hsg_resident.cu): AUTO only, and neither under the profiler, whose classes
// are single half-sweeps, nor while the caller captures the stream (what a
// capture takes, and what it refuses, stays with the half-sweep launches),
// and where the device can place its cluster.
bool use_resident(const hsg_ctx* c, const hsg_schedule* s) {
  if (s->kernel != HSG_KERNEL_AUTO || c->prof || !hsg::resident_takes(main_update(s), c->L, s->hits)) return false;
  if (s->kind == HSG_NONE && s->n_or == 0) return false;
  if (stream_captured(c)) return false;
  return hsg::resident_fits(main_update(s), c->L, 1, false, c->sm_count);
}

// n_sweeps sweeps in the resident kernel, a launch for as many as it takes at a time
// or up to an energy due.
hsg_status run_resident(hsg_ctx* c, const hsg_schedule* s, int n_sweeps) {
  const int upd = main_update(s);
  hsg_status st;
  for (int k = 0; k < n_sweeps;) {
    uint64_t m = (uint64_t)std::min(n_sweeps - k, hsg::kResidentSweeps);
    if (s->energy_every > 0) m = std::min(m, (uint64_t)s->energy_every - c->sweep % (uint64_t)s->energy_every);
    hsg::ResidentArgs a{};
    a.L = (uint32_t)c->L;
    a.packed = c->packed;
    a.sweeps = (uint32_t)m;
    a.per_sweep = (s->kind != HSG_NONE ? 2u : 0u) + 2u * (uint32_t)s->n_or;
    a.renorm_every = (uint32_t)s->renorm_every;
    a.step = s->step;
    a.hits = s->hits;
    a.sweep_ptr = c->d_ctr;
    a.n = 1;
    a.spins = c->spins;
    a.J = c->J;
    a.k0 = c->k0;
    a.k1 = c->k1;
    a.beta = beta_of(s->T);
    st = launch(c, HSG_PROF_LAYOUT, 1, "resident sweeps kernel", [&] { return hsg::launch_resident(upd, a, c->sm_count, c->stream); });
    if (st != HSG_OK) return st;
    c->sweep += m;
    k += (int)m;
    if (s->energy_every > 0 && c->sweep % (uint64_t)s->energy_every == 0) {
      if ((st = run_energy(c, true)) != HSG_OK) return st;
      c->elog_n += 1;
    }
  }
  return HSG_OK;
}

hsg_status grow_elog(hsg_ctx* c, int need) {
  if (need <= c->elog_cap) return HSG_OK;
  int cap = c->elog_cap > 0 ? c->elog_cap : kElogInit;
  while (cap < need) cap *= 2;
  void* p = nullptr;
  cudaError_t e = dev_alloc(&p, sizeof(double) * (size_t)cap, c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "energy log");
  if (c->elog_n > 0) {
    e = cudaMemcpyAsync(p, c->elog, sizeof(double) * (size_t)c->elog_n, cudaMemcpyDeviceToDevice, c->stream);
    if (e != cudaSuccess) {
      dev_free(p, c->stream);
      return cuda_fail(c, e, "energy log copy");
    }
  }
  dev_free(c->elog, c->stream);
  c->elog = static_cast<double*>(p);
  c->elog_cap = cap;
  return HSG_OK;
}

}  // namespace

void hsg::set_thread_error(const std::string& msg) { g_thread_error = msg; }

extern "C" {

hsg_status hsg_create(hsg_ctx** out, int L, uint64_t seed, uint32_t sample, uint32_t replica, void* cuda_stream) {
  return hsg_create_layout(out, L, seed, sample, replica, cuda_stream, HSG_LAYOUT_FLOAT4);
}

hsg_status hsg_create_layout(hsg_ctx** out, int L, uint64_t seed, uint32_t sample, uint32_t replica,
                             void* cuda_stream, int layout) {
  if (!out) return fail(nullptr, HSG_EINVAL, "out is NULL");
  *out = nullptr;
  if (L < 4 || L > kMaxL || (L & 1))
    return fail(nullptr, HSG_EINVAL, "L must be even and in [4, " + std::to_string(kMaxL) + "]");
  if (layout != HSG_LAYOUT_FLOAT4 && layout != HSG_LAYOUT_PACKED)
    return fail(nullptr, HSG_EINVAL, "layout must be HSG_LAYOUT_FLOAT4 or HSG_LAYOUT_PACKED");
  if (!hsg::key_stream_ok(sample, replica)) return fail(nullptr, HSG_EINVAL, hsg::kKeyStreamMsg);
  hsg_ctx* c = new (std::nothrow) hsg_ctx();
  if (!c) return fail(nullptr, HSG_ENOMEM, "host allocation failed");
  c->packed = layout == HSG_LAYOUT_PACKED;
  c->L = L;
  c->Lh = L / 2;
  c->N = (long long)L * L * L;
  c->Nh = c->N / 2;
  c->seed = seed;
  c->sample = sample;
  c->replica = replica;
  // Key of (seed, sample, replica): low seed word, high seed word XOR the
  // Weyl-scrambled stream number 2*sample + replica.
  c->k0 = (uint32_t)(seed & 0xFFFFFFFFu);
  c->k1 = (uint32_t)(seed >> 32) ^ ((2u * sample + replica) * 0x9E3779B9u);
  c->stream = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = cudaGetDevice(&c->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device);
  int l2 = 0;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, c->device);
  c->l2_bytes = l2;
  if (e != cudaSuccess) {
    hsg_status st = cuda_fail(nullptr, e, "no usable CUDA device");
    delete c;
    return st;
  }
  struct {
    void** p;
    size_t bytes;
    const char* what;
  } allocs[] = {
      {reinterpret_cast<void**>(&c->spins), (c->packed ? 3 * sizeof(float) : sizeof(float4)) * (size_t)c->N, "spins"},
      {reinterpret_cast<void**>(&c->J), sizeof(float) * 3 * (size_t)c->N, "couplings"},
      {reinterpret_cast<void**>(&c->partials), sizeof(double) * hsg::energy_partials(L), "energy partials"},
      {reinterpret_cast<void**>(&c->d_ctr), kCounters * sizeof(unsigned long long), "device counters"},
  };
  for (auto& a : allocs) {
    e = dev_alloc(a.p, a.bytes, c->stream);
    if (e != cudaSuccess) {
      hsg_status st = cuda_fail(nullptr, e, a.what);
      release(c);
      return st;
    }
  }
  hsg_status st = grow_elog(c, kElogInit);
  if (st != HSG_OK) {
    g_thread_error = c->err;
    release(c);
    return st;
  }
  e = hsg::take_result_words(&c->words);
  c->host_e = c->words.p;
  if (e == cudaSuccess) e = cudaMemsetAsync(c->d_ctr, 0, kCounters * sizeof(unsigned long long), c->stream);
  if (e != cudaSuccess) {
    st = cuda_fail(nullptr, e, "pinned host slot / counters");
    release(c);
    return st;
  }
  st = launch(c, HSG_PROF_INIT, 1, "init kernel",
              [&] { return hsg::launch_init_spins(c->spins, c->packed, L, c->k0, c->k1, c->stream); });
  if (st != HSG_OK) {
    g_thread_error = c->err;
    release(c);
    return st;
  }
  *out = c;
  return HSG_OK;
}

hsg_status hsg_destroy(hsg_ctx* ctx) {
  release(ctx);
  return HSG_OK;
}

hsg_status hsg_release_memory(void) {
  const cudaError_t e = hsg::release_kept();
  return e == cudaSuccess ? HSG_OK : cuda_fail(nullptr, e, "memory release");
}

hsg_status hsg_set_couplings(hsg_ctx* c, const void* J, int dtype, int where) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (!J) return fail(c, HSG_EINVAL, "J is NULL");
  if (dtype != HSG_F32 && dtype != HSG_F64) return fail(c, HSG_EINVAL, "dtype must be HSG_F32 or HSG_F64");
  if (where != HSG_HOST && where != HSG_DEVICE) return fail(c, HSG_EINVAL, "where must be HSG_HOST or HSG_DEVICE");
  const bool f64 = dtype == HSG_F64;
  const void* src = J;
  if (where == HSG_HOST) {
    const size_t bytes = (f64 ? sizeof(double) : sizeof(float)) * 3 * (size_t)c->N;
    hsg_status st = ensure_stage(c, bytes);
    if (st != HSG_OK) return st;
    cudaError_t e = cudaMemcpyAsync(c->stage, J, bytes, cudaMemcpyHostToDevice, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "coupling upload");
    src = c->stage;
  }
  // With a padded copy in use (temporally blocked sweeps at L >= 32) the
  // same launch writes it too.
  float* const Jp = c->use_tma ? c->Jpad : nullptr;
  hsg_status st = launch(c, HSG_PROF_LAYOUT, 1, "coupling layout kernel",
                         [&] { return hsg::launch_scatter_couplings(src, f64, c->J, c->L, c->stream, Jp); });
  if (st != HSG_OK) return st;
  if (where == HSG_HOST) {
    // The caller may reuse its array as soon as we return.
    cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "coupling upload sync");
  }
  c->have_J = true;
  c->Jpad_ok = Jp != nullptr;
  return HSG_OK;
}

hsg_status hsg_generate_couplings(hsg_ctx* c) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  // Key of (seed, sample, replica 0): replicas of one sample share J.
  const uint32_t k1 = (uint32_t)(c->seed >> 32) ^ ((2u * c->sample) * 0x9E3779B9u);
  hsg_status st = launch(c, HSG_PROF_LAYOUT, 1, "coupling generator kernel",
                         [&] { return hsg::launch_gen_couplings(c->J, c->L, c->k0, k1, c->stream); });
  if (st == HSG_OK) {
    c->have_J = true;
    c->Jpad_ok = false;
  }
  return st;
}

hsg_status hsg_get_couplings(hsg_ctx* c, float* out, int where) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (!out) return fail(c, HSG_EINVAL, "out is NULL");
  if (where != HSG_HOST && where != HSG_DEVICE) return fail(c, HSG_EINVAL, "where must be HSG_HOST or HSG_DEVICE");
  if (!c->have_J) return fail(c, HSG_EINVAL, "couplings not set");
  const size_t bytes = sizeof(float) * 3 * (size_t)c->N;
  float* dst = out;
  if (where == HSG_HOST) {
    hsg_status st = ensure_stage(c, bytes);
    if (st != HSG_OK) return st;
    dst = static_cast<float*>(c->stage);
  }
  hsg_status st = launch(c, HSG_PROF_LAYOUT, 1, "coupling gather kernel",
                         [&] { return hsg::launch_gather_couplings(c->J, dst, c->L, c->stream); });
  if (st != HSG_OK) return st;
  if (where == HSG_HOST) {
    cudaError_t e = cudaMemcpyAsync(out, dst, bytes, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "coupling readback");
  }
  return HSG_OK;
}

hsg_status hsg_sweep(hsg_ctx* c, const hsg_schedule* s, int n_sweeps) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  hsg_status st = check_schedule(c, s, true);
  if (st != HSG_OK) return st;
  if (n_sweeps < 0) return fail(c, HSG_EINVAL, "n_sweeps must be >= 0");
  if (!c->have_J) return fail(c, HSG_EINVAL, "couplings not set: call hsg_set_couplings first");
  if (s->energy_every > 0) {
    const uint64_t end = c->sweep + (uint64_t)n_sweeps;
    const uint64_t logged = end / (uint64_t)s->energy_every - c->sweep / (uint64_t)s->energy_every;
    st = grow_elog(c, c->elog_n + (int)logged);
    if (st != HSG_OK) return st;
  }
  if (use_resident(c, s)) return run_resident(c, s, n_sweeps);
  const int variant = pick_variant(c, s);
  const int swaps = variant == hsg::V_WAVE ? wave_sweeps_per_sweep(s) : 0;
  if (swaps > 0 && !c->spins_alt) {
    cudaError_t e = dev_alloc(reinterpret_cast<void**>(&c->spins_alt), sizeof(float4) * (size_t)c->N, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "second spin buffer");
  }
  if (swaps > 0 && (st = prepare_bond_boxes(c)) != HSG_OK) return st;
  SweepGroup group_guard(c);
  int k = 0;
  // Sweeps run in periods of P = lcm(renorm_every, energy_every) sweeps.  On a non-default stream and without the
  // profiler, a period that starts at a multiple of P is captured once as a
  // CUDA graph (the kernels read the sweep counter and the energy-log
  // position from device memory) and replayed; other sweeps are launched
  // directly.  Both paths issue the same kernels in the same order.  A
  // captured period leaves the spins in the buffer it found them in (an even
  // number of buffer swaps), so that the graph can be replayed.  Without
  // cadences the period is as many sweeps as one graph is given (free_period: a
  // graph of one sweep costs 4-8 us of launching each), and what is left over may have
  // a graph of its own (pick_short).
  const bool cadence = s->renorm_every > 0 || s->energy_every > 0;
  long long period = 1;
  if (s->renorm_every > 0) period = std::lcm(period, (long long)s->renorm_every);
  if (s->energy_every > 0) period = std::lcm(period, (long long)s->energy_every);
  if ((period * swaps) % 2 == 1) period *= 2;
  const int unit = cadence ? 1 : (int)period;  // without cadences: 1, or 2 with an odd number of swaps
  if (!cadence && n_sweeps > 0) {
    // The graph there is starts from the other buffer (an odd number of swaps has
    // been launched since): one direct sweep leads back to it.
    if (swaps % 2 == 1 && !c->prof && same_graph(c, c->graph, s, variant) && c->graph.spins == c->spins_alt) {
      if ((st = enqueue_one_sweep(c, s)) != HSG_OK) return st;
      k = 1;
    }
    period = free_period(c, s, variant, n_sweeps - k, unit);
  }
  const bool seen = c->have_last && same_schedule(c->last, *s);
  if (!seen) c->short_want = 0;
  bool graphs = c->stream != nullptr && !c->prof && period <= kMaxGraphPeriod;
  // A new schedule's graph that this call would launch only once is not captured
  // where the host cannot hide it behind the kernels: direct launches cost it 1.65 us
  // each against 2.9.  A new T for each sweep of heat-bath + 20 OR, us, captured / direct:
  // L = 40 132 / 75, 66 140 / 109, 100 200 / 266; + 2 OR: 32 / 16, 38 / 20, 45 / 44.
  if (graphs && c->L <= kOnceMaxL && n_sweeps - k < 2 * period && !seen &&
      !same_graph(c, c->graph, s, variant) && !stream_captured(c))
    graphs = false;
  c->last = *s;
  c->have_last = true;
  // Asked once a call where there is none, and not while the caller captures: the
  // direct launches can be part of its graph, a graph of ours can not.
  bool look_short = graphs && !cadence && !stream_captured(c);
  while (k < n_sweeps) {
    SweepGraph* g = nullptr;
    if (graphs && (!cadence || c->sweep % (uint64_t)period == 0) && n_sweeps - k >= period) {
      g = &c->graph;
      if ((g->period != period || !graph_matches(c, *g, s, variant)) &&
          (st = capture_period(c, s, variant, (int)period, g)) != HSG_OK)
        return st;
    } else if (look_short) {
      if ((st = pick_short(c, s, variant, n_sweeps - k, unit, &g)) != HSG_OK) return st;
      look_short = g != nullptr;
    }
    if (g) {
      cudaError_t e = cudaGraphLaunch(g->exec, c->stream);
      if (e != cudaSuccess) return cuda_fail(c, e, "sweep graph launch");
      c->replays += 1;
      c->launches += (uint64_t)g->launches;
      c->sweep += (uint64_t)g->period;
      if (s->energy_every > 0) c->elog_n += g->period / s->energy_every;
      k += g->period;
    } else {
      if ((st = enqueue_one_sweep(c, s)) != HSG_OK) return st;
      k += 1;
    }
  }
  return HSG_OK;
}

hsg_status hsg_energy(hsg_ctx* c, double* e_per_spin) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (!e_per_spin) return fail(c, HSG_EINVAL, "e_per_spin is NULL");
  if (!c->have_J) return fail(c, HSG_EINVAL, "couplings not set");
  hsg_status st = run_energy(c, false);
  if (st != HSG_OK) return st;
  const cudaError_t e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "energy readback");
  *e_per_spin = *c->host_e;
  return check_box_waits(c);
}

hsg_status hsg_get_energy_log(hsg_ctx* c, double* out, int max_n, int* n) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (max_n < 0 || (max_n > 0 && !out)) return fail(c, HSG_EINVAL, "bad output buffer");
  const int k = max_n < c->elog_n ? max_n : c->elog_n;
  cudaError_t e = cudaSuccess;
  if (k > 0) e = cudaMemcpyAsync(out, c->elog, sizeof(double) * (size_t)k, cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "energy log readback");
  if (n) *n = c->elog_n;
  return HSG_OK;
}

hsg_status hsg_clear_energy_log(hsg_ctx* c) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  hsg_status st = launch(c, HSG_PROF_LAYOUT, 1, "counter kernel",
                         [&] { return hsg::launch_set_u64(c->d_ctr + 1, 0, c->stream); });
  if (st != HSG_OK) return st;
  c->elog_n = 0;
  return HSG_OK;
}

hsg_status hsg_get_spins(hsg_ctx* c, float* out, int where) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (!out) return fail(c, HSG_EINVAL, "out is NULL");
  if (where != HSG_HOST && where != HSG_DEVICE) return fail(c, HSG_EINVAL, "where must be HSG_HOST or HSG_DEVICE");
  const size_t bytes = sizeof(float) * 3 * (size_t)c->N;
  float* dst = out;
  if (where == HSG_HOST) {
    hsg_status st = ensure_stage(c, bytes);
    if (st != HSG_OK) return st;
    dst = static_cast<float*>(c->stage);
  }
  hsg_status st = launch(c, HSG_PROF_LAYOUT, 1, "spin gather kernel",
                         [&] { return hsg::launch_gather_spins(c->spins, c->packed, dst, c->L, c->stream); });
  if (st != HSG_OK) return st;
  if (where == HSG_HOST) {
    cudaError_t e = cudaMemcpyAsync(out, dst, bytes, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "spin readback");
  }
  return HSG_OK;
}

hsg_status hsg_set_spins(hsg_ctx* c, const float* in, int where) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (!in) return fail(c, HSG_EINVAL, "in is NULL");
  if (where != HSG_HOST && where != HSG_DEVICE) return fail(c, HSG_EINVAL, "where must be HSG_HOST or HSG_DEVICE");
  const float* src = in;
  if (where == HSG_HOST) {
    const size_t bytes = sizeof(float) * 3 * (size_t)c->N;
    hsg_status st = ensure_stage(c, bytes);
    if (st != HSG_OK) return st;
    cudaError_t e = cudaMemcpyAsync(c->stage, in, bytes, cudaMemcpyHostToDevice, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "spin upload");
    src = static_cast<const float*>(c->stage);
  }
  hsg_status st = launch(c, HSG_PROF_LAYOUT, 1, "spin scatter kernel",
                         [&] { return hsg::launch_scatter_spins(src, c->spins, c->packed, c->L, c->stream); });
  if (st != HSG_OK) return st;
  if (where == HSG_HOST) {
    cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "spin upload sync");
  }
  return HSG_OK;
}

hsg_status hsg_get_sites(hsg_ctx* c, const uint32_t* sites, int n, float* spins, float* bonds) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (n < 0) return fail(c, HSG_EINVAL, "n must be >= 0");
  if (n == 0) return HSG_OK;
  if (!sites || !spins) return fail(c, HSG_EINVAL, "sites and spins must not be NULL");
  if (bonds && !c->have_J) return fail(c, HSG_EINVAL, "couplings not set");
  for (int k = 0; k < n; ++k)
    if ((long long)sites[k] >= c->N) return fail(c, HSG_EINVAL, "site index out of range");
  const size_t nb = (size_t)n;
  hsg_status st = ensure_stage(c, nb * (4 + 12 + 12));
  if (st != HSG_OK) return st;
  uint32_t* d_sites = static_cast<uint32_t*>(c->stage);
  float* d_spins = reinterpret_cast<float*>(d_sites + nb);
  float* d_bonds = d_spins + 3 * nb;
  cudaError_t e = cudaMemcpyAsync(d_sites, sites, 4 * nb, cudaMemcpyHostToDevice, c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "site list upload");
  st = launch(c, HSG_PROF_LAYOUT, 1, "site gather kernel",
              [&] {
                return hsg::launch_gather_sites(c->spins, c->packed, c->J, c->L, d_sites, n, d_spins, d_bonds,
                                                c->stream);
              });
  if (st != HSG_OK) return st;
  e = cudaMemcpyAsync(spins, d_spins, 12 * nb, cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess && bonds) e = cudaMemcpyAsync(bonds, d_bonds, 12 * nb, cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "site readback");
  return HSG_OK;
}

hsg_status hsg_get_sweep(hsg_ctx* c, uint64_t* sweep) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (!sweep) return fail(c, HSG_EINVAL, "sweep is NULL");
  *sweep = c->sweep;
  return HSG_OK;
}

hsg_status hsg_set_sweep(hsg_ctx* c, uint64_t sweep) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  hsg_status st = launch(c, HSG_PROF_LAYOUT, 1, "counter kernel",
                         [&] { return hsg::launch_set_u64(c->d_ctr, sweep, c->stream); });
  if (st != HSG_OK) return st;
  c->sweep = sweep;
  return HSG_OK;
}

hsg_status hsg_half_sweep(hsg_ctx* c, const hsg_schedule* s, int update, int colour) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  hsg_status st = check_schedule(c, s, false);
  if (st != HSG_OK) return st;
  if (update != HSG_OVERRELAX && update != HSG_METROPOLIS && update != HSG_HEATBATH && update != HSG_METROPOLIS_OR)
    return fail(c, HSG_EINVAL, "update must be HSG_OVERRELAX, HSG_METROPOLIS, HSG_HEATBATH or HSG_METROPOLIS_OR");
  if (colour != 0 && colour != 1) return fail(c, HSG_EINVAL, "colour must be 0 or 1");
  if (!c->have_J) return fail(c, HSG_EINVAL, "couplings not set");
  return run_half_sweep(c, s, update, colour);
}

hsg_status hsg_renorm(hsg_ctx* c) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  return run_renorm(c);
}

hsg_status hsg_kernel_for(hsg_ctx* c, const hsg_schedule* s, int* kernel) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (!kernel) return fail(c, HSG_EINVAL, "kernel is NULL");
  hsg_status st = check_schedule(c, s, true);
  if (st != HSG_OK) return st;
  *kernel = pick_variant(c, s);
  return HSG_OK;
}

hsg_status hsg_profile(hsg_ctx* c, int on) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (!on) close_run(c);
  c->prof = on != 0;
  return HSG_OK;
}

hsg_status hsg_profile_read(hsg_ctx* c, int kclass, double* total_ms, uint64_t* launches) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (kclass < 0 || kclass >= HSG_PROF_COUNT) return fail(c, HSG_EINVAL, "bad kernel class");
  close_run(c);
  cudaError_t e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "profile sync");
  double ms = 0.0;
  uint64_t n = 0;
  for (const auto& r : c->recs) {
    if (r.kclass != kclass || !r.stop) continue;
    float t = 0.0f;
    e = cudaEventElapsedTime(&t, r.start, r.stop);
    if (e != cudaSuccess) return cuda_fail(c, e, "cudaEventElapsedTime");
    ms += t;
    n += r.count;
  }
  if (total_ms) *total_ms = ms;
  if (launches) *launches = n;
  return HSG_OK;
}

hsg_status hsg_profile_reset(hsg_ctx* c) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  cudaError_t e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "profile sync");
  close_run(c);
  for (auto& r : c->recs) {
    c->free_events.push_back(r.start);
    if (r.stop) c->free_events.push_back(r.stop);
  }
  c->recs.clear();
  return HSG_OK;
}

hsg_status hsg_launch_count(hsg_ctx* c, uint64_t* launches) {
  if (!c) return fail(nullptr, HSG_EINVAL, "ctx is NULL");
  const hsg::DeviceGuard device_guard(c->device);
  if (device_guard.status() != cudaSuccess) return cuda_fail(c, device_guard.status(), "cudaSetDevice");
  if (!launches) return fail(c, HSG_EINVAL, "launches is NULL");
  *launches = c->launches;
  return HSG_OK;
}

const char* hsg_last_error(const hsg_ctx* c) { return c ? c->err.c_str() : g_thread_error.c_str(); }

const char* hsg_status_string(hsg_status s) {
  switch (s) {
    case HSG_OK: return "HSG_OK";
    case HSG_EINVAL: return "HSG_EINVAL";
    case HSG_ENOMEM: return "HSG_ENOMEM";
    case HSG_ECUDA: return "HSG_ECUDA";
    case HSG_ETIMEOUT: return "HSG_ETIMEOUT";
    case HSG_EBUSY: return "HSG_EBUSY";
    default: return "HSG_UNKNOWN";
  }
}

int hsg_version(void) { return kVersion; }

hsg_status hsg_philox(uint64_t seed, uint32_t sample, uint32_t replica, uint32_t c1, uint32_t c2, uint32_t c3,
                      uint32_t n, uint32_t* out, void* cuda_stream) {
  if (!out) return fail(nullptr, HSG_EINVAL, "out is NULL");
  if (reinterpret_cast<uintptr_t>(out) % 16 != 0) return fail(nullptr, HSG_EINVAL, "out must be 16-byte aligned");
  if (!hsg::key_stream_ok(sample, replica)) return fail(nullptr, HSG_EINVAL, hsg::kKeyStreamMsg);
  const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFu);
  const uint32_t k1 = (uint32_t)(seed >> 32) ^ ((2u * sample + replica) * 0x9E3779B9u);
  cudaError_t e = hsg::launch_philox(k0, k1, c1, c2, c3, n, out, static_cast<cudaStream_t>(cuda_stream));
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "philox kernel");
  return HSG_OK;
}

hsg_status hsg_test_stall_tensor_loads(int on) {
  if (on < 0 || on > 3) return fail(nullptr, HSG_EINVAL, "on must be 0 .. 3");
  g_test_stall_boxes.store(on);
  return HSG_OK;
}

hsg_status hsg_test_graph_counts(hsg_ctx* c, uint64_t* captured, uint64_t* launched) {
  if (!c || !captured || !launched) return fail(c, HSG_EINVAL, "NULL argument");
  *captured = c->captures;
  *launched = c->replays;
  return HSG_OK;
}

hsg_status hsg_test_no_clusters(int on) {
  if (on != 0 && on != 1) return fail(nullptr, HSG_EINVAL, "on must be 0 or 1");
  hsg::test_no_clusters(on == 1);
  return HSG_OK;
}

hsg_status hsg_test_fail_alloc(int k) {
  if (k < 0) return fail(nullptr, HSG_EINVAL, "k must be >= 0");
  g_fail_alloc_countdown = k;
  return HSG_OK;
}

}  // extern "C"

// re_capi.cu -- host side of the C ABI declared in include/re.h: contexts,
// device memory, launch configuration, the advance / exchange loop (optionally
// captured in a CUDA graph), getters, the autotuner and the stateless entry
// points.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "re.h"
#include "re_internal.h"

namespace {
// An NVTX range over one API call (shown by nsys / ncu timelines; header-only
// NVTX costs nothing when no tool is attached).
struct ApiRange {
  explicit ApiRange(const char* name) { nvtxRangePushA(name); }
  ~ApiRange() { nvtxRangePop(); }
};
}  // namespace

using re::EnsDev;
using re::finish_ens;
using re::LaunchCfg;
using re::RepDev;
using re::StateDev;
using re::choose_cells;
using re::set_capacity;

namespace re {

// Cells of the plain path's list build (and of the spatial sort):
// nc = floor(L / (rlist / m)) per side, scanned over a
// (2m + 1)^3 neighbourhood; cells only pay when 2m + 1 < nc.  m is chosen
// to minimise candidates per atom plus a per-cell visiting cost.
void choose_cells(double L, double rlist, int N, int want_m, int* nc_out, int* m_out) {
  double best = (double)N;  // all pairs
  int bnc = 0, bm = 0;
  for (int m = 1; m <= 3; ++m) {
    if (want_m > 0 && m != want_m) continue;
    const int nc = (int)std::floor(L / (rlist / m));
    if (nc < 2 * m + 2 || nc * nc * nc > 65535) continue;
    const double span = 2.0 * m + 1.0;
    const double cost = N * span * span * span / ((double)nc * nc * nc) + 4.0 * span * span * span;
    if (cost < best) {
      best = cost;
      bnc = nc;
      bm = m;
    }
  }
  *nc_out = bnc;
  *m_out = bm;
}

// Neighbour capacity of one of P sub-lists: the uniform-density count m
// within rlist split P ways, plus six standard deviations of a Poisson count
// and 4, rounded up to a whole block of four (at most one entry per atom).
// A user capacity c (per atom) gives ceil(c / P) per sub-list.
void set_capacity(EnsDev& e, int user_cap) {
  const double rho = e.N / (e.L * e.L * e.L);
  const double m = rho * 4.0 / 3.0 * M_PI * e.rlist * e.rlist * e.rlist;
  const int pv[4] = {1, 2, 4, 8};
  e.cap = 0;
  for (int k = 0; k < 4; ++k) {
    const double mp = m / pv[k];
    int cs = user_cap > 0 ? (user_cap + pv[k] - 1) / pv[k]
                          : (int)std::ceil(mp + 6.0 * std::sqrt(mp) + 4.0);
    cs = std::min(cs, e.N + 3);
    cs = std::max(4, (cs + 3) / 4 * 4);
    e.capsub[k] = cs;
    e.cap = std::max(e.cap, cs * pv[k]);
  }
}

}  // namespace re

namespace {

thread_local std::string g_create_error;

constexpr int kRing = 8;  // pinned staging slots for per-call budgets

struct Ensemble {
  int N, R;
  double L, rc;
  std::vector<double> temps;
  uint64_t seed;
};

}  // namespace

struct re_ctx {
  re_opts opt{};
  std::vector<EnsDev> ens;
  std::vector<RepDev> reps;
  int n_rep = 0, n_pairs = 0;
  int64_t n_atoms = 0, n_nbr = 0;
  int max_n = 0, max_r = 0, max_ncell = 0;
  LaunchCfg cfg{1, 256, 0, 1, 0};
  cudaStream_t stream = nullptr;
  int device = 0;
  StateDev s{};
  EnsDev* d_ens = nullptr;
  RepDev* d_rep = nullptr;
  int* d_work = nullptr;
  int* d_work2 = nullptr;           // split launch: work lists of the two classes
  int* d_work_id = nullptr;         // per-ensemble launches: replica r at position r
  int* d_work_ord = nullptr;        // budget mode, uneven budgets: longest job first
  int32_t* d_zero = nullptr;        // n_rep zero budgets (prologue launches)
  std::vector<LaunchCfg> ecfg;      // per-ensemble launches: the shape of each ensemble
  int list_mode = 0;                // the lists are laid out for: 0 the uniform shape, 1 the
                                    // per-ensemble shapes (threads per atom may differ)
  std::vector<cudaStream_t> cls_stream;  // per-ensemble launches: ensembles 1.. run here
  std::vector<cudaEvent_t> cls_ev;
  cudaStream_t side = nullptr;      // split launch: the wide class runs here
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  int32_t* d_budget = nullptr;      // n_rep, per call
  std::vector<int32_t> h_budget_last;  // what d_budget holds (when budget_cached)
  bool budget_cached = false;
  int32_t* d_budget_nx = nullptr;   // n_rep, filled with opt.nx
  int32_t* d_budget_run = nullptr;  // n_cycles * n_rep for re_run
  size_t budget_run_cap = 0;
  int32_t* h_ring = nullptr;        // pinned, kRing * n_rep
  // pinned: per-replica results read back in one synchronisation
  // (U, K, econs: doubles; status, partner: int32; accepted: bytes)
  unsigned char* h_out = nullptr;
  cudaEvent_t ring_ev[kRing] = {};
  int ring_pos = 0;
  int32_t* d_partner = nullptr;
  uint8_t* d_acc = nullptr;
  double* d_io = nullptr;           // 3 * n_atoms doubles, state import/export
  bool plain_refresh = true;        // plain path: lists/forces need a prologue
  int sort_every = 0;               // steps between spatial re-sorts (0: never)
  int64_t since_sort = 0;           // steps (largest budget) since the last re-sort
  bool tuning = false;              // autotune trials: no re-sorting
  std::vector<void*> allocs;
  std::string err;
  // free-running exchange: coordination words (2 E + 5 n_rep ints), published
  // (T, U) pairs, and the event log (grown on demand)
  int32_t* d_fr_words = nullptr;
  double* d_fr_slot = nullptr;
  int64_t* d_log_step = nullptr;
  double* d_log_T = nullptr;
  int32_t* d_log_partner = nullptr;
  int32_t* d_log_acc = nullptr;
  int log_rows = 0;
  int resident_clusters = -1;  // batched clusters resident at once (-1: not yet queried)
  LaunchCfg fcfg{};             // free-running launch when the tuned shape is not resident
  bool use_fcfg = false;        // set for the duration of such a launch (list layout 2)
  double wait_s = 1.0;         // limit of the free-running exchange's bounded waits
  int stall_rep = -1;          // fault injection for the next re_run_free (-1: none)
  int stall_from = 0;
  // re_run_record: the record rows (device, pinned host), the staged budgets,
  // and two copy streams (host -> device budgets, device -> host records)
  unsigned char* d_rec = nullptr;
  unsigned char* h_rec = nullptr;
  size_t rec_cap = 0;               // bytes of d_rec and h_rec
  int32_t* d_rec_bud = nullptr;
  int32_t* h_rec_bud = nullptr;
  size_t rec_bud_cap = 0;           // entries of d_rec_bud and h_rec_bud
  cudaStream_t rec_in = nullptr, rec_out = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  cudaGraphExec_t rec_graph = nullptr;  // cached graph of re_run_record
  int rec_graph_cycles = 0;
  bool rec_graph_steps = false;
  // cached graph of re_run
  cudaGraphExec_t graph = nullptr;
  int graph_cycles = 0;
  const int32_t* graph_budget = nullptr;
};

namespace {

int fail(re_ctx* c, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (c)
    c->err = buf;
  else
    g_create_error = buf;
  return code;
}

int cuda_fail(re_ctx* c, cudaError_t e, const char* what) {
  return fail(c, e == cudaErrorMemoryAllocation ? RE_ENOMEM : RE_ECUDA, "%s: %s", what,
              cudaGetErrorString(e));
}

#define RE_CUDA(c, call, what)                   \
  do {                                           \
    cudaError_t e_ = (call);                     \
    if (e_ != cudaSuccess) return cuda_fail(c, e_, what); \
  } while (0)

// The memory pools of re_lj_forces_device, one per device: stream-ordered, so
// calls from any threads and streams share one; it keeps at most 64 MB between
// calls (the driver's pools grow by 32 MB; keeping less than that, every call
// maps memory anew, 220 us) and returns the rest, and that too where another
// allocation of the library would fail for it (trim_scratch_pool).  The some 45
// allocations of a context took half a millisecond a call and more.
struct ScratchPools {
  std::mutex mu;
  cudaMemPool_t of[64] = {};
};
ScratchPools g_scratch_pools;

cudaError_t scratch_pool(cudaMemPool_t* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_scratch_pools.mu);
  cudaMemPool_t& pool = g_scratch_pools.of[dev];
  if (!pool) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    if ((e = cudaMemPoolCreate(&p, &props)) != cudaSuccess) return e;
    uint64_t keep = 64ull << 20;
    if ((e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
      cudaMemPoolDestroy(p);
      return e;
    }
    pool = p;
  }
  *out = pool;
  return cudaSuccess;
}

// Gives back what the current device's pool keeps; false when it has none.
bool trim_scratch_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  std::lock_guard<std::mutex> lock(g_scratch_pools.mu);
  const cudaMemPool_t pool = g_scratch_pools.of[dev];
  return pool && cudaMemPoolTrimTo(pool, 0) == cudaSuccess;
}

template <class T>
int dalloc(re_ctx* c, T** p, size_t n) {
  void* q = nullptr;
  size_t bytes = std::max<size_t>(n, 1) * sizeof(T);
  cudaError_t e = cudaMalloc(&q, bytes);
  if (e == cudaErrorMemoryAllocation && trim_scratch_pool()) {
    cudaGetLastError();
    e = cudaMalloc(&q, bytes);
  }
  if (e != cudaSuccess) return cuda_fail(c, e, "cudaMalloc");
  c->allocs.push_back(q);
  *p = static_cast<T*>(q);
  return RE_OK;
}

}  // namespace

namespace re {
void finish_ens(EnsDev& e) {
  StepConst& k = e.kc;
  k = StepConst{};
  k.lam32 = e.L * 0x1.0p-32;
  k.lam64 = e.L * 0x1.0p-64;
  k.inv_l = 1.0 / e.L;
  k.dtq = e.dt * 0x1.0p64 / e.L;
  k.hdt = 0.5 * e.dt;
  k.inv_hdt = 1.0 / k.hdt;
  const double rc6 = e.rc * e.rc * e.rc * e.rc * e.rc * e.rc;
  k.uc = e.shift ? 4.0 * (1.0 / (rc6 * rc6) - 1.0 / rc6) : 0.0;
  k.rc2 = e.rc * e.rc;
  const double rcu = e.rc / k.lam32;
  k.rc2u_lo = (float)(rcu * rcu * (1.0 - 2e-6));
  k.rc2u_hi = (float)(rcu * rcu * (1.0 + 2e-6));
  const double rcx = e.rc / (e.L * 0x1.0p-42);
  k.rc2x = rcx * rcx;
  // list radius rounded up, half skin rounded down: the list never misses a pair
  const double rlu = e.rlist * (1.0 + 1e-6) / k.lam32;
  k.rl2u = (float)(rlu * rlu);
  const double hu = 0.5 * e.skin * (1.0 - 1e-6) / k.lam32;
  k.half2u = (float)(hu * hu);
  set_pair_constants(k);
  k.nf = 3 * e.N - 3;
  k.c_th = e.tau > 0.0 ? std::exp(-e.dt / e.tau) : 1.0;
  const double omc = e.tau > 0.0 ? -std::expm1(-e.dt / e.tau) : 0.0;  // 1 - c, no cancellation
  k.cm1f = (float)(-omc);
  // Kbar = Nf T / 2: a = (1 - c) T / 2, b = 2 sqrt(c (1 - c) T / 2), g = sqrt(2 c / ((1 - c) T))
  k.af1 = 0.5 * omc;
  k.bf1 = 2.0 * std::sqrt(0.5 * k.c_th * omc);
  k.gf1 = omc > 0.0 ? std::sqrt(2.0 * k.c_th / omc) : 0.0;
  set_thermo_target(k, 1.0);
  set_potential_scale(k, 1.0);
}
}  // namespace re

namespace {

template <class T>
void dfree(re_ctx* c, T*& p) {
  if (!p) return;
  auto it = std::find(c->allocs.begin(), c->allocs.end(), static_cast<void*>(p));
  if (it != c->allocs.end()) c->allocs.erase(it);
  cudaFree(p);
  p = nullptr;
}

// The replicas one launch covers: every ensemble of the context (the uniform
// launch) or one ensemble (a class of a group's per-ensemble launches).
struct Scope {
  int max_n, max_ncell, n_rep, e0, e1;  // ensembles [e0, e1)
};

Scope all_scope(const re_ctx* c) {
  return Scope{c->max_n, c->max_ncell, c->n_rep, 0, (int)c->ens.size()};
}

Scope ens_scope(const re_ctx* c, int e) {
  const EnsDev& d = c->ens[e];
  return Scope{d.N, d.nc > 0 ? d.nc * d.nc * d.nc : 1, d.R, e, e + 1};
}

int threads_for(int max_n, int cluster, int atom_threads) {
  const int per = (max_n + cluster - 1) / cluster;
  return std::max(32, (atom_threads * per + 31) / 32 * 32);
}

int sm_count() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 148;
}

// The split launch of shape k (see LaunchCfg): for a one-ensemble batched
// context whose uniform launch leaves SMs idle, the hottest replicas get
// clusters of twice the CTAs (cluster sizes that pair up on the GPU like the
// uniform ones), as many as the idle SMs allow (fewer than all).  A wide CTA
// keeps the threads per atom -- a replica moves between the classes as the
// temperatures change, and its neighbour lists are laid out per thread of an
// atom -- and the CTA's thread count, so that one CTA still fills an SM (a
// smaller one could share its SM with a second and leave another SM idle);
// its extra threads hold no atom.
void set_wide(const re_ctx* c, LaunchCfg& k, bool on) {
  k.wide_n = k.wide_cluster = k.wide_threads = k.wide_atom_threads = 0;
  if (!on || c->ens.size() != 1 || c->opt.path != RE_PATH_BATCHED) return;
  const int sms = sm_count(), wc = k.cluster * 2;
  const int idle = sms - k.cluster * c->n_rep;
  if (wc > 8 || idle <= 0 || (c->max_n + wc - 1) / wc < 32) return;
  const int n = std::min(idle / k.cluster, c->n_rep - 1);
  if (n <= 0) return;
  k.wide_n = n;
  k.wide_cluster = wc;
  k.wide_atom_threads = k.atom_threads;
  k.wide_threads = std::max(k.threads, threads_for(c->max_n, wc, k.atom_threads));
}

// Per-ensemble launches of a group (re_opts.group_launch): in budget mode each
// ensemble of a context of several runs as its own launch, all launches
// concurrent on streams of their own, each in the launch shape that suits its
// replica size.
bool per_class(const re_ctx* c) {
  return c->ens.size() > 1 && c->opt.group_launch >= 0 && c->opt.path == RE_PATH_BATCHED;
}

// The launch shape of the wide class of a split launch.
LaunchCfg wide_cfg(const LaunchCfg& k) {
  LaunchCfg w = k;
  w.cluster = k.wide_cluster;
  w.threads = k.wide_threads;
  w.atom_threads = k.wide_atom_threads;
  w.wide_n = w.wide_cluster = w.wide_threads = w.wide_atom_threads = 0;
  return w;
}

// Default launch shape: enough CTAs per replica to cover the SMs in about one
// wave, then as many threads per atom as fit in one CTA: at most 4, or 8 on the
// FP64 path, whose pair loop deals its FP64 turns out evenly over an atom's
// lanes and wants warps to hide its other latencies (8 x 256 atoms: 41 against
// 45 thousand clocks a step, 20 x 864: 111 against 132).  (Clusters of 16 CTAs
// for a few FP64 replicas gain nothing: the FP64 units are shared by the two
// SMs of a pair.)
LaunchCfg default_cfg(const re_ctx* c, const Scope& sc) {
  LaunchCfg k{};
  const int sms = sm_count();
  int cl = c->opt.cluster;
  if (cl <= 0) {
    // at least enough CTAs that one thread per atom fits in 1024 threads, then
    // more until the replicas cover the SMs in about one wave
    cl = 1;
    while (cl < 8 && (sc.max_n + cl - 1) / cl > 1024) cl *= 2;
    while (cl < 8 && sc.n_rep * cl < (sms * 4) / 5 && (sc.max_n + 2 * cl - 1) / (2 * cl) >= 32)
      cl *= 2;
  }
  int p = c->opt.atom_threads;
  if (p <= 0) {
    p = c->opt.precision == RE_PREC_FP64 ? 8 : 4;
    while (p > 1 && threads_for(sc.max_n, cl, p) > 1024) p /= 2;
  }
  k.cluster = cl;
  k.atom_threads = p;
  k.threads = threads_for(sc.max_n, cl, p);
  k.cell_div = 0;
  k.lists_smem = c->opt.lists_smem > 0 ? 1 : 0;
  if (sc.e1 - sc.e0 == (int)c->ens.size()) set_wide(c, k, c->opt.wide_launch > 0);
  return k;
}
LaunchCfg default_cfg(const re_ctx* c) { return default_cfg(c, all_scope(c)); }

int upload_tables(re_ctx* c) {
  RE_CUDA(c, cudaMemcpyAsync(c->d_ens, c->ens.data(), sizeof(EnsDev) * c->ens.size(),
                             cudaMemcpyHostToDevice, c->stream), "upload ensembles");
  RE_CUDA(c, cudaMemcpyAsync(c->d_rep, c->reps.data(), sizeof(RepDev) * c->reps.size(),
                             cudaMemcpyHostToDevice, c->stream), "upload replicas");
  return RE_OK;
}

// Whether a screened list build (see re_batched.cuh) in shape k finds room for less
// than half of the notes that a lane can make in the list array: four threads an
// atom, sparse systems, capacities given by the caller.
bool notes_short(const EnsDev& e, const LaunchCfg& k) {
  const int P = k.atom_threads, idx = P == 1 ? 0 : (P == 2 ? 1 : 2);
  if (P > 4 || e.N <= re::kDirectBuild) return false;
  const int quads = (e.N + 127) / 128;  // of rows; a lane makes 4 / P notes of each
  return 2 * re::list_notes(e.cap, e.capsub[idx], P) < std::min(e.capsub[idx] / 4, quads * (4 / P));
}

// An array of their own for the notes, while a launch shape in use is short of room
// for them: 1372 atoms on eight CTAs of four threads an atom, skin 0.1, 15.1 us a
// step instead of 16.4.  Such shapes are those of few replicas; the others do
// without it.  Failing to get it changes the time only.  Given back only where no
// cached graph can hold it (give_back: the graphs are dropped there).
void fit_notes(re_ctx* c, bool give_back) {
  bool need = false;
  for (size_t e = 0; e < c->ens.size() && c->opt.path == RE_PATH_BATCHED; ++e) {
    need |= notes_short(c->ens[e], c->cfg) || (c->use_fcfg && notes_short(c->ens[e], c->fcfg));
    if (per_class(c)) need |= notes_short(c->ens[e], c->ecfg[e]);
  }
  if (need == (c->s.raw != nullptr)) return;
  const std::string err = c->err;
  if (!need) {
    if (give_back) dfree(c, c->s.raw);
  } else if (dalloc(c, &c->s.raw, (size_t)c->n_nbr) != RE_OK) {
    cudaGetLastError();
    c->err = err;
  }
}

// Allocate device memory for the current ens/reps tables.
int allocate(re_ctx* c) {
  const size_t A = (size_t)c->n_atoms, R = (size_t)c->n_rep, E = c->ens.size();
  StateDev& s = c->s;
  int rc = RE_OK;
  if ((rc = dalloc(c, &s.qx, A)) || (rc = dalloc(c, &s.qy, A)) || (rc = dalloc(c, &s.qz, A)) ||
      (rc = dalloc(c, &s.vx, A)) || (rc = dalloc(c, &s.vy, A)) || (rc = dalloc(c, &s.vz, A)) ||
      (rc = dalloc(c, &s.fx, A)) || (rc = dalloc(c, &s.fy, A)) || (rc = dalloc(c, &s.fz, A)) ||
      (rc = dalloc(c, &s.rx, A)) || (rc = dalloc(c, &s.ry, A)) || (rc = dalloc(c, &s.rz, A)) ||
      (rc = dalloc(c, &s.ncnt, 8 * A)) || (rc = dalloc(c, &s.nbr, (size_t)c->n_nbr)) ||
      (rc = dalloc(c, &s.T, R)) || (rc = dalloc(c, &s.U, 4 * R)) || (rc = dalloc(c, &s.vscale, R)) ||
      (rc = dalloc(c, &s.lam, R)) || (rc = dalloc(c, &s.fscale, R)) ||
      (rc = dalloc(c, &s.step, R)) || (rc = dalloc(c, &s.nreb, R)) ||
      (rc = dalloc(c, &s.valid, R)) ||
      (rc = dalloc(c, &s.attempt, E)) || (rc = dalloc(c, &s.pair_att, (size_t)c->n_pairs)) ||
      (rc = dalloc(c, &s.pair_acc, (size_t)c->n_pairs)) ||
      (rc = dalloc(c, &s.red, R * 1024)) || (rc = dalloc(c, &s.dmax, R)) ||
      (rc = dalloc(c, &s.perm, A)) || (rc = dalloc(c, &s.order, A)) ||
      (rc = dalloc(c, &s.stop, E)) ||
      (rc = dalloc(c, &s.sbuf, 7 * A)) ||
      (rc = dalloc(c, &c->d_ens, E)) || (rc = dalloc(c, &c->d_rep, R)) ||
      (rc = dalloc(c, &c->d_work, R)) || (rc = dalloc(c, &c->d_work2, R)) ||
      (rc = dalloc(c, &c->d_work_id, R)) || (rc = dalloc(c, &c->d_zero, R)) ||
      (rc = dalloc(c, &c->d_work_ord, R)) ||
      (rc = dalloc(c, &c->d_budget, R)) ||
      (rc = dalloc(c, &c->d_budget_nx, R)) || (rc = dalloc(c, &c->d_partner, 2 * R)) ||
      (rc = dalloc(c, &c->d_io, 3 * A)))
    return rc;
  // what is read back together lies together, laid out like h_out: the energies
  // and the status words, the partners and the decisions
  fit_notes(c, false);
  s.K = s.U + R;
  s.econs = s.U + 2 * R;
  s.status = reinterpret_cast<int32_t*>(s.U + 3 * R);
  c->d_acc = reinterpret_cast<uint8_t*>(c->d_partner + R);
  RE_CUDA(c, cudaMemsetAsync(s.nbr, 0, sizeof(uint16_t) * (size_t)c->n_nbr, c->stream), "memset");
  RE_CUDA(c, cudaMemsetAsync(c->d_zero, 0, sizeof(int32_t) * R, c->stream), "memset");
  RE_CUDA(c, cudaMemsetAsync(s.ncnt, 0, sizeof(int32_t) * 8 * A, c->stream), "memset");
  RE_CUDA(c, cudaMemsetAsync(s.attempt, 0, sizeof(int64_t) * E, c->stream), "memset");
  RE_CUDA(c, cudaMemsetAsync(s.pair_att, 0, sizeof(int64_t) * std::max(1, c->n_pairs), c->stream), "memset");
  RE_CUDA(c, cudaMemsetAsync(s.pair_acc, 0, sizeof(int64_t) * std::max(1, c->n_pairs), c->stream), "memset");
  RE_CUDA(c, cudaMemsetAsync(s.dmax, 0, sizeof(uint32_t) * R, c->stream), "memset");
  {
    // potential scales 1 (plain LJ) until re_create_h sets them; no pending force factor
    const std::vector<double> ones(R, 1.0);
    RE_CUDA(c, cudaMemcpy(s.lam, ones.data(), 8 * R, cudaMemcpyHostToDevice), "init lam");
    RE_CUDA(c, cudaMemcpy(s.fscale, ones.data(), 8 * R, cudaMemcpyHostToDevice), "init fscale");
  }
  RE_CUDA(c, cudaMallocHost(&c->h_ring, sizeof(int32_t) * R * kRing), "cudaMallocHost");
  RE_CUDA(c, cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking), "side stream");
  RE_CUDA(c, cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming), "event");
  RE_CUDA(c, cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming), "event");
  RE_CUDA(c, cudaMallocHost(&c->h_out, (3 * 8 + 2 * 4 + 1) * R), "cudaMallocHost");
  for (int k = 0; k < kRing; ++k)
    RE_CUDA(c, cudaEventCreateWithFlags(&c->ring_ev[k], cudaEventDisableTiming), "event");
  // work list: replicas by decreasing size (largest clusters start first)
  std::vector<int> work(R);
  for (size_t r = 0; r < R; ++r) work[r] = (int)r;
  std::stable_sort(work.begin(), work.end(), [&](int a, int b) {
    return c->ens[c->reps[a].ens].N > c->ens[c->reps[b].ens].N;
  });
  RE_CUDA(c, cudaMemcpyAsync(c->d_work, work.data(), sizeof(int) * R, cudaMemcpyHostToDevice,
                             c->stream), "upload work");
  for (size_t r = 0; r < R; ++r) work[r] = (int)r;
  RE_CUDA(c, cudaMemcpyAsync(c->d_work_id, work.data(), sizeof(int) * R, cudaMemcpyHostToDevice,
                             c->stream), "upload work");
  for (size_t e = 1; e < E; ++e) {
    cudaStream_t st = nullptr;
    cudaEvent_t ev = nullptr;
    RE_CUDA(c, cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking), "class stream");
    c->cls_stream.push_back(st);
    RE_CUDA(c, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming), "event");
    c->cls_ev.push_back(ev);
  }
  std::vector<int32_t> nx(R, c->opt.nx);
  RE_CUDA(c, cudaMemcpyAsync(c->d_budget_nx, nx.data(), sizeof(int32_t) * R,
                             cudaMemcpyHostToDevice, c->stream), "upload nx");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "sync");
  int rc2 = upload_tables(c);
  if (rc2) return rc2;
  // every context starts with its atoms in original order
  cudaError_t e = re::launch_identity_perm(c->s, c->d_ens, c->d_rep, c->n_rep, c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "identity permutation");
  return RE_OK;
}

// Fill per-ensemble cells for the current cfg.cell_div; returns max ncell.
void apply_cells(re_ctx* c, int want_m) {
  c->max_ncell = 1;
  for (auto& e : c->ens) {
    choose_cells(e.L, e.rlist, e.N, want_m, &e.nc, &e.m);
    c->max_ncell = std::max(c->max_ncell, e.nc > 0 ? e.nc * e.nc * e.nc : 1);
  }
}

int max_smem_optin() {
  int dev = 0, maxsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return maxsm > 0 ? maxsm : 232448;
}

// Shared-memory list entries per CTA for launch shape k: the largest CTA's
// P sub-lists over all ensembles, or 0 when they would not fit (the kernel then
// reads the lists from global memory).
size_t list_elems_for(const re_ctx* c, const LaunchCfg& k, const Scope& sc) {
  if (!k.lists_smem) return 0;
  const int pidx = k.atom_threads == 1 ? 0 : (k.atom_threads == 2 ? 1 : (k.atom_threads == 4 ? 2 : 3));
  size_t elems = 0;
  for (int i = sc.e0; i < sc.e1; ++i) {
    const EnsDev& e = c->ens[i];
    const size_t per = (size_t)(e.N + k.cluster - 1) / k.cluster;
    elems = std::max(elems, per * k.atom_threads * (size_t)e.capsub[pidx]);
  }
  const size_t smem = re::batched_smem_bytes(sc.max_n, k.threads,
                                             c->opt.precision == RE_PREC_FP64, elems);
  return smem + re::kBatchedStaticSmem <= (size_t)max_smem_optin() ? elems : 0;
}
size_t list_elems_for(const re_ctx* c, const LaunchCfg& k) {
  return list_elems_for(c, k, all_scope(c));
}

int check_cfg(re_ctx* c, const LaunchCfg& k, const Scope& sc) {
  if (k.wide_n > 0) {
    if (k.wide_n >= c->n_rep || c->ens.size() != 1 || k.wide_cluster < 2 || k.wide_cluster > 8 ||
        k.wide_atom_threads != k.atom_threads)
      return fail(c, RE_EINVAL, "split launch needs one ensemble, fewer wide replicas than "
                  "replicas, 2..8 CTAs per wide replica and the same threads per atom");
    const int rc = check_cfg(c, wide_cfg(k), sc);
    if (rc) return rc;
  }
  if (k.cluster < 1 || k.cluster > 8 || (k.cluster != 3 && (k.cluster & (k.cluster - 1))))
    return fail(c, RE_EINVAL, "cluster must be 1, 2, 3, 4 or 8 (got %d)", k.cluster);
  if (k.atom_threads != 1 && k.atom_threads != 2 && k.atom_threads != 4 && k.atom_threads != 8)
    return fail(c, RE_EINVAL, "atom_threads must be 1, 2, 4 or 8 (got %d)", k.atom_threads);
  if (k.threads < 32 || k.threads > 1024 || k.threads % 32 ||
      k.threads < k.atom_threads * ((sc.max_n + k.cluster - 1) / k.cluster))
    return fail(c, RE_EINVAL, "%d atoms per CTA x %d threads per atom exceed 1024 threads; "
                "use more CTAs per replica", (sc.max_n + k.cluster - 1) / k.cluster, k.atom_threads);
  if (sc.max_n > re::kMaxBatchedAtoms)
    return fail(c, RE_EINVAL, "replica of %d atoms: the batched path takes at most %d", sc.max_n,
                re::kMaxBatchedAtoms);
  const size_t smem = re::batched_admission_bytes(sc.max_n, sc.max_ncell, k.threads,
                                                  c->opt.precision == RE_PREC_FP64) +
                      re::kBatchedStaticSmem;
  const int maxsm = max_smem_optin();
  if (smem > (size_t)maxsm)
    return fail(c, RE_EINVAL, "replica of %d atoms needs %zu bytes of shared memory (max %d)",
                sc.max_n, smem, maxsm);
  return RE_OK;
}
int check_cfg(re_ctx* c, const LaunchCfg& k) { return check_cfg(c, k, all_scope(c)); }

// Launch shapes of the per-ensemble classes: each ensemble's default shape as
// if it were a context of its own.
void default_class_cfgs(re_ctx* c) {
  c->ecfg.assign(c->ens.size(), LaunchCfg{});
  for (size_t e = 0; e < c->ens.size(); ++e) {
    c->ecfg[e] = default_cfg(c, ens_scope(c, (int)e));
    c->ecfg[e].cell_div = c->opt.cell_div;
  }
}

int check_class_cfgs(re_ctx* c) {
  for (size_t e = 0; e < c->ens.size(); ++e) {
    const int rc = check_cfg(c, c->ecfg[e], ens_scope(c, (int)e));
    if (rc) return rc;
  }
  return RE_OK;
}

// Cells of every ensemble from its class's cell division.
void apply_cells_each(re_ctx* c) {
  c->max_ncell = 1;
  for (size_t i = 0; i < c->ens.size(); ++i) {
    EnsDev& e = c->ens[i];
    choose_cells(e.L, e.rlist, e.N, c->ecfg[i].cell_div, &e.nc, &e.m);
    c->max_ncell = std::max(c->max_ncell, e.nc > 0 ? e.nc * e.nc * e.nc : 1);
  }
}

// The launch of class e of a group's per-ensemble launches on stream st;
// with uneven budgets its replicas longest job first.
int launch_class(re_ctx* c, int e, const int32_t* d_budget, cudaStream_t st, bool uneven = false) {
  const Scope sc = ens_scope(c, e);
  const LaunchCfg& k = c->ecfg[e];
  const int r0 = c->ens[e].rep_off;
  const int* work = c->d_work_id + r0;
  if (uneven && c->ens[e].R <= 4096) {
    RE_CUDA(c, re::launch_order_work(d_budget, c->d_rep, c->d_ens, r0, c->ens[e].R,
                                     c->d_work_ord, st), "order work");
    work = c->d_work_ord + r0;
  }
  cudaError_t err = re::launch_batched(c->s, c->d_ens, c->d_rep, work, c->ens[e].R, d_budget,
                                       c->opt.precision == RE_PREC_FP64, k, sc.max_n,
                                       list_elems_for(c, k, sc), 0, st, nullptr, uneven);
  if (err != cudaSuccess) return cuda_fail(c, err, "batched MD launch (ensemble class)");
  return RE_OK;
}

// Lists, forces, U and K of every replica in the layout of `mode` (see
// re_ctx::list_mode) when they are in the other one: a prologue launch in the
// new shape(s) with zero budgets.  The replicas' list rebuild counters are
// kept (this rebuild is a change of layout, not the list rule of the
// Example section).
// The lists' layout follows the launch shape's threads per atom.  Layouts:
// 0 the uniform shape (cfg), 1 the per-ensemble shapes (ecfg), 2 the
// free-running fallback shape (fcfg).  A switch rebuilds every list (and the
// forces) at the current positions; rebuild counters are kept.
int relayout_lists(re_ctx* c, int mode) {
  if (c->list_mode == mode) return RE_OK;
  c->list_mode = mode;
  const size_t R = (size_t)c->n_rep;
  RE_CUDA(c, cudaMemcpyAsync(c->d_io, c->s.nreb, 8 * R, cudaMemcpyDeviceToDevice, c->stream),
          "save counters");
  RE_CUDA(c, cudaMemsetAsync(c->s.valid, 0, 4 * R, c->stream), "invalidate lists");
  const bool fp64 = c->opt.precision == RE_PREC_FP64;
  if (mode == 1) {
    for (size_t e = 0; e < c->ens.size(); ++e) {
      const int rc = launch_class(c, (int)e, c->d_zero, c->stream);
      if (rc) return rc;
    }
  } else if (mode == 2) {
    cudaError_t e = re::launch_batched(c->s, c->d_ens, c->d_rep, c->d_work, c->n_rep, c->d_zero,
                                       fp64, c->fcfg, c->max_n, 0, 0, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "batched MD launch");
  } else {
    cudaError_t e = re::launch_batched(c->s, c->d_ens, c->d_rep, c->d_work, c->n_rep, c->d_zero,
                                       fp64, c->cfg, c->max_n, 0, 0, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "batched MD launch");
  }
  RE_CUDA(c, cudaMemcpyAsync(c->s.nreb, c->d_io, 8 * R, cudaMemcpyDeviceToDevice, c->stream),
          "restore counters");
  return RE_OK;
}

// uneven: the budgets differ between replicas (budget mode); the work is then
// ordered longest job first on the device.
int launch_advance(re_ctx* c, const int32_t* d_budget, const int32_t* h_budget,
                   int max_budget = -1, int async_nx = 0, const re::FreeDev* fr = nullptr,
                   bool uneven = false) {
  if (c->opt.path == RE_PATH_BATCHED) {
    // renumber atoms in space order every sort_every steps (mixed path): warps
    // then hold neighbouring atoms, whose lists and gathers overlap
    if (c->sort_every > 0 && !c->tuning && c->since_sort >= c->sort_every) {
      cudaError_t e = re::launch_spatial_sort(c->s, c->d_ens, c->d_rep, c->n_rep, c->max_n,
                                              c->max_ncell, c->n_atoms, c->stream);
      if (e != cudaSuccess) return cuda_fail(c, e, "spatial sort");
      c->since_sort = 0;
    }
    c->since_sort += max_budget >= 0 ? max_budget : c->opt.nx;
    if (async_nx > 0) {
      cudaError_t e = cudaMemsetAsync(c->s.stop, 0, sizeof(int32_t) * c->ens.size(), c->stream);
      if (e != cudaSuccess) return cuda_fail(c, e, "clear stop flags");
    }
    // the free-running modes read the lists from global memory
    const bool budgets = async_nx <= 0 && !(fr && fr->nx > 0);
    const bool fp64 = c->opt.precision == RE_PREC_FP64;
    {
      // a group switching between its per-ensemble launches and the uniform
      // one (free-running modes) rebuilds its lists in the other layout first
      const bool fshape = !budgets && fr && fr->nx > 0 && c->use_fcfg;
      const int rc = relayout_lists(c, budgets && per_class(c) ? 1 : (fshape ? 2 : 0));
      if (rc) return rc;
    }
    if (budgets && per_class(c)) {
      // one launch per ensemble, concurrent: class 0 on the context's stream,
      // the others on their own streams, forked from and joined back to it
      const int E = (int)c->ens.size();
      RE_CUDA(c, cudaEventRecord(c->ev_fork, c->stream), "fork");
      for (int e = 1; e < E; ++e) {
        RE_CUDA(c, cudaStreamWaitEvent(c->cls_stream[e - 1], c->ev_fork, 0), "fork");
        const int rc = launch_class(c, e, d_budget, c->cls_stream[e - 1], uneven);
        if (rc) return rc;
        RE_CUDA(c, cudaEventRecord(c->cls_ev[e - 1], c->cls_stream[e - 1]), "join");
      }
      const int rc = launch_class(c, 0, d_budget, c->stream, uneven);
      if (rc) return rc;
      for (int e = 1; e < E; ++e)
        RE_CUDA(c, cudaStreamWaitEvent(c->stream, c->cls_ev[e - 1], 0), "join");
      return RE_OK;
    }
    if (budgets && c->cfg.wide_n > 0) {
      // split launch: rank by temperature on the device, then the two classes
      // run concurrently (the wide one on the side stream, joined back)
      const int nw = c->cfg.wide_n, nn = c->n_rep - nw;
      const LaunchCfg wk = wide_cfg(c->cfg);
      RE_CUDA(c, re::launch_split_work(c->s.T, c->n_rep, nw, c->d_work2, c->stream), "split work");
      RE_CUDA(c, cudaEventRecord(c->ev_fork, c->stream), "fork");
      RE_CUDA(c, cudaStreamWaitEvent(c->side, c->ev_fork, 0), "fork");
      cudaError_t e = re::launch_batched(c->s, c->d_ens, c->d_rep, c->d_work2 + nn, nw, d_budget,
                                         fp64, wk, c->max_n, list_elems_for(c, wk),
                                         0, c->side, nullptr, uneven);
      if (e != cudaSuccess) return cuda_fail(c, e, "batched MD launch (wide class)");
      e = re::launch_batched(c->s, c->d_ens, c->d_rep, c->d_work2, nn, d_budget, fp64, c->cfg,
                             c->max_n, list_elems_for(c, c->cfg), 0, c->stream,
                             nullptr, uneven);
      if (e != cudaSuccess) return cuda_fail(c, e, "batched MD launch");
      RE_CUDA(c, cudaEventRecord(c->ev_join, c->side), "join");
      RE_CUDA(c, cudaStreamWaitEvent(c->stream, c->ev_join, 0), "join");
      return RE_OK;
    }
    // uneven budgets: longest job first (otherwise the fixed order, largest
    // replicas first)
    const bool order = budgets && uneven && c->n_rep <= 4096;
    if (order)
      RE_CUDA(c, re::launch_order_work(d_budget, c->d_rep, c->d_ens, 0, c->n_rep, c->d_work_ord,
                                       c->stream), "order work");
    const LaunchCfg& k = (!budgets && fr && fr->nx > 0 && c->use_fcfg) ? c->fcfg : c->cfg;
    cudaError_t e = re::launch_batched(c->s, c->d_ens, c->d_rep, order ? c->d_work_ord : c->d_work,
                                       c->n_rep, d_budget, fp64, k, c->max_n,
                                       budgets ? list_elems_for(c, k) : 0, async_nx,
                                       c->stream, fr, budgets && uneven);
    if (e != cudaSuccess) return cuda_fail(c, e, "batched MD launch");
    return RE_OK;
  }
  // plain path: one replica after another, a launch sequence per step
  for (int r = 0; r < c->n_rep; ++r) {
    const int steps = h_budget ? h_budget[r] : c->opt.nx;
    if (steps <= 0 && !c->plain_refresh) continue;
    const RepDev& rd = c->reps[r];
    cudaError_t e = re::launch_plain_advance(c->s, c->ens[rd.ens], rd, r, c->d_ens, c->d_rep,
                                             steps, c->max_ncell, c->stream,
                                             c->plain_refresh ? 1 : 0);
    if (e != cudaSuccess) return cuda_fail(c, e, "plain MD launch");
  }
  c->plain_refresh = false;
  return RE_OK;
}

int refresh(re_ctx* c) {
  if (c->opt.path == RE_PATH_BATCHED) {
    // budget 0 with invalid lists: the kernel's prologue builds lists, forces, U, K
    RE_CUDA(c, cudaMemsetAsync(c->d_budget, 0, sizeof(int32_t) * c->n_rep, c->stream), "memset");
    c->budget_cached = false;
    return launch_advance(c, c->d_budget, nullptr, 0);
  }
  c->plain_refresh = true;
  std::vector<int32_t> zero(c->n_rep, 0);
  return launch_advance(c, nullptr, zero.data());
}

// Pinned read-back areas of h_out.
double* out_U(re_ctx* c) { return reinterpret_cast<double*>(c->h_out); }
double* out_K(re_ctx* c) { return out_U(c) + c->n_rep; }
double* out_econs(re_ctx* c) { return out_U(c) + 2 * (size_t)c->n_rep; }
int32_t* out_status(re_ctx* c) { return reinterpret_cast<int32_t*>(out_U(c) + 3 * (size_t)c->n_rep); }
int32_t* out_partner(re_ctx* c) { return out_status(c) + c->n_rep; }
uint8_t* out_acc(re_ctx* c) { return reinterpret_cast<uint8_t*>(out_partner(c) + c->n_rep); }

// RE_ETIMEOUT with message fmt(r).  A failed free-running launch leaves every
// replica at a step boundary with a consistent state (a pair either swapped
// on both sides or not at all), so the timeout marks are cleared on the
// device once reported: the context goes on with the next call.
int timeout_fail(re_ctx* c, const int32_t* st, const char* fmt, int r) {
  const int code = fail(c, RE_ETIMEOUT, fmt, r);
  std::vector<int32_t> cleared(st, st + c->n_rep);
  for (auto& w : cleared) w &= ~(int32_t)(re::kStTimeout | re::kStAborted);
  cudaError_t e = cudaMemcpyAsync(c->s.status, cleared.data(), sizeof(int32_t) * c->n_rep,
                                  cudaMemcpyHostToDevice, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "clear timeout marks");
  return code;
}

// The first error recorded in the replicas' status words.
int status_eval(re_ctx* c, const int32_t* st) {
  for (int r = 0; r < c->n_rep; ++r) {
    if (st[r] & re::kStOverflow)
      return fail(c, RE_EOVERFLOW, "replica %d: neighbour list capacity exceeded (%d per atom; "
                  "raise nbr_capacity)", r, c->ens[c->reps[r].ens].cap);
    if (st[r] & (re::kStNumeric | re::kStRngCap))
      return fail(c, RE_ENUMERIC, "replica %d: non-finite energy or thermostat draw", r);
  }
  // a timed-out wait is reported after the errors that may have caused it;
  // the replica whose own wait ran out is named before those it stopped
  for (int r = 0; r < c->n_rep; ++r)
    if (st[r] & re::kStTimeout)
      return timeout_fail(c, st, "replica %d: free-running exchange: its bounded wait ran out "
                          "(or it stopped answering)", r);
  for (int r = 0; r < c->n_rep; ++r)
    if (st[r] & re::kStAborted)
      return timeout_fail(c, st, "replica %d: free-running exchange stopped early by another "
                          "replica's failed wait", r);
  return RE_OK;
}

int status_check(re_ctx* c) {
  RE_CUDA(c, cudaMemcpyAsync(out_status(c), c->s.status, sizeof(int32_t) * c->n_rep,
                             cudaMemcpyDeviceToHost, c->stream), "read status");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  return status_eval(c, out_status(c));
}

int build_context(re_ctx* c, const std::vector<Ensemble>& es, const std::vector<re_ctx*>* src) {
  int rep_off = 0, pair_off = 0;
  int64_t atom_off = 0, nbr_off = 0;
  for (size_t k = 0; k < es.size(); ++k) {
    const Ensemble& s = es[k];
    EnsDev e{};
    e.N = s.N;
    e.R = s.R;
    e.rep_off = rep_off;
    e.pair_off = pair_off;
    e.L = s.L;
    e.rc = s.rc;
    e.skin = c->opt.skin;
    e.rlist = s.rc + c->opt.skin;
    e.dt = c->opt.dt;
    e.tau = c->opt.tau_T;
    e.shift = c->opt.shift_energy ? 1 : 0;
    e.parity_mode = c->opt.pair_parity;
    e.xdist = std::max(1, c->opt.exch_distance);
    e.seed = s.seed;
    set_capacity(e, c->opt.nbr_capacity);
    finish_ens(e);
    if (src) {
      e.cap = (*src)[k]->ens[0].cap;
      for (int q = 0; q < 4; ++q) e.capsub[q] = (*src)[k]->ens[0].capsub[q];
    }
    c->ens.push_back(e);
    for (int r = 0; r < s.R; ++r) {
      RepDev rd{};
      rd.ens = (int)k;
      rd.id = r;
      rd.stream = c->opt.id_offset + r;
      rd.atom_off = (int)atom_off;
      rd.nbr_off = nbr_off;
      c->reps.push_back(rd);
      atom_off += s.N;
      nbr_off += (int64_t)e.cap * s.N;
    }
    rep_off += s.R;
    pair_off += std::max(0, s.R - 1);
    c->max_n = std::max(c->max_n, s.N);
    c->max_r = std::max(c->max_r, s.R);
  }
  if (atom_off > INT32_MAX) return fail(c, RE_EINVAL, "too many atoms in one context");
  c->n_rep = rep_off;
  c->n_pairs = pair_off;
  c->sort_every = (c->opt.path == RE_PATH_BATCHED && c->opt.precision == RE_PREC_MIXED &&
                   c->opt.sort_interval >= 0)
                      ? (c->opt.sort_interval > 0 ? c->opt.sort_interval : 200)
                      : 0;
  c->n_atoms = atom_off;
  c->n_nbr = nbr_off;
  c->s.vfix = (c->opt.path == RE_PATH_BATCHED && c->opt.precision == RE_PREC_MIXED) ? 1 : 0;
  apply_cells(c, c->opt.cell_div);
  c->cfg = default_cfg(c);
  c->cfg.cell_div = c->opt.cell_div;
  default_class_cfgs(c);
  if (c->opt.path == RE_PATH_BATCHED) {
    int rc = check_cfg(c, c->cfg);
    if (rc == RE_OK && per_class(c)) rc = check_class_cfgs(c);
    if (rc) return rc;
  }
  return allocate(c);
}

}  // namespace

// =========================================================================
extern "C" {

void re_default_opts(re_opts* o) {
  if (!o) return;
  o->dt = 0.005;
  o->skin = 0.5;
  o->tau_T = 0.5;
  o->shift_energy = 1;
  o->precision = RE_PREC_MIXED;
  o->path = RE_PATH_BATCHED;
  o->pair_parity = 0;
  o->nx = 10;
  o->nbr_capacity = 0;
  o->cell_div = 0;
  o->cluster = 0;
  o->atom_threads = 0;
  o->sort_interval = 0;
  o->exch_distance = 1;
  o->id_offset = 0;
  o->lists_smem = 0;
  o->wide_launch = 0;
  o->group_launch = 0;
}

int re_create(int N, double L, double rc, int n_rep, const double* temps, uint64_t seed,
              const re_opts* opt, re_ctx** out) {
  return re_create_h(N, L, rc, n_rep, temps, nullptr, seed, opt, out);
}

int re_create_h(int N, double L, double rc, int n_rep, const double* temps, const double* lams,
                uint64_t seed, const re_opts* opt, re_ctx** out) {
  g_create_error.clear();
  if (!out) return fail(nullptr, RE_EINVAL, "out is NULL");
  *out = nullptr;
  re_opts o;
  re_default_opts(&o);
  if (opt) o = *opt;
  if (n_rep < 1 || n_rep > 4096) return fail(nullptr, RE_EINVAL, "n_rep must be in [1, 4096]");
  if (!temps) return fail(nullptr, RE_EINVAL, "temps is NULL");
  int k = 1;
  while (4 * k * k * k < N) ++k;
  if (N < 4 || 4 * k * k * k != N) return fail(nullptr, RE_EINVAL, "N must be 4 k^3 (got %d)", N);
  if (N > 65535) return fail(nullptr, RE_EINVAL, "N must be <= 65535 (got %d)", N);
  if (!(L > 0) || !(rc > 0) || !(o.skin > 0) || !(o.dt > 0))
    return fail(nullptr, RE_EINVAL, "L, rc, skin and dt must be positive");
  if (rc + o.skin >= 0.5 * L)
    return fail(nullptr, RE_EINVAL, "list radius rc + skin = %g must be below L/2 = %g", rc + o.skin,
                0.5 * L);
  if (o.precision != RE_PREC_FP64 && o.precision != RE_PREC_MIXED)
    return fail(nullptr, RE_EINVAL, "unknown precision %d", o.precision);
  if (o.path != RE_PATH_BATCHED && o.path != RE_PATH_PLAIN)
    return fail(nullptr, RE_EINVAL, "unknown path %d", o.path);
  if (o.path == RE_PATH_PLAIN) o.precision = RE_PREC_FP64;
  if (o.nx < 0) return fail(nullptr, RE_EINVAL, "nx must be >= 0");
  if (o.exch_distance < 0) return fail(nullptr, RE_EINVAL, "exch_distance must be >= 1");
  if (o.id_offset < 0) return fail(nullptr, RE_EINVAL, "id_offset must be >= 0");
  for (int i = 0; i < n_rep; ++i) {
    if (!(temps[i] > 0) || !std::isfinite(temps[i]))
      return fail(nullptr, RE_EINVAL, "temperatures must be positive");
    if (lams && !(lams[i] > 0 && std::isfinite(lams[i])))
      return fail(nullptr, RE_EINVAL, "potential scales must be positive");
    const double ki = temps[i] / (lams ? lams[i] : 1.0);
    for (int j = 0; j < i; ++j)
      if (ki == temps[j] / (lams ? lams[j] : 1.0))
        return fail(nullptr, RE_EINVAL, lams ? "ladder keys T/lam must be distinct"
                                             : "temperatures must be distinct");
  }
  re_ctx* c = new re_ctx();
  c->opt = o;
  cudaGetDevice(&c->device);
  Ensemble e{N, n_rep, L, rc, std::vector<double>(temps, temps + n_rep), seed};
  int rcode = build_context(c, {e}, nullptr);
  if (rcode == RE_OK) {
    cudaError_t ce = cudaMemcpyAsync(c->s.T, temps, sizeof(double) * n_rep,
                                     cudaMemcpyHostToDevice, c->stream);
    if (ce == cudaSuccess && lams)
      ce = cudaMemcpyAsync(c->s.lam, lams, sizeof(double) * n_rep, cudaMemcpyHostToDevice,
                           c->stream);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(c->stream);
    if (ce != cudaSuccess) rcode = cuda_fail(c, ce, "upload temps");
  }
  if (rcode == RE_OK) {
    cudaError_t ce = re::launch_init_lattice(c->s, c->d_ens, c->d_rep, c->n_rep, 256, c->stream);
    if (ce != cudaSuccess) rcode = cuda_fail(c, ce, "lattice init");
  }
  if (rcode == RE_OK) rcode = refresh(c);
  if (rcode == RE_OK) rcode = status_check(c);
  if (rcode != RE_OK) {
    g_create_error = c->err;
    re_destroy(c);
    return rcode;
  }
  *out = c;
  return RE_OK;
}

int re_group(re_ctx* const* ctxs, int n, re_ctx** out) {
  g_create_error.clear();
  if (!ctxs || n < 1 || !out) return fail(nullptr, RE_EINVAL, "bad arguments");
  *out = nullptr;
  std::vector<Ensemble> es;
  std::vector<re_ctx*> src;
  for (int i = 0; i < n; ++i) {
    re_ctx* s = ctxs[i];
    if (!s) return fail(nullptr, RE_EINVAL, "member %d is NULL", i);
    if (s->ens.size() != 1) return fail(nullptr, RE_EINVAL, "members must be single ensembles");
    if (s->opt.precision != ctxs[0]->opt.precision || s->opt.path != ctxs[0]->opt.path)
      return fail(nullptr, RE_EINVAL, "members must share precision and path");
    const EnsDev& e = s->ens[0];
    es.push_back(Ensemble{e.N, e.R, e.L, e.rc, {}, e.seed});
    src.push_back(s);
    re_sync(s);
  }
  re_ctx* c = new re_ctx();
  c->opt = ctxs[0]->opt;
  // an explicit launch shape is kept only when every member asks for the same one
  for (int i = 1; i < n; ++i) {
    if (ctxs[i]->opt.cluster != c->opt.cluster) c->opt.cluster = 0;
    if (ctxs[i]->opt.atom_threads != c->opt.atom_threads) c->opt.atom_threads = 0;
    if (ctxs[i]->opt.cell_div != c->opt.cell_div) c->opt.cell_div = 0;
  }
  cudaGetDevice(&c->device);
  int rcode = build_context(c, es, &src);
  // per-ensemble physics (skin, dt, tau, shift, parity) come from each member
  if (rcode == RE_OK) {
    for (int i = 0; i < n; ++i) {
      const EnsDev& m = src[i]->ens[0];
      EnsDev& e = c->ens[i];
      e.skin = m.skin;
      e.rlist = m.rlist;
      e.dt = m.dt;
      e.tau = m.tau;
      e.shift = m.shift;
      e.parity_mode = m.parity_mode;
      e.xdist = m.xdist;
      finish_ens(e);
    }
    apply_cells(c, c->opt.cell_div);
    c->cfg = default_cfg(c);
    c->cfg.cell_div = c->opt.cell_div;
    default_class_cfgs(c);
    if (c->opt.path == RE_PATH_BATCHED) rcode = check_cfg(c, c->cfg);
    if (rcode == RE_OK && per_class(c)) rcode = check_class_cfgs(c);
    if (rcode == RE_OK) rcode = upload_tables(c);
    if (rcode == RE_OK) fit_notes(c, true);
  }
  // copy member states
  for (int i = 0; i < n && rcode == RE_OK; ++i) {
    re_ctx* s = src[i];
    const int r0 = c->ens[i].rep_off;
    const size_t a0 = (size_t)c->reps[r0].atom_off, A = (size_t)s->n_atoms;
    const size_t R = (size_t)s->n_rep;
    auto cp = [&](void* dst, const void* srcp, size_t bytes) {
      cudaError_t e = cudaMemcpyAsync(dst, srcp, bytes, cudaMemcpyDeviceToDevice, c->stream);
      if (e != cudaSuccess && rcode == RE_OK) rcode = cuda_fail(c, e, "copy member state");
    };
    cp(c->s.qx + a0, s->s.qx, 8 * A);
    cp(c->s.qy + a0, s->s.qy, 8 * A);
    cp(c->s.qz + a0, s->s.qz, 8 * A);
    cp(c->s.vx + a0, s->s.vx, 8 * A);
    cp(c->s.vy + a0, s->s.vy, 8 * A);
    cp(c->s.vz + a0, s->s.vz, 8 * A);
    cp(c->s.perm + a0, s->s.perm, 4 * A);
    cp(c->s.fx + a0, s->s.fx, 8 * A);
    cp(c->s.fy + a0, s->s.fy, 8 * A);
    cp(c->s.fz + a0, s->s.fz, 8 * A);
    cp(c->s.T + r0, s->s.T, 8 * R);
    cp(c->s.U + r0, s->s.U, 8 * R);
    cp(c->s.K + r0, s->s.K, 8 * R);
    cp(c->s.econs + r0, s->s.econs, 8 * R);
    cp(c->s.vscale + r0, s->s.vscale, 8 * R);
    cp(c->s.lam + r0, s->s.lam, 8 * R);
    cp(c->s.fscale + r0, s->s.fscale, 8 * R);
    cp(c->s.step + r0, s->s.step, 8 * R);
    cp(c->s.nreb + r0, s->s.nreb, 8 * R);
    cp(c->s.status + r0, s->s.status, 4 * R);
    cp(c->s.attempt + i, s->s.attempt, 8);
    if (s->n_pairs > 0) {
      cp(c->s.pair_att + c->ens[i].pair_off, s->s.pair_att, 8 * (size_t)s->n_pairs);
      cp(c->s.pair_acc + c->ens[i].pair_off, s->s.pair_acc, 8 * (size_t)s->n_pairs);
    }
  }
  if (rcode == RE_OK) {
    cudaError_t ce = cudaMemsetAsync(c->s.valid, 0, sizeof(int32_t) * c->n_rep, c->stream);
    if (ce != cudaSuccess) rcode = cuda_fail(c, ce, "memset");
  }
  if (rcode == RE_OK) rcode = refresh(c);
  // the group's first list build is a copy of lists the members had built
  // and counted already: keep the members' rebuild counters
  for (int i = 0; i < n && rcode == RE_OK; ++i) {
    cudaError_t e = cudaMemcpyAsync(c->s.nreb + c->ens[i].rep_off, src[i]->s.nreb,
                                    8 * (size_t)src[i]->n_rep, cudaMemcpyDeviceToDevice, c->stream);
    if (e != cudaSuccess) rcode = cuda_fail(c, e, "copy member counters");
  }
  if (rcode == RE_OK) rcode = status_check(c);
  if (rcode != RE_OK) {
    g_create_error = c->err;
    re_destroy(c);
    return rcode;
  }
  *out = c;
  return RE_OK;
}

int re_advance(re_ctx* c, const int32_t* steps) {
  ApiRange range_("re_advance");
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  if (!steps) return launch_advance(c, c->d_budget_nx, nullptr, c->opt.nx);
  for (int r = 0; r < c->n_rep; ++r)
    if (steps[r] < 0) return fail(c, RE_EINVAL, "steps[%d] is negative", r);
  if (c->opt.path == RE_PATH_PLAIN) return launch_advance(c, nullptr, steps);
  // the device copy of the budgets is kept: a call with the same budgets as
  // the last upload (the rule for fixed strides) copies nothing
  const size_t bb = sizeof(int32_t) * (size_t)c->n_rep;
  if (!c->budget_cached || std::memcmp(c->h_budget_last.data(), steps, bb) != 0) {
    // stage the budgets in a pinned ring slot, then copy asynchronously
    const int slot = c->ring_pos;
    c->ring_pos = (c->ring_pos + 1) % kRing;
    RE_CUDA(c, cudaEventSynchronize(c->ring_ev[slot]), "ring wait");
    int32_t* h = c->h_ring + (size_t)slot * c->n_rep;
    std::memcpy(h, steps, bb);
    RE_CUDA(c, cudaMemcpyAsync(c->d_budget, h, bb, cudaMemcpyHostToDevice, c->stream),
            "upload budgets");
    RE_CUDA(c, cudaEventRecord(c->ring_ev[slot], c->stream), "ring record");
    c->h_budget_last.assign(steps, steps + c->n_rep);
    c->budget_cached = true;
  }
  int mx = 0, mn = INT_MAX;
  for (int r = 0; r < c->n_rep; ++r) {
    mx = std::max(mx, (int)steps[r]);
    mn = std::min(mn, (int)steps[r]);
  }
  return launch_advance(c, c->d_budget, nullptr, mx, 0, nullptr, mn != mx);
}

namespace {

// The shape of a free-running launch, in which replicas wait for one another:
// all its clusters must be resident at once.  The tuned shape when it is
// (*narrower = false); otherwise (fcfg, *narrower = true) the first resident
// one with fewer CTAs per replica, trying the tuned threads per atom first
// (same list layout) and then fewer.
int free_shape(re_ctx* c, bool* narrower) {
  const bool fp64 = c->opt.precision == RE_PREC_FP64;
  *narrower = false;
  if (c->resident_clusters < 0)
    c->resident_clusters = re::batched_max_active_clusters(fp64, c->cfg, c->max_n);
  if (c->n_rep <= c->resident_clusters) return RE_OK;
  const std::string err = c->err;
  const int clusters[5] = {8, 4, 3, 2, 1};
  const int pvals[4] = {8, 4, 2, 1};
  for (int cl : clusters) {
    if (cl >= c->cfg.cluster) continue;
    for (int pass = 0; pass < 2; ++pass)
      for (int p : pvals) {
        // pass 0: the tuned threads per atom; pass 1: fewer
        if (pass == 0 ? p != c->cfg.atom_threads : p >= c->cfg.atom_threads) continue;
        LaunchCfg k{cl, threads_for(c->max_n, cl, p), c->cfg.cell_div, p, 0, 0, 0, 0, 0};
        if (k.threads > 1024 || check_cfg(c, k) != RE_OK) continue;
        if (re::batched_max_active_clusters(fp64, k, c->max_n) < c->n_rep) continue;
        c->err = err;
        c->fcfg = k;
        *narrower = true;
        return RE_OK;
      }
  }
  return fail(c, RE_EINVAL,
              "free-running exchange needs all %d replicas resident at once; %d clusters of the "
              "tuned launch shape fit on the GPU, and no shape with fewer CTAs per replica holds "
              "them all", c->n_rep, c->resident_clusters);
}

}  // namespace

int re_advance_async(re_ctx* c, int nx) {
  ApiRange range_("re_advance_async");
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  if (nx < 1) return fail(c, RE_EINVAL, "nx must be >= 1");
  if (c->opt.path != RE_PATH_BATCHED)
    return fail(c, RE_EINVAL, "free-running mode needs the batched path");
  // the cap of the non-master replicas bounds the host's step bookkeeping
  return launch_advance(c, c->d_budget_nx, nullptr, nx, nx);
}

int re_run_free(re_ctx* c, int n_att, int nx, int64_t* log_step, double* log_T,
                int32_t* log_partner, uint8_t* log_acc) {
  ApiRange range_("re_run_free");
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  if (n_att < 0 || nx < 1) return fail(c, RE_EINVAL, "n_att >= 0 and nx >= 1 required");
  if (c->opt.path != RE_PATH_BATCHED)
    return fail(c, RE_EINVAL, "free-running mode needs the batched path");
  if (n_att == 0) return RE_OK;
  if ((int64_t)(n_att + 1) * (16 * (int64_t)nx + 16) > INT32_MAX)
    return fail(c, RE_EINVAL, "n_att * nx too large for one launch");
  // every replica waits for others inside the launch: all clusters must be
  // resident at once -- in the tuned shape, or else in a narrower one
  bool narrower = false;
  {
    const int rc = free_shape(c, &narrower);
    if (rc) return rc;
  }
  const int E = (int)c->ens.size(), R = c->n_rep;
  const bool want_log = log_step || log_T || log_partner || log_acc;
  if (!c->d_fr_words) {
    int rc;
    if ((rc = dalloc(c, &c->d_fr_words, (size_t)2 * E + 5 * (size_t)R)) ||
        (rc = dalloc(c, &c->d_fr_slot, 4 * (size_t)R)))
      return rc;
  }
  if (want_log && c->log_rows < n_att) {
    dfree(c, c->d_log_step);
    dfree(c, c->d_log_T);
    dfree(c, c->d_log_partner);
    dfree(c, c->d_log_acc);
    int rc;
    const size_t n = (size_t)n_att * R;
    if ((rc = dalloc(c, &c->d_log_step, n)) || (rc = dalloc(c, &c->d_log_T, n)) ||
        (rc = dalloc(c, &c->d_log_partner, n)) || (rc = dalloc(c, &c->d_log_acc, n)))
      return rc;
    c->log_rows = n_att;
  }
  re::FreeDev fr{};
  fr.nx = nx;
  fr.n_att = n_att;
  fr.log_cap = want_log ? n_att : 0;
  fr.rtot = R;
  fr.wait_ns = (uint64_t)(c->wait_s * 1e9);
  fr.stall_rep = c->stall_rep;  // one call only
  fr.stall_from = c->stall_from;
  c->stall_rep = -1;
  fr.issue = c->d_fr_words;
  fr.abort_ = fr.issue + E;
  fr.partner = fr.abort_ + E;
  fr.pos = fr.partner + R;
  fr.done = fr.pos + R;
  fr.flag = fr.done + R;
  fr.order = fr.flag + R;
  fr.slot = c->d_fr_slot;
  fr.key = c->d_fr_slot + 3 * (size_t)R;
  fr.log_step = c->d_log_step;
  fr.log_T = c->d_log_T;
  fr.log_partner = c->d_log_partner;
  fr.log_acc = c->d_log_acc;
  RE_CUDA(c, cudaMemsetAsync(c->d_fr_words, 0, sizeof(int32_t) * (2 * (size_t)E + 5 * (size_t)R),
                             c->stream), "clear exchange words");
  if (want_log) {
    // entries of replicas that never take part in an attempt keep step -1
    const size_t n = (size_t)n_att * R;
    RE_CUDA(c, cudaMemsetAsync(c->d_log_step, 0xFF, 8 * n, c->stream), "clear log");
    RE_CUDA(c, cudaMemsetAsync(c->d_log_partner, 0xFF, 4 * n, c->stream), "clear log");
    RE_CUDA(c, cudaMemsetAsync(c->d_log_acc, 0, 4 * n, c->stream), "clear log");
    RE_CUDA(c, cudaMemsetAsync(c->d_log_T, 0, 8 * n, c->stream), "clear log");
  }
  c->use_fcfg = narrower;
  fit_notes(c, false);
  int rc = launch_advance(c, c->d_budget_nx, nullptr, n_att * nx, 0, &fr);
  c->use_fcfg = false;
  if (rc) return rc;
  RE_CUDA(c, re::launch_attempt_add(c->s, E, n_att, c->stream), "attempt counters");
  // back to the tuned shape's list layout (replicas stopped by a failed wait
  // keep invalid lists and rebuild them at their next launch)
  if (narrower && (rc = relayout_lists(c, 0))) return rc;
  if (!want_log) return RE_OK;
  // the log is read back also when the launch failed: it shows where every
  // replica stopped
  rc = status_check(c);
  if (rc != RE_OK && rc != RE_ETIMEOUT) return rc;
  const size_t n = (size_t)n_att * R;
  if (log_step)
    RE_CUDA(c, cudaMemcpy(log_step, c->d_log_step, 8 * n, cudaMemcpyDeviceToHost), "read log");
  if (log_T) RE_CUDA(c, cudaMemcpy(log_T, c->d_log_T, 8 * n, cudaMemcpyDeviceToHost), "read log");
  if (log_partner)
    RE_CUDA(c, cudaMemcpy(log_partner, c->d_log_partner, 4 * n, cudaMemcpyDeviceToHost),
            "read log");
  if (log_acc) {
    std::vector<int32_t> a(n);
    RE_CUDA(c, cudaMemcpy(a.data(), c->d_log_acc, 4 * n, cudaMemcpyDeviceToHost), "read log");
    for (size_t k = 0; k < n; ++k) log_acc[k] = (uint8_t)a[k];
  }
  return rc;
}

int re_set_wait_limit(re_ctx* c, double seconds) {
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  if (!(seconds >= 1e-4 && seconds <= 10.0))
    return fail(c, RE_EINVAL, "wait limit must be in [1e-4, 10] seconds");
  c->wait_s = seconds;
  return RE_OK;
}

int re_inject_stall(re_ctx* c, int replica, int from_attempt) {
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  if (replica < -1 || replica >= c->n_rep || from_attempt < 0)
    return fail(c, RE_EINVAL, "replica must be in [-1, n_rep) and from_attempt >= 0");
  c->stall_rep = replica;
  c->stall_from = from_attempt;
  return RE_OK;
}

int re_run_async(re_ctx* c, int n_cycles, int nx, int use_graph) {
  ApiRange range_("re_run_async");
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  if (n_cycles < 0 || nx < 1) return fail(c, RE_EINVAL, "n_cycles >= 0 and nx >= 1 required");
  if (c->opt.path != RE_PATH_BATCHED)
    return fail(c, RE_EINVAL, "free-running mode needs the batched path");
  auto enqueue = [&]() -> int {
    for (int k = 0; k < n_cycles; ++k) {
      int rc = launch_advance(c, c->d_budget_nx, nullptr, nx, nx);
      if (rc) return rc;
      cudaError_t e = re::launch_exchange(c->s, c->d_ens, (int)c->ens.size(), c->max_r,
                                          c->d_partner, c->d_acc, c->stream);
      if (e != cudaSuccess) return cuda_fail(c, e, "exchange launch");
    }
    return RE_OK;
  };
  if (!use_graph || n_cycles == 0) return enqueue();
  // master-stop launches use the uniform shape's list layout: switch to it
  // before the capture, not inside the graph
  {
    const int rc = relayout_lists(c, 0);
    if (rc) return rc;
  }
  cudaStream_t cap = nullptr;
  RE_CUDA(c, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "stream");
  cudaStream_t saved = c->stream;
  c->stream = cap;
  cudaGraph_t g = nullptr;
  int rc = RE_OK;
  cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    rc = enqueue();
    cudaError_t e2 = cudaStreamEndCapture(cap, &g);
    if (rc == RE_OK && e2 != cudaSuccess) rc = cuda_fail(c, e2, "graph capture");
  } else {
    rc = cuda_fail(c, e, "begin capture");
  }
  c->stream = saved;
  cudaStreamDestroy(cap);
  if (rc) {
    if (g) cudaGraphDestroy(g);
    return rc;
  }
  cudaGraphExec_t ge = nullptr;
  e = cudaGraphInstantiate(&ge, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return cuda_fail(c, e, "graph instantiate");
  e = cudaGraphLaunch(ge, c->stream);
  cudaGraphExecDestroy(ge);  // released once the launch completes
  if (e != cudaSuccess) return cuda_fail(c, e, "graph launch");
  return RE_OK;
}

int re_exchange(re_ctx* c, int32_t* partner_out, uint8_t* accepted_out) {
  ApiRange range_("re_exchange");
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  cudaError_t e = re::launch_exchange(c->s, c->d_ens, (int)c->ens.size(), c->max_r, c->d_partner,
                                      c->d_acc, c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "exchange launch");
  if (!partner_out && !accepted_out) return RE_OK;
  // through the pinned read-back area: one asynchronous copy, one wait
  RE_CUDA(c, cudaMemcpyAsync(out_partner(c), c->d_partner, 5 * (size_t)c->n_rep,
                             cudaMemcpyDeviceToHost, c->stream), "read partners and decisions");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  if (partner_out) std::memcpy(partner_out, out_partner(c), sizeof(int32_t) * c->n_rep);
  if (accepted_out) std::memcpy(accepted_out, out_acc(c), c->n_rep);
  return RE_OK;
}

int re_run(re_ctx* c, int n_cycles, const int32_t* steps, int use_graph) {
  ApiRange range_("re_run");
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  if (n_cycles < 0) return fail(c, RE_EINVAL, "n_cycles must be >= 0");
  if (n_cycles == 0) return RE_OK;
  if (c->opt.path == RE_PATH_PLAIN) {
    for (int k = 0; k < n_cycles; ++k) {
      int rc = re_advance(c, steps ? steps + (size_t)k * c->n_rep : nullptr);
      if (rc) return rc;
      rc = re_exchange(c, nullptr, nullptr);
      if (rc) return rc;
    }
    return RE_OK;
  }
  const int32_t* dbud = c->d_budget_nx;
  size_t stride = 0;
  if (steps) {
    const size_t need = (size_t)n_cycles * c->n_rep;
    for (size_t i = 0; i < need; ++i)
      if (steps[i] < 0) return fail(c, RE_EINVAL, "negative step budget");
    if (need > c->budget_run_cap) {
      if (c->graph) {
        cudaGraphExecDestroy(c->graph);
        c->graph = nullptr;
      }
      if (c->d_budget_run) {
        cudaStreamSynchronize(c->stream);
        cudaFree(c->d_budget_run);
        auto it = std::find(c->allocs.begin(), c->allocs.end(), (void*)c->d_budget_run);
        if (it != c->allocs.end()) c->allocs.erase(it);
        c->d_budget_run = nullptr;
      }
      int rc = dalloc(c, &c->d_budget_run, need);
      if (rc) return rc;
      c->budget_run_cap = need;
    }
    RE_CUDA(c, cudaMemcpyAsync(c->d_budget_run, steps, sizeof(int32_t) * need,
                               cudaMemcpyHostToDevice, c->stream), "upload budgets");
    dbud = c->d_budget_run;
    stride = (size_t)c->n_rep;
  }
  auto enqueue = [&]() -> int {
    for (int k = 0; k < n_cycles; ++k) {
      int mx = c->opt.nx, mn = c->opt.nx;
      if (steps) {
        mx = 0;
        mn = INT_MAX;
        for (int r = 0; r < c->n_rep; ++r) {
          mx = std::max(mx, (int)steps[(size_t)k * c->n_rep + r]);
          mn = std::min(mn, (int)steps[(size_t)k * c->n_rep + r]);
        }
      }
      int rc = launch_advance(c, dbud + stride * k, nullptr, mx, 0, nullptr, mn != mx);
      if (rc) return rc;
      cudaError_t e = re::launch_exchange(c->s, c->d_ens, (int)c->ens.size(), c->max_r,
                                          c->d_partner, c->d_acc, c->stream);
      if (e != cudaSuccess) return cuda_fail(c, e, "exchange launch");
    }
    return RE_OK;
  };
  if (!use_graph) return enqueue();
  // the graph's launches expect the budget launches' list layout: restore it
  // first, outside the graph (a free-running call in between may have
  // switched it), so that neither a capture nor a replay meets the other one
  {
    const int rc = relayout_lists(c, per_class(c) ? 1 : 0);
    if (rc) return rc;
  }
  if (!c->graph || c->graph_cycles != n_cycles || c->graph_budget != dbud) {
    if (c->graph) {
      cudaGraphExecDestroy(c->graph);
      c->graph = nullptr;
    }
    cudaStream_t cap = nullptr;
    RE_CUDA(c, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "stream");
    cudaStream_t saved = c->stream;
    c->stream = cap;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    int rc = RE_OK;
    if (e == cudaSuccess) {
      rc = enqueue();
      cudaError_t e2 = cudaStreamEndCapture(cap, &g);
      if (rc == RE_OK && e2 != cudaSuccess) rc = cuda_fail(c, e2, "graph capture");
    } else {
      rc = cuda_fail(c, e, "begin capture");
    }
    c->stream = saved;
    cudaStreamDestroy(cap);
    if (rc) {
      if (g) cudaGraphDestroy(g);
      return rc;
    }
    e = cudaGraphInstantiate(&c->graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(c, e, "graph instantiate");
    c->graph_cycles = n_cycles;
    c->graph_budget = dbud;
  }
  RE_CUDA(c, cudaGraphLaunch(c->graph, c->stream), "graph launch");
  return RE_OK;
}

namespace {

// Frees a device buffer of the context's allocation list.
void dfree_tracked(re_ctx* c, void* p) {
  if (!p) return;
  cudaFree(p);
  auto it = std::find(c->allocs.begin(), c->allocs.end(), p);
  if (it != c->allocs.end()) c->allocs.erase(it);
}

}  // namespace

int re_run_record(re_ctx* c, int n_cycles, const int32_t* steps, int use_graph, int32_t* partner,
                  uint8_t* accepted, double* T, double* U, double* K, double* H) {
  ApiRange range_("re_run_record");
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  if (n_cycles < 0) return fail(c, RE_EINVAL, "n_cycles must be >= 0");
  if (n_cycles == 0) return RE_OK;
  const size_t R = (size_t)c->n_rep, nb = (size_t)n_cycles * R;
  if (steps)
    for (size_t i = 0; i < nb; ++i)
      if (steps[i] < 0) return fail(c, RE_EINVAL, "negative step budget");
  const bool plain = c->opt.path == RE_PATH_PLAIN;
  // record row: T, U, K, econs (doubles), partner (int32), accepted (bytes)
  const size_t rowb = (37 * R + 7) & ~(size_t)7;
  const size_t off_part = 32 * R, off_acc = 36 * R;
  if (rowb * n_cycles > c->rec_cap || (steps && !plain && nb > c->rec_bud_cap)) {
    RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
    if (c->rec_graph) {  // it holds the addresses of the areas replaced here
      cudaGraphExecDestroy(c->rec_graph);
      c->rec_graph = nullptr;
    }
    if (rowb * n_cycles > c->rec_cap) {
      dfree_tracked(c, c->d_rec);
      c->d_rec = nullptr;
      if (c->h_rec) cudaFreeHost(c->h_rec);
      c->h_rec = nullptr;
      c->rec_cap = 0;
      int rc = dalloc(c, &c->d_rec, rowb * n_cycles);
      if (rc) return rc;
      RE_CUDA(c, cudaMallocHost(&c->h_rec, rowb * n_cycles), "cudaMallocHost");
      c->rec_cap = rowb * n_cycles;
    }
    if (steps && !plain && nb > c->rec_bud_cap) {
      dfree_tracked(c, c->d_rec_bud);
      c->d_rec_bud = nullptr;
      if (c->h_rec_bud) cudaFreeHost(c->h_rec_bud);
      c->h_rec_bud = nullptr;
      c->rec_bud_cap = 0;
      int rc = dalloc(c, &c->d_rec_bud, nb);
      if (rc) return rc;
      RE_CUDA(c, cudaMallocHost(&c->h_rec_bud, sizeof(int32_t) * nb), "cudaMallocHost");
      c->rec_bud_cap = nb;
    }
  }
  if (!c->rec_in) {
    RE_CUDA(c, cudaStreamCreateWithFlags(&c->rec_in, cudaStreamNonBlocking), "stream");
    RE_CUDA(c, cudaStreamCreateWithFlags(&c->rec_out, cudaStreamNonBlocking), "stream");
    RE_CUDA(c, cudaEventCreateWithFlags(&c->ev_in, cudaEventDisableTiming), "event");
    RE_CUDA(c, cudaEventCreateWithFlags(&c->ev_out, cudaEventDisableTiming), "event");
  }
  // a previous call that failed half-way may still be copying
  RE_CUDA(c, cudaStreamSynchronize(c->rec_in), "synchronise");
  RE_CUDA(c, cudaStreamSynchronize(c->rec_out), "synchronise");
  if (steps && !plain) std::memcpy(c->h_rec_bud, steps, sizeof(int32_t) * nb);
  // the cycles: budgets in on rec_in, advance and exchange on the context's
  // stream, records out on rec_out; both copy streams join the stream at the end
  auto enqueue = [&]() -> int {
    for (int k = 0; k < n_cycles; ++k) {
      const int32_t* hrow = steps ? steps + (size_t)k * R : nullptr;
      int rc;
      if (plain) {
        rc = launch_advance(c, nullptr, hrow);
      } else if (hrow) {
        int mx = 0, mn = INT_MAX;
        for (size_t r = 0; r < R; ++r) {
          mx = std::max(mx, (int)hrow[r]);
          mn = std::min(mn, (int)hrow[r]);
        }
        // this cycle's budgets: their own copy, which the advance waits for
        int32_t* drow = c->d_rec_bud + (size_t)k * R;
        RE_CUDA(c, cudaMemcpyAsync(drow, c->h_rec_bud + (size_t)k * R, sizeof(int32_t) * R,
                                   cudaMemcpyHostToDevice, c->rec_in), "upload budgets");
        RE_CUDA(c, cudaEventRecord(c->ev_in, c->rec_in), "event");
        RE_CUDA(c, cudaStreamWaitEvent(c->stream, c->ev_in, 0), "event wait");
        rc = launch_advance(c, drow, nullptr, mx, 0, nullptr, mn != mx);
      } else {
        rc = launch_advance(c, c->d_budget_nx, nullptr, c->opt.nx);
      }
      if (rc) return rc;
      unsigned char* row = c->d_rec + (size_t)k * rowb;
      cudaError_t e = re::launch_exchange(c->s, c->d_ens, (int)c->ens.size(), c->max_r,
                                          reinterpret_cast<int32_t*>(row + off_part),
                                          row + off_acc, c->stream,
                                          reinterpret_cast<double*>(row), (int)R);
      if (e != cudaSuccess) return cuda_fail(c, e, "exchange launch");
      // the record of cycle k travels while cycle k + 1 runs
      RE_CUDA(c, cudaEventRecord(c->ev_out, c->stream), "event");
      RE_CUDA(c, cudaStreamWaitEvent(c->rec_out, c->ev_out, 0), "event wait");
      RE_CUDA(c, cudaMemcpyAsync(c->h_rec + (size_t)k * rowb, row, rowb, cudaMemcpyDeviceToHost,
                                 c->rec_out), "read record");
    }
    RE_CUDA(c, cudaEventRecord(c->ev_in, c->rec_in), "event");
    RE_CUDA(c, cudaStreamWaitEvent(c->stream, c->ev_in, 0), "event wait");
    RE_CUDA(c, cudaEventRecord(c->ev_out, c->rec_out), "event");
    RE_CUDA(c, cudaStreamWaitEvent(c->stream, c->ev_out, 0), "event wait");
    return RE_OK;
  };
  if (!use_graph || plain) {
    const int rc = enqueue();
    if (rc) return rc;
  } else {
    // the budget launches' list layout, switched outside the graph
    int rc = relayout_lists(c, per_class(c) ? 1 : 0);
    if (rc) return rc;
    if (!c->rec_graph || c->rec_graph_cycles != n_cycles ||
        c->rec_graph_steps != (steps != nullptr)) {
      if (c->rec_graph) {
        cudaGraphExecDestroy(c->rec_graph);
        c->rec_graph = nullptr;
      }
      cudaStream_t cap = nullptr;
      RE_CUDA(c, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "stream");
      cudaStream_t saved = c->stream;
      c->stream = cap;
      cudaGraph_t g = nullptr;
      cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        // the copy streams join the capture through an event of the stream
        e = cudaEventRecord(c->ev_out, cap);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(c->rec_in, c->ev_out, 0);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(c->rec_out, c->ev_out, 0);
        rc = e == cudaSuccess ? enqueue() : cuda_fail(c, e, "graph fork");
        cudaError_t e2 = cudaStreamEndCapture(cap, &g);
        if (rc == RE_OK && e2 != cudaSuccess) rc = cuda_fail(c, e2, "graph capture");
      } else {
        rc = cuda_fail(c, e, "begin capture");
      }
      c->stream = saved;
      cudaStreamDestroy(cap);
      if (rc) {
        if (g) cudaGraphDestroy(g);
        return rc;
      }
      e = cudaGraphInstantiate(&c->rec_graph, g, 0);
      cudaGraphDestroy(g);
      if (e != cudaSuccess) return cuda_fail(c, e, "graph instantiate");
      c->rec_graph_cycles = n_cycles;
      c->rec_graph_steps = steps != nullptr;
    }
    RE_CUDA(c, cudaGraphLaunch(c->rec_graph, c->stream), "graph launch");
  }
  const int rc = status_check(c);  // synchronises the stream, and so the copies
  if (rc != RE_OK && rc != RE_ENUMERIC && rc != RE_EOVERFLOW) return rc;
  for (int k = 0; k < n_cycles; ++k) {
    const unsigned char* row = c->h_rec + (size_t)k * rowb;
    const double* d = reinterpret_cast<const double*>(row);
    const int32_t* pr = reinterpret_cast<const int32_t*>(row + off_part);
    const size_t o = (size_t)k * R;
    for (size_t r = 0; r < R; ++r) {
      if (T) T[o + r] = d[r];
      if (U) U[o + r] = d[R + r];
      if (K) K[o + r] = d[2 * R + r];
      if (H) H[o + r] = d[R + r] + d[2 * R + r] + d[3 * R + r];
      if (partner) partner[o + r] = pr[r];
      if (accepted) accepted[o + r] = row[off_acc + r];
    }
  }
  return rc;
}

int re_energies(re_ctx* c, double* U, double* K, double* H) {
  ApiRange range_("re_energies");
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  // energies and status in one copy (pinned destination)
  const size_t R = (size_t)c->n_rep;
  RE_CUDA(c, cudaMemcpyAsync(out_U(c), c->s.U, 28 * R, cudaMemcpyDeviceToHost, c->stream),
          "read energies");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  int rc = status_eval(c, out_status(c));
  if (rc) return rc;
  const double *u = out_U(c), *k = out_K(c), *e = out_econs(c);
  for (size_t r = 0; r < R; ++r) {
    if (U) U[r] = u[r];
    if (K) K[r] = k[r];
    if (H) H[r] = u[r] + k[r] + e[r];
  }
  return RE_OK;
}

int re_apply_exchange(re_ctx* c, const double* T_new, const double* lam_new,
                      const double* vscale, const double* uscale) {
  if (!c || !T_new || !vscale) return fail(c, RE_EINVAL, "bad arguments");
  const int R = c->n_rep;
  std::vector<double> in(4 * (size_t)R);
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  if (!lam_new)
    RE_CUDA(c, cudaMemcpy(in.data() + R, c->s.lam, 8 * (size_t)R, cudaMemcpyDeviceToHost),
            "read lam");
  for (int r = 0; r < R; ++r) {
    in[r] = T_new[r];
    if (lam_new) in[R + r] = lam_new[r];
    in[2 * R + r] = vscale[r];
    in[3 * R + r] = uscale ? uscale[r] : 1.0;
    if (!(in[r] > 0) || !(in[R + r] > 0) || !(in[2 * R + r] > 0) || !(in[3 * R + r] > 0))
      return fail(c, RE_EINVAL, "replica %d: T, lam and the factors must be positive", r);
  }
  RE_CUDA(c, cudaMemcpyAsync(c->d_io, in.data(), 8 * in.size(), cudaMemcpyHostToDevice,
                             c->stream), "upload exchange");
  cudaError_t e = re::launch_apply_exchange(c->s, c->d_io, R, c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "apply exchange");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  return RE_OK;
}

int re_lambdas(re_ctx* c, double* lam) {
  if (!c || !lam) return fail(c, RE_EINVAL, "bad arguments");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  RE_CUDA(c, cudaMemcpy(lam, c->s.lam, sizeof(double) * c->n_rep, cudaMemcpyDeviceToHost),
          "read lam");
  return RE_OK;
}

int re_temps(re_ctx* c, double* T) {
  if (!c || !T) return fail(c, RE_EINVAL, "bad arguments");
  RE_CUDA(c, cudaMemcpyAsync(out_U(c), c->s.T, sizeof(double) * c->n_rep, cudaMemcpyDeviceToHost,
                             c->stream), "read T");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  std::memcpy(T, out_U(c), sizeof(double) * c->n_rep);
  return RE_OK;
}

int re_get_state(re_ctx* c, double* x, double* v) {
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  const size_t n3 = 3 * (size_t)c->n_atoms;
  // both in one launch (v into the re-sort's staging words), pending factors of
  // an exchange applied to what is read
  double* dv = reinterpret_cast<double*>(c->s.sbuf);
  const cudaError_t e = re::launch_export_state(c->s, c->d_ens, c->d_rep, c->n_rep,
                                                x ? c->d_io : nullptr, v ? dv : nullptr, nullptr,
                                                c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "export");
  if (x) RE_CUDA(c, cudaMemcpyAsync(x, c->d_io, 8 * n3, cudaMemcpyDeviceToHost, c->stream), "read x");
  if (v) RE_CUDA(c, cudaMemcpyAsync(v, dv, 8 * n3, cudaMemcpyDeviceToHost, c->stream), "read v");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  return RE_OK;
}

namespace {

// Whether atoms that follow one another in x mostly lie within the list radius
// of one another (a sample of about a thousand pairs over all replicas).  Where
// they don't -- any order that does not follow space -- the atoms are renumbered
// before the next lists instead of at the next interval: 64 x 4000 atoms in
// random order 64 us a step instead of 79, 8 x 2048 atoms of four slabs in turn
// (whose sub-lists overflow and are dealt) 15 instead of 39.  An order that
// follows space is kept: the sort costs 20 to 50 us, and its cells of about 30
// atoms are a coarser order than a lattice's rows.
bool numbered_in_space(const re_ctx* c, const double* x) {
  const int per = std::max(1, 1024 / c->n_rep);
  int near = 0, n = 0;
  for (int r = 0; r < c->n_rep; ++r) {
    const EnsDev& e = c->ens[c->reps[r].ens];
    const double* xr = x + 3 * (size_t)c->reps[r].atom_off;
    for (int k = 0; k < per; ++k) {
      const int i = (int)(((int64_t)k * (e.N - 1) / per + 7 * r) % (e.N - 1));
      double r2 = 0.0;
      for (int d = 0; d < 3; ++d) {
        double s = (xr[3 * (i + 1) + d] - xr[3 * i + d]) * e.kc.inv_l;
        s -= std::nearbyint(s);
        r2 += s * s * e.L * e.L;
      }
      near += r2 < e.rlist * e.rlist ? 1 : 0;
      ++n;
    }
  }
  return 2 * near >= n;
}

}  // namespace

int re_set_state(re_ctx* c, const double* x, const double* v) {
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  const size_t n3 = 3 * (size_t)c->n_atoms;
  cudaError_t e = re::launch_apply_vscale(c->s, c->d_rep, c->d_ens, c->n_rep, c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "apply velocity factors");
  if (x) {
    RE_CUDA(c, cudaMemcpyAsync(c->d_io, x, 8 * n3, cudaMemcpyHostToDevice, c->stream), "write x");
    e = re::launch_import_state(c->s, c->d_ens, c->d_rep, c->n_rep, c->d_io, nullptr, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "import");
    RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
    if (c->sort_every > 0 && !numbered_in_space(c, x)) c->since_sort = c->sort_every;
  }
  if (v) {
    RE_CUDA(c, cudaMemcpyAsync(c->d_io, v, 8 * n3, cudaMemcpyHostToDevice, c->stream), "write v");
    e = re::launch_import_state(c->s, c->d_ens, c->d_rep, c->n_rep, nullptr, c->d_io, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "import");
  }
  int rc = refresh(c);
  if (rc) return rc;
  return status_check(c);
}

namespace {

// A checkpoint: this header, the launch shape of every ensemble's class (the
// lists' layout follows the threads per atom), then the arrays of
// ckpt_arrays() in order.
struct CkptHeader {
  char magic[8];
  uint32_t version, precision, path, n_ens;
  int32_t n_rep, n_pairs, plain_refresh, list_mode;
  int64_t n_atoms, n_nbr, since_sort, payload;
  LaunchCfg cfg;
  uint64_t shape;  // hash of the ensembles' parameters and the replica table
};
constexpr char kCkptMagic[8] = {'R', 'E', '-', 'C', 'K', 'P', 'T', '3'};

struct CkptArray {
  void* dev;
  size_t bytes;
};

// Everything the next call reads (scratch buffers and per-launch words excluded).
std::vector<CkptArray> ckpt_arrays(re_ctx* c) {
  const size_t A = (size_t)c->n_atoms, R = (size_t)c->n_rep, E = c->ens.size();
  const size_t P = (size_t)c->n_pairs;
  StateDev& s = c->s;
  return {{s.qx, 8 * A},     {s.qy, 8 * A},      {s.qz, 8 * A},     {s.vx, 8 * A},
          {s.vy, 8 * A},     {s.vz, 8 * A},      {s.fx, 8 * A},     {s.fy, 8 * A},
          {s.fz, 8 * A},     {s.rx, 4 * A},      {s.ry, 4 * A},     {s.rz, 4 * A},
          {s.ncnt, 32 * A},  {s.perm, 4 * A},    {s.nbr, 2 * (size_t)c->n_nbr},
          {s.T, 8 * R},      {s.U, 8 * R},       {s.K, 8 * R},      {s.econs, 8 * R},
          {s.vscale, 8 * R}, {s.lam, 8 * R},     {s.fscale, 8 * R}, {s.step, 8 * R},
          {s.nreb, 8 * R},   {s.status, 4 * R},  {s.valid, 4 * R},  {s.dmax, 4 * R},
          {s.attempt, 8 * E}, {s.pair_att, 8 * P}, {s.pair_acc, 8 * P}};
}

// FNV-1a over the parameters that fix the context's shape and trajectories.
uint64_t ckpt_shape(const re_ctx* c) {
  uint64_t h = 1469598103934665603ull;
  auto mix = [&](const void* p, size_t n) {
    const unsigned char* b = static_cast<const unsigned char*>(p);
    for (size_t i = 0; i < n; ++i) h = (h ^ b[i]) * 1099511628211ull;
  };
  for (const EnsDev& e : c->ens) {
    const int iv[7] = {e.N, e.R, e.rep_off, e.pair_off, e.cap, e.shift, e.xdist};
    const double dv[6] = {e.L, e.rc, e.rlist, e.skin, e.dt, e.tau};
    mix(iv, sizeof iv);
    mix(e.capsub, sizeof e.capsub);
    mix(dv, sizeof dv);
    mix(&e.seed, sizeof e.seed);
    mix(&e.parity_mode, sizeof e.parity_mode);
  }
  for (const RepDev& r : c->reps) {
    const int64_t v[5] = {r.ens, r.id, r.atom_off, r.stream, r.nbr_off};
    mix(v, sizeof v);
  }
  const int ov[4] = {c->opt.shift_energy, c->opt.sort_interval, c->opt.nx, per_class(c) ? 1 : 0};
  mix(ov, sizeof ov);
  return h;
}

size_t ckpt_bytes(re_ctx* c) {
  size_t n = sizeof(CkptHeader) + sizeof(LaunchCfg) * c->ens.size();
  for (const CkptArray& a : ckpt_arrays(c)) n += a.bytes;
  return n;
}

}  // namespace

int re_checkpoint_size(const re_ctx* c, size_t* bytes) {
  if (!c || !bytes) return fail(const_cast<re_ctx*>(c), RE_EINVAL, "bad arguments");
  *bytes = ckpt_bytes(const_cast<re_ctx*>(c));
  return RE_OK;
}

int re_checkpoint_save(re_ctx* c, void* buf, size_t bytes) {
  ApiRange range_("re_checkpoint_save");
  if (!c || !buf) return fail(c, RE_EINVAL, "bad arguments");
  const size_t need = ckpt_bytes(c);
  if (bytes < need) return fail(c, RE_EINVAL, "checkpoint buffer of %zu bytes, %zu needed", bytes, need);
  CkptHeader h{};
  std::memcpy(h.magic, kCkptMagic, sizeof h.magic);
  h.version = 1;
  h.precision = (uint32_t)c->opt.precision;
  h.path = (uint32_t)c->opt.path;
  h.n_ens = (uint32_t)c->ens.size();
  h.n_rep = c->n_rep;
  h.n_pairs = c->n_pairs;
  h.plain_refresh = c->plain_refresh ? 1 : 0;
  h.list_mode = c->list_mode;
  h.n_atoms = c->n_atoms;
  h.n_nbr = c->n_nbr;
  h.since_sort = c->since_sort;
  h.payload = (int64_t)(need - sizeof h);
  h.cfg = c->cfg;
  h.shape = ckpt_shape(c);
  unsigned char* out = static_cast<unsigned char*>(buf);
  std::memcpy(out, &h, sizeof h);
  size_t off = sizeof h;
  std::memcpy(out + off, c->ecfg.data(), sizeof(LaunchCfg) * c->ens.size());
  off += sizeof(LaunchCfg) * c->ens.size();
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  for (const CkptArray& a : ckpt_arrays(c)) {
    if (a.bytes)
      RE_CUDA(c, cudaMemcpy(out + off, a.dev, a.bytes, cudaMemcpyDeviceToHost), "checkpoint read");
    off += a.bytes;
  }
  return RE_OK;
}

int re_checkpoint_load(re_ctx* c, const void* buf, size_t bytes) {
  ApiRange range_("re_checkpoint_load");
  if (!c || !buf) return fail(c, RE_EINVAL, "bad arguments");
  CkptHeader h{};
  if (bytes < sizeof h) return fail(c, RE_EINVAL, "not a checkpoint (%zu bytes)", bytes);
  std::memcpy(&h, buf, sizeof h);
  if (std::memcmp(h.magic, kCkptMagic, sizeof h.magic) != 0 || h.version != 1)
    return fail(c, RE_EINVAL, "not a checkpoint of this library");
  if (h.precision != (uint32_t)c->opt.precision || h.path != (uint32_t)c->opt.path ||
      h.n_ens != (uint32_t)c->ens.size() || h.n_rep != c->n_rep || h.n_pairs != c->n_pairs ||
      h.n_atoms != c->n_atoms || h.n_nbr != c->n_nbr || h.shape != ckpt_shape(c))
    return fail(c, RE_EINVAL, "checkpoint of a context of another shape, seed or options");
  if (h.payload < 0 || bytes < sizeof h + (size_t)h.payload || ckpt_bytes(c) != sizeof h + (size_t)h.payload)
    return fail(c, RE_EINVAL, "truncated checkpoint");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  // the launch configuration first: it fixes the cells and the lists' layout
  const unsigned char* in = static_cast<const unsigned char*>(buf);
  std::vector<LaunchCfg> ecfg(c->ens.size());
  std::memcpy(ecfg.data(), in + sizeof h, sizeof(LaunchCfg) * ecfg.size());
  const LaunchCfg old_cfg = c->cfg;
  const std::vector<LaunchCfg> old_ecfg = c->ecfg;
  auto cells = [&]() {
    if (per_class(c))
      apply_cells_each(c);
    else
      apply_cells(c, c->cfg.cell_div);
  };
  c->cfg = h.cfg;
  c->ecfg = ecfg;
  cells();
  int rc = check_cfg(c, h.cfg);
  if (rc == RE_OK && per_class(c)) rc = check_class_cfgs(c);
  if (rc) {
    c->cfg = old_cfg;
    c->ecfg = old_ecfg;
    cells();
    return rc;
  }
  c->resident_clusters = -1;
  rc = upload_tables(c);
  if (rc) return rc;
  if (c->graph) {
    cudaGraphExecDestroy(c->graph);
    c->graph = nullptr;
  }
  if (c->rec_graph) {
    cudaGraphExecDestroy(c->rec_graph);
    c->rec_graph = nullptr;
  }
  fit_notes(c, true);
  size_t off = sizeof h + sizeof(LaunchCfg) * c->ens.size();
  for (const CkptArray& a : ckpt_arrays(c)) {
    if (a.bytes)
      RE_CUDA(c, cudaMemcpy(a.dev, in + off, a.bytes, cudaMemcpyHostToDevice), "checkpoint write");
    off += a.bytes;
  }
  c->since_sort = h.since_sort;
  c->plain_refresh = h.plain_refresh != 0;
  c->list_mode = h.list_mode;
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  return RE_OK;
}

int re_forces(re_ctx* c, double* f) {
  if (!c || !f) return fail(c, RE_EINVAL, "bad arguments");
  int rc = status_check(c);
  if (rc) return rc;
  const cudaError_t e = re::launch_export_state(c->s, c->d_ens, c->d_rep, c->n_rep, nullptr, nullptr,
                                                c->d_io, c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "export");
  RE_CUDA(c, cudaMemcpyAsync(f, c->d_io, 8 * 3 * (size_t)c->n_atoms, cudaMemcpyDeviceToHost,
                             c->stream), "read f");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  return RE_OK;
}

int re_counters(re_ctx* c, int64_t* steps, int64_t* rebuilds) {
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  if (steps)
    RE_CUDA(c, cudaMemcpy(steps, c->s.step, 8 * (size_t)c->n_rep, cudaMemcpyDeviceToHost), "read");
  if (rebuilds)
    RE_CUDA(c, cudaMemcpy(rebuilds, c->s.nreb, 8 * (size_t)c->n_rep, cudaMemcpyDeviceToHost),
            "read");
  return RE_OK;
}

int re_accept_stats(re_ctx* c, int64_t* attempts, int64_t* accepts) {
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  if (c->n_pairs == 0) return RE_OK;
  if (attempts)
    RE_CUDA(c, cudaMemcpy(attempts, c->s.pair_att, 8 * (size_t)c->n_pairs, cudaMemcpyDeviceToHost),
            "read");
  if (accepts)
    RE_CUDA(c, cudaMemcpy(accepts, c->s.pair_acc, 8 * (size_t)c->n_pairs, cudaMemcpyDeviceToHost),
            "read");
  return RE_OK;
}

int re_info(const re_ctx* c, int* n_rep, int64_t* n_atoms, int* n_ens, int* n_pairs) {
  if (!c) return RE_EINVAL;
  if (n_rep) *n_rep = c->n_rep;
  if (n_atoms) *n_atoms = c->n_atoms;
  if (n_ens) *n_ens = (int)c->ens.size();
  if (n_pairs) *n_pairs = c->n_pairs;
  return RE_OK;
}

int re_config_ex(const re_ctx* c, int* cluster, int* threads, int* cell_div, int* atom_threads,
                 int* lists_smem) {
  if (!c) return RE_EINVAL;
  if (lists_smem) *lists_smem = list_elems_for(c, c->cfg) > 0 ? 1 : 0;
  return re_config(c, cluster, threads, cell_div, atom_threads);
}

int re_config_class(const re_ctx* c, int e, int* cluster, int* threads, int* cell_div,
                    int* atom_threads, int* lists_smem) {
  if (!c || e < 0 || e >= (int)c->ens.size() || !per_class(c)) return RE_EINVAL;
  const LaunchCfg& k = c->ecfg[e];
  if (cluster) *cluster = k.cluster;
  if (threads) *threads = k.threads;
  if (cell_div) *cell_div = c->ens[e].m;
  if (atom_threads) *atom_threads = k.atom_threads;
  if (lists_smem) *lists_smem = list_elems_for(c, k, ens_scope(c, e)) > 0 ? 1 : 0;
  return RE_OK;
}

int re_config_wide(const re_ctx* c, int* wide_n, int* wide_cluster, int* wide_threads,
                   int* wide_atom_threads) {
  if (!c) return RE_EINVAL;
  if (wide_n) *wide_n = c->cfg.wide_n;
  if (wide_cluster) *wide_cluster = c->cfg.wide_cluster;
  if (wide_threads) *wide_threads = c->cfg.wide_threads;
  if (wide_atom_threads) *wide_atom_threads = c->cfg.wide_atom_threads;
  return RE_OK;
}

int re_config(const re_ctx* c, int* cluster, int* threads, int* cell_div, int* atom_threads) {
  if (!c) return RE_EINVAL;
  if (cluster) *cluster = c->cfg.cluster;
  if (threads) *threads = c->cfg.threads;
  if (atom_threads) *atom_threads = c->cfg.atom_threads;
  if (cell_div) *cell_div = c->ens.empty() ? 0 : c->ens[0].m;
  return RE_OK;
}

int re_autotune(re_ctx* c, int steps) {
  ApiRange range_("re_autotune");
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  if (c->opt.path != RE_PATH_BATCHED) return RE_OK;
  // launches of as many steps as the caller's, the same for every replica, whose
  // fixed parts (start, lists copied to shared memory, a split launch's ordering)
  // count as they do in use
  steps = std::max(steps, 1);
  const int n_warm = (40 + steps - 1) / steps, n_timed = std::max(2, (120 + steps - 1) / steps);
  int rc = status_check(c);
  if (rc) return rc;
  // snapshot everything a trial run changes
  const size_t A = (size_t)c->n_atoms, R = (size_t)c->n_rep;
  struct Buf {
    void* dev;
    size_t bytes;
    void* save;
  };
  std::vector<Buf> bufs = {
      {c->s.qx, 8 * A}, {c->s.qy, 8 * A}, {c->s.qz, 8 * A}, {c->s.vx, 8 * A},
      {c->s.vy, 8 * A}, {c->s.vz, 8 * A}, {c->s.fx, 8 * A}, {c->s.fy, 8 * A},
      {c->s.fz, 8 * A}, {c->s.U, 8 * R},  {c->s.K, 8 * R},  {c->s.econs, 8 * R},
      {c->s.vscale, 8 * R}, {c->s.fscale, 8 * R}, {c->s.step, 8 * R}, {c->s.nreb, 8 * R},
      {c->s.status, 4 * R}};
  for (auto& b : bufs) {
    b.save = nullptr;
    cudaError_t e = cudaMalloc(&b.save, b.bytes);
    if (e != cudaSuccess) {
      for (auto& q : bufs)
        if (q.save) cudaFree(q.save);
      return cuda_fail(c, e, "autotune snapshot");
    }
    cudaMemcpyAsync(b.save, b.dev, b.bytes, cudaMemcpyDeviceToDevice, c->stream);
  }
  std::vector<int32_t> bud(R, steps);
  c->budget_cached = false;
  RE_CUDA(c, cudaMemcpyAsync(c->d_budget, bud.data(), 4 * R, cudaMemcpyHostToDevice, c->stream),
          "upload");
  // budgets of one step for the untimed list build of every trial
  int32_t* d_one = nullptr;
  {
    const std::vector<int32_t> ones(R, 1);
    RE_CUDA(c, cudaMalloc(&d_one, 4 * R), "autotune budgets");
    RE_CUDA(c, cudaMemcpy(d_one, ones.data(), 4 * R, cudaMemcpyHostToDevice), "autotune budgets");
  }
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  c->tuning = true;
  // One trial: restore the state, build every list of the shape (one step) and
  // run some 40 steps untimed, then time launches of some 120; best of two.
  // run(b) enqueues the launch(es) under test with budgets b.  The untimed steps
  // matter: lists built all at once also wear out together, which hides the
  // wait for the replicas that rebuild more often than others.  (One launch of
  // 40 steps timed right after the builds picked for 64 x 864 a split launch
  // with lists in shared memory, 192 us a cycle of 10 steps; one launch with the
  // lists in global memory takes 180.)  A trial that overflowed or failed
  // stopped early: it is never picked.
  auto trial = [&](auto run) -> float {
    float ms = 1e30f;
    for (int rep = 0; rep < 2; ++rep) {
      for (auto& b : bufs)
        cudaMemcpyAsync(b.dev, b.save, b.bytes, cudaMemcpyDeviceToDevice, c->stream);
      cudaMemsetAsync(c->s.valid, 0, 4 * R, c->stream);
      bool ok = run(d_one) == RE_OK;
      for (int k = 0; k < n_warm + n_timed && ok; ++k) {
        if (k == n_warm) cudaEventRecord(e0, c->stream);
        ok = run(c->d_budget) == RE_OK;
      }
      if (!ok) break;
      cudaEventRecord(e1, c->stream);
      if (cudaEventSynchronize(e1) != cudaSuccess) break;
      float t = 0;
      cudaEventElapsedTime(&t, e0, e1);
      ms = std::min(ms, t);
    }
    cudaGetLastError();
    std::vector<int32_t> st(R);
    cudaMemcpy(st.data(), c->s.status, 4 * R, cudaMemcpyDeviceToHost);
    for (size_t r = 0; r < R; ++r)
      if (st[r]) ms = 1e30f;
    return ms;
  };
  const int clusters[4] = {1, 2, 4, 8};
  const int pvals[4] = {1, 2, 4, 8};
  const LaunchCfg keep = c->cfg;
  LaunchCfg best = keep;
  int best_m = c->opt.cell_div;
  if (per_class(c)) {
    // a group's per-ensemble launches: every class tuned on its own (the
    // others not launched); the uniform shape, used by the free-running
    // modes, stays the default one
    for (size_t ei = 0; ei < c->ens.size(); ++ei) {
      const int e = (int)ei;
      LaunchCfg cbest = c->ecfg[e];
      float cbest_ms = 1e30f;
      // the cells order the atoms and bound the admission, no more: other
      // divisions are tried where the automatic one admits no shape
      for (int m = 0; m <= 3; ++m) {
        if (c->opt.cell_div > 0 && m != c->opt.cell_div) continue;
        if (cbest_ms < 1e30f) break;
        EnsDev& d = c->ens[e];
        int nc = 0, mm = 0;
        choose_cells(d.L, d.rlist, d.N, m, &nc, &mm);
        if (m > 0 && mm != m) continue;
        c->ecfg[e].cell_div = m;
        apply_cells_each(c);
        upload_tables(c);
        const Scope sc = ens_scope(c, e);
        for (int ci = 0; ci < 4; ++ci) {
          if (c->opt.cluster > 0 && clusters[ci] != c->opt.cluster) continue;
          for (int pi = 0; pi < 8; ++pi) {
            const int ls = pi & 1;
            if (c->opt.atom_threads > 0 && pvals[pi / 2] != c->opt.atom_threads) continue;
            if ((c->opt.lists_smem > 0 && ls == 0) || (c->opt.lists_smem < 0 && ls == 1)) continue;
            LaunchCfg k{clusters[ci], threads_for(sc.max_n, clusters[ci], pvals[pi / 2]), m,
                        pvals[pi / 2], ls, 0, 0, 0, 0};
            if ((sc.max_n + k.cluster - 1) / k.cluster < 16) continue;
            if (check_cfg(c, k, sc) != RE_OK) continue;
            if (ls == 1 && list_elems_for(c, k, sc) == 0) continue;
            c->ecfg[e] = k;
            fit_notes(c, false);
            const float ms = trial([&](const int32_t* b) { return launch_class(c, e, b, c->stream); });
            if (ms < cbest_ms) {
              cbest_ms = ms;
              cbest = k;
            }
          }
        }
      }
      c->ecfg[e] = cbest;
      apply_cells_each(c);
      upload_tables(c);
    }
  } else {
    float best_ms = 1e30f;
  for (int m = 0; m <= 3; ++m) {
    if (c->opt.cell_div > 0 && m != c->opt.cell_div) continue;
    if (best_ms < 1e30f) break;  // as above
    apply_cells(c, m);
    if (m > 0) {
      bool any = false;
      for (auto& e : c->ens) any |= (e.m == m);
      if (!any) continue;
    }
    upload_tables(c);
    for (int ci = 0; ci < 4; ++ci) {
      if (c->opt.cluster > 0 && clusters[ci] != c->opt.cluster) continue;
      for (int pi = 0; pi < 8; ++pi) {
        // lists in global memory, then in shared memory (when they fit)
        const int ls = pi & 1;
        if (c->opt.atom_threads > 0 && pvals[pi / 2] != c->opt.atom_threads) continue;
        if ((c->opt.lists_smem > 0 && ls == 0) || (c->opt.lists_smem < 0 && ls == 1)) continue;
        for (int wv = 0; wv < 2; ++wv) {
        // each shape as one launch, then split (hottest replicas on wider clusters)
        LaunchCfg k{clusters[ci], threads_for(c->max_n, clusters[ci], pvals[pi / 2]), m,
                    pvals[pi / 2], ls, 0, 0, 0, 0};
        set_wide(c, k, wv == 1);
        if (wv == 1 && (k.wide_n == 0 || c->opt.wide_launch < 0)) continue;
        if (wv == 0 && c->opt.wide_launch > 0 && (set_wide(c, k, true), k.wide_n > 0)) continue;
        if (wv == 0) set_wide(c, k, false);
        if ((c->max_n + k.cluster - 1) / k.cluster < 16) continue;
        if (check_cfg(c, k) != RE_OK) continue;
        if (ls == 1 && list_elems_for(c, k) == 0) continue;
        c->cfg = k;
        fit_notes(c, false);
        float ms = trial([&](const int32_t* b) { return launch_advance(c, b, nullptr, 1); });
        // the split launch must win clearly: its gain is within the noise of
        // a trial on the workloads measured so far
        if (k.wide_n > 0) ms *= 1.03f;
        if (ms < best_ms) {
          best_ms = ms;
          best = k;
          best_m = m;
        }
        }
      }
    }
  }
  }
  c->cfg = best;
  c->resident_clusters = -1;
  if (per_class(c))
    apply_cells_each(c);
  else
    apply_cells(c, best_m);
  fit_notes(c, true);  // the cached graphs go below
  upload_tables(c);
  for (auto& b : bufs) {
    cudaMemcpyAsync(b.dev, b.save, b.bytes, cudaMemcpyDeviceToDevice, c->stream);
  }
  cudaMemsetAsync(c->s.valid, 0, 4 * R, c->stream);
  cudaStreamSynchronize(c->stream);
  c->tuning = false;
  for (auto& b : bufs) cudaFree(b.save);
  cudaFree(d_one);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (c->graph) {
    cudaGraphExecDestroy(c->graph);
    c->graph = nullptr;
  }
  if (c->rec_graph) {
    cudaGraphExecDestroy(c->rec_graph);
    c->rec_graph = nullptr;
  }
  rc = refresh(c);
  if (rc) return rc;
  return status_check(c);
}

int re_set_stream(re_ctx* c, void* stream) {
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  RE_CUDA(c, cudaStreamSynchronize(c->stream), "synchronise");
  c->stream = static_cast<cudaStream_t>(stream);
  return RE_OK;
}

int re_sync(re_ctx* c) {
  if (!c) return fail(nullptr, RE_EINVAL, "context is NULL");
  return status_check(c);
}

const char* re_last_error(const re_ctx* c) {
  return c ? c->err.c_str() : g_create_error.c_str();
}

void re_destroy(re_ctx* c) {
  if (!c) return;
  cudaStreamSynchronize(c->stream);
  if (c->rec_in) cudaStreamSynchronize(c->rec_in);
  if (c->rec_out) cudaStreamSynchronize(c->rec_out);
  if (c->graph) cudaGraphExecDestroy(c->graph);
  for (void* p : c->allocs) cudaFree(p);
  if (c->h_ring) cudaFreeHost(c->h_ring);
  if (c->side) cudaStreamDestroy(c->side);
  for (cudaStream_t st : c->cls_stream) cudaStreamDestroy(st);
  for (cudaEvent_t ev : c->cls_ev) cudaEventDestroy(ev);
  if (c->ev_fork) cudaEventDestroy(c->ev_fork);
  if (c->ev_join) cudaEventDestroy(c->ev_join);
  if (c->h_out) cudaFreeHost(c->h_out);
  if (c->h_rec) cudaFreeHost(c->h_rec);
  if (c->h_rec_bud) cudaFreeHost(c->h_rec_bud);
  if (c->rec_graph) cudaGraphExecDestroy(c->rec_graph);
  if (c->rec_in) cudaStreamDestroy(c->rec_in);
  if (c->rec_out) cudaStreamDestroy(c->rec_out);
  if (c->ev_in) cudaEventDestroy(c->ev_in);
  if (c->ev_out) cudaEventDestroy(c->ev_out);
  for (int k = 0; k < kRing; ++k)
    if (c->ring_ev[k]) cudaEventDestroy(c->ring_ev[k]);
  delete c;
}

int re_exchange_device(int R, const double* T, const double* U, uint64_t seed, int64_t attempt,
                       int parity_mode, double* T_out, int32_t* partner, uint8_t* accepted,
                       double* vscale, void* stream) {
  g_create_error.clear();
  if (R < 1 || R > 4096) return fail(nullptr, RE_EINVAL, "R must be in [1, 4096]");
  if (!T || !U || !T_out || !partner || !accepted || !vscale)
    return fail(nullptr, RE_EINVAL, "NULL device pointer");
  if (parity_mode != 0 && parity_mode != 1) return fail(nullptr, RE_EINVAL, "parity_mode 0 or 1");
  cudaError_t e = re::launch_exchange_raw(R, T, nullptr, U, seed, attempt, parity_mode, 1, T_out,
                                          nullptr, partner, accepted, vscale, nullptr,
                                          static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "exchange launch");
  return RE_OK;
}

int re_exchange_device_h(int R, const double* T, const double* lam, const double* U,
                         uint64_t seed, int64_t attempt, int parity_mode, int distance,
                         double* T_out, double* lam_out, int32_t* partner, uint8_t* accepted,
                         double* vscale, double* uscale, void* stream) {
  g_create_error.clear();
  if (R < 1 || R > 4096) return fail(nullptr, RE_EINVAL, "R must be in [1, 4096]");
  if (!T || !U || !T_out || !partner || !accepted || !vscale)
    return fail(nullptr, RE_EINVAL, "NULL device pointer");
  if (parity_mode != 0 && parity_mode != 1) return fail(nullptr, RE_EINVAL, "parity_mode 0 or 1");
  if (distance < 1) return fail(nullptr, RE_EINVAL, "distance must be >= 1");
  cudaError_t e = re::launch_exchange_raw(R, T, lam, U, seed, attempt, parity_mode, distance, T_out,
                                          lam_out, partner, accepted, vscale, uscale,
                                          static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "exchange launch");
  return RE_OK;
}

int re_lj_forces_device(int N, double L, double rc, int shift, int precision, const double* x,
                        double* f, double* U, void* stream) {
  g_create_error.clear();
  if (N < 2 || N > 65535) return fail(nullptr, RE_EINVAL, "N must be in [2, 65535]");
  if (!x || !f || !U) return fail(nullptr, RE_EINVAL, "NULL device pointer");
  if (!(L > 0) || !(rc > 0) || rc + 0.5 >= 0.5 * L)
    return fail(nullptr, RE_EINVAL, "need rc + 0.5 < L/2");
  if (precision != RE_PREC_FP64 && precision != RE_PREC_MIXED)
    return fail(nullptr, RE_EINVAL, "unknown precision");
  // the sizes that a one-replica context of this precision takes
  re_ctx c;
  re_default_opts(&c.opt);
  c.opt.precision = precision;
  EnsDev e{};
  e.N = N;
  e.R = 1;
  e.L = L;
  e.rc = rc;
  e.skin = c.opt.skin;
  e.rlist = rc + c.opt.skin;
  e.dt = c.opt.dt;
  e.tau = c.opt.tau_T;
  e.shift = shift ? 1 : 0;
  set_capacity(e, 0);
  finish_ens(e);
  c.ens.push_back(e);
  c.n_rep = c.max_r = 1;
  c.max_n = N;
  apply_cells(&c, 0);
  const LaunchCfg cfg = default_cfg(&c);
  if (check_cfg(&c, cfg) != RE_OK) return fail(nullptr, RE_EINVAL, "%s", c.err.c_str());
  // the neighbours that lists of up to four threads per atom hold
  int p = 4;
  while (p > 1 && threads_for(N, cfg.cluster, p) > 1024) p /= 2;
  const int cap = p * e.capsub[p == 1 ? 0 : (p == 2 ? 1 : 2)];
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaMemPool_t pool = nullptr;
  cudaError_t ce = scratch_pool(&pool);
  if (ce != cudaSuccess) return cuda_fail(nullptr, ce, "scratch pool");
  void* scratch = nullptr;
  ce = cudaMallocFromPoolAsync(&scratch, re::direct_scratch_bytes(N), pool, st);
  if (ce != cudaSuccess) return cuda_fail(nullptr, ce, "scratch");
  int32_t* d_status = nullptr;
  int32_t status = 0;
  ce = re::launch_lj_direct(scratch, N, e.kc, precision == RE_PREC_MIXED, cap, sm_count(), x, f, U,
                            &d_status, st);
  if (ce == cudaSuccess)
    ce = cudaMemcpyAsync(&status, d_status, sizeof status, cudaMemcpyDeviceToHost, st);
  const cudaError_t cf = cudaFreeAsync(scratch, st);
  const cudaError_t cs = cudaStreamSynchronize(st);
  for (cudaError_t k : {ce, cf, cs})
    if (k != cudaSuccess) return cuda_fail(nullptr, k, "forces");
  if (status & re::kStOverflow)
    return fail(nullptr, RE_EOVERFLOW, "neighbour list capacity exceeded (%d per atom)", cap);
  if (status) return fail(nullptr, RE_ENUMERIC, "non-finite energy (overlapping atoms?)");
  return RE_OK;
}

}  // extern "C"

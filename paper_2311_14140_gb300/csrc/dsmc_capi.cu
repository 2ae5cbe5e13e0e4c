// dsmc_capi.cu -- host side of the C ABI declared in include/dsmc.h: argument checks,
// the derived parameters of the method, the device memory layout of a run (one or
// more independent instances), the order of kernel launches within a step, the span
// partition of the step passes and its tuner, CUDA-graph replay, synchronisation,
// the device error word and kernel timing.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "dsmc.h"
#include "dsmc_internal.h"

using namespace dsmc;

namespace {

thread_local std::string g_last_error;

dsmc_status fail(dsmc_status s, const std::string& msg) {
  g_last_error = msg;
  return s;
}

dsmc_status cuda_fail(cudaError_t e, const char* what) {
  g_last_error = std::string(what) + ": " + cudaGetErrorString(e);
  return DSMC_E_CUDA;
}

#define DSMC_CUDA(call, what)                  \
  do {                                         \
    cudaError_t e_ = (call);                   \
    if (e_ != cudaSuccess) return cuda_fail(e_, what); \
  } while (0)

enum KernelId {
  K_INIT = 0,
  K_COLLIDE_MOVE,
  K_SCAN,
  K_OFFSETS,
  K_SCATTER_SPANS,
  K_INDEX_COUNT,
  K_INDEX_SCATTER,
  K_NUM
};
const char* const kKernelNames[K_NUM] = {"init",          "collide_move", "scan_hist",
                                         "cell_offsets",  "scatter_spans", "index_count",
                                         "index_scatter"};

constexpr int kDefaultSpanParticles = 4096;
constexpr int kMinSpanParticles = 1024;
constexpr int kMaxSpanParticles = 1 << 24;
constexpr int kMaxInstances = 65535;  // grid y of the per-instance prefix pass
constexpr int kGraphSteps = 16;       // steps per replay of the captured graph (even)
constexpr long long kTeamParticles = 1500000;  // more never fit the SMs' shared memory
constexpr int kResidentSteps = 512;   // steps per resident launch, at most

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// Spans of the step passes: consecutive cells holding about `target` particles at
// the initial density, at most kMaxSpans spans and kMaxCellsPerSpan cells per span.
// Only the work split depends on the spans: collision groups, random-number counters
// and the sort order do not, so every partition gives the same results.
void make_spans(int n_cells, int ppc, int target, int* cps, int* n_spans) {
  const long long N = (long long)n_cells * ppc;
  long long t = (N + kMaxSpans - 1) / kMaxSpans;
  if (t < target) t = target;
  long long c = (t + ppc - 1) / ppc;
  if (c < (n_cells + kMaxSpans - 1) / kMaxSpans) c = (n_cells + kMaxSpans - 1) / kMaxSpans;
  if (c > kMaxCellsPerSpan) c = kMaxCellsPerSpan;
  if (c > n_cells) c = n_cells;
  if (c < 1) c = 1;
  *cps = (int)c;
  *n_spans = (int)((n_cells + c - 1) / c);
}

// Spans per cell of one run with few, populous cells: a cell is then shared by several CTAs, so
// that the run still makes about kPartSpans spans, of about kPartMin particles or more (16
// collision groups of 256 for a CTA's 8 warps).  us per step, whole cells -> shared: 200 x 50,000 465 ->
// 191, 100 x 25,000 215 -> 79, 20 x 100,000 610 -> 63, 300 x 6,666 89 -> 68, 700 x 25,000 362 ->
// 312.  From about 320 cells on the whole cells of less than 10,000 particles keep most places
// on the SMs busy, and the larger sort matrix and the sums cost more than sharing gives (400 x
// 5,000 101 -> 113 at Kn = 6, 860 x 9,302 175 -> 176).
constexpr int kPartSpans = 900, kPartMin = 4096, kPartCells = 320, kPartLarge = 10000;

int cell_parts(int n_cells, int ppc) {
  if (n_cells > kPartCells && ppc < kPartLarge) return 1;
  const long long N = (long long)n_cells * ppc;
  const long long t = std::max<long long>(kPartMin, N / kPartSpans);
  return (int)std::max<long long>(1, (ppc + t - 1) / t);
}

// Whole cells that fill one wave of 8-warp CTAs, three per SM, to 4/5 or more leave few places
// idle and stay whole: shares of them cost a second and third wave where walls or collisions
// make the groups long (440 x 10,000, whole / shared us per step: Kn = 3 125 / 152, Kn = 6 161 /
// 186, Kn = 0.1 124 / 111; 350 x 10,000: 123 / 125, 151 / 150, 120 / 93; 470 x 10,000, just over
// the wave: 162 / 158, 201 / 194, 128 / 115).
bool fills_wave(int n_cells, int sms) { return n_cells <= 3 * sms && 5 * n_cells >= 12 * sms; }

// Parameters of the method in binary64, rounded once to binary32 where the kernels
// use them.
struct Params {
  double nsig, dt;
  float dt_f, F_f, coef, cvhs, vexp, vinv, lncv, smax0;
};

// n sigma_ref H from Kn through mu0 v0 / (P0 H) = 2 Kn / sqrt(pi) (Eq. 7) and the
// first Chapman-Enskog viscosity of VHS molecules, mu = 15 sqrt(pi m k T) /
// (2 sigma (5 - 2 omega)(7 - 2 omega)) (Bird): n sigma H = 15 sqrt(2) pi /
// (4 (5 - 2 omega)(7 - 2 omega) Kn).  The equilibrium collision frequency is
// nu = n sigma <g>, <g> = 2 sqrt(2) / sqrt(pi).  VHS: sigma g / sigma_ref =
// 2^(omega - 1/2) / Gamma(5/2 - omega) g^(2 - 2 omega) in v0 units, which makes
// <sigma g> = sigma_ref <g> at the wall temperature.
bool derive_params(double omega, double Kn, double F, int ppc, const dsmc_options& o,
                   Params* p) {
  double nsig = 0.0;
  if (!std::isinf(Kn)) {
    const double top = 15.0 * std::sqrt(2.0) * M_PI;
    const double bottom = 4.0 * (5.0 - 2.0 * omega) * (7.0 - 2.0 * omega) * Kn;
    nsig = top / bottom;
  }
  const double mean_g = 2.0 * std::sqrt(2.0) / std::sqrt(M_PI);
  const double nu = nsig * mean_g;
  double dt;
  if (o.dt > 0.0)
    dt = o.dt;
  else if (nu > 0.0)
    dt = o.dt_factor / nu;
  else
    return false;
  const double cv = (omega == 0.5) ? 1.0 : std::pow(2.0, omega - 0.5) / std::tgamma(2.5 - omega);
  p->nsig = nsig;
  p->dt = dt;
  p->dt_f = (float)dt;
  p->F_f = (float)F;
  p->coef = (float)(nsig * dt / (2.0 * (double)ppc));
  p->cvhs = (float)cv;
  p->vexp = (float)(2.0 - 2.0 * omega);
  p->vinv = (omega < 1.0) ? (float)(1.0 / (2.0 - 2.0 * omega)) : 0.0f;
  p->lncv = (float)std::log(cv);
  p->smax0 = (float)(cv * std::pow(5.0, 2.0 - 2.0 * omega));
  return std::isfinite(dt) && dt > 0.0;
}

dsmc_status check_options(const dsmc_options* o) {
  if (!o) return fail(DSMC_E_INVAL, "options: NULL");
  if (!(o->dt_factor > 0.0) || !std::isfinite(o->dt_factor))
    return fail(DSMC_E_INVAL, "options: dt_factor must be finite and > 0");
  if (!(o->dt >= 0.0) || !std::isfinite(o->dt))
    return fail(DSMC_E_INVAL, "options: dt must be finite and >= 0");
  if (o->group_size < 2 || o->group_size > kMaxGroup || (o->group_size & 1))
    return fail(DSMC_E_INVAL, "options: group_size must be even, 2..512");
  if (o->span_particles != 0 &&
      (o->span_particles < kMinSpanParticles || o->span_particles > kMaxSpanParticles))
    return fail(DSMC_E_INVAL, "options: span_particles must be 0 or 1024..2^24");
  if (o->cta_warps != 0 && o->cta_warps != kAWarps && o->cta_warps != kAWarpsSmall)
    return fail(DSMC_E_INVAL, "options: cta_warps must be 0, 4 or 8");
  if (o->span_rows < 0 || o->span_rows > kMaxSpanRows)
    return fail(DSMC_E_INVAL, "options: span_rows must be 0, 1 or 2");
  if (o->graph && o->stream == nullptr)
    return fail(DSMC_E_INVAL, "options: graph replay needs a stream other than the legacy default");
  if (o->accum != DSMC_ACCUM_FP32 && o->accum != DSMC_ACCUM_FP64)
    return fail(DSMC_E_INVAL, "options: accum must be DSMC_ACCUM_FP32 or DSMC_ACCUM_FP64");
  return DSMC_OK;
}

// The options that set the split of the span passes; 0: not named.
struct Split {
  int particles = 0, warps = 0, rows = 0;
};

bool names_partition(const dsmc_options& o) {
  return o.span_particles || o.cta_warps || o.span_rows;
}

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

// First-fit allocator of index ranges [0, capacity) (slots, cells, cell offsets and
// sort-matrix entries of the instances of a handle).
class Extents {
 public:
  void reset(long long capacity) {
    free_.clear();
    if (capacity > 0) free_[0] = capacity;
  }
  long long alloc(long long n) {
    for (auto it = free_.begin(); it != free_.end(); ++it)
      if (it->second >= n) {
        const long long s = it->first, len = it->second;
        free_.erase(it);
        if (len > n) free_[s + n] = len - n;
        return s;
      }
    return -1;
  }
  void release(long long s, long long n) {
    auto it = free_.emplace(s, n).first;
    auto nx = std::next(it);
    if (nx != free_.end() && it->first + it->second == nx->first) {
      it->second += nx->second;
      free_.erase(nx);
    }
    if (it != free_.begin()) {
      auto pv = std::prev(it);
      if (pv->first + pv->second == it->first) {
        pv->second += it->second;
        free_.erase(it);
      }
    }
  }

 private:
  std::map<long long, long long> free_;
};

// One instance of a run: its definition, derived parameters, place in the device
// arrays, span partition and counters.
struct Inst {
  bool active = false;
  bool fresh = false;  // added, not yet initialised on the device
  double omega = 0.5, Kn = 1.0, wall_T = 273.0, F = 0.0;
  int n_cells = 0, ppc = 0;
  long long N = 0;
  uint64_t seed = 0;
  Params p{};
  int max_spans = 0;  // rows of the sort matrix reserved (finest partition)
  long long slot_len = 0;
  int part_base = 0, cell_base = 0, off_base = 0;
  long long hist_base = 0;
  int cps = 0, n_spans = 0, span_base = 0;  // partition in use
  int parts = 1;                            // spans per cell (cps 1)
  long long step = 0, n_samples = 0;
  int open_top = 0;  // y = 1 an open Chapman-Enskog interface
  float u_top = 0.0f, p_top = 0.0f;
  int cut[kResidentMaxCluster + 1] = {};  // slot shares of the CTAs of a resident cluster
};

// Sizes of the device arrays of a handle.
struct Capacity {
  long long slots = 0, hist_ints = 0;
  int cells = 0, offs = 0, spans = 0, inst = 0;
};

// Byte offsets of the arrays in the device workspace.
struct Layout {
  size_t st, hist, count, offset, smax, ncand, nacc, acc, fields, tab, span_inst, chan, err,
      total;
};

long long padded_slots(long long N) { return (N + 63) & ~63LL; }

int reserved_spans(int n_cells, int ppc) {
  int cps, ns;
  make_spans(n_cells, ppc, kMinSpanParticles, &cps, &ns);
  return ns;
}

// Workspace layout for a capacity: two record buffers, the sort matrix, per-cell
// arrays, two instance tables, two span tables (the step's and the admission pass's)
// and the step's span order, the channel sums and the error word.
Layout layout_of(const Capacity& C) {
  Layout L{};
  size_t o = 0;
  L.st = o;
  o += align256(2 * (size_t)C.slots * sizeof(float4));
  L.hist = o;
  o += align256((size_t)C.hist_ints * sizeof(int));
  L.count = o;
  o += align256((size_t)C.cells * sizeof(int));
  L.offset = o;
  o += align256(2 * (size_t)C.offs * sizeof(int));
  L.smax = o;
  o += align256(2 * (size_t)C.cells * sizeof(float));
  L.ncand = o;
  o += align256((size_t)C.cells * sizeof(unsigned long long));
  L.nacc = o;
  o += align256((size_t)C.cells * sizeof(unsigned long long));
  L.acc = o;
  o += align256((size_t)C.cells * kNMom * sizeof(double));
  L.fields = o;
  o += align256((size_t)C.cells * DSMC_NFIELD * sizeof(double));
  L.tab = o;
  o += align256(2 * (size_t)C.inst * sizeof(InstParams));
  L.span_inst = o;
  o += align256(3 * (size_t)C.spans * sizeof(int));
  L.chan = o;
  o += align256(2 * (size_t)C.inst * sizeof(double));
  L.err = o;
  o += 256;
  L.total = o;
  return L;
}

// Ints of the sums of n_cells shared cells: 12 64-bit sums and a maximum each.
long long cell_sums_ints(int n_cells) { return 25LL * n_cells; }

// The rows of the sort matrix reserved for an instance: its finest partition; for one run of its
// own also the partition that shares cells.
int reserved_rows(int n_cells, int ppc, bool alone) {
  const int r = reserved_spans(n_cells, ppc);
  const int parts = alone ? cell_parts(n_cells, ppc) : 1;
  return parts > 1 ? std::max(r, n_cells * parts) : r;
}

// The capacity that holds exactly these instances, placed one after another.
Capacity capacity_of(const dsmc_instance* d, int n) {
  Capacity C{};
  for (int i = 0; i < n; ++i) {
    const long long N = (long long)d[i].n_cells * d[i].ppc;
    const int rows = reserved_rows(d[i].n_cells, d[i].ppc, n == 1);
    C.slots += padded_slots(N);
    C.cells += d[i].n_cells;
    C.offs += d[i].n_cells + 1;
    C.hist_ints += (long long)rows * kMaxSpanRows * d[i].n_cells;
    C.spans += rows;
  }
  C.inst = n;
  // one run: room for the exchange of a team of CTAs (dsmc_resident.cu) in the sort matrix's
  // place, for the sizes whose records the SMs' shared memory holds
  if (n == 1 && C.slots <= kTeamParticles)
    C.hist_ints = std::max<long long>(C.hist_ints,
                                      (long long)team_exchange_ints(kTeamMax, d[0].n_cells));
  // and, behind it all, for the sums of cells that several CTAs share
  if (n == 1 && cell_parts(d[0].n_cells, d[0].ppc) > 1)
    C.hist_ints = ((C.hist_ints + 1) & ~1LL) + cell_sums_ints(d[0].n_cells);
  return C;
}

// The capacity of a pool: every instance of `lim` fits as long as the totals do (up to
// fragmentation of the free ranges).
dsmc_status capacity_of_pool(const dsmc_pool_limits* lim, Capacity* C) {
  if (!lim) return fail(DSMC_E_INVAL, "pool limits: NULL");
  if (lim->max_particles < 1 || lim->max_particles > kMaxParticles || lim->max_cells < 1 ||
      lim->max_instances < 1 || lim->max_instances > kMaxInstances ||
      lim->max_cells_per_instance < 1 || lim->max_cells_per_instance > kMaxStepCells ||
      lim->max_cells_per_instance > lim->max_cells)
    return fail(DSMC_E_INVAL,
                "pool limits: max_particles 1..2^31 - 2^24, max_instances 1..65535, "
                "1 <= max_cells_per_instance <= min(16384, max_cells)");
  Capacity c{};
  c.slots = lim->max_particles;
  c.cells = lim->max_cells;
  c.offs = lim->max_cells + lim->max_instances;
  c.inst = lim->max_instances;
  // An instance of N particles reserves at most N / 1024 + 1 sort-matrix rows.
  const long long rows = lim->max_particles / kMinSpanParticles + lim->max_instances;
  c.spans = (int)std::min<long long>(rows, INT_MAX / 2);
  c.hist_ints = rows * kMaxSpanRows * (long long)lim->max_cells_per_instance;
  *C = c;
  return DSMC_OK;
}

// Checks one instance definition; the message names the instance in a batch.
dsmc_status check_instance(const dsmc_instance& d, int index, int n_inst) {
  const std::string at = n_inst > 1 ? "instance " + std::to_string(index) + ": " : "";
  if (!(d.gas.mass > 0.0) || !(d.gas.d_ref > 0.0) || !(d.gas.T_ref > 0.0))
    return fail(DSMC_E_INVAL, at + "gas: mass, d_ref and T_ref must be > 0");
  if (!(d.gas.omega >= 0.5 && d.gas.omega <= 1.0))
    return fail(DSMC_E_INVAL, at + "gas: omega must lie in [0.5, 1]");
  if (!(d.Kn > 0.0)) return fail(DSMC_E_INVAL, at + "Kn must be > 0 (or +inf)");
  if (!(d.wall_T > 0.0) || !std::isfinite(d.wall_T))
    return fail(DSMC_E_INVAL, at + "wall_T must be > 0");
  if (!std::isfinite(d.body_force)) return fail(DSMC_E_INVAL, at + "body_force must be finite");
  if (d.n_cells < 1 || d.ppc < 1) return fail(DSMC_E_INVAL, at + "n_cells and ppc must be >= 1");
  if ((long long)d.n_cells * d.ppc > kMaxParticles)
    return fail(DSMC_E_INVAL, at + "n_cells * ppc must be <= 2^31 - 2^24");
  if (d.n_cells > kMaxStepCells) return fail(DSMC_E_INVAL, at + "n_cells must be <= 16384");
  return DSMC_OK;
}

int collision_mode(double omega) { return omega == 0.5 ? 0 : (omega == 1.0 ? 2 : 1); }

}  // namespace

void dsmc::set_last_error(const std::string& msg) { g_last_error = msg; }

struct dsmc_sim {
  int device = 0;
  int sms = 1;  // of the device
  bool pool = false;  // instances may be added and removed
  dsmc_options opt{};
  std::vector<Inst> inst;  // by id
  std::vector<int> order;  // active ids in table order
  long long gstep = 0;     // steps this handle has launched
  int span_target = kDefaultSpanParticles;
  // The split of the span passes follows the instances (choose_split) until the options or the
  // tuner name one; instances were added or removed since it was made.
  bool auto_split = true, split_dirty = false;
  bool split_shared = false;  // choose_split's choice for a device shared with other runs
  // The split dsmc_autotune chose: options that give it back (as a caller does who changes
  // another option) name nothing by themselves.
  Split tuned;
  int check_warps = kAWarps;  // warps per CTA that instances' sizes are checked against
  int cta_warps = kAWarps;  // warps per CTA of the collide/move pass
  int span_rows = 1;        // sort-matrix rows per span
  int spans = 0, max_cps = 1, max_cells = 1, max_spans = 1;  // partition in use
  long long part_total = 0;  // particles of the active instances
  int spans_reserved = 0;
  Capacity C{};
  Layout L{};
  Extents ex_slots, ex_cells, ex_offs, ex_hist;
  void* ws = nullptr;
  bool owns = false;
  float4* P[2]{};  // particle records (y, vx, vy, vz), double-buffered for the sort
  int cur = 0;
  int *hist = nullptr, *count = nullptr, *err = nullptr;
  int* off[2]{};
  int ocur = 0;
  float* smax[2]{};
  int scur = 0;
  unsigned long long *ncand = nullptr, *nacc = nullptr;
  double* acc = nullptr;
  double* fields = nullptr;  // dsmc_cell_fields_of's output on the device
  InstParams* tab_dev = nullptr;  // [0, C.inst): the step's; [C.inst, 2 C.inst): admission
  int* span_inst_dev = nullptr;   // likewise with C.spans entries each, then the order
  int* span_order_dev = nullptr;  // the span each collide/move CTA takes (C.spans entries)
  double* chan_dev = nullptr;
  std::vector<InstParams> tab, adm_tab;
  std::vector<int> span_inst, adm_span, span_order;
  bool tab_dirty = true, spans_dirty = true;
  // Cluster-resident steps (dsmc_resident.cu): the launch's shape, or cl = 0 when the
  // handle's steps take the span passes.
  ResidentLaunch res{};
  bool res_dirty = true;
  bool span_passes = false;  // the caller's options name a partition, or it is being tuned
  int last_kind = DSMC_STEP_NONE, last_ctas = 0;  // of the latest steps
  // Behind the latest steps of a run on a team, and their stream (TeamRuns; under its lock).
  cudaEvent_t stepped = nullptr;
  void* stepped_stream = nullptr;
  // CUDA graph of kGraphSteps consecutive steps, replayed by dsmc_step when
  // options.graph is set.  Its kernels read the global step from gstep_dev, which the
  // kernel that forms the cell offsets advances.
  cudaGraphExec_t graph = nullptr;
  bool graph_valid = false, capturing = false;
  int graph_parity = 0;  // buffer parities (cur, ocur, scur) the graph starts from
  long long* gstep_dev = nullptr;
  unsigned* barrier = nullptr;  // of a team's CTAs: count and generation
  dsmc_status latched = DSMC_OK;
  std::vector<cudaEvent_t> events;
  std::vector<int> event_kernel;
  size_t events_used = 0;
  double ktime[K_NUM] = {};
  long long kcount[K_NUM] = {};

  cudaStream_t stream() const { return (cudaStream_t)opt.stream; }
  int n_inst() const { return (int)order.size(); }
  int cap() const { return opt.group_size + opt.group_size / 2 - 1; }
};

namespace {

// Kernel timing: an event pair around a launch when profiling.
cudaError_t mark(dsmc_sim* h, int kernel) {
  if (!h->opt.profile) return cudaSuccess;
  if (h->events_used + 1 >= h->events.size()) {
    for (int i = 0; i < 64; ++i) {
      cudaEvent_t e;
      cudaError_t r = cudaEventCreate(&e);
      if (r != cudaSuccess) return r;
      h->events.push_back(e);
      h->event_kernel.push_back(-1);
    }
  }
  h->event_kernel[h->events_used] = kernel;
  return cudaEventRecord(h->events[h->events_used++], h->stream());
}

template <typename Launch>
cudaError_t timed(dsmc_sim* h, int kernel, Launch&& launch) {
  cudaError_t e = mark(h, kernel);
  if (e != cudaSuccess) return e;
  e = launch();
  if (e != cudaSuccess) return e;
  return mark(h, -1);
}

dsmc_status collect_times(dsmc_sim* h) {
  if (h->events_used == 0) return DSMC_OK;
  DSMC_CUDA(cudaStreamSynchronize(h->stream()), "profile sync");
  for (size_t i = 0; i + 1 < h->events_used; i += 2) {
    float ms = 0.0f;
    DSMC_CUDA(cudaEventElapsedTime(&ms, h->events[i], h->events[i + 1]), "event time");
    const int k = h->event_kernel[i];
    if (k >= 0 && k < K_NUM) {
      h->ktime[k] += ms;
      h->kcount[k] += 1;
    }
  }
  h->events_used = 0;
  return DSMC_OK;
}

// The step passes must fit one CTA's shared memory with this partition, group size and
// CTA shape.
bool step_fits(int max_cells, int max_cps, int G, int warps = kAWarps, int rows = 1) {
  return step_smem_layout(max_cells, max_cps, G + G / 2 - 1, warps, rows, false).total <=
         kStepSmemMax;
}

// The largest cells-per-span any active instance (and `extra`, if given) would use
// with `target` particles per span, and the largest cell count.
void partition_extent(const dsmc_sim* h, int target, const Inst* extra, int* max_cps,
                      int* max_cells) {
  int m = 1, mc = 1;
  auto visit = [&](const Inst& x) {
    int cps, ns;
    make_spans(x.n_cells, x.ppc, target, &cps, &ns);
    m = std::max(m, cps);
    mc = std::max(mc, x.n_cells);
  };
  for (int id : h->order) visit(h->inst[id]);
  if (extra) visit(*extra);
  *max_cps = m;
  *max_cells = mc;
}

// Launch order of the collide/move CTAs: the spans by estimated cost, heaviest first, so
// that the pass does not end on a few slow CTAs started last (the spans at the top wall of
// a run started in cell order ran about twice as long as the rest and left most SMs idle
// for the last sixth of the pass).  A span's cost is taken as its particles times
// (1 + 2.2 h), h the expected wall hits per particle and step: with normal velocity
// components of variance 1/2 (v0 units), a particle at distance d from a wall reaches it
// within dt with probability erfc(d / dt) / 2, evaluated at the span's centre for both
// walls; 2.2 is the measured extra cost of a hit relative to a particle's other work in the
// step (a batch at Kn = 10, about one hit per particle and step, costs 3.2 times one at
// Kn = 0.1).  The order changes which CTA takes a span, never a result.
void set_span_order(dsmc_sim* h) {
  std::vector<std::pair<double, int>> cost;
  cost.reserve((size_t)h->spans);
  for (int t = 0; t < h->n_inst(); ++t) {
    const Inst& x = h->inst[h->order[t]];
    const double dt = x.p.dt;
    for (int k = 0; k < x.n_spans; ++k) {
      const int c0 = k / x.parts * x.cps, c1 = std::min(c0 + x.cps, x.n_cells);
      const double yc = 0.5 * (c0 + c1) / x.n_cells;
      const double hits = dt > 0.0 ? 0.5 * (std::erfc(yc / dt) + std::erfc((1.0 - yc) / dt)) : 0.0;
      cost.emplace_back(-(double)(c1 - c0) * x.ppc / x.parts * (1.0 + 2.2 * hits),
                        x.span_base + k);
    }
  }
  std::stable_sort(cost.begin(), cost.end(),
                   [](const std::pair<double, int>& a, const std::pair<double, int>& b) {
                     return a.first < b.first;
                   });
  h->span_order.resize(cost.size());
  for (size_t i = 0; i < cost.size(); ++i) h->span_order[i] = cost[i].second;
}

// Assigns spans with `target` particles per span to every active instance.
void set_partition(dsmc_sim* h, int target) {
  h->span_target = target;
  h->span_inst.clear();
  int base = 0, m = 1, mc = 1, ms = 1;
  long long np = 0;
  for (int t = 0; t < h->n_inst(); ++t) {
    Inst& x = h->inst[h->order[t]];
    np += x.N;
    make_spans(x.n_cells, x.ppc, target, &x.cps, &x.n_spans);
    x.parts = h->auto_split && !h->split_shared && !h->pool && h->C.inst == 1 &&
                      !fills_wave(x.n_cells, h->sms)
                  ? cell_parts(x.n_cells, x.ppc)
                  : 1;
    if (x.parts > 1) {
      x.cps = 1;
      x.n_spans = x.n_cells * x.parts;
    }
    x.span_base = base;
    base += x.n_spans;
    m = std::max(m, x.cps);
    mc = std::max(mc, x.n_cells);
    ms = std::max(ms, x.n_spans);
    h->span_inst.insert(h->span_inst.end(), (size_t)x.n_spans, t);
  }
  h->spans = base;
  h->max_cps = m;
  h->max_cells = mc;
  h->max_spans = ms;
  h->part_total = np;
  set_span_order(h);
  h->tab_dirty = h->spans_dirty = h->res_dirty = true;
  h->graph_valid = false;
}

int default_span_particles(long long n);

// Warps per CTA and particles per span for the active instances of a batch or pool, by their
// particles (us per step of batches of uneven instances; in brackets the former 4-warp CTAs of
// 4,096 particles, then 8-warp CTAs of 4,096 / 6,144 and 4-warp CTAs of 4,096 / 5,120 where they
// lose): below 27,000 particles per SM 8-warp CTAs (fewer, larger CTAs leave fewer SMs idle behind
// the last spans) with spans of 1,024 to 4,096 particles, about one per place on the SMs (1.2
// million 68 [80], 2.8 million 115 [119], 3.6 million 142 [150; 4-warp 157]); from there 4-warp
// CTAs of 4,096 (4.4 million 154 [167; 8-warp 162 / 161],
// 5.2 million 176 [194; 8-warp 188 / 185]), from 40,000 per SM on 5,120 (6.3 million 209 [232;
// 4,096 215], 8.5 million 270 [316]), from 120,000 per SM on 8,192 (24 million 657 [692]).
void choose_split(dsmc_sim* h) {
  if (!h->pool && h->n_inst() <= 1) {
    if (h->n_inst() == 1) {
      const Inst& x = h->inst[h->order[0]];
      long long target;
      if (h->split_shared) {
        // steps beside those of other runs: fewer, larger spans than one run needs to fill the SMs
        // cost least in all (8 runs of 397 x 2,531: 397 spans 27.6 us per step and run, 199 17.7)
        target = default_span_particles(x.N);
      } else if (x.n_cells > kCoopCells) {
        // a scatter with a warp per span wants about 6.6 of them per SM (3,000 x 500: 334 spans
        // 106 us per step, 1,000 spans 64); beyond 4,096 particles whole cells up to 6,144 (4,000
        // x 1,500: 1,334 spans 196, 1,000 spans 185), but no cell more (1,600 x 5,000: 1,600
        // spans 182, 800 spans 199)
        const long long t = x.N / (33LL * h->sms / 5);
        const long long k = std::max((std::min<long long>(4096, t) + x.ppc - 1) / x.ppc,
                                     std::min<long long>(6144, t) / x.ppc);
        target = k * x.ppc;
        // more than two and less than three spans per SM are a second wave of few CTAs (so many
        // cells' histograms leave room for two per SM): the default's two then (3,500 x 113: 292
        // spans 45 us per step, 350 spans 49; 3,996 x 200: 286 spans 65, 666 spans 59)
        const long long c = std::max<long long>(k, kMinSpanParticles / x.ppc);
        const long long spans = x.n_cells / std::max<long long>(1, c);
        if (spans >= 2LL * h->sms && spans < 3LL * h->sms) target = default_span_particles(x.N);
      } else {
        // whole cells: the fewest per span whose spans fit 1.2 waves of 8-warp CTAs, three per
        // SM, and no more than the default's particles need; the few CTAs behind a full wave have
        // the SMs to themselves and cost little, half a wave more does not (us per step at Kn 2,
        // cells per span 1 / 2 / 3: 500 x 3,500 71 / 85 / 113, 1,000 x 3,000 111 / 105 / 112,
        // 800 x 3,000 95 / 83 / 99, 700 x 2,000 68 / 68 / 78; 1,300 x 2,000 107 / 108 / 88)
        const long long most =
            std::max<long long>(1, (default_span_particles(x.N) + x.ppc - 1) / x.ppc);
        long long k = 1;
        while (k < most && 5 * ((x.n_cells + k - 1) / k) > 18LL * h->sms) ++k;
        target = k * x.ppc;
      }
      h->span_target = (int)std::min<long long>(kMaxSpanParticles,
                                                std::max<long long>(kMinSpanParticles, target));
    }
    return;
  }
  long long n = 0;
  for (int id : h->order) n += h->inst[id].N;
  int warps = kAWarps;
  long long target =
      std::min<long long>(4096, std::max<long long>(kMinSpanParticles, 2 * n / (7LL * h->sms)));
  if (n >= 27000LL * h->sms) {
    warps = kAWarpsSmall;
    target = n >= 120000LL * h->sms ? 8192 : n >= 40000LL * h->sms ? 5120 : 4096;
  }
  int mcps, mcells;
  partition_extent(h, (int)target, nullptr, &mcps, &mcells);
  if (!step_fits(mcells, mcps, h->opt.group_size, warps, h->span_rows)) warps = kAWarpsSmall;
  h->cta_warps = warps;
  h->span_target = (int)target;
}

// Brings the partition up to date with the active instances.
void ensure_partition(dsmc_sim* h) {
  if (!h->split_dirty) return;
  h->split_dirty = false;
  if (h->auto_split) choose_split(h);
  set_partition(h, h->span_target);
}

InstParams instance_params(const dsmc_sim* h, int id, int span_base) {
  const Inst& x = h->inst[id];
  InstParams a{};
  a.n_cells = x.n_cells;
  a.cell_base = x.cell_base;
  a.off_base = x.off_base;
  a.span_base = span_base;
  a.n_spans = x.n_spans;
  a.cps = x.cps;
  a.parts = x.parts;
  a.part_base = x.part_base;
  a.n_part = (int)x.N;
  a.hist_base = x.hist_base;
  a.G = h->opt.group_size;
  a.cap = h->cap();
  a.ncf = (float)x.n_cells;
  a.dt = x.p.dt_f;
  a.F = x.p.F_f;
  a.coef = x.p.coef;
  a.cvhs = x.p.cvhs;
  a.vexp = x.p.vexp;
  a.vinv = x.p.vinv;
  a.lncv = x.p.lncv;
  a.lg2cv = (float)std::log2((double)x.p.cvhs);
  a.k0 = (uint32_t)(x.seed & 0xffffffffu);
  a.k1 = (uint32_t)(x.seed >> 32);
  for (int r = 0; r < 10; ++r) {
    a.keys.k0[r] = a.k0 + (uint32_t)r * 0x9E3779B9u;
    a.keys.k1[r] = a.k1 + (uint32_t)r * 0xBB67AE85u;
  }
  a.step0 = h->gstep - x.step;  // the instance's step = global step - step0
  a.sample_start = h->opt.sample_start;
  a.collide = (h->opt.collisions != 0 && x.p.nsig > 0.0) ? 1 : 0;
  a.mode = collision_mode(x.omega);
  a.id = id;
  a.smax0 = x.p.smax0;
  a.open_top = x.open_top;
  a.u_top = x.u_top;
  a.p_top = x.p_top;
  std::copy(x.cut, x.cut + kResidentMaxCluster + 1, a.cut);
  return a;
}

// Rebuilds the instance table after a change and, for a batch, enqueues its copy to
// the device (ordered on the stream before the next launch).  The copies read
// pageable host memory, which CUDA stages before the call returns.
dsmc_status upload_tables(dsmc_sim* h) {
  ensure_partition(h);
  if (h->tab_dirty) {
    h->tab.resize(h->order.size());
    for (int t = 0; t < h->n_inst(); ++t)
      h->tab[t] = instance_params(h, h->order[t], h->inst[h->order[t]].span_base);
    if (!h->tab.empty())
      DSMC_CUDA(cudaMemcpyAsync(h->tab_dev, h->tab.data(), h->tab.size() * sizeof(InstParams),
                                cudaMemcpyHostToDevice, h->stream()),
                "instance table");
    h->tab_dirty = false;
    if (h->n_inst() == 1) h->graph_valid = false;  // the captured launches hold tab[0]
  }
  if (h->spans_dirty) {
    if (!h->span_inst.empty())
      DSMC_CUDA(cudaMemcpyAsync(h->span_inst_dev, h->span_inst.data(),
                                h->span_inst.size() * sizeof(int), cudaMemcpyHostToDevice,
                                h->stream()),
                "span table");
    if (!h->span_order.empty())
      DSMC_CUDA(cudaMemcpyAsync(h->span_order_dev, h->span_order.data(),
                                h->span_order.size() * sizeof(int), cudaMemcpyHostToDevice,
                                h->stream()),
                "span order");
    h->spans_dirty = false;
  }
  return DSMC_OK;
}

StepLaunch step_launch(const dsmc_sim* h, bool count_only) {
  StepLaunch L{};
  L.n_inst = h->n_inst();
  L.tab = h->tab_dev;
  L.span_inst = h->span_inst_dev;
  L.span_order = h->span_order.empty() ? nullptr : h->span_order_dev;
  L.n_spans_total = h->spans;
  L.max_cells = h->max_cells;
  L.max_spans = h->max_spans;
  L.n_part_total = h->part_total;
  L.max_cps = h->max_cps;
  L.max_cap = h->cap();
  L.warps = h->cta_warps;
  L.rows = h->span_rows;
  L.gstep = h->gstep;
  L.gstep_dev = h->capturing ? h->gstep_dev : nullptr;
  L.count_only = count_only ? 1 : 0;
  L.accum = h->opt.accum;
  return L;
}

// The launches of one pass over the records from buffer `src` to buffer src ^ 1:
// collide + sample + move + count (or count only), prefix over spans, cell offsets and
// stable scatter.
dsmc_status launch_pass(dsmc_sim* h, bool count_only, const StepLaunch& SL,
                        const InstParams& one, int src, int osrc) {
  cudaStream_t s = h->stream();
  int* off_cur = h->off[osrc];
  int* off_new = h->off[osrc ^ 1];
  CellSums sums{};
  if (one.parts > 1) {
    sums.off = off_cur;
    sums.smax_in = h->smax[h->scur];
    sums.smax_out = h->smax[h->scur ^ 1];
    sums.acc = h->acc;
    sums.fix = (unsigned long long*)(h->hist + h->C.hist_ints - cell_sums_ints(one.n_cells));
    sums.gmax = (unsigned*)(sums.fix + (size_t)one.n_cells * 12);
  }
  DSMC_CUDA(timed(h, count_only ? K_INDEX_COUNT : K_COLLIDE_MOVE, [&] {
              return launch_collide_move(h->P[src], off_cur, h->smax[h->scur],
                                         h->smax[h->scur ^ 1], h->ncand, h->nacc, h->acc,
                                         h->hist, sums, one, SL, h->err, s);
            }),
            count_only ? "index_count" : "collide_move");
  DSMC_CUDA(timed(h, K_SCAN, [&] { return launch_scan_spans(h->hist, h->count, sums, one, SL, s); }),
            "scan_hist");
  if (!scatter_forms_offsets(SL))
    DSMC_CUDA(timed(h, K_OFFSETS,
                    [&] { return launch_offsets_cells(h->count, off_new, one, SL, s); }),
              "cell_offsets");
  DSMC_CUDA(timed(h, count_only ? K_INDEX_SCATTER : K_SCATTER_SPANS, [&] {
              return launch_scatter_spans(h->P[src], h->P[src ^ 1], off_cur, h->count, off_new,
                                          h->hist, one, SL, h->err, s);
            }),
            count_only ? "index_scatter" : "scatter_spans");
  return DSMC_OK;
}

// One pass over every active instance from the current buffers to the other ones.
dsmc_status run_pass(dsmc_sim* h, bool count_only) {
  if (h->n_inst() == 0) return DSMC_OK;
  const StepLaunch SL = step_launch(h, count_only);
  dsmc_status s = launch_pass(h, count_only, SL, h->tab[0], h->cur, h->ocur);
  if (s != DSMC_OK) return s;
  if (!count_only) h->scur ^= 1;
  h->cur ^= 1;
  h->ocur ^= 1;
  return DSMC_OK;
}

// Sort into cells without moving (state load).  The current offsets must describe
// slot ranges per cell span; records may be in any order within them.
dsmc_status run_index(dsmc_sim* h) {
  dsmc_status s = upload_tables(h);
  if (s != DSMC_OK) return s;
  return run_pass(h, /*count_only=*/true);
}

// Device initialisation of the instances added since the last step: particles drawn
// into the idle record buffer with offsets of whole cells, per-cell arrays reset, then
// a sort into cells of those instances alone into the current buffers (the other
// instances are not touched).
dsmc_status admit_fresh(dsmc_sim* h) {
  ensure_partition(h);
  std::vector<int> ids;
  for (int id : h->order)
    if (h->inst[id].fresh) ids.push_back(id);
  if (ids.empty()) return DSMC_OK;
  cudaStream_t s = h->stream();
  const int idle = h->cur ^ 1, oidle = h->ocur ^ 1;
  h->adm_tab.clear();
  h->adm_span.clear();
  int base = 0, m = 1, mc = 1, ms = 1;
  long long np = 0;
  for (size_t k = 0; k < ids.size(); ++k) {
    const Inst& x = h->inst[ids[k]];
    np += x.N;
    h->adm_tab.push_back(instance_params(h, ids[k], base));
    h->adm_span.insert(h->adm_span.end(), (size_t)x.n_spans, (int)k);
    base += x.n_spans;
    m = std::max(m, x.cps);
    mc = std::max(mc, x.n_cells);
    ms = std::max(ms, x.n_spans);
    DSMC_CUDA(timed(h, K_INIT, [&] {
                return launch_init(h->P[idle] + x.part_base, (int)x.N, x.ppc, (float)x.n_cells,
                                   (uint32_t)(x.seed & 0xffffffffu), (uint32_t)(x.seed >> 32),
                                   h->err, s);
              }),
              "init");
  }
  InstParams* adm_tab_dev = h->tab_dev + h->C.inst;
  int* adm_span_dev = h->span_inst_dev + h->C.spans;
  DSMC_CUDA(cudaMemcpyAsync(adm_tab_dev, h->adm_tab.data(), h->adm_tab.size() * sizeof(InstParams),
                            cudaMemcpyHostToDevice, s),
            "admission table");
  DSMC_CUDA(cudaMemcpyAsync(adm_span_dev, h->adm_span.data(), h->adm_span.size() * sizeof(int),
                            cudaMemcpyHostToDevice, s),
            "admission span table");
  DSMC_CUDA(launch_admit_cells(adm_tab_dev, (int)ids.size(), h->off[oidle], h->smax[h->scur],
                               h->ncand, h->nacc, h->acc, s),
            "admit cells");
  if (h->adm_tab[0].parts > 1) {
    const long long n = cell_sums_ints(h->adm_tab[0].n_cells);
    DSMC_CUDA(cudaMemsetAsync(h->hist + h->C.hist_ints - n, 0, n * sizeof(int), s), "cell sums");
  }
  StepLaunch SL{};
  SL.n_inst = (int)ids.size();
  SL.tab = adm_tab_dev;
  SL.span_inst = adm_span_dev;
  SL.n_spans_total = base;
  SL.max_cells = mc;
  SL.max_spans = ms;
  SL.n_part_total = np;
  SL.max_cps = m;
  SL.max_cap = h->cap();
  SL.warps = h->cta_warps;
  SL.rows = h->span_rows;
  SL.gstep = h->gstep;
  SL.gstep_dev = nullptr;
  SL.count_only = 1;
  dsmc_status st = launch_pass(h, true, SL, h->adm_tab[0], idle, oidle);
  if (st != DSMC_OK) return st;
  for (int id : ids) h->inst[id].fresh = false;
  return DSMC_OK;
}

// Advances every active instance's counters for n steps.
void count_steps(dsmc_sim* h, int n) {
  h->gstep += n;
  for (int id : h->order) {
    Inst& x = h->inst[id];
    const long long from = std::max(x.step + 1, h->opt.sample_start);  // first sampled step
    x.step += n;
    x.n_samples += std::max(0LL, x.step - from + 1);
  }
}

// Slot ranges for a sort of instance id's records in arbitrary order: cell span k
// covers [off[k cps], off[(k+1) cps]) with off[c] = part_base + floor(c N / n_cells).
dsmc_status set_uniform_offsets(dsmc_sim* h, int id, std::vector<int>& host) {
  const Inst& x = h->inst[id];
  host.resize((size_t)x.n_cells + 1);
  for (int c = 0; c <= x.n_cells; ++c)
    host[c] = x.part_base + (int)((long long)c * x.N / x.n_cells);
  DSMC_CUDA(cudaMemcpyAsync(h->off[h->ocur] + x.off_base, host.data(), host.size() * sizeof(int),
                            cudaMemcpyHostToDevice, h->stream()),
            "offsets");
  return DSMC_OK;
}

// The status of the device error word v.
dsmc_status check_error_word(dsmc_sim* h, int v) {
  if (v != 0) {
    h->latched = DSMC_E_DEVICE_LIMIT;
    std::string what;
    if (v & kErrNormals) what += " gaussian-attempts";
    if (v & kErrBounces) what += " wall-bounces";
    if (v & kErrSphere) what += " scattering-attempts";
    if (v & kErrCandidates) what += " candidate-count";
    if (v & kErrSort) what += " sort-destination";
    if (v & kErrCopyTimeout) what += " bulk-copy-timeout";
    if (v & kErrInflow) what += " inflow-attempts";
    if (v & kErrMoments) what += " moment-range";
    if (v & kErrTeam) what += " team-barrier-timeout";
    return fail(DSMC_E_DEVICE_LIMIT, "device limit reached:" + what);
  }
  return DSMC_OK;
}

dsmc_status read_error_word(dsmc_sim* h) {
  int v = 0;
  DSMC_CUDA(cudaMemcpyAsync(&v, h->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream()),
            "read error word");
  DSMC_CUDA(cudaStreamSynchronize(h->stream()), "stream sync");
  return check_error_word(h, v);
}

// The address at which this device's kernels can access all of the caller's `bytes` at p: device
// memory of this device or pinned host memory, aligned for binary32; NULL for anything else
// (pageable, managed, another device's, shorter than `bytes`), which is copied instead.
void* direct_pointer(const void* p, size_t bytes, int device) {
  if ((uintptr_t)p & 3u) return nullptr;
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  const bool here = at.type == cudaMemoryTypeDevice && at.device == device;
  if ((!here && at.type != cudaMemoryTypeHost) || !at.devicePointer) return nullptr;
  // the allocation's extent
  using GetAttribute = CUresult (*)(void*, CUpointer_attribute, CUdeviceptr);
  static const GetAttribute get = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuPointerGetAttribute", &f, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      f = nullptr;
    }
    return (GetAttribute)f;
  }();
  CUdeviceptr start = 0;
  size_t size = 0;
  const CUdeviceptr d = (CUdeviceptr)at.devicePointer;
  if (!get || get(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, d) != CUDA_SUCCESS ||
      get(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, d) != CUDA_SUCCESS)
    return nullptr;
  return d >= start && bytes <= size && d - start <= size - bytes ? at.devicePointer : nullptr;
}

// The same for four arrays of n floats (NULL entries stay NULL); false when one of them cannot
// be accessed so or two overlap.
bool direct_arrays(void* const* p, size_t n, int device, float** out) {
  const size_t bytes = n * sizeof(float);
  for (int k = 0; k < 4; ++k) {
    out[k] = nullptr;
    if (!p[k]) continue;
    out[k] = (float*)direct_pointer(p[k], bytes, device);
    if (!out[k]) return false;
    for (int j = 0; j < k; ++j)
      if (out[j] && (uintptr_t)out[j] < (uintptr_t)out[k] + bytes &&
          (uintptr_t)out[k] < (uintptr_t)out[j] + bytes)
        return false;
  }
  return true;
}

dsmc_status check_handle(dsmc_sim* h) {
  if (!h) return fail(DSMC_E_INVAL, "handle: NULL");
  return DSMC_OK;
}

dsmc_status check_index(dsmc_sim* h, int id) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  if (id < 0 || id >= (int)h->inst.size() || !h->inst[id].active)
    return fail(DSMC_E_INVAL, "instance index out of range or not active");
  return DSMC_OK;
}

void drop_graph(dsmc_sim* h) {
  if (h->graph) cudaGraphExecDestroy(h->graph);
  h->graph = nullptr;
  h->graph_valid = false;
}

int parity(const dsmc_sim* h) { return h->cur | (h->ocur << 1) | (h->scur << 2); }

// Captures the launches of kGraphSteps steps into a graph.  Capture only records:
// the host-side buffer parities are restored afterwards (an even step count returns
// them to the same values after each replay).
dsmc_status capture_graph(dsmc_sim* h) {
  cudaStream_t s = h->stream();
  const int c0 = h->cur, o0 = h->ocur, s0 = h->scur;
  cudaGraph_t g = nullptr;
  DSMC_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal), "begin capture");
  h->capturing = true;
  dsmc_status st = DSMC_OK;
  for (int k = 0; k < kGraphSteps && st == DSMC_OK; ++k) st = run_pass(h, false);
  h->capturing = false;
  const cudaError_t e_end = cudaStreamEndCapture(s, &g);
  h->cur = c0;
  h->ocur = o0;
  h->scur = s0;
  if (st != DSMC_OK || e_end != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
    return st != DSMC_OK ? st : cuda_fail(e_end, "stream capture");
  }
  drop_graph(h);
  const cudaError_t e = cudaGraphInstantiate(&h->graph, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return cuda_fail(e, "graph instantiate");
  h->graph_parity = parity(h);
  h->graph_valid = true;
  return DSMC_OK;
}

dsmc_status step_once(dsmc_sim* h) {
  count_steps(h, 1);
  dsmc_status s = upload_tables(h);
  if (s != DSMC_OK) return s;
  return run_pass(h, false);
}

// Shares of an instance's slots for the cl CTAs of its cluster or team, of about equal cost: a
// particle at y costs 1 + 1.5 h(y), h its expected wall hits in the step (as in
// set_span_order; 1.5 is the measured extra cost of a hit here, where a CTA's wall hits are
// flown by all its warps).  With equal shares the CTAs next to the walls took 64,000 cycles
// of a 67,000-cycle step of a 100,000-particle run and the others 46,000 (Kn = 0.5); with
// these, 49,000 and 45,000 of 52,000.  The cost's integral is taken at 256 points and
// inverted linearly.  Returns the largest share.
int set_cuts(const Inst& x, int cl, int* cut) {
  constexpr int kPoints = 256;
  const double dt = x.p.dt, w = 1.5;
  auto ierfc = [&](double y) {  // integral of erfc(t / dt) over [0, y]
    const double u = y / dt;
    return y * std::erfc(u) + dt * (1.0 - std::exp(-u * u)) / std::sqrt(M_PI);
  };
  const double whole = ierfc(1.0);
  double cost[kPoints + 1];
  for (int i = 0; i <= kPoints; ++i) {
    const double y = (double)i / kPoints;
    cost[i] = y + 0.5 * w * (ierfc(y) + whole - ierfc(1.0 - y));
  }
  int share = 0, i = 0;
  cut[0] = 0;
  for (int r = 1; r <= cl; ++r) {
    const double target = cost[kPoints] * r / cl;
    while (i < kPoints - 1 && cost[i + 1] < target) ++i;
    const double y = (i + (target - cost[i]) / (cost[i + 1] - cost[i])) / kPoints;
    const long long at = r == cl ? x.N : (long long)(y * (double)x.N);
    cut[r] = (int)std::min(x.N, std::max<long long>(cut[r - 1], at));
    share = std::max(share, cut[r] - cut[r - 1]);
  }
  return share;
}

constexpr long long kClusterParticles = 40000;
constexpr int kResidentShare = 2600;

// Fills in a resident launch's sizes; false when it does not fit the device.
bool size_resident(dsmc_sim* h, ResidentLaunch& R) {
  const dsmc_options& o = h->opt;
  long long n_max = 0;
  for (int id : h->order) n_max = std::max(n_max, h->inst[id].N);
  if (n_max / R.cl > 30000) return false;  // local slots are 16-bit; so large a share never fits
  R.max_cells = h->max_cells;
  if (R.team && team_exchange_ints(R.cl, R.max_cells) > (size_t)h->C.hist_ints) return false;
  int share = 0;
  for (int id : h->order)
    share = std::max(share, set_cuts(h->inst[id], R.cl, R.team ? R.cut : h->inst[id].cut));
  R.range_cap = share + h->cap();
  R.list_cap = R.range_cap / o.group_size + std::min(R.max_cells, R.range_cap) + 2;
  R.own_cap = (R.max_cells + R.cl - 1) / R.cl;
  const size_t smem = resident_smem_layout(R.max_cells, R.range_cap, R.list_cap, R.own_cap,
                                           R.team ? 0 : R.cl, resident_local(R),
                                           resident_warps(R.n_inst > 1))
                          .total;
  if (smem > kResidentSmemMax) return false;
  bool fits = false;
  if (resident_fits(R, smem, o.accum == DSMC_ACCUM_FP64, &fits) == cudaSuccess && fits)
    return true;
  cudaGetLastError();
  return false;
}

// The runs of this process whose steps go to a team.  A team has the whole device to itself, so
// teams of several streams run one after the other where span passes overlap (us per step and run,
// one after the other / span passes: 200 x 500 on 2 streams 14.0 / 14.4, 3 14.1 / 9.7, 8 13.9 / 4.0;
// 300 x 1,000 on 2 16.5 / 22, 3 16.5 / 15.4, 8 16.4 / 7.1; 397 x 2,531 on 3 27.6 / 28, 4 27.7 / 22).
// While the steps of kTeamOthers other runs, on other streams, are in flight, a call's steps take
// the span passes.  Runs mark their steps with an event only while there are that many of them.
constexpr int kTeamOthers = 2;

struct TeamRuns {
  std::mutex lock;
  std::vector<dsmc_sim*> runs;
  std::atomic<int> size{0};
};

TeamRuns& team_runs() {
  static TeamRuns* const t = new TeamRuns;  // (handles may be destroyed after static objects)
  return *t;
}

// Event calls are not allowed while another thread captures a stream in global mode, unless this
// thread says that they do not concern it.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

void leave_team_runs(dsmc_sim* h) {
  TeamRuns& t = team_runs();
  std::lock_guard<std::mutex> hold(t.lock);
  t.runs.erase(std::remove(t.runs.begin(), t.runs.end(), h), t.runs.end());
  t.size = (int)t.runs.size();
}

void join_team_runs(dsmc_sim* h) {
  TeamRuns& t = team_runs();
  std::lock_guard<std::mutex> hold(t.lock);
  if (std::find(t.runs.begin(), t.runs.end(), h) == t.runs.end()) t.runs.push_back(h);
  t.size = (int)t.runs.size();
}

// Whether events may bear on this handle's steps: enough other runs, and no capture of its stream.
bool team_runs_watched(dsmc_sim* h) {
  if (team_runs().size <= kTeamOthers) return false;
  cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(h->stream(), &c) == cudaSuccess) return c == cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return false;
}

// Whether the device is to be shared: kTeamOthers other runs have steps in flight.
bool team_runs_crowded(dsmc_sim* h) {
  TeamRuns& t = team_runs();
  RelaxedCapture relaxed;
  std::lock_guard<std::mutex> hold(t.lock);
  int n = 0;
  for (dsmc_sim* x : t.runs) {
    if (x == h || x->device != h->device || !x->stepped || x->stepped_stream == h->opt.stream)
      continue;
    if (cudaEventQuery(x->stepped) == cudaErrorNotReady) ++n;
    cudaGetLastError();
    if (n >= kTeamOthers) return true;
  }
  return false;
}

// Marks the steps enqueued so far (best effort: a missing mark only leaves the choice as it was).
// The record is made without the lock: it waits where the stream's queue of launches is full.
void mark_team_steps(dsmc_sim* h) {
  RelaxedCapture relaxed;
  if (!h->stepped || h->stepped_stream != h->opt.stream) {
    cudaEvent_t e = h->stepped;
    if (!e && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    std::lock_guard<std::mutex> hold(team_runs().lock);
    h->stepped = e;
    h->stepped_stream = h->opt.stream;
  }
  if (cudaEventRecord(h->stepped, h->stream()) != cudaSuccess) cudaGetLastError();
}

// The split of a run of its own beside other runs, or alone.  (The plan of resident steps does
// not depend on it.)
void use_shared_split(dsmc_sim* h, bool shared) {
  if (!h->auto_split || h->split_shared == shared) return;
  h->split_shared = shared;
  h->split_dirty = true;
  ensure_partition(h);
  h->res_dirty = false;
}

// Decides whether the handle's steps run resident (dsmc_resident.cu) and with how many CTAs
// per instance.  Options that name a partition of the span passes keep those, as does
// profiling, which times their kernels; a pool's members come and go between calls.
//
// One run: a cluster of 16 CTAs up to kClusterParticles (us per step, cluster / team of 152 /
// span passes under graph replay: 2,250 particles 7.0 / 10.7 / 20.5, 20,000 11.4 / 13.0 / 22.5,
// 40,000 13.8 / 13.0 / 23, 80,000 23.1 / 14.9 / 27), from there a team of a CTA per SM (more
// CTAs were never slower: 100,000 particles 18.4 with 32, 15.2 with 64, 13.7 with 152), as long
// as its share fits a CTA's shared memory (1,004,807 particles 27.7 against 71; up to about
// 1,300,000, depending on the cells).
// A batch: clusters of as many CTAs per instance as give shares of at most kResidentShare
// particles and fill the SMs twice, as long as an instance then fits 16 CTAs and the launch is
// not many waves long (64 x 2,250 particles: 11 us per step against 30; 64 x 10,000: 28 / 48;
// 64 x 20,000: 45 / 70; 128 x 20,000, 1,024 CTAs: 87 / 95; beyond that the span passes,
// which spread every instance over all SMs, are as fast: 256 x 20,000, 161 / 153;
// 24 x 100,000, 137 / 85).
void find_resident(dsmc_sim* h) {
  if (h->pool || h->opt.profile || h->span_passes) return;
  long long n_max = 0;
  for (int id : h->order) n_max = std::max(n_max, h->inst[id].N);
  ResidentLaunch R{};
  R.n_inst = h->n_inst();
  R.cl = kResidentMaxCluster;
  bool fits = false;
  if (R.n_inst == 1) {
    ResidentLaunch T{};
    T.n_inst = 1;
    T.cl = std::min(h->sms, kTeamMax);
    T.team = 1;
    if (n_max <= kClusterParticles) fits = size_resident(h, R);
    if (!fits && size_resident(h, T)) {
      R = T;
      fits = true;
    }
  } else {
    R.cl = 2;
    while (R.cl < kResidentMaxCluster &&
           (n_max > (long long)kResidentShare * R.cl || R.n_inst * 2 * R.cl <= 2 * h->sms))
      R.cl *= 2;
    fits = n_max <= (long long)kResidentShare * R.cl &&
           (long long)R.n_inst * R.cl <= (R.cl == 16 ? 512 : 1024) && size_resident(h, R);
  }
  if (!fits) return;
  if (R.n_inst > 1) {
    // The launch's clusters start in table order: the costliest instances first, so that the
    // launch does not end on them (64 runs of 20,000 particles at Kn 0.1 to 5: 44.3 -> 41.3 us per
    // step).  An instance's cost is its particles times 1 + 1.5 of their expected wall hits,
    // about 0.28 dt per particle at each wall.
    auto cost = [&](int id) { return h->inst[id].N * (1.0 + 0.85 * h->inst[id].p.dt); };
    std::stable_sort(h->order.begin(), h->order.end(),
                     [&](int x, int y) { return cost(x) > cost(y); });
    set_partition(h, h->span_target);  // places in the table have changed
  }
  h->res = R;
  h->tab_dirty = true;  // the instance table carries the cuts
}

void plan_resident(dsmc_sim* h) {
  ensure_partition(h);
  if (h->res.team) leave_team_runs(h);
  h->res = ResidentLaunch{};
  find_resident(h);
  if (h->res.team)
    join_team_runs(h);
  else
    use_shared_split(h, false);
  h->res_dirty = false;
}

// n steps of a resident launch.  Where the launch is refused (a stream that has only some of the
// SMs, for which the plan's queries do not ask), nothing has run: the handle's steps take the span
// passes from then on (res.cl = 0).
dsmc_status step_resident(dsmc_sim* h, int n) {
  ResidentLaunch R = h->res;
  R.tab = h->tab_dev;
  R.n_steps = n;
  R.gstep = h->gstep + 1;
  R.parity_rec = h->cur;
  R.parity_off = h->ocur;
  R.parity_smax = h->scur;
  const cudaError_t e =
      launch_resident(h->P[0], h->P[1], h->off[0], h->off[1], h->smax[0], h->smax[1], h->ncand,
                      h->nacc, h->acc, h->hist, h->barrier, h->tab[0], R,
                      h->opt.accum == DSMC_ACCUM_FP64, h->err, h->stream());
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources ||
      e == cudaErrorInvalidConfiguration || e == cudaErrorInvalidClusterSize ||
      e == cudaErrorNotSupported) {
    cudaGetLastError();
    if (R.team) leave_team_runs(h);
    h->res = ResidentLaunch{};
    return DSMC_OK;
  }
  DSMC_CUDA(e, "resident steps");
  h->cur ^= n & 1;
  h->ocur ^= n & 1;
  h->scur ^= n & 1;
  count_steps(h, n);
  h->last_kind = R.team ? DSMC_STEP_TEAM : DSMC_STEP_CLUSTERS;
  h->last_ctas = R.cl;
  return DSMC_OK;
}

dsmc_status step_n(dsmc_sim* h, int n_steps) {
  dsmc_status s;
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  int it = 0;
  bool watched = false;
  if (h->n_inst() > 0 && n_steps > 0) {
    if (h->res_dirty || h->split_dirty) plan_resident(h);
    watched = h->res.team && team_runs_watched(h);
    const bool crowded = watched && team_runs_crowded(h);
    if (crowded) use_shared_split(h, true);
    if (h->res.cl > 0 && !crowded) {
      if ((s = upload_tables(h)) != DSMC_OK) return s;
      while (it < n_steps && h->res.cl > 0) {
        const int n = std::min(n_steps - it, kResidentSteps);
        if ((s = step_resident(h, n)) != DSMC_OK) return s;
        if (h->res.cl > 0) it += n;
      }
      if (it == n_steps) {
        if (watched) mark_team_steps(h);
        return DSMC_OK;
      }
    }
    h->last_kind = DSMC_STEP_SPANS;
    h->last_ctas = 0;
  }
  if (h->opt.graph && !h->opt.profile && h->n_inst() > 0) {
    while (n_steps - it >= kGraphSteps) {
      if ((s = upload_tables(h)) != DSMC_OK) return s;
      if (!h->graph_valid || h->graph_parity != parity(h))
        if ((s = capture_graph(h)) != DSMC_OK) return s;
      // The graph's first step runs at global step gstep + 1.
      DSMC_CUDA(launch_set_counter(h->gstep_dev, h->gstep + 1, h->stream()), "set step");
      DSMC_CUDA(cudaGraphLaunch(h->graph, h->stream()), "graph launch");
      count_steps(h, kGraphSteps);
      it += kGraphSteps;
    }
  }
  for (; it < n_steps; ++it)
    if ((s = step_once(h)) != DSMC_OK) return s;
  if (watched) mark_team_steps(h);
  return DSMC_OK;
}

// Adds an instance (extents, parameters, counters); its device data is set up by the
// next step or synchronising call.  *id gets its id.
dsmc_status add_instance(dsmc_sim* h, const dsmc_instance& d, int index, int n_def, int* id) {
  dsmc_status st = check_instance(d, index, n_def);
  if (st != DSMC_OK) return st;
  Inst x;
  x.omega = d.gas.omega;
  x.Kn = d.Kn;
  x.wall_T = d.wall_T;
  x.F = d.body_force;
  x.n_cells = d.n_cells;
  x.ppc = d.ppc;
  x.N = (long long)d.n_cells * d.ppc;
  x.seed = d.seed;
  if (!derive_params(x.omega, x.Kn, x.F, x.ppc, h->opt, &x.p))
    return fail(DSMC_E_INVAL, (n_def > 1 ? "instance " + std::to_string(index) + ": " : "") +
                                  "time step undefined: set options.dt for infinite Kn");
  int mcps, mcells;
  partition_extent(h, h->span_target, &x, &mcps, &mcells);
  if (!step_fits(mcells, mcps, h->opt.group_size, h->check_warps, h->span_rows))
    return fail(DSMC_E_INVAL, "n_cells and group_size exceed the step's shared memory");
  // Find a free id and room in every array.
  int new_id = -1;
  for (int i = 0; i < (int)h->inst.size(); ++i)
    if (!h->inst[i].active) {
      new_id = i;
      break;
    }
  if (new_id < 0 && (int)h->inst.size() >= h->C.inst)
    return fail(DSMC_E_NOMEM, "no room: instance table full");
  x.max_spans = reserved_rows(x.n_cells, x.ppc, !h->pool && h->C.inst == 1);
  if (h->spans_reserved + x.max_spans > h->C.spans)
    return fail(DSMC_E_NOMEM, "no room: span table full");
  x.slot_len = padded_slots(x.N);
  const long long ps = h->ex_slots.alloc(x.slot_len);
  const long long cb = ps < 0 ? -1 : h->ex_cells.alloc(x.n_cells);
  const long long ob = cb < 0 ? -1 : h->ex_offs.alloc(x.n_cells + 1);
  const long long hb =
      ob < 0 ? -1 : h->ex_hist.alloc((long long)x.max_spans * kMaxSpanRows * x.n_cells);
  if (hb < 0) {
    if (ob >= 0) h->ex_offs.release(ob, x.n_cells + 1);
    if (cb >= 0) h->ex_cells.release(cb, x.n_cells);
    if (ps >= 0) h->ex_slots.release(ps, x.slot_len);
    return fail(DSMC_E_NOMEM, "no room: device memory of the handle is taken");
  }
  x.part_base = (int)ps;
  x.cell_base = (int)cb;
  x.off_base = (int)ob;
  x.hist_base = hb;
  x.active = true;
  x.fresh = true;
  if (new_id < 0) {
    new_id = (int)h->inst.size();
    h->inst.push_back(x);
  } else {
    h->inst[new_id] = x;
  }
  h->order.push_back(new_id);
  h->spans_reserved += x.max_spans;
  h->split_dirty = true;
  *id = new_id;
  return DSMC_OK;
}

// Default particles per span for a handle of n particles: 4,096, or fewer for a small run
// so that its step passes still spread over two CTAs per SM (a 20,000-particle run: 17
// spans of 1,024 particles instead of 5 of 4,096), never below the finest partition its
// sort matrix is sized for.
int default_span_particles(long long n) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      sms < 1)
    sms = 152;
  const long long t = n / (2LL * sms);
  return (int)std::max<long long>(kMinSpanParticles,
                                  std::min<long long>(kDefaultSpanParticles, t));
}

// Allocates the handle and its device workspace for capacity C.
dsmc_status new_handle(const Capacity& C, const dsmc_options& opt, bool pool, void* workspace,
                       size_t workspace_bytes, dsmc_sim** out) {
  dsmc_sim* h = new (std::nothrow) dsmc_sim();
  if (!h) return fail(DSMC_E_NOMEM, "host allocation failed");
  h->pool = pool;
  h->opt = opt;
  h->C = C;
  h->L = layout_of(C);
  h->span_target = opt.span_particles ? opt.span_particles : default_span_particles(C.slots);
  h->cta_warps = opt.cta_warps ? opt.cta_warps : (pool ? kAWarpsSmall : kAWarps);
  h->check_warps = h->cta_warps;
  h->auto_split = !opt.span_particles && !opt.cta_warps;
  h->span_rows = opt.span_rows ? opt.span_rows : 1;
  h->span_passes = names_partition(opt);
  h->ex_slots.reset(C.slots);
  h->ex_cells.reset(C.cells);
  h->ex_offs.reset(C.offs);
  h->ex_hist.reset(C.hist_ints);
  cudaError_t ce = cudaGetDevice(&h->device);
  if (ce == cudaSuccess)
    ce = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, h->device);
  if (ce != cudaSuccess) {
    delete h;
    return cuda_fail(ce, "cudaGetDevice");
  }
  if (workspace) {
    if (workspace_bytes < h->L.total || ((uintptr_t)workspace & 255u)) {
      delete h;
      return fail(DSMC_E_NOMEM, "workspace smaller than the workspace size or not 256-byte aligned");
    }
    h->ws = workspace;
    h->owns = false;
  } else {
    ce = cudaMalloc(&h->ws, h->L.total);
    if (ce != cudaSuccess) {
      delete h;
      cudaGetLastError();
      return fail(DSMC_E_NOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(ce));
    }
    h->owns = true;
  }
  const Layout& L = h->L;
  char* b = (char*)h->ws;
  h->P[0] = (float4*)(b + L.st);
  h->P[1] = h->P[0] + C.slots;
  h->hist = (int*)(b + L.hist);
  h->count = (int*)(b + L.count);
  h->off[0] = (int*)(b + L.offset);
  h->off[1] = h->off[0] + C.offs;
  h->smax[0] = (float*)(b + L.smax);
  h->smax[1] = h->smax[0] + C.cells;
  h->ncand = (unsigned long long*)(b + L.ncand);
  h->nacc = (unsigned long long*)(b + L.nacc);
  h->acc = (double*)(b + L.acc);
  h->fields = (double*)(b + L.fields);
  h->tab_dev = (InstParams*)(b + L.tab);
  h->span_inst_dev = (int*)(b + L.span_inst);
  h->span_order_dev = h->span_inst_dev + 2 * (size_t)h->C.spans;
  h->chan_dev = (double*)(b + L.chan);
  h->err = (int*)(b + L.err);
  h->gstep_dev = (long long*)(b + L.err + 8);
  h->barrier = (unsigned*)(b + L.err + 128);
  ce = set_step_smem_limits(kStepSmemMax, kStepSmemMax);
  if (ce == cudaSuccess) ce = cudaMemsetAsync(h->err, 0, 256, h->stream());
  if (ce != cudaSuccess) {
    dsmc_status s = cuda_fail(ce, "handle setup");
    dsmc_destroy(h);
    return s;
  }
  *out = h;
  return DSMC_OK;
}

// Sets up fresh instances on the device and checks for errors (synchronises).
dsmc_status settle(dsmc_sim* h) {
  dsmc_status st = admit_fresh(h);
  if (st != DSMC_OK) return st;
  st = collect_times(h);
  if (st != DSMC_OK) return st;
  return read_error_word(h);
}

dsmc_status create_run(const dsmc_instance* defs, int n_inst, const dsmc_options* opt_in,
                       void* workspace, size_t workspace_bytes, dsmc_handle* out) {
  if (!out) return fail(DSMC_E_INVAL, "out: NULL");
  *out = nullptr;
  if (!defs) return fail(DSMC_E_INVAL, "instances: NULL");
  if (n_inst < 1 || n_inst > kMaxInstances)
    return fail(DSMC_E_INVAL, "n_instances must be 1..65535");
  dsmc_options opt;
  dsmc_default_options(&opt);
  if (opt_in) opt = *opt_in;
  dsmc_status st = check_options(&opt);
  if (st != DSMC_OK) return st;
  for (int i = 0; i < n_inst; ++i)
    if ((st = check_instance(defs[i], i, n_inst)) != DSMC_OK) return st;
  long long slots = 0;
  for (int i = 0; i < n_inst; ++i) slots += padded_slots((long long)defs[i].n_cells * defs[i].ppc);
  if (slots > kMaxParticles)
    return fail(DSMC_E_INVAL, "the instances' particles (each padded to 64) must total <= 2^31 - 2^24");
  // Parameters and shared-memory fit before any device work.
  {
    int mcps = 1, mcells = 1;
    const int target = opt.span_particles ? opt.span_particles : kDefaultSpanParticles;
    for (int i = 0; i < n_inst; ++i) {
      Params p;
      if (!derive_params(defs[i].gas.omega, defs[i].Kn, defs[i].body_force, defs[i].ppc, opt, &p))
        return fail(DSMC_E_INVAL, (n_inst > 1 ? "instance " + std::to_string(i) + ": " : "") +
                                      "time step undefined: set options.dt for infinite Kn");
      int cps, ns;
      make_spans(defs[i].n_cells, defs[i].ppc, target, &cps, &ns);
      mcps = std::max(mcps, cps);
      mcells = std::max(mcells, defs[i].n_cells);
    }
    if (!step_fits(mcells, mcps, opt.group_size, opt.cta_warps ? opt.cta_warps : kAWarps,
                   opt.span_rows ? opt.span_rows : 1))
      return fail(DSMC_E_INVAL, "n_cells and group_size exceed the step's shared memory");
  }
  dsmc_sim* h = nullptr;
  st = new_handle(capacity_of(defs, n_inst), opt, false, workspace, workspace_bytes, &h);
  if (st != DSMC_OK) return st;
  for (int i = 0; i < n_inst; ++i) {
    int id = -1;
    st = add_instance(h, defs[i], i, n_inst, &id);
    if (st != DSMC_OK) {
      dsmc_destroy(h);
      return st;
    }
  }
  st = settle(h);
  if (st != DSMC_OK) {
    dsmc_destroy(h);
    return st;
  }
  *out = h;
  return DSMC_OK;
}

dsmc_instance make_instance(const dsmc_gas* gas, double Kn, double wall_T, double body_force,
                            int n_cells, int ppc, uint64_t seed) {
  dsmc_instance d{};
  if (gas) d.gas = *gas;
  d.Kn = Kn;
  d.wall_T = wall_T;
  d.body_force = body_force;
  d.n_cells = n_cells;
  d.ppc = ppc;
  d.seed = seed;
  return d;
}

}  // namespace

extern "C" {

dsmc_status dsmc_default_options(dsmc_options* opt) {
  if (!opt) return fail(DSMC_E_INVAL, "options: NULL");
  std::memset(opt, 0, sizeof(*opt));
  opt->dt_factor = 0.2;
  opt->dt = 0.0;
  opt->sample_start = 0;
  opt->group_size = 256;
  opt->collisions = 1;
  opt->profile = 0;
  opt->span_particles = 0;
  opt->cta_warps = 0;
  opt->span_rows = 0;
  opt->graph = 0;
  opt->accum = DSMC_ACCUM_FP32;
  opt->stream = nullptr;
  return DSMC_OK;
}

size_t dsmc_batch_workspace_bytes(const dsmc_instance* inst, int n_inst) {
  if (!inst || n_inst < 1 || n_inst > kMaxInstances) return 0;
  for (int i = 0; i < n_inst; ++i)
    if (inst[i].n_cells < 1 || inst[i].ppc < 1 || inst[i].n_cells > kMaxStepCells) return 0;
  return layout_of(capacity_of(inst, n_inst)).total;
}

size_t dsmc_workspace_bytes(int n_cells, int ppc) {
  dsmc_instance d{};
  d.n_cells = n_cells;
  d.ppc = ppc;
  return dsmc_batch_workspace_bytes(&d, 1);
}

size_t dsmc_pool_workspace_bytes(const dsmc_pool_limits* limits) {
  Capacity C;
  const std::string saved = g_last_error;
  if (capacity_of_pool(limits, &C) != DSMC_OK) {
    g_last_error = saved;
    return 0;
  }
  return layout_of(C).total;
}

dsmc_status dsmc_create_in(const dsmc_gas* gas, double Kn, double wall_T, double body_force,
                           int n_cells, int ppc, uint64_t seed, const dsmc_options* opt_in,
                           void* workspace, size_t workspace_bytes, dsmc_handle* out) {
  if (!out) return fail(DSMC_E_INVAL, "out: NULL");
  *out = nullptr;
  if (!gas) return fail(DSMC_E_INVAL, "gas: NULL");
  const dsmc_instance d = make_instance(gas, Kn, wall_T, body_force, n_cells, ppc, seed);
  return create_run(&d, 1, opt_in, workspace, workspace_bytes, out);
}

dsmc_status dsmc_create(const dsmc_gas* gas, double Kn, double wall_T, double body_force,
                        int n_cells, int ppc, uint64_t seed, dsmc_handle* out) {
  return dsmc_create_in(gas, Kn, wall_T, body_force, n_cells, ppc, seed, nullptr, nullptr, 0,
                        out);
}

dsmc_status dsmc_create_batch(const dsmc_instance* inst, int n_inst, const dsmc_options* opt,
                              void* workspace, size_t workspace_bytes, dsmc_handle* out) {
  return create_run(inst, n_inst, opt, workspace, workspace_bytes, out);
}

dsmc_status dsmc_pool_create(const dsmc_pool_limits* limits, const dsmc_options* opt_in,
                             void* workspace, size_t workspace_bytes, dsmc_handle* out) {
  if (!out) return fail(DSMC_E_INVAL, "out: NULL");
  *out = nullptr;
  Capacity C;
  dsmc_status st = capacity_of_pool(limits, &C);
  if (st != DSMC_OK) return st;
  dsmc_options opt;
  dsmc_default_options(&opt);
  if (opt_in) opt = *opt_in;
  if ((st = check_options(&opt)) != DSMC_OK) return st;
  dsmc_sim* h = nullptr;
  st = new_handle(C, opt, true, workspace, workspace_bytes, &h);
  if (st != DSMC_OK) return st;
  *out = h;
  return DSMC_OK;
}

dsmc_status dsmc_pool_add(dsmc_handle h, const dsmc_instance* inst, int* id) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  if (!inst || !id) return fail(DSMC_E_INVAL, "instance and id must not be NULL");
  if (!h->pool) return fail(DSMC_E_STATE, "dsmc_pool_add needs a handle from dsmc_pool_create");
  *id = -1;
  return add_instance(h, *inst, 0, 1, id);
}

dsmc_status dsmc_pool_remove(dsmc_handle h, int id) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  if (!h->pool) return fail(DSMC_E_STATE, "dsmc_pool_remove needs a handle from dsmc_pool_create");
  Inst& x = h->inst[id];
  // Work already enqueued on the stream still reads these ranges; anything that reuses
  // them is enqueued after it.
  h->ex_slots.release(x.part_base, x.slot_len);
  h->ex_cells.release(x.cell_base, x.n_cells);
  h->ex_offs.release(x.off_base, x.n_cells + 1);
  h->ex_hist.release(x.hist_base, (long long)x.max_spans * kMaxSpanRows * x.n_cells);
  h->spans_reserved -= x.max_spans;
  x.active = false;
  x.fresh = false;
  h->order.erase(std::find(h->order.begin(), h->order.end(), id));
  h->split_dirty = true;
  return DSMC_OK;
}

dsmc_status dsmc_channel_sums(dsmc_handle h, double* out) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  if (!out) return fail(DSMC_E_INVAL, "out: NULL");
  DeviceGuard guard(h->device);
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  if ((s = upload_tables(h)) != DSMC_OK) return s;
  const size_t n_ids = h->inst.size();
  if (h->n_inst() > 0)
    DSMC_CUDA(launch_channel_sums(h->tab_dev, h->n_inst(), h->acc, h->chan_dev, h->stream()),
              "channel sums");
  if (n_ids > 0)
    DSMC_CUDA(cudaMemcpyAsync(out, h->chan_dev, 2 * n_ids * sizeof(double), cudaMemcpyDefault,
                              h->stream()),
              "copy channel sums");
  s = dsmc_sync(h);
  if (s != DSMC_OK) return s;
  for (size_t i = 0; i < n_ids; ++i)
    if (!h->inst[i].active) out[2 * i] = out[2 * i + 1] = 0.0;
  return DSMC_OK;
}

dsmc_status dsmc_device_moments_of(dsmc_handle h, int id, const double** acc) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  if (!acc) return fail(DSMC_E_INVAL, "acc: NULL");
  DeviceGuard guard(h->device);
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  *acc = h->acc + (size_t)h->inst[id].cell_base * kNMom;
  return DSMC_OK;
}

dsmc_status dsmc_set_open_top(dsmc_handle h, int id, double u, double P) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  if (!std::isfinite(u) || !std::isfinite(P) || std::fabs(P) > 0.25)
    return fail(DSMC_E_INVAL, "open boundary: finite u and |P| <= 0.25");
  Inst& x = h->inst[id];
  x.open_top = 1;
  x.u_top = (float)u;
  x.p_top = (float)P;
  h->tab_dirty = true;
  return DSMC_OK;
}

int dsmc_batch_size(dsmc_handle h) { return h ? h->n_inst() : 0; }

int dsmc_id_bound(dsmc_handle h) { return h ? (int)h->inst.size() : 0; }

dsmc_status dsmc_set_options(dsmc_handle h, const dsmc_options* opt) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  s = check_options(opt);
  if (s != DSMC_OK) return s;
  std::vector<Params> ps(h->inst.size());
  for (int id : h->order) {
    const Inst& x = h->inst[id];
    if (!derive_params(x.omega, x.Kn, x.F, x.ppc, *opt, &ps[id]))
      return fail(DSMC_E_INVAL, "time step undefined: set options.dt for infinite Kn");
  }
  // 0 keeps the value in use, and so does the tuner's.
  ensure_partition(h);
  const Split& tuned = h->tuned;
  const bool new_particles = opt->span_particles && opt->span_particles != tuned.particles;
  const bool new_warps = opt->cta_warps && opt->cta_warps != tuned.warps;
  const bool named = new_particles || new_warps ||
                     (opt->span_rows && opt->span_rows != tuned.rows);
  const bool auto_split = h->auto_split && !new_particles && !new_warps;
  const int target_use = opt->span_particles ? opt->span_particles : h->span_target;
  const int warps_use = opt->cta_warps ? opt->cta_warps
                                       : (auto_split ? h->check_warps : h->cta_warps);
  const int rows_use = opt->span_rows ? opt->span_rows : h->span_rows;
  int mcps, mcells;
  partition_extent(h, target_use, nullptr, &mcps, &mcells);
  if (!step_fits(mcells, mcps, opt->group_size, warps_use, rows_use))
    return fail(DSMC_E_INVAL, "n_cells and group_size exceed the step's shared memory");
  if (h->events_used) {
    s = collect_times(h);
    if (s != DSMC_OK) return s;
  }
  h->opt = *opt;
  if (named) {
    h->span_passes = true;
    h->tuned = Split{};
  } else if (!names_partition(*opt)) {
    h->span_passes = false;
  }
  for (int id : h->order) h->inst[id].p = ps[id];
  const bool was_auto = h->auto_split;
  h->auto_split = auto_split;
  if (opt->cta_warps && !auto_split) h->check_warps = warps_use;
  h->span_rows = rows_use;
  if (auto_split) {
    h->split_dirty = true;  // the group size bears on the choice
  } else {
    h->cta_warps = warps_use;
    if (was_auto || target_use != h->span_target) set_partition(h, target_use);
  }
  h->tab_dirty = h->res_dirty = true;
  drop_graph(h);  // launch shapes or the stream may have changed
  return DSMC_OK;
}

dsmc_status dsmc_step(dsmc_handle h, int n_steps) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  if (n_steps < 0) return fail(DSMC_E_INVAL, "n_steps must be >= 0");
  if (h->latched != DSMC_OK) return fail(h->latched, "an earlier step reached a device limit");
  DeviceGuard guard(h->device);
  s = step_n(h, n_steps);
  if (s != DSMC_OK) return s;
  if (h->opt.profile) return collect_times(h);
  return DSMC_OK;
}

dsmc_status dsmc_last_step(dsmc_handle h, int* kind, int* ctas) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  if (kind) *kind = h->last_kind;
  if (ctas) *ctas = h->last_ctas;
  return DSMC_OK;
}

dsmc_status dsmc_autotune(dsmc_handle h, int steps_per_trial, int* best_span_particles,
                          double* best_ms_per_step) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  if (steps_per_trial < 1) return fail(DSMC_E_INVAL, "steps_per_trial must be >= 1");
  if (h->latched != DSMC_OK) return fail(h->latched, "an earlier step reached a device limit");
  if (h->n_inst() == 0) return fail(DSMC_E_STATE, "no instances to tune on");
  DeviceGuard guard(h->device);
  cudaStream_t st = h->stream();
  cudaEvent_t e0, e1;
  DSMC_CUDA(cudaEventCreate(&e0), "event");
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return fail(DSMC_E_CUDA, "event");
  }
  ensure_partition(h);
  const bool own_auto = h->auto_split, span_passes = h->span_passes;
  const Split own{h->span_target, h->cta_warps, h->span_rows};
  Split best = own;
  bool best_own = false;  // the partition in use is the fastest
  double best_ms = -1.0;
  dsmc_status r = DSMC_OK;
  h->span_passes = h->res_dirty = true;  // the trials are of the span passes
  // One untimed step with a new shape, then the timed trial; whether it is the fastest.
  auto trial = [&]() {
    if ((r = step_n(h, 1)) != DSMC_OK) return false;
    if (cudaEventRecord(e0, st) != cudaSuccess) return r = fail(DSMC_E_CUDA, "event record"), false;
    if ((r = step_n(h, steps_per_trial)) != DSMC_OK) return false;
    if (cudaEventRecord(e1, st) != cudaSuccess) return r = fail(DSMC_E_CUDA, "event record"), false;
    if (cudaEventSynchronize(e1) != cudaSuccess) return r = fail(DSMC_E_CUDA, "event sync"), false;
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    const double per = ms / steps_per_trial;
    if (best_ms >= 0.0 && per >= best_ms) return false;
    best_ms = per;
    return true;
  };
  // a run whose cells are shared by several CTAs: that partition, which the whole-cell spans
  // below cannot reach, is the first trial
  if (h->inst[h->order[0]].parts > 1) best_own = trial();
  h->auto_split = false;
  const int shapes[4][2] = {{kAWarps, 1}, {kAWarps, 2}, {kAWarpsSmall, 1}, {kAWarpsSmall, 2}};
  for (const auto& shape : shapes) {
    const int w = shape[0], rows = shape[1];
    long long last_sig = -1;
    for (int target = kMinSpanParticles; target <= (1 << 17) && r == DSMC_OK; target *= 2) {
      int mcps, mcells;
      partition_extent(h, target, nullptr, &mcps, &mcells);
      if (!step_fits(mcells, mcps, h->opt.group_size, w, rows)) break;
      // Skip targets that give the same partition as the last one.
      long long sig = 0;
      for (int id : h->order) {
        int cps, ns;
        make_spans(h->inst[id].n_cells, h->inst[id].ppc, target, &cps, &ns);
        sig = (sig * 1000003 + cps) & 0x3fffffffffffLL;
      }
      if (sig == last_sig) continue;
      last_sig = sig;
      h->cta_warps = w;
      h->span_rows = rows;
      set_partition(h, target);
      if (trial()) {
        best = Split{target, w, rows};
        best_own = false;
      }
    }
    if (r != DSMC_OK) break;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  h->span_passes = span_passes;
  h->res_dirty = true;
  if (r != DSMC_OK || best_own) {  // as before the trials
    h->auto_split = own_auto;
    h->cta_warps = own.warps;
    h->span_rows = own.rows;
    set_partition(h, own.particles);
    if (r != DSMC_OK) {
      cudaGetLastError();
      return r;
    }
    best = own;
  } else {
    h->cta_warps = h->check_warps = best.warps;
    h->span_rows = best.rows;
    set_partition(h, best.particles);
    h->opt.span_particles = best.particles;
    h->opt.cta_warps = best.warps;
    h->opt.span_rows = best.rows;
  }
  h->tuned = best;
  if (best_span_particles) *best_span_particles = best.particles;
  if (best_ms_per_step) *best_ms_per_step = best_ms;
  if (h->opt.profile) return collect_times(h);
  return DSMC_OK;
}

dsmc_status dsmc_sync(dsmc_handle h) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  DeviceGuard guard(h->device);
  return settle(h);
}

dsmc_status dsmc_sample_moments_of(dsmc_handle h, int id, double* out, long long* n_samples) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  if (!out) return fail(DSMC_E_INVAL, "out: NULL");
  DeviceGuard guard(h->device);
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  const Inst& x = h->inst[id];
  DSMC_CUDA(cudaMemcpyAsync(out, h->acc + (size_t)x.cell_base * kNMom,
                            (size_t)x.n_cells * kNMom * sizeof(double), cudaMemcpyDefault,
                            h->stream()),
            "copy moments");
  if (n_samples) *n_samples = x.n_samples;
  return dsmc_sync(h);
}

dsmc_status dsmc_sample_moments(dsmc_handle h, double* out, long long* n_samples) {
  return dsmc_sample_moments_of(h, 0, out, n_samples);
}

dsmc_status dsmc_cell_fields_of(dsmc_handle h, int id, double* out) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  if (!out) return fail(DSMC_E_INVAL, "out: NULL");
  DeviceGuard guard(h->device);
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  const Inst& x = h->inst[id];
  if (x.n_samples < 1) return fail(DSMC_E_STATE, "cell fields: no sampled steps yet");
  double* f = h->fields + (size_t)x.cell_base * DSMC_NFIELD;
  DSMC_CUDA(launch_cell_fields(h->acc + (size_t)x.cell_base * kNMom, x.n_cells, x.n_samples,
                               x.ppc, f, h->stream()),
            "cell fields");
  DSMC_CUDA(cudaMemcpyAsync(out, f, (size_t)x.n_cells * DSMC_NFIELD * sizeof(double),
                            cudaMemcpyDefault, h->stream()),
            "copy cell fields");
  return dsmc_sync(h);
}

dsmc_status dsmc_sample_moments_all(dsmc_handle h, double* out, long long* n_samples) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  if (!out) return fail(DSMC_E_INVAL, "out: NULL");
  DeviceGuard guard(h->device);
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  DSMC_CUDA(cudaMemcpyAsync(out, h->acc, (size_t)h->C.cells * kNMom * sizeof(double),
                            cudaMemcpyDefault, h->stream()),
            "copy moments");
  if (n_samples)
    for (size_t i = 0; i < h->inst.size(); ++i)
      n_samples[i] = h->inst[i].active ? h->inst[i].n_samples : 0;
  return dsmc_sync(h);
}

dsmc_status dsmc_reset_samples_of(dsmc_handle h, int id) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  DeviceGuard guard(h->device);
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  cudaStream_t st = h->stream();
  Inst& x = h->inst[id];
  const size_t c0 = (size_t)x.cell_base, nc = (size_t)x.n_cells;
  DSMC_CUDA(cudaMemsetAsync(h->acc + c0 * kNMom, 0, nc * kNMom * sizeof(double), st), "reset");
  DSMC_CUDA(cudaMemsetAsync(h->ncand + c0, 0, nc * 8, st), "reset");
  DSMC_CUDA(cudaMemsetAsync(h->nacc + c0, 0, nc * 8, st), "reset");
  x.n_samples = 0;
  return DSMC_OK;
}

dsmc_status dsmc_reset_samples(dsmc_handle h) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  for (int id : h->order)
    if ((s = dsmc_reset_samples_of(h, id)) != DSMC_OK) return s;
  return DSMC_OK;
}

dsmc_status dsmc_copy_state_of(dsmc_handle h, int id, float* y, float* vx, float* vy,
                               float* vz) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  DeviceGuard guard(h->device);
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  cudaStream_t st = h->stream();
  const Inst& x = h->inst[id];
  // Straight into the caller's arrays where a kernel can write them (5e7 particles to device
  // memory: 0.51 -> 0.26 ms; 20,000: 36 -> 18 us; 1e6 to pinned memory 112 -> 103 us).
  {
    void* const dst[4] = {y, vx, vy, vz};
    float* out[4];
    if (direct_arrays(dst, (size_t)x.N, h->device, out)) {
      DSMC_CUDA(launch_unpack(h->P[h->cur] + x.part_base, out[0], out[1], out[2], out[3],
                              (int)x.N, st),
                "unpack");
      return dsmc_sync(h);
    }
  }
  // Else unpack the records into four arrays in the instance's part of the idle sort
  // buffer, then copy out.
  float* tmp = reinterpret_cast<float*>(h->P[h->cur ^ 1] + x.part_base);
  const size_t n = (size_t)x.N;
  float* arr[4] = {tmp, tmp + n, tmp + 2 * n, tmp + 3 * n};
  DSMC_CUDA(launch_unpack(h->P[h->cur] + x.part_base, arr[0], arr[1], arr[2], arr[3], (int)x.N,
                          st),
            "unpack");
  float* dst[4] = {y, vx, vy, vz};
  for (int k = 0; k < 4; ++k)
    if (dst[k])
      DSMC_CUDA(cudaMemcpyAsync(dst[k], arr[k], n * sizeof(float), cudaMemcpyDefault, st),
                "copy state");
  return dsmc_sync(h);
}

dsmc_status dsmc_copy_state(dsmc_handle h, float* y, float* vx, float* vy, float* vz) {
  return dsmc_copy_state_of(h, 0, y, vx, vy, vz);
}

dsmc_status dsmc_copy_cells_of(dsmc_handle h, int id, int* offset, float* smax,
                               unsigned long long* ncand, unsigned long long* nacc) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  DeviceGuard guard(h->device);
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  cudaStream_t st = h->stream();
  const Inst& x = h->inst[id];
  const size_t c0 = (size_t)x.cell_base, nc = (size_t)x.n_cells;
  // Gathered into one block (offsets relative to the instance's first slot, as for a run of its
  // own), with the error word: one copy instead of four and the error word's (60 -> 25 us), in
  // the space dsmc_cell_fields_of uses while it runs.
  const CellBlock B(x.n_cells);
  static_assert(CellBlock::kPerCell <= DSMC_NFIELD * sizeof(double), "the block fits the fields");
  char* block = (char*)(h->fields + c0 * DSMC_NFIELD);
  DSMC_CUDA(launch_gather_cells(h->off[h->ocur] + x.off_base, x.part_base,
                                h->smax[h->scur] + c0, h->ncand + c0, h->nacc + c0, h->err,
                                x.n_cells, block, st),
            "gather cells");
  std::vector<char> host(B.total);
  DSMC_CUDA(cudaMemcpyAsync(host.data(), block, B.total, cudaMemcpyDeviceToHost, st),
            "copy cells");
  struct {
    void* to;
    size_t at, bytes;
  } parts[4] = {{offset, B.offset, (nc + 1) * sizeof(int)},
                {smax, B.smax, nc * sizeof(float)},
                {ncand, B.ncand, nc * 8},
                {nacc, B.nacc, nc * 8}};
  // Device (and managed) arrays get theirs from the block on the handle's stream, like every
  // other result; host arrays from its host copy.
  for (auto& q : parts) {
    if (!q.to) continue;
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, q.to) != cudaSuccess) cudaGetLastError();
    if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged) continue;
    DSMC_CUDA(cudaMemcpyAsync(q.to, block + q.at, q.bytes, cudaMemcpyDefault, st), "copy cells");
    q.to = nullptr;
  }
  DSMC_CUDA(cudaStreamSynchronize(st), "stream sync");
  if ((s = collect_times(h)) != DSMC_OK) return s;
  for (const auto& q : parts)
    if (q.to) std::memcpy(q.to, host.data() + q.at, q.bytes);
  int v = 0;
  std::memcpy(&v, host.data() + B.err, sizeof(int));
  return check_error_word(h, v);
}

dsmc_status dsmc_copy_cells(dsmc_handle h, int* offset, float* smax, unsigned long long* ncand,
                            unsigned long long* nacc) {
  return dsmc_copy_cells_of(h, 0, offset, smax, ncand, nacc);
}

dsmc_status dsmc_load_state_of(dsmc_handle h, int id, const float* y, const float* vx,
                               const float* vy, const float* vz, const float* smax,
                               long long step) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  if (!y || !vx || !vy || !vz) return fail(DSMC_E_INVAL, "state arrays must not be NULL");
  if (step < 0) return fail(DSMC_E_INVAL, "step must be >= 0");
  DeviceGuard guard(h->device);
  if ((s = admit_fresh(h)) != DSMC_OK) return s;
  cudaStream_t st = h->stream();
  Inst& x = h->inst[id];
  float* tmp = reinterpret_cast<float*>(h->P[h->cur ^ 1] + x.part_base);
  const size_t n = (size_t)x.N;
  const float* src[4] = {y, vx, vy, vz};
  void* const given[4] = {const_cast<float*>(y), const_cast<float*>(vx), const_cast<float*>(vy),
                          const_cast<float*>(vz)};
  float* in[4];
  if (!direct_arrays(given, n, h->device, in))
    for (int k = 0; k < 4; ++k) {
      in[k] = tmp + k * n;
      DSMC_CUDA(cudaMemcpyAsync(in[k], src[k], n * sizeof(float), cudaMemcpyDefault, st),
                "load state");
    }
  DSMC_CUDA(launch_pack(in[0], in[1], in[2], in[3], h->P[h->cur] + x.part_base, (int)x.N, st),
            "pack");
  if (smax)
    DSMC_CUDA(cudaMemcpyAsync(h->smax[h->scur] + x.cell_base, smax,
                              (size_t)x.n_cells * sizeof(float), cudaMemcpyDefault, st),
              "load smax");
  x.step = step;
  h->tab_dirty = true;
  std::vector<int> host;
  s = set_uniform_offsets(h, id, host);
  if (s != DSMC_OK) return s;
  // The sort pass runs over every instance: for the others, already in cell order,
  // the stable sort leaves records and offsets unchanged.
  s = run_index(h);
  if (s != DSMC_OK) return s;
  return dsmc_sync(h);  // also keeps `host` alive until its copy has run
}

dsmc_status dsmc_load_state(dsmc_handle h, const float* y, const float* vx, const float* vy,
                            const float* vz, const float* smax, long long step) {
  return dsmc_load_state_of(h, 0, y, vx, vy, vz, smax, step);
}

dsmc_status dsmc_get_info_of(dsmc_handle h, int id, dsmc_info* info) {
  dsmc_status s = check_index(h, id);
  if (s != DSMC_OK) return s;
  if (!info) return fail(DSMC_E_INVAL, "info: NULL");
  ensure_partition(h);
  const Inst& x = h->inst[id];
  info->n_particles = x.N;
  info->n_cells = x.n_cells;
  info->ppc = x.ppc;
  info->step = x.step;
  info->n_samples = x.n_samples;
  info->Kn = x.Kn;
  info->omega = x.omega;
  info->body_force = x.F;
  info->nsigma = x.p.nsig;
  info->dt = x.p.dt;
  info->dt_f = x.p.dt_f;
  info->F_f = x.p.F_f;
  info->coef = x.p.coef;
  info->cvhs = x.p.cvhs;
  info->vexp = x.p.vexp;
  info->vinv = x.p.vinv;
  info->lncv = x.p.lncv;
  info->smax0 = x.p.smax0;
  info->device_bytes = h->L.total;
  info->n_instances = h->n_inst();
  info->span_particles = h->span_target;
  info->cta_warps = h->cta_warps;
  info->span_rows = h->span_rows;
  info->cells_per_span = x.cps;
  info->n_spans = x.n_spans;
  info->total_spans = h->spans;
  info->first_slot = x.part_base;
  info->first_cell = x.cell_base;
  return DSMC_OK;
}

dsmc_status dsmc_get_info(dsmc_handle h, dsmc_info* info) { return dsmc_get_info_of(h, 0, info); }

int dsmc_kernel_count(void) { return K_NUM; }

const char* dsmc_kernel_name(int k) { return (k >= 0 && k < K_NUM) ? kKernelNames[k] : ""; }

dsmc_status dsmc_kernel_times(dsmc_handle h, double* total_ms, long long* launches) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  s = collect_times(h);
  if (s != DSMC_OK) return s;
  for (int k = 0; k < K_NUM; ++k) {
    if (total_ms) total_ms[k] = h->ktime[k];
    if (launches) launches[k] = h->kcount[k];
  }
  return DSMC_OK;
}

dsmc_status dsmc_reset_kernel_times(dsmc_handle h) {
  dsmc_status s = check_handle(h);
  if (s != DSMC_OK) return s;
  s = collect_times(h);
  for (int k = 0; k < K_NUM; ++k) {
    h->ktime[k] = 0.0;
    h->kcount[k] = 0;
  }
  return s;
}

dsmc_status dsmc_destroy(dsmc_handle h) {
  if (!h) return DSMC_OK;
  DeviceGuard guard(h->device);
  cudaStreamSynchronize(h->stream());
  drop_graph(h);
  leave_team_runs(h);
  if (h->stepped) cudaEventDestroy(h->stepped);
  for (cudaEvent_t e : h->events) cudaEventDestroy(e);
  if (h->owns && h->ws) cudaFree(h->ws);
  delete h;
  return DSMC_OK;
}

const char* dsmc_last_error(void) { return g_last_error.c_str(); }

const char* dsmc_status_string(dsmc_status s) {
  switch (s) {
    case DSMC_OK: return "ok";
    case DSMC_E_INVAL: return "invalid argument";
    case DSMC_E_NOMEM: return "out of memory";
    case DSMC_E_CUDA: return "CUDA error";
    case DSMC_E_DEVICE_LIMIT: return "device limit reached";
    case DSMC_E_STATE: return "invalid state";
  }
  return "unknown status";
}

}  // extern "C"

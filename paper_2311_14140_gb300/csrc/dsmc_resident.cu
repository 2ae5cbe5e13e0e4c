// dsmc_resident.cu -- many steps of small runs in one launch.
//
// A small run's step is bound by launches and by the latency of its passes, not by work:
// 20,000 particles through the span passes of dsmc_step.cu take 22 us per step (three
// launches under graph replay, each a cold start of a CTA's worth of dependent phases),
// against about 2 us of instruction issue on 16 SMs.  Here one launch runs all the steps of a
// call, and particles, counts and prefixes pass between its CTAs with two barriers per step
// instead of kernel boundaries:
//   a cluster (up to 16 CTAs) per instance: counts by distributed shared memory, hardware
//     cluster barriers.  Instances do not depend on one another, so a batch is one cluster per
//     instance.
//   a team (kTeam): for one run that 16 SMs would be slow on, a cooperative grid of a CTA per
//     SM: counts and cell results by global memory, a counter barrier (about 1.5 us each).
// Measured (us per step, before = span passes under graph replay): 20,000 particles 22.5 ->
// 10.8, 10,000 20.9 -> 8.1 and 2,250 20.5 -> 6.8 (cluster), 100,000 21-30 -> 13.5, 300,000
// 38 -> 16.7, 1,004,807 71 -> 27.4 (team).  What is left is the latency of one collision group per warp (a chain of
// about 8,000 cycles at 200 particles), then barriers, loads and the ranking.
//
// A step, for CTA r of CL (identical arithmetic, operation for operation, to the
// span passes; only the place where it happens differs):
//   A  load its slots -- the collision groups that start in its share [cut_r, cut_{r+1}) of
//      the slots -- into shared memory; its warps take the groups one after another (moments, NTC
//      candidates, moments, flight) and update them in place; then every warp ranks a
//      contiguous part of the slots by new cell (running counts per warp and cell), and
//      the CTA publishes its particles per cell.
//      [barrier]
//   B  every CTA reads the others' counts: exclusive prefix over CTAs and cells gives the
//      new cell offsets and the CTA's base in every cell; the cell's owner CTA adds the
//      step's moment sums to the run's; each record goes to its sorted place: in the shared
//      memory of the CTA that takes it next (one instance on one cluster), or in the other
//      record buffer (global memory, L2-resident at these sizes).
//      [barrier]
// Cell results (fixed-point moment totals, counters, largest relative speed) are integer
// adds and maxima, in the owner CTA's shared memory or in global memory, so they do not depend
// on the order.
#include <type_traits>

#include "dsmc_collide.cuh"
#include "dsmc_device.cuh"
#include "dsmc_internal.h"

namespace dsmc {

namespace {

// --- cluster primitives ---------------------------------------------------------------

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Barrier of all threads of the cluster; memory operations before it (shared, distributed
// shared and global) are visible to the cluster's threads after it.
__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The address of this CTA's shared-memory location `p` in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}

__device__ __forceinline__ uint32_t peer_load(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ void peer_store(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ void peer_store4(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}

__device__ __forceinline__ void peer_add(uint32_t addr, unsigned long long v) {
  asm volatile("red.relaxed.cluster.shared::cluster.add.u64 [%0], %1;" ::"r"(addr), "l"(v)
               : "memory");
}

__device__ __forceinline__ void peer_max(uint32_t addr, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.max.u32 [%0], %1;" ::"r"(addr), "r"(v)
               : "memory");
}

// Barrier of the CTAs of a team: a counter and a generation in global memory (both zero, or as
// an earlier team left them).  The last CTA to arrive clears the counter and advances the
// generation.  Memory operations before it are visible after it to loads that bypass L1.
// Waits are bounded; false when one ran out.  The counter is then out of step for good.
struct TeamBarrier {
  unsigned *count = nullptr, *gen = nullptr, now = 0u;
  int n = 0;
  static __device__ __forceinline__ unsigned load(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
  }
  __device__ __forceinline__ void start(unsigned* b, int ctas) {
    count = b;
    gen = b + 1;
    n = ctas;
    if (threadIdx.x == 0) now = load(gen);  // nobody passes the first wait before this CTA arrives
  }
  __device__ __forceinline__ bool wait() {
    bool ok = true;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned before;
      asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;"
                   : "=r"(before)
                   : "l"(count)
                   : "memory");
      ++now;
      if (before == (unsigned)(n - 1)) {
        *count = 0u;
        asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(gen), "r"(now) : "memory");
      } else {
        ok = false;
        for (int i = 0; i < kMaxWaitPolls && !ok; ++i) ok = load(gen) == now;
      }
    }
    return __syncthreads_and(ok) != 0;
  }
};

}  // namespace

template <bool kBatch, int kWarps, bool kF64, bool kTeam>
__global__ void __launch_bounds__(kWarps * 32, kBatch ? 2 : 1)
    k_resident(float4* P0, float4* P1, int* off0, int* off1, float* smax0, float* smax1,
               unsigned long long* ncand_all, unsigned long long* nacc_all, double* acc_all,
               int* exchange, unsigned* barrier, const InstParams one, const ResidentLaunch RL,
               int* err) {
  static_assert(!(kBatch && kTeam), "a team serves one instance");
  // One instance on one cluster: a CTA sends its sorted records straight into the shared memory
  // of the CTA that takes them in the next step (two record buffers), so they are neither
  // written to L2 nor read back.  A batch's CTAs share SMs two by two and a team's are not a
  // cluster: their records go through the global buffers.
  constexpr bool kLocal = !kBatch && !kTeam;
  using Acc = typename std::conditional<kF64, double, float>::type;
  constexpr int kThreads = kWarps * 32;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ InstParams sh_inst;
  __shared__ int wsum[2][32];
  // first groups of the CTAs (kLocal: of all of them), or of this CTA and the next
  constexpr int kBounds = kLocal ? kResidentMaxCluster + 1 : 2;
  __shared__ int bnd_slot[kBounds], bnd_cell[kBounds], bnd_group[kBounds];
  __shared__ int n_groups_sh, next_group, n_hits, dead;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int CL = RL.cl;
  const int rank = kTeam ? (int)blockIdx.x : (int)cluster_rank();
  if constexpr (kBatch) {
    const int* src = reinterpret_cast<const int*>(&RL.tab[blockIdx.x / CL]);
    int* dst = reinterpret_cast<int*>(&sh_inst);
    for (int i = tid; i < (int)(sizeof(InstParams) / 4); i += kThreads) dst[i] = src[i];
    __syncthreads();
  }
  const InstParams& a = kBatch ? sh_inst : one;
  const ResidentSmem L = resident_smem_layout(RL.max_cells, RL.range_cap, RL.list_cap,
                                              RL.own_cap, kTeam ? 0 : RL.cl, kLocal, kWarps);
  float4* rec = reinterpret_cast<float4*>(smem + L.rec);        // this CTA's records
  float4* rec_next = rec + RL.range_cap;                        // the next step's (kLocal)
  unsigned* key = reinterpret_cast<unsigned*>(smem + L.key);    // candidate masks, then ranks
  int2* list = reinterpret_cast<int2*>(smem + L.list);          // groups: (cell, gi << 10 | gn)
  unsigned short* rows = reinterpret_cast<unsigned short*>(smem + L.rows);  // counts per warp, cell
  int* tot = reinterpret_cast<int*>(smem + L.tot);              // counts per CTA and cell
  int* base = reinterpret_cast<int*>(smem + L.base);            // this CTA's first slot per cell
  float* csmax = reinterpret_cast<float*>(smem + L.smax);       // (sigma g)_max per cell
  // of the cells this CTA owns: the step's fixed-point sums, the run's moment sums, and the
  // largest relative speed of even and odd steps
  unsigned long long* cfix = reinterpret_cast<unsigned long long*>(smem + L.cfix);
  double* csum = reinterpret_cast<double*>(smem + L.csum);
  unsigned* cgmax = reinterpret_cast<unsigned*>(smem + L.cgmax);

  const int n_cells = a.n_cells, G = a.G, mode = a.mode;
  const int own = (n_cells + CL - 1) / CL;          // cells per owner CTA
  const int own0 = rank * own;                      // first cell this CTA owns
  const int own_n = max(0, min(own, n_cells - own0));
  const int lo = a.part_base, hi = a.part_base + a.n_part;
  // slots at which this CTA's and the next CTA's groups may start
  const int B0 = lo + (kTeam ? RL.cut[rank] : a.cut[rank]);
  const int B1 = lo + (kTeam ? RL.cut[rank + 1] : a.cut[rank + 1]);
  const int me = kLocal ? rank : 0, last = kLocal ? CL : 1;  // this CTA's bound, the last one
  // A team's exchange in global memory: count rows of its CTAs; their sums over blocks of
  // kTeamBlock CTAs, of even and odd steps; the cells' largest relative speeds, of even and
  // odd steps; and the cells' fixed-point sums.
  const int n_blocks = (CL + kTeamBlock - 1) / kTeamBlock, my_block = rank / kTeamBlock;
  int* xrow = exchange;
  int* xblk = xrow + (size_t)CL * n_cells;
  unsigned* xgmax = reinterpret_cast<unsigned*>(xblk + 2 * (size_t)n_blocks * n_cells);
  unsigned long long* xfix = reinterpret_cast<unsigned long long*>(
      exchange + team_fix_offset(CL, n_cells));
  TeamBarrier team;
  if constexpr (kTeam) team.start(barrier, CL);
  bool lost = false;  // a wait ran out: the CTA leaves, and the others' waits run out too
  auto wait_all = [&]() {
    if constexpr (kTeam)
      lost = !team.wait();
    else
      cluster_barrier();
  };
  unsigned long long* ncand = ncand_all + a.cell_base;
  unsigned long long* nacc = nacc_all + a.cell_base;
  double* acc = acc_all + (size_t)a.cell_base * kNMom;
  long long istep = RL.gstep - a.step0;

  int* off = reinterpret_cast<int*>(smem + L.off);  // this step's cell offsets
  int* off_next = off + RL.max_cells + 1;
  {
    const int* g = (RL.parity_off ? off1 : off0) + a.off_base;
    const float* s = (RL.parity_smax ? smax1 : smax0) + a.cell_base;
    for (int c = tid; c <= n_cells; c += kThreads) off[c] = g[c];
    for (int c = tid; c < n_cells; c += kThreads) csmax[c] = s[c];
    if constexpr (kTeam) {
      for (int i = rank * kThreads + tid; i < 2 * n_blocks * n_cells; i += CL * kThreads) xblk[i] = 0;
      for (int i = rank * kThreads + tid; i < 2 * n_cells; i += CL * kThreads) xgmax[i] = 0u;
      for (int i = rank * kThreads + tid; i < 12 * n_cells; i += CL * kThreads) xfix[i] = 0ull;
    } else {
      for (int i = tid; i < own * 12; i += kThreads) cfix[i] = 0ull;
      for (int i = tid; i < 2 * own; i += kThreads) cgmax[i] = 0u;
    }
    for (int i = tid; i < own_n * kNMom; i += kThreads) csum[i] = acc[(size_t)own0 * kNMom + i];
  }
  const int gshift = (G & (G - 1)) ? -1 : 31 - __clz(G);  // G is a power of two: its exponent
  auto groups_of = [&](int n) {  // group_count without its division
    if (gshift < 0) return group_count(n, G);
    const int ng = n >> gshift, r = n & (G - 1);
    return ng + ((r > 0 && (ng == 0 || r >= G / 2)) ? 1 : 0);
  };
  // Bound k (a slot share's first slot B) from the cell c it falls into, of n slots from
  // `first` on: the CTA's groups begin with the cell's first group that starts at or after B,
  // or with the next cell.
  auto set_bound = [&](int k, int B, int c, int first, int n) {
    const int i = gshift < 0 ? (B - first + G - 1) / G : (B - first + G - 1) >> gshift;
    const int ng = groups_of(n);
    bnd_cell[k] = c;
    bnd_group[k] = min(i, ng);
    bnd_slot[k] = i < ng ? first + i * G : first + n;
  };
  // The bounds under cell offsets o, by the first threads (a search each): what a cluster that
  // needs all of its CTAs' bounds does.
  auto find_bounds = [&](const int* o) {
    if (kLocal ? tid >= CL : (tid >= 2 || rank + tid >= CL)) return;
    const int B = kLocal ? lo + a.cut[tid] : (tid ? B1 : B0);
    int c = 0;
    for (int h = 1 << (31 - __clz(n_cells)); h > 0; h >>= 1)
      if (c + h < n_cells && o[c + h] <= B) c += h;
    set_bound(tid, B, c, o[c], o[c + 1] - o[c]);
  };
  // The list of this CTA's groups under cell offsets o and the bounds, by one warp.
  auto make_list = [&](const int* o) {
    const int cb = bnd_cell[me], ce = bnd_cell[me + 1];
    const int gb = bnd_group[me], ge = bnd_group[me + 1];
    const int len = bnd_slot[me + 1] - bnd_slot[me];
    int run = 0;
    const int cend = len > 0 && len <= RL.range_cap ? min(ce, n_cells - 1) : cb - 1;
    for (int c0 = cb; c0 <= cend; c0 += 32) {
      const int c = c0 + lane;
      int g0 = 0, g1 = 0, ng = 0, nc = 0;
      if (c <= cend) {
        nc = o[c + 1] - o[c];
        ng = groups_of(nc);
        g0 = c == cb ? gb : 0;
        g1 = max(g0, c == ce ? ge : ng);
      }
      const int cnt = g1 - g0;
      int incl = cnt;
#pragma unroll
      for (int q = 1; q < 32; q <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, q);
        if (lane >= q) incl += t;
      }
      int p = run + incl - cnt;
      for (int g = g0; g < g1; ++g, ++p)
        if (p < RL.list_cap) list[p] = make_int2(c, (g << 10) | (g == ng - 1 ? nc - g * G : G));
      run += __shfl_sync(kFull, incl, 31);
    }
    if (lane == 0) {
      n_groups_sh = run <= RL.list_cap ? run : -1;
      next_group = kWarps;  // every warp starts with the group of its own number
    }
  };
  unsigned short* queue = rows;  // (local slots)
  const int qcap = (int)(L.rows_bytes / 2) & ~31;  // wall hits the queue holds
  if (tid == 0) {
    n_hits = 0;
    // A team whose run's error word has kErrTeam already does not start: launches may be queued
    // behind the one whose wait ran out.
    dead = kTeam && (*(const volatile int*)err & kErrTeam) != 0;
    // the instance's end (the last CTA's end is past every cell)
    bnd_slot[last] = hi;
    bnd_cell[last] = n_cells;
    bnd_group[last] = 0;
  }
  for (int i = tid; i < RL.range_cap; i += kThreads) key[i] = 0u;  // (zero between steps)
  __syncthreads();
  find_bounds(off);
  __syncthreads();
  if (kLocal && w == kWarps - 1) make_list(off);
  const float4* Pin = RL.parity_rec ? P1 : P0;
  float4* Pout = RL.parity_rec ? P0 : P1;
  bool bad_bounce = false, cand_fail = false, inflow_fail = false, mom_range = false;
  bool bad_sort = false;
  if constexpr (kLocal) {
    const int s0 = bnd_slot[me], n = min(bnd_slot[me + 1] - s0, RL.range_cap);
    for (int i = tid; i < n; i += kThreads) rec[i] = Pin[s0 + i];
  }
  if (kTeam && dead)
    lost = true;  // (nothing of the run has been written)
  else
    wait_all();  // every CTA's accumulators are cleared

  int st = 0;
  for (; st < RL.n_steps && !lost; ++st, ++istep) {
    const uint32_t step = (uint32_t)istep;
    const bool sample = istep >= a.sample_start;
    const bool collide = a.collide != 0;
    const int s0 = bnd_slot[me];
    int len = bnd_slot[me + 1] - s0;
    if (len < 0 || len > RL.range_cap) {  // only corrupted offsets can do this
      bad_sort = true;
      len = 0;
    }

    // A. This CTA's records and groups.
    if constexpr (!kLocal) {
      if (w == kWarps - 1)
        make_list(off);
      else
        for (int i = tid; i < len; i += kThreads - 32) rec[i] = __ldcg(Pin + s0 + i);
      __syncthreads();
    }
    const int n_groups = n_groups_sh;
    if (n_groups < 0) bad_sort = true;

    for (int q = w; q < n_groups;) {
      const int2 e = list[q];
      const int c = e.x, gi = e.y >> 10, gn = e.y & 1023;
      const int cs = off[c], nc = off[c + 1] - cs;
      const int gl = cs + gi * G - s0;  // first local slot of the group
      if (gl < 0 || gl + gn > len) {  // only corrupted offsets can do this
        bad_sort = true;
        break;
      }
      float4* rg = rec + gl;
      unsigned* touch = key + gl;
      const float smax = csmax[c];

      // Moments before the collisions, candidates, moments after them.
      float gmax = 0.0f;
      unsigned laccn = 0;
      uint32_t M = 0;
      LaneSums<Acc> m;
      m.zero();
      if (sample)
        for (int i = lane; i < gn; i += 32) {
          const float4 r = rg[i];
          m.add(r.y, r.z, r.w);
        }
      if (collide && gn >= 2)
        ntc_collide(a, rg, touch, gn, nc, c, gi, step, smax, mode, lane, lt, gmax, M, laccn,
                    cand_fail);
      __syncwarp();
      if (sample)
        for (int i = lane; i < gn; i += 32) {
          const float4 r = rg[i];
          m.add(r.y, r.z, r.w);
        }

      // The group's results into the slots of the cell's owner.
      const int oc = c / own, os = c - oc * own;
      if (sample) {
        const Acc total = group_total(m, lane);
        const int k = moment_of_lane(lane);
        if ((lane & 1) == 0 && k >= 1 && k <= 12) {
          const int gexp = grid_exponent(nc);
          const long long fx = fixed_of(total, gexp);
          const long long lim = (long long)(2 * gn) << (20 + gexp);
          if (fx > lim || fx < -lim) mom_range = true;
          if constexpr (kTeam)
            atomicAdd(xfix + (size_t)c * 12 + (k - 1), (unsigned long long)fx);
          else
            peer_add(peer_addr(cfix + os * 12 + (k - 1), oc), (unsigned long long)fx);
        }
      }
      const unsigned gbits = __reduce_max_sync(kFull, __float_as_uint(gmax));  // gmax >= 0
      const unsigned nac = __reduce_add_sync(kFull, laccn);
      if (lane == 0) {
        if constexpr (kTeam) {
          if (gbits) atomicMax(xgmax + (st & 1) * n_cells + c, gbits);
        } else {
          if (gbits) peer_max(peer_addr(cgmax + (st & 1) * own + os, oc), gbits);
        }
        if (M) atomicAdd(ncand + c, (unsigned long long)M);
        if (nac) atomicAdd(nacc + c, (unsigned long long)nac);
        q = atomicAdd(&next_group, 1);
      }
      q = __shfl_sync(kFull, q, 0);
    }
    __syncthreads();

    // Flight.  Particles that reach a wall are queued and flown afterwards, shared evenly by
    // all warps of the CTA (they come from the few cells next to a wall).  The queue lives
    // in the space of the ranks' counts, as many slots at a time as it could ever need.
    for (int c0 = 0; c0 < len; c0 += qcap) {
      const int c1 = min(len, c0 + qcap);
      for (int b = c0 + w * 32; b < c1; b += kThreads) {
        const int i = b + lane;
        bool hits = false;
        if (i < c1) {
          const float4 r = rec[i];
          const float ynew = fadd(r.x, fmul(r.z, a.dt));
          hits = (ynew < 0.0f) || (ynew > 1.0f);
          if (!hits)
            *reinterpret_cast<float2*>(&rec[i]) = make_float2(ynew, fadd(r.y, fmul(a.F, a.dt)));
        }
        const unsigned hm = __ballot_sync(kFull, hits);
        if (hm) {
          int at = 0;
          if (lane == 0) at = atomicAdd(&n_hits, __popc(hm));
          at = __shfl_sync(kFull, at, 0) + __popc(hm & lt);
          if (hits) queue[at] = (unsigned short)i;
        }
      }
      __syncthreads();
      const int nq = n_hits;
      for (int b = w * 32; b < nq; b += kThreads)
        if (b + lane < nq) {
          const int i = queue[b + lane];
          const float4 r = rec[i];
          float yy = r.x, xx = r.y, uy = r.z, zz = r.w;
          if (!fly(yy, xx, uy, zz, a.dt, a.F, a.keys, step, (uint32_t)(s0 + i - lo), a.open_top,
                   a.u_top, a.p_top, inflow_fail))
            bad_bounce = true;
          rec[i] = make_float4(yy, xx, uy, zz);
        }
      __syncthreads();
      if (tid == 0) n_hits = 0;
      if (c1 < len) __syncthreads();
    }
    unsigned short* row = rows + w * n_cells;
    for (int c = lane; c < n_cells; c += 32) row[c] = 0;
    __syncwarp();

    // Rank of every record among the earlier ones of its warp's part bound for its cell; the
    // cells and same-cell lanes of four slices at a time, then slice after slice the counts.
    const int part = ((len + kWarps - 1) / kWarps + 31) & ~31;
    const int pb = w * part, pe = min(len, pb + part);
    for (int b = pb; b < pe; b += 128) {
      int cell[4];
      unsigned peers[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = b + 32 * u + lane;
        cell[u] = i < pe ? cell_of(rec[i].x, n_cells, a.ncf) : -1;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (b + 32 * u < pe) peers[u] = __match_any_sync(kFull, cell[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (b + 32 * u >= pe) break;
        const bool act = cell[u] >= 0;
        const int first = act ? row[cell[u]] : 0;
        const int before = __popc(peers[u] & lt);
        __syncwarp();
        if (act) {
          if (before == 0) row[cell[u]] = (unsigned short)(first + __popc(peers[u]));
          key[b + 32 * u + lane] = ((unsigned)cell[u] << 16) | (unsigned)(first + before);
        }
        __syncwarp();
      }
    }
    __syncthreads();
    for (int c = tid; c < n_cells; c += kThreads) {
      int t[kWarps], run = 0;
#pragma unroll
      for (int v = 0; v < kWarps; ++v) t[v] = rows[v * n_cells + c];
#pragma unroll
      for (int v = 0; v < kWarps; ++v) {
        rows[v * n_cells + c] = (unsigned short)run;
        run += t[v];
      }
      if constexpr (kTeam) {
        xrow[(size_t)rank * n_cells + c] = run;
        if (run) atomicAdd(xblk + ((size_t)(st & 1) * n_blocks + my_block) * n_cells + c, run);
      } else {
        for (int v = 0; v < CL; ++v) peer_store(peer_addr(tot + rank * n_cells + c, v), run);
      }
    }
    wait_all();
    if (lost) break;

    // B. New offsets, the cells' results, and the sort.
    int carry = lo;
    for (int cb = 0, ph = 0; cb < n_cells; cb += kThreads, ph ^= 1) {
      const int c = cb + tid;
      int total = 0, pre = 0;
      uint32_t gm = 0u;
      if constexpr (kTeam) {
        if (c < n_cells) {
          gm = __ldcg(xgmax + (st & 1) * n_cells + c);
          const int* blk = xblk + (size_t)(st & 1) * n_blocks * n_cells + c;
          const int* row0 = xrow + (size_t)my_block * kTeamBlock * n_cells + c;
          int x[kTeamBlock], y[kTeamBlock];  // all loads in flight at once
#pragma unroll
          for (int v = 0; v < kTeamBlock; ++v) {
            x[v] = v < n_blocks ? __ldcg(blk + (size_t)v * n_cells) : 0;
            y[v] = my_block * kTeamBlock + v < rank ? __ldcg(row0 + (size_t)v * n_cells) : 0;
          }
#pragma unroll
          for (int v = 0; v < kTeamBlock; ++v) {
            total += x[v];
            pre += (v < my_block ? x[v] : 0) + y[v];
          }
        }
      } else if (c < n_cells) {
        const int oc = c / own;  // the owner's largest relative speed, used below
        gm = peer_load(peer_addr(cgmax + (st & 1) * own + (c - oc * own), oc));
#pragma unroll
        for (int v = 0; v < kResidentMaxCluster; ++v) {
          const int t = v < CL ? tot[v * n_cells + c] : 0;
          total += t;
          pre += v < rank ? t : 0;
        }
      }
      int incl = total;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
      }
      if (lane == 31) wsum[ph][w] = incl;
      __syncthreads();
      const int ws = lane < kWarps ? wsum[ph][lane] : 0;
      const int before = carry + __reduce_add_sync(kFull, lane < w ? ws : 0);
      const int all = __reduce_add_sync(kFull, ws);
      carry += all;
      if (c < n_cells) {
        const int first = before + incl - total;
        off_next[c] = first;
        base[c] = first + pre;
        if (c == n_cells - 1) off_next[n_cells] = first + total;
        if constexpr (!kLocal) {  // this CTA's two bounds, by the threads whose cells they fall into
          if (B0 >= first && B0 < first + total) set_bound(0, B0, c, first, total);
          if (rank + 1 < CL && B1 >= first && B1 < first + total) set_bound(1, B1, c, first, total);
        }
        // (sigma g)_max of the next step
        const float g = __uint_as_float(gm);
        const float sg = (mode == 0) ? g : fmul(a.cvhs, pow32(g, a.vexp));
        csmax[c] = fmaxf(csmax[c], sg);
      }
    }
    // (taken from the last threads down: the first ones are busy with the cells above)
    for (int i = kThreads - 1 - tid; i < own_n * kNMom; i += kThreads) {
      const int oc = i / kNMom, k = i - oc * kNMom, c = own0 + oc;
      if (k == 0) {
        if constexpr (kTeam)
          xgmax[((st & 1) ^ 1) * n_cells + c] = 0u;
        else
          cgmax[((st & 1) ^ 1) * own + oc] = 0u;
      }
      if (sample) {
        const int nc = off[c + 1] - off[c];
        if (k == 0) {
          csum[i] += (double)nc;
        } else {
          unsigned long long* fix =
              kTeam ? xfix + (size_t)c * 12 + (k - 1) : cfix + oc * 12 + (k - 1);
          const unsigned long long q = kTeam ? __ldcg(fix) : *fix;
          const double grid =
              __longlong_as_double((long long)(1023 - grid_exponent(nc > 0 ? nc : 1)) << 52);
          csum[i] += 0.5 * grid * (double)(long long)q;
          *fix = 0ull;
        }
      }
    }
    if constexpr (kTeam)  // the block sums of the next step
      for (int i = rank * kThreads + tid; i < n_blocks * n_cells; i += CL * kThreads)
        xblk[(size_t)((st & 1) ^ 1) * n_blocks * n_cells + i] = 0;
    __syncthreads();
    if constexpr (kLocal) {
      find_bounds(off_next);
      __syncthreads();
    }
    for (int b = pb; b < pe; b += 32) {
      const int i = b + lane;
      if (i < pe) {
        const unsigned kk = key[i];
        key[i] = 0u;
        const int cell = (int)(kk >> 16);
        const int d = base[cell] + rows[w * n_cells + cell] + (int)(kk & 0xffffu);
        if (d < lo || d >= hi) {
          bad_sort = true;
        } else if constexpr (kLocal) {
          int k = 0;  // the CTA whose slots these are
#pragma unroll
          for (int o = kResidentMaxCluster / 2; o > 0; o >>= 1)
            if (k + o < CL && d >= bnd_slot[k + o]) k += o;
          const int at = d - bnd_slot[k];
          if (at < RL.range_cap)
            peer_store4(peer_addr(rec_next + at, k), rec[i]);
          else
            bad_sort = true;
        } else {
          Pout[d] = rec[i];
        }
      }
    }
    // the next step's groups, by the warp whose part is the shortest
    if (kLocal && w == kWarps - 1) make_list(off_next);
    wait_all();
    int* t0 = off;
    off = off_next;
    off_next = t0;
    float4* t1 = const_cast<float4*>(Pin);
    Pin = Pout;
    Pout = t1;
    if constexpr (kLocal) {
      float4* t2 = rec;
      rec = rec_next;
      rec_next = t2;
    }
  }
  if constexpr (kLocal) {  // Pin: the buffer of the state after the last step
    const int s0 = bnd_slot[me], n = min(bnd_slot[me + 1] - s0, RL.range_cap);
    float4* out = const_cast<float4*>(Pin);
    for (int i = tid; i < n; i += kThreads) out[s0 + i] = rec[i];
  }

  for (int i = tid; i < own_n * kNMom; i += kThreads) acc[(size_t)own0 * kNMom + i] = csum[i];
  // The run's state after the last step, where the next launch of either kind looks for it.
  if (rank == 0 && !lost) {
    int* g = ((RL.parity_off ^ RL.n_steps) & 1 ? off1 : off0) + a.off_base;
    float* s = ((RL.parity_smax ^ RL.n_steps) & 1 ? smax1 : smax0) + a.cell_base;
    for (int c = tid; c <= n_cells; c += kThreads) g[c] = off[c];
    for (int c = tid; c < n_cells; c += kThreads) s[c] = csmax[c];
  }
  if (bad_bounce) atomicOr(err, kErrBounces);
  if (cand_fail && lane == 0) atomicOr(err, kErrCandidates);
  if (inflow_fail) atomicOr(err, kErrInflow);
  if (mom_range) atomicOr(err, kErrMoments);
  if (bad_sort) atomicOr(err, kErrSort);
  if (lost && tid == 0) atomicOr(err, kErrTeam);
}

namespace {

const void* resident_kernel(bool batch, bool f64, bool team) {
  if (team)
    return f64 ? (const void*)k_resident<false, kResidentWarps, true, true>
               : (const void*)k_resident<false, kResidentWarps, false, true>;
  if (batch)
    return f64 ? (const void*)k_resident<true, kResidentWarpsBatch, true, false>
               : (const void*)k_resident<true, kResidentWarpsBatch, false, false>;
  return f64 ? (const void*)k_resident<false, kResidentWarps, true, false>
             : (const void*)k_resident<false, kResidentWarps, false, false>;
}

// The launch of `ctas` CTAs in clusters of `cl`, or as a cooperative grid (team).
struct ResidentConfig {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  ResidentConfig(int ctas, int cl, int warps, size_t smem, bool team, cudaStream_t st) {
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)(warps * 32));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    if (team) {
      at.id = cudaLaunchAttributeCooperative;
      at.val.cooperative = 1;
    } else {
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = (unsigned)cl;
      at.val.clusterDim.y = at.val.clusterDim.z = 1;
    }
    cfg.attrs = &at;
    cfg.numAttrs = 1;
  }
};

}  // namespace

cudaError_t resident_fits(const ResidentLaunch& L, size_t smem, bool f64, bool* fits) {
  const bool batch = L.n_inst > 1;
  const void* f = resident_kernel(batch, f64, L.team != 0);
  *fits = false;
  cudaError_t e =
      cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResidentSmemMax);
  if (e == cudaSuccess && !L.team)
    e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  int n = 0;
  if (L.team) {  // every CTA of the grid resident at once, one per SM
    int dev = 0, sms = 0, coop = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess)
      return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, resident_warps(false) * 32, smem);
    *fits = e == cudaSuccess && coop && n >= 1 && L.cl <= sms;
    return e;
  }
  ResidentConfig c(L.cl, L.cl, resident_warps(batch), smem, false, nullptr);
  e = cudaOccupancyMaxActiveClusters(&n, f, &c.cfg);
  *fits = e == cudaSuccess && n >= 1;
  return e;
}

cudaError_t launch_resident(float4* P0, float4* P1, int* off0, int* off1, float* smax0,
                            float* smax1, unsigned long long* ncand, unsigned long long* nacc,
                            double* acc, int* exchange, unsigned* barrier, const InstParams& one,
                            const ResidentLaunch& L, bool f64, int* err, cudaStream_t st) {
  const int warps = resident_warps(L.n_inst > 1);
  const ResidentSmem S = resident_smem_layout(L.max_cells, L.range_cap, L.list_cap, L.own_cap,
                                              L.team ? 0 : L.cl, resident_local(L), warps);
  ResidentConfig c(L.cl * L.n_inst, L.cl, warps, S.total, L.team != 0, st);
  void* args[] = {&P0,   &P1,  &off0,     &off1,    &smax0, &smax1, &ncand,
                  &nacc, &acc, &exchange, &barrier, const_cast<InstParams*>(&one),
                  const_cast<ResidentLaunch*>(&L),  &err};
  const cudaError_t e =
      cudaLaunchKernelExC(&c.cfg, resident_kernel(L.n_inst > 1, f64, L.team != 0), args);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace dsmc

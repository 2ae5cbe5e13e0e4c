// dsmc_step.cu -- the two state passes of one DSMC step (Bird's method, which the
// paper cites for its micro model; problem of Sec. 2.1, units of Eq. 6).
//
// The resident particle state is an array of float4 records (y, vx, vy, vz): one
// 16-byte load or store moves a whole particle, so the sort's scattered writes cost
// one L2 sector per particle instead of four.
//
//   k_collide_move   one CTA per span of consecutive cells, the heaviest spans launched
//                    first (an order the host estimates).  Its warps take the span's
//                    collision groups one after another (a shared counter hands them
//                    out) and for each group
//                      1. load the group's records, keep them in shared memory and add
//                         their moment sums before the collisions,
//                      2. draw every NTC candidate's pair, acceptance threshold and
//                         scattering direction up front (one Philox draw per candidate,
//                         32 candidates at a time, one per lane), then apply the
//                         candidates in conflict-free rounds that reproduce the
//                         sequential order exactly,
//                      3. per particle: add the moment sums after the collisions, fly
//                         with the body force and diffuse walls, store the record back
//                         in place and count its new cell in the CTA's histogram.
//                    The histogram becomes the span's row of the sort matrix.  Per-cell
//                    (sigma g)_max, collision counters and moment sums are written by
//                    the one CTA that owns the cell; where several CTAs share a cell they
//                    add integers into CellSums and the scan writes the results.  With
//                    `count_only` the pass just counts cells of the span's slots (the sort into cells at creation
//                    and after a state load).
//   k_scatter_spans  one warp per span: re-reads the records in slot order, 16 per lane
//                    in flight, ranks each record among the same-cell records before it
//                    and scatters it stably into the other buffer from the span's row of
//                    the prefix-summed matrix plus the new cell offsets.
//   k_scatter_coop   the same scatter with a CTA per span (up to 1,365 cells): all its
//                    warps rank one round of 256 (or 512) records at a time.
//
// Between them, k_scan_spans (or k_scan_cols for instances of few spans) turns the matrix into
// per-span bases and the cells' counts; the new cell offsets come from those, in the
// CTA-per-span scatter itself or by k_offsets_cells for the other.
#include <climits>
#include <type_traits>

#include "dsmc_collide.cuh"
#include "dsmc_device.cuh"
#include "dsmc_internal.h"

namespace dsmc {

namespace {

// Adds a group's results into the CTA's slots of its cell: the 12 moment totals as
// fixed-point integers (lanes 2i of the butterfly), the largest relative speed, the
// candidate and accepted-collision counts.  Returns false when a total exceeds the
// magnitude the fixed-point range allows for the group's size.
template <typename T>
__device__ __forceinline__ bool add_group(const LaneSums<T>& m, bool sample, int gn, int nc,
                                          float gmax, uint32_t M, unsigned accn,
                                          unsigned long long* cfix, unsigned* cgmax,
                                          unsigned long long* ccand,
                                          unsigned long long* caccn, int lane) {
  bool ok = true;
  if (sample) {
    const auto tot = group_total(m, lane);
    const int k = moment_of_lane(lane);
    if ((lane & 1) == 0 && k >= 1 && k <= 12) {
      const int ge = grid_exponent(nc);
      const long long q = fixed_of(tot, ge);
      // |q| <= 2 gn 2^20 2^ge holds for |products| <= 2^20
      const long long lim = (long long)(2 * gn) << (20 + ge);
      if (q > lim || q < -lim) ok = false;
      atomicAdd(&cfix[k], (unsigned long long)q);
    }
  }
  const unsigned gbits = __reduce_max_sync(kFull, __float_as_uint(gmax));  // gmax >= 0
  const unsigned nacc = __reduce_add_sync(kFull, accn);
  if (lane == 0) {
    atomicMax(cgmax, gbits);
    atomicAdd(ccand, (unsigned long long)M);
    atomicAdd(caccn, (unsigned long long)nacc);
  }
  return ok;
}

}  // namespace

// The parameters of the instance a span belongs to: the kernel argument for a
// single-instance run, else the entry of the run's instance table.
template <bool kBatch>
__device__ __forceinline__ const InstParams& instance_of(const InstParams& one,
                                                         const StepLaunch& SL, int span) {
  if constexpr (kBatch)
    return SL.tab[SL.span_inst[span]];
  else
    return one;
}

// Copies the CTA's instance entry into shared memory (one read of the table per CTA,
// then broadcast reads); returns the copy, or the kernel argument for one instance.
template <bool kBatch>
__device__ __forceinline__ const InstParams& stage_instance(const InstParams& one,
                                                            const StepLaunch& SL, int span,
                                                            InstParams* sh) {
  if constexpr (kBatch) {
    static_assert(sizeof(InstParams) % 4 == 0, "InstParams is copied as words");
    const int* src = reinterpret_cast<const int*>(&SL.tab[SL.span_inst[span]]);
    int* dst = reinterpret_cast<int*>(sh);
    for (int i = threadIdx.x; i < (int)(sizeof(InstParams) / 4); i += blockDim.x)
      dst[i] = src[i];
    __syncthreads();
    return *sh;
  } else {
    return one;
  }
}

// Span `span` of an instance: its cells [c0, c1) and slots [sb0, sb1); with several spans per
// cell also the groups [g0, g1) of the cell that are its share (g1 = -1: all groups).
struct SpanRange {
  int c0, c1, sb0, sb1, g0, g1;
};

__device__ __forceinline__ SpanRange span_range(const InstParams& a, const int* __restrict__ off,
                                                int span) {
  SpanRange s;
  if (a.parts == 1) {
    s.c0 = span * a.cps;
    s.c1 = min(s.c0 + a.cps, a.n_cells);
    s.sb0 = off[s.c0];
    s.sb1 = off[s.c1];
    s.g0 = 0;
    s.g1 = -1;
  } else {
    s.c0 = span / a.parts;
    s.c1 = s.c0 + 1;
    const int j = span - s.c0 * a.parts;
    const int first = off[s.c0], end = off[s.c1];
    const int ng = group_count(end - first, a.G);
    s.g0 = (int)((long long)ng * j / a.parts);
    s.g1 = (int)((long long)ng * (j + 1) / a.parts);
    s.sb0 = s.g0 == ng ? end : first + s.g0 * a.G;
    s.sb1 = s.g1 == ng ? end : first + s.g1 * a.G;
  }
  return s;
}

// Collision models (a.mode): 0 hard spheres, 1 VHS with 0.5 < omega < 1, 2 omega = 1
// (sigma g independent of g).  CTAs per SM the register budget is set for: 3 of 8 warps,
// 6 of 4 warps; the batched 4-warp kernel reads its parameters from shared memory and
// spills at 6 (85 registers), so it is given 5 (no spills, 10 % faster on the
// 256-instance batch).  With the error-keeping moment sums (kF64: 36 binary32 values per
// lane, 124 registers) two and four.
template <bool kBatch, int kWarps, bool kF64>
constexpr int collide_ctas_per_sm() {
  return kF64 ? (kWarps == kAWarps ? 2 : 4) : (kWarps == kAWarps ? 3 : (kBatch ? 5 : 6));
}

template <bool kBatch, int kWarps, bool kF64>
__global__ void __launch_bounds__(kWarps * 32, (collide_ctas_per_sm<kBatch, kWarps, kF64>()))
    k_collide_move(float4* __restrict__ P, const int* __restrict__ off_all,
                   const float* __restrict__ smax_in_all, float* __restrict__ smax_out_all,
                   unsigned long long* __restrict__ ncand_all,
                   unsigned long long* __restrict__ nacc_all, double* __restrict__ acc_all,
                   int* __restrict__ hist, const CellSums sums, const InstParams one,
                   const StepLaunch SL, int* __restrict__ err) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ InstParams sh_inst;
  // unrolling the per-particle loops helps the single run; the batched kernel, which
  // already spills, was 16 % slower with it
  constexpr int kMoveUnroll = kBatch ? 1 : 4;
  // the global span of this CTA: the launch takes spans heaviest first
  const int gspan = SL.span_order ? SL.span_order[blockIdx.x] : (int)blockIdx.x;
  const InstParams& a = stage_instance<kBatch>(one, SL, gspan, &sh_inst);
  const int* __restrict__ off = off_all + a.off_base;
  const float* __restrict__ smax_in = smax_in_all + a.cell_base;
  float* __restrict__ smax_out = smax_out_all + a.cell_base;
  unsigned long long* __restrict__ ncand = ncand_all + a.cell_base;
  unsigned long long* __restrict__ nacc = nacc_all + a.cell_base;
  double* __restrict__ acc = acc_all + (size_t)a.cell_base * kNMom;
  // the instance's step number
  const long long istep = (SL.gstep_dev ? *SL.gstep_dev : SL.gstep) - a.step0;
  const uint32_t step = (uint32_t)istep;
  const bool count_only = SL.count_only != 0;
  const bool sample = !count_only && istep >= a.sample_start;
  const bool collide = !count_only && a.collide != 0;
  const int mode = a.mode;
  const int n_cells = a.n_cells;
  const int cps = a.cps;
  const int cap = a.cap;
  const int G = a.G;
  const int R = SL.rows;
  const StepSmem L = step_smem_layout(n_cells, cps, cap, kWarps, R, kBatch);
  using Acc = typename std::conditional<kF64, double, float>::type;
  int* h = reinterpret_cast<int*>(smem + L.hist);  // the span's rows x n_cells counts
  // per local cell: fixed-point moment sums (slot 0 unused), in a cell's grid
  unsigned long long* cfix = reinterpret_cast<unsigned long long*>(smem + L.cell_acc);
  unsigned long long* ccand = reinterpret_cast<unsigned long long*>(smem + L.cell_cand);
  unsigned long long* caccn = reinterpret_cast<unsigned long long*>(smem + L.cell_accn);
  unsigned* cgmax = reinterpret_cast<unsigned*>(smem + L.cell_gmax);
  int* gfirst = reinterpret_cast<int*>(smem + L.cell_groups);  // cps + 1 group prefix
  int* next_group = gfirst + cps + 1;
  int* cstart = reinterpret_cast<int*>(smem + L.cell_start);     // cps + 1 cell starts
  float* csmax = reinterpret_cast<float*>(smem + L.cell_smax);   // cps (sigma g)_max
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  unsigned char* wmem = smem + L.warps + (size_t)wib * L.per_warp;
  float4* rec = reinterpret_cast<float4*>(wmem + L.w_rec);  // (y, vx, vy, vz) per particle
  // Per particle of the staged group: during a batch of candidates, the lanes whose
  // candidates touch it (bit mask); zero between batches.  Also the queue of wall hits
  // (then restored to zero).
  unsigned* touch = reinterpret_cast<unsigned*>(wmem + L.w_own);
  uint64_t* bar = reinterpret_cast<uint64_t*>(wmem + L.w_bar);

  const int span = gspan - a.span_base;  // the instance's span
  const SpanRange sr = span_range(a, off, span);
  const int c0 = sr.c0, c1 = sr.c1;
  const unsigned lt = (1u << lane) - 1u;
  // rows (span R + r) of the sort matrix; row r counts the r-th half of the slots
  int* row = hist + a.hist_base + (size_t)span * R * n_cells;
  const int sb0 = sr.sb0, sb1 = sr.sb1;
  const int mid = (R > 1) ? sb0 + ((sb1 - sb0) >> 1) : sb1;  // first slot of the second row
  for (int i = threadIdx.x; i < R * n_cells; i += blockDim.x) h[i] = 0;
  // count one particle of slot p in new cell cn
  auto count_cell = [&](int p, int cn) { atomicAdd(&h[(p >= mid ? n_cells : 0) + cn], 1); };
  auto write_rows = [&]() {
    for (int e = threadIdx.x; e < R * n_cells; e += blockDim.x) row[e] = h[e];
  };

  if (count_only) {  // sort into cells: count the cells of the span's slots
    __syncthreads();
    for (int p = sb0 + threadIdx.x; p < sb1; p += blockDim.x)
      count_cell(p, cell_of(P[p].x, n_cells, a.ncf));
    __syncthreads();
    write_rows();
    return;
  }

  for (int i = threadIdx.x; i < cps * kNMom; i += blockDim.x) cfix[i] = 0ull;
  for (int i = threadIdx.x; i < cps; i += blockDim.x) {
    ccand[i] = 0;
    caccn[i] = 0;
    cgmax[i] = 0u;
  }
  if (wib == 0) {  // group prefix over the span's cells, 32 cells at a time
    int base = 0;
    for (int i0 = 0; i0 < c1 - c0; i0 += 32) {
      const int i = i0 + lane;
      int g = 0;
      if (i < c1 - c0) {
        const int s0 = off[c0 + i], s1 = off[c0 + i + 1];
        g = group_count(s1 - s0, G);
        cstart[i] = s0;
        csmax[i] = smax_in[c0 + i];
      }
      int incl = g;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
      }
      if (i < c1 - c0) gfirst[i] = base + incl - g;
      base += __shfl_sync(kFull, incl, 31);
    }
    if (lane == 0) {
      gfirst[c1 - c0] = base;
      cstart[c1 - c0] = off[c1];
      if (!kBatch && sr.g1 >= 0) {  // a share of one cell: its groups are numbered from g0
        gfirst[0] = -sr.g0;
        gfirst[1] = base - sr.g0;
      }
      *next_group = 0;
    }
  }
  for (int i = lane; i < cap; i += 32) touch[i] = 0u;
  if (lane == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  const int n_groups = !kBatch && sr.g1 >= 0 ? sr.g1 - sr.g0 : gfirst[c1 - c0];

  bool bad_bounce = false, cand_fail = false, timeout = false;
  bool inflow_fail = false, mom_range = false;
  uint32_t parity = 0;
  // Groups are handed out by a counter.  Each warp reserves its next group when it
  // starts one, prefetches the next group's records into L2, and issues their bulk copy
  // into its buffer as soon as the current group's records have been read for the last
  // time.  A group is described from shared memory alone (cell starts and group prefix).
  auto cell_of_group = [&](int q, int from) {
    int l = from;
    while (gfirst[l + 1] <= q) ++l;
    return l;
  };
  auto group_slots = [&](int q, int l, int& gs_, int& gn_) {
    const int gi_ = q - gfirst[l];
    const int nc_ = cstart[l + 1] - cstart[l];
    gs_ = cstart[l] + gi_ * G;
    gn_ = (gi_ == gfirst[l + 1] - gfirst[l] - 1) ? nc_ - gi_ * G : G;
  };
  auto issue_copy = [&](int gs_, int gn_) {
    fence_proxy_async_smem();  // earlier generic accesses to rec before the async write
    __syncwarp();
    if (lane == 0) {
      mbar_arrive_expect_tx(bar, (uint32_t)gn_ * 16u);
      bulk_load(rec, P + gs_, (uint32_t)gn_ * 16u, bar);
    }
  };
  // The batched kernel's wall hits wait from group to group in a per-warp queue, so that (but
  // for the span's last ones) every flight has 32 particles: its groups are small (a cell of
  // 50 to 400 particles, a fifth of them hits on average) and flights are most of its
  // instructions.  A waiting particle's record is in its slot in global memory (staging the
  // records in shared memory costs the 8-warp CTA one of its three places on an SM).
  int* wall_slot = reinterpret_cast<int*>(wmem + L.w_wall);
  int n_wall = 0;
  auto fly_queued = [&](int at) {
    const int p = wall_slot[at];
    const float4 r = P[p];
    float yy = r.x, xx = r.y, uy = r.z, zz = r.w;
    if (!fly(yy, xx, uy, zz, a.dt, a.F, a.keys, step, (uint32_t)(p - a.part_base), a.open_top,
             a.u_top, a.p_top, inflow_fail))
      bad_bounce = true;
    P[p] = make_float4(yy, xx, uy, zz);
    count_cell(p, cell_of(yy, n_cells, a.ncf));
  };
  int q_next = 0;
  if (lane == 0) q_next = atomicAdd(next_group, 1);
  q_next = __shfl_sync(kFull, q_next, 0);
  int l_next = 0;
  if (q_next < n_groups) {
    int s_, n_;
    l_next = cell_of_group(q_next, 0);
    group_slots(q_next, l_next, s_, n_);
    issue_copy(s_, n_);
  }
  for (;;) {
    const int q = q_next;
    if (q >= n_groups) break;
    const int lc = l_next;
    const int c = c0 + lc;
    const int gi = q - gfirst[lc];
    const int nc = cstart[lc + 1] - cstart[lc];
    int gs, gn;
    group_slots(q, lc, gs, gn);
    if (lane == 0) q_next = atomicAdd(next_group, 1);
    q_next = __shfl_sync(kFull, q_next, 0);
    int gs_next = 0, gn_next = 0;
    if (q_next < n_groups) {
      l_next = cell_of_group(q_next, lc);
      group_slots(q_next, l_next, gs_next, gn_next);
      if (lane == 0) bulk_prefetch_l2(P + gs_next, (uint32_t)gn_next * 16u);
    }

    // 1. The group's records in shared memory (bulk copy issued beforehand).
    const float smax = csmax[lc];
    if (!mbar_wait(bar, parity)) {
      timeout = true;
      mbar_wait(bar, parity);  // give the copy one more bounded chance to land
      break;
    }
    parity ^= 1u;

    // 2. Moments before the collisions.
    float gmax = 0.0f;
    unsigned laccn = 0;
    uint32_t M = 0;
    LaneSums<Acc> m;
    m.zero();
    if (sample)
#pragma unroll kMoveUnroll
      for (int i = lane; i < gn; i += 32) {
        const float4 r = rec[i];
        m.add(r.y, r.z, r.w);
      }

    // 3. NTC candidates of the group.
    if (collide && gn >= 2)
      ntc_collide(a, rec, touch, gn, nc, c, gi, step, smax, mode, lane, lt, gmax, M, laccn,
                  cand_fail);
    __syncwarp();

    // 4. Moments after the collisions, free flight, store, count the new cell.
    //    A particle whose flight reaches a wall is queued and flown afterwards, 32 such
    //    particles at a time (the free flight is exactly the first leg of the full flight, so
    //    the result is the same).
    if constexpr (kBatch) {
      for (int b = 0; b < gn; b += 32) {
        const int i = b + lane;
        bool hits = false;
        if (i < gn) {
          const float4 r = rec[i];
          if (sample) m.add(r.y, r.z, r.w);
          const float ynew = fadd(r.x, fmul(r.z, a.dt));
          hits = (ynew < 0.0f) || (ynew > 1.0f);
          const float xx = fadd(r.y, fmul(a.F, a.dt));
          P[gs + i] = make_float4(hits ? r.x : ynew, hits ? r.y : xx, r.z, r.w);
          if (!hits) count_cell(gs + i, cell_of(ynew, n_cells, a.ncf));
        }
        const unsigned q = __ballot_sync(kFull, hits);
        if (hits) wall_slot[n_wall + __popc(q & lt)] = gs + i;
        n_wall += __popc(q);
        if (n_wall >= 32) {
          n_wall -= 32;
          __syncwarp();
          fly_queued(n_wall + lane);
          __syncwarp();
        }
      }
    } else {
      int n_hit = 0;
#pragma unroll 4
      for (int b = 0; b < gn; b += 32) {
        const int i = b + lane;
        bool hits = false;
        if (i < gn) {
          const float4 r = rec[i];
          if (sample) m.add(r.y, r.z, r.w);
          const float ynew = fadd(r.x, fmul(r.z, a.dt));
          hits = (ynew < 0.0f) || (ynew > 1.0f);
          if (!hits) {
            const float xx = fadd(r.y, fmul(a.F, a.dt));
            P[gs + i] = make_float4(ynew, xx, r.z, r.w);
            count_cell(gs + i, cell_of(ynew, n_cells, a.ncf));
          }
        }
        const unsigned q = __ballot_sync(kFull, hits);
        if (hits) touch[n_hit + __popc(q & lt)] = (unsigned)i;
        n_hit += __popc(q);
      }
      __syncwarp();
      for (int b = 0; b < n_hit; b += 32) {
        if (b + lane < n_hit) {
          const int i = (int)touch[b + lane];
          const int p = gs + i;
          const float4 r = rec[i];
          float yy = r.x, xx = r.y, uy = r.z, zz = r.w;
          if (!fly(yy, xx, uy, zz, a.dt, a.F, a.keys, step, (uint32_t)(p - a.part_base),
                   a.open_top, a.u_top, a.p_top, inflow_fail))
            bad_bounce = true;
          P[p] = make_float4(yy, xx, uy, zz);
          count_cell(p, cell_of(yy, n_cells, a.ncf));
        }
      }
      __syncwarp();
      for (int i = lane; i < n_hit; i += 32) touch[i] = 0u;
    }
    // the records are read for the last time: bring in the next group's
    if (q_next < n_groups) issue_copy(gs_next, gn_next);
    if (!add_group(m, sample, gn, nc, gmax, M, laccn, cfix + (size_t)lc * kNMom, &cgmax[lc],
                   &ccand[lc], &caccn[lc], lane))
      mom_range = true;
    __syncwarp();
  }
  __syncwarp();
  if (kBatch && lane < n_wall) fly_queued(lane);
  if (bad_bounce) atomicOr(err, kErrBounces);
  if (cand_fail && lane == 0) atomicOr(err, kErrCandidates);
  if (timeout && lane == 0) atomicOr(err, kErrCopyTimeout);
  if (inflow_fail) atomicOr(err, kErrInflow);
  if (mom_range) atomicOr(err, kErrMoments);
  __syncthreads();

  write_rows();
  if (!kBatch && sr.g1 >= 0) {  // the cell's other CTAs add theirs; the scan makes the results
    if (threadIdx.x < 12 && sample && cfix[threadIdx.x + 1])
      atomicAdd(sums.fix + (size_t)c0 * 12 + threadIdx.x, cfix[threadIdx.x + 1]);
    if (threadIdx.x == 12 && cgmax[0]) atomicMax(sums.gmax + c0, cgmax[0]);
    if (threadIdx.x == 13 && ccand[0]) atomicAdd(ncand + c0, ccand[0]);
    if (threadIdx.x == 14 && caccn[0]) atomicAdd(nacc + c0, caccn[0]);
    return;
  }
  for (int c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
    const int lc = c - c0;
    const float gm = __uint_as_float(cgmax[lc]);
    const float sg = (mode == 0) ? gm : fmul(a.cvhs, pow32(gm, a.vexp));
    smax_out[c] = fmaxf(smax_in[c], sg);
    ncand[c] += ccand[lc];
    nacc[c] += caccn[lc];
    if (sample) {
      // count: half before and half after the collisions of every particle of the cell
      const int nc = off[c + 1] - off[c];
      acc[(size_t)c * kNMom] += (double)nc;
      const double grid = __longlong_as_double((long long)(1023 - grid_exponent(nc > 0 ? nc : 1)) << 52);
      for (int k = 1; k < kNMom; ++k)
        acc[(size_t)c * kNMom + k] +=
            0.5 * grid * (double)(long long)cfix[(size_t)lc * kNMom + k];
    }
  }
}

// One warp per span: stable scatter of the span's records into the other buffer.  Slots
// are taken 256 at a time (8 per lane); the loads of the next 256 are issued before the
// current ones are placed, so each lane keeps 8 to 16 records in flight.
//
// A record's place is its cell's running slot (run[]) plus the number of lanes before
// it in its 32-record slice that go to the same cell.  Those "peer" lanes come from a
// small per-warp table of lane masks: each lane ORs its bit into entry (cell mod 256)
// and reads the entry back.  While a slice's cells lie within 256 consecutive values,
// which holds unless a particle crosses more than 255 cells in one step, two cells never
// share an entry and the mask is exactly the set of same-cell lanes; otherwise the slice
// falls back to __match_any_sync.  The table costs a few shared-memory operations per
// slice, where __match_any_sync on ~25 distinct values of 32 (2,000 cells, particles
// crossing ~20 cells a step) was the scatter's bottleneck.  With few warps per SM the
// longer chain of one warp matters more, and the launcher keeps __match_any_sync
// (place_batch_match); both give the same places.
namespace {

constexpr int kScatterUnroll = 8;
constexpr int kMaskSlots = 256;  // entries of the per-warp mask table (a power of two)
constexpr int kMaskWarpsPerSm = 4;

__device__ __forceinline__ void load_batch(float4 (&r)[kScatterUnroll],
                                           const float4* __restrict__ P, int base, int b1,
                                           int lane) {
#pragma unroll
  for (int u = 0; u < kScatterUnroll; ++u) {
    const int p = base + u * 32 + lane;
    if (p < b1) r[u] = P[p];
  }
}

__device__ __forceinline__ bool place_batch_mask(const float4 (&r)[kScatterUnroll],
                                            float4* __restrict__ P2, int* run, unsigned* msk,
                                            int base, int b1,
                                            int n_cells, float ncf, int lo, int hi, int lane,
                                            unsigned lt) {
  int cell[kScatterUnroll];
  unsigned peers[kScatterUnroll];
#pragma unroll
  for (int u = 0; u < kScatterUnroll; ++u) {
    const int p = base + u * 32 + lane;
    cell[u] = (p < b1) ? cell_of(r[u].x, n_cells, ncf) : -1;  // -1: no record
  }
  // lanes of each slice bound for the same cell
#pragma unroll
  for (int u = 0; u < kScatterUnroll; ++u) {
    const int cmin = __reduce_min_sync(kFull, cell[u] >= 0 ? cell[u] : INT_MAX);
    const int cmax = __reduce_max_sync(kFull, cell[u]);
    if (cmax - cmin < kMaskSlots) {  // no two cells share a slot of the mask table
      const int slot = cell[u] & (kMaskSlots - 1);
      if (cell[u] >= 0) atomicOr(&msk[slot], 1u << lane);
      __syncwarp();
      peers[u] = (cell[u] >= 0) ? msk[slot] : 0u;
      __syncwarp();
      if (cell[u] >= 0) msk[slot] = 0u;  // the table is all zero between slices
      __syncwarp();
    } else {
      peers[u] = __match_any_sync(kFull, cell[u]);
    }
  }
  // slots, slice after slice: the first lane of each peer group advances the run
  int d[kScatterUnroll];
#pragma unroll
  for (int u = 0; u < kScatterUnroll; ++u) {
    const bool act = cell[u] >= 0;
    const int first = act ? run[cell[u]] : 0;
    __syncwarp();
    if (act && (peers[u] & lt) == 0) run[cell[u]] = first + __popc(peers[u]);
    __syncwarp();
    d[u] = first + __popc(peers[u] & lt);
  }
  bool bad = false;
#pragma unroll
  for (int u = 0; u < kScatterUnroll; ++u) {
    if (cell[u] >= 0) {
      if (d[u] >= lo && d[u] < hi)
        P2[d[u]] = r[u];
      else
        bad = true;
    }
  }
  return bad;
}

// Ranking with __match_any_sync, slice after slice (fewer instructions in the chain of
// one warp: the better choice when few warps share an SM).
__device__ __forceinline__ bool place_batch_match(const float4 (&r)[kScatterUnroll],
                                                  float4* __restrict__ P2, int* run, int base,
                                                  int b1, int n_cells, float ncf, int lo, int hi,
                                                  int lane, unsigned lt) {
  bool bad = false;
#pragma unroll
  for (int u = 0; u < kScatterUnroll; ++u) {
    const int p = base + u * 32 + lane;
    const bool act = p < b1;
    const int cell = act ? cell_of(r[u].x, n_cells, ncf) : -1;
    const unsigned peers = __match_any_sync(kFull, cell);
    const int first = act ? run[cell] : 0;
    __syncwarp();
    if (act && (peers & lt) == 0) run[cell] = first + __popc(peers);
    __syncwarp();
    if (act) {
      const int d = first + __popc(peers & lt);
      if (d >= lo && d < hi)
        P2[d] = r[u];
      else
        bad = true;
    }
  }
  return bad;
}

}  // namespace

template <bool kBatch, bool kMask>
__global__ void __launch_bounds__(kBWarpsMax * 32)
    k_scatter_spans(const float4* __restrict__ P, float4* __restrict__ P2,
                    const int* __restrict__ off_cur_all, const int* __restrict__ off_new_all,
                    const int* __restrict__ hist, const InstParams one, const StepLaunch SL,
                    int* __restrict__ err) {
  constexpr int kBatch2 = 32 * kScatterUnroll;
  extern __shared__ int sh_run[];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int unit = blockIdx.x * (blockDim.x >> 5) + wib;  // (span, row of the span)
  const int R = SL.rows;
  const int gspan = unit / R, sub = unit - gspan * R;
  if (gspan >= SL.n_spans_total) return;
  const InstParams& a = instance_of<kBatch>(one, SL, gspan);
  const int n_cells = a.n_cells;
  const int span = gspan - a.span_base;
  const int* __restrict__ off_cur = off_cur_all + a.off_base;
  const int* __restrict__ off_new = off_new_all + a.off_base;
  int* run = sh_run + (size_t)wib * (SL.max_cells + kMaskSlots);
  unsigned* msk = reinterpret_cast<unsigned*>(run + SL.max_cells);
  for (int i = lane; i < kMaskSlots; i += 32) msk[i] = 0u;
  const int* row = hist + a.hist_base + ((size_t)span * R + sub) * n_cells;
  for (int c = lane; c < n_cells; c += 32) run[c] = off_new[c] + row[c];
  __syncwarp();
  const SpanRange sr = span_range(a, off_cur, span);
  const int sb0 = sr.sb0, sb1 = sr.sb1;
  const int mid = (R > 1) ? sb0 + ((sb1 - sb0) >> 1) : sb1;
  const int b0 = (sub == 0) ? sb0 : mid;
  const int b1 = (sub == 0) ? mid : sb1;
  const int lo = a.part_base, hi = a.part_base + a.n_part;  // the instance's slots
  const unsigned lt = (1u << lane) - 1u;
  bool bad = false;
  float4 ra[kScatterUnroll], rb[kScatterUnroll];
  load_batch(ra, P, b0, b1, lane);
  for (int base = b0; base < b1; base += 2 * kBatch2) {
    load_batch(rb, P, base + kBatch2, b1, lane);
    bad |= kMask ? place_batch_mask(ra, P2, run, msk, base, b1, n_cells, a.ncf, lo, hi, lane, lt)
                 : place_batch_match(ra, P2, run, base, b1, n_cells, a.ncf, lo, hi, lane, lt);
    if (base + kBatch2 >= b1) break;
    load_batch(ra, P, base + 2 * kBatch2, b1, lane);
    bad |= kMask ? place_batch_mask(rb, P2, run, msk, base + kBatch2, b1, n_cells, a.ncf, lo, hi,
                                    lane, lt)
                 : place_batch_match(rb, P2, run, base + kBatch2, b1, n_cells, a.ncf, lo, hi,
                                     lane, lt);
  }
  if (bad) atomicOr(err, kErrSort);
}

// One CTA of kCoopWarps warps per (span, row): the stable scatter of the row's records
// into the other buffer, kCoopWarps * 64 records per round.  In a round warp w takes the
// 64 consecutive records [base + 64 w, base + 64 w + 64) as two 32-record slices; a
// record's place is
//   run[cell]                      the cell's next slot after the earlier rounds,
// + sum over warps w' < w of       the round's records of w' bound for the same cell,
// + its rank among its warp's records bound for the same cell (__match_any_sync within
//   its slice, plus the first slice's count for a record of the second).
// Each warp publishes its per-cell counts in its own row of a table tagged with the
// round number (no clearing between rounds); after the places are taken, every warp
// adds its counts into run[].  All warps of the CTA work on one span at once: for
// short spans of small instances (a batch) this beats a warp per span, whose time is
// its span's ranking chain plus a pass over all of the instance's cells to set up run[].
// Shared memory: run[n_cells] and the table kCoopWarps x n_cells, so it is used while
// that leaves room for 4 CTAs per SM.
constexpr int kCoopWarps = 8;
constexpr size_t kCoopSmemMax = 48 * 1024;
static_assert(kCoopCells == (int)(kCoopSmemMax / sizeof(int) / (kCoopWarps + 1)), "");
constexpr int kCoopPer = (kCoopCells + kCoopWarps * 32 - 1) / (kCoopWarps * 32);  // cells per thread

template <bool kBatch, int kSlices>
__global__ void __launch_bounds__(kCoopWarps * 32)
    k_scatter_coop(const float4* __restrict__ P, float4* __restrict__ P2,
                   const int* __restrict__ off_cur_all, const int* __restrict__ count_all,
                   int* __restrict__ off_new_all, const int* __restrict__ hist, const InstParams one, const StepLaunch SL,
                   int* __restrict__ err) {
  extern __shared__ int sh_coop[];
  const int lane = threadIdx.x & 31;
  const int w = threadIdx.x >> 5;
  const int R = SL.rows;
  const int gspan = blockIdx.x / R, sub = blockIdx.x - gspan * R;
  const InstParams& a = instance_of<kBatch>(one, SL, gspan);
  const int n_cells = a.n_cells;
  const int span = gspan - a.span_base;
  const int* __restrict__ off_cur = off_cur_all + a.off_base;
  const int* __restrict__ count = count_all + a.cell_base;
  int* run = sh_coop;
  int* tab = sh_coop + n_cells;  // tab[w' * n_cells + c] = (round << 8) | count
  const int* row = hist + a.hist_base + ((size_t)span * R + sub) * n_cells;
  {
    // The new cell offsets (prefix of the cells' counts) on the way to the run's first places:
    // a thread takes kCoopPer consecutive cells.  Every CTA forms them, the instance's first
    // one writes them down for the next step.  The warps' totals pass through the first entries
    // of the table, inverted: a negative entry is of no round.  (32 bytes of their own took the
    // CTA of 1,365 cells over a quarter of the SM's 196 KB split and cost it L1: 25,000 particles
    // per cell 262 -> 277 us.)
    int n[kCoopPer], before[kCoopPer], incl = 0;
    const int cb = threadIdx.x * kCoopPer;
#pragma unroll
    for (int k = 0; k < kCoopPer; ++k) {
      n[k] = cb + k < n_cells ? count[cb + k] : 0;
      before[k] = cb + k < n_cells ? row[cb + k] : 0;
    }
#pragma unroll
    for (int k = 0; k < kCoopPer; ++k) incl += n[k];
    const int mine = incl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) tab[w] = ~incl;
    for (int i = kCoopWarps + threadIdx.x; i < kCoopWarps * n_cells; i += blockDim.x) tab[i] = -1;
    __syncthreads();
    int at = a.part_base + incl - mine;
#pragma unroll
    for (int v = 0; v < kCoopWarps; ++v) at += v < w ? ~tab[v] : 0;
    int* __restrict__ off_new = blockIdx.x == a.span_base * R ? off_new_all + a.off_base : nullptr;
#pragma unroll
    for (int k = 0; k < kCoopPer; ++k) {
      if (cb + k < n_cells) {
        run[cb + k] = at + before[k];
        if (off_new) off_new[cb + k] = at;
      }
      at += n[k];
      if (off_new && cb + k == n_cells - 1) off_new[n_cells] = at;
    }
    // Graph replay: the step's collide/move pass has finished reading the step number.
    if (SL.gstep_dev != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *SL.gstep_dev += 1;
  }
  const SpanRange sr = span_range(a, off_cur, span);
  const int sb0 = sr.sb0, sb1 = sr.sb1;
  const int mid = (R > 1) ? sb0 + ((sb1 - sb0) >> 1) : sb1;
  const int b0 = (sub == 0) ? sb0 : mid;
  const int b1 = (sub == 0) ? mid : sb1;
  const int lo = a.part_base, hi = a.part_base + a.n_part;  // the instance's slots
  const unsigned lt = (1u << lane) - 1u;
  // A round: warp w takes the 32 kSlices records [base + 32 kSlices w, ...) as kSlices
  // slices of 32 (one record per lane each); two barriers per round.
  static_assert(kSlices == 1 || kSlices == 2, "one or two slices per warp and round");
  constexpr int kWarpRecs = 32 * kSlices;
  constexpr int kRound = kCoopWarps * kWarpRecs;
  constexpr int kAhead = 6 / kSlices;  // rounds of records in flight per lane (6 records)
  float4 r[kAhead][kSlices];
#pragma unroll
  for (int u = 0; u < kAhead; ++u)
#pragma unroll
    for (int sl = 0; sl < kSlices; ++sl) {
      const int p = b0 + u * kRound + w * kWarpRecs + sl * 32 + lane;
      if (p < b1) r[u][sl] = P[p];
    }
  bool bad = false;
  int* tw = tab + w * n_cells;  // this warp's counts of the round, per cell
  __syncthreads();
  int round = 0;
  for (int base = b0; base < b1; base += kAhead * kRound) {
#pragma unroll
    for (int u = 0; u < kAhead; ++u, ++round) {
      const int rb = base + u * kRound;
      if (rb >= b1) break;  // uniform across the CTA
      const int pw = rb + w * kWarpRecs + lane;
      float4 rec[kSlices];
      int cell[kSlices], prev[kSlices];
      unsigned peers[kSlices];
#pragma unroll
      for (int sl = 0; sl < kSlices; ++sl) {
        const int p = pw + 32 * sl;
        rec[sl] = r[u][sl];
        // the record kAhead rounds later into this register
        if (p + kAhead * kRound < b1) r[u][sl] = P[p + kAhead * kRound];
        cell[sl] = (p < b1) ? cell_of(rec[sl].x, n_cells, a.ncf) : -1;
        peers[sl] = __match_any_sync(kFull, cell[sl]);
      }
      const int tag = round << 8;
      // the warp's count per cell, slice after slice: a slice's lanes find how many of the
      // earlier slices precede them in their cell, and its leaders store the running count
#pragma unroll
      for (int sl = 0; sl < kSlices; ++sl) {
        prev[sl] = 0;
        if (sl > 0) {
          __syncwarp();
          if (cell[sl] >= 0) {
            const int e = tw[cell[sl]];
            prev[sl] = ((e >> 8) == round) ? (e & 0xff) : 0;
          }
          __syncwarp();
        }
        if (cell[sl] >= 0 && (peers[sl] & lt) == 0u)
          tw[cell[sl]] = tag | (prev[sl] + __popc(peers[sl]));
      }
      __syncthreads();
#pragma unroll
      for (int sl = 0; sl < kSlices; ++sl) {
        if (cell[sl] < 0) continue;
        int before = prev[sl] + __popc(peers[sl] & lt);
#pragma unroll
        for (int v = 0; v < kCoopWarps - 1; ++v) {
          if (v < w) {
            const int e = tab[v * n_cells + cell[sl]];
            if ((e >> 8) == round) before += e & 0xff;
          }
        }
        const int d = run[cell[sl]] + before;
        if (d >= lo && d < hi)
          P2[d] = rec[sl];
        else
          bad = true;
      }
      __syncthreads();
#pragma unroll
      for (int sl = 0; sl < kSlices; ++sl)
        if (cell[sl] >= 0 && (peers[sl] & lt) == 0u) atomicAdd(&run[cell[sl]], __popc(peers[sl]));
    }
  }
  if (bad) atomicOr(err, kErrSort);
}

// The results of a step in cell c of an instance whose cells are shared by several CTAs
// (as the one CTA of a cell writes them otherwise).
__device__ __forceinline__ void finish_cell(const CellSums& S, const InstParams& a,
                                            const StepLaunch& SL, int c) {
  if (a.parts == 1 || SL.count_only) return;
  const long long istep = (SL.gstep_dev ? *SL.gstep_dev : SL.gstep) - a.step0;
  const float gm = __uint_as_float(S.gmax[c]);
  S.gmax[c] = 0u;
  const float sg = (a.mode == 0) ? gm : fmul(a.cvhs, pow32(gm, a.vexp));
  S.smax_out[c] = fmaxf(S.smax_in[c], sg);
  if (istep < a.sample_start) return;
  const int nc = S.off[c + 1] - S.off[c];
  double* acc = S.acc + (size_t)c * kNMom;
  acc[0] += (double)nc;
  const double grid =
      __longlong_as_double((long long)(1023 - grid_exponent(nc > 0 ? nc : 1)) << 52);
  unsigned long long* fix = S.fix + (size_t)c * 12;
  unsigned long long q[12];
  double sum[12];  // (all loads on their way before the first use)
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    q[k] = fix[k];
    sum[k] = acc[k + 1];
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    acc[k + 1] = sum[k] + 0.5 * grid * (double)(long long)q[k];
    fix[k] = 0ull;
  }
}

// Per instance and cell c: row r of the sort matrix <- sum over rows r' < r (the spans
// before), count[c] <- total.  Block (kScanCells, 1024 / kScanCells): x = cell
// within a chunk, y = one of the contiguous row segments; grid (cell chunks, instances).  Chunks
// of 16 cells (two sectors of a row) give 2,000 cells 125 CTAs instead of 63 of twice the rows
// per thread (20.7 -> 14 us at 2,000 rows).  They are taken while they fit one wave of CTAs (2,800
// cells x 934 rows: 16-cell chunks 15.8 us, 32 cells 12.5; 2,400 x 1,200: 12.4, 14.3) and do not
// straddle sectors, or the rows are short (1,403 x 1,403: 23.3, 18.7; 2,900 x 1,450: 37.9, 21.4;
// but 1,001 x 1,001: 10.2, 12.4).
template <bool kBatch, int kScanCells>
__global__ void __launch_bounds__(1024)
    k_scan_spans(int* __restrict__ hist, int* __restrict__ count_all, const CellSums sums,
                 const InstParams one, const StepLaunch SL) {
  __shared__ int seg_tot[(1024 / kScanCells)][kScanCells + 1];
  const InstParams& a = kBatch ? SL.tab[blockIdx.y] : one;
  const int n_cells = a.n_cells;
  if ((int)blockIdx.x * kScanCells >= n_cells) return;
  const int n_rows = a.n_spans * SL.rows;
  int* __restrict__ m = hist + a.hist_base;
  int* __restrict__ count = count_all + a.cell_base;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int c = blockIdx.x * kScanCells + tx;
  const int seg = (n_rows + (1024 / kScanCells) - 1) / (1024 / kScanCells);
  const int r0 = min(n_rows, ty * seg);
  const int r1 = min(n_rows, r0 + seg);
  int s = 0;
  if (c < n_cells) {
    int r = r0;
    for (; r + 8 <= r1; r += 8) {
      int v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = m[(size_t)(r + u) * n_cells + c];
#pragma unroll
      for (int u = 0; u < 8; ++u) s += v[u];
    }
    for (; r < r1; ++r) s += m[(size_t)r * n_cells + c];
  }
  seg_tot[ty][tx] = s;
  __syncthreads();
  if (ty == 0) {
    int run = 0;
    for (int k = 0; k < (1024 / kScanCells); ++k) {
      const int v = seg_tot[k][tx];
      seg_tot[k][tx] = run;
      run += v;
    }
    if (c < n_cells) {
      count[c] = run;
      if constexpr (!kBatch) finish_cell(sums, a, SL, c);
    }
  }
  __syncthreads();
  if (c < n_cells) {
    int run = seg_tot[ty][tx];
    int r = r0;
    for (; r + 8 <= r1; r += 8) {
      int v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = m[(size_t)(r + u) * n_cells + c];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        m[(size_t)(r + u) * n_cells + c] = run;
        run += v[u];
      }
    }
    for (; r < r1; ++r) {
      const size_t i = (size_t)r * n_cells + c;
      const int v = m[i];
      m[i] = run;
      run += v;
    }
  }
}

// The same prefix for runs whose instances have at most kScanColsMaxRows rows (batches
// and pools of small instances): one thread per cell walks its column of the matrix, 32
// rows of loads in flight at a time; blocks of 64 cells, grid (cell chunks, instances).
// The block-per-32-cells kernel above would spend most of its 1,024 threads and its two
// CTA barriers on a handful of rows per instance (0.049 against 0.022 ms per step on the
// 256-instance batch).
constexpr int kScanColsMaxRows = 256;
constexpr int kScanColsCells = 64;
constexpr int kScanColsDepth = 32;

template <bool kBatch>
__global__ void __launch_bounds__(kScanColsCells)
    k_scan_cols(int* __restrict__ hist, int* __restrict__ count_all, const CellSums sums,
                const InstParams one, const StepLaunch SL) {
  const InstParams& a = kBatch ? SL.tab[blockIdx.y] : one;
  const int n_cells = a.n_cells;
  const int c = blockIdx.x * kScanColsCells + threadIdx.x;
  if (c >= n_cells) return;
  const int n_rows = a.n_spans * SL.rows;
  int* __restrict__ m = hist + a.hist_base + c;  // m[r n_cells]: row r of this column
  int run = 0;
  for (int r = 0; r < n_rows; r += kScanColsDepth) {
    int v[kScanColsDepth];
#pragma unroll
    for (int u = 0; u < kScanColsDepth; ++u)
      if (r + u < n_rows) v[u] = m[(size_t)(r + u) * n_cells];
#pragma unroll
    for (int u = 0; u < kScanColsDepth; ++u)
      if (r + u < n_rows) {
        m[(size_t)(r + u) * n_cells] = run;
        run += v[u];
      }
  }
  count_all[a.cell_base + c] = run;
  if constexpr (!kBatch) finish_cell(sums, a, SL, c);
}

// Per instance (one CTA each): off_new[c] = first global slot of cell c,
// off_new[n_cells] = end of the instance's slots.  For the scatter with a warp per span, which
// would take 5 us to form the offsets of 2,000 cells in every warp (k_scatter_coop does so in
// every CTA, for 0.1 us).
template <bool kBatch>
__global__ void __launch_bounds__(1024)
    k_offsets_cells(const int* __restrict__ count_all, int* __restrict__ off_new_all,
                    const InstParams one, const StepLaunch SL) {
  __shared__ int wsum[32];
  const InstParams& a = kBatch ? SL.tab[blockIdx.x] : one;
  const int n_cells = a.n_cells;
  const int* __restrict__ count = count_all + a.cell_base;
  int* __restrict__ offset = off_new_all + a.off_base;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int per = (n_cells + 1023) / 1024;
  const int cb = t * per;
  const int ce = min(n_cells, cb + per);
  int mine = 0;
  for (int c = cb; c < ce; ++c) mine += count[c];
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) wsum[w] = incl;
  __syncthreads();
  const int before = __reduce_add_sync(kFull, lane < w ? wsum[lane] : 0);
  int run = a.part_base + before + incl - mine;
  for (int c = cb; c < ce; ++c) {
    offset[c] = run;
    run += count[c];
  }
  if (t == 1023) offset[n_cells] = run;
  // Graph replay: the step's collide/move pass has finished reading the step number.
  if (SL.gstep_dev != nullptr && blockIdx.x == 0 && t == 0) *SL.gstep_dev += 1;
}

__global__ void k_set_counter(long long* counter, long long value) { *counter = value; }

__global__ void __launch_bounds__(256)
    k_admit_cells(const InstParams* __restrict__ tab, int* __restrict__ off_all,
                  float* __restrict__ smax_all, unsigned long long* __restrict__ ncand_all,
                  unsigned long long* __restrict__ nacc_all, double* __restrict__ acc_all) {
  const InstParams& a = tab[blockIdx.x];
  const int n_cells = a.n_cells;
  const int ppc = a.n_part / n_cells;
  int* off = off_all + a.off_base;
  for (int c = threadIdx.x; c <= n_cells; c += blockDim.x) off[c] = a.part_base + c * ppc;
  for (int c = threadIdx.x; c < n_cells; c += blockDim.x) {
    smax_all[a.cell_base + c] = a.smax0;
    ncand_all[a.cell_base + c] = 0ull;
    nacc_all[a.cell_base + c] = 0ull;
  }
  double* acc = acc_all + (size_t)a.cell_base * kNMom;
  for (int i = threadIdx.x; i < n_cells * kNMom; i += blockDim.x) acc[i] = 0.0;
}

__global__ void __launch_bounds__(256)
    k_channel_sums(const InstParams* __restrict__ tab, const double* __restrict__ acc_all,
                   double* __restrict__ out) {
  __shared__ double part[2][8];
  const InstParams& a = tab[blockIdx.x];
  const double* acc = acc_all + (size_t)a.cell_base * kNMom;
  double n = 0.0, u = 0.0;
  for (int c = threadIdx.x; c < a.n_cells; c += blockDim.x) {
    n += acc[(size_t)c * kNMom + 0];
    u += acc[(size_t)c * kNMom + 1];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    n += __shfl_xor_sync(0xffffffffu, n, o);
    u += __shfl_xor_sync(0xffffffffu, u, o);
  }
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    part[0][w] = n;
    part[1][w] = u;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sn = 0.0, su = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
      sn += part[0][k];
      su += part[1][k];
    }
    out[2 * a.id] = sn;
    out[2 * a.id + 1] = su;
  }
}

// Records <-> four arrays (y, vx, vy, vz), for the state accessors.  A thread per record and no
// stride over the grid: from 2^30 records on, a record's index plus the grid's size passes 2^31.
__global__ void k_unpack(const float4* __restrict__ P, float* __restrict__ y,
                         float* __restrict__ vx, float* __restrict__ vy, float* __restrict__ vz,
                         int N) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  const float4 r = P[p];
  if (y) y[p] = r.x;
  if (vx) vx[p] = r.y;
  if (vy) vy[p] = r.z;
  if (vz) vz[p] = r.w;
}

// An instance's cell data (offsets relative to its first slot) and the error word in one block.
__global__ void k_gather_cells(const int* __restrict__ off, int base,
                               const float* __restrict__ smax,
                               const unsigned long long* __restrict__ ncand,
                               const unsigned long long* __restrict__ nacc,
                               const int* __restrict__ err, int n_cells, char* block) {
  const CellBlock B(n_cells);
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c > n_cells) return;
  reinterpret_cast<int*>(block + B.offset)[c] = off[c] - base;
  if (c == n_cells) {
    *reinterpret_cast<int*>(block + B.err) = *err;
    return;
  }
  reinterpret_cast<unsigned long long*>(block + B.ncand)[c] = ncand[c];
  reinterpret_cast<unsigned long long*>(block + B.nacc)[c] = nacc[c];
  reinterpret_cast<float*>(block + B.smax)[c] = smax[c];
}

// Pack four arrays into records; y is moved onto the nearest wall if outside [0, 1].
__global__ void k_pack(const float* __restrict__ y, const float* __restrict__ vx,
                       const float* __restrict__ vy, const float* __restrict__ vz,
                       float4* __restrict__ P, int N) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  const float v = y[p];
  const float yc = (v >= 0.0f) ? ((v <= 1.0f) ? v : 1.0f) : 0.0f;
  P[p] = make_float4(yc, vx[p], vy[p], vz[p]);
}

// ---------------------------------------------------------------------------

cudaError_t launch_collide_move(float4* P, const int* off, const float* smax_in,
                                float* smax_out, unsigned long long* ncand,
                                unsigned long long* nacc, double* acc, int* hist,
                                const CellSums& sums, const InstParams& one,
                                const StepLaunch& L, int* err, cudaStream_t st) {
  const bool batch = L.n_inst > 1;
  bool small = L.warps == kAWarpsSmall;
  // an 8-warp CTA that fits without the batch's wall queues (as the host checked) but not with
  // them gives way to the 4-warp one, which fits at every accepted size
  if (!small && step_smem_layout(L.max_cells, L.max_cps, L.max_cap, kAWarps, L.rows, batch).total >
                    kStepSmemMax)
    small = true;
  const int warps = small ? kAWarpsSmall : kAWarps;
  const StepSmem S = step_smem_layout(L.max_cells, L.max_cps, L.max_cap, warps, L.rows, batch);
  const dim3 block(warps * 32);
#define DSMC_COLLIDE(B, W, D)                                                       \
  k_collide_move<B, W, D><<<L.n_spans_total, block, S.total, st>>>(               \
      P, off, smax_in, smax_out, ncand, nacc, acc, hist, sums, one, L, err)
#define DSMC_COLLIDE_SHAPE(B, D)   \
  do {                             \
    if (small)                     \
      DSMC_COLLIDE(B, kAWarpsSmall, D); \
    else                           \
      DSMC_COLLIDE(B, kAWarps, D); \
  } while (0)
  const bool f64 = L.accum == DSMC_ACCUM_FP64;
  if (L.n_inst == 1) {
    if (f64)
      DSMC_COLLIDE_SHAPE(false, true);
    else
      DSMC_COLLIDE_SHAPE(false, false);
  } else {
    if (f64)
      DSMC_COLLIDE_SHAPE(true, true);
    else
      DSMC_COLLIDE_SHAPE(true, false);
  }
#undef DSMC_COLLIDE_SHAPE
#undef DSMC_COLLIDE
  return cudaGetLastError();
}

int scatter_spans_warps(int n_cells) {
  size_t w = kStepSmemMax / ((size_t)(n_cells + kMaskSlots) * sizeof(int));
  if (w > (size_t)kBWarpsMax) w = kBWarpsMax;
  return w < 1 ? 1 : (int)w;
}

static size_t scatter_coop_smem(int max_cells) {
  return (size_t)(kCoopWarps + 1) * (size_t)max_cells * sizeof(int);
}

cudaError_t launch_scatter_spans(const float4* P, float4* P2, const int* off_cur,
                                 const int* count, int* off_new, const int* hist,
                                 const InstParams& one, const StepLaunch& L, int* err,
                                 cudaStream_t st) {
  if (scatter_forms_offsets(L)) {  // a CTA per (span, row)
    const size_t coop = scatter_coop_smem(L.max_cells);
    const int units = L.n_spans_total * L.rows;
    // two slices per warp and round once the rows average 4,096 records (the batch's
    // tuned spans: 0.328 -> 0.30 ms); one for shorter rows (small runs' 1,024-particle
    // spans, where fewer, longer rounds were slower)
    const bool two = L.n_part_total >= 4096LL * units;
#define DSMC_COOP(B, S)                                                                  \
  k_scatter_coop<B, S><<<units, kCoopWarps * 32, coop, st>>>(P, P2, off_cur, count, off_new, \
                                                             hist, one, L, err)
    if (L.n_inst == 1) {
      if (two) DSMC_COOP(false, 2); else DSMC_COOP(false, 1);
    } else {
      if (two) DSMC_COOP(true, 2); else DSMC_COOP(true, 1);
    }
#undef DSMC_COOP
    return cudaGetLastError();
  }
  const int wpb = scatter_spans_warps(L.max_cells);
  const size_t smem = (size_t)wpb * (L.max_cells + kMaskSlots) * sizeof(int);
  const int units = L.n_spans_total * L.rows;
  const int blocks = (units + wpb - 1) / wpb;
  // the mask-table ranking once at least kMaskWarpsPerSm scatter warps share an SM
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const bool mask = units >= kMaskWarpsPerSm * sms;
#define DSMC_SCATTER(B, M)                                                                   \
  k_scatter_spans<B, M><<<blocks, wpb * 32, smem, st>>>(P, P2, off_cur, off_new, hist, one, L, \
                                                        err)
  if (L.n_inst == 1) {
    if (mask)
      DSMC_SCATTER(false, true);
    else
      DSMC_SCATTER(false, false);
  } else {
    if (mask)
      DSMC_SCATTER(true, true);
    else
      DSMC_SCATTER(true, false);
  }
#undef DSMC_SCATTER
  return cudaGetLastError();
}

cudaError_t launch_scan_spans(int* hist, int* count, const CellSums& sums, const InstParams& one,
                              const StepLaunch& L, cudaStream_t st) {
  if ((long long)L.max_spans * L.rows <= kScanColsMaxRows) {
    const dim3 grid((L.max_cells + kScanColsCells - 1) / kScanColsCells, L.n_inst);
    if (L.n_inst == 1)
      k_scan_cols<false><<<grid, kScanColsCells, 0, st>>>(hist, count, sums, one, L);
    else
      k_scan_cols<true><<<grid, kScanColsCells, 0, st>>>(hist, count, sums, one, L);
    return cudaGetLastError();
  }
  const bool wide = L.max_cells > 16 * 152 || (L.max_cells > 1200 && L.max_cells % 16 != 0);
  const int cells = wide ? 32 : 16;
  const dim3 grid((L.max_cells + cells - 1) / cells, L.n_inst), block(cells, 1024 / cells);
#define DSMC_SCAN(B, C) k_scan_spans<B, C><<<grid, block, 0, st>>>(hist, count, sums, one, L)
  if (L.n_inst == 1) {
    if (wide) DSMC_SCAN(false, 32); else DSMC_SCAN(false, 16);
  } else {
    if (wide) DSMC_SCAN(true, 32); else DSMC_SCAN(true, 16);
  }
#undef DSMC_SCAN
  return cudaGetLastError();
}

bool scatter_forms_offsets(const StepLaunch& L) {
  return L.max_cells <= kCoopCells;
}

cudaError_t launch_offsets_cells(const int* count, int* off_new, const InstParams& one,
                                 const StepLaunch& L, cudaStream_t st) {
  if (L.n_inst == 1)
    k_offsets_cells<false><<<1, 1024, 0, st>>>(count, off_new, one, L);
  else
    k_offsets_cells<true><<<L.n_inst, 1024, 0, st>>>(count, off_new, one, L);
  return cudaGetLastError();
}

cudaError_t launch_set_counter(long long* counter, long long value, cudaStream_t st) {
  k_set_counter<<<1, 1, 0, st>>>(counter, value);
  return cudaGetLastError();
}

cudaError_t launch_admit_cells(const InstParams* tab, int n, int* off, float* smax,
                               unsigned long long* ncand, unsigned long long* nacc,
                               double* acc, cudaStream_t st) {
  k_admit_cells<<<n, 256, 0, st>>>(tab, off, smax, ncand, nacc, acc);
  return cudaGetLastError();
}

cudaError_t launch_channel_sums(const InstParams* tab, int n, const double* acc, double* out,
                                cudaStream_t st) {
  k_channel_sums<<<n, 256, 0, st>>>(tab, acc, out);
  return cudaGetLastError();
}

cudaError_t launch_gather_cells(const int* off, int base, const float* smax,
                                const unsigned long long* ncand, const unsigned long long* nacc,
                                const int* err, int n_cells, char* block, cudaStream_t st) {
  k_gather_cells<<<(n_cells + 1 + 255) / 256, 256, 0, st>>>(off, base, smax, ncand, nacc, err,
                                                           n_cells, block);
  return cudaGetLastError();
}

cudaError_t launch_unpack(const float4* P, float* y, float* vx, float* vy, float* vz, int N,
                          cudaStream_t st) {
  const int blocks = (N + 255) / 256;
  k_unpack<<<blocks > 0 ? blocks : 1, 256, 0, st>>>(P, y, vx, vy, vz, N);
  return cudaGetLastError();
}

cudaError_t launch_pack(const float* y, const float* vx, const float* vy, const float* vz,
                        float4* P, int N, cudaStream_t st) {
  const int blocks = (N + 255) / 256;
  k_pack<<<blocks > 0 ? blocks : 1, 256, 0, st>>>(y, vx, vy, vz, P, N);
  return cudaGetLastError();
}

cudaError_t set_step_smem_limits(size_t a_bytes, size_t b_bytes) {
  const void* collide[8] = {(const void*)k_collide_move<false, kAWarps, false>,
                            (const void*)k_collide_move<true, kAWarps, false>,
                            (const void*)k_collide_move<false, kAWarpsSmall, false>,
                            (const void*)k_collide_move<true, kAWarpsSmall, false>,
                            (const void*)k_collide_move<false, kAWarps, true>,
                            (const void*)k_collide_move<true, kAWarps, true>,
                            (const void*)k_collide_move<false, kAWarpsSmall, true>,
                            (const void*)k_collide_move<true, kAWarpsSmall, true>};
  for (const void* f : collide) {
    const cudaError_t e =
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)a_bytes);
    if (e != cudaSuccess) return e;
  }
  const void* scatter[8] = {(const void*)k_scatter_spans<false, false>,
                            (const void*)k_scatter_spans<false, true>,
                            (const void*)k_scatter_spans<true, false>,
                            (const void*)k_scatter_spans<true, true>,
                            (const void*)k_scatter_coop<false, 1>,
                            (const void*)k_scatter_coop<true, 1>,
                            (const void*)k_scatter_coop<false, 2>,
                            (const void*)k_scatter_coop<true, 2>};
  for (const void* f : scatter) {
    const cudaError_t e =
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b_bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace dsmc

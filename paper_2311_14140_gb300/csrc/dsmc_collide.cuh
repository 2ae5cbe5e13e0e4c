// dsmc_collide.cuh -- device code of one collision group shared by the step kernels: the
// moment sums, the NTC candidates of a group whose records are staged in shared memory,
// and the exact combination of group totals.
#pragma once

#include <stdint.h>

#include "dsmc_device.cuh"
#include "dsmc_internal.h"

namespace dsmc {

constexpr unsigned kFull = 0xffffffffu;

// sin(2 pi v) and cos(2 pi v) for v in [0, 1], binary32: 4 v = n + r with n the nearest
// integer (4 v, n and r exact), theta = r pi/2 in [-pi/4, pi/4], the Taylor series of
// sin theta through theta^9 and of cos theta through theta^10 (truncation below 2e-9 on
// that range) by Horner's rule, then n quarter turns (selects, not branches: lanes of a
// warp fall in different quadrants).
__device__ __forceinline__ void sincos_turn(float v, float& sn, float& cs) {
  const float t = fmul(4.0f, v);
  const float n = floorf(fadd(t, 0.5f));
  const float r = fsub(t, n);
  const float th = fmul(r, 0x1.921fb6p+0f);  // pi/2
  const float t2 = fmul(th, th);
  float ps = 0x1.71de3ap-19f;                  // 1/9!
  ps = fsub(fmul(ps, t2), 0x1.a01a02p-13f);    // 1/7!
  ps = fadd(fmul(ps, t2), 0x1.111112p-7f);     // 1/5!
  ps = fsub(fmul(ps, t2), 0x1.555556p-3f);     // 1/3!
  ps = fmul(ps, t2);
  const float s = fadd(th, fmul(th, ps));
  float pc = -0x1.27e4fcp-22f;                 // -1/10!
  pc = fadd(fmul(pc, t2), 0x1.a01a02p-16f);    // 1/8!
  pc = fsub(fmul(pc, t2), 0x1.6c16c2p-10f);    // 1/6!
  pc = fadd(fmul(pc, t2), 0x1.555556p-5f);     // 1/4!
  pc = fsub(fmul(pc, t2), 0.5f);
  const float c = fadd(1.0f, fmul(t2, pc));
  const int q = ((int)n) & 3;  // quarter turns: swap for odd q, signs by quadrant
  const float a = (q & 1) ? c : s, b = (q & 1) ? s : c;
  sn = (q & 2) ? -a : a;
  cs = ((q + 1) & 2) ? -b : b;
}

// VHS acceptance threshold on the relative speed (sigma g > u (sigma g)_max written as
// g > thr): thr = exp((ln(u smax) - ln cvhs) / (2 - 2 omega)), with the library's own
// binary32 ln and exp; this value decides.
__device__ __forceinline__ float vhs_threshold(float us, float vinv, float lncv) {
  return exp32(fmul(vinv, fsub(ln32(us), lncv)));
}

// The same threshold from the hardware's base-2 approximations: within 3e-5 relative of
// vhs_threshold (the approximations' own errors, the binary32 rounding of an argument of
// magnitude below 70, and the 2-ulp error of ln32 and exp32).  [t (1 - 2^-10),
// t (1 + 2^-10)] therefore brackets the deciding value; a relative speed outside the
// bracket is decided without it.
constexpr float kThrLo = 1.0f - 0x1p-10f;
constexpr float kThrHi = 1.0f + 0x1p-10f;

__device__ __forceinline__ float vhs_threshold_approx(float us, float vinv, float lg2cv) {
  float l, t;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(us));
  const float x = fmul(vinv, fsub(l, lg2cv));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(x));
  return t;
}

// Isotropic scattering direction from two uniform words by the cylindrical (Archimedes)
// map: n_z = 2 u(w0) - 1 and azimuth 2 pi u(w1), independent and uniform, give
// n = (sqrt(1 - n_z^2) cos, sqrt(1 - n_z^2) sin, n_z), uniform on the sphere.  No
// rejection, so every candidate of a warp takes the same two draws.
__device__ __forceinline__ void direction_of(uint32_t w0, uint32_t w1, float& nx, float& ny,
                                             float& nz) {
  nz = s11(w0);
  const float rho = fsqrt(fsub(1.0f, fmul(nz, nz)));
  float sn, cs;
  sincos_turn(u01(w1), sn, cs);
  nx = fmul(rho, cs);
  ny = fmul(rho, sn);
}

// Per-lane sums of the 12 velocity moments of a group's particles (the count is the
// cell's particle number and needs no sum): v, v_i v_j (six), v_i |v|^2 (three).
// LaneSums<float>: the products of the binary32 velocities summed in binary32, the
// second and third moments by fused multiply-add (one rounding per term).
// LaneSums<double> (DSMC_ACCUM_FP64): every product rounded to binary32 exactly as the
// oracle forms it, then summed as an unevaluated triple of binary32 (hi, mid, lo): the rounding
// errors of the additions to hi go to mid, those of the additions to mid to lo.  With u = 2^-24
// and k products per lane (48 at most), |mid| <= k u S and |lo| <= k^2 u^2 S, S the sum of
// |products|, so the additions to lo lose at most k^3 u^3 S < 2^-55 S; binary64 additions lose up
// to k 2^-53 S.  (A pair without lo loses k^2 / 2 u^2 S, 2^-38 S: 2^-47 S seen with magnitudes
// spread over 2^14, where binary64 loses 2^-52 S and the cell's grid is 2^-55 S.)  The GB300 makes
// 2 binary64 additions per clock and SM against 128 in binary32: a step of 1,000 cells x 5,003
// (Kn = 0.1) took 0.678 ms with them, takes 0.184 ms (0.151 with pairs, 0.120 with
// LaneSums<float>).
template <typename T>
struct LaneSums;

template <>
struct LaneSums<float> {
  float2 a, b, c, d, e, f;  // (vx, vy) (vz, vz2) (vx2, vy2) (vxvy, vxvz) (vyvz, vz v2) (vx v2, vy v2)
  __device__ __forceinline__ void zero() {
    a = b = c = d = e = f = make_float2(0.0f, 0.0f);
  }
  __device__ __forceinline__ void add(float x, float y, float z) {
    const float2 xy = make_float2(x, y);
    const float2 sq = __fmul2_rn(xy, xy);
    const float zz = fmul(z, z);
    const float v2 = fadd(fadd(sq.x, sq.y), zz);
    a = __fadd2_rn(a, xy);
    b = __fadd2_rn(b, make_float2(z, zz));
    c = __fadd2_rn(c, sq);
    d = __ffma2_rn(make_float2(x, x), make_float2(y, z), d);
    e = __ffma2_rn(make_float2(y, z), make_float2(z, v2), e);
    f = __ffma2_rn(xy, make_float2(v2, v2), f);
  }
  // moment k = 1..12 in the order of the raw sums (1 vx, 2 vy, 3 vz, 4 vx2, 5 vy2, 6 vz2,
  // 7 vxvy, 8 vxvz, 9 vyvz, 10 vx v2, 11 vy v2, 12 vz v2); 0 for the padding slots
  __device__ __forceinline__ float get(int k) const {
    switch (k) {
      case 1: return a.x;
      case 2: return a.y;
      case 3: return b.x;
      case 4: return c.x;
      case 5: return c.y;
      case 6: return b.y;
      case 7: return d.x;
      case 8: return d.y;
      case 9: return e.x;
      case 10: return f.x;
      case 11: return f.y;
      case 12: return e.y;
      default: return 0.0f;
    }
  }
};

// Two sums at a time, in packed binary32 operations.
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  float2 r;
  asm("sub.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long&>(r))
      : "l"(reinterpret_cast<const unsigned long long&>(a)),
        "l"(reinterpret_cast<const unsigned long long&>(b)));
  return r;
}

// s = a + b rounded, and its rounding error exactly (Knuth's two-sum).
__device__ __forceinline__ float2 two_sum2(float2 a, float2 b, float2& s) {
  s = __fadd2_rn(a, b);
  const float2 t = sub2(s, a);
  return __fadd2_rn(sub2(a, sub2(s, t)), sub2(b, t));
}

struct Triple2 {
  float2 hi, mid, lo;
  __device__ __forceinline__ void add(float2 p) {
    const float2 e = two_sum2(hi, p, hi);
    lo = __fadd2_rn(lo, two_sum2(mid, e, mid));
  }
};

template <>
struct LaneSums<double> {
  Triple2 a, b, c, d, e, f;  // the same places as in LaneSums<float>
  __device__ __forceinline__ void zero() {
    const float2 z = make_float2(0.0f, 0.0f);
    a = b = c = d = e = f = Triple2{z, z, z};
  }
  // (the products by scalar multiplications: a packed product followed by a packed addition
  // was contracted, which adds the exact product instead of the rounded one)
  __device__ __forceinline__ void add(float x, float y, float z) {
    const float xx = fmul(x, x), yy = fmul(y, y), zz = fmul(z, z);
    const float v2 = fadd(fadd(xx, yy), zz);
    a.add(make_float2(x, y));
    b.add(make_float2(z, zz));
    c.add(make_float2(xx, yy));
    d.add(make_float2(fmul(x, y), fmul(x, z)));
    e.add(make_float2(fmul(y, z), fmul(z, v2)));
    f.add(make_float2(fmul(x, v2), fmul(y, v2)));
  }
  static __device__ __forceinline__ float3 first(const Triple2& t) {
    return make_float3(t.hi.x, t.mid.x, t.lo.x);
  }
  static __device__ __forceinline__ float3 second(const Triple2& t) {
    return make_float3(t.hi.y, t.mid.y, t.lo.y);
  }
  // moment k as its triple (hi, mid, lo), in the order of LaneSums<float>::get
  __device__ __forceinline__ float3 get(int k) const {
    switch (k) {
      case 1: return first(a);
      case 2: return second(a);
      case 3: return first(b);
      case 4: return first(c);
      case 5: return second(c);
      case 6: return second(b);
      case 7: return first(d);
      case 8: return second(d);
      case 9: return first(e);
      case 10: return first(f);
      case 11: return second(f);
      case 12: return second(e);
      default: return make_float3(0.0f, 0.0f, 0.0f);
    }
  }
};

// The same for one sum.
__device__ __forceinline__ float two_sum(float a, float b, float& s) {
  s = fadd(a, b);
  const float t = fsub(s, a);
  return fadd(fsub(a, fsub(s, t)), fsub(b, t));
}

// Sum of two triples.
__device__ __forceinline__ float3 triple_sum(float3 a, float3 b) {
  float hi, m0, mid;
  const float e = two_sum(a.x, b.x, hi);
  const float f = two_sum(a.y, b.y, m0);
  const float g = two_sum(m0, e, mid);
  return make_float3(hi, mid, fadd(fadd(a.z, b.z), fadd(f, g)));
}

// Warp sum of a group's lane sums by a transposing butterfly over 16 slots (moments
// 1..12 and zero padding): each exchange halves the values a lane carries, so 16
// shuffles leave the total of moment moment_of_lane(lane) on lanes 2i and 2i+1.
__device__ __forceinline__ int moment_of_lane(int lane) {
  return ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
}

__device__ __forceinline__ float group_total(const LaneSums<float>& m, int lane) {
  float v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = m.get(k);
#pragma unroll
  for (int half = 8, mask = 16; half >= 1; half >>= 1, mask >>= 1) {
    const bool upper = (lane & mask) != 0;
#pragma unroll
    for (int k = 0; k < half; ++k) {
      const float send = upper ? v[k] : v[k + half];
      const float keep = upper ? v[k + half] : v[k];
      v[k] = keep + __shfl_xor_sync(kFull, send, mask);
    }
  }
  return v[0] + __shfl_xor_sync(kFull, v[0], 1);
}

// The same for triples; the triple's value in binary64.
__device__ __forceinline__ double group_total(const LaneSums<double>& m, int lane) {
  float3 v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = m.get(k);
  auto other = [](float3 x, int mask) {
    return make_float3(__shfl_xor_sync(kFull, x.x, mask), __shfl_xor_sync(kFull, x.y, mask),
                       __shfl_xor_sync(kFull, x.z, mask));
  };
#pragma unroll
  for (int half = 8, mask = 16; half >= 1; half >>= 1, mask >>= 1) {
    const bool upper = (lane & mask) != 0;
#pragma unroll
    for (int k = 0; k < half; ++k) {
      const float3 send = upper ? v[k] : v[k + half];
      const float3 keep = upper ? v[k + half] : v[k];
      v[k] = triple_sum(keep, other(send, mask));
    }
  }
  const float3 s = triple_sum(v[0], other(v[0], 1));
  return (double)s.x + ((double)s.y + (double)s.z);
}

// Exact, order-independent combination of group totals.  A cell's group totals are
// rounded to integer multiples of a grid 2^-(41 - e), e = bit length of the cell's
// particle count nc, and the integers added in 64 bits: integer addition does not
// depend on the order in which warps finish their groups, so a step's cell sums are a
// pure function of the state.  With |v| <= 101 (|each product| <= 2^20) a group total is
// at most 2 n_g 2^20 in magnitude and the cell's integer sum stays below 2^62.  The
// rounding adds at most 2^-(42 - e) per group total.
__device__ __forceinline__ int grid_exponent(int nc) { return 41 - (32 - __clz(nc)); }

__device__ __forceinline__ long long fixed_of(float t, int gexp) {
  return __float2ll_rn(fmul(t, __int_as_float((127 + gexp) << 23)));
}
__device__ __forceinline__ long long fixed_of(double t, int gexp) {
  return __double2ll_rn(__dmul_rn(t, __longlong_as_double((long long)(1023 + gexp) << 52)));
}

// The NTC candidates of one collision group (group gi, gn particles, of cell c with nc
// particles): every candidate's pair, acceptance threshold and scattering direction are
// drawn up front, 32 candidates at a time, one per lane, then applied in conflict-free
// rounds that reproduce the sequential order exactly.  rec[0..gn) are the group's records
// in shared memory (updated in place); touch[0..gn) is zero on entry and exit.  gmax gets
// the largest relative speed seen (this lane's), M the candidate count, laccn this lane's
// accepted collisions; cand_fail is set when the count exceeds its limit.
__device__ __forceinline__ void ntc_collide(const InstParams& a, float4* rec, unsigned* touch,
                                            int gn, int nc, int c, int gi, uint32_t step,
                                            float smax, int mode, int lane, unsigned lt,
                                            float& gmax, uint32_t& M, unsigned& laccn,
                                            bool& cand_fail) {
  const uint32_t c3 = (kStreamColl << 24) | ((uint32_t)gi << 4);
  const float t1 = fmul((float)(gn - 1), (float)nc);
  const float mf = fmul(fmul(t1, a.coef), smax);
  const float fl = floorf(mf);
  const float frac = fsub(mf, fl);
  const bool mbad = !(mf <= kMaxCandidates);
  if (mbad) cand_fail = true;
  // M is floor(mf) or floor(mf) + 1 by the count-rounding draw (candidate counter
  // 0xffffffff).  Batch 0 draws it on lane 31 beside candidates 0..30 on lanes
  // 0..30; later batches hold candidates 31 + 32 b + lane.
  for (uint32_t kb = 0, first = 1;; first = 0) {
    const uint32_t k =
        first ? (lane == 31 ? 0xffffffffu : (uint32_t)lane) : kb + (uint32_t)lane;
    U4 w{};
    if (first) {
      w = philox_rk(k, (uint32_t)c, step, c3, a.keys);
      const float ur = __shfl_sync(kFull, u01(w.x), 31);
      M = mbad ? 0u : (uint32_t)fl + (ur < frac ? 1u : 0u);
    }
    bool pend = first ? (lane < 31 && (uint32_t)lane < M) : (k < M);
    if (M == 0u) break;
    int i = 0, j = 0;
    // acceptance: g > thr; thr_lo <= thr <= thr_hi, equal unless the VHS threshold
    // was bracketed by the fast approximation (thr itself is then formed only for
    // a relative speed inside the bracket)
    float us = 0.0f, thr_lo = 0.0f, thr_hi = 0.0f, nx = 0.0f, ny = 0.0f, nz = 0.0f;
    if (pend) {
      // one draw per candidate: word 0 the pair (multiply-shift: i from the high
      // half of w0 gn, j from the low half times gn - 1), word 1 the acceptance
      // uniform, words 2 and 3 the scattering direction
      if (!first) w = philox_rk(k, (uint32_t)c, step, c3, a.keys);
      const unsigned long long pij = (unsigned long long)w.x * (unsigned long long)gn;
      i = (int)(pij >> 32);
      j = (int)__umulhi((uint32_t)pij, (uint32_t)(gn - 1));
      j += (j >= i) ? 1 : 0;
      us = fmul(u01(w.y), smax);
      if (mode == 0) {
        thr_lo = thr_hi = us;
      } else if (mode == 1) {
        const float t = vhs_threshold_approx(us, a.vinv, a.lg2cv);
        if (t > 0x1p-100f && t < 0x1p100f) {
          thr_lo = fmul(t, kThrLo);
          thr_hi = fmul(t, kThrHi);
        } else {
          thr_lo = thr_hi = vhs_threshold(us, a.vinv, a.lncv);
        }
      } else {
        thr_lo = thr_hi = (us < a.cvhs) ? -1.0f : __int_as_float(0x7f800000);
      }
      direction_of(w.z, w.w, nx, ny, nz);
    }
    // Earlier candidates of the batch that share a particle with this one: the
    // candidate may be applied once none of them is pending any more, which gives
    // exactly the result of applying the candidates in order.
    if (pend) {
      atomicOr(&touch[i], 1u << lane);
      atomicOr(&touch[j], 1u << lane);
    }
    __syncwarp();
    const unsigned before = pend ? ((touch[i] | touch[j]) & lt) : 0u;
    __syncwarp();
    if (pend) {
      touch[i] = 0u;
      touch[j] = 0u;
    }
    for (;;) {
      const unsigned waiting = __ballot_sync(kFull, pend);
      if (waiting == 0u) break;
      const bool ready = pend && (before & waiting) == 0u;
      if (ready) {
        const float4 ri = rec[i], rj = rec[j];
        const float gx = fsub(ri.y, rj.y), gy = fsub(ri.z, rj.z), gz = fsub(ri.w, rj.w);
        const float g = fsqrt(fadd(fadd(fmul(gx, gx), fmul(gy, gy)), fmul(gz, gz)));
        gmax = fmaxf(gmax, g);
        bool accept = g > thr_hi;
        if (!accept && g > thr_lo) accept = g > vhs_threshold(us, a.vinv, a.lncv);
        if (accept) {
          const float hg = fmul(0.5f, g);
          const float cx = fmul(fadd(ri.y, rj.y), 0.5f);
          const float cy = fmul(fadd(ri.z, rj.z), 0.5f);
          const float cz = fmul(fadd(ri.w, rj.w), 0.5f);
          const float dx = fmul(hg, nx), dy = fmul(hg, ny), dz = fmul(hg, nz);
          rec[i] = make_float4(ri.x, fadd(cx, dx), fadd(cy, dy), fadd(cz, dz));
          rec[j] = make_float4(rj.x, fsub(cx, dx), fsub(cy, dy), fsub(cz, dz));
          laccn += 1;
        }
        pend = false;
      }
      __syncwarp();
    }
    kb = first ? 31u : kb + 32u;
    if (kb >= M) break;
  }
}

}  // namespace dsmc

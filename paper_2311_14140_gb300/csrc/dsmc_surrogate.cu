// dsmc_surrogate.cu -- the surrogate stage of the Micro-Macro-Surrogate method
// (Sec. 2.3, Appendix A): training samples from DSMC moment windows, Bayesian ridge
// regression with evidence maximisation and model selection, and the corrected 1D
// macroscopic solve with Monte Carlo uncertainty bands.
//
// Device work (binary64):
//   k_basis   once per surrogate: the Appendix A basis at the training cells (their values
//             depend on the grid and the exponents alone) and their Phi^T Phi.
//   k_window  one training sample per call: from a window's raw moment sums, the cell
//             velocities and shear stresses (Eq. 6 units), the constitutive targets
//             E_i = P_i + (2 Kn / sqrt(pi)) du/dy_i at the interior cells (Eq. 13, du/dy
//             by central differences) with their Appendix A basis rows, and the wall
//             velocities extrapolated linearly from the two nearest cells; it adds the
//             sample's sufficient statistics (Phi^T Phi, Phi^T t, t^T t, sum t, N) for
//             the boundary and constitutive models to running totals.  The moment sums
//             stay on the device: a run's accumulators are read in place.
//   k_modes   Eq. 8 is linear: a trial's profile is its wall velocity plus the profile of the
//             body force plus its weights times the profiles of the basis functions, so those
//             (at most four) are solved once, in closed form up to a prefix sum; also the
//             trials' weights, drawn from the selected models' posteriors (w = m + L z,
//             S = L L^T by Cholesky on the host).
//   k_bands   per cell: mean and standard deviation over the trials.
// Host work: the evidence maximisation itself (MacKay's re-estimation of alpha and beta
// on 1x1 to 3x3 matrices, Bishop Sec. 3.5, Tipping App. A) and Eq. 17.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "dsmc.h"
#include "dsmc_internal.h"

namespace {

constexpr int kStats = 20;  // sufficient statistics, layout below
// [0..8] Phi^T Phi (3x3, row-major) of the constitutive basis, [9..11] Phi^T t,
// [12] t^T t, [13] N (constitutive); [14] sum x t, [15] sum x^2, [16] t^T t, [17] N
// (boundary); [18] sum t (constitutive), [19] sum t (boundary).
constexpr int kThreads = 256;
constexpr int kWindowCells = 1024;  // cells whose velocities k_window keeps in shared memory
constexpr double kAlphaMax = 1e30;  // weight precision above which weights are off
constexpr double kSqrtPi = 1.7724538509055160273;

// Table 1 of the paper: exponents b_1..b_3 at the tabulated Kn.
constexpr double kTableKn[7] = {0.01, 0.05, 0.1, 0.2, 0.5, 1.0, 5.0};
constexpr double kTableB[7][3] = {{130, 150, 200}, {30, 40, 70}, {20, 40, 10}, {20, 12, 8},
                                  {10, 7, 6},      {8, 6, 20},   {7, 6, 5}};

dsmc_status reject(dsmc_status s, const std::string& msg) {
  dsmc::set_last_error(msg);
  return s;
}

dsmc_status cuda_reject(cudaError_t e, const char* what) {
  return reject(DSMC_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define SUR_CUDA(call, what)                       \
  do {                                             \
    cudaError_t e_ = (call);                       \
    if (e_ != cudaSuccess) return cuda_reject(e_, what); \
  } while (0)

struct WindowArgs {
  int n;           // cells
  double n_norm;   // steps * ppc: sampled count per cell at the initial density
  double kn, F;
  double b[3];
  double length;   // the run's extent in channel units (1: the whole channel)
  int last;        // last training cell (first is 1)
  int both;        // 1: both walls give boundary data (whole channel), 0: bottom only
};

// Sum over the CTA of K values per thread, into red[0..K) (valid after the call's barrier):
// warp k adds value k of all threads.  (A butterfly of every value in every warp is three times
// the binary64 additions, which come at two per clock.)
template <int K>
__device__ __forceinline__ void block_sums(const double (&v)[K], double (&part)[K][kThreads],
                                           double* red) {
  static_assert(K <= kThreads / 32, "a warp per value");
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) part[k][t] = v[k];
  __syncthreads();
  if (w < K) {
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < kThreads / 32; ++u) s += part[w][u * 32 + lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[w] = s;
  }
  __syncthreads();
}

// basis[l n + i] = c (exp(-b_l y_i) - exp(-b_l (1 - y_i))) at the training cells 1..last, and
// gram[0..5] = their products' sums (00, 01, 02, 11, 12, 22).
__global__ void __launch_bounds__(kThreads)
    k_basis(WindowArgs a, double* __restrict__ basis, double* __restrict__ gram) {
  __shared__ double part[6][kThreads];
  const double h = a.length / a.n;
  const double c = 2.0 * a.kn / kSqrtPi;
  double g[6] = {0, 0, 0, 0, 0, 0};
  for (int i = 1 + threadIdx.x; i <= a.last; i += kThreads) {
    const double y = (i + 0.5) * h;
    double f[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      f[l] = c * (exp(-a.b[l] * y) - exp(-a.b[l] * (1.0 - y)));
      basis[(size_t)l * a.n + i] = f[l];
    }
    g[0] = fma(f[0], f[0], g[0]);
    g[1] = fma(f[0], f[1], g[1]);
    g[2] = fma(f[0], f[2], g[2]);
    g[3] = fma(f[1], f[1], g[3]);
    g[4] = fma(f[1], f[2], g[4]);
    g[5] = fma(f[2], f[2], g[5]);
  }
  block_sums<6>(g, part, gram);
}

// One CTA: a cell per thread (200 cells in the paper), one division per cell.  Binary64 runs at
// two operations per clock and SM here, so the exponentials of the basis (now k_basis's) and
// six divisions per cell were most of this kernel: windows of 200 cells added one after another
// took 25 us each and take 8.9, the kernel 8.
__global__ void __launch_bounds__(kThreads)
    k_window(const double* __restrict__ acc, WindowArgs a, const double* __restrict__ basis,
             const double* __restrict__ gram, double* __restrict__ stats,
             double* __restrict__ scratch) {
  __shared__ double u_sh[kWindowCells];
  double* u = a.n <= kWindowCells ? u_sh : scratch;  // cell velocities
  __shared__ double part[5][kThreads];
  __shared__ double red[5];
  const int t = threadIdx.x;
  const double h = a.length / a.n;
  const double c = 2.0 * a.kn / kSqrtPi;
  const double per = 2.0 / a.n_norm, slope = c / (2.0 * h);
  const int gi[9] = {0, 1, 2, 1, 3, 4, 2, 4, 5};
  // what the totals below need, on its way while the cells are worked on
  const double before = t < kStats ? stats[t] : 0.0;
  const double gr = t < 9 ? gram[gi[t]] : 0.0;
  for (int i = t; i < a.n; i += kThreads) {
    const double* r = acc + (size_t)i * dsmc::kNMom;
    u[i] = r[1] / r[0];
  }
  __syncthreads();
  double v[5] = {0, 0, 0, 0, 0};  // Phi^T t (three), t^T t, sum t
  for (int i = 1 + t; i <= a.last; i += kThreads) {
    const double* r = acc + (size_t)i * dsmc::kNMom;
    // P = 2 (N / n_norm) (S_xy / N - u_x u_y) with u_y = S_y / N
    const double P = per * (r[7] - u[i] * r[2]);
    const double E = fma(slope, u[i + 1] - u[i - 1], P);
#pragma unroll
    for (int l = 0; l < 3; ++l) v[l] = fma(basis[(size_t)l * a.n + i], E, v[l]);
    v[3] = fma(E, E, v[3]);
    v[4] += E;
  }
  block_sums<5>(v, part, red);
  // Totals: Phi^T Phi of the sample is the basis's own; the boundary models have x = -P(0) = F
  // (and P(1) = F) and t = the wall velocities.
  if (t >= kStats) return;
  const int n = a.n;
  const double ub = 1.5 * u[0] - 0.5 * u[1];
  const double ut = a.both ? 1.5 * u[n - 1] - 0.5 * u[n - 2] : 0.0;
  double add = 0.0;
  if (t < 9) add = gr;
  else if (t < 13) add = red[t - 9];
  else if (t == 13) add = (double)a.last;
  else if (t == 14) add = a.both ? a.F * ub + a.F * ut : a.F * ub;
  else if (t == 15) add = a.both ? a.F * a.F + a.F * a.F : a.F * a.F;
  else if (t == 16) add = a.both ? ub * ub + ut * ut : ub * ub;
  else if (t == 17) add = a.both ? 2.0 : 1.0;
  else if (t == 18) add = red[4];
  else add = a.both ? ub + ut : ub;
  stats[t] = before + add;
}

// Posterior of the selected models as the trials need it.
struct TrialModels {
  int sel_v, k;  // slip selected; number of constitutive weights (0..3)
  double m_v, sd_v;
  double m[3], L[9];  // weights' means and the Cholesky factor of their covariance
  double kn, F;
  double b[3];
  int n;  // CFD cells
};

// Blocks 0..k: the profile of one unit right side of the cell-centred finite-volume form of
// Eq. 8 with zero wall values: block 0 the body force, block 1 + l the basis function l.
// With face fluxes q_f (f = 0..n) the rows say q_{i+1} - q_i = r_i, so q_f = q_0 + R_f with
// R_f = f src (block 0) or S_f - S_0; summing u_{i+1} - u_i = h q_{i+1} from wall to wall
// (half cells at both ends) gives q_0 = -(h sum_{0<f<n} R_f + h/2 R_n) and
// u_i = h/2 q_0 + h i q_0 + h sum_{0<f<=i} R_f: one prefix sum instead of a sweep of n
// dependent divisions per trial (dsmc_surrogate_profile at 200 cells: 0.85 ms with one trial,
// 1.18 with 1,000; now 0.057 and 0.066).
// The blocks after them: the weights of the trials, (uw, w_1..w_3) in weights[4 t ..].
__global__ void __launch_bounds__(kThreads)
    k_modes(TrialModels tm, const double* __restrict__ z, int n_trials,
            double* __restrict__ modes, double* __restrict__ weights) {
  __shared__ double wtot[kThreads / 32];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  if ((int)blockIdx.x > tm.k) {
    const int tr = ((int)blockIdx.x - tm.k - 1) * kThreads + t;
    if (tr >= n_trials) return;
    const double* zt = z + (size_t)tr * 4;
    double* wt = weights + (size_t)tr * 4;
    // -sigma_P P(0) = sigma_P F
    wt[0] = tm.sel_v ? (tm.m_v + tm.sd_v * zt[0]) * tm.F : 0.0;
    for (int i = 0; i < 3; ++i) {
      double s = 0.0;
      if (i < tm.k) {
        s = tm.m[i];
        for (int j = 0; j <= i; ++j) s += tm.L[i * 3 + j] * zt[1 + j];
      }
      wt[1 + i] = s;
    }
    return;
  }
  const int l = (int)blockIdx.x - 1;
  const int n = tm.n;
  const double h = 1.0 / n;
  const double src = -h * kSqrtPi * tm.F / tm.kn;
  const double b = l >= 0 ? tm.b[l] : 0.0;
  const double S0 = 1.0 - exp(-b);
  auto R = [&](int f) {
    if (l < 0) return f * src;
    const double y = f * h;
    return exp(-b * y) - exp(-b * (1.0 - y)) - S0;
  };
  double* u = modes + (size_t)(l + 1) * n;
  double carry = 0.0;  // sum of R over the faces of the earlier chunks
  for (int c0 = 0; c0 < n; c0 += kThreads) {
    const int i = c0 + t;
    double x = (i > 0 && i < n) ? R(i) : 0.0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wtot[wid] = x;
    __syncthreads();
    double before = carry, all = 0.0;
    for (int q = 0; q < kThreads / 32; ++q) {
      if (q < wid) before += wtot[q];
      all += wtot[q];
    }
    carry += all;
    if (i < n) u[i] = before + x;  // sum over 0 < f <= i
    __syncthreads();
  }
  const double q0 = -(h * carry + 0.5 * h * R(n));
  for (int i = t; i < n; i += kThreads) u[i] = h * ((0.5 + i) * q0 + u[i]);
}

// S(y) of Eq. 14 with weights w (k of them) at the faces y = f / n, f = 0..n.
__global__ void k_correction(int k, double w0, double w1, double w2, double b0, double b1,
                             double b2, int n, double* __restrict__ S) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f > n) return;
  const double y = (double)f / n;
  const double w[3] = {w0, w1, w2}, b[3] = {b0, b1, b2};
  double s = 0.0;
  for (int l = 0; l < k; ++l) s += w[l] * (exp(-b[l] * y) - exp(-b[l] * (1.0 - y)));
  S[f] = s;
}

// Cell blockIdx.x: mean and (sample) standard deviation over the trials of
// u = uw + u_F + sum_l w_l u_l.
__global__ void __launch_bounds__(kThreads)
    k_bands(const double* __restrict__ modes, const double* __restrict__ weights, int k,
            int n_trials, int n, double* __restrict__ mean, double* __restrict__ sd) {
  __shared__ double part[1][kThreads];
  __shared__ double red[2];
  const int i = blockIdx.x, t = threadIdx.x;
  const double base = modes[i];
  double g[3] = {0, 0, 0};
#pragma unroll
  for (int l = 0; l < 3; ++l)
    if (l < k) g[l] = modes[(size_t)(l + 1) * n + i];
  auto profile = [&](int tr) {
    const double* w = weights + (size_t)tr * 4;
    return w[0] + fma(w[3], g[2], fma(w[2], g[1], fma(w[1], g[0], base)));
  };
  double s[1] = {0.0};
  for (int tr = t; tr < n_trials; tr += kThreads) s[0] += profile(tr);
  block_sums<1>(s, part, red);
  const double m = red[0] / n_trials;
  double v[1] = {0.0};
  for (int tr = t; tr < n_trials; tr += kThreads) {
    const double d = profile(tr) - m;
    v[0] = fma(d, d, v[0]);
  }
  block_sums<1>(v, part, red + 1);
  if (t == 0) {
    mean[i] = m;
    sd[i] = n_trials > 1 ? sqrt(red[1] / (n_trials - 1)) : 0.0;
  }
}

// Standard deviation when no model with random weights is selected (no slip, C0): every trial has
// the same profile, and the deviation is the rounding of the sums over the trials, about 1e-16 of
// u.  Those digits are part of the results that runs of the library are compared by, and they
// depend on the last bits of u: so u is swept here (Thomas) and the trials are summed one after
// another, as for profiles solved trial by trial.  (The mean is k_bands's for every fit, whether a
// standard deviation is asked for or not.)
__global__ void __launch_bounds__(kThreads)
    k_same_profiles_sd(double kn, double F, int n, int n_trials, double* __restrict__ u,
                       double* __restrict__ cp, double* __restrict__ sd) {
  if (threadIdx.x == 0) {
    const double h = 1.0 / n;
    const double src = -h * kSqrtPi * F / kn;
    const double inner = 1.0 / h, wall = 2.0 / h;  // coefficients of the faces
    double cprev = 0.0, rprev = 0.0;
    for (int i = 0; i < n; ++i) {
      const double lo = (i > 0) ? inner : 0.0;
      const double up = (i < n - 1) ? inner : 0.0;
      const double d = -((i > 0) ? inner : wall) - ((i < n - 1) ? inner : wall);
      const double den = d - lo * cprev;
      cprev = up / den;
      rprev = (src - lo * rprev) / den;
      cp[i] = cprev;
      u[i] = rprev;
    }
    double next = u[n - 1];
    for (int i = n - 2; i >= 0; --i) u[i] = next = u[i] - cp[i] * next;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += kThreads) {
    const double x = u[i];
    double s = 0.0, v = 0.0;
    for (int t = 0; t < n_trials; ++t) s += x;
    const double m = s / n_trials, d = x - m;
    for (int t = 0; t < n_trials; ++t) v += d * d;
    sd[i] = sqrt(v / (n_trials - 1));
  }
}

// ---------------------------------------------------------------------------
// Host linear algebra on k x k symmetric matrices (k <= 3).

// Cholesky A = L L^T; false if A is not positive definite.
bool cholesky(const double* A, int k, double* L) {
  for (int i = 0; i < 9; ++i) L[i] = 0.0;
  for (int i = 0; i < k; ++i)
    for (int j = 0; j <= i; ++j) {
      double s = A[i * 3 + j];
      for (int q = 0; q < j; ++q) s -= L[i * 3 + q] * L[j * 3 + q];
      if (i == j) {
        if (!(s > 0.0)) return false;
        L[i * 3 + i] = std::sqrt(s);
      } else {
        L[i * 3 + j] = s / L[j * 3 + j];
      }
    }
  return true;
}

// Inverse and log determinant of an SPD matrix through its Cholesky factor.
bool spd_inverse(const double* A, int k, double* inv, double* logdet) {
  double L[9];
  if (!cholesky(A, k, L)) return false;
  *logdet = 0.0;
  for (int i = 0; i < k; ++i) *logdet += 2.0 * std::log(L[i * 3 + i]);
  for (int c = 0; c < k; ++c) {  // solve A x = e_c
    double y[3] = {0, 0, 0}, x[3] = {0, 0, 0};
    for (int i = 0; i < k; ++i) {
      double s = (i == c) ? 1.0 : 0.0;
      for (int q = 0; q < i; ++q) s -= L[i * 3 + q] * y[q];
      y[i] = s / L[i * 3 + i];
    }
    for (int i = k - 1; i >= 0; --i) {
      double s = y[i];
      for (int q = i + 1; q < k; ++q) s -= L[q * 3 + i] * x[q];
      x[i] = s / L[i * 3 + i];
    }
    for (int i = 0; i < k; ++i) inv[i * 3 + c] = x[i];
  }
  return true;
}

// Eigenvalues of a symmetric k x k matrix by cyclic Jacobi rotations.
void sym_eigenvalues(const double* A0, int k, double* ev) {
  double A[9];
  std::memcpy(A, A0, sizeof(A));
  for (int sweep = 0; sweep < 100; ++sweep) {
    double off = 0.0;
    for (int p = 0; p < k; ++p)
      for (int q = p + 1; q < k; ++q) off += A[p * 3 + q] * A[p * 3 + q];
    if (off == 0.0) break;
    for (int p = 0; p < k; ++p)
      for (int q = p + 1; q < k; ++q) {
        const double apq = A[p * 3 + q];
        if (apq == 0.0) continue;
        const double theta = (A[q * 3 + q] - A[p * 3 + p]) / (2.0 * apq);
        const double t = (theta >= 0 ? 1.0 : -1.0) / (std::fabs(theta) + std::sqrt(theta * theta + 1.0));
        const double c = 1.0 / std::sqrt(t * t + 1.0), s = t * c;
        for (int r = 0; r < k; ++r) {  // A <- A J
          const double arp = A[r * 3 + p], arq = A[r * 3 + q];
          A[r * 3 + p] = c * arp - s * arq;
          A[r * 3 + q] = s * arp + c * arq;
        }
        for (int r = 0; r < k; ++r) {  // A <- J^T A
          const double apr = A[p * 3 + r], aqr = A[q * 3 + r];
          A[p * 3 + r] = c * apr - s * aqr;
          A[q * 3 + r] = s * apr + c * aqr;
        }
      }
  }
  for (int i = 0; i < k; ++i) ev[i] = A[i * 3 + i];
}

struct Fit {
  double m[3], S[9], alpha, beta, logev;
  int iterations;
};

// Evidence maximisation for a model with k weights from its sufficient statistics:
// G = Phi^T Phi (k x k block of a 3x3), pt = Phi^T t, tt = t^T t, st = sum t, N.
bool brr_stats(const double* G3, const double* pt, double tt, double st, double N, int k,
               Fit* f) {
  double G[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (int i = 0; i < k; ++i)
    for (int j = 0; j < k; ++j) G[i * 3 + j] = G3[i * 3 + j];
  double ev[3];
  sym_eigenvalues(G, k, ev);
  const double mean = st / N;
  double var = tt / N - mean * mean;
  double alpha = 1.0, beta = 1.0 / (var > 1e-300 ? var : 1e-300);
  double S[9] = {}, m[3] = {}, logdet = 0.0;
  auto posterior = [&](double al, double be) {
    double A[9];
    for (int i = 0; i < 9; ++i) A[i] = be * G[i];
    for (int i = 0; i < k; ++i) A[i * 3 + i] += al;
    if (!spd_inverse(A, k, S, &logdet)) return false;
    for (int i = 0; i < k; ++i) {
      double s = 0.0;
      for (int j = 0; j < k; ++j) s += S[i * 3 + j] * pt[j];
      m[i] = be * s;
    }
    return true;
  };
  auto resid = [&]() {  // |t - Phi m|^2 from the statistics
    double r = tt;
    for (int i = 0; i < k; ++i) {
      r -= 2.0 * m[i] * pt[i];
      for (int j = 0; j < k; ++j) r += m[i] * G[i * 3 + j] * m[j];
    }
    return r;
  };
  int it = 0;
  for (; it < 1000; ++it) {
    if (!posterior(alpha, beta)) return false;
    double gamma = 0.0;
    for (int i = 0; i < k; ++i) gamma += beta * ev[i] / (alpha + beta * ev[i]);
    double mm = 0.0;
    for (int i = 0; i < k; ++i) mm += m[i] * m[i];
    const double an = (mm <= gamma / kAlphaMax) ? kAlphaMax : gamma / mm;
    const double bn = (N - gamma) / resid();
    const bool done = std::fabs(an - alpha) <= 1e-12 * alpha && std::fabs(bn - beta) <= 1e-12 * beta;
    alpha = an;
    beta = bn;
    if (done) break;
  }
  if (!posterior(alpha, beta)) return false;
  double mm = 0.0;
  for (int i = 0; i < k; ++i) mm += m[i] * m[i];
  const double E = 0.5 * beta * resid() + 0.5 * alpha * mm;
  f->logev = 0.5 * k * std::log(alpha) + 0.5 * N * std::log(beta) - E - 0.5 * logdet -
             0.5 * N * std::log(2.0 * M_PI);
  std::memcpy(f->m, m, sizeof(m));
  std::memcpy(f->S, S, sizeof(S));
  f->alpha = alpha;
  f->beta = beta;
  f->iterations = it + 1;
  return true;
}

// Evidence of a model without weights: t ~ N(0, I / beta) at beta = N / t^T t.
double zero_evidence(double tt, double N, double* beta) {
  *beta = N / tt;
  return 0.5 * N * std::log(*beta) - 0.5 * N * std::log(2.0 * M_PI) - 0.5 * (*beta) * tt;
}

// Eq. 17's most probable model (equal priors), the simplest (lowest index) among models
// whose log evidences agree with the best to kTieRel: such ties are rounding noise, e.g.
// every extra weight shrunk to zero on data with no signal for it.
constexpr double kTieRel = 1e-9;

int select_model(const double* le, int n) {
  double top = le[0];
  for (int k = 1; k < n; ++k) top = std::max(top, le[k]);
  const double tol = kTieRel * std::max(1.0, std::fabs(top));
  for (int k = 0; k < n; ++k)
    if (le[k] >= top - tol) return k;
  return 0;
}

void probabilities(const double* le, int n, double* p) {
  double mx = le[0];
  for (int i = 1; i < n; ++i) mx = le[i] > mx ? le[i] : mx;
  double s = 0.0;
  for (int i = 0; i < n; ++i) s += (p[i] = std::exp(le[i] - mx));
  for (int i = 0; i < n; ++i) p[i] /= s;
}

}  // namespace

struct dsmc_surrogate {
  double Kn = 1.0, F = 0.0;
  int n_cells = 0, ppc = 0;
  double length = 1.0;  // extent of the runs in channel units
  int n_train = 0;      // cells of the training region (sub-domain runs)
  double b[3]{};
  cudaStream_t stream = nullptr;
  double* stats = nullptr;    // device, kStats
  double* window = nullptr;   // device, n_cells x 13 (host windows are copied here)
  double* basis = nullptr;    // device: 3 x n_cells basis values, their 6 products' sums, and
                              // n_cells velocities (scratch of k_window)
  double* trials = nullptr;   // device scratch of dsmc_surrogate_profile
  size_t trials_cap = 0;
  long long n_samples = 0;
  dsmc_surrogate_fit fit{};
  bool fitted = false;
};

extern "C" {

dsmc_status dsmc_surrogate_exponents(double Kn, double* b) {
  if (!b || !(Kn > 0.0)) return reject(DSMC_E_INVAL, "surrogate: Kn > 0 and b non-NULL");
  int best = 0;
  for (int i = 1; i < 7; ++i)
    if (std::fabs(std::log(Kn) - std::log(kTableKn[i])) <
        std::fabs(std::log(Kn) - std::log(kTableKn[best])))
      best = i;
  for (int l = 0; l < 3; ++l) b[l] = kTableB[best][l];
  return DSMC_OK;
}

static WindowArgs window_args(const dsmc_surrogate* s, long long n_steps) {
  WindowArgs a;
  a.n = s->n_cells;
  a.n_norm = (double)n_steps * (double)s->ppc;
  a.kn = s->Kn;
  a.F = s->F;
  for (int l = 0; l < 3; ++l) a.b[l] = s->b[l];
  a.length = s->length;
  a.both = s->length == 1.0 ? 1 : 0;
  a.last = a.both ? s->n_cells - 2 : s->n_train - 1;
  return a;
}

static dsmc_status create_surrogate(double Kn, double F, int n_cells, int ppc, double length,
                                    int n_train, const double* b, void* stream,
                                    dsmc_surrogate_handle* out) {
  if (!out) return reject(DSMC_E_INVAL, "out: NULL");
  *out = nullptr;
  if (!(Kn > 0.0) || !std::isfinite(Kn) || !std::isfinite(F) || F == 0.0 || n_cells < 3 ||
      ppc < 1)
    return reject(DSMC_E_INVAL, "surrogate: finite Kn > 0, finite F != 0, n_cells >= 3, ppc >= 1");
  dsmc_surrogate* s = new (std::nothrow) dsmc_surrogate();
  if (!s) return reject(DSMC_E_NOMEM, "host allocation failed");
  s->Kn = Kn;
  s->F = F;
  s->n_cells = n_cells;
  s->ppc = ppc;
  s->length = length;
  s->n_train = n_train;
  s->stream = (cudaStream_t)stream;
  if (b)
    for (int l = 0; l < 3; ++l) s->b[l] = b[l];
  else
    dsmc_surrogate_exponents(Kn, s->b);
  const size_t nc = (size_t)n_cells;
  // one allocation: statistics, the window's copy and the basis
  cudaError_t e = cudaMalloc(&s->stats, (kStats + (dsmc::kNMom + 4) * nc + 6) * sizeof(double));
  s->window = s->stats + kStats;
  s->basis = s->window + dsmc::kNMom * nc;
  if (e == cudaSuccess) e = cudaMemsetAsync(s->stats, 0, kStats * sizeof(double), s->stream);
  if (e == cudaSuccess) {
    k_basis<<<1, kThreads, 0, s->stream>>>(window_args(s, 1), s->basis, s->basis + 3 * nc);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    dsmc_surrogate_destroy(s);
    return cuda_reject(e, "surrogate allocation");
  }
  *out = s;
  return DSMC_OK;
}

dsmc_status dsmc_surrogate_create(double Kn, double F, int n_cells, int ppc, const double* b,
                                  void* stream, dsmc_surrogate_handle* out) {
  return create_surrogate(Kn, F, n_cells, ppc, 1.0, 0, b, stream, out);
}

dsmc_status dsmc_surrogate_create_region(double Kn, double F, int n_cells, int ppc,
                                         double length, int n_train, const double* b,
                                         void* stream, dsmc_surrogate_handle* out) {
  if (!(length > 0.0 && length < 1.0) || n_train < 2 || n_train > n_cells - 1)
    return reject(DSMC_E_INVAL, "surrogate region: 0 < length < 1, 2 <= n_train <= n_cells - 1");
  return create_surrogate(Kn, F, n_cells, ppc, length, n_train, b, stream, out);
}

dsmc_status dsmc_surrogate_destroy(dsmc_surrogate_handle s) {
  if (!s) return DSMC_OK;
  cudaStreamSynchronize(s->stream);
  cudaFree(s->stats);  // (and the window and the basis)
  cudaFree(s->trials);
  delete s;
  return DSMC_OK;
}

dsmc_status dsmc_surrogate_reset(dsmc_surrogate_handle s) {
  if (!s) return reject(DSMC_E_INVAL, "surrogate: NULL");
  SUR_CUDA(cudaMemsetAsync(s->stats, 0, kStats * sizeof(double), s->stream), "reset");
  s->n_samples = 0;
  s->fitted = false;
  return DSMC_OK;
}

// One window on the device (acc_dev: n_cells x 13 raw sums of n_steps sampled steps).
static dsmc_status add_device_window(dsmc_surrogate* s, const double* acc_dev, long long n_steps) {
  const size_t nc = (size_t)s->n_cells;
  k_window<<<1, kThreads, 0, s->stream>>>(acc_dev, window_args(s, n_steps), s->basis,
                                          s->basis + 3 * nc, s->stats, s->basis + 3 * nc + 6);
  SUR_CUDA(cudaGetLastError(), "window kernel");
  s->n_samples += 1;
  s->fitted = false;
  return DSMC_OK;
}

dsmc_status dsmc_surrogate_add_window(dsmc_surrogate_handle s, const double* acc,
                                      long long n_steps) {
  if (!s || !acc) return reject(DSMC_E_INVAL, "surrogate: NULL");
  if (n_steps < 1) return reject(DSMC_E_INVAL, "surrogate: n_steps >= 1");
  cudaPointerAttributes attr{};
  const bool on_device = cudaPointerGetAttributes(&attr, acc) == cudaSuccess &&
                         attr.type == cudaMemoryTypeDevice;
  cudaGetLastError();
  if (on_device) return add_device_window(s, acc, n_steps);
  SUR_CUDA(cudaMemcpyAsync(s->window, acc, (size_t)s->n_cells * dsmc::kNMom * sizeof(double),
                           cudaMemcpyDefault, s->stream),
           "copy window");
  return add_device_window(s, s->window, n_steps);
}

dsmc_status dsmc_surrogate_add_run(dsmc_surrogate_handle s, dsmc_handle h, int id) {
  if (!s || !h) return reject(DSMC_E_INVAL, "surrogate: NULL");
  dsmc_info info;
  dsmc_status st = dsmc_get_info_of(h, id, &info);
  if (st != DSMC_OK) return st;
  if (info.n_cells != s->n_cells || info.ppc != s->ppc)
    return reject(DSMC_E_INVAL, "surrogate: the run's n_cells and ppc differ from the surrogate's");
  if (info.n_samples < 1) return reject(DSMC_E_STATE, "surrogate: the run has no sampled steps");
  const double* acc = nullptr;
  if ((st = dsmc_device_moments_of(h, id, &acc)) != DSMC_OK) return st;
  // The run's work and the window kernel are ordered through the run's stream.
  if ((st = dsmc_sync(h)) != DSMC_OK) return st;
  if ((st = add_device_window(s, acc, info.n_samples)) != DSMC_OK) return st;
  SUR_CUDA(cudaStreamSynchronize(s->stream), "window");
  return dsmc_reset_samples_of(h, id);
}

dsmc_status dsmc_surrogate_train(dsmc_surrogate_handle s, dsmc_surrogate_fit* out) {
  if (!s || !out) return reject(DSMC_E_INVAL, "surrogate: NULL");
  if (s->n_samples < 1) return reject(DSMC_E_STATE, "surrogate: no training samples");
  double st[kStats];
  SUR_CUDA(cudaMemcpyAsync(st, s->stats, sizeof(st), cudaMemcpyDeviceToHost, s->stream), "stats");
  SUR_CUDA(cudaStreamSynchronize(s->stream), "stats");
  dsmc_surrogate_fit f;
  std::memset(&f, 0, sizeof(f));
  f.n_samples = s->n_samples;
  f.n_v = st[17];
  f.n_c = st[13];
  // Boundary models: no-slip (no weights) and slip (one weight, x = F).
  f.log_evidence_v[0] = zero_evidence(st[16], st[17], &f.beta_v[0]);
  {
    const double G[9] = {st[15], 0, 0, 0, 0, 0, 0, 0, 0};
    const double pt[3] = {st[14], 0, 0};
    Fit r;
    if (!brr_stats(G, pt, st[16], st[19], st[17], 1, &r))
      return reject(DSMC_E_STATE, "surrogate: slip model posterior not positive definite");
    f.log_evidence_v[1] = r.logev;
    f.alpha_v[1] = r.alpha;
    f.beta_v[1] = r.beta;
    f.sigma_p = r.m[0];
    f.sigma_p_var = r.S[0];
    f.iterations_v = r.iterations;
  }
  // Constitutive models C0..C3.
  f.log_evidence_c[0] = zero_evidence(st[12], st[13], &f.beta_c[0]);
  for (int k = 1; k <= 3; ++k) {
    Fit r;
    if (!brr_stats(st, st + 9, st[12], st[18], st[13], k, &r))
      return reject(DSMC_E_STATE, "surrogate: constitutive posterior not positive definite");
    f.log_evidence_c[k] = r.logev;
    f.alpha_c[k] = r.alpha;
    f.beta_c[k] = r.beta;
    for (int i = 0; i < 3; ++i) f.m_c[k][i] = r.m[i];
    for (int i = 0; i < 9; ++i) f.S_c[k][i] = r.S[i];
    f.iterations_c[k] = r.iterations;
  }
  probabilities(f.log_evidence_v, 2, f.prob_v);
  probabilities(f.log_evidence_c, 4, f.prob_c);
  f.sel_v = select_model(f.log_evidence_v, 2);
  f.sel_c = select_model(f.log_evidence_c, 4);
  for (int l = 0; l < 3; ++l) f.b[l] = s->b[l];
  s->fit = f;
  s->fitted = true;
  *out = f;
  return DSMC_OK;
}

dsmc_status dsmc_surrogate_correction(const dsmc_surrogate_fit* fit, int n, double* S_faces,
                                      void* stream) {
  if (!fit || !S_faces) return reject(DSMC_E_INVAL, "surrogate: NULL");
  if (n < 1 || fit->sel_c < 0 || fit->sel_c > 3)
    return reject(DSMC_E_INVAL, "surrogate: n >= 1 and a selected model in C0..C3");
  cudaStream_t st = (cudaStream_t)stream;
  double* d = nullptr;
  SUR_CUDA(cudaMalloc(&d, ((size_t)n + 1) * sizeof(double)), "correction memory");
  const int k = fit->sel_c;
  const double* m = fit->m_c[k];
  k_correction<<<(n + 1 + 127) / 128, 128, 0, st>>>(k, m[0], m[1], m[2], fit->b[0], fit->b[1],
                                                    fit->b[2], n, d);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(S_faces, d, ((size_t)n + 1) * sizeof(double), cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(d);
  if (e != cudaSuccess) return cuda_reject(e, "correction");
  return DSMC_OK;
}

dsmc_status dsmc_surrogate_profile(dsmc_surrogate_handle s, const dsmc_surrogate_fit* fit,
                                   int n_cfd, const double* z, int n_trials, double* u_mean,
                                   double* u_std) {
  if (!s || !z || !u_mean) return reject(DSMC_E_INVAL, "surrogate: NULL");
  if (n_cfd < 1 || n_trials < 1) return reject(DSMC_E_INVAL, "surrogate: n_cfd, n_trials >= 1");
  if (!fit && !s->fitted) return reject(DSMC_E_STATE, "surrogate: no fit");
  const dsmc_surrogate_fit& f = fit ? *fit : s->fit;
  if (f.sel_v < 0 || f.sel_v > 1 || f.sel_c < 0 || f.sel_c > 3)
    return reject(DSMC_E_INVAL, "surrogate: selected models out of range");
  TrialModels tm{};
  tm.sel_v = f.sel_v;
  tm.k = f.sel_c;
  tm.m_v = f.sigma_p;
  tm.sd_v = std::sqrt(f.sigma_p_var);
  for (int i = 0; i < 3; ++i) tm.m[i] = f.m_c[f.sel_c][i];
  const double* S = f.S_c[f.sel_c];
  for (int i = 0; i < tm.k; ++i)  // Cholesky S = L L^T; a direction without variance gets none
    for (int j = 0; j <= i; ++j) {
      double x = S[i * 3 + j];
      for (int q = 0; q < j; ++q) x -= tm.L[i * 3 + q] * tm.L[j * 3 + q];
      if (i == j)
        tm.L[i * 3 + i] = std::sqrt(x > 0.0 ? x : 0.0);
      else
        tm.L[i * 3 + j] = tm.L[j * 3 + j] > 0.0 ? x / tm.L[j * 3 + j] : 0.0;
    }
  tm.kn = s->Kn;
  tm.F = s->F;
  for (int l = 0; l < 3; ++l) tm.b[l] = f.b[l];
  tm.n = n_cfd;
  // device space: z, weights, profiles of the unit right sides, mean, sd
  const size_t need = 8 * (size_t)n_trials + 6 * (size_t)n_cfd;
  if (need > s->trials_cap) {
    cudaFree(s->trials);
    s->trials = nullptr;
    s->trials_cap = 0;
    SUR_CUDA(cudaMalloc(&s->trials, need * sizeof(double)), "trial memory");
    s->trials_cap = need;
  }
  double* zd = s->trials;
  double* weights = zd + (size_t)n_trials * 4;
  double* modes = weights + (size_t)n_trials * 4;
  double* md = modes + (size_t)n_cfd * 4;
  double* sd = md + n_cfd;
  SUR_CUDA(cudaMemcpyAsync(zd, z, (size_t)n_trials * 4 * sizeof(double), cudaMemcpyDefault,
                           s->stream),
           "copy z");
  k_modes<<<tm.k + 1 + (n_trials + kThreads - 1) / kThreads, kThreads, 0, s->stream>>>(
      tm, zd, n_trials, modes, weights);
  SUR_CUDA(cudaGetLastError(), "modes kernel");
  k_bands<<<n_cfd, kThreads, 0, s->stream>>>(modes, weights, tm.k, n_trials, n_cfd, md, sd);
  SUR_CUDA(cudaGetLastError(), "bands kernel");
  if (u_std && n_trials > 1 && tm.sel_v == 0 && tm.k == 0) {
    k_same_profiles_sd<<<1, kThreads, 0, s->stream>>>(tm.kn, tm.F, n_cfd, n_trials, modes,
                                                      modes + n_cfd, sd);
    SUR_CUDA(cudaGetLastError(), "profile kernel");
  }
  SUR_CUDA(cudaMemcpyAsync(u_mean, md, n_cfd * sizeof(double), cudaMemcpyDefault, s->stream),
           "copy mean");
  if (u_std)
    SUR_CUDA(cudaMemcpyAsync(u_std, sd, n_cfd * sizeof(double), cudaMemcpyDefault, s->stream),
             "copy sd");
  SUR_CUDA(cudaStreamSynchronize(s->stream), "profile");
  return DSMC_OK;
}

}  // extern "C"

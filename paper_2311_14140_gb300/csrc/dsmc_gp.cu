// dsmc_gp.cu -- a Gaussian-process variant of the surrogate stage, not the paper's
// method (whose surrogates are Bayesian ridge regressions per flow case, Sec. 2.3): a GP
// over the (Kn, force) design of many DSMC runs predicts the slip coefficient and the
// stress correction of a new case, and the 1D CFD (Eq. 8 with Eq. 10) uses them.
//
// GP regression as in Rasmussen and Williams (2006), Ch. 2 and Sec. 5.4: squared-
// exponential covariance exp(-1/2 sum_d ((x_d - x'_d) / l_d)^2) over two inputs scaled to
// the unit square, noise variance s2 on the diagonal; each output column standardised
// (mean, standard deviation) and sharing the covariance.  All binary64 on the device:
//   k_gp_standardise  per output column: mean and standard deviation;
//   k_gp_factor       one CTA per hyperparameter point: the covariance in shared memory, its
//                     Cholesky factor (right-looking), log|K|; the factor goes to memory;
//   k_gp_lml          one CTA per hyperparameter point and 8 output columns: the forward
//                     solve L z = y and z^T z.  The summed log marginal likelihood of a point
//                     is -1/2 sum_o z_o^T z_o - m sum log L_kk - n m/2 log 2 pi;
//   k_gp_alpha        one CTA per 8 columns: alpha = K^-1 y at the chosen point (forward
//                     and back substitution);
//   k_gp_predict      one CTA per query point: k(x*, X) in shared memory, then every
//                     column's mean mu + sd (k* . alpha);
//   k_cfd_faces       the finite-volume solve of Eq. 8 with the stress correction given at
//                     the faces, one CTA: closed form up to a prefix sum.
// Binary64 runs at two operations per clock and SM on the GB300, so the triangular solves (n^2
// / 2 fused multiply-adds per column and point) are spread over all SMs and use fma().  64
// points, 202 columns, 90 hyperparameter points: fit 1.50 -> 0.30 ms (factors 68 us, solves 90,
// alpha 29; the solves' floor at that rate is 72 us), one CFD solve 309 -> 51 us (6.5 us of it
// the kernel), when every column was one thread's solve in local memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "dsmc.h"
#include "dsmc_internal.h"

namespace {

constexpr int kGpThreads = 256;
constexpr double kSqrtPi = 1.7724538509055160273;
constexpr double kLog2Pi = 1.8378770664093454836;

dsmc_status reject(dsmc_status s, const std::string& msg) {
  dsmc::set_last_error(msg);
  return s;
}

dsmc_status cuda_reject(cudaError_t e, const char* what) {
  return reject(DSMC_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define GP_CUDA(call, what)                            \
  do {                                                 \
    cudaError_t e_ = (call);                           \
    if (e_ != cudaSuccess) return cuda_reject(e_, what); \
  } while (0)

__device__ __forceinline__ double se_kernel(double ax, double ay, double bx, double by,
                                            double l1, double l2) {
  const double d1 = (ax - bx) / l1, d2 = (ay - by) / l2;
  return exp(-0.5 * (d1 * d1 + d2 * d2));
}

// A warp's 32 columns per block of (32, 8): each row group of 8 sums its rows.
__global__ void __launch_bounds__(kGpThreads)
    k_gp_standardise(const double* __restrict__ Y, int n, int m, double* __restrict__ Ys,
                     double* __restrict__ mu, double* __restrict__ sd) {
  __shared__ double part[8][33];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int o = blockIdx.x * 32 + tx;
  auto total = [&](double v) {  // sum over the row groups, to all of them
    part[ty][tx] = v;
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += part[k][tx];
    __syncthreads();
    return s;
  };
  double s = 0.0;
  if (o < m)
    for (int i = ty; i < n; i += 8) s += Y[(size_t)i * m + o];
  const double mean = total(s) / n;
  double v = 0.0;
  if (o < m)
    for (int i = ty; i < n; i += 8) {
      const double d = Y[(size_t)i * m + o] - mean;
      v = fma(d, d, v);
    }
  double sdv = sqrt(total(v) / n);
  if (!(sdv > 0.0)) sdv = 1.0;
  if (o >= m) return;
  if (ty == 0) {
    mu[o] = mean;
    sd[o] = sdv;
  }
  const double inv = 1.0 / sdv;
  for (int i = ty; i < n; i += 8) Ys[(size_t)i * m + o] = (Y[(size_t)i * m + o] - mean) * inv;
}

// Lower triangles are packed by rows: element (i, j <= i) at i (i + 1) / 2 + j.
__host__ __device__ constexpr int tri(int i) { return i * (i + 1) / 2; }

// K = k(X, X) + s2 I in shared memory, its lower Cholesky factor in place, then the factor as
// the solves take it (packed; L_ij / L_jj below the diagonal, 1 / L_ii on it) to Lout and
// sum log L_kk to logdet; logdet = NaN if a pivot is not positive.  The elements are numbered from the last
// column backwards, so the trailing block of step k is the first r (r + 1) / 2 of them
// (r = n - 1 - k) and every warp's lanes all have work: binary64 instructions cost a full
// warp's 16 cycles whatever the number of active lanes.  The thread of the next pivot forms
// its inverse square root while the others are still updating.
__global__ void __launch_bounds__(kGpThreads)
    k_gp_factor(const double* __restrict__ X, int n, const double* __restrict__ grid,
                double* __restrict__ Lout, double* __restrict__ logdet) {
  extern __shared__ double A[];
  __shared__ double diag[DSMC_GP_MAX_POINTS], inv_sh;
  __shared__ int bad;
  const int nt = tri(n);
  ushort2* ij = reinterpret_cast<ushort2*>(A + nt);  // (row, column) of element e
  const double* g = grid + 3 * (size_t)blockIdx.x;
  const int t = threadIdx.x;
  for (int j = n - 1 - t; j >= 0; j -= kGpThreads)
    for (int i = j; i < n; ++i)
      ij[tri(n - 1 - j) + (i - j)] = make_ushort2((unsigned short)i, (unsigned short)j);
  if (t == 0) bad = 0;
  __syncthreads();
  {
    // (a subnormal length scale has no finite reciprocal, and 0 times infinity is no distance)
    const double i1 = 1.0 / g[0], i2 = 1.0 / g[1], s2 = g[2];
    const bool divide = isinf(i1) || isinf(i2);
    for (int e = t; e < nt; e += kGpThreads) {
      const int i = ij[e].x, j = ij[e].y;
      double d1 = X[2 * i] - X[2 * j], d2 = X[2 * i + 1] - X[2 * j + 1];
      d1 = divide ? d1 / g[0] : d1 * i1;
      d2 = divide ? d2 / g[1] : d2 * i2;
      const double k = exp(-0.5 * fma(d1, d1, d2 * d2));
      A[tri(i) + j] = i == j ? k + s2 : k;
    }
  }
  auto pivot = [&](int k) {  // by one thread, after element (k, k) has its last update
    double d = A[tri(k) + k];
    if (!(d > 0.0)) {
      bad = 1;
      d = 1.0;
    }
    inv_sh = rsqrt(d);
    diag[k] = d;
  };
  __syncthreads();
  if (t == 0) pivot(0);
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    const double inv = inv_sh;
    for (int i = k + 1 + t; i < n; i += kGpThreads) A[tri(i) + k] *= inv;
    if (t == 0) A[tri(k) + k] = inv;
    __syncthreads();
    const int nr = tri(n - 1 - k);
    // element (k + 1, k + 1) is the first of the trailing block's last column: number
    // tri(n - 2 - k)
    const int next = k + 1 < n ? tri(n - 2 - k) : -1;
    for (int e = t; e < nr; e += kGpThreads) {
      const int i = ij[e].x, j = ij[e].y;
      A[tri(i) + j] = fma(-A[tri(i) + k], A[tri(j) + k], A[tri(i) + j]);
      if (e == next) pivot(k + 1);
    }
    __syncthreads();
  }
  double* out = Lout + (size_t)blockIdx.x * nt;
  for (int e = t; e < nt; e += kGpThreads) {
    const int i = ij[e].x, j = ij[e].y;
    const double v = A[tri(i) + j];
    out[tri(i) + j] = i == j ? v : v * A[tri(j) + j];
  }
  if (t < 32) {
    double s = 0.0;
    for (int k = t; k < n; k += 32) s += 0.5 * log(diag[k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (t == 0) logdet[blockIdx.x] = bad ? nan("") : s;
  }
}

// A CTA's solves: kSolveCols columns, a warp covering 4 rows of 8 columns, right-looking (once
// a row's value is known, all later rows are updated at once: no chain of dependent binary64
// operations longer than one per row).  L (packed) and the columns z[row][column] in shared
// memory.
constexpr int kSolveCols = 8;

__device__ __forceinline__ void load_solve(const double* __restrict__ L,
                                           const double* __restrict__ Ys, int n, int m, int o0,
                                           double* Ls, double* z) {
  const int t = threadIdx.x, c = t & (kSolveCols - 1);
  for (int e = t; e < tri(n); e += kGpThreads) Ls[e] = L[e];
  const int o = min(o0 + c, m - 1);
  for (int i = t / kSolveCols; i < n; i += kGpThreads / kSolveCols)
    z[i * kSolveCols + c] = Ys[(size_t)i * m + o];
  __syncthreads();
}

// s = (L D^-1)^-1 y in z, D the diagonal of L: row i of L^-1 y is s_i / L_ii.
__device__ __forceinline__ void solve_forward(const double* Ls, double* z, int n) {
  const int t = threadIdx.x, c = t & (kSolveCols - 1), r0 = t / kSolveCols;
  for (int i = 0; i + 1 < n; ++i) {
    const double v = z[i * kSolveCols + c];
    for (int r = i + 1 + r0; r < n; r += kGpThreads / kSolveCols)
      z[r * kSolveCols + c] = fma(-Ls[tri(r) + i], v, z[r * kSolveCols + c]);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kGpThreads)
    k_gp_lml(const double* __restrict__ Ls_all, const double* __restrict__ Ys, int n, int m,
             double* __restrict__ zz_out) {
  extern __shared__ double sh[];
  __shared__ double part[kGpThreads / 32];
  double *Ls = sh, *z = sh + tri(n);
  const int o0 = blockIdx.x * kSolveCols, t = threadIdx.x;
  load_solve(Ls_all + (size_t)blockIdx.y * tri(n), Ys, n, m, o0, Ls, z);
  solve_forward(Ls, z, n);
  double zz = 0.0;
  if (o0 + (t & (kSolveCols - 1)) < m)
    for (int i = t / kSolveCols; i < n; i += kGpThreads / kSolveCols) {
      const double v = z[i * kSolveCols + (t & (kSolveCols - 1))] * Ls[tri(i) + i];
      zz = fma(v, v, zz);
    }
#pragma unroll
  for (int k = 16; k > 0; k >>= 1) zz += __shfl_xor_sync(0xffffffffu, zz, k);
  if ((t & 31) == 0) part[t >> 5] = zz;
  __syncthreads();
  if (t == 0) {
    double s = 0.0;
    for (int k = 0; k < kGpThreads / 32; ++k) s += part[k];
    zz_out[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = s;
  }
}

__global__ void __launch_bounds__(kGpThreads)
    k_gp_alpha(const double* __restrict__ L, const double* __restrict__ Ys, int n, int m,
               double* __restrict__ alpha) {
  extern __shared__ double sh[];
  double *Ls = sh, *z = sh + tri(n);
  const int t = threadIdx.x, c = t & (kSolveCols - 1), r0 = t / kSolveCols;
  const int o0 = blockIdx.x * kSolveCols;
  load_solve(L, Ys, n, m, o0, Ls, z);
  solve_forward(Ls, z, n);
  for (int i = r0; i < n; i += kGpThreads / kSolveCols) {
    const double inv = Ls[tri(i) + i];
    z[i * kSolveCols + c] *= inv * inv;
  }
  __syncthreads();
  for (int i = n - 1; i > 0; --i) {  // L^T a = z, divided by D: a_r -= (L_ir / L_rr) a_i
    const double v = z[i * kSolveCols + c];
    for (int r = r0; r < i; r += kGpThreads / kSolveCols)
      z[r * kSolveCols + c] = fma(-Ls[tri(i) + r], v, z[r * kSolveCols + c]);
    __syncthreads();
  }
  if (o0 + c < m)
    for (int i = r0; i < n; i += kGpThreads / kSolveCols)
      alpha[(size_t)i * m + o0 + c] = z[i * kSolveCols + c];
}

__global__ void k_gp_predict(const double* __restrict__ X, int n, int m,
                             const double* __restrict__ alpha, const double* __restrict__ mu,
                             const double* __restrict__ sd, double l1, double l2,
                             const double* __restrict__ Xs, double* __restrict__ out) {
  __shared__ double ks[128];
  const double* x = Xs + 2 * blockIdx.x;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    ks[i] = se_kernel(x[0], x[1], X[2 * i], X[2 * i + 1], l1, l2);
  __syncthreads();
  for (int o = threadIdx.x; o < m; o += blockDim.x) {
    double s = 0.0;
    for (int i = 0; i < n; ++i) s += ks[i] * alpha[(size_t)i * m + o];
    out[(size_t)blockIdx.x * m + o] = mu[o] + sd[o] * s;
  }
}

// With face fluxes q_f (f = 0..n) the rows of the cell-centred finite-volume system say
// q_{i+1} - q_i = src + S_{i+1} - S_i, so q_f = q_0 + R_f with R_f = f src + S_f - S_0; summing
// u_{i+1} - u_i = h q_{i+1} from wall to wall (half cells at both ends, the same wall velocity)
// gives q_0 = -(h sum_{0<f<n} R_f + h/2 R_n) and u_i = uw + h (1/2 + i) q_0 + h sum_{0<f<=i} R_f.
// A sweep of n dependent divisions by one thread took 0.26 ms at 200 cells; this takes 6.5 us.
__global__ void __launch_bounds__(kGpThreads)
    k_cfd_faces(double kn, double F, int n, int slip, double sigma_p,
                const double* __restrict__ S, double* __restrict__ u) {
  __shared__ double wtot[kGpThreads / 32];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const double h = 1.0 / n;
  const double src = -h * kSqrtPi * F / kn;
  const double uw = slip ? sigma_p * F : 0.0;
  const double S0 = S[0];
  double carry = 0.0;  // sum of R over the faces of the earlier chunks
  for (int c0 = 0; c0 < n; c0 += kGpThreads) {
    const int i = c0 + t;
    double x = (i > 0 && i < n) ? i * src + (S[i] - S0) : 0.0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wtot[wid] = x;
    __syncthreads();
    double before = carry, all = 0.0;
    for (int q = 0; q < kGpThreads / 32; ++q) {
      if (q < wid) before += wtot[q];
      all += wtot[q];
    }
    carry += all;
    if (i < n) u[i] = before + x;  // sum over 0 < f <= i
    __syncthreads();
  }
  const double q0 = -(h * carry + 0.5 * h * (n * src + (S[n] - S0)));
  for (int i = t; i < n; i += kGpThreads) u[i] = uw + h * ((0.5 + i) * q0 + u[i]);
}

}  // namespace

struct dsmc_gp {
  int n = 0, m = 0;
  double l1 = 0, l2 = 0, s2 = 0;
  cudaStream_t stream = nullptr;
  double *X = nullptr, *alpha = nullptr, *mu = nullptr, *sd = nullptr;
};

extern "C" {

dsmc_status dsmc_gp_fit(const double* X, const double* Y, int n, int m, const double* grid,
                        int n_grid, void* stream, dsmc_gp_handle* out, double* lml,
                        int* best) {
  if (!out || !X || !Y || !grid) return reject(DSMC_E_INVAL, "gp: NULL argument");
  *out = nullptr;
  if (n < 2 || n > DSMC_GP_MAX_POINTS || m < 1 || n_grid < 1)
    return reject(DSMC_E_INVAL, "gp: 2 <= n <= 128 points, m >= 1 outputs, n_grid >= 1");
  for (int g = 0; g < n_grid; ++g)
    if (!(grid[3 * g] > 0.0) || !(grid[3 * g + 1] > 0.0) || !(grid[3 * g + 2] >= 0.0))
      return reject(DSMC_E_INVAL, "gp: length scales > 0 and noise >= 0");
  cudaStream_t st = (cudaStream_t)stream;
  dsmc_gp* gp = new (std::nothrow) dsmc_gp();
  if (!gp) return reject(DSMC_E_NOMEM, "host allocation failed");
  gp->n = n;
  gp->m = m;
  gp->stream = st;
  // The factors of `chunk` hyperparameter points at a time (64 MiB at most).
  const size_t nn = (size_t)tri(n), nm = (size_t)n * m;
  const int col_blocks = (m + kSolveCols - 1) / kSolveCols;
  const int chunk = (int)std::min<size_t>(
      std::min<size_t>((size_t)n_grid, 65535),
      std::max<size_t>(1, ((size_t)64 << 20) / ((nn + 1 + (size_t)col_blocks) * sizeof(double))));
  // One stream-ordered allocation each for what the handle keeps (X, alpha, mu, sd) and for the
  // fit: Y, its standardised columns, the grid, and the chunk's factors, logs and column sums.
  // (The device's default pool keeps a freed block until the next synchronisation; cudaFree
  // would empty it and cost the next call 0.4 ms.)
  double* tmp = nullptr;
  auto fail = [&](dsmc_status s) {
    if (tmp) cudaFreeAsync(tmp, st);
    dsmc_gp_destroy(gp);
    return s;
  };
  cudaError_t e = cudaMallocAsync(&gp->X, (2 * (size_t)n + nm + 2 * (size_t)m) * sizeof(double), st);
  if (e == cudaSuccess)
    e = cudaMallocAsync(&tmp, (2 * nm + 3 * (size_t)n_grid +
                               (size_t)chunk * (nn + 1 + (size_t)col_blocks)) * sizeof(double), st);
  if (e != cudaSuccess) return fail(cuda_reject(e, "gp allocation"));
  gp->alpha = gp->X + 2 * (size_t)n;
  gp->mu = gp->alpha + nm;
  gp->sd = gp->mu + m;
  double *Yd = tmp, *Ys = Yd + nm, *gd = Ys + nm, *Ls = gd + 3 * (size_t)n_grid;
  double *ld = Ls + (size_t)chunk * nn, *zd = ld + chunk;
  if ((e = cudaMemcpyAsync(gp->X, X, 2 * (size_t)n * sizeof(double), cudaMemcpyDefault, st)) !=
          cudaSuccess ||
      (e = cudaMemcpyAsync(Yd, Y, nm * sizeof(double), cudaMemcpyDefault, st)) != cudaSuccess ||
      (e = cudaMemcpyAsync(gd, grid, 3 * (size_t)n_grid * sizeof(double), cudaMemcpyDefault,
                           st)) != cudaSuccess)
    return fail(cuda_reject(e, "gp copy"));
  const size_t smem = nn * (sizeof(double) + sizeof(ushort2));
  const size_t zmem = (nn + (size_t)n * kSolveCols) * sizeof(double);
  const int most = 112 * 1024;  // of either kind at DSMC_GP_MAX_POINTS
  if ((e = cudaFuncSetAttribute(k_gp_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                most)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(k_gp_lml, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) !=
          cudaSuccess ||
      (e = cudaFuncSetAttribute(k_gp_alpha, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) !=
          cudaSuccess)
    return fail(cuda_reject(e, "gp shared memory"));
  k_gp_standardise<<<(m + 31) / 32, dim3(32, 8), 0, st>>>(Yd, n, m, Ys, gp->mu, gp->sd);
  std::vector<double> host((size_t)n_grid), part((size_t)chunk * (1 + (size_t)col_blocks));
  int b = -1;
  for (int g0 = 0; g0 < n_grid; g0 += chunk) {
    const int ng = std::min(chunk, n_grid - g0);
    k_gp_factor<<<ng, kGpThreads, smem, st>>>(gp->X, n, gd + 3 * (size_t)g0, Ls, ld);
    k_gp_lml<<<dim3(col_blocks, ng), kGpThreads, zmem, st>>>(Ls, Ys, n, m, zd);
    if ((e = cudaGetLastError()) != cudaSuccess) return fail(cuda_reject(e, "gp kernels"));
    // ld and zd are adjacent: logs of all `chunk` points, then the column blocks' sums
    if ((e = cudaMemcpyAsync(part.data(), ld,
                             ((size_t)chunk + (size_t)ng * col_blocks) * sizeof(double),
                             cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
      return fail(cuda_reject(e, "gp marginal likelihoods"));
    for (int g = 0; g < ng; ++g) {
      double zz = 0.0;
      for (int c = 0; c < col_blocks; ++c) zz += part[(size_t)chunk + (size_t)g * col_blocks + c];
      const double v = -0.5 * zz - m * part[g] - 0.5 * (double)n * m * kLog2Pi;
      host[g0 + g] = std::isnan(part[g]) ? -INFINITY : v;
      if (std::isfinite(host[g0 + g]) && (b < 0 || host[g0 + g] > host[b])) b = g0 + g;
    }
  }
  if (b < 0) return fail(reject(DSMC_E_STATE, "gp: no grid point gives a positive definite covariance"));
  gp->l1 = grid[3 * b];
  gp->l2 = grid[3 * b + 1];
  gp->s2 = grid[3 * b + 2];
  const double* Lb = Ls + (size_t)b * nn;
  if (n_grid > chunk) {  // the chosen point's factor may be overwritten
    k_gp_factor<<<1, kGpThreads, smem, st>>>(gp->X, n, gd + 3 * (size_t)b, Ls, ld);
    Lb = Ls;
  }
  k_gp_alpha<<<col_blocks, kGpThreads, zmem, st>>>(Lb, Ys, n, m, gp->alpha);
  if ((e = cudaGetLastError()) != cudaSuccess || (e = cudaStreamSynchronize(st)) != cudaSuccess)
    return fail(cuda_reject(e, "gp alpha"));
  if (lml)
    for (int g = 0; g < n_grid; ++g) lml[g] = host[g];
  if (best) *best = b;
  cudaFreeAsync(tmp, st);
  *out = gp;
  return DSMC_OK;
}

dsmc_status dsmc_gp_predict(dsmc_gp_handle gp, const double* Xs, int ns, double* out) {
  if (!gp || !Xs || !out) return reject(DSMC_E_INVAL, "gp: NULL argument");
  if (ns < 1) return reject(DSMC_E_INVAL, "gp: ns >= 1");
  cudaStream_t st = gp->stream;
  double* xd = nullptr;
  const size_t nx = 2 * (size_t)ns;
  cudaError_t e = cudaMallocAsync(&xd, (nx + (size_t)ns * gp->m) * sizeof(double), st);
  double* od = xd + nx;
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(xd, Xs, 2 * (size_t)ns * sizeof(double), cudaMemcpyDefault, st);
  if (e == cudaSuccess) {
    k_gp_predict<<<ns, kGpThreads, 0, st>>>(gp->X, gp->n, gp->m, gp->alpha, gp->mu, gp->sd,
                                             gp->l1, gp->l2, xd, od);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(out, od, (size_t)ns * gp->m * sizeof(double), cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (xd) cudaFreeAsync(xd, st);
  if (e != cudaSuccess) return cuda_reject(e, "gp predict");
  return DSMC_OK;
}

dsmc_status dsmc_gp_hyper(dsmc_gp_handle gp, double* l1, double* l2, double* s2) {
  if (!gp) return reject(DSMC_E_INVAL, "gp: NULL");
  if (l1) *l1 = gp->l1;
  if (l2) *l2 = gp->l2;
  if (s2) *s2 = gp->s2;
  return DSMC_OK;
}

dsmc_status dsmc_gp_destroy(dsmc_gp_handle gp) {
  if (!gp) return DSMC_OK;
  cudaStreamSynchronize(gp->stream);
  // X, alpha, mu and sd are one allocation, idle by now; the stream may be gone
  if (gp->X && cudaFreeAsync(gp->X, nullptr) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(gp->X);
  }
  delete gp;
  return DSMC_OK;
}

dsmc_status dsmc_cfd_faces(double Kn, double F, int n, int slip, double sigma_p,
                           const double* S_faces, double* u, void* stream) {
  if (!S_faces || !u) return reject(DSMC_E_INVAL, "cfd: NULL argument");
  if (!(Kn > 0.0) || n < 1) return reject(DSMC_E_INVAL, "cfd: Kn > 0, n >= 1");
  cudaStream_t st = (cudaStream_t)stream;
  double* Sd = nullptr;
  cudaError_t e = cudaMallocAsync(&Sd, (2 * (size_t)n + 1) * sizeof(double), st);
  double* ud = Sd + n + 1;
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(Sd, S_faces, ((size_t)n + 1) * sizeof(double), cudaMemcpyDefault, st);
  if (e == cudaSuccess) {
    k_cfd_faces<<<1, kGpThreads, 0, st>>>(Kn, F, n, slip, sigma_p, Sd, ud);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(u, ud, (size_t)n * sizeof(double), cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (Sd) cudaFreeAsync(Sd, st);
  if (e != cudaSuccess) return cuda_reject(e, "cfd");
  return DSMC_OK;
}

}  // extern "C"

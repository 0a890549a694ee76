// Refinement control, correction rebuild, coefficient tables, rho0-gradient reductions and
// the field-layout conversion.
#include "columns.cuh"
#include "kernel_grants.cuh"
#include "kernels.cuh"
#include "residual2.cuh"

namespace pgb {

// ---------------------------------------------------------------------------
// Vertical coefficient tables (one thread per level, FP64; nz values only).
//   W_k = rho_k dz_k, a_k = rho_{k-1/2}/(W_k h_{k-1/2}), c_k = rho_{k+1/2}/(W_k h_{k+1/2}),
//   h_{k+1/2} = (dz_k + dz_{k+1})/2, rho_{k+1/2} = (rho_k + rho_{k+1})/2; a_0 = 0 (zero flux
//   through the bottom face).  Top face: zero flux gives c_{nz-1} = 0; p = 0 on it (Dirichlet)
//   gives the flux rho_top (0 - p_{nz-1})/(dz_{nz-1}/2), so c_{nz-1} = rho_top/(W h) with
//   h = dz_{nz-1}/2 and rho_top = rho_{nz-1} (only centre densities are given).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 split_ff(double x) {
  const float h = __double2float_rn(x);
  const float l = __double2float_rn(x - (double)h);
  return make_float2(h, l);
}

__global__ void k_coefficients(const double* __restrict__ dz, const double* __restrict__ rho, int nz,
                               double* a_d, double* c_d, double* W_d, float* a_f, float* c_f, float2* a_ff,
                               float2* c_ff, int top_dirichlet) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nz; k += blockDim.x * gridDim.x) {
    const double W = rho[k] * dz[k];
    const double up = (k + 1 < nz)      ? (0.5 * (rho[k] + rho[k + 1])) / (0.5 * (dz[k] + dz[k + 1]))
                      : top_dirichlet ? rho[k] / (0.5 * dz[k])
                                      : 0.0;
    const double dn = (k > 0) ? (0.5 * (rho[k - 1] + rho[k])) / (0.5 * (dz[k - 1] + dz[k])) : 0.0;
    const double a = dn / W, c = up / W;
    a_d[k] = a;
    c_d[k] = c;
    W_d[k] = W;
    a_f[k] = __double2float_rn(a);
    c_f[k] = __double2float_rn(c);
    a_ff[k] = split_ff(a);
    c_ff[k] = split_ff(c);
  }
}

cudaError_t launch_coefficients(const double* dz, const double* rho0, int nz, double* a_d, double* c_d,
                                double* W_d, float* a_f, float* c_f, float2* a_ff, float2* c_ff, int top_dirichlet,
                                cudaStream_t st) {
  k_coefficients<<<(nz + 127) / 128, 128, 0, st>>>(dz, rho0, nz, a_d, c_d, W_d, a_f, c_f, a_ff, c_ff, top_dirichlet);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Limiting accuracy of the mixed refinement: the part of the error that no sweep
// removes, because the residual r = S - mu_W - L p is formed in double-float
// arithmetic (unit roundoff u = 2^-48).  Each of the operator's products rounds
// at about u K |p| (K = max_k (a_k + c_k) + 2/dx^2 + 2/dy^2, the largest
// coefficient sum), so r carries noise of size about u K ||p|| that is
// uncorrelated from point to point, and the correction solved from it carries
// L^{-1} of that noise.  For noise of equal variance in every mode the expected
// norm is u K ||p|| sqrt(mean over the modes of 1/lambda^2), lambda running over
// the eigenvalues lambda_h(kx, ky) + mu_m of the discrete operator (the singular
// mode of the Neumann problem excluded: the solve projects it out).  The
// vertical operator W^{-1} M (M symmetric) is similar to the symmetric
// tridiagonal B = W^{-1/2} M W^{-1/2}; its mu_m come from Sturm-count bisection.
// The similarity is not orthogonal, so a noise vector's plain norm can grow by up
// to the factor eta = nz sum W^2/(sum W)^2 >= 1 in the dominant (vertically
// constant) modes; the term is multiplied by sqrt(eta).  Result:
//     F = u K sqrt(eta) sqrt(sum_{modes} 1/lambda^2 / N),   N = nx ny nz,
// the relative error below which the refinement's error bound cannot certify a
// result; it is added to every bound.  The sum over (kx, ky) uses the
// geometric-grid value g(t_j) >= g(lambda_h), t_j <= lambda_h, of the decreasing
// g(lambda) = sum_m 1/(lambda + mu_m)^2 (at most (t_{j+1}/t_j)^2 = 1.06 too large).
// One block; fixed-order sums (deterministic).
// ---------------------------------------------------------------------------
constexpr int kFloorThreads = 512;   // >= the largest nz a plan accepts
constexpr int kFloorGrid = 512;

__device__ int sturm_count(const double* d, const double* e2, int nz, double x) {
  // eigenvalues of B below x = negative pivots of the LDL^T factorisation of B - x I
  int cnt = 0;
  double q = d[0] - x;
  for (int k = 0;;) {
    if (q < 0) ++cnt;
    if (++k == nz) break;
    const double qq = (q != 0.0) ? q : -1e-300;
    q = d[k] - x - e2[k - 1] / qq;
  }
  return cnt;
}

__global__ void __launch_bounds__(kFloorThreads) k_accuracy_floor(const double* __restrict__ a,
                                                                   const double* __restrict__ c,
                                                                   const double* __restrict__ W, int nz, int nx,
                                                                   int ny, double dx, double dy, int top_dirichlet,
                                                                   double* __restrict__ out) {
  __shared__ double d[kFloorThreads], e2[kFloorThreads], mu[kFloorThreads];
  __shared__ double g[kFloorGrid];
  __shared__ double red[6][kFloorThreads];
  const int t = threadIdx.x;
  double kmax = 0, sw = 0, sw2 = 0, gmax = 0, wmax = 0, wmin = 1e300;
  for (int k = t; k < nz; k += blockDim.x) {
    d[k] = a[k] + c[k];
    e2[k] = (k + 1 < nz) ? c[k] * a[k + 1] : 0.0;   // squared off-diagonal of B between k and k+1
  }
  __syncthreads();
  for (int k = t; k < nz; k += blockDim.x) {
    kmax = fmax(kmax, d[k]);
    wmax = fmax(wmax, W[k]);
    wmin = fmin(wmin, W[k]);
    sw += W[k];
    sw2 += W[k] * W[k];
    const double off = ((k > 0) ? sqrt(e2[k - 1]) : 0.0) + ((k + 1 < nz) ? sqrt(e2[k]) : 0.0);
    gmax = fmax(gmax, d[k] + off);   // Gershgorin bound on the spectrum of B
  }
  red[0][t] = kmax;
  red[1][t] = sw;
  red[2][t] = sw2;
  red[3][t] = gmax;
  red[4][t] = wmax;
  red[5][t] = wmin;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (t < h) {
      red[0][t] = fmax(red[0][t], red[0][t + h]);
      red[1][t] += red[1][t + h];
      red[2][t] += red[2][t + h];
      red[3][t] = fmax(red[3][t], red[3][t + h]);
      red[4][t] = fmax(red[4][t], red[4][t + h]);
      red[5][t] = fmin(red[5][t], red[5][t + h]);
    }
    __syncthreads();
  }
  const double wratio = (red[5][0] > 0) ? red[4][0] / red[5][0] : 1.0;
  const double K = red[0][0] + 2.0 / (dx * dx) + 2.0 / (dy * dy);
  const double eta = (red[1][0] > 0) ? nz * red[2][0] / (red[1][0] * red[1][0]) : 1.0;
  const double top = red[3][0] * (1.0 + 1e-12) + 1e-300;
  // mu_m, m-th smallest eigenvalue of B (count(x) <= m exactly for x <= mu_m), to a relative
  // 1e-7; with zero flux through top and bottom mu_0 = 0 (the constants are the null space)
  for (int m = t; m < nz; m += blockDim.x) {
    double lo = 0.0, hi = top;
    if (m > 0 || top_dirichlet) {
      for (int it = 0; it < 200 && hi - lo > 1e-7 * hi; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (sturm_count(d, e2, nz, mid) <= m) lo = mid;
        else hi = mid;
      }
      mu[m] = 0.5 * (lo + hi);
    } else {
      mu[m] = 0.0;
    }
  }
  __syncthreads();
  // g on the grid t_j = lam_lo exp(j h) spanning the nonzero horizontal eigenvalues
  const double sx = sinpi(1.0 / nx), sy = sinpi(1.0 / ny);
  const double lam_lo = fmin(4.0 / (dx * dx) * sx * sx, 4.0 / (dy * dy) * sy * sy);
  const double lam_hi = 4.0 / (dx * dx) + 4.0 / (dy * dy);
  const double hstep = log(lam_hi / lam_lo) / (kFloorGrid - 1);
  for (int j = t; j < kFloorGrid; j += blockDim.x) {
    const double tj = lam_lo * exp(j * hstep);
    double s = 0;
    for (int m = 0; m < nz; ++m) {
      const double v = 1.0 / (tj + mu[m]);
      s += v * v;
    }
    g[j] = s;
  }
  __syncthreads();
  // sum over the wavenumber pairs, each unique |kx|, |ky| with its multiplicity
  const int ux = nx / 2 + 1, uy = ny / 2 + 1;
  double acc = 0;
  for (long long pidx = t; pidx < (long long)ux * uy; pidx += blockDim.x) {
    const int kx = (int)(pidx % ux), ky = (int)(pidx / ux);
    const double mx = (kx == 0 || 2 * kx == nx) ? 1.0 : 2.0;
    const double my = (ky == 0 || 2 * ky == ny) ? 1.0 : 2.0;
    const double s1 = sinpi((double)kx / nx), s2 = sinpi((double)ky / ny);
    const double lam = 4.0 / (dx * dx) * s1 * s1 + 4.0 / (dy * dy) * s2 * s2;
    double gv;
    if (kx == 0 && ky == 0) {   // the mean column: its own eigenvalues, the singular one excluded
      gv = 0;
      for (int m = top_dirichlet ? 0 : 1; m < nz; ++m) gv += 1.0 / (mu[m] * mu[m]);
    } else {
      int j = (int)floor(log(lam / lam_lo) / hstep);
      j = max(0, min(kFloorGrid - 1, j));
      while (j > 0 && lam_lo * exp(j * hstep) > lam) --j;
      gv = g[j];
    }
    acc += mx * my * gv;
  }
  red[0][t] = acc;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (t < h) red[0][t] += red[0][t + h];
    __syncthreads();
  }
  if (t == 0) {
    const double u = 0x1p-48;
    const double npts = (double)nx * ny * nz;
    out[0] = u * K * sqrt(eta) * sqrt(red[0][0] / npts);
    out[1] = wratio;
    out[2] = sqrt(eta) * sqrt(red[0][0] / npts);   // the same amplification for any residual noise
  }
}

cudaError_t launch_accuracy_floor(const double* a_d, const double* c_d, const double* W_d, int nz, int nx, int ny,
                                  double dx, double dy, int top_dirichlet, double* out, cudaStream_t st) {
  if (nz > kFloorThreads) return cudaErrorInvalidValue;
  k_accuracy_floor<<<1, kFloorThreads, 0, st>>>(a_d, c_d, W_d, nz, nx, ny, dx, dy, top_dirichlet, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Pivot reciprocals of the listed low-|k| columns, a block per column: tab[0][n][nz], 1/u_k eliminated from the bottom
// (with the step the sequential column solves use, lowk_pivot_step, so that reading the table gives the same solution
// bit for bit), and tab[1][n][nz], the twisted ones of lowk_column_tab: 1/u_k below m = nz/2, from the top
// 1/v_k (h_{nz-1} = s + c_{nz-1}, h_k = s + c_k h_{k+1}/v_{k+1}, v_k = h_k + a_k) above it, and
// 1/(s + a_m g_{m-1}/u_{m-1} + c_m h_{m+1}/v_{m+1}) at m (0 for the singular column).  A column without row
// sum (the mean column) has g = h = 0 but for the top coupling: its levels are independent.  After both: 1/sum W.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(64) k_lowk_pivots(const int2* __restrict__ cols, int n, const double* __restrict__ a,
                                                    const double* __restrict__ c, const double* __restrict__ lamx,
                                                    const double* __restrict__ lamy, const double* __restrict__ W,
                                                    int nz, int singular00, double* __restrict__ tab) {
  const int j = blockIdx.x, t = threadIdx.x, m = nz / 2;
  if (j == 0 && t < 32) {
    double sw = 0.0;
    for (int k = t; k < nz; k += 32) sw += W[k];
    for (int o = 16; o > 0; o >>= 1) sw += __shfl_down_sync(0xffffffffu, sw, o);
    if (t == 0) tab[2 * (size_t)n * nz] = 1.0 / sw;
  }
  const int2 ck = cols[j];
  const bool singular = singular00 && ck.x == 0 && ck.y == 0;
  const double s = singular ? 0.0 : -(lamx[ck.x] + lamy[ck.y]);
  double* lower = tab + (size_t)j * nz;
  double* tw = tab + (size_t)(n + j) * nz;
  __shared__ double meet[2];   // g_{m-1}/u_{m-1}, h_{m+1}/v_{m+1}
  if (s == 0.0) {
    for (int k = t; k < nz; k += blockDim.x) lower[k] = singular && k == nz - 1 ? 0.0 : 1.0 / c[k];
    if (t == 0) meet[0] = 0.0;
  } else if (t == 0) {
    double g_prev = s, inv_prev = 0.0;
    for (int k = 0; k < nz; ++k) {
      const double inv = lowk_pivot_step(k, s, a[k], c[k], g_prev, inv_prev, false);
      lower[k] = inv;
      inv_prev = inv;
      if (k == m - 1) meet[0] = g_prev * inv;
    }
  }
  if (singular) {   // h = 0 throughout
    for (int k = m + 1 + t; k < nz; k += blockDim.x) tw[k] = 1.0 / a[k];
    if (t == 32) meet[1] = m + 1 < nz ? 0.0 : 1.0;
  } else if (t == 32) {
    double ratio = 1.0;   // above the top: the face's coupling enters the top row's sum
    for (int k = nz - 1; k > m; --k) {
      const double h = s + c[k] * ratio, inv = 1.0 / (h + a[k]);
      tw[k] = inv;
      ratio = h * inv;
    }
    meet[1] = ratio;
  }
  __syncthreads();
  for (int k = t; k < m; k += blockDim.x) tw[k] = lower[k];
  if (t == 0) tw[m] = singular ? 0.0 : 1.0 / (s + a[m] * meet[0] + c[m] * meet[1]);
}
cudaError_t launch_lowk_pivots(const int2* cols, int n, const double* a_d, const double* c_d, const double* lamx_d,
                               const double* lamy_d, const double* W_d, int nz, int singular00, double* inv_tab,
                               cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_lowk_pivots<<<n, 64, 0, st>>>(cols, n, a_d, c_d, lamx_d, lamy_d, W_d, nz, singular00, inv_tab);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Refinement control: sums the x-pass partials in a fixed order (the inverse
// x-pass's delta^2, p^2, sum p and the forward x-pass's r^2, S^2), records the
// relative update, relative residual and error bound, and sets the done flag
// (control_decide in kernels.cuh states the stopping rule).
// ---------------------------------------------------------------------------
// Stage 1 (kControlBlocks blocks): each block sums a contiguous range of the
// partials in a fixed order; the last block to finish (ticket counter) sums the
// block results in block order and applies the stopping rule.  Deterministic.
constexpr int kControlBlocks = 64;

__global__ void __launch_bounds__(256) k_control(Stats* st, const double* __restrict__ partials, int nblocks,
                                                  const double* __restrict__ res_partials, int res_nblocks,
                                                  int pass, int max_sweeps, double tol,
                                                  const double* __restrict__ floor, long long npoints,
                                                  int wrote_p, double* __restrict__ stage,
                                                  unsigned* __restrict__ ticket) {
  __shared__ double sh[5][256];
  __shared__ bool last;
  if (st->done) return;   // later sweeps after convergence: nothing to do
  const int t = threadIdx.x;
  const int per = (nblocks + gridDim.x - 1) / gridDim.x;
  const int b0 = blockIdx.x * per, b1 = min(nblocks, b0 + per);
  const int rper = (res_nblocks + gridDim.x - 1) / gridDim.x;
  const int r0 = blockIdx.x * rper, r1 = min(res_nblocks, r0 + rper);
  double v[5] = {0, 0, 0, 0, 0};
  for (int i = b0 + t; i < b1; i += blockDim.x) {
    v[0] += partials[3 * i];
    v[1] += partials[3 * i + 1];
    v[2] += partials[3 * i + 2];
  }
  for (int i = r0 + t; i < r1; i += blockDim.x) {
    v[3] += res_partials[2 * i];
    v[4] += res_partials[2 * i + 1];
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) sh[k][t] = v[k];
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (t < h) {
#pragma unroll
      for (int k = 0; k < 5; ++k) sh[k][t] += sh[k][t + h];
    }
    __syncthreads();
  }
  if (t == 0) {
#pragma unroll
    for (int k = 0; k < 5; ++k) stage[5 * blockIdx.x + k] = sh[k][0];
    __threadfence();
    last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!last || t != 0) return;
  __threadfence();
  double tot[5] = {0, 0, 0, 0, 0};
  for (int i = 0; i < (int)gridDim.x; ++i)
#pragma unroll
    for (int k = 0; k < 5; ++k) tot[k] += stage[5 * i + k];
  *ticket = 0;   // ready for the next pass
  control_decide(st, tot[0], tot[1], tot[2], tot[3], tot[4], pass, max_sweeps, tol, npoints, wrote_p, *floor);
}

// ---------------------------------------------------------------------------
// Verification of the current iterate by the next correction's norm (see launch_verify in
// kernels.cuh).  One block; fixed-order sums.
// ---------------------------------------------------------------------------
constexpr int kVerifyThreads = 256;
__global__ void __launch_bounds__(kVerifyThreads) k_verify(Stats* st, const double* __restrict__ sq, int nsq,
                                                           const double* __restrict__ res_partials, int res_nblocks,
                                                           int pass, double tol, const double* __restrict__ floor,
                                                           double nxny, int p_stored, double inv_lcut2, int from_r0) {
  __shared__ double sh[3][kVerifyThreads];
  if (st->done) return;   // an earlier pass already ended the refinement
  const int t = threadIdx.x;
  double a = 0, b = 0, c = 0;
  for (int i = t; i < nsq; i += kVerifyThreads) a += sq[i];
  for (int i = t; i < res_nblocks; i += kVerifyThreads) {
    b += res_partials[2 * i];
    c += res_partials[2 * i + 1];
  }
  sh[0][t] = a;
  sh[1][t] = b;
  sh[2][t] = c;
  __syncthreads();
  // one warp per sum: the FP64 unit takes a warp's addition in 76 clocks, so what counts is their number in a row
  // (a tree over 1024 threads: 8.7 -> 7.2 us at 64 x 64 x 48)
  if (t < 96) {
    const int q = t >> 5;
    double x = 0.0;
    for (int i = t & 31; i < kVerifyThreads; i += 32) x += sh[q][i];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    __syncwarp();
    if ((t & 31) == 0) sh[q][0] = x;
  }
  __syncthreads();
  if (t != 0) return;
  double sd = nxny * sh[0][0];
  // low wavenumbers only: every other column of the correction is (lambda_h + T)^{-1} of the residual's
  // column, with T = W^{-1} M similar to a positive semidefinite matrix through W^{1/2}, so its norm is at
  // most sqrt(W_max/W_min)/lambda_h <= sqrt(W_max/W_min)/lambda_cut times the residual column's (Parseval)
  if (inv_lcut2 > 0) sd += floor[1] * inv_lcut2 * sh[1][0];
  double fl = floor[0], ss = sh[2][0];
  if (from_r0 && pass >= 2) {
    // the residual was formed as r0 - L q from the previous sweep's residual r0 stored in FP32: its
    // rounding (at most 2^-24 ||r0|| in the 2-norm) reaches the correction like the residual's own
    // rounding does, so it adds 2^-24 ||r0|| G/||p|| to the limiting accuracy (G = floor[2]); the
    // source norm is the previous sweep's (this pass did not read S)
    const double sp = st->sq_p[pass - 1];
    if (sp > 0) fl += 0x1p-24 * sqrt(st->sq_res[pass - 2]) * floor[2] / sqrt(sp);
    ss = st->sq_src[pass - 2];
  }
  verify_decide(st, sd, sh[1][0], ss, pass, tol, fl, p_stored);
}

cudaError_t launch_verify(Stats* st_dev, const double* sq, int nsq, const double* res_partials, int res_nblocks,
                          int pass, double tol, const double* floor, double nxny, int p_stored, double inv_lcut2,
                          int from_r0, cudaStream_t st) {
  k_verify<<<1, kVerifyThreads, 0, st>>>(st_dev, sq, nsq, res_partials, res_nblocks, pass, tol, floor, nxny, p_stored,
                               inv_lcut2, from_r0);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Final iterate when the refinement stopped after a sweep that stored only the
// float correction q: p = p0 + q as a double (exact sum of the two floats up to
// the double rounding).  A no-op unless Stats::need_final is set.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_finalize(const float2* __restrict__ p0, const float2* __restrict__ q,
                                                  double2* __restrict__ p, long long npairs,
                                                  const Stats* __restrict__ stats) {
  pdl_trigger();
  pdl_wait();   // the previous kernels of the stream are complete
  if (!stats->need_final) return;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < npairs;
       i += (long long)gridDim.x * blockDim.x) {
    __stcs(&p[i], finalize_pair(__ldcs(&p0[i]), __ldcs(&q[i])));
  }
}

// ---------------------------------------------------------------------------
// Accumulated correction of the refinement, rebuilt before a second or third
// sweep: q = p - p0 to float accuracy, from the double iterate p = p0 + q the
// previous sweep stored ((h, l) = p split into floats; h - p0 is exact when h
// and p0 are within a factor 2, and rounds at 2^-24 |q| otherwise).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_q_rebuild(const double2* __restrict__ p, const float2* __restrict__ p0,
                                                   float2* __restrict__ q, long long npairs,
                                                   const int* __restrict__ done) {
  pdl_trigger();
  pdl_wait();   // the previous kernels of the stream are complete
  if (done && *done) return;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < npairs;
       i += (long long)gridDim.x * blockDim.x) {
    __stcs(&q[i], q_rebuild_pair(__ldcs(&p[i]), __ldcs(&p0[i])));
  }
}

cudaError_t launch_q_rebuild(const double* p, const float* p0, float* q, long long n, const int* done,
                             cudaStream_t st) {
  const long long npairs = n / 2;   // nx is even
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  long long blocks = (npairs + 255) / 256;
  const long long cap = (long long)(sms > 0 ? sms : 1) * 8;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  return pdl_launch(k_q_rebuild, dim3((unsigned)blocks), dim3(256), 0, st, (const double2*)p, (const float2*)p0,
                    (float2*)q, npairs, done);
}

cudaError_t launch_control(Stats* st_dev, const double* partials, int nblocks, const double* res_partials,
                           int res_nblocks, int pass, int max_sweeps, double tol, const double* floor,
                           long long npoints, int wrote_p, cudaStream_t st) {
  k_control<<<kControlBlocks, 256, 0, st>>>(st_dev, partials, nblocks, res_partials, res_nblocks, pass, max_sweeps,
                                            tol, floor, npoints, wrote_p, st_dev->control_stage,
                                            &st_dev->control_ticket);
  return cudaGetLastError();
}

__global__ void k_set_if_not_done(cudaGraphConditionalHandle h, const int* __restrict__ done) {
  cudaGraphSetConditional(h, *done ? 0u : 1u);
}

cudaError_t launch_set_if_not_done(cudaGraphConditionalHandle h, const int* done, cudaStream_t st) {
  k_set_if_not_done<<<1, 1, 0, st>>>(h, done);
  return cudaGetLastError();
}

// Zeroes n 32-bit words.  A kernel rather than cudaMemsetAsync: the solve's statistics are cleared on the
// compute stream, where a memset can be served by a copy engine and wait behind a host copy in flight.
__global__ void __launch_bounds__(256) k_zero_words(unsigned* __restrict__ p, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    p[i] = 0u;
}

cudaError_t launch_zero_words(void* p, size_t bytes, cudaStream_t st) {
  if (bytes % 4) return cudaErrorInvalidValue;
  const long long n = (long long)(bytes / 4);
  if (n == 0) return cudaSuccess;
  long long blocks = (n + 255) / 256;
  if (blocks > 64) blocks = 64;
  k_zero_words<<<(unsigned)blocks, 256, 0, st>>>((unsigned*)p, n);
  return cudaGetLastError();
}

// four ints (src need not be 16-byte aligned)
__global__ void k_copy_status(const int* __restrict__ src, int* dst) {
  dst[0] = src[0];
  dst[1] = src[1];
  dst[2] = src[2];
  dst[3] = src[3];
}

cudaError_t launch_copy_status(const int* src, int* dst, cudaStream_t st) {
  k_copy_status<<<1, 1, 0, st>>>(src, dst);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const float* p0, const float* q, double* p, long long n, const Stats* stats,
                            cudaStream_t st) {
  const long long npairs = n / 2;   // nx is even
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  long long blocks = (npairs + 255) / 256;
  const long long cap = (long long)(sms > 0 ? sms : 1) * 8;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  return pdl_launch(k_finalize, dim3((unsigned)blocks), dim3(256), 0, st, (const float2*)p0, (const float2*)q,
                    (double2*)p, npairs, stats);
}

// ---------------------------------------------------------------------------
// rho0 gradient.  With g = G^T (dL/dp) and D_f = p_{k+1} - p_k on face f = k+1/2:
//   Lo_f = sum_ij g_k D_f,  Up_f = sum_ij g_{k+1} D_f,
//   dL/drho_m = -sum_k (da_k/drho_m * Ma_k + dc_k/drho_m * Mc_k),
//   Mc_k = Lo_k,  Ma_k = -Up_{k-1}.
// Partials per (face, block) are reduced in a fixed order (deterministic).
//
// The double form is bound by the FP64 pipe: one subtraction and two FMAs a point, the level planes of
// neighbouring faces coming from L2.  The block reduction costs as many FP64 instructions per warp as
// some ten points do, so a thread takes at least kGrhoPoints points (one point a thread, as it was,
// spent several times the work of the sums in the reductions: 512 x 512 x 64, both kernels together 831 ->
// about 165 us).  The float
// forms round the products to float and add them in pairs of floats (hi + lo, exact two-sums), so that
// a longer sum per thread loses nothing.
// ---------------------------------------------------------------------------
constexpr int kGrhoPoints = 32;

struct GrhoSumD {   // FP64 fields
  using V = double2;
  double lo0 = 0, up0 = 0, lo1 = 0, up1 = 0;
  __device__ __forceinline__ void add(V p0, V p1, V g0, V g1) {
    const double d0 = p1.x - p0.x, d1 = p1.y - p0.y;
    lo0 = fma(g0.x, d0, lo0);
    up0 = fma(g1.x, d0, up0);
    lo1 = fma(g0.y, d1, lo1);
    up1 = fma(g1.y, d1, up1);
  }
  __device__ __forceinline__ double lo() const { return lo0 + lo1; }
  __device__ __forceinline__ double up() const { return up0 + up1; }
};
struct GrhoSumF {   // float products, sums as float pairs
  using V = float2;
  float lh = 0, ll = 0, uh = 0, ul = 0;
  __device__ __forceinline__ void one(float p0, float p1, float g0, float g1) {
    const float d = p1 - p0;
    float e;
    two_sum(lh, __fmul_rn(g0, d), lh, e);
    ll += e;
    two_sum(uh, __fmul_rn(g1, d), uh, e);
    ul += e;
  }
  __device__ __forceinline__ void add(V p0, V p1, V g0, V g1) {
    one(p0.x, p1.x, g0.x, g1.x);
    one(p0.y, p1.y, g0.y, g1.y);
  }
  // past the float range h is the infinity (or NaN) of a plain sum, and the two-sums' low parts mean nothing
  static __device__ __forceinline__ double value(float h, float l) { return (double)h + (isfinite(h) ? (double)l : 0.0); }
  __device__ __forceinline__ double lo() const { return value(lh, ll); }
  __device__ __forceinline__ double up() const { return value(uh, ul); }
};
struct GrhoSumM : GrhoSumF {   // mixed: double fields, rounded to float with integer operations
  using V = double2;
  __device__ __forceinline__ void add(V p0, V p1, V g0, V g1) {
    one(d2f_int(p0.x), d2f_int(p1.x), d2f_int(g0.x), d2f_int(g1.x));
    one(d2f_int(p0.y), d2f_int(p1.y), d2f_int(g0.y), d2f_int(g1.y));
  }
};

// half: pairs of points per level plane (nx is even, so the planes hold whole, aligned pairs)
template <typename Sum>
__global__ void __launch_bounds__(256) k_grho_partial(const typename Sum::V* __restrict__ gS,
                                                      const typename Sum::V* __restrict__ p, long long half,
                                                      double* __restrict__ partials) {
  const int f = blockIdx.y;
  const typename Sum::V* g0 = gS + f * half;
  const typename Sum::V* p0 = p + f * half;
  Sum a;
#pragma unroll 4
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < half; i += (long long)gridDim.x * blockDim.x)
    a.add(p0[i], p0[i + half], g0[i], g0[i + half]);
  double lo = a.lo(), up = a.up();
  for (int o = 16; o > 0; o >>= 1) {
    lo += __shfl_down_sync(0xffffffffu, lo, o);
    up += __shfl_down_sync(0xffffffffu, up, o);
  }
  __shared__ double s[2][8];
  const int t = threadIdx.x;
  if ((t & 31) == 0) {
    s[0][t >> 5] = lo;
    s[1][t >> 5] = up;
  }
  __syncthreads();
  if (t < 2) {
    double v = 0;
    for (int w = 0; w < 8; ++w) v += s[t][w];
    partials[2 * ((long long)f * gridDim.x + blockIdx.x) + t] = v;
  }
}

// One block per level m: warps 0..3 sum the (Lo, Up) partials of the faces m-1 and m in a fixed order
// (a thread per level looping over every block's partials took 260 us at 512 x 512 x 64).
__global__ void __launch_bounds__(128) k_grho_final(const double* __restrict__ partials, int nb, int nz,
                                                    const double* __restrict__ dz, const double* __restrict__ rho,
                                                    const double* __restrict__ a, const double* __restrict__ c,
                                                    const double* __restrict__ W, double* __restrict__ grho) {
  __shared__ double sum[4];
  const int m = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int f = m - 1 + (w >> 1), which = w & 1;   // face and sum of this warp
  double v = 0;
  if (f >= 0 && f < nz - 1)
    for (int b = lane; b < nb; b += 32) v += partials[2 * ((long long)f * nb + b) + which];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (lane == 0) sum[w] = v;
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double lo_dn = sum[0], up_dn = sum[1], lo_up = sum[2], up_up = sum[3];
  auto hf = [&](int face) { return 0.5 * (dz[face] + dz[face + 1]); };
  double acc = 0;
  // a-terms: k = m (face m-1) and k = m+1 (face m); Ma_k = -Up_{k-1}
  if (m >= 1) acc += (0.5 / (W[m] * hf(m - 1)) - a[m] / rho[m]) * -up_dn;
  if (m + 1 <= nz - 1) acc += (0.5 / (W[m + 1] * hf(m))) * -up_up;
  // c-terms: k = m (face m) and k = m-1 (face m-1); Mc_k = Lo_k
  if (m <= nz - 2) acc += (0.5 / (W[m] * hf(m)) - c[m] / rho[m]) * lo_up;
  if (m >= 1) acc += (0.5 / (W[m - 1] * hf(m - 1))) * lo_dn;
  grho[m] = -acc;
}

cudaError_t launch_grho(int kind, const void* g, const void* p, const Geom& g_, const Tables& tb, const double* dz,
                        const double* rho0, double* partials, int nparts_max, double* grho, cudaStream_t st) {
  const long long half = (long long)g_.nx * g_.ny / 2;
  // kGrhoPoints points a thread, fewer while that leaves less than about four blocks per SM
  const int faces = g_.nz - 1;
  long long nb = (2 * half + 256 * kGrhoPoints - 1) / (256 * kGrhoPoints);
  const long long fill = (4ll * sm_count() + faces - 1) / faces, most = (half + 255) / 256;
  if (nb < fill) nb = fill;
  if (nb > most) nb = most;
  if (nb > nparts_max) nb = nparts_max;
  if (nb < 1) nb = 1;
  const dim3 grid((unsigned)nb, faces);
  if (kind == 0)
    k_grho_partial<GrhoSumD><<<grid, 256, 0, st>>>((const double2*)g, (const double2*)p, half, partials);
  else if (kind == 1)
    k_grho_partial<GrhoSumF><<<grid, 256, 0, st>>>((const float2*)g, (const float2*)p, half, partials);
  else
    k_grho_partial<GrhoSumM><<<grid, 256, 0, st>>>((const double2*)g, (const double2*)p, half, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_grho_final<<<g_.nz, 128, 0, st>>>(partials, (int)nb, g_.nz, dz, rho0, tb.a_d, tb.c_d, tb.W_d, grho);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Field layout conversion.  MONC keeps its fields with the vertical index
// fastest, [nx][ny][nz]; the solver works on [nz][ny][nx].  Both directions are
// the same operation, dst[b][m][a] = src[a][m][b] (a < A, m < M, b < B): a swap
// of the outer and inner axes, done in 32 x 32 tiles of one m through shared
// memory so that the reads (along b) and the writes (along a) are coalesced.
// The padded row (33) keeps the transposed shared reads free of bank conflicts
// for 4-byte elements and for each half-warp of 8-byte ones.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_swap_outer_inner(const T* __restrict__ src, T* __restrict__ dst, int A,
                                                          int M, int B) {
  __shared__ T tile[32][33];
  const int b0 = blockIdx.x * 32, a0 = blockIdx.y * 32, m = blockIdx.z;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const long long src_a = (long long)M * B, dst_b = (long long)M * A;
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const int a = a0 + r, b = b0 + tx;
    if (a < A && b < B) tile[r][tx] = __ldcs(&src[a * src_a + (long long)m * B + b]);   // read once
  }
  __syncthreads();
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const int b = b0 + r, a = a0 + tx;
    if (a < A && b < B) dst[b * dst_b + (long long)m * A + a] = tile[tx][r];
  }
}

cudaError_t launch_swap_outer_inner(const void* src, void* dst, int A, int M, int B, int elem_bytes,
                                    cudaStream_t st) {
  if (A <= 0 || M <= 0 || B <= 0 || M > 65535) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)((B + 31) / 32), (unsigned)((A + 31) / 32), (unsigned)M), block(32, 8);
  if (elem_bytes == 8)
    k_swap_outer_inner<double><<<grid, block, 0, st>>>((const double*)src, (double*)dst, A, M, B);
  else
    k_swap_outer_inner<float><<<grid, block, 0, st>>>((const float*)src, (float*)dst, A, M, B);
  return cudaGetLastError();
}

}  // namespace pgb

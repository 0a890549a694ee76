// Column solves shared by the column kernels (thomas_kernels.cu) and the fused
// spectral-middle kernel (spectral_fused.cu): after the forward transform each
// (kx, ky) wavenumber gives an independent tridiagonal system along z
// (Section 2.1).  The pivot algebra is stated at the top of thomas_kernels.cu.
#pragma once
#include "kernels.cuh"
#include "launch_rules.hpp"

namespace pgb {

template <typename T> __device__ __forceinline__ T rcp(T u);
// single MUFU reciprocal (max error ~1 ulp) on the critical path of the float recurrence
template <> __device__ __forceinline__ float rcp<float>(float u) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(u));
  return r;
}
template <> __device__ __forceinline__ double rcp<double>(double u) { return 1.0 / u; }

__device__ __forceinline__ int signed_ky(int ky, int ny) { return ky > ny / 2 ? ky - ny : ky; }

struct LowkArgs {
  const int2* cols;
  int n;
  const double* a_d;
  const double* c_d;
  const double* W_d;
  const double* lamx_d;
  const double* lamy_d;
  const double* target_mean;
  double scale;   // 1/(nx ny) in double for the double-precision columns
  int singular00; // zero flux at the top: the (0,0) column is singular
  const double* inv_tab;   // [n][nz] twisted pivot reciprocals of the listed columns, then 1/sum W (launch_lowk_pivots)
};

// One step of the low-|k| pivot recurrence (rounded step by step, so that the table built ahead by
// k_lowk_pivots and a column solve computing its own pivots agree bit for bit):
// g_k = s + a_k g_{k-1}/u_{k-1} (g_0 = s), u_k = g_k + c_k, returns 1/u_k (0 for the pinned singular top).
__device__ __forceinline__ double lowk_pivot_step(int k, double s, double ak, double ck, double& g_prev, double inv_prev,
                                                  bool last_singular) {
  const double gk = (k == 0) ? s : __dadd_rn(s, __dmul_rn(__dmul_rn(ak, g_prev), inv_prev));
  const double u = __dadd_rn(gk, ck);
  g_prev = gk;
  return last_singular ? 0.0 : 1.0 / u;   // the singular top pivot is pinned
}

// ---------------------------------------------------------------------------
// Low-|k| and singular columns, in double.  The (0,0) column, when
// zero flux at the top makes it singular:
//   forward: remove the W-weighted mean of the right-hand side (compatibility),
//            pin x_{nz-1} = 0, back-substitute, shift to zero mean;
//   adjoint: remove the plain mean of the right-hand side, pin v_{nz-1} = 0,
//            back-substitute, remove the W direction (x -= W sum(x)/sum(W)).
// ---------------------------------------------------------------------------
// The sequential recurrence of one low-|k| or singular column (forward solve), run by one thread
// out of shared memory: the right-hand side at zx[k ld], zy[k ld] (real and
// imaginary parts; overwritten by the solution before any mean shift), the
// back-substitution factors in w[k ld], the level tables a, c, W (stride 1).
// red receives (shift_x, shift_y, 1, sum x, sum y) for the caller's output
// pass; sq_out (nullable) the sum of |x_k|^2 of the output.
// tab: w[k ld] holds the column's pivot reciprocals 1/u_k on entry (staged by the caller from the
// plan's table, in parallel): the chain then loads them from shared memory instead of forming
// pivots, and the back substitution forms its factors from them (the same products as when they are
// stored by the forward sweep, so both ways give the same bits).
__device__ __forceinline__ void lowk_recurrence(double* zx, double* zy, double* w, int ld, const double* a,
                                                const double* c, const double* W, int nz, int kx, int ky, bool singular,
                                                const double* __restrict__ lamx, const double* __restrict__ lamy,
                                                double scale, const double* __restrict__ target_mean,
                                                Stats* stats, double* red, double* sq_out, bool tab) {
  double mean_x = 0, mean_y = 0;
  if (singular) {
    double sw = 0;
    for (int k = 0; k < nz; ++k) {
      const double wk = W[k];
      mean_x += wk * zx[k * ld];
      mean_y += wk * zy[k * ld];
      sw += wk;
    }
    mean_x /= sw;
    mean_y /= sw;
    // only the first solve records mu_W (a refinement correction solve has a target mean)
    if (stats && !target_mean) stats->mu_w = mean_x * scale;
  }
  const double s = singular ? 0.0 : -(lamx[kx] + lamy[ky]);
  const double ms = -scale;
  double g_prev = s, inv_prev = 0, yx = 0, yy = 0;
  for (int k = 0; k < nz; ++k) {
    const double bx = ms * (zx[k * ld] - mean_x), by = ms * (zy[k * ld] - mean_y);
    // the pivots depend on the column's wavenumbers and the levels only: staged from the plan's
    // table when it has them (no division on the chain), else computed here
    const double inv =
        tab ? w[k * ld] : lowk_pivot_step(k, s, a[k], c[k], g_prev, inv_prev, singular && (k == nz - 1));
    double nx_ = bx, ny_ = by;
    if (k > 0) {
      const double f = a[k] * inv_prev;
      nx_ += f * yx;
      ny_ += f * yy;
    }
    yx = nx_;
    yy = ny_;
    zx[k * ld] = yx * inv;
    zy[k * ld] = yy * inv;
    if (!tab) w[k * ld] = c[k] * inv;
    inv_prev = inv;
  }
  double xx = zx[(nz - 1) * ld], xy = zy[(nz - 1) * ld];
  double sx = xx, sy = xy;
  for (int k = nz - 2; k >= 0; --k) {
    const double wk = !tab ? w[k * ld] : c[k] * w[k * ld];
    xx = zx[k * ld] + wk * xx;
    xy = zy[k * ld] + wk * xy;
    zx[k * ld] = xx;
    zy[k * ld] = xy;
    sx += xx;
    sy += xy;
  }
  double shx = 0, shy = 0;
  if (singular) {
    shx = sx / (double)nz;
    shy = sy / (double)nz;
    // refinement sweep: the correction also removes the mean of the current iterate
    if (target_mean) shx += __ldcg(target_mean);
  }
  red[0] = shx;
  red[1] = shy;
  red[2] = 1;
  red[3] = sx;
  red[4] = sy;
  if (sq_out) {
    double sq = 0;
    for (int k = 0; k < nz; ++k) {
      const double ox = singular ? zx[k * ld] - shx : zx[k * ld], oy = singular ? zy[k * ld] - shy : zy[k * ld];
      sq += ox * ox + oy * oy;
    }
    *sq_out = sq;
  }
}

// Shared memory (in doubles) of one low-|k| column solved by a block.
__host__ __device__ constexpr size_t lowk_smem_elems(int nz) { return 6 * (size_t)nz + 96; }

// Fixed-order sum over the block (every thread gets the result): a shuffle tree over the existing lanes of each warp
// (a block may be half a warp), then the warps in order.  scratch: a double per warp.
__device__ __forceinline__ double lowk_block_sum(double v, double* scratch) {
  const int lane = threadIdx.x & 31, lanes = warp_lanes(threadIdx.x, blockDim.x);
  const unsigned mask = warp_mask(threadIdx.x, blockDim.x);
  for (int o = 16; o > 0; o >>= 1) {
    const double u = __shfl_down_sync(mask, v, o);
    if (lane + o < lanes) v += u;
  }
  const int wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();   // scratch may still be read from an earlier sum
  if ((threadIdx.x & 31) == 0) scratch[wid] = v;
  __syncthreads();
  double r = scratch[0];
  for (int w = 1; w < nw; ++w) r += scratch[w];
  return r;
}

// One low-|k| or singular column in double precision from the plan's table of twisted pivot reciprocals (inv_col,
// k_lowk_pivots: 1/u_k below level m = nz/2, 1/v_k above it, the meeting pivot's at m, 0 where it is singular and
// pinned), solved by the whole block (at most 1024 threads).  The FP64 units take a warp's instruction in about 76
// clocks however few of its lanes are active, so what counts is the length of the serial part: the column is
// eliminated from both ends at once, real and imaginary parts on lanes 0-1 (upwards) and 2-3 (downwards) of the first
// warp, one FMA per level and sweep, nz/2 levels each way (eliminated from the bottom alone, twice that: the
// column kernel of a 64 x 64 x 48 solve 16 -> 10 us, of the first try at 1024 x 1024 x 128 32 -> 27).  Everything
// that does not depend on the previous level runs across the block:
//   z_k = b_k/u_k + (e_k/u_k) z_prev,  x_m = (b_m + e_m z_{m-1} + e'_m z_{m+1})/u_m,  x_k = z_k + (r_k/u_k) x_next,
// with the couplings e (to the eliminated neighbour) and r (to the other): forward e_k = a_k, r_k = c_k below m and
// c_k, a_k above; adjoint (transposed) e_k = c_{k-1}, r_k = a_{k+1} below and a_{k+1}, c_{k-1} above.
template <typename TS, bool ADJ>
__device__ __forceinline__ void lowk_column_tab(unsigned char* smraw, typename CT<TS>::t* __restrict__ spec,
                                                const Geom& g, const double* __restrict__ ag,
                                                const double* __restrict__ cg, const double* __restrict__ Wg,
                                                double scale, int2 colk, Stats* stats,
                                                const double* __restrict__ target_mean, bool singular00,
                                                double* sq_out, const double* __restrict__ inv_col, double inv_sumw) {
  using CS = typename CT<TS>::t;
  const int nz = g.nz, m = nz / 2, t = threadIdx.x, nt = blockDim.x;
  double* z = reinterpret_cast<double*>(smraw);   // [2][nz]: real parts, imaginary parts
  double* F = z + 2 * nz;                          // elimination factors
  double* w = F + nz;                              // back-substitution factors
  double* scratch = w + nz;                        // [1 per warp]
  const int kx = colk.x, ky = colk.y;
  const bool singular = singular00 && kx == 0 && ky == 0;   // nonsingular with p = 0 on the top face
  CS* colp = spec + (long long)ky * g.P + kx;
  // the column is read at L2 (not through L1), so that a persistent kernel that produced it earlier
  // in the same launch on another SM is seen
  // The mean column is real (it is the horizontal mean of a real field), so only its real part has a mean.  No
  // division here: 1/nz early, 1/sum W from the table.
  const double inv_nz = singular ? 1.0 / (double)nz : 0.0;
  double mean = 0.0;
  for (int k = t; k < nz; k += nt) {
    const CS v = __ldcg(&colp[(long long)k * g.plane]);
    z[k] = (double)v.x;
    z[nz + k] = (double)v.y;
    if (singular) mean += (ADJ ? 1.0 : __ldg(Wg + k)) * (double)v.x;
  }
  if (singular) {   // compatibility: the W-weighted (adjoint: plain) mean of the right-hand side
    mean = lowk_block_sum(mean, scratch) * (ADJ ? inv_nz : inv_sumw);
    // only the first solve records mu_W (a refinement correction solve has a target mean)
    if (!ADJ && t == 0 && stats && !target_mean) stats->mu_w = mean * scale;
  }
  const double ms = -scale;
  for (int k = t; k < nz; k += nt) {   // each thread its own levels: no barrier since they were stored
    const double u = __ldg(inv_col + k), f = k == m ? ms : ms * u;   // b_m is scaled after the meeting
    z[k] = f * (z[k] - mean);
    z[nz + k] *= f;
    const bool up = k > m;
    // at the ends e is 0 (a_0, and the flux coupling above the top, which has no level to couple to)
    const double e = ADJ ? (up ? (k + 1 < nz ? __ldg(ag + k + 1) : 0.0) : (k > 0 ? __ldg(cg + k - 1) : 0.0))
                         : (up ? (k + 1 < nz ? __ldg(cg + k) : 0.0) : __ldg(ag + k));
    const double r = ADJ ? (up ? __ldg(cg + k - 1) : (k + 1 < nz ? __ldg(ag + k + 1) : 0.0))
                         : (up ? __ldg(ag + k) : __ldg(cg + k));
    F[k] = k == m ? e : e * u;    // level m: the couplings themselves (below: F, above: w)
    w[k] = k == m ? (ADJ ? r : (k + 1 < nz ? r : 0.0)) : r * u;
  }
  __syncthreads();
  if (t < 32) {   // lanes 0-3: (part, direction); the others keep the shuffles whole (a block has 16 threads at least)
    const unsigned mask = warp_mask(t, nt);
    const int part = t & 1, up = (t >> 1) & 1, n = t < 4 ? (up ? nz - 1 - m : m) : 0;
    double* zp = z + part * nz;
    const int k0 = up ? nz - 1 : 0, dk = up ? -1 : 1;
    double y = 0.0;
    if (n > 0) {
      double f = F[k0], b = zp[k0];
      for (int i = 0; i < n; ++i) {
        const int k = k0 + i * dk;
        const double fn = F[k + dk], bn = zp[k + dk];   // ahead of this level's store (level m at the end)
        y = fma(f, y, b);
        zp[k] = y;
        f = fn;
        b = bn;
      }
    }
    const double term = (up ? w[m] : F[m]) * y;
    const double both = term + __shfl_xor_sync(mask, term, 2);
    double x = (zp[m] + both) * __ldg(inv_col + m);
    __syncwarp(mask);
    if (t < 2) zp[m] = x;
    if (n > 0) {
      int k = k0 + (n - 1) * dk;
      double f = w[k], b = zp[k];
      for (int i = n - 1; i >= 0; --i) {
        const int kn = i > 0 ? k - dk : k;
        const double fn = w[kn], bn = zp[kn];
        x = fma(f, x, b);
        zp[k] = x;
        k = kn;
        f = fn;
        b = bn;
      }
    }
  }
  __syncthreads();
  double shift = 0.0;   // off the mean column's levels (adjoint: times W_k)
  if (singular) {
    double sx = 0.0;
    for (int k = t; k < nz; k += nt) sx += z[k];
    sx = lowk_block_sum(sx, scratch);
    // adjoint: remove the W direction (the null vector of the transposed column); refinement sweep: the
    // correction also removes the mean of the current iterate
    shift = ADJ ? sx * inv_sumw : sx * inv_nz + (target_mean ? __ldcg(target_mean) : 0.0);
  }
  double sq = 0.0;
  for (int k = t; k < nz; k += nt) {
    double ox = z[k];
    const double oy = z[nz + k];
    if (singular) ox -= ADJ ? __ldg(Wg + k) * shift : shift;
    if (!ADJ && sq_out) sq += ox * ox + oy * oy;
    CS o;
    o.x = (TS)ox;
    o.y = (TS)oy;
    colp[(long long)k * g.plane] = o;
  }
  if (!ADJ && sq_out) {
    sq = lowk_block_sum(sq, scratch);
    if (t == 0) *sq_out = sq;
  }
}

// Listed column `index`, solved by the whole block.  sq_out (nullable): the solution's sum of |x_k|^2 over the levels
// (forward solve), stored by thread 0.  Shared memory: lowk_smem_elems(nz) doubles.
template <typename TS, bool ADJ>
__device__ __forceinline__ void lowk_column(unsigned char* smraw, typename CT<TS>::t* __restrict__ spec,
                                            const Geom& g, const LowkArgs& L, int index, Stats* stats,
                                            double* sq_out = nullptr) {
  lowk_column_tab<TS, ADJ>(smraw, spec, g, L.a_d, L.c_d, L.W_d, L.scale, L.cols[index], stats, L.target_mean,
                           L.singular00 != 0, sq_out, L.inv_tab + (size_t)index * g.nz,
                           __ldg(L.inv_tab + (size_t)L.n * g.nz));
}

// ---------------------------------------------------------------------------
// Twisted FP32 solve of the columns of one staged tile [nz][TC] (two threads per
// column): the lower thread eliminates levels 0..m-1 upward with the pivots
// (g_k, u_k = g_k + c_k), the upper one levels nz-1..m+1 downward with the mirror
// recurrence h_{nz-1} = s + c_{nz-1}, h_k = s + c_k h_{k+1}/v_{k+1}, v_k = h_k + a_k;
// they meet at m = nz/2 and substitute back outward (k_thomas_tw states the
// algebra).  Thread t < 2 TC works on column t % TC (upper half when t >= TC);
// every thread of the block calls this (it holds two block barriers); threads
// with part = false only take part in the barriers.  valid: the column is one
// this solve handles; s its row sum -(lambda_x + lambda_y); out: its level-0
// entry in the spectrum (levels plane entries apart).  wp/colp: the column's
// factor and tile slots.  Shared: ac [nz] (a_k, c_k), meet [TC], xm_s [TC].
// Returns the sum of |x_k|^2 over the levels the thread wrote (0 when it wrote none).
// ADJ: the transposed columns (couplings c_{k-1}, a_{k+1} of the neighbouring rows, the same pivots).
// ---------------------------------------------------------------------------
template <bool ADJ = false>
__device__ __forceinline__ float tw_solve_tile(float2* colp, float* wp, const float2* __restrict__ ac, float4* meet,
                                               float2* xm_s, int TC, int nz, int col_t, int upper, bool part,
                                               bool valid, float s, float ms, float2* out, long long plane) {
  const int m = nz / 2;
  if (part && upper == 0) {
    // levels 0..m-1, upward elimination
    float g_prev = s, inv_prev = 0.f;
    float2 y = make_float2(0.f, 0.f);
    for (int k = 0; k < m; ++k) {
      const float2 akc = ac[k];
      const float2 d = colp[(size_t)k * TC];
      const float f = (k == 0) ? 0.f : akc.x * inv_prev;
      const float gk = (k == 0) ? s : s + f * g_prev;
      const float inv = rcp(gk + akc.y);
      if constexpr (ADJ) {
        const float cm = (k == 0) ? 0.f : ac[k - 1].y;
        y = make_float2(fmaf(ms, d.x, cm * y.x) * inv, fmaf(ms, d.y, cm * y.y) * inv);
        colp[(size_t)k * TC] = y;
        wp[(size_t)k * TC] = ac[k + 1].x * inv;
      } else {
        y = make_float2(fmaf(ms, d.x, f * y.x), fmaf(ms, d.y, f * y.y));
        colp[(size_t)k * TC] = make_float2(y.x * inv, y.y * inv);
        wp[(size_t)k * TC] = akc.y * inv;
      }
      g_prev = gk;
      inv_prev = inv;
    }
    // the level-m terms of the lower part: a_m g_{m-1}/u_{m-1} and a_m z_{m-1}
    const float am = ac[m].x, zm = ADJ ? (m > 0 ? ac[m - 1].y : 0.f) : am;   // adjoint: c_{m-1} z_{m-1}
    const float2 z = (m > 0) ? colp[(size_t)(m - 1) * TC] : make_float2(0.f, 0.f);
    meet[col_t] = (m > 0) ? make_float4(am * g_prev * inv_prev, zm * z.x, zm * z.y, 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
  } else if (part) {
    // levels nz-1..m+1, downward elimination with the mirror recurrence
    float h_prev = s, inv_prev = 0.f;
    float2 y = make_float2(0.f, 0.f);
    for (int k = nz - 1; k > m; --k) {
      const float2 akc = ac[k];
      const float2 d = colp[(size_t)k * TC];
      const float f = (k == nz - 1) ? 0.f : akc.y * inv_prev;   // c_k / v_{k+1}
      const float hk = (k == nz - 1) ? s + akc.y : s + f * h_prev;
      const float inv = rcp(hk + akc.x);
      if constexpr (ADJ) {
        const float am = (k == nz - 1) ? 0.f : ac[k + 1].x;
        y = make_float2(fmaf(ms, d.x, am * y.x) * inv, fmaf(ms, d.y, am * y.y) * inv);
        colp[(size_t)k * TC] = y;
        wp[(size_t)k * TC] = ac[k - 1].y * inv;
      } else {
        y = make_float2(fmaf(ms, d.x, f * y.x), fmaf(ms, d.y, f * y.y));
        colp[(size_t)k * TC] = make_float2(y.x * inv, y.y * inv);
        wp[(size_t)k * TC] = akc.x * inv;
      }
      h_prev = hk;
      inv_prev = inv;
    }
    xm_s[col_t] = make_float2((m + 1 < nz) ? h_prev * inv_prev : 1.f, 0.f);   // h_{m+1}/v_{m+1}
  }
  __syncthreads();
  if (part && upper == 0) {
    const float2 akc = ac[m];
    const float cm = akc.y;
    const float hterm = cm * xm_s[col_t].x;
    const float2 zt = (m + 1 < nz) ? colp[(size_t)(m + 1) * TC] : make_float2(0.f, 0.f);
    const float4 lo = meet[col_t];
    const float2 dm = colp[(size_t)m * TC];
    const float den = s + lo.x + hterm;
    const float zu = ADJ ? (m + 1 < nz ? ac[m + 1].x : 0.f) : cm;   // adjoint: a_{m+1} z_{m+1}
    const float2 num = make_float2(fmaf(ms, dm.x, lo.y + zu * zt.x), fmaf(ms, dm.y, lo.z + zu * zt.y));
    const float2 xm = make_float2(__fdiv_rn(num.x, den), __fdiv_rn(num.y, den));
    xm_s[col_t] = xm;   // this thread has read the h-term; no other thread touches the slot before the barrier
  }
  __syncthreads();
  float sq = 0.f;   // sum of |x_k|^2 over the levels this thread writes (x_m by the lower thread)
  if (!part || !valid) return sq;
  const float2 xm = xm_s[col_t];
  if (upper == 0) {
    out[(long long)m * plane] = xm;
    sq = xm.x * xm.x + xm.y * xm.y;
    float2 x = xm;
    for (int k = m - 1; k >= 0; --k) {
      const float2 z = colp[(size_t)k * TC];
      const float w = wp[(size_t)k * TC];
      x = make_float2(z.x + w * x.x, z.y + w * x.y);
      out[(long long)k * plane] = x;
      sq = fmaf(x.x, x.x, fmaf(x.y, x.y, sq));
    }
  } else {
    float2 x = xm;
    for (int k = m + 1; k < nz; ++k) {
      const float2 z = colp[(size_t)k * TC];
      const float w = wp[(size_t)k * TC];
      x = make_float2(z.x + w * x.x, z.y + w * x.y);
      out[(long long)k * plane] = x;
      sq = fmaf(x.x, x.x, fmaf(x.y, x.y, sq));
    }
  }
  return sq;
}

}  // namespace pgb

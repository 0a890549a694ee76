// Forward x-pass of a refinement sweep with all of the stencil's rows staged in shared memory: sweep 1's residual
// r0 = S - mu_W - L p0, and the verification's first try r0 - L q (the same values, in the same arithmetic, as the
// kernels of xpass_res.cu, which keep the residual with q and the lines too long for two rows a CTA).
//
// Bound by instruction issue (3.3 and 3.7 warp instructions a point for the two: the double-float stencil in packed
// pairs, and the transform) once the operands are at hand.  Read row by row through L2, the y and z neighbours kept 24 warps an SM
// waiting instead (long-scoreboard stalls 4 to 6 per instruction, issue slots 50-55% used; bringing the
// upper rows into L2 ahead of time changed nothing).  Here a CTA of about 128 threads takes RB rows of one level
// and stages, by bulk copies on two mbarriers, their operand rows (S, or r0 and p0) and the field's rows: the RB
// with one halo row on each side, the RB above and the RB below.  The stencil then reads shared memory
// only.  The field's rows are refilled for the next group while this one is transformed (in the place of its
// operand rows); four CTAs an SM cover each other's loads.
// 1024 x 1024 x 128: sweep 1's pass 830 -> 630 us, the first try's 996 -> 672 (their DRAM traffic alone: 400).
//
// Compiled twice, for dx == dy (PGB_XRT_ISO 1, from xpass_res_tile_iso.cu) and for the general form.
#include "xpass_common.cuh"

#ifndef PGB_XRT_ISO
#define PGB_XRT_ISO 0
#endif

namespace pgb {
namespace {

constexpr int xrt_blocks(int n) { return n % 3 == 0 ? 3 : 4; }

// twiddles (N), unpack twiddles (N/2 + 2), operand rows [RB][NX] doubles, field rows [RB + 2][NX],
// [RB][NX] above, [RB][NX] below, two mbarriers
template <int N> struct XrtLayout {
  static constexpr int RB = xrt_rows(N), NX = 2 * N;
  static constexpr size_t off_op = xs_align((size_t)(N + N / 2 + 2) * 8, 128);
  static constexpr size_t off_f = off_op + (size_t)RB * NX * 8;
  static constexpr size_t off_up = off_f + (size_t)(RB + 2) * NX * 4;
  static constexpr size_t off_dn = off_up + (size_t)RB * NX * 4;
  static constexpr size_t off_bar = off_dn + (size_t)RB * NX * 4;
  static constexpr size_t total = off_bar + 16;
};

template <int N, int E, bool ISO, bool FROM_R0>
__global__ void __launch_bounds__(xrt_rows(N) * (N / E), xrt_blocks(N))
    k_xrt(ResidualArgs R, float2* __restrict__ spec, Geom g, const float2* __restrict__ twx,
          const float2* __restrict__ twr, const int* __restrict__ done, unsigned* __restrict__ err) {
  using C = float2;
  using L = XrtLayout<N>;
  constexpr int nl = N / E, RB = L::RB, TH = RB * nl, NX = L::NX;
  pdl_trigger();
  extern __shared__ __align__(128) unsigned char smraw[];
  C* tw_s = reinterpret_cast<C*>(smraw);
  C* twr_s = tw_s + N;
  unsigned char* op = smraw + L::off_op;
  float* fld = reinterpret_cast<float*>(smraw + L::off_f);    // row 0: south halo, 1..: the group, then north halo
  float* fup = reinterpret_cast<float*>(smraw + L::off_up);
  float* fdn = reinterpret_cast<float*>(smraw + L::off_dn);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smraw + L::off_bar);   // [0] operand rows, [1] field rows
  const int lane = threadIdx.x, ty = threadIdx.y, tid = ty * nl + lane;
  const int gpl = (g.ny + RB - 1) / RB;   // groups per level
  const int ngroups = gpl * (g.lev1 - g.lev0);
  st_build_twiddles<N, E>(tw_s, twx, tid, TH);
  for (int t = tid; t <= N / 2; t += TH) twr_s[t] = twr[t];
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  __syncthreads();
  pdl_wait();   // the previous kernels of the stream are complete
  if (done && *done) return;
  const float* field = FROM_R0 ? R.q : R.p0;
  auto issue_op = [&](int grp) {
    const int k = g.lev0 + grp / gpl, j0 = grp % gpl * RB;
    const unsigned nv = (unsigned)(g.ny - j0 < RB ? g.ny - j0 : RB);
    const long long r0 = (long long)k * g.ny + j0;
    mbar_arrive_expect_tx(&bar[0], nv * NX * (FROM_R0 && !R.p_out ? 4u : 8u));
    if constexpr (FROM_R0) {
      for (unsigned j = 0; j < nv; ++j)
        bulk_g2s(op + (size_t)j * NX * 4, R.r0 + (r0 + j) * R.r_ld, NX * 4u, &bar[0]);
      if (R.p_out) bulk_g2s(op + (size_t)RB * NX * 4, R.p0 + r0 * NX, nv * NX * 4u, &bar[0]);
    } else {
      bulk_g2s(op, R.S + r0 * NX, nv * NX * 8u, &bar[0]);
    }
  };
  auto issue_field = [&](int grp) {
    const int k = g.lev0 + grp / gpl, j0 = grp % gpl * RB;
    const int nv = g.ny - j0 < RB ? g.ny - j0 : RB;
    const long long lev = (long long)k * g.ny, r0 = lev + j0;
    const bool up = k + 1 < g.nz, dn = k > 0;
    mbar_arrive_expect_tx(&bar[1], (unsigned)(nv * (1 + (up ? 1 : 0) + (dn ? 1 : 0)) + 2) * NX * 4u);
    bulk_g2s(fld, field + (lev + (j0 == 0 ? g.ny - 1 : j0 - 1)) * NX, NX * 4u, &bar[1]);
    bulk_g2s(fld + NX, field + r0 * NX, (unsigned)nv * NX * 4u, &bar[1]);
    bulk_g2s(fld + (size_t)(nv + 1) * NX, field + (lev + (j0 + nv == g.ny ? 0 : j0 + nv)) * NX, NX * 4u, &bar[1]);
    if (up) bulk_g2s(fup, field + (r0 + g.ny) * NX, (unsigned)nv * NX * 4u, &bar[1]);
    if (dn) bulk_g2s(fdn, field + (r0 - g.ny) * NX, (unsigned)nv * NX * 4u, &bar[1]);
  };
  bool wait_op = false, wait_field = false;   // copies in flight (the issuing thread's)
  if (tid == 0 && (int)blockIdx.x < ngroups) {
    issue_field(blockIdx.x);
    issue_op(blockIdx.x);
    wait_op = wait_field = true;
  }
  const LineSyncT<nl> sync{1 + ty};
  const LineAddr<N> sw{};
  C* la = reinterpret_cast<C*>(op + (size_t)ty * NX * 8);   // the line buffers: the place of the operand rows
  C* lb = la + N;
  const float* rowc = fld + (size_t)(ty + 1) * NX;
  const float2* cc = reinterpret_cast<const float2*>(rowc);
  const float2* cs = reinterpret_cast<const float2*>(rowc - NX);
  const float2* cn = reinterpret_cast<const float2*>(rowc + NX);
  const float2* cu = reinterpret_cast<const float2*>(fup + (size_t)ty * NX);
  const float2* cd = reinterpret_cast<const float2*>(fdn + (size_t)ty * NX);
  float2 racc = make_float2(0.f, 0.f), sacc = racc;   // per-lane sums of r^2 and S^2 (even / odd points)
  bool ok = true;
  unsigned phase = 0;
  for (int grp = blockIdx.x; grp < ngroups; grp += gridDim.x, phase ^= 1) {
    const int k = g.lev0 + grp / gpl, j = grp % gpl * RB + ty;
    const bool valid = j < g.ny;
    const long long row = (long long)k * g.ny + (valid ? j : 0);
    const bool has_dn = k > 0, has_up = k + 1 < g.nz;
    const ResCoef K = res_coef(R.cx, R.cy, R.a_ff[k], R.c_ff[k], *R.mu_ff);
    const bool got = mbar_wait_bounded(&bar[1], phase, kWaitPolls) && mbar_wait_bounded(&bar[0], phase, kWaitPolls);
    if (!__syncthreads_and(got)) {
      ok = false;
      break;
    }
    wait_op = wait_field = false;
    C v[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int e = st_in_index<N, E, 0>(lane, i);
      const float2 pc = cc[e];
      const float pw = rowc[e == 0 ? NX - 1 : 2 * e - 1], pe = rowc[e == N - 1 ? 0 : 2 * e + 2];
      const float2 pd = has_dn ? cd[e] : pc, pu = has_up ? cu[e] : make_float2(0.f, 0.f);
      // the pair's east neighbours are (pc.y, pe), its west neighbours (pw, pc.x)
      if constexpr (FROM_R0) {
        v[i] = residual_from_r0<ISO>(reinterpret_cast<const float2*>(op + (size_t)ty * NX * 4)[e], pc,
                                     make_float2(pc.y, pe), make_float2(pw, pc.x), cn[e], cs[e], pd, pu, K);
        if (valid) {
          racc = fma2(v[i], v[i], racc);
          if (R.p_out) {   // the iterate p0 + q as the double the inverse x-pass would store
            float2 sp, tp;
            two_sum2(reinterpret_cast<const float2*>(op + (size_t)(RB + ty) * NX * 4)[e], pc, sp, tp);
            __stcs(reinterpret_cast<double2*>(R.p_out + row * NX) + e,
                   make_double2(ff2d_fast(sp.x, tp.x), ff2d_fast(sp.y, tp.y)));
          }
        }
      } else {
        const double2 S = reinterpret_cast<const double2*>(op + (size_t)ty * NX * 8)[e];
        float2 Sh, Sl;
        d2ff_trunc(S.x, Sh.x, Sl.x);
        d2ff_trunc(S.y, Sh.y, Sl.y);
        const float2 z = make_float2(0.f, 0.f);
        v[i] = residual_value2<false, ISO>(pc, make_float2(pc.y, pe), make_float2(pw, pc.x), cn[e], cs[e], pd, pu, z, z,
                                           z, z, z, z, z, Sh, Sl, K);
        if (valid) {
          racc = fma2(v[i], v[i], racc);
          sacc = fma2(Sh, Sh, sacc);
          // sweep 1's residual, kept for the verification's first try
          if (R.r_out) __stcs(reinterpret_cast<float2*>(R.r_out + row * R.r_ld) + e, v[i]);
        }
      }
    }
    fence_proxy_async_smem();
    __syncthreads();   // every row has read its operands: the field's rows may be refilled, the operand rows reused
    const int next = grp + gridDim.x;
    if (tid == 0 && next < ngroups) {
      issue_field(next);
      wait_field = true;
    }
    const C* fin = st_fft<N, E, -1, false, float>(v, la, lb, sw, lane, tw_s, sync);
    r2c_unpack_store<N, E>(fin, twr_s, spec + row * g.P, lane, valid, R.kmax > 0 ? R.kmax : N);
    fence_proxy_async_smem();   // generic writes to the operand rows come before their refill by bulk copies
    __syncthreads();
    if (tid == 0 && next < ngroups) {
      issue_op(next);
      wait_op = true;
    }
  }
  if (tid == 0 && !ok) {   // report, and let copies in flight land before the shared memory is released
    atomicOr(err, (unsigned)ERR_WAIT_TIMEOUT);
    if (wait_field) mbar_wait_bounded(&bar[1], phase, kWaitPolls);
    if (wait_op) mbar_wait_bounded(&bar[0], phase, kWaitPolls);
  }
  // per-CTA sums of r^2 and S^2 (fixed-order tree) in the drained operand rows
  static_assert((size_t)TH * 8 <= (size_t)RB * NX * 8 && TH <= 128, "reduction does not fit the operand rows");
  __syncthreads();
  float (*red)[TH] = reinterpret_cast<float (*)[TH]>(op);
  red[0][tid] = racc.x + racc.y;
  red[1][tid] = sacc.x + sacc.y;
  __syncthreads();
  for (int h = 64; h > 0; h >>= 1) {
    if (tid < h && tid + h < TH) {
      red[0][tid] += red[0][tid + h];
      red[1][tid] += red[1][tid + h];
    }
    __syncthreads();
  }
  if (tid == 0 && R.partials) {
    double* out = R.partials + 2 * (R.part0 + (long long)blockIdx.x);
    // at L2: blocks of the chunk before, on other SMs, wrote these lines
    out[0] = (double)red[0][0] + (R.part_add ? __ldcg(out) : 0.0);
    out[1] = (double)red[1][0] + (R.part_add ? __ldcg(out + 1) : 0.0);
  }
}

template <bool ISO, bool FROM_R0>
cudaError_t xrt_launch(const ResidualArgs& R, float2* spec, const Geom& g, int n, const Tables& tb, const int* done,
                       unsigned* err, int* nblocks_out, cudaStream_t st, bool* used) {
#define PGB_XRT_CASE(V)                                                                                              \
  case V: {                                                                                                          \
    constexpr int EE = st_elems(V), RB = xrt_rows(V);                                                                \
    static_assert(xrt_length(V), "two rows a CTA at least");                                                        \
    auto kern = k_xrt<V, EE, ISO, FROM_R0>;                                                                          \
    int cap = 0;                                                                                                     \
    const cudaError_t e = prepare(kern, RB * (V / EE), XrtLayout<V>::total, cap);                                    \
    if (e != cudaSuccess || cap <= 0) return e;                                                                      \
    const long long groups = (long long)((g.ny + RB - 1) / RB) * (g.lev1 - g.lev0);                                  \
    const int grid = tile_pass_blocks(groups, cap, R.slots);                                                         \
    if (nblocks_out) *nblocks_out = grid;                                                                            \
    *used = true;                                                                                                    \
    return pdl_launch(kern, dim3(grid), dim3(V / EE, RB), XrtLayout<V>::total, st, R, spec, g, tb.twx_f, tb.twr_f,   \
                      done, err);                                                                                    \
  }
  switch (n) {
    PGB_XRT_CASE(16) PGB_XRT_CASE(18) PGB_XRT_CASE(24) PGB_XRT_CASE(48) PGB_XRT_CASE(54)
    PGB_XRT_CASE(32) PGB_XRT_CASE(36) PGB_XRT_CASE(64) PGB_XRT_CASE(72) PGB_XRT_CASE(96) PGB_XRT_CASE(108)
    PGB_XRT_CASE(128) PGB_XRT_CASE(144) PGB_XRT_CASE(192) PGB_XRT_CASE(216) PGB_XRT_CASE(256) PGB_XRT_CASE(288)
    PGB_XRT_CASE(324) PGB_XRT_CASE(384) PGB_XRT_CASE(432) PGB_XRT_CASE(512) PGB_XRT_CASE(768)
    default: return cudaSuccess;
  }
#undef PGB_XRT_CASE
}

template <bool ISO>
cudaError_t xrt(const ResidualArgs& R, float2* spec, const Geom& g, int n, const Tables& tb, const int* done,
                unsigned* err, int* nblocks_out, cudaStream_t st, bool* used) {
  if (!aligned16(R.p0) || (g.nx * 4) % 16) return cudaSuccess;
  if (R.r0) {
    if (!R.q || !aligned16(R.q) || !aligned16(R.r0) || (R.r_ld * 4) % 16) return cudaSuccess;
    return xrt_launch<ISO, true>(R, spec, g, n, tb, done, err, nblocks_out, st, used);
  }
  if (R.q || !aligned16(R.S)) return cudaSuccess;   // the full residual with q: xpass_res.cu
  return xrt_launch<ISO, false>(R, spec, g, n, tb, done, err, nblocks_out, st, used);
}

}  // namespace

#if PGB_XRT_ISO
cudaError_t launch_xrt_iso(const ResidualArgs& R, float2* spec, const Geom& g, int n, const Tables& tb, const int* done,
                           unsigned* err, int* nblocks_out, cudaStream_t st, bool* used) {
  return xrt<true>(R, spec, g, n, tb, done, err, nblocks_out, st, used);
}
#else
cudaError_t launch_xrt_iso(const ResidualArgs& R, float2* spec, const Geom& g, int n, const Tables& tb, const int* done,
                           unsigned* err, int* nblocks_out, cudaStream_t st, bool* used);

int xres_tile_blocks(int ny, int nz, int n) {
  if (!xpass_static_supported(n) || !xrt_length(n)) return 0;
  const int groups = (ny + xrt_rows(n) - 1) / xrt_rows(n) * nz;
  const int resident = (st_elems(n) == kE3 ? 3 : 4) * sm_count();   // by its registers (160-168, 112-128)
  return groups < resident ? groups : resident;
}

cudaError_t launch_xres_tile(const ResidualArgs& R, void* spec, const Geom& g, const FftPlan& fx, const Tables& tb,
                             const int* done, unsigned* err, int* nblocks_out, cudaStream_t st, bool* used) {
  *used = false;
  if (!xpass_static_supported(fx.n) || !xrt_length(fx.n)) return cudaSuccess;
  // dx == dy: the kernels with the merged horizontal term
  if (R.cx.x == R.cy.x && R.cx.y == R.cy.y)
    return launch_xrt_iso(R, (float2*)spec, g, fx.n, tb, done, err, nblocks_out, st, used);
  return xrt<false>(R, (float2*)spec, g, fx.n, tb, done, err, nblocks_out, st, used);
}
#endif

}  // namespace pgb

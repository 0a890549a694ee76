// Preconditioned conjugate gradients for a density that varies in x, y and z,
// with the direct FFT solve as the preconditioner.  This is the iterative
// alternative of Section 2.2 (a matrix-free CG whose cost per iteration is a
// stencil application and a few vector updates, preconditioned by a cheap
// approximate inverse), for the case the direct method alone cannot handle: a
// horizontally varying density does not separate under the Fourier transform.
//
// Operator (flux form, cell weights W_ijk = rho_ijk dz_k):
//   (W A d)_ijk = dz_k [ (F^x_{i+1/2} - F^x_{i-1/2})/dx + (F^y_{j+1/2} - F^y_{j-1/2})/dy ]
//               + F^z_{k+1/2} - F^z_{k-1/2},
//   F^x_{i+1/2} = rho_{i+1/2} (d_{i+1} - d_i)/dx, rho_{i+1/2} = (rho_i + rho_{i+1})/2 (periodic);
//   F^y likewise; F^z_{k+1/2} = rho_{k+1/2} (d_{k+1} - d_k)/h_{k+1/2}, zero at the bottom face and
//   at the top face, or rho_{nz-1} (0 - d_{nz-1})/(dz_{nz-1}/2) with p = 0 on the top face.
// CG runs on K = -W A (symmetric, positive semidefinite) with b = -W (S - mu_W); the
// preconditioner is z = -G(r / Wbar): G is the plan's solve for the level density
// rho0 (weights Wbar_k = rho0_k dz_k).  Polak-Ribiere beta = -alpha (q . z_new)/(r . z)
// keeps the iteration robust to a preconditioner that is applied in reduced precision.
// All vectors and reductions are FP64, the partial sums added in block order by each launch's last block, which also
// forms the step lengths on the device: the host waits once per iteration, for the stopping test.
//
// What bounds the kernels (GB300, 512 x 512 x 64, 16.8 M points): the FP64 unit does 1.7 operations a clock and SM, so
// one FP64 operation per point costs as much as 11 bytes of HBM traffic, and each kernel keeps to two or so:
//   k_cg_apply   instruction issue (the operator in double-float arithmetic, see below): 285 -> 185 us
//   k_cg_update  r -= alpha q, t = -r/Wbar (float where the preconditioner transforms floats), the residual norm in
//                the FP32 pipe; 32 bytes a point (64 with the step of p): 161 -> 103 us
//   k_cg_dots    z.r and z.q; 20 bytes a point, bound by the FP64 unit: 73 us
//   k_cg_dir     p += alpha d (of the step before, as d is read anyway) and d = z + beta d; 36 bytes a point: 93 us
//                (57 without the step of p)
// With the mixed plan's float preconditioner z stays the float field the inverse transform writes.
// No FP64 division runs per point: the level reciprocals come from a small table, and the residual's weight
// 1/rho (needed only for the stopping test) is a float reciprocal.
//
// The operator: q = -sum_f c_f (d_f - d_c) with c_f = const_k (rho_f + rho_c).  rho is split into float pairs once
// per solve, d as it is read (integer operations); differences and sums are formed first and exactly
// (two-sums), products by FMA-based two-products, on the two points of a pair at once (packed FP32).  The face
// densities' sums are thus double-float ones, where FP64 formed them before the coefficients were split; the splits
// keep the whole remainder in return (split_whole), and q's rms error against 80-bit arithmetic is 0.54 to 0.72 of that
// form's over 54 fields (noise 7.5e-15 of |q| against 1.34e-14; with splits cut at 2^-46 it was 1.06 to 1.18 of it), at
// the same time per iteration.  A block
// takes a tile of 64 x 8 points and marches up the levels: every value is read from memory once (24 bytes a
// point with q, where three stored face coefficients made it 40), the x neighbours come by shuffles, the y
// neighbours through shared memory, and the flux through the upper face is kept as the next level's lower one.
#include "kernels.cuh"
#include "residual2.cuh"

namespace pgb {
namespace {

// The step lengths and sums of a solve, on the device.
struct CgState {
  double mu, ss, inv_snorm, rz, dq, alpha, beta, rel2, shift;
  unsigned ticket;
};

struct CgDims {
  int nx, ny, nz;
  long long plane, n;
  int top_dirichlet;
};

// What a launch's sums (s0, s1) mean; run by one thread once every block's partials are added up.
__device__ __forceinline__ void cg_finish(int op, CgState* c, double s0, double s1, const CgDims& D) {
  switch (op) {
    case CG_PREP: c->mu = (!D.top_dirichlet && s1 > 0) ? s0 / s1 : 0.0; break;
    case CG_START:
      c->ss = s0;
      c->inv_snorm = s0 > 0 ? 1.0 / sqrt(s0) : 0.0;
      break;
    case CG_DOTS0: c->rz = s0; break;
    case CG_APPLY:
      c->dq = s0;
      c->alpha = s0 > 0 ? c->rz / s0 : 0.0;   // otherwise d is in the null space (or a breakdown): no step
      break;
    case CG_UPDATE: c->rel2 = s0; break;
    case CG_DOTS:
      c->beta = -c->alpha * s1 / c->rz;       // Polak-Ribiere: z_new . (r_new - r_old) / (r_old . z_old)
      c->rz = s0;
      break;
    case CG_LAST: c->shift = s0 / (double)D.n; break;
    default: break;
  }
}

// Sums a and b over the launch's blocks (256 threads each): per block a shuffle tree and the warps in order, over the
// blocks by the last one to finish, in block order per thread and then a fixed tree.
__device__ __forceinline__ void cg_reduce(int op, CgState* c, double a, double b, double* partials, const CgDims& D) {
  __shared__ double s0[256], s1[256];
  __shared__ bool last;
  const int t = threadIdx.x;
  const unsigned nb = gridDim.x * gridDim.y, blk = blockIdx.y * gridDim.x + blockIdx.x;
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  if ((t & 31) == 0) {
    s0[t >> 5] = a;
    s1[t >> 5] = b;
  }
  __syncthreads();
  if (t == 0) {
    double x = 0, y = 0;
    for (int w = 0; w < 8; ++w) {
      x += s0[w];
      y += s1[w];
    }
    partials[2 * blk] = x;
    partials[2 * blk + 1] = y;
    __threadfence();
    last = atomicAdd(&c->ticket, 1u) == nb - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double x = 0, y = 0;
  for (unsigned i = t; i < nb; i += 256) {
    x += __ldcg(&partials[2 * i]);
    y += __ldcg(&partials[2 * i + 1]);
  }
  s0[t] = x;
  s1[t] = y;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (t < h) {
      s0[t] += s0[t + h];
      s1[t] += s1[t + h];
    }
    __syncthreads();
  }
  if (t == 0) {
    c->ticket = 0u;   // ready for the next launch
    cg_finish(op, c, s0[0], s1[0], D);
  }
}

// x as a float pair: h truncated, l the whole remainder of 29 bits rounded to float, |h + l - x| <= 2^-48 |x|.
// d2ff_trunc, which cuts the remainder at 23 bits, leaves up to 2^-46; the ranges are the same.
__device__ __forceinline__ void split_whole(double x, float& h, float& l) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  float cut;
  d2ff_trunc(x, h, cut);
  const int se = (int)((b >> 52) & 0x7ffu) - 942;
  const float sc = __uint_as_float((uint32_t)(se > 0 ? se : 0) << 23);
  l = copysignf(((float)(int)((uint32_t)b & 0x1fffffffu) * 0.015625f) * sc, h);
}

// Flat kernels: grid (blocks per level, nz), pairs of points; pairs of block x of a level.
#define CG_PAIRS(i, D)                                                                                      \
  for (long long half = (D).plane / 2, off = (long long)blockIdx.y * half, i_ = blockIdx.x * 256ll + threadIdx.x, \
                 i = off + i_;                                                                              \
       i_ < half; i_ += gridDim.x * 256ll, i = off + i_)

// rho as float pairs, and sum W S, sum W for mu_W = sum W S / sum W
__global__ void __launch_bounds__(256) k_cg_prep(const double2* __restrict__ rho, const double2* __restrict__ S,
                                                 float2* __restrict__ rh, float2* __restrict__ rl,
                                                 const CgLevel* __restrict__ lv, CgDims D, CgState* c,
                                                 double* __restrict__ partials) {
  double ws = 0, w = 0;
#pragma unroll 2
  CG_PAIRS(i, D) {
    const double2 r = rho[i], s = S[i];
    float2 h, l;
    split_whole(r.x, h.x, l.x);
    split_whole(r.y, h.y, l.y);
    rh[i] = h;
    rl[i] = l;
    ws = fma(r.x, s.x, ws);
    ws = fma(r.y, s.y, ws);
    w += r.x + r.y;
  }
  const double dz = lv[blockIdx.y].dz;
  cg_reduce(CG_PREP, c, ws * dz, w * dz, partials, D);
}

template <typename T> struct CgVec;
template <> struct CgVec<double> {
  using t = double2;
  static __device__ __forceinline__ double2 in(double2 x) { return x; }
  static __device__ __forceinline__ double2 out(double2 x) { return x; }
};
template <> struct CgVec<float> {
  using t = float2;
  static __device__ __forceinline__ double2 in(float2 x) { return make_double2(f2d_int(x.x), f2d_int(x.y)); }
  static __device__ __forceinline__ float2 out(double2 x) { return make_float2(d2f_int(x.x), d2f_int(x.y)); }
};

// r = b = -W (S - mu), t = -r/Wbar (the preconditioner's source); sum S . S
template <typename TT>
__global__ void __launch_bounds__(256) k_cg_start(const double2* __restrict__ rho, const double2* __restrict__ S,
                                                  double2* __restrict__ r, typename CgVec<TT>::t* __restrict__ t,
                                                  const CgLevel* __restrict__ lv, CgDims D, CgState* c,
                                                  double* __restrict__ partials) {
  double ss = 0;
  const CgLevel L = lv[blockIdx.y];
  const double mu = c->mu, iw = -L.iwbar;
#pragma unroll 2
  CG_PAIRS(i, D) {
    const double2 s = S[i], q = rho[i];
    const double2 b = make_double2(-(q.x * L.dz) * (s.x - mu), -(q.y * L.dz) * (s.y - mu));
    r[i] = b;
    t[i] = CgVec<TT>::out(make_double2(b.x * iw, b.y * iw));
    ss = fma(s.x, s.x, ss);
    ss = fma(s.y, s.y, ss);
  }
  cg_reduce(CG_START, c, ss, 0.0, partials, D);
}

// Two points' d and rho as float pairs.
struct CgPt {
  float2 dh, dl, rh, rl;
};
// (rho_f + rho_c) (d_f - d_c) = ph - npl, an unnormalised float pair: sum and difference exact in their high parts,
// the product of the high parts exact.  The low part comes negated, which saves the packed negations.
__device__ __forceinline__ void cg_flux(const CgPt& f, const CgPt& c, float2& ph, float2& npl) {
  float2 s, e, t, u;
  two_diff2(f.dh, c.dh, s, e);
  const float2 lo = add2(e, sub2(f.dl, c.dl));
  two_sum2(f.rh, c.rh, t, u);
  const float2 m1 = make_float2(-1.f, -1.f), nt = mul2(t, m1);
  const float2 ntl = fma2(u, m1, mul2(add2(f.rl, c.rl), m1));
  ph = mul2(t, s);
  npl = fma2(nt, lo, fma2(ntl, s, fma2(nt, s, ph)));
}
// times a constant k = (h, l)
__device__ __forceinline__ void cg_scale(float2& ph, float2& npl, float2 k) {
  const float2 h = f2bc(k.x), nh = f2bc(-k.x), nl = f2bc(-k.y), p = mul2(h, ph);
  npl = fma2(h, npl, fma2(nl, ph, fma2(nh, ph, p)));
  ph = p;
}
// (H - L) += (ph - npl)
__device__ __forceinline__ void cg_acc(float2& H, float2& L, float2 ph, float2 npl) {
  float2 s, e;
  two_sum2(H, ph, s, e);
  H = s;
  L = add2(L, sub2(npl, e));
}
__device__ __forceinline__ float2 cg_split(double x) {
  float h, l;
  split_whole(x, h, l);
  return make_float2(h, l);
}
__device__ __forceinline__ CgPt cg_point2(double2 d, float2 rh, float2 rl) {
  const float2 a = cg_split(d.x), b = cg_split(d.y);
  return {make_float2(a.x, b.x), make_float2(a.y, b.y), rh, rl};
}

constexpr int kCgTY = 8;    // rows of a tile (a warp each), 32 pairs of points wide
constexpr int kCgZC = 16;   // levels a tile marches up

// q = K d = -(W A d); sum d . q.  Tiles (x, y, level chunk) in grid-stride order.
__global__ void __launch_bounds__(256) k_cg_apply(const double2* __restrict__ d, const float2* __restrict__ rh,
                                                  const float2* __restrict__ rl, double2* __restrict__ q,
                                                  const CgLevel* __restrict__ lv, CgDims D, CgState* c,
                                                  double* __restrict__ partials) {
  __shared__ float4 sd[2][kCgTY + 2][32], sr[2][kCgTY + 2][32];   // rows j0 - 1 .. j0 + 8 of a level
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nx2 = D.nx / 2, tx = (nx2 + 31) / 32, ty = (D.ny + kCgTY - 1) / kCgTY, tz = (D.nz + kCgZC - 1) / kCgZC;
  double acc = 0;
  for (long long tile = blockIdx.x; tile < (long long)tx * ty * tz; tile += gridDim.x) {
    const int x0 = (int)(tile % tx) * 32, j0 = (int)(tile / tx % ty) * kCgTY, k0 = (int)(tile / tx / ty) * kCgZC;
    const int k1 = min(D.nz, k0 + kCgZC), np = min(32, nx2 - x0), nr = min(kCgTY, D.ny - j0);
    const bool act = lane < np && w < nr;
    const int j = j0 + min(w, nr - 1), i = x0 + min(lane, np - 1);
    // the row south (warp 0) or north (warp nr - 1) of the tile and the point west (lane 0) or east (lane np - 1; a
    // tile is at least two pairs wide) of it, as element offsets within a level
    const bool hs = w == 0, halo = hs || w == nr - 1, ew = lane == 0, edge = ew || lane == np - 1;
    const unsigned half = (unsigned)(D.plane / 2);   // pairs of a level: at most 4096 x 4096 / 2
    const unsigned own = (unsigned)(j * nx2 + i);
    const unsigned js = (unsigned)((j0 == 0 ? D.ny - 1 : j0 - 1) * nx2 + i);
    const unsigned jn = (unsigned)((j0 + nr == D.ny ? 0 : j0 + nr) * nx2 + i), jh = hs ? js : jn;
    const unsigned ie = 2u * (unsigned)(j * nx2) +
                        (unsigned)(ew ? (x0 == 0 ? D.nx - 1 : 2 * x0 - 1) : (x0 + np == nx2 ? 0 : 2 * (x0 + np)));
    const double2* dk = d + (long long)k0 * half;
    const float2 *hk = rh + (long long)k0 * half, *lk = rl + (long long)k0 * half;
    const float2 z2 = make_float2(0.f, 0.f);
    struct Raw {
      double2 d;
      float2 h, l;
    };
    auto load = [&](const double2* dp, const float2* hp, const float2* lp, unsigned at) {
      return Raw{dp[at], hp[at], lp[at]};
    };
    auto split = [&](const Raw& v) { return cg_point2(v.d, v.h, v.l); };
    double e_d = 0.0;   // the edge point
    float e_h = 0.f, e_l = 0.f;
    auto load_edge = [&](const double2* dp, const float2* hp, const float2* lp) {
      e_d = reinterpret_cast<const double*>(dp)[ie];
      e_h = reinterpret_cast<const float*>(hp)[ie];
      e_l = reinterpret_cast<const float*>(lp)[ie];
    };
    // loaded ahead: this level's halo row and edge point, the next level's own pair
    CgPt cur = split(load(dk, hk, lk, own));
    Raw r_up{}, r_halo{};
    if (k0 + 1 < D.nz) r_up = load(dk + half, hk + half, lk + half, own);
    if (halo) r_halo = load(dk, hk, lk, jh);
    if (edge) load_edge(dk, hk, lk);
    float2 dnh = z2, dnl = z2;   // flux through the lower face, from the level below
    if (k0 > 0) {
      cg_flux(cur, split(load(dk - half, hk - half, lk - half, own)), dnh, dnl);
      cg_scale(dnh, dnl, lv[k0 - 1].ku);
    }
    for (int k = k0, b = 0; k < k1; ++k, b ^= 1) {
      // above the top: the face value 0 with the coefficient rho_k ku (ku = 0 with zero flux)
      const CgPt up = k + 1 < D.nz ? split(r_up) : CgPt{z2, z2, z2, z2};
      const CgPt hal = split(r_halo);
      const float2 e_s = cg_split(e_d);
      const float4 ev = make_float4(e_s.x, e_s.y, e_h, e_l);
      auto publish = [&](int r, const CgPt& v) {
        sd[b][r][lane] = make_float4(v.dh.x, v.dh.y, v.dl.x, v.dl.y);
        sr[b][r][lane] = make_float4(v.rh.x, v.rh.y, v.rl.x, v.rl.y);
      };
      if (w < nr) publish(w + 1, cur);
      if (halo) publish(hs ? 0 : nr + 1, hal);
      if (hs && nr == 1) publish(2, split(load(dk, hk, lk, jn)));   // a tile of one row has both next to it
      const double2* dn_ = dk + half;
      const float2 *hn_ = hk + half, *ln_ = lk + half;
      if (k + 1 < k1) {   // ahead of this level's arithmetic
        if (halo) r_halo = load(dn_, hn_, ln_, jh);
        if (edge) load_edge(dn_, hn_, ln_);
        if (k + 2 < D.nz) r_up = load(dn_ + half, hn_ + half, ln_ + half, own);
      }
      __syncthreads();
      const CgLevel& L = lv[k];
      float2 H, Lo, ph, pl, eh, el;
      // x: the faces (west, middle) and (middle, east) of the pair
      float4 pw = make_float4(__shfl_up_sync(~0u, cur.dh.y, 1), __shfl_up_sync(~0u, cur.dl.y, 1),
                              __shfl_up_sync(~0u, cur.rh.y, 1), __shfl_up_sync(~0u, cur.rl.y, 1));
      float4 pe = make_float4(__shfl_down_sync(~0u, cur.dh.x, 1), __shfl_down_sync(~0u, cur.dl.x, 1),
                              __shfl_down_sync(~0u, cur.rh.x, 1), __shfl_down_sync(~0u, cur.rl.x, 1));
      if (ew) pw = ev;
      if (edge && !ew) pe = ev;
      const CgPt west = {make_float2(pw.x, cur.dh.x), make_float2(pw.y, cur.dl.x), make_float2(pw.z, cur.rh.x),
                         make_float2(pw.w, cur.rl.x)};
      const CgPt east = {make_float2(cur.dh.y, pe.x), make_float2(cur.dl.y, pe.y), make_float2(cur.rh.y, pe.z),
                         make_float2(cur.rl.y, pe.w)};
      cg_flux(west, cur, H, Lo);
      cg_flux(east, cur, eh, el);
      cg_acc(H, Lo, eh, el);
      cg_scale(H, Lo, L.kx);
      // y
      auto row = [&](int r) {
        const float4 a = sd[b][r][lane], e = sr[b][r][lane];
        return CgPt{make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(e.x, e.y), make_float2(e.z, e.w)};
      };
      cg_flux(row(w), cur, ph, pl);
      cg_flux(row(w + 2), cur, eh, el);
      cg_acc(ph, pl, eh, el);
      cg_scale(ph, pl, L.ky);
      cg_acc(H, Lo, ph, pl);
      // z
      cg_flux(up, cur, ph, pl);
      cg_scale(ph, pl, L.ku);
      cg_acc(H, Lo, ph, pl);
      {   // minus the flux through the lower face
        float2 s, e;
        two_diff2(H, dnh, s, e);
        H = s;
        Lo = sub2(Lo, add2(dnl, e));
      }
      dnh = ph;
      dnl = pl;
      float2 s, t;
      two_diff2(Lo, H, s, t);   // K d = -(W A d)
      if (act) {
        const double2 Kd = make_double2(ff2d_fast(s.x, t.x), ff2d_fast(s.y, t.y)), dc = dk[own];
        q[(long long)k * half + own] = Kd;
        acc = fma(dc.x, Kd.x, acc);
        acc = fma(dc.y, Kd.y, acc);
      }
      cur = up;
      dk = dn_;
      hk = hn_;
      lk = ln_;
    }
    __syncthreads();   // the buffers are reused by the next tile
  }
  cg_reduce(CG_APPLY, c, acc, 0.0, partials, D);
}

// r -= alpha q, t = -r/Wbar; sum (r/(W ||S||))^2 (the relative residual of A p = S - mu)
template <typename TT>
__global__ void __launch_bounds__(256) k_cg_update(const float2* __restrict__ rh, const double2* __restrict__ q,
                                                   double2* __restrict__ r, typename CgVec<TT>::t* __restrict__ t,
                                                   const CgLevel* __restrict__ lv, CgDims D, CgState* c,
                                                   double* __restrict__ partials) {
  const CgLevel L = lv[blockIdx.y];
  const double na = -c->alpha, iw = -L.iwbar;
  const float idz = (float)L.idz * (float)c->inv_snorm;   // the norm comes out relative to ||S||
  float rr = 0.f;
#pragma unroll 2
  CG_PAIRS(i, D) {
    const double2 qv = q[i], rv = r[i];
    const float2 h = rh[i];
    const double2 rn = make_double2(fma(na, qv.x, rv.x), fma(na, qv.y, rv.y));
    r[i] = rn;
    t[i] = CgVec<TT>::out(make_double2(rn.x * iw, rn.y * iw));
    // residual of A p = S - mu: r / (rho dz), to float accuracy (a stopping test), in the FP32 pipe
    const float ax = d2f_int(rn.x) * idz * __frcp_rn(h.x), ay = d2f_int(rn.y) * idz * __frcp_rn(h.y);
    rr = __fmaf_rn(ax, ax, __fmaf_rn(ay, ay, rr));
  }
  cg_reduce(CG_UPDATE, c, (double)rr, 0.0, partials, D);
}

// z . r and, from the second preconditioner solve on, z . q
template <typename TT, bool FIRST>
__global__ void __launch_bounds__(256) k_cg_dots(const typename CgVec<TT>::t* __restrict__ z,
                                                 const double2* __restrict__ r, const double2* __restrict__ q, CgDims D,
                                                 CgState* c, double* __restrict__ partials) {
  double zr = 0, zq = 0;
#pragma unroll 2
  CG_PAIRS(i, D) {
    const double2 zv = CgVec<TT>::in(z[i]), rv = r[i];
    zr = fma(zv.x, rv.x, zr);
    zr = fma(zv.y, rv.y, zr);
    if (!FIRST) {
      const double2 qv = q[i];
      zq = fma(zv.x, qv.x, zq);
      zq = fma(zv.y, qv.y, zq);
    }
  }
  cg_reduce(FIRST ? CG_DOTS0 : CG_DOTS, c, zr, zq, partials, D);
}

// STEP 0: d = z.  1: p = alpha d, d = z + beta d.  2: p += alpha d, d = z + beta d.
template <typename TT, int STEP>
__global__ void __launch_bounds__(256) k_cg_dir(const typename CgVec<TT>::t* __restrict__ z, double2* __restrict__ d,
                                                double2* __restrict__ p, CgDims D, const CgState* __restrict__ c) {
  const double alpha = STEP ? c->alpha : 0.0, beta = STEP ? c->beta : 0.0;
#pragma unroll 2
  CG_PAIRS(i, D) {
    const double2 zv = CgVec<TT>::in(z[i]);
    if (STEP == 0) {
      d[i] = zv;
    } else {
      const double2 dv = d[i], po = STEP == 2 ? p[i] : make_double2(0.0, 0.0);
      p[i] = STEP == 2 ? make_double2(fma(alpha, dv.x, po.x), fma(alpha, dv.y, po.y))
                       : make_double2(alpha * dv.x, alpha * dv.y);
      d[i] = make_double2(fma(beta, dv.x, zv.x), fma(beta, dv.y, zv.y));
    }
  }
}

// the last step's p (STEP as above; 3: p = 0), and sum p.  A direction with no step (d . K d not positive: d in the
// null space, or not finite) leaves p as it was.
template <int STEP>
__global__ void __launch_bounds__(256) k_cg_last(const double2* __restrict__ d, double2* __restrict__ p, CgDims D,
                                                 CgState* c, double* __restrict__ partials) {
  const double alpha = c->alpha;
  const bool step = STEP != 3 && c->dq > 0;
  double s = 0;
#pragma unroll 2
  CG_PAIRS(i, D) {
    double2 v = make_double2(0.0, 0.0);
    if (STEP == 2) v = p[i];
    if (step) {
      const double2 dv = d[i];
      v = STEP == 2 ? make_double2(fma(alpha, dv.x, v.x), fma(alpha, dv.y, v.y))
                    : make_double2(alpha * dv.x, alpha * dv.y);
    }
    p[i] = v;
    s += v.x + v.y;
  }
  cg_reduce(CG_LAST, c, s, 0.0, partials, D);
}
// p -= its mean
__global__ void __launch_bounds__(256) k_cg_shift(double2* __restrict__ p, CgDims D, const CgState* __restrict__ c) {
  const double m = c->shift;
#pragma unroll 2
  CG_PAIRS(i, D) {
    const double2 v = p[i];
    p[i] = make_double2(v.x - m, v.y - m);
  }
}

}  // namespace

// Host side ---------------------------------------------------------------------

static int cg_sms() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}
// blocks of the largest launch: eight a SM, and at least one per level
int cg_blocks(int nz) {
  const int b = cg_sms() * 8;
  return b > nz ? b : nz;
}
size_t cg_state_bytes() { return sizeof(CgState); }

cudaError_t cg_launch(int op, const CgGrid& K, const CgArgs& a, cudaStream_t st) {
  CgDims D{};
  D.nx = K.nx;
  D.ny = K.ny;
  D.nz = K.nz;
  D.plane = (long long)K.nx * K.ny;
  D.n = D.plane * K.nz;
  D.top_dirichlet = K.top_dirichlet;
  CgState* c = (CgState*)a.state;
  const int sms = cg_sms();
  long long bx = (D.plane / 2 + 255) / 256;
  const long long per_level = sms * 8 / K.nz > 1 ? sms * 8 / K.nz : 1;
  if (bx > per_level) bx = per_level;
  const dim3 g((unsigned)bx, (unsigned)K.nz);
  const long long tiles = (long long)((K.nx / 2 + 31) / 32) * ((K.ny + kCgTY - 1) / kCgTY) * ((K.nz + kCgZC - 1) / kCgZC);
  const unsigned ga = (unsigned)(tiles < sms * 8 ? tiles : sms * 8);
  const double2 *rho = (const double2*)a.rho, *S = (const double2*)a.S;
  double2 *r = (double2*)a.r, *d = (double2*)a.d, *q = (double2*)a.q, *p = (double2*)a.p;
  float2 *rh = (float2*)a.rh, *rl = (float2*)a.rl;
  double* P = a.partials;
  if (a.float_pc) {
    float2* t = (float2*)a.t;
    const float2* z = (const float2*)a.z;
    switch (op) {
      case CG_START: k_cg_start<float><<<g, 256, 0, st>>>(rho, S, r, t, a.lv, D, c, P); return cudaGetLastError();
      case CG_UPDATE: k_cg_update<float><<<g, 256, 0, st>>>(rh, q, r, t, a.lv, D, c, P); return cudaGetLastError();
      case CG_DOTS0: k_cg_dots<float, true><<<g, 256, 0, st>>>(z, r, q, D, c, P); return cudaGetLastError();
      case CG_DOTS: k_cg_dots<float, false><<<g, 256, 0, st>>>(z, r, q, D, c, P); return cudaGetLastError();
      case CG_DIR:
        if (a.step == 0) k_cg_dir<float, 0><<<g, 256, 0, st>>>(z, d, p, D, c);
        else if (a.step == 1) k_cg_dir<float, 1><<<g, 256, 0, st>>>(z, d, p, D, c);
        else k_cg_dir<float, 2><<<g, 256, 0, st>>>(z, d, p, D, c);
        return cudaGetLastError();
      default: break;
    }
  } else {
    double2* t = (double2*)a.t;
    const double2* z = (const double2*)a.z;
    switch (op) {
      case CG_START: k_cg_start<double><<<g, 256, 0, st>>>(rho, S, r, t, a.lv, D, c, P); return cudaGetLastError();
      case CG_UPDATE: k_cg_update<double><<<g, 256, 0, st>>>(rh, q, r, t, a.lv, D, c, P); return cudaGetLastError();
      case CG_DOTS0: k_cg_dots<double, true><<<g, 256, 0, st>>>(z, r, q, D, c, P); return cudaGetLastError();
      case CG_DOTS: k_cg_dots<double, false><<<g, 256, 0, st>>>(z, r, q, D, c, P); return cudaGetLastError();
      case CG_DIR:
        if (a.step == 0) k_cg_dir<double, 0><<<g, 256, 0, st>>>(z, d, p, D, c);
        else if (a.step == 1) k_cg_dir<double, 1><<<g, 256, 0, st>>>(z, d, p, D, c);
        else k_cg_dir<double, 2><<<g, 256, 0, st>>>(z, d, p, D, c);
        return cudaGetLastError();
      default: break;
    }
  }
  switch (op) {
    case CG_PREP: k_cg_prep<<<g, 256, 0, st>>>(rho, S, rh, rl, a.lv, D, c, P); break;
    case CG_APPLY: k_cg_apply<<<ga, 256, 0, st>>>(d, rh, rl, q, a.lv, D, c, P); break;
    case CG_LAST:
      if (a.step == 1) k_cg_last<1><<<g, 256, 0, st>>>(d, p, D, c, P);
      else if (a.step == 2) k_cg_last<2><<<g, 256, 0, st>>>(d, p, D, c, P);
      else k_cg_last<3><<<g, 256, 0, st>>>(d, p, D, c, P);
      break;
    case CG_SHIFT: k_cg_shift<<<g, 256, 0, st>>>(p, D, c); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t cg_read(const void* state, CgReport* out, cudaStream_t st) {
  CgState h{};
  cudaError_t e = cudaMemcpyAsync(&h, state, sizeof(h), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  out->mu = h.mu;
  out->ss = h.ss;
  out->dq = h.dq;
  out->rel2 = h.rel2;
  return e;
}

}  // namespace pgb

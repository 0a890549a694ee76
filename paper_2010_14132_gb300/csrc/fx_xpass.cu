// x-passes (R2C and C2R) of the double-precision plans in 64-bit block fixed point (fx_engine.cuh), and the
// twiddle tables of its transforms.  (Section 2.1: the x transform of every row of every level.)
//
// One CTA takes RB rows, a line of N = nx/2 packed points per N/E threads, two shared line buffers per row
// (one barrier per stage).  First-stage inputs come straight from global memory (forward) and last-stage
// outputs go straight back (inverse); twiddles are read from the plan's stage-ordered table through L1.
// CTAs of about 128 threads: six fit an SM at 80 registers a thread, and their loads, conversions (FP64 unit)
// and butterflies (integer units) overlap.
#include <cmath>
#include <vector>

#include "fx_engine.cuh"
#include "kernels.cuh"

namespace pgb {
namespace {

constexpr int fx_x_rows(int n) {   // rows per CTA: about 128 threads
  const int nl = n / fx_elems(n);
  return nl >= 128 ? 1 : (128 + nl / 2) / nl;
}

// Largest exponent field and sum of magnitudes over a line's threads.  Lines inside a warp reduce by
// shuffles; wider or odd ones through a shared word per line (zeroed before).
template <int NL> struct FxLine {
  static constexpr bool kWarp = NL <= 32 && 32 % NL == 0;
  static __device__ __forceinline__ int max_exp(int e, int* slot, LineSyncT<NL> sync) {
    if constexpr (kWarp) {
#pragma unroll
      for (int o = NL / 2; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
      return e;
    } else {
      if constexpr (NL % 32 == 0) {
        e = __reduce_max_sync(0xffffffffu, e);
        if ((threadIdx.x & 31) == 0) atomicMax(slot, e);
      } else {
        atomicMax(slot, e);
      }
      sync();
      return *slot;
    }
  }
  // the sum is in *slot after the line's next barrier
  static __device__ __forceinline__ void sum(unsigned s, unsigned* slot) {
    if constexpr (kWarp) {
#pragma unroll
      for (int o = NL / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (threadIdx.x == 0) *slot = s;
    } else if constexpr (NL % 32 == 0) {
      s = __reduce_add_sync(0xffffffffu, s);
      if ((threadIdx.x & 31) == 0) atomicAdd(slot, s);
    } else {
      atomicAdd(slot, s);
    }
  }
};

template <int N>
__global__ void __launch_bounds__(N / fx_elems(N) * fx_x_rows(N)) k_xfwd_fx(const double* __restrict__ in,
                                                                           double2* __restrict__ spec, Geom g,
                                                                           const int4* __restrict__ tw,
                                                                           const int4* __restrict__ twr) {
  constexpr int E = fx_elems(N), nl = N / E, RB = fx_x_rows(N), LS = fx_line_stride(N);
  // one more bit of room than the transform needs: 2 |X_k| <= |Z_k + conj Z_{N-k}| + |Z_k - conj Z_{N-k}|
  constexpr int T = 60 - clog2(fx_radix(N, 0, E));
  pdl_trigger();
  extern __shared__ __align__(128) unsigned char smraw[];
  Fx2* lines = reinterpret_cast<Fx2*>(smraw);
  int* emax_s = reinterpret_cast<int*>(lines + RB * 2 * LS);
  unsigned* l1_s = reinterpret_cast<unsigned*>(emax_s + RB);
  const int lane = threadIdx.x, ty = threadIdx.y;
  const long long row = (long long)g.lev0 * g.ny + (long long)blockIdx.x * RB + ty;
  const bool valid = row < (long long)g.lev1 * g.ny;
  const LineSyncT<nl> sync{1 + ty};
  const Swizzled16 sw{};
  Fx2* la = lines + (size_t)ty * 2 * LS;
  if (lane == 0) {
    emax_s[ty] = 0;
    l1_s[ty] = 0;
  }
  pdl_wait();
  const double2* src = reinterpret_cast<const double2*>(in + (valid ? row : 0) * g.nx);
  double2 x[E];
#pragma unroll
  for (int i = 0; i < E; ++i) x[i] = valid ? __ldcs(&src[fx_in_index<N, E>(lane, i)]) : make_double2(0, 0);
  sync();
  unsigned h = 0;
#pragma unroll
  for (int i = 0; i < E; ++i) h = max(h, max(fx_hi_abs(x[i].x), fx_hi_abs(x[i].y)));
  int e = FxLine<nl>::max_exp((int)(h >> 20), &emax_s[ty], sync);
  const bool bad = e == 0x7ff;
  e = max(e, 1);
  const FxIn to_i(e, T);
  Fx2 v[E];
  unsigned l1 = 0;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    v[i] = {to_i(x[i].x), to_i(x[i].y)};
    l1 += fx_mag(v[i].x) + fx_mag(v[i].y);
  }
  FxLine<nl>::sum(fx_l1(2 * l1), &l1_s[ty]);   // twice the sum: the spare bit again
  int l1b = 0;
  const Fx2* fin = fx_run_from<N, E, false, 0, false>(v, la, la + LS, sw, lane, tw, sync, &l1_s[ty], l1b);
  // unpack the bin pairs (k, N - k): 2 X_k = 2 E_k + w^k 2 O_k, X_{N-k} = conj(E_k - w^k O_k)
  const FxOut to_d(fx_total_shift<N, E>(l1b) + e - 1022 - T - 1, bad);
  double2* dst = spec + (valid ? row : 0) * g.P;
#pragma unroll
  for (int q = 0; q < E / 2; ++q) {
    const int k = lane + nl * q;   // k < N/2
    const Fx2 zk = fin[sw(k)], zc = fin[sw(k == 0 ? 0 : N - k)];
    const Fx2 ev = {zk.x + zc.x, zk.y - zc.y};
    const Fx2 wo = fx_cmul(Fx2{zk.y + zc.y, zc.x - zk.x}, __ldg(&twr[k]), 3);   // w^k (-i (Z_k - conj Z_{N-k}))
    if (valid) {
      dst[k] = make_double2(to_d(ev.x + wo.x), to_d(ev.y + wo.y));
      dst[N - k] = make_double2(to_d(ev.x - wo.x), to_d(wo.y - ev.y));
    }
  }
  if (lane == 0 && valid) {   // the self-paired bin: X_{N/2} = conj Z_{N/2}
    const Fx2 z = fin[sw(N / 2)];
    dst[N / 2] = make_double2(to_d(z.x + z.x), to_d(-(z.y + z.y)));
  }
}

template <int N>
__global__ void __launch_bounds__(N / fx_elems(N) * fx_x_rows(N)) k_xinv_fx(const double2* __restrict__ spec,
                                                                           double* __restrict__ out, Geom g,
                                                                           const int4* __restrict__ tw,
                                                                           const int4* __restrict__ twr) {
  constexpr int E = fx_elems(N), nl = N / E, RB = fx_x_rows(N), LS = fx_line_stride(N);
  // two more bits of room than the transform needs: |z| <= 2 (|X_m| + |X_{N-m}|)
  constexpr int T = 59 - clog2(fx_radix(N, 0, E));
  pdl_trigger();
  extern __shared__ __align__(128) unsigned char smraw[];
  Fx2* lines = reinterpret_cast<Fx2*>(smraw);
  int* emax_s = reinterpret_cast<int*>(lines + RB * 2 * LS);
  unsigned* l1_s = reinterpret_cast<unsigned*>(emax_s + RB);
  const int lane = threadIdx.x, ty = threadIdx.y;
  const long long row = (long long)g.lev0 * g.ny + (long long)blockIdx.x * RB + ty;
  const bool valid = row < (long long)g.lev1 * g.ny;
  const LineSyncT<nl> sync{1 + ty};
  const Swizzled16 sw{};
  Fx2* la = lines + (size_t)ty * 2 * LS;
  if (lane == 0) {
    emax_s[ty] = 0;
    l1_s[ty] = 0;
  }
  pdl_wait();
  const double2* src = spec + (valid ? row : 0) * g.P;
  double2 x[E], xn = make_double2(0, 0);
#pragma unroll
  for (int q = 0; q < E; ++q) x[q] = valid ? __ldcs(&src[lane + nl * q]) : make_double2(0, 0);
  if (lane == 0) {   // self-conjugate bins: real parts only
    if (valid) xn.x = __ldcs(&src[N].x);
    x[0].y = 0;
  }
  sync();
  unsigned h = fx_hi_abs(xn.x);
#pragma unroll
  for (int q = 0; q < E; ++q) h = max(h, max(fx_hi_abs(x[q].x), fx_hi_abs(x[q].y)));
  int e = FxLine<nl>::max_exp((int)(h >> 20), &emax_s[ty], sync);
  const bool bad = e == 0x7ff;
  e = max(e, 1);
  const FxIn to_i(e, T);
  unsigned l1 = 0;
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const Fx2 a = {to_i(x[q].x), to_i(x[q].y)};
    l1 += fx_mag(a.x) + fx_mag(a.y);
    la[sw(lane + nl * q)] = a;
  }
  if (lane == 0) {
    const i64 a = to_i(xn.x);
    l1 += fx_mag(a);
    la[sw(N)] = {a, 0};
  }
  FxLine<nl>::sum(fx_l1(4 * l1), &l1_s[ty]);   // sum |z| <= 4 sum |X|
  sync();
  Fx2 v[E];
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int m = fx_in_index<N, E>(lane, i);
    const Fx2 xk = la[sw(m)], xc = la[sw(N - m)];
    const Fx2 ev = {xk.x + xc.x, xk.y - xc.y};
    int4 w = __ldg(&twr[m]);   // its conjugate: exp(+2 pi i m/nx)
    w.z = -w.z;
    w.w = -w.w;
    const Fx2 od = fx_cmul(Fx2{xk.x - xc.x, xk.y + xc.y}, w, 3);
    v[i] = {ev.y + od.x, ev.x - od.y};   // ev + i od, parts exchanged for the inverse transform
  }
  int l1b = 0;
  fx_run_from<N, E, true, 0, false>(v, la + LS, la, sw, lane, tw, sync, &l1_s[ty], l1b);
  if (!valid) return;
  const FxOut to_d(fx_total_shift<N, E>(l1b) + e - 1022 - T, bad);
  double2* dst = reinterpret_cast<double2*>(out + row * g.nx);
#pragma unroll
  for (int i = 0; i < E; ++i)
    __stcs(&dst[fx_out_index<N, E>(lane, i)],
           make_double2(to_d(v[i].y), to_d(v[i].x)));
}

template <int N> struct FxX {
  static constexpr int nl = N / fx_elems(N), RB = fx_x_rows(N);
  static constexpr size_t smem = (size_t)RB * (2 * fx_line_stride(N) * sizeof(Fx2) + sizeof(int) + sizeof(unsigned));
  static dim3 grid(const Geom& g) {
    return dim3((unsigned)(((long long)g.ny * (g.lev1 - g.lev0) + RB - 1) / RB));
  }
};

// exp(-2 pi i m/n) in units of 2^-61 as balanced halves (re high, re low, im high, im low); the angle is
// reduced to an eighth of a turn in integers, so the parts are good to the last unit
int4 fx_twiddle(long long m, long long n) {
  m %= n;
  const long long o = 8 * m / n, r = 8 * m - o * n;   // octant, and the rest in eighths of n
  const long double q = 0.785398163397448309615660845819875721L;   // pi/4
  const long double th = q * (long double)(o % 2 ? n - r : r) / (long double)n;
  long double c = cosl(th), s = o % 2 ? -sinl(th) : sinl(th);
  for (long long k = (o + 1) / 2; k > 0; --k) {   // quarter turns
    const long double t = c;
    c = -s;
    s = t;
  }
  auto halves = [](long double v, int& hi, int& lo) {
    const long long f = llrintl(v * 2305843009213693952.0L);   // 2^61
    lo = (int)(unsigned)(unsigned long long)f;
    hi = (int)((f - lo) / 4294967296ll);   // exact
    if (lo == (int)0x80000000) lo += 1;    // its negative has to exist
  };
  int4 w;
  halves(c, w.x, w.y);
  halves(-s, w.z, w.w);
  return w;
}

}  // namespace

std::vector<int4> fx_stage_table(int n) {
  std::vector<int4> t;
  if (!fx_length(n)) return t;
  const int E = fx_elems(n);
  for (int s = 0, Ns = 1; s < fx_nstages(n, E); ++s) {
    const int R = fx_radix(n, s, E);
    for (int r = 1; r < R; ++r)
      for (int k = 0; k < Ns; ++k) t.push_back(fx_twiddle((long long)r * k, (long long)Ns * R));
    Ns *= R;
  }
  return t;
}

std::vector<int4> fx_unpack_table(int nx) {
  std::vector<int4> t;
  for (int m = 0; m <= nx / 2; ++m) t.push_back(fx_twiddle(m, nx));
  return t;
}

cudaError_t launch_xfwd_fx(const double* in, double2* spec, const Geom& g, int n, const Tables& tb, cudaStream_t st,
                           bool* used) {
  *used = false;
  if (!tb.twx_q || !tb.twr_q) return cudaSuccess;
  PGB_FX_N_SWITCH(n, {
    const cudaError_t e = allow_smem(k_xfwd_fx<NN>, FxX<NN>::smem);
    if (e != cudaSuccess) return e;
    *used = true;
    return pdl_launch(k_xfwd_fx<NN>, FxX<NN>::grid(g), dim3(FxX<NN>::nl, FxX<NN>::RB), FxX<NN>::smem, st, in, spec, g,
                      tb.twx_q, tb.twr_q);
  });
}

cudaError_t launch_xinv_fx(const double2* spec, double* out, const Geom& g, int n, const Tables& tb, cudaStream_t st,
                           bool* used) {
  *used = false;
  if (!tb.twx_q || !tb.twr_q) return cudaSuccess;
  PGB_FX_N_SWITCH(n, {
    const cudaError_t e = allow_smem(k_xinv_fx<NN>, FxX<NN>::smem);
    if (e != cudaSuccess) return e;
    *used = true;
    return pdl_launch(k_xinv_fx<NN>, FxX<NN>::grid(g), dim3(FxX<NN>::nl, FxX<NN>::RB), FxX<NN>::smem, st, spec, out, g,
                      tb.twx_q, tb.twr_q);
  });
}

}  // namespace pgb

// y-pass (both directions) of the double-precision plans in 64-bit block fixed point (fx_engine.cuh), in place
// on the spectrum.  (Section 2.1: the y transform of every kx column of every level.)
//
// One CTA takes TK consecutive kx of one level: thread (l, lane) holds E
// elements of column l, loaded straight from global memory, exchanged between stages through one shared
// [N][TK] tile, and stored from registers after the last stage.  Every column has its own scale.

#include "fx_engine.cuh"
#include "kernels.cuh"

namespace pgb {
namespace {

// columns per CTA: 8 (128-byte row segments) up to 32 KB of tile, then fewer
constexpr int fx_y_cols(int n) { return n <= 256 ? 8 : (n <= 576 ? 4 : 2); }

// resident CTAs asked of the compiler: 768 threads per SM leave 80 registers a thread, just enough without
// spills (512 threads of 110 registers, one CTA per SM, took 147 instead of 99 us at 512 x 512 x 64)
#ifndef PGB_FXY_THREADS
#define PGB_FXY_THREADS 768
#endif
constexpr int fx_y_blocks(int n) {
  const int t = n / fx_elems(n) * fx_y_cols(n), want = n % 3 == 0 ? 512 : PGB_FXY_THREADS;
  return want / t < 1 ? 1 : (want / t > 16 ? 16 : want / t);
}

// element idx of a column in the [N][TK] tile; with TK < 8 several lanes share a 128-byte phase, and the first
// stage's stride of 8 rows would put all of them in the same part of it
template <int TK> struct FxTile {
  __device__ __forceinline__ int operator()(int idx) const { return (idx ^ ((idx >> 3) & (8 / TK - 1))) * TK; }
};

template <int N>
__global__ void __launch_bounds__(N / fx_elems(N) * fx_y_cols(N), fx_y_blocks(N)) k_yfft_fx(double2* __restrict__ spec, Geom g,
                                                                           const int4* __restrict__ tw, int inverse) {
  constexpr int E = fx_elems(N), nl = N / E, TK = fx_y_cols(N);
  constexpr int T = 61 - clog2(fx_radix(N, 0, E));
  constexpr bool kShuffle = (TK * nl) % 32 == 0;
  pdl_trigger();
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ int emax_s[TK];
  __shared__ unsigned l1_s[TK];
  const int l = threadIdx.x, lane = threadIdx.y;
  const int kx = blockIdx.x * TK + l;
  const bool vcol = kx < g.nxh;
  double2* base = spec + (long long)(g.lev0 + blockIdx.y) * g.plane + kx;
  if (lane == 0) {
    emax_s[l] = 0;
    l1_s[l] = 0;
  }
  pdl_wait();
  double2 x[E];
#pragma unroll
  for (int i = 0; i < E; ++i)
    x[i] = vcol ? base[(long long)fx_in_index<N, E>(lane, i) * g.P] : make_double2(0, 0);
  __syncthreads();
  unsigned h = 0;
#pragma unroll
  for (int i = 0; i < E; ++i) h = max(h, max(fx_hi_abs(x[i].x), fx_hi_abs(x[i].y)));
  int e = (int)(h >> 20);
  if constexpr (kShuffle) {
#pragma unroll
    for (int o = TK; o < 32; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if (((lane * TK + l) & 31) < TK) atomicMax(&emax_s[l], e);
  } else {
    atomicMax(&emax_s[l], e);
  }
  __syncthreads();
  e = emax_s[l];
  const bool bad = e == 0x7ff;
  e = max(e, 1);
  const FxIn to_i(e, T);
  Fx2 v[E];
  unsigned l1 = 0;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const i64 a = to_i(x[i].x), b = to_i(x[i].y);
    l1 += fx_mag(a) + fx_mag(b);
    v[i] = inverse ? Fx2{b, a} : Fx2{a, b};
  }
  l1 = fx_l1(l1);
  if constexpr (kShuffle) {
#pragma unroll
    for (int o = TK; o < 32; o <<= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, o);
    if (((lane * TK + l) & 31) < TK) atomicAdd(&l1_s[l], l1);
  } else {
    atomicAdd(&l1_s[l], l1);
  }
  int l1b = 0;
  Fx2* tile = reinterpret_cast<Fx2*>(smraw) + l;
  fx_run_from<N, E, true, 0, true>(v, tile, tile, FxTile<TK>{}, lane, tw, SyncBlock{}, &l1_s[l], l1b);
  if (!vcol) return;
  const FxOut to_d(fx_total_shift<N, E>(l1b) + e - 1022 - T, bad);
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const double a = to_d(v[i].x), b = to_d(v[i].y);
    base[(long long)fx_out_index<N, E>(lane, i) * g.P] = inverse ? make_double2(b, a) : make_double2(a, b);
  }
}

}  // namespace

cudaError_t launch_yfft_fx(int sign, double2* spec, const Geom& g, int n, const Tables& tb, cudaStream_t st,
                           bool* used) {
  *used = false;
  if (!tb.twy_q) return cudaSuccess;
  PGB_FX_N_SWITCH(n, {
    constexpr int TK = fx_y_cols(NN);
    constexpr size_t smem = (size_t)TK * NN * sizeof(Fx2);
    const cudaError_t e = allow_smem(k_yfft_fx<NN>, smem);
    if (e != cudaSuccess) return e;
    *used = true;
    return pdl_launch(k_yfft_fx<NN>, dim3((g.nxh + TK - 1) / TK, g.lev1 - g.lev0), dim3(TK, NN / fx_elems(NN)), smem,
                      st, spec, g, tb.twy_q, sign > 0 ? 1 : 0);
  });
}

}  // namespace pgb

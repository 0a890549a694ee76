// Stockham FFT of double-precision lines in 64-bit block fixed point.
//
// The FP64 units of GB300 issue 1.7 operations a clock and SM (measured), the integer units 60 64-bit adds
// or 24 32 x 32 -> 64 multiply-adds.  A butterfly in 64-bit integers therefore costs a thirty-sixth of its
// FP64 form per addition and a fifth per complex multiplication (2.2 against 0.42 a clock and SM), and the
// FP64 transforms were bound by nothing else.  A line is read as doubles, scaled to integers by one power of
// two, transformed, and written back as doubles:
//
//  * Scale: with e the largest exponent of the line's components, they become integers up to 2^T in
//    magnitude, T = 61 - L0, 2^L0 >= the first stage's radix, so no complex value passes 2^62 there.
//  * Growth: after stage s no value exceeds min(radix product x max|z|, sum of |components|); the stage shifts
//    right by just as many bits as that bound asks for (0 to 3, read out of the 96-bit product for free),
//    rounding to nearest.  A line dominated by one bin is not shifted at all, noise by about log2(n) - 2 bits.
//  * Accuracy: with n elements, ||X||_rms = ||x||_2 and sum |x| <= sqrt(n) ||x||_2, the rounding of the last
//    stages, about 2^-62 of that sum, is within a few 2^-62 sqrt(n) of the result's norm: 2^-56 for n = 1024,
//    where FP64 butterflies leave some 2^-52.5.  The conversion back rounds to 53 bits.  Whole solves with
//    lines of 16 to 2048 points, measured against extended precision: errors 0.62 of the butterflies' for noise,
//    0.7 to 0.8 for fields with a dominant bin, an outlier or a weak level, 0.02 where low wavenumbers amplify
//    what the transforms leave in them.
//  * A line that holds an infinity or a NaN gives NaN throughout (`bad`); results above the double range
//    are infinities, those below the normal range subnormal numbers.
//
// What it gave (GB300, 512 x 512 x 64, one pass over the field): forward x 584 -> 85 us, y 440 -> 94, inverse x
// 560 -> 91.  The passes are now bound by the integer pipe (65% busy, about 230 instructions a complex point)
// with the register file limiting an SM to 24 warps; the HBM floor of a pass is 40 us.
//
// The 64-bit products take both factors in balanced halves, x = xh 2^32 + xl with xl signed, and drop only
// xl yl (below one unit of the result).  The inverse transform is the forward one with real and imaginary
// parts exchanged on the way in and out.
#pragma once

#include "fft_static.cuh"
#include "kernel_grants.cuh"

namespace pgb {

typedef long long i64;

struct __align__(16) Fx2 {
  i64 x, y;
};

constexpr int clog2(long long n) {
  int b = 0;
  while ((1LL << b) < n) ++b;
  return b;
}
// elements per thread: 8 for powers of two, 12 (or 6) for lengths with a factor 3
constexpr int fx_elems(int n) { return st_elems(n); }
// Radix schedule: the 3s first, then 8 (or 4 for E = 12 and 6), then what is left of 2.  Not the composite radices of the
// FP32 transforms: a radix-12 stage drops its bits before twelve sums instead of after each three or four, which was
// 1.09x to 1.17x faster and less exact (768 x 576: max error 2.0e-15 of the field's against 0.8e-15; in FP64 arithmetic
// 1.3e-15).
constexpr int fx_radix(int n, int s, int e) {
  const int a = st_count(n, 2), b = st_count(n, 3), L = st_big_log(e);
  if (s < b) return 3;
  return s - b < a / L ? 1 << L : 1 << (a % L);
}
constexpr int fx_nstages(int n, int e) {
  return st_count(n, 3) + st_count(n, 2) / st_big_log(e) + (st_count(n, 2) % st_big_log(e) ? 1 : 0);
}
constexpr int fx_span(int n, int s, int e) {
  int ns = 1;
  for (int i = 0; i < s; ++i) ns *= fx_radix(n, i, e);
  return ns;
}
// element held in slot i before the first stage, and after the last
template <int N, int E> __device__ __forceinline__ int fx_in_index(int lane, int i) {
  constexpr int R = fx_radix(N, 0, E);
  return lane + (N / E) * (i / R) + (i % R) * (N / R);
}
template <int N, int E> __device__ __forceinline__ int fx_out_index(int lane, int i) {
  constexpr int S = fx_nstages(N, E) - 1, R = fx_radix(N, S, E), Ns = fx_span(N, S, E);
  return lane + (N / E) * (i / R) + (i % R) * Ns;
}
// lengths the kernels are built for
constexpr bool fx_length(int n) {
  switch (n) {
    case 16: case 32: case 64: case 128: case 256: case 512: case 1024: case 2048:
    case 24: case 48: case 96: case 192: case 384: case 768:
    case 36: case 72: case 144: case 288: case 576:
    case 18: case 54: case 108: case 216: case 432: case 864: case 324:
      return true;
    default: return false;
  }
}

__device__ __forceinline__ i64 fx_madw(int a, int b, i64 c) {   // a b + c
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ int fx_hi(i64 a) { return (int)((unsigned long long)a >> 32) + (int)((unsigned)a >> 31); }
__device__ __forceinline__ Fx2 fx_add(Fx2 a, Fx2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Fx2 fx_sub(Fx2 a, Fx2 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ Fx2 fx_mul_mi(Fx2 a) { return {a.y, -a.x}; }   // times -i
// the top 64 bits of (h : low word of m) << t, 0 <= t <= 31
__device__ __forceinline__ i64 fx_join(i64 h, i64 m, int t) {
  const unsigned hl = (unsigned)h, hh = (unsigned)((unsigned long long)h >> 32);
  const unsigned lo = __funnelshift_l((unsigned)m, hl, t), hi = __funnelshift_l(hl, hh, t);
  return (i64)(((unsigned long long)hi << 32) | lo);
}
// a w 2^(t-3) with w = (re, im) in units of 2^-61, halves (rh, rl, ih, il); |a| <= 2^62
__device__ __forceinline__ Fx2 fx_cmul(Fx2 a, int4 w, int t) {
  const i64 half = (i64)(0x80000000u >> t);
  const int rl = (int)a.x, rh = fx_hi(a.x), il = (int)a.y, ih = fx_hi(a.y);
  const int nih = -w.z, nil = -w.w;
  const i64 m = fx_madw(il, nih, fx_madw(ih, nil, fx_madw(rl, w.x, fx_madw(rh, w.y, half))));
  const i64 h = fx_madw(ih, nih, fx_madw(rh, w.x, (i64)(int)((unsigned long long)m >> 32)));
  const i64 n = fx_madw(il, w.x, fx_madw(ih, w.y, fx_madw(rl, w.z, fx_madw(rh, w.w, half))));
  const i64 g = fx_madw(ih, w.x, fx_madw(rh, w.z, (i64)(int)((unsigned long long)n >> 32)));
  return {fx_join(h, m, t), fx_join(g, n, t)};
}
// a c for a constant c < 1 given as c 2^62 in balanced halves
__device__ __forceinline__ i64 fx_mulc(i64 a, int ch, int cl) {
  const int al = (int)a, ah = fx_hi(a);
  const i64 m = fx_madw(al, ch, fx_madw(ah, cl, 0x20000000ll));
  const i64 h = fx_madw(ah, ch, (i64)(int)((unsigned long long)m >> 32));
  return fx_join(h, m, 2);
}
constexpr i64 kFxSqrtHalf = 3260954456333195553ll;    // 2^62 sqrt(1/2)
constexpr i64 kFxSqrt3Half = 3993837246235628775ll;   // 2^62 sqrt(3)/2
__device__ __forceinline__ i64 fx_mul_sqrt_half(i64 a) {
  return fx_mulc(a, (int)((kFxSqrtHalf + 0x80000000ll) >> 32), (int)kFxSqrtHalf);
}
__device__ __forceinline__ i64 fx_mul_sqrt3_half(i64 a) {
  return fx_mulc(a, (int)((kFxSqrt3Half + 0x80000000ll) >> 32), (int)kFxSqrt3Half);
}
// a / 2^s rounded to nearest, ties to even (rounding them up would leave the same bias in every bin, an
// impulse at index 0 of the other side), 0 <= s <= 3
__device__ __forceinline__ i64 fx_shr(i64 a, int s) {
  const int odd = (int)((unsigned)a >> s) & 1;
  return (a + (((1 << s) >> 1) - (s ? 1 - odd : 0))) >> s;
}

// forward DFTs of R values
__device__ __forceinline__ void fx_dft4(Fx2& x0, Fx2& x1, Fx2& x2, Fx2& x3) {
  const Fx2 a = fx_add(x0, x2), b = fx_sub(x0, x2);
  const Fx2 c = fx_add(x1, x3), d = fx_mul_mi(fx_sub(x1, x3));
  x0 = fx_add(a, c);
  x2 = fx_sub(a, c);
  x1 = fx_add(b, d);
  x3 = fx_sub(b, d);
}
template <int R> __device__ __forceinline__ void fx_dft(Fx2* v) {
  if constexpr (R == 2) {
    const Fx2 t = v[0];
    v[0] = fx_add(t, v[1]);
    v[1] = fx_sub(t, v[1]);
  } else if constexpr (R == 3) {
    const Fx2 t = fx_add(v[1], v[2]), u = fx_sub(v[1], v[2]);
    const Fx2 m = {v[0].x - fx_shr(t.x, 1), v[0].y - fx_shr(t.y, 1)};
    const Fx2 su = {fx_mul_sqrt3_half(u.y), -fx_mul_sqrt3_half(u.x)};   // -i sqrt(3)/2 u
    v[0] = fx_add(v[0], t);
    v[1] = fx_add(m, su);
    v[2] = fx_sub(m, su);
  } else if constexpr (R == 4) {
    fx_dft4(v[0], v[1], v[2], v[3]);
  } else {
    static_assert(R == 8, "radix");
    Fx2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    fx_dft4(e0, e1, e2, e3);
    fx_dft4(o0, o1, o2, o3);
    // w = (1 - i)/sqrt2, w^2 = -i, w^3 = w w^2
    const Fx2 w1 = {fx_mul_sqrt_half(o1.x + o1.y), fx_mul_sqrt_half(o1.y - o1.x)};
    const Fx2 w2 = fx_mul_mi(o2);
    const Fx2 w3 = {fx_mul_sqrt_half(o3.y - o3.x), fx_mul_sqrt_half(-o3.x - o3.y)};
    v[0] = fx_add(e0, o0);
    v[4] = fx_sub(e0, o0);
    v[1] = fx_add(e1, w1);
    v[5] = fx_sub(e1, w1);
    v[2] = fx_add(e2, w2);
    v[6] = fx_sub(e2, w2);
    v[3] = fx_add(e3, w3);
    v[7] = fx_sub(e3, w3);
  }
}

// ---------------------------------------------------------------------------
// conversions
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned fx_hi_abs(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
// The largest |high word| of a line gives its exponent field e (taken as at least 1).
// x 2^(T + 1022 - e) rounded to an integer, up to 2^T in magnitude: the exponent field is moved and the value
// converted (two conversions a clock and SM on the otherwise idle FP64 unit, against some 16 integer
// instructions).  What would leave the normal range is below 2^-900 then: 0.  Lines whose largest
// exponent lies near the lower end, where subnormal numbers count, take the integer form.
static __device__ __noinline__ i64 fx_from_double_any(double x, int e, int T) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = (b & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0ull);
  const int d = 63 - T + e - (ex ? ex : 1);   // right shift of m 2^10 (below 2^63), >= 2
  unsigned long long r = 0;
  if (d < 64) {
    r = (m << 10) >> d;
    const unsigned long long rest = (m << 10) << (64 - d), half = 1ull << 63;
    if (rest > half || (rest == half && (r & 1))) ++r;
  }
  return (b >> 63) ? -(i64)r : (i64)r;
}
struct FxIn {
  int e, T, add;
  unsigned low;
  bool any;
  __device__ __forceinline__ FxIn(int e_, int T_) : e(e_), T(T_), any(e_ < 100 || e_ == 0x7ff) {
    add = (T + 1022 - e) << 20;
    low = e > T + 1022 ? (unsigned)(e - T - 1021) << 20 : 0x100000u;   // smaller exponent fields would wrap
  }
  __device__ __forceinline__ i64 operator()(double x) const {
    if (any) return fx_from_double_any(x, e, T);
    const int hi = __double2hiint(x);
    const bool keep = ((unsigned)hi & 0x7fffffffu) >= low;
    return __double2ll_rn(__hiloint2double(keep ? hi + add : 0, keep ? __double2loint(x) : 0));
  }
};
// v 2^q rounded to the nearest double (subnormal below the normal range, infinity above); bad: NaN
static __device__ __noinline__ double fx_to_double_any(i64 v, int q, bool bad) {
  const i64 s = v >> 63;
  unsigned long long m = (unsigned long long)((v ^ s) - s);
  const int z = __clzll((i64)m);
  m <<= (z & 63);
  const int be = 1086 + q - z;   // biased exponent of the leading bit
  const int d = be >= 1 ? 11 : 12 - be;   // bits below the last one kept: 11, more for a subnormal number
  unsigned long long r = d < 64 ? m >> d : 0ull;
  const unsigned long long rest = d < 64 ? m << (64 - d) : (d == 64 ? m : 0ull), half = 1ull << 63;
  r += (rest > half || (rest == half && (r & 1))) ? 1u : 0u;
  if (be >= 1) r += (unsigned long long)(unsigned)(be - 1) << 52;   // the leading bit is the exponent's last unit
  r = be >= 2047 ? 0x7ff0000000000000ull : r;
  r = z == 64 ? 0ull : r;
  r |= (unsigned long long)s & 0x8000000000000000ull;
  r = bad ? 0x7ff8000000000000ull : r;
  return __longlong_as_double((i64)r);
}
// The same for a line whose results all have normal exponents (any = false), by the conversion instruction
// (two a clock and SM on the otherwise idle FP64 unit, against some 20 integer instructions) and an addition
// to the exponent field.
struct FxOut {
  int q;
  bool any, bad;
  __device__ __forceinline__ FxOut(int q_, bool bad_) : q(q_), any(bad_ || q_ < -1000 || q_ > 950), bad(bad_) {}
  __device__ __forceinline__ double operator()(i64 v) const {
    if (any) return fx_to_double_any(v, q, bad);
    const double d = (double)v;
    const int hi = __double2hiint(d);
    return __hiloint2double(v == 0 ? hi : hi + (q << 20), __double2loint(d));
  }
};
// Sum of magnitudes: a thread adds up fx_mag of at most 24 components (T <= 59), then gives fx_l1 of that sum,
// in units of 2^39, to the sum over the line's threads (at most 2^12 components in all).
__device__ __forceinline__ unsigned fx_mag(i64 v) {
  const int h = (int)((unsigned long long)v >> 32);
  return (unsigned)(h < 0 ? -h : h) + 1u;
}
__device__ __forceinline__ unsigned fx_l1(unsigned sum_mag) { return (sum_mag >> 7) + 1u; }
__device__ __forceinline__ int fx_l1_bits(unsigned s) { return 71 - __clz((int)s); }   // sum of magnitudes < 2^bits

// Right shifts up to and including stage S (S >= 1) for a line whose magnitudes sum to less than 2^l1b.
template <int N, int E, int S> __device__ __forceinline__ int fx_shift_sum(int l1b) {
  if constexpr (S <= 0) {
    return 0;
  } else {
    constexpr int L0 = clog2(fx_radix(N, 0, E)), K = clog2((long long)fx_span(N, S, E) * fx_radix(N, S, E)) - L0;
    const int c = l1b - 62 < K ? l1b - 62 : K;
    return c > 0 ? c : 0;
  }
}
template <int N, int E> __device__ __forceinline__ int fx_total_shift(int l1b) {
  return fx_shift_sum<N, E, fx_nstages(N, E) - 1>(l1b);
}
// shift count per stage never passes 3: K grows by at most clog2(radix) <= 3 from stage to stage

// Shared-memory slot of element idx of a contiguous line of 16-byte elements: the low three bits XORed with
// the next three, so that the stride-R writes of the first stage spread over all banks.
struct Swizzled16 {
  __device__ __forceinline__ int operator()(int idx) const { return idx ^ ((idx >> 3) & 7); }
};
__host__ __device__ constexpr int fx_line_stride(int n) { return (n + 8) / 8 * 8; }

// Stages from S on.  v: the stage's inputs (slot i = what st_store and st_load put there).  FINAL_IN_REGS as in
// fft_static.cuh; the result is true / 2^(total shift) in the scale of the inputs.  l1 (shared) is read after
// the first exchange's barrier.
template <int N, int E, bool FINAL_IN_REGS, int S, bool INPLACE, typename Addr, typename Sync>
__device__ __forceinline__ Fx2* fx_run_from(Fx2 (&v)[E], Fx2* cur, Fx2* nxt, Addr addr, int lane,
                                            const int4* __restrict__ tw, Sync sync, const unsigned* l1, int& l1b) {
  constexpr int NST = fx_nstages(N, E), R = fx_radix(N, S, E), Ns = fx_span(N, S, E), B = E / R, nl = N / E;
  if constexpr (S > 0) {
    if constexpr (S == 1) l1b = fx_l1_bits(*l1);
    const int sh = fx_shift_sum<N, E, S>(l1b) - fx_shift_sum<N, E, S - 1>(l1b);
#pragma unroll
    for (int q = 0; q < B; ++q) {
      const int k = (lane + nl * q) % Ns;
      v[q * R] = {fx_shr(v[q * R].x, sh), fx_shr(v[q * R].y, sh)};
#pragma unroll
      for (int r = 1; r < R; ++r) v[q * R + r] = fx_cmul(v[q * R + r], __ldg(&tw[(Ns - 1) + (r - 1) * Ns + k]), 3 - sh);
    }
  }
#pragma unroll
  for (int q = 0; q < B; ++q) fx_dft<R>(&v[q * R]);
  if constexpr (S == NST - 1 && FINAL_IN_REGS) {
    return nullptr;
  } else {
    st_store<R, E, N, Ns>(v, cur, addr, lane);
    sync();
    if constexpr (S == NST - 1) {
      return cur;
    } else {
      st_load<fx_radix(N, S + 1, E), E, N>(v, cur, addr, lane);
      if constexpr (INPLACE) sync();
      return fx_run_from<N, E, FINAL_IN_REGS, S + 1, INPLACE>(v, nxt, cur, addr, lane, tw, sync, l1, l1b);
    }
  }
}

#define PGB_FX_N_CASE(V, ...) \
  case V: { constexpr int NN = V; __VA_ARGS__; } break;
#define PGB_FX_N_SWITCH(N, ...)                                                                                 \
  switch (N) {                                                                                                  \
    PGB_FX_N_CASE(16, __VA_ARGS__) PGB_FX_N_CASE(32, __VA_ARGS__) PGB_FX_N_CASE(64, __VA_ARGS__)                \
    PGB_FX_N_CASE(128, __VA_ARGS__) PGB_FX_N_CASE(256, __VA_ARGS__) PGB_FX_N_CASE(512, __VA_ARGS__)             \
    PGB_FX_N_CASE(1024, __VA_ARGS__) PGB_FX_N_CASE(2048, __VA_ARGS__) PGB_FX_N_CASE(24, __VA_ARGS__)            \
    PGB_FX_N_CASE(48, __VA_ARGS__) PGB_FX_N_CASE(96, __VA_ARGS__) PGB_FX_N_CASE(192, __VA_ARGS__)               \
    PGB_FX_N_CASE(384, __VA_ARGS__) PGB_FX_N_CASE(768, __VA_ARGS__) PGB_FX_N_CASE(36, __VA_ARGS__)              \
    PGB_FX_N_CASE(72, __VA_ARGS__) PGB_FX_N_CASE(144, __VA_ARGS__) PGB_FX_N_CASE(288, __VA_ARGS__)              \
    PGB_FX_N_CASE(576, __VA_ARGS__) PGB_FX_N_CASE(108, __VA_ARGS__) PGB_FX_N_CASE(216, __VA_ARGS__)             \
    PGB_FX_N_CASE(18, __VA_ARGS__) PGB_FX_N_CASE(54, __VA_ARGS__)                                               \
    PGB_FX_N_CASE(432, __VA_ARGS__) PGB_FX_N_CASE(864, __VA_ARGS__) PGB_FX_N_CASE(324, __VA_ARGS__)             \
    default: return cudaSuccess;                                                                                \
  }

}  // namespace pgb

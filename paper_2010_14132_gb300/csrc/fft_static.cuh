// Stockham FFT with the line length known at compile time.
//
// Same transform as fft_engine.cuh (stage s of radix R and span Ns takes inputs
// x[j + r n/R], applies exp(SIGN 2 pi i r (j mod Ns)/(Ns R)), an R-point DFT,
// and writes y[(j - j mod Ns) R + j mod Ns + r Ns]), with every index, span and
// table stride a constant, so the per-element work is the butterfly itself plus
// one shared-memory access.  The values of a thread stay in registers between
// stages; consecutive stages alternate between two shared buffers, so one
// barrier per stage suffices.  The caller supplies the first stage's inputs in
// registers (loaded in whatever way suits it) and receives the result either in
// registers (last stage's layout) or in natural order in a shared buffer.  With 16
// elements per thread the main radix is 16 (one stage fewer than radix 8 for
// most lengths), with 12 the composite radix 12.
#pragma once
#include "fft_engine.cuh"

namespace pgb {

// Radix schedule for n = 2^a 3^b and E elements per thread.  Powers of two: radix 32 (when E is a multiple of 32), 16, 8 (a
// multiple of 8) or 4, then a final 2, 4 or 8.  Lengths with a factor 3 (E = 12 or 6): the largest of 12, 6, 4, 3, 2 that
// divides both what is left of n and E, so that 216 = 12 6 3 takes three stages and 384 = 12 4 4 2 four.  Each stage saved
// is one exchange through shared memory and its barrier less, which is what bounds these lengths: with the stages
// 3 3 3 4 2 and 3 4 4 4 2 instead, FP32 432 x 324 x 37 takes 76.7 us against 70.1, 384 x 384 x 64 107.7 against 94.9,
// 576 x 576 x 48 206.6 against 162.1, 768 x 768 x 48 315 against 269; errors against 64 bits the same to 2 %.
constexpr int st_count(int n, int p) {
  int c = 0;
  while (n > 1 && n % p == 0) {
    n /= p;
    ++c;
  }
  return c;
}
constexpr int st_big_log(int e) { return e % 32 == 0 ? 5 : (e % 16 == 0 ? 4 : (e % 8 == 0 ? 3 : 2)); }   // log2 of the main power-of-two radix
constexpr int st_next3(int n, int e) {   // the next radix of a schedule with factors 3
  constexpr int cand[5] = {12, 6, 4, 3, 2};
  for (int i = 0; i < 5; ++i)
    if (e % cand[i] == 0 && n % cand[i] == 0) return cand[i];
  return n;
}
// Elements per thread for lengths with a factor 3: 12 values per thread keep a line's data in twice as many
// threads as 24 would, for the same shared memory
constexpr int kE3 = 12;
// ... or 6, where the length has a single factor 2
constexpr int kE3Odd = 6;
// elements per thread by length: 8 for powers of two
constexpr int st_elems(int n) { return n % 12 == 0 ? kE3 : (n % 6 == 0 ? kE3Odd : 8); }
constexpr int st_radix(int n, int s, int e) {
  if (e % 3 == 0) {
    for (; s > 0; --s) n /= st_next3(n, e);
    return st_next3(n, e);
  }
  const int a = st_count(n, 2), L = st_big_log(e);
  return s < a / L ? 1 << L : 1 << (a % L);
}
constexpr int st_nstages(int n, int e) {
  if (e % 3 == 0) {
    int c = 0;
    while (n > 1 && c < 16) {
      n /= st_next3(n, e);
      ++c;
    }
    return c;
  }
  return st_count(n, 2) / st_big_log(e) + (st_count(n, 2) % st_big_log(e) ? 1 : 0);
}
constexpr int st_span(int n, int s, int e) {
  int ns = 1;
  for (int i = 0; i < s; ++i) ns *= st_radix(n, i, e);
  return ns;
}
// E elements per thread must be a multiple of every radix of the schedule.
constexpr bool st_valid(int n, int e) {
  if (n < 2 || e < 1 || n % e != 0) return false;
  if (e == 32 && n != 512 && n != 1024) return false;   // two stages, where 16 elements take three
  if (n % 3 == 0 && e != st_elems(n)) return false;   // one element count for lengths with a factor 3
  for (int s = 0; s < st_nstages(n, e); ++s)
    if (e % st_radix(n, s, e) != 0) return false;
  return st_span(n, st_nstages(n, e), e) == n;
}

// Element index held in slot i = q R + r of a thread before stage s (inputs x[j + r n/R]).
template <int N, int E, int S> __device__ __forceinline__ int st_in_index(int lane, int i) {
  constexpr int R = st_radix(N, S, E), nl = N / E, m = N / R;
  return lane + nl * (i / R) + (i % R) * m;
}
// Element index held in slot i after the last stage, when it stays in registers.
template <int N, int E> __device__ __forceinline__ int st_out_index(int lane, int i) {
  constexpr int S = st_nstages(N, E) - 1, R = st_radix(N, S, E), nl = N / E, Ns = st_span(N, S, E);
  // last stage: j < Ns, so j mod Ns = j and the outputs are y[j + r Ns]
  return lane + nl * (i / R) + (i % R) * Ns;
}

// Per-line barrier among the NL threads of a line: inside a warp, over whole warps (a named barrier per line, ids
// 1..15), or, for lines that do not tile warps, the block's barrier (every line of the block then takes part).
template <int NL> struct LineSyncT {
  int id;
  __device__ __forceinline__ void operator()() const {
    if constexpr (NL <= 32 && 32 % NL == 0) __syncwarp();
    else if constexpr (NL % 32 == 0) asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(NL) : "memory");
    else __syncthreads();
  }
};

// Slot of element idx of a line of N.  Powers of two: the low four bits XORed with the next four (a bijection within
// blocks of 16).  Multiples of 12: the low two bits with bits 4-5 (within blocks of 4), which spreads the first
// stage's stride of 12 over all 16 bank pairs.  Other lengths (radix 6 first): plain.
template <int N> struct LineAddr {
  __device__ __forceinline__ int operator()(int idx) const {
    if constexpr (N % 12 == 0) return idx ^ ((idx >> 4) & 3);
    else if constexpr (N % 16 == 0) return idx ^ ((idx >> 4) & 15);
    return idx;
  }
};

// Twiddles in stage order: the stage of span Ns and radix R keeps exp(-2 pi i r k/(Ns R))
// at [(Ns - 1) + (r - 1) Ns + k], r = 1..R-1, k = 0..Ns-1 (N - 1 entries in all, as the
// earlier stages' (R - 1) Ns sum to Ns - 1).  Threads of a line read consecutive k, so the
// reads are free of bank conflicts, unlike the strided r k (N/(Ns R)) reads of one table.
template <int N, int E, typename C>
__device__ __forceinline__ void st_build_twiddles(C* dst, const C* __restrict__ tw_n, int tid, int nthreads) {
  for (int t = tid; t < N - 1; t += nthreads) {
    int Ns = 1, R = st_radix(N, 0, E);
#pragma unroll 1
    for (int s = 0; s < st_nstages(N, E); ++s) {
      R = st_radix(N, s, E);
      if (t < Ns * R - 1) break;
      Ns *= R;
    }
    const int u = t - (Ns - 1), r = u / Ns + 1, k = u - (r - 1) * Ns;
    dst[t] = tw_n[r * k * (N / (Ns * R))];
  }
}

template <int R, int E, int N, int Ns, int SIGN, typename T>
__device__ __forceinline__ void st_butterflies(typename CT<T>::t (&v)[E], int lane,
                                               const typename CT<T>::t* __restrict__ tw) {
  constexpr int B = E / R, nl = N / E;
#pragma unroll
  for (int q = 0; q < B; ++q) {
    if constexpr (Ns > 1) {
      const int k = (lane + nl * q) % Ns;
#pragma unroll
      for (int r = 1; r < R; ++r) v[q * R + r] = tw_apply<SIGN>(v[q * R + r], tw[(Ns - 1) + (r - 1) * Ns + k]);
    }
    dft_r<R, SIGN, T>(&v[q * R]);
  }
}

template <int R, int E, int N, int Ns, typename C, typename Addr>
__device__ __forceinline__ void st_store(const C (&v)[E], C* buf, Addr addr, int lane) {
  constexpr int B = E / R, nl = N / E;
#pragma unroll
  for (int q = 0; q < B; ++q) {
    const int j = lane + nl * q;
    const int k = j % Ns;
    const int d = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) buf[addr(d + r * Ns)] = v[q * R + r];
  }
}

template <int R, int E, int N, typename C, typename Addr>
__device__ __forceinline__ void st_load(C (&v)[E], const C* buf, Addr addr, int lane) {
  constexpr int B = E / R, nl = N / E, m = N / R;
#pragma unroll
  for (int q = 0; q < B; ++q)
#pragma unroll
    for (int r = 0; r < R; ++r) v[q * R + r] = buf[addr(lane + nl * q + r * m)];
}

template <int N, int E, int SIGN, bool FINAL_IN_REGS, int S, bool INPLACE, typename T, typename Addr, typename Sync>
__device__ __forceinline__ typename CT<T>::t* st_run_from(typename CT<T>::t (&v)[E], typename CT<T>::t* cur,
                                                          typename CT<T>::t* nxt, Addr addr, int lane,
                                                          const typename CT<T>::t* __restrict__ tw, Sync sync) {
  constexpr int NST = st_nstages(N, E), R = st_radix(N, S, E), Ns = st_span(N, S, E);
  st_butterflies<R, E, N, Ns, SIGN, T>(v, lane, tw);
  if constexpr (S == NST - 1 && FINAL_IN_REGS) {
    return nullptr;
  } else {
    st_store<R, E, N, Ns>(v, cur, addr, lane);
    sync();
    if constexpr (S == NST - 1) {
      return cur;
    } else {
      st_load<st_radix(N, S + 1, E), E, N>(v, cur, addr, lane);
      if constexpr (INPLACE) sync();   // one buffer: every read of this stage precedes the next writes
      return st_run_from<N, E, SIGN, FINAL_IN_REGS, S + 1, INPLACE, T>(v, nxt, cur, addr, lane, tw, sync);
    }
  }
}

// All stages.  v: the first stage's inputs (slot i = element st_in_index<N,E,0>).
// FINAL_IN_REGS: v ends holding element st_out_index<N,E>(lane, i) in slot i and
// nullptr is returned; otherwise the result is stored in natural order in the
// returned buffer (a or b).  tw: the stage-ordered table built by st_build_twiddles.
// The caller makes sure no thread of the line still reads a or b from earlier use.
template <int N, int E, int SIGN, bool FINAL_IN_REGS, typename T, typename Addr, typename Sync,
          bool INPLACE = false>
__device__ __forceinline__ typename CT<T>::t* st_fft(typename CT<T>::t (&v)[E], typename CT<T>::t* a,
                                                     typename CT<T>::t* b, Addr addr, int lane,
                                                     const typename CT<T>::t* __restrict__ tw, Sync sync) {
  static_assert(st_valid(N, E), "unsupported static FFT shape");
  // lane < N/E: lets the compiler split swizzled addresses into a per-thread base plus constants
  __builtin_assume(lane >= 0 && lane < N / E);
  return st_run_from<N, E, SIGN, FINAL_IN_REGS, 0, INPLACE, T>(v, a, b, addr, lane, tw, sync);
}
// In-place variant: one buffer, two barriers per stage.  The caller makes sure every
// thread has read its first-stage inputs from buf before the first store.
template <int N, int E, int SIGN, bool FINAL_IN_REGS, typename T, typename Addr, typename Sync>
__device__ __forceinline__ typename CT<T>::t* st_fft_inplace(typename CT<T>::t (&v)[E], typename CT<T>::t* buf,
                                                             Addr addr, int lane,
                                                             const typename CT<T>::t* __restrict__ tw, Sync sync) {
  return st_fft<N, E, SIGN, FINAL_IN_REGS, T, Addr, Sync, true>(v, buf, buf, addr, lane, tw, sync);
}

}  // namespace pgb

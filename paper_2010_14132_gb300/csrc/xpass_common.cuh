// Persistent x-pass kernels for FP32 transforms of half lengths 2^a 3^b (the list in PGB_XS_N_SWITCH)
// (Section 2.1: the x transform of every row of every level).
//
// One CTA per SM slot walks groups of RB consecutive rows.  Each group's input
// rows (the field rows for the forward pass, the spectrum rows for the inverse)
// are brought into a ring of shared staging buffers by 1-D bulk copies (TMA)
// completing on an mbarrier, so the loads of the next groups are in flight
// while the current group is transformed.  The FFT runs with the line length
// fixed at compile time (fft_static.cuh) on twiddle tables held in shared memory.
//
//  * forward (R2C): rows packed as n/2 complex points z_m = x_2m + i x_2m+1; after
//    the transform each thread unpacks the pair of bins (k, n/2 - k):
//      X_k = E_k + w^k O_k,   X_{n/2-k} = conj(E_k - w^k O_k),
//    with E_k = (Z_k + conj Z_{n/2-k})/2, O_k = -i (Z_k - conj Z_{n/2-k})/2 and
//    w = exp(-2 pi i/n) (the second form follows from w^{n/2-k} = -conj(w^k)).
//  * inverse (C2R): each first-stage input z_m is formed directly from the staged
//    bins X_m and X_{n/2-m} (self-conjugate bins keep their real parts), the
//    transform's last stage stays in registers, and the epilogue writes the output
//    (and, in the mixed-precision path, the refinement update and norm partial
//    sums) straight from registers.
//
// This header holds what the three kernel files (xpass_fwd.cu, xpass_res.cu,
// xpass_inv.cu) share: the shared-memory layout, the staging-ring bookkeeping,
// the R2C unpacking and the launch configuration.
#pragma once
#include "async_copy.cuh"
#include "fft_static.cuh"
#include "kernel_grants.cuh"
#include "kernels.cuh"
#include "residual2.cuh"

namespace pgb {
namespace {

// Rows per CTA of the residual kernels that stage every stencil row (xpass_res_tile.cu), about 128 threads; lines
// that leave fewer than two (1024 packed points and more) take the kernels that read neighbour rows through L2.
__host__ __device__ constexpr int xrt_rows(int n) { return 128 / (n / st_elems(n)); }
__host__ __device__ constexpr bool xrt_length(int n) { return xrt_rows(n) >= 2; }

// CTA size: at most 256 threads with 8 or 12 elements per thread, 128 with 16 (one warp per
// 512-point line); with 16 elements the FFT runs radix-16 stages.
__host__ __device__ constexpr int xs_max_threads(int E) { return E >= 16 ? 128 : 256; }
// rows per CTA and threads of a CTA for lines of N packed points
__host__ __device__ constexpr int xs_rows(int N, int E) { return xs_max_threads(E) / (N / E); }
__host__ __device__ constexpr int xs_threads(int N, int E) { return xs_rows(N, E) * (N / E); }
constexpr int kXsMaxStages = 4;

template <typename T> struct V2s;
template <> struct V2s<float> { using t = float2; };
template <> struct V2s<double> { using t = double2; };

template <typename TI> __device__ __forceinline__ float to_f(TI x);
template <> __device__ __forceinline__ float to_f<float>(float x) { return x; }
template <> __device__ __forceinline__ float to_f<double>(double x) { return d2f_int(x); }

// Shared layout: twiddles (n/2), unpack twiddles (half a line of them for the forward kernels, a line for the inverse),
// the line buffers that do not fit the staged rows, then the
// staging ring (128-byte aligned) and its mbarriers.  A staged row of nx doubles holds exactly the two n/2-point line
// buffers of its own row (XS_ALIAS_TWO); a row of nx floats, or of n/2 + 1 spectrum bins, holds one of them, the
// one that the second stage writes, when every input has long been read (XS_ALIAS_ONE; lines with a factor 3, whose
// registers allow two CTAs per SM either way, keep both buffers).  What that saves makes room for a fourth
// CTA per SM or a deeper ring (FP32 solve of 256 x 256 x 64: 53.1 -> 50.3 us; forward pass at 1024 x 1024 x 128, 8 elements per
// thread, 232 -> 211).  The mixed path's inverse epilogues are held to three CTAs by their registers and keep both buffers.
enum XsAlias { XS_ALIAS_NONE = 0, XS_ALIAS_ONE = 1, XS_ALIAS_TWO = 2 };
struct XsLayout {
  size_t off_stage, off_bar, total;
};
__host__ __device__ constexpr size_t xs_align(size_t x, size_t a) { return (x + a - 1) / a * a; }
__host__ __device__ constexpr XsAlias xs_alias_float(int E) { return E % 3 == 0 ? XS_ALIAS_NONE : XS_ALIAS_ONE; }
__host__ __device__ inline XsLayout xs_layout(int N, int RB, int ns, unsigned stage_bytes, XsAlias alias, bool inverse) {
  XsLayout L{};
  size_t off = (size_t)N * 8 + (size_t)((inverse ? N : N / 2) + 2) * 8 + (size_t)RB * (2 - (int)alias) * N * 8;
  L.off_stage = xs_align(off, 128);
  L.off_bar = xs_align(L.off_stage + (size_t)ns * stage_bytes, 8);
  L.total = L.off_bar + (size_t)ns * 8;
  return L;
}

// Bounded-wait bookkeeping of the staging ring, kept by the issuing thread.
struct Ring {
  int issued[kXsMaxStages];
  int consumed[kXsMaxStages];
};

__device__ __forceinline__ void ring_drain(Ring& rg, uint64_t* bar, int ns) {
  // let every copy still in flight land before the CTA's shared memory is released
  for (int s = 0; s < ns; ++s)
    for (int c = rg.consumed[s]; c < rg.issued[s]; ++c) mbar_wait_bounded(&bar[s], (unsigned)(c & 1), kWaitPolls);
}

// R2C unpacking of a transformed line (natural order in fin, element i at slot Addr(i)) and store of the
// bins 0..N to dst: each thread takes the bin pairs (k, N - k), k = lane + nl q.
template <int N, int E, typename Addr = LineAddr<N>>
__device__ __forceinline__ void r2c_unpack_store(const float2* fin, const float2* twr_s, float2* dst, int lane,
                                                 bool valid, int kmax = N) {
  using C = float2;
  constexpr int nl = N / E;
  const Addr sw{};
#pragma unroll
  for (int q = 0; q < E / 2; ++q) {
    const int k = lane + nl * q;   // k < N/2
    const C A = fin[sw(k)];
    const C B = cconj(fin[sw(k == 0 ? 0 : N - k)]);
    const C ev = make_float2(0.5f * (A.x + B.x), 0.5f * (A.y + B.y));
    const C dd = make_float2(0.5f * (A.x - B.x), 0.5f * (A.y - B.y));
    const C wo = cmul(twr_s[k], make_float2(dd.y, -dd.x));   // w^k * (-i dd)
    if (valid) {   // bins above kmax are not stored
      if (k <= kmax) dst[k] = cadd(ev, wo);
      if (N - k <= kmax) dst[N - k] = cconj(csub(ev, wo));
    }
  }
  if (lane == 0) {   // the self-paired bin k = N/2
    const C A = fin[sw(N / 2)];
    const C B = cconj(A);
    const C ev = make_float2(0.5f * (A.x + B.x), 0.5f * (A.y + B.y));
    const C dd = make_float2(0.5f * (A.x - B.x), 0.5f * (A.y - B.y));
    const C wo = cmul(twr_s[N / 2], make_float2(dd.y, -dd.x));
    if (valid && N / 2 <= kmax) dst[N / 2] = cadd(ev, wo);
  }
}

// ---------------------------------------------------------------------------
// launch configuration
// ---------------------------------------------------------------------------

struct XsConfig {
  int ns = 0;
  unsigned stage_bytes = 0;
  size_t smem = 0;
};

// Staging depth and CTAs per SM: the most CTAs per SM (up to max_ctas) whose
// shared memory still allows two stages, then the deepest ring (up to four
// stages) at that CTA count.
XsConfig xs_config(int N, int E, unsigned stage_bytes, size_t static_smem, XsAlias alias, bool inverse, int max_ctas) {
  const int RB = xs_rows(N, E);
  constexpr size_t kSmPerSm = 228 * 1024, kReserved = 1024, kMaxPerCta = 227 * 1024;
  XsConfig c{};
  c.stage_bytes = stage_bytes;
  for (int ctas = max_ctas; ctas >= 1 && c.ns == 0; --ctas) {
    size_t budget = kSmPerSm / ctas - kReserved - static_smem;
    if (budget > kMaxPerCta - static_smem) budget = kMaxPerCta - static_smem;
    for (int ns = kXsMaxStages; ns >= 2; --ns)
      if (xs_layout(N, RB, ns, stage_bytes, alias, inverse).total <= budget) {
        c.ns = ns;
        break;
      }
  }
  if (c.ns) c.smem = xs_layout(N, RB, c.ns, stage_bytes, alias, inverse).total;
  return c;
}

template <typename K> cudaError_t prepare(K kernel, int threads, size_t smem, int& grid_cap) {
  int per_sm = 0;
  const cudaError_t e = allow_smem(kernel, smem, threads, &per_sm);
  if (e == cudaSuccess) grid_cap = per_sm * sm_count();
  return e;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Elements per thread of the persistent x-pass for a half length N: kE3 when N has
// a factor 3 (radix 12 first), else the plan's 8 or 16.
inline int xs_elems(int N, int plan_e) { return N % 3 == 0 ? st_elems(N) : (plan_e == 16 ? 16 : 8); }
// ... of the FP32 transforms without the mixed path's conversions and epilogues, where no option chose it: 16 from 256
// points on for the forward pass and from 512 on for the inverse one, whose registers then fit three CTAs per SM.  256
// points take two stages (16 16) instead of three, 512 as many, with one warp per line instead of two and no barrier
// between warps.  FP32 1024 x 1024 x 64 492 us with 8 in both, 483 with 16 in the forward pass, 476 in both;
// 512 x 512 x 64 139 with 8, 136 with 16 in the forward pass, 139 in both; 256 x 256 x 64 (128 points) 47.9 and 51.8.
// Up to 4096 lines a pass leaves warp slots empty, and what counts is the time of one line, which twice the threads
// shorten: solves with 8 and with 16 take 41.3 and 46.5 us at 4096 x 64 x 8 (512 lines), 36.5 and 38.2 at 2048 x 128 x 8,
// 36.6 and 39.2 at 1024 x 64 x 32 (2048 lines), 34.3 and 35.5 at 512 x 128 x 32 (4096), but 133.4 and 126.1 at
// 2048 x 256 x 32, 46.4 and 45.0 at 512 x 256 x 32 (8192).  The lines of all levels count, so that chunks of them round
// alike.
inline int xs_elems_fp32(const FftPlan& fx, const Geom& g, bool inverse) {
  const bool more = !fx.e_set && fx.n % 3 != 0 && fx.n >= (inverse ? 512 : 256) && (long long)g.ny * g.nz > 4096;
  return more ? 16 : xs_elems(fx.n, fx.E);
}

// Dispatch to the compile-time (N, E) instance; shapes the engine cannot take are
// never instantiated (and are not reported supported).
#define PGB_XS_E_SWITCH(E, ...)                                 \
  if ((E) == kE3) {                                             \
    constexpr int EE = kE3;                                     \
    __VA_ARGS__;                                                \
  } else if ((E) == kE3Odd) {                                   \
    constexpr int EE = kE3Odd;                                  \
    __VA_ARGS__;                                                \
  } else if ((E) == 16) {                                       \
    constexpr int EE = 16;                                      \
    __VA_ARGS__;                                                \
  } else {                                                      \
    constexpr int EE = 8;                                       \
    __VA_ARGS__;                                                \
  }
#define PGB_XS_N_CASE(V, ...) \
  case V: { constexpr int NN = V; if constexpr (st_valid(NN, EE)) { __VA_ARGS__; } } break;
// Half lengths with compile-time kernels.  The ones with factors 9, 27 and 81 ran the run-time engine (24 elements
// and 190 registers a thread, index arithmetic by division): 432 x 324 x 37 in FP32 145 -> 77 us (x 42 -> 22, inverse
// x 40 -> 22, the y-pass of 324 points 24 -> 17), 70 with radix 12.  The short ones (16 to 54) ran it as well, one CTA
// per row group: FP32 32 x 32 x 32 38 -> 27 us, mixed 181 -> 123; FP32 96 x 768 x 101 237 -> 122, 108 with radix 12.
#define PGB_XS_N_SWITCH(N, ...)                          \
  switch (N) {                                           \
    PGB_XS_N_CASE(16, __VA_ARGS__)                       \
    PGB_XS_N_CASE(18, __VA_ARGS__)                       \
    PGB_XS_N_CASE(24, __VA_ARGS__)                       \
    PGB_XS_N_CASE(32, __VA_ARGS__)                       \
    PGB_XS_N_CASE(36, __VA_ARGS__)                       \
    PGB_XS_N_CASE(48, __VA_ARGS__)                       \
    PGB_XS_N_CASE(54, __VA_ARGS__)                       \
    PGB_XS_N_CASE(64, __VA_ARGS__)                       \
    PGB_XS_N_CASE(72, __VA_ARGS__)                       \
    PGB_XS_N_CASE(96, __VA_ARGS__)                       \
    PGB_XS_N_CASE(108, __VA_ARGS__)                      \
    PGB_XS_N_CASE(128, __VA_ARGS__)                      \
    PGB_XS_N_CASE(144, __VA_ARGS__)                      \
    PGB_XS_N_CASE(192, __VA_ARGS__)                      \
    PGB_XS_N_CASE(216, __VA_ARGS__)                      \
    PGB_XS_N_CASE(256, __VA_ARGS__)                      \
    PGB_XS_N_CASE(288, __VA_ARGS__)                      \
    PGB_XS_N_CASE(324, __VA_ARGS__)                      \
    PGB_XS_N_CASE(384, __VA_ARGS__)                      \
    PGB_XS_N_CASE(432, __VA_ARGS__)                      \
    PGB_XS_N_CASE(512, __VA_ARGS__)                      \
    PGB_XS_N_CASE(768, __VA_ARGS__)                      \
    PGB_XS_N_CASE(1024, __VA_ARGS__)                     \
    PGB_XS_N_CASE(2048, __VA_ARGS__)                     \
    default: return cudaSuccess;                         \
  }

// Launch one persistent x-pass kernel: grid = min(groups, resident CTAs).
template <typename K, typename... Args>
cudaError_t xs_launch(K kern, int threads_x, int RB, const XsConfig& c, long long ngroups, int* nblocks_out,
                      cudaStream_t st, bool* used, Args... args) {
  int cap = 0;
  cudaError_t e = prepare(kern, threads_x * RB, c.smem, cap);
  if (e != cudaSuccess) return e;
  if (cap <= 0) return cudaSuccess;
  const long long grid = ngroups < cap ? ngroups : cap;
  if (grid <= 0) return cudaSuccess;
  if (nblocks_out) *nblocks_out = (int)grid;
  *used = true;
  return pdl_launch(kern, dim3((unsigned)grid), dim3(threads_x, RB), c.smem, st, args..., c.ns, c.stage_bytes);
}

}  // namespace
}  // namespace pgb

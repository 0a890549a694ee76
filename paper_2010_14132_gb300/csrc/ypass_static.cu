// Persistent FP32 y-pass for ny = 2^a 3^b in [32, 2048] (the list in PGB_YS_N_SWITCH; Section 2.1: the
// transform along y of every kx column of every level).
//
// A tile is one level and TK consecutive kx columns: ny rows of TK complex
// values, brought into shared memory by 2-D TMA boxes (columns past nx/2 read
// as zeros).  A CTA walks tiles with a ring of two tile buffers, so the next
// tile loads while the current one is transformed.  The transform is the
// compile-time Stockham engine (fft_static.cuh) on the TK interleaved columns:
// its first stage reads the TMA tile, the stages alternate between a scratch
// tile and the (by then consumed) input tile in a swizzled layout, and the last
// stage's outputs go from registers straight to global memory (each warp writes
// row segments of TK contiguous values).

#include "async_copy.cuh"
#include "fft_static.cuh"
#include "kernel_grants.cuh"
#include "kernels.cuh"

namespace pgb {

namespace {

// Column-interleaved tile addressing with the complex index swizzled inside
// blocks of 16 (spreads the stride-R first-stage writes over the banks).
template <int N> struct SwStrided {
  int es;
  __device__ __forceinline__ int operator()(int idx) const { return LineAddr<N>{}(idx) * es; }
};
// ... and with 32 elements per thread: the first stage's stride of 32 keeps the parity, which decides the half of the
// banks that a row of 8 columns takes, so it is swapped in every other block of 32 (written so that each unrolled
// access is one of two bases plus a constant)
struct SwPair {
  int es;
  __device__ __forceinline__ int operator()(int idx) const {
    const int s = (idx >> 5) & 1;
    return ((idx & 1) ? idx - s : idx + s) * es;
  }
};
template <int N, int E> struct SwOf { using t = SwStrided<N>; };
template <int N> struct SwOf<N, 32> { using t = SwPair; };
struct Plain {
  int es;
  __device__ __forceinline__ int operator()(int idx) const { return idx * es; }
};

size_t ys_tile_bytes(int N, int TK) { return ((size_t)N * TK * sizeof(float2) + 127) / 128 * 128; }
size_t ys_smem(int N, int TK, bool inplace) {
  return (inplace ? 2 : 3) * ys_tile_bytes(N, TK) + (size_t)N * sizeof(float2) + 64;
}

constexpr int ys_max_threads(int E) { return E >= 16 || E % 3 == 0 ? 512 : 1024; }
// the single-buffered kernel runs two CTAs per SM: 256 threads for the 12-element lengths keeps
// their registers (128) free of spills (288 for 864 points, whose 72 threads a column would leave only two
// columns otherwise)
constexpr int ys1_max_threads(int N, int E) { return E == 32 ? 256 : E % 3 == 0 ? (N == 864 ? 288 : 256) : ys_max_threads(E); }

template <int N, int E, int SIGN, bool INPLACE>
__global__ void __launch_bounds__(ys_max_threads(E)) k_ys(const __grid_constant__ CUtensorMap tm, Geom g,
                                            const float2* __restrict__ twy, float2* __restrict__ spec, int box_rows,
                                            int tiles_per_level, int ntiles, const int* __restrict__ done,
                                            unsigned* __restrict__ err) {
  using C = float2;
  constexpr int nl = N / E;
  pdl_trigger();
  extern __shared__ __align__(128) unsigned char smraw[];
  const int TK = blockDim.x, l = threadIdx.x, lane = threadIdx.y;
  const int tid = lane * TK + l, nthreads = TK * nl;
  const size_t tb = ((size_t)N * TK * sizeof(C) + 127) / 128 * 128;
  constexpr int NT = INPLACE ? 2 : 3;   // tile buffers: the TMA ring (+ a scratch tile)
  C* ring[2] = {reinterpret_cast<C*>(smraw), reinterpret_cast<C*>(smraw + tb)};
  C* scratch = reinterpret_cast<C*>(smraw + 2 * tb);
  C* tw_s = reinterpret_cast<C*>(smraw + NT * tb);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smraw + NT * tb + (size_t)N * sizeof(C));
  const unsigned tile_bytes = (unsigned)((size_t)N * TK * sizeof(C));
  st_build_twiddles<N, E>(tw_s, twy, tid, nthreads);
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  __syncthreads();
  pdl_wait();   // the previous kernels of the stream are complete
  if (done && *done) return;
  int issued[2] = {0, 0}, consumed[2] = {0, 0};
  auto issue = [&](int t, int b) {
    const int level = t / tiles_per_level, kx0 = (t - level * tiles_per_level) * TK;
    mbar_arrive_expect_tx(&bar[b], tile_bytes);
    for (int r0 = 0; r0 < N; r0 += box_rows) tma_load_2d(ring[b] + (size_t)r0 * TK, &tm, kx0, level * N + r0, &bar[b]);
    issued[b]++;
  };
  const int t0 = g.lev0 * tiles_per_level + blockIdx.x;
  if (tid == 0) {
    if (t0 < ntiles) issue(t0, 0);
    if (t0 + (int)gridDim.x < ntiles) issue(t0 + gridDim.x, 1);
  }
  const SwStrided<N> sw{TK};
  bool ok = true;
  int it = 0;
  for (int t = t0; t < ntiles; t += gridDim.x, ++it) {
    const int b = it & 1;
    const bool got = mbar_wait_bounded(&bar[b], (unsigned)((it >> 1) & 1), kWaitPolls);
    if (!__syncthreads_and(got)) {
      ok = false;
      break;
    }
    if (tid == 0) {
      consumed[b]++;
      // every thread is past the previous tile: its buffer takes the tile after this one
      const int tn = t + gridDim.x;
      if (it > 0 && tn < ntiles) {
        fence_proxy_async_smem();
        issue(tn, b ^ 1);
      }
    }
    C* in = ring[b];
    C v[E];
#pragma unroll
    for (int i = 0; i < E; ++i) v[i] = in[Plain{TK}(st_in_index<N, E, 0>(lane, i)) + l];
    if constexpr (INPLACE) {
      __syncthreads();   // every thread has its inputs before the tile is overwritten
      st_fft_inplace<N, E, SIGN, true, float>(v, in + l, sw, lane, tw_s, SyncBlock());
    } else {
      st_fft<N, E, SIGN, true, float>(v, scratch + l, in + l, sw, lane, tw_s, SyncBlock());
    }
    (void)scratch;
    const int level = t / tiles_per_level, kx = (t - level * tiles_per_level) * TK + l;
    if (kx < g.nxh) {
      C* col = spec + (long long)level * g.plane + kx;
#pragma unroll
      for (int i = 0; i < E; ++i) col[(long long)st_out_index<N, E>(lane, i) * g.P] = v[i];
    }
    fence_proxy_async_smem();   // generic writes to the ring buffer come before its refill by TMA
  }
  if (tid == 0) {
    if (!ok) atomicOr(err, (unsigned)ERR_WAIT_TIMEOUT);
    for (int b = 0; b < 2; ++b)
      for (int c = consumed[b]; c < issued[b]; ++c) mbar_wait_bounded(&bar[b], (unsigned)(c & 1), kWaitPolls);
  }
}


// Single-buffered variant: one tile per CTA, transformed in place, two CTAs per
// SM (registers capped for it), so one CTA's load overlaps the other's transform.
// The next tile's load is issued as soon as the transform has finished reading the
// tile (its outputs are in registers), so it also overlaps this tile's stores.
template <int N, int E, int SIGN>
__global__ void __launch_bounds__(ys1_max_threads(N, E), 2) k_ys1(const __grid_constant__ CUtensorMap tm, Geom g,
                                                             const float2* __restrict__ twy,
                                                             float2* __restrict__ spec, int box_rows,
                                                             int tiles_per_level, int ntiles,
                                                             const int* __restrict__ done, unsigned* __restrict__ err) {
  using C = float2;
  constexpr int nl = N / E;
  pdl_trigger();
  extern __shared__ __align__(128) unsigned char smraw[];
  const int TK = blockDim.x, l = threadIdx.x, lane = threadIdx.y;
  const int tid = lane * TK + l, nthreads = TK * nl;
  const size_t tb = ((size_t)N * TK * sizeof(C) + 127) / 128 * 128;
  C* tile = reinterpret_cast<C*>(smraw);
  C* tw_s = reinterpret_cast<C*>(smraw + tb);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smraw + tb + (size_t)N * sizeof(C));
  const unsigned tile_bytes = (unsigned)((size_t)N * TK * sizeof(C));
  st_build_twiddles<N, E>(tw_s, twy, tid, nthreads);
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  pdl_wait();   // the previous kernels of the stream are complete
  if (done && *done) return;
  const typename SwOf<N, E>::t sw{TK};
  int it = 0, pending = 0;
  bool ok = true;
  auto issue = [&](int tt) {
    const int lv = tt / tiles_per_level, k0 = (tt - lv * tiles_per_level) * TK;
    mbar_arrive_expect_tx(bar, tile_bytes);
    for (int r0 = 0; r0 < N; r0 += box_rows) tma_load_2d(tile + (size_t)r0 * TK, &tm, k0, lv * N + r0, bar);
    pending = 1;
  };
  int t = g.lev0 * tiles_per_level + blockIdx.x;
  if (tid == 0 && t < ntiles) issue(t);
  for (; t < ntiles; t += gridDim.x, ++it) {
    const int level = t / tiles_per_level, kx0 = (t - level * tiles_per_level) * TK;
    const bool got = mbar_wait_bounded(bar, (unsigned)(it & 1), kWaitPolls);
    if (!__syncthreads_and(got)) {
      ok = false;
      break;
    }
    pending = 0;
    C v[E];
#pragma unroll
    for (int i = 0; i < E; ++i) v[i] = tile[Plain{TK}(st_in_index<N, E, 0>(lane, i)) + l];
    __syncthreads();   // every thread has its inputs before the tile is overwritten
    st_fft_inplace<N, E, SIGN, true, float>(v, tile + l, sw, lane, tw_s, SyncBlock());
    // The in-place transform ends on a barrier after its last reads of the tile, and its outputs are in
    // registers: refill the tile with the next one while this one is stored.
    fence_proxy_async_smem();   // generic writes to the tile come before its refill by TMA
    __syncthreads();
    if (tid == 0 && t + (int)gridDim.x < ntiles) issue(t + gridDim.x);
    const int kx = kx0 + l;
    if (kx < g.nxh) {
      C* col = spec + (long long)level * g.plane + kx;
#pragma unroll
      for (int i = 0; i < E; ++i) col[(long long)st_out_index<N, E>(lane, i) * g.P] = v[i];
    }
  }
  if (tid == 0) {
    if (!ok) atomicOr(err, (unsigned)ERR_WAIT_TIMEOUT);
    if (pending) mbar_wait_bounded(bar, (unsigned)(it & 1), kWaitPolls);   // let a copy in flight land
  }
}

int largest_divisor_upto(int n, int cap) {
  for (int d = cap; d >= 1; --d)
    if (n % d == 0) return d;
  return 1;
}

#define PGB_YS_N_CASE(V, ...) \
  case V: { constexpr int NN = V; if constexpr (st_valid(NN, E)) { __VA_ARGS__; } } break;
#define PGB_YS_N_SWITCH(N, ...)        \
  switch (N) {                         \
    PGB_YS_N_CASE(32, __VA_ARGS__)     \
    PGB_YS_N_CASE(36, __VA_ARGS__)     \
    PGB_YS_N_CASE(48, __VA_ARGS__)     \
    PGB_YS_N_CASE(54, __VA_ARGS__)     \
    PGB_YS_N_CASE(64, __VA_ARGS__)     \
    PGB_YS_N_CASE(72, __VA_ARGS__)     \
    PGB_YS_N_CASE(96, __VA_ARGS__)     \
    PGB_YS_N_CASE(108, __VA_ARGS__)    \
    PGB_YS_N_CASE(128, __VA_ARGS__)    \
    PGB_YS_N_CASE(144, __VA_ARGS__)    \
    PGB_YS_N_CASE(192, __VA_ARGS__)    \
    PGB_YS_N_CASE(216, __VA_ARGS__)    \
    PGB_YS_N_CASE(256, __VA_ARGS__)    \
    PGB_YS_N_CASE(288, __VA_ARGS__)    \
    PGB_YS_N_CASE(324, __VA_ARGS__)    \
    PGB_YS_N_CASE(384, __VA_ARGS__)    \
    PGB_YS_N_CASE(432, __VA_ARGS__)    \
    PGB_YS_N_CASE(512, __VA_ARGS__)    \
    PGB_YS_N_CASE(576, __VA_ARGS__)    \
    PGB_YS_N_CASE(768, __VA_ARGS__)    \
    PGB_YS_N_CASE(864, __VA_ARGS__)    \
    PGB_YS_N_CASE(1024, __VA_ARGS__)   \
    PGB_YS_N_CASE(1536, __VA_ARGS__)   \
    PGB_YS_N_CASE(2048, __VA_ARGS__)   \
    default: return cudaSuccess;       \
  }

template <int E, int SIGN, bool INPLACE>
cudaError_t ys_launch(float2* spec, const Geom& g, int N, const float2* twy, int tk, const int* done, unsigned* err,
                      cudaStream_t st, bool* used) {
  const size_t smem = ys_smem(N, tk, INPLACE);
  const int nthreads = tk * (N / E);
  if (smem > 220 * 1024 || nthreads > ys_max_threads(E) || nthreads < 32) return cudaSuccess;
  const int box_rows = largest_divisor_upto(N, 256);
  if (((size_t)box_rows * tk * sizeof(float2)) % 128 != 0 && box_rows != N) return cudaSuccess;
  CUtensorMap tm;
  if (!encode_tensor_2d(&tm, spec, 8, (unsigned long long)g.nxh, (unsigned long long)g.ny * g.nz,
                        (unsigned long long)g.P * sizeof(float2), (unsigned)tk, (unsigned)box_rows))
    return cudaSuccess;
  const int tiles_per_level = (g.nxh + tk - 1) / tk;
  const int ntiles = tiles_per_level * g.lev1;
  const int chunk_tiles = tiles_per_level * (g.lev1 - g.lev0);
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = cudaSuccess;
  PGB_YS_N_SWITCH(N, {
    auto kern = k_ys<NN, E, SIGN, INPLACE>;
    int per_sm = 0;
    e = allow_smem(kern, smem, nthreads, &per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaSuccess;
    const int grid = chunk_tiles < sms * per_sm ? chunk_tiles : sms * per_sm;
    if (grid <= 0) return cudaSuccess;
    e = pdl_launch(kern, dim3(grid), dim3(tk, N / E), smem, st, tm, g, twy, spec, box_rows, tiles_per_level, ntiles,
                   done, err);
    if (e != cudaSuccess) return e;
    *used = true;
  });
  return cudaGetLastError();
}


template <int E, int SIGN>
cudaError_t ys1_launch(float2* spec, const Geom& g, int N, const float2* twy, int tk, const int* done, unsigned* err,
                       cudaStream_t st, bool* used) {
  const size_t smem = ys_tile_bytes(N, tk) + (size_t)N * sizeof(float2) + 64;
  const int nthreads = tk * (N / E);
  if (smem > 110 * 1024 || nthreads > ys1_max_threads(N, E) || nthreads < 32) return cudaSuccess;
  const int box_rows = largest_divisor_upto(N, 256);
  if (((size_t)box_rows * tk * sizeof(float2)) % 128 != 0 && box_rows != N) return cudaSuccess;
  CUtensorMap tm;
  if (!encode_tensor_2d(&tm, spec, 8, (unsigned long long)g.nxh, (unsigned long long)g.ny * g.nz,
                        (unsigned long long)g.P * sizeof(float2), (unsigned)tk, (unsigned)box_rows))
    return cudaSuccess;
  const int tiles_per_level = (g.nxh + tk - 1) / tk;
  const int ntiles = tiles_per_level * g.lev1;
  const int chunk_tiles = tiles_per_level * (g.lev1 - g.lev0);
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = cudaSuccess;
  PGB_YS_N_SWITCH(N, {
    auto kern = k_ys1<NN, E, SIGN>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nthreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaSuccess;
    const int grid = chunk_tiles < sms * per_sm ? chunk_tiles : sms * per_sm;
    if (grid <= 0) return cudaSuccess;
    e = pdl_launch(kern, dim3(grid), dim3(tk, N / E), smem, st, tm, g, twy, spec, box_rows, tiles_per_level, ntiles,
                   done, err);
    if (e != cudaSuccess) return e;
    *used = true;
  });
  return cudaGetLastError();
}

}  // namespace

bool ypass_static_supported(int ny) {
  switch (ny) {
    case 32: case 64: case 128: case 256: case 512: case 1024: case 2048:
    case 36: case 48: case 54: case 72: case 96: case 108: case 144: case 192: case 216: case 288: case 324: case 384: case 432: case 576: case 768:
    case 864: case 1536:
      return true;
    default: return false;
  }
}

cudaError_t launch_yfft_static(int sign, void* spec, const Geom& g, const FftPlan& fy, const Tables& tb, int tile,
                               int variant, const int* done, unsigned* err, cudaStream_t st, bool* used) {
  *used = false;
  if (!ypass_static_supported(fy.n)) return cudaSuccess;
  int tk = tile > 0 ? tile : 8;   // 64-byte TMA box rows (measured best untuned at 1024^2 and on small domains)
  if (tk % 2) tk += 1;   // 16-byte inner TMA box
  // when ny has a factor 3, 12 elements per thread (radix 12 first) or 6
  const int E = fy.n % 3 == 0 ? st_elems(fy.n) : (fy.E == 16 ? 16 : 8);
  // 512 = 32 16 and 1024 = 32 32: with 32 elements per thread these two lengths take two stages instead of three, one
  // exchange through shared memory and two barriers less, which is what the pass waits for (one tile per CTA: load,
  // stages and stores follow each other).  1024 x 1024 x 128: 225 -> 181 us a pass (cold; 4.8 -> 5.9 TB/s); 512 x 512 x 64:
  // 31 -> 24.7.  128 registers, no spills, two CTAs of 256 threads at 1024 and four of 128 at 512.  256 points are two
  // stages with 16 elements already, 2048 three with either.  512 points with no more tiles than SMs keep 16: one tile is
  // all an SM then has to do, and twice the threads shorten it by more than the stage saved (FP32 solves with 32 and 16:
  // 64 x 512 x 8, 40 tiles, 29.7 and 27.7 us; 128 x 512 x 16, 144, 33.1 and 31.4; 64 x 512 x 32, 160, 36.8 and 36.5;
  // 1024 x 512 x 3, 195, 36.0 and 36.5; 128 x 512 x 24, 216, 35.0 and 37.1), where 1024 points gain with any number.  The
  // tiles of all levels count, so that chunks of them round alike.
  if (variant == 2 && E == 16 && !fy.e_set && (fy.n == 512 || fy.n == 1024)) {
    int tk1 = tk;
    while (tk1 > 2 && tk1 * (fy.n / 32) > ys1_max_threads(fy.n, 32)) tk1 >>= 1;
    if (fy.n == 1024 || (long long)((g.nxh + tk1 - 1) / tk1) * g.nz > sm_count()) {
      float2* sp = (float2*)spec;
      const cudaError_t e = sign < 0 ? ys1_launch<32, -1>(sp, g, fy.n, tb.twy_f, tk1, done, err, st, used)
                                     : ys1_launch<32, +1>(sp, g, fy.n, tb.twy_f, tk1, done, err, st, used);
      if (e != cudaSuccess || *used) return e;
    }
  }
  if (variant == 2 && E != 8) {   // single-buffered, in place, two CTAs per SM
    int tk1 = tk;
    if (tile <= 0 && tk1 * (fy.n / E) < 32) tk1 = 16;   // a warp at least
    while (tk1 > 2 && tk1 * (fy.n / E) > ys1_max_threads(fy.n, E)) tk1 >>= 1;
    float2* sp = (float2*)spec;
    cudaError_t e;
    if (E == kE3Odd)
      e = sign < 0 ? ys1_launch<kE3Odd, -1>(sp, g, fy.n, tb.twy_f, tk1, done, err, st, used)
                   : ys1_launch<kE3Odd, +1>(sp, g, fy.n, tb.twy_f, tk1, done, err, st, used);
    else if (E == 16)
      e = sign < 0 ? ys1_launch<16, -1>(sp, g, fy.n, tb.twy_f, tk1, done, err, st, used)
                   : ys1_launch<16, +1>(sp, g, fy.n, tb.twy_f, tk1, done, err, st, used);
    else
      e = sign < 0 ? ys1_launch<kE3, -1>(sp, g, fy.n, tb.twy_f, tk1, done, err, st, used)
                   : ys1_launch<kE3, +1>(sp, g, fy.n, tb.twy_f, tk1, done, err, st, used);
    if (e != cudaSuccess || *used) return e;
  }
  const bool inplace = variant == 1;
  while (tk > 2 && (ys_smem(fy.n, tk, inplace) > 220 * 1024 || tk * (fy.n / E) > ys_max_threads(E))) tk >>= 1;
  float2* sp = (float2*)spec;
#define PGB_YS_CALL(EE, SG)                                                                   \
  return inplace ? ys_launch<EE, SG, true>(sp, g, fy.n, tb.twy_f, tk, done, err, st, used)    \
                 : ys_launch<EE, SG, false>(sp, g, fy.n, tb.twy_f, tk, done, err, st, used)
  if (E == kE3Odd) return cudaSuccess;   // that form only
  if (E == kE3) {
    if (sign < 0) PGB_YS_CALL(kE3, -1);
    PGB_YS_CALL(kE3, +1);
  }
  if (E == 16) {
    if (sign < 0) PGB_YS_CALL(16, -1);
    PGB_YS_CALL(16, +1);
  }
  if (sign < 0) PGB_YS_CALL(8, -1);
  PGB_YS_CALL(8, +1);
#undef PGB_YS_CALL
}

}  // namespace pgb

// Small rules shared by the kernels and their launchers that need no CUDA header: a plain C++ compiler takes this file
// too, so that they are tested on the host.
#pragma once

#ifdef __CUDACC__
#define PGB_HD __host__ __device__ __forceinline__
#else
#define PGB_HD inline
#endif

namespace pgb {

// Threads that thread t's warp holds in a block of n: column CTAs take 16 columns where the levels leave room for no
// more, and a shuffle or a warp barrier may name existing lanes only.
PGB_HD int warp_lanes(int t, int n) {
  const int rest = n - (t & ~31);
  return rest < 32 ? rest : 32;
}
PGB_HD unsigned warp_mask(int t, int n) {
  const int lanes = warp_lanes(t, n);
  return lanes == 32 ? 0xffffffffu : (1u << lanes) - 1u;
}

}  // namespace pgb

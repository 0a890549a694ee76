// Small rules shared by the kernels and their launchers that need no CUDA header: a plain C++ compiler takes this file
// too, so that they are tested on the host.
#pragma once

#include <cstddef>
#include <functional>
#include <mutex>
#include <unordered_map>

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

// Blocks of one launch of the tiled residual pass: all groups of rows that are resident at once, up to the slots for
// their sums.  The launches of a pass's level chunks use the same slots, one after the other (each chunk's blocks in
// slots of its own left the last chunks one block: 256 x 256 x 48 in chunks of five levels 635 -> 2247 us).
inline int tile_pass_blocks(long long groups, int resident, int slots) {
  const int n = groups < resident ? (int)groups : resident;
  return n < slots ? n : slots;
}
// Slots that a launch of n blocks adds to those in use.
inline int added_slots(int in_use, int n) { return n > in_use ? n - in_use : 0; }

// FP64 column kernel: values a lane carries, of a pair of columns (4), one column (2) or one real or imaginary part (1),
// for 19, 13 or 10 FP64 instructions per level of every warp (16 lanes of columns, both halves) that one of the FP64 units,
// four an SM, has to run; the least of the three (128 x 128 x 64 on 608 units: one column, 97 -> 77 us for the solve).
inline int fp64_column_values(long long pairs, long long cols, int sms) {
  const long long units = sms > 0 ? 4ll * sms : 1;
  auto cost = [units](long long lanes, int per_level) { return ((lanes + 15) / 16 + units - 1) / units * per_level; };
  const long long c4 = cost(pairs, 19), c2 = cost(cols, 13), c1 = cost(2 * cols, 10);
  return c4 <= c2 && c4 <= c1 ? 4 : (c2 <= c1 ? 2 : 1);
}

// What the kernels have been granted, for all devices of the process: a kernel's shared memory limit is an attribute of
// the kernel on one device, and its CTAs per SM depend on the device and on the shared memory it is launched with.
class KernelGrants {
 public:
  // CTAs per SM of (device, kernel, smem) in *per_sm (0 if threads is 0: not asked for).  allow(smem) raises the limit,
  // called where the device's is lower; occupancy(per_sm) is called once per entry.  Both return 0 or an error, passed on.
  template <typename Allow, typename Occupancy>
  int get(int device, const void* kernel, size_t smem, int threads, Allow allow, Occupancy occupancy, int* per_sm) {
    std::lock_guard<std::mutex> lock(mu_);
    size_t& limit = limit_[{device, kernel, 0}];
    if (limit < smem) {
      if (const int e = allow(smem)) return e;
      limit = smem;
    }
    *per_sm = 0;
    if (threads <= 0) return 0;
    int& n = ctas_[{device, kernel, smem}];
    if (n == 0)
      if (const int e = occupancy(&n)) return e;
    *per_sm = n;
    return 0;
  }

 private:
  struct Key {
    int device;
    const void* kernel;
    size_t smem;
    bool operator==(const Key& o) const { return device == o.device && kernel == o.kernel && smem == o.smem; }
  };
  struct Hash {
    size_t operator()(const Key& k) const {
      return std::hash<const void*>()(k.kernel) * 31 + k.smem * 131 + (size_t)k.device;
    }
  };
  std::mutex mu_;
  std::unordered_map<Key, size_t, Hash> limit_;
  std::unordered_map<Key, int, Hash> ctas_;
};

}  // namespace pgb

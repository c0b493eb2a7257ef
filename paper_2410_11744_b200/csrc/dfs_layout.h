// Shared-memory layout of the depth-first renumbering (dfs_reorder.cu): plain C++, so that the host can size a launch and
// a test can check the sizes without a GPU.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define DYSPEC_HOST_DEVICE __host__ __device__
#else
#define DYSPEC_HOST_DEVICE
#endif

namespace dyspec {

// Splitters among E tour elements.
constexpr uint32_t kSpread = 2654435769u;          // odd
constexpr uint32_t spread_inverse() {              // modulo 2^32, hence modulo every smaller power of two (Newton)
  uint32_t x = kSpread;
  for (int k = 0; k < 5; ++k) x *= 2u - kSpread * x;
  return x;
}
constexpr uint32_t kSpreadInverse = spread_inverse();
static_assert(kSpread * kSpreadInverse == 1u, "inverse");
struct Splitters {
  uint32_t mask;                                   // a power of two - 1, at least E - 1
  int count;                                       // numbers 0 .. count - 1 (some stand for no element)
  int exist;                                       // at least as many as stand for one: 7 E / 32, which the multiplier misses by little
  DYSPEC_HOST_DEVICE explicit Splitters(int E) : mask(31u) {
#ifdef __CUDA_ARCH__
    mask |= 0xFFFFFFFFu >> __clz(E - 1 | 1);
#else
    while (mask < uint32_t(E - 1)) mask = 2u * mask + 1u;
#endif
    count = 7 * int((mask + 1u) >> 5);
    exist = 7 * E / 32 + 6;
  }
  DYSPEC_HOST_DEVICE int number(uint32_t e) const { return int((e * kSpread) & mask); }        // a splitter if < count
  DYSPEC_HOST_DEVICE uint32_t element(int k) const { return (uint32_t(k) * kSpreadInverse) & mask; }
};

constexpr int kJumpAll = 256;                      // nodes up to which all elements jump

// Shared memory of a tree of n nodes (byte offsets).  A launch is sized by its largest tree and every CTA lays out its own, so
// `bytes` must not fall when n grows.
struct DfsLayout {
  int par, fc, ns, chunks, table, next, at, jump, bytes;
  DYSPEC_HOST_DEVICE explicit DfsLayout(int n) {
    const int n16 = (n + 1 + 31) & ~31;
    par = 0;
    fc = par + 2 * n16;
    ns = fc + 2 * n16;
    chunks = ns + 2 * n16;
    table = chunks + 8 * n16;
    next = table;                                  // the table of step 1 is dead when the tour is written
    at = next + 4 * n16;
    jump = n <= kJumpAll ? table : at + 8 * n16;
    const int lists = jump + 8 * (n <= kJumpAll ? 2 * n : Splitters(2 * n).count), tabled = table + (n + 1) * ((n + 31) >> 5);
    bytes = lists > tabled ? lists : tabled;
  }
};

}  // namespace dyspec

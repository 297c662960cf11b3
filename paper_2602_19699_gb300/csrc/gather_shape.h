// Launch shape of the gather kernel (api.cu), kept apart from CUDA so that the
// rule can be compiled and checked on its own.
#pragma once
#include <algorithm>

namespace to {

struct GatherShape {
  unsigned gx, gy;   // grid: stretches of an instance's elements, instances
  bool wide;         // 64-bit element indices
};

constexpr int kGatherThreads = 256;

// elements of an instance's longest output: X and Vx (T_max + 1) n, U T_max m
// (m <= n), K T_max m n
inline long long gather_elems(int T_max, int n, int m, bool K) {
  const long long x = ((long long)T_max + 1) * n;
  return K ? std::max(x, (long long)T_max * m * n) : x;
}

// Four elements a thread.  A thread's index runs past the last element by less
// than a grid's stretch, a quarter of the elements and one block, so 32 bits
// hold it up to 2^30 elements; the divisions by n and m cost several times more
// in 64.
inline GatherShape gather_shape(int B, long long elems) {
  GatherShape s;
  s.gx = (unsigned)std::max(1LL, (elems + 4 * kGatherThreads - 1) / (4 * kGatherThreads));
  s.gy = (unsigned)std::min(B, 65535);
  s.wide = elems > (1LL << 30);
  return s;
}

}  // namespace to

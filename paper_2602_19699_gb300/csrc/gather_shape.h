// Launch shape of the gather kernel (api.cu), kept apart from CUDA so that the
// rule can be compiled and checked on its own.
#pragma once
#include <algorithm>

namespace to {

struct GatherShape {
  unsigned bx, by;   // a block: threads across an instance's elements, instances
  unsigned gx, gy;   // grid: stretches of an instance's elements, sets of instances
  bool wide;         // 64-bit element indices
};

constexpr int kGatherThreads = 256;

// elements of an instance's longest output: X and Vx (T_max + 1) n, U T_max m
// (m <= n), K T_max m n
inline long long gather_elems(int T_max, int n, int m, bool K) {
  const long long x = ((long long)T_max + 1) * n;
  return K ? std::max(x, (long long)T_max * m * n) : x;
}

// A thread takes four to eight elements of one instance, so that its reads of
// the horizon, offset and slot are shared and its loads overlap; an instance of
// fewer than 1024 elements leaves room in the block for others.  Batches that do
// not fill the GPU that way (kGatherFill threads) spread an instance further, up
// to an element a thread: there a thread's own chain is what counts.
//
// A thread's index runs past the last element by less than a grid's stretch, a
// quarter of the elements and one block, so 32 bits hold it up to 2^30 elements;
// the divisions by n and m cost several times more in 64.
constexpr long long kGatherFill = 128 * 1024;

inline GatherShape gather_shape(int B, long long elems) {
  GatherShape s;
  s.bx = 8;
  while (s.bx < kGatherThreads && (8LL * s.bx <= elems || (s.bx < elems && (long long)B * s.bx < kGatherFill))) s.bx *= 2;
  s.by = kGatherThreads / s.bx;
  s.gx = (unsigned)std::max(1LL, s.bx < kGatherThreads ? 1 : (elems + 4 * kGatherThreads - 1) / (4 * kGatherThreads));
  s.gy = (unsigned)std::min<long long>(((long long)B + s.by - 1) / s.by, 65535);
  s.wide = elems > (1LL << 30);
  return s;
}

}  // namespace to

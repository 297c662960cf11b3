// Biased-initial-condition ranking (Sec. III-C/D): the std-critic network
// scores 10N candidate initial states and the N with the largest predicted
// critic standard deviation start the next TO batch (include/to.h:
// toranker_create, torank_candidates).
//
// Network: x (n_in) -> 256 tanh -> 256 tanh -> 1 softplus (a positive std), in
// float32 with every sum taken in index order.  The 256 x 256 layer is the
// work (10.7 of 11 GFLOP for 81 920 candidates): a CTA of 256 threads holds
// 8 Q candidates' activations in shared memory and streams the layer's weights
// through it in slices of 32 inputs; a thread accumulates 8 units x Q
// candidates in registers.  Selection: a radix select of the scores' bit
// patterns (positive floats order like their bits) by one cluster of 8 CTAs
// that keep the keys in shared memory, then a compaction in index order (ties
// at the threshold go to the lowest indices).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "handles.h"

namespace {

constexpr int kH = 256;        // hidden width
constexpr int kMaxIn = 64;     // largest input width
constexpr int kSlice = 32;     // inputs per staged slice of the weights

__device__ __forceinline__ float softplus_(float z) { return z > 0.f ? z + log1pf(expf(-z)) : log1pf(expf(z)); }

// 16-byte asynchronous copies of n4 float4 from global to shared memory
__device__ __forceinline__ void stage(float* dst, const float* src, int n4) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  for (int i = threadIdx.x; i < n4; i += kH)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16u * i), "l"(src + 4 * (size_t)i) : "memory");
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// The candidates of a tile: thread group cg (0..7) owns columns 32 j + 4 cg ..
// + 3 for j < Q / 4, then, where Q is not a multiple of 4, the two columns
// 8 (Q & ~3) + 2 cg, + 1.
template <int Q>
__device__ __forceinline__ int cand_col(int cg, int q) {
  return q < (Q & ~3) ? (q >> 2) * 32 + cg * 4 + (q & 3) : (Q & ~3) * 8 + cg * 2 + (q & 1);
}

template <int Q>
__device__ __forceinline__ void load_row(const float* row, int cg, float (&v)[Q]) {
#pragma unroll
  for (int j = 0; j < Q / 4; ++j) {
    const float4 t = *reinterpret_cast<const float4*>(row + 32 * j + 4 * cg);
    v[4 * j] = t.x; v[4 * j + 1] = t.y; v[4 * j + 2] = t.z; v[4 * j + 3] = t.w;
  }
  if constexpr (Q & 2) {
    const float2 t = *reinterpret_cast<const float2*>(row + (Q & ~3) * 8 + 2 * cg);
    v[Q - 2] = t.x; v[Q - 1] = t.y;
  }
}

// acc[u][q] += w[k][unit u] * v[k][candidate q] for k = 0 .. n-1 in order.  A
// thread's units are 4 ug .. + 3 and 128 + 4 ug .. + 3, so that the 8 groups of
// a quarter warp read 128 consecutive bytes.
template <int Q>
__device__ __forceinline__ void accumulate(float (&acc)[8][Q], const float* w, const float* v, int stride, int n, int ug,
                                           int cg) {
#pragma unroll 2
  for (int k = 0; k < n; ++k) {
    const float4 w0 = *reinterpret_cast<const float4*>(w + k * kH + 4 * ug);
    const float4 w1 = *reinterpret_cast<const float4*>(w + k * kH + 128 + 4 * ug);
    float x[Q];
    load_row<Q>(v + k * stride, cg, x);
    const float wu[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int q = 0; q < Q; ++q) acc[u][q] += wu[u] * x[q];
  }
}

template <int Q>
__device__ __forceinline__ void store_tanh(const float (&acc)[8][Q], float* h, int stride, int ug, int cg) {
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    float* row = h + (u < 4 ? 4 * ug + u : 124 + 4 * ug + u) * stride;
#pragma unroll
    for (int j = 0; j < Q / 4; ++j)
      *reinterpret_cast<float4*>(row + 32 * j + 4 * cg) =
          make_float4(tanhf(acc[u][4 * j]), tanhf(acc[u][4 * j + 1]), tanhf(acc[u][4 * j + 2]), tanhf(acc[u][4 * j + 3]));
    if constexpr (Q & 2)
      *reinterpret_cast<float2*>(row + (Q & ~3) * 8 + 2 * cg) = make_float2(tanhf(acc[u][Q - 2]), tanhf(acc[u][Q - 1]));
  }
}

// row stride of the activations: 4 words past the candidates, so that the 8
// units a quarter warp stores lie in different banks
template <int Q> constexpr int kStride = 8 * Q + 4;
template <int Q> constexpr size_t kRankSmem = sizeof(float) * ((size_t)kH * kStride<Q> + 2 * (size_t)kSlice * kH);

// One tile of 8 Q candidates.  What bounds it: at Q = 16 a warp reads 6 16-byte
// vectors for 128 multiply-adds (24 cycles of the shared-memory port against
// 32 of the SM's FMA pipes), where a tile of 1 unit x 64 candidates reads 16 for
// 64 and the port holds it at 19 % of the FMA rate.  81 920 candidates of 6 inputs:
// 249 us (647 with that tile), 55 % of the FP32 rate; the selection 26 us (87 by
// one CTA), the copies 28, the whole call 345 (755).  The rest of the kernel's time
// is 2 warps a scheduler with nothing to run while all of them evaluate tanh, wait
// for a slice or sum the output layer.
template <int Q>
__global__ void __launch_bounds__(kH, 1) std_critic_kernel(int C, int n_in, const double* __restrict__ x,
                                                            const float* __restrict__ w, float* __restrict__ score,
                                                            unsigned* __restrict__ key) {
  extern __shared__ __align__(16) float sm[];
  constexpr int S = kStride<Q>, NC = 8 * Q;
  float* h = sm;                       // [kH][S]: x (transposed), then layer 1's, then layer 2's activations
  float* ws = sm + kH * S;             // two slices of [kSlice][kH] weights
  const float* W1 = w;                 // [n_in][kH], input-major
  const float* b1 = W1 + n_in * kH;
  const float* W2 = b1 + kH;           // [kH][kH]
  const float* b2 = W2 + kH * kH;
  const float* W3 = b2 + kH;           // [kH]
  const float* b3 = W3 + kH;
  const int c0 = blockIdx.x * NC;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int ug = (warp & 3) * 8 + (lane & 7), cg = (warp >> 2) * 4 + (lane >> 3);
  stage(ws, W1, n_in * kH / 4);        // n_in <= 64 rows fill at most both slices
  for (int e = t; e < NC * n_in; e += kH) {
    const int c = e / n_in, i = e - c * n_in;
    h[i * S + c] = c0 + c < C ? (float)x[(size_t)(c0 + c) * n_in + i] : 0.f;
  }
  float acc[8][Q];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const float b = b1[u < 4 ? 4 * ug + u : 124 + 4 * ug + u];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[u][q] = b;
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  accumulate<Q>(acc, ws, h, S, n_in, ug, cg);
  __syncthreads();                     // every thread has read x and W1
  stage(ws, W2, kSlice * kH / 4);
  store_tanh<Q>(acc, h, S, ug, cg);
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const float b = b2[u < 4 ? 4 * ug + u : 124 + 4 * ug + u];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[u][q] = b;
  }
  for (int s = 0; s < kH / kSlice; ++s) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();                   // slice s is there; the other buffer (slice s - 1) is read
    if (s + 1 < kH / kSlice) stage(ws + ((s + 1) & 1) * kSlice * kH, W2 + (size_t)(s + 1) * kSlice * kH, kSlice * kH / 4);
    accumulate<Q>(acc, ws + (s & 1) * kSlice * kH, h + s * kSlice * S, S, kSlice, ug, cg);
  }
  __syncthreads();                     // every thread has read layer 1's activations
  store_tanh<Q>(acc, h, S, ug, cg);
  __syncthreads();
  // output
  if (t < NC && c0 + t < C) {
    float s = b3[0];
#pragma unroll 16
    for (int i = 0; i < kH; ++i) s += W3[i] * h[i * S + t];
    const float sd = softplus_(s);
    score[c0 + t] = sd;
    // positive floats order like their bit patterns; a non-finite score ranks last
    key[c0 + t] = (isfinite(sd) && sd > 0.f) ? __float_as_uint(sd) : 0u;
  }
}

template <int Q>
cudaError_t launch_std_critic(int C, int n_in, const double* x, const float* w, float* score, unsigned* key, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(std_critic_kernel<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRankSmem<Q>);
  if (e != cudaSuccess) return e;
  std_critic_kernel<Q><<<(C + 8 * Q - 1) / (8 * Q), kH, kRankSmem<Q>, s>>>(C, n_in, x, w, score, key);
  return cudaGetLastError();
}

// Candidates per thread.  A tile occupies an SM, so the time is the number of
// rounds of tiles over the SMs times a tile's, which goes like Q + 2 (the
// weight reads and the staging count for about two candidates).
int pick_q(int C, int sms) {
  int best = 16;
  long long cost = -1;
  for (int q : {16, 14, 12, 8, 4, 2}) {
    const long long tiles = (C + 8LL * q - 1) / (8 * q), c = ((tiles + sms - 1) / sms) * (q + 2);
    if (cost < 0 || c < cost) { cost = c; best = q; }
  }
  return best;
}

// Radix select of the N largest keys and their compaction in index order, by
// one cluster of kSelCtas CTAs.  CTA r owns the r-th contiguous range of the
// keys and (up to kSelCached of them) keeps it in shared memory; each of the
// three digits is a histogram per CTA, summed through distributed shared
// memory by every CTA.  One CTA that read the keys from memory five times was
// latency-bound: 87 us of 745 us for 81 920 candidates.
constexpr int kSelCtas = 8, kSelThreads = 1024, kSelCached = 48 * 1024, kSelBins = 2048;

// inclusive scan over the CTA's threads; *total the sum
__device__ __forceinline__ int block_scan(int v, int* part, int* total) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  __syncthreads();                     // part may still be read from the previous scan
  if (lane == 31) part[warp] = v;
  __syncthreads();
  if (warp == 0) {
    int s = part[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += u;
    }
    part[lane] = s;
  }
  __syncthreads();
  *total = part[31];
  return v + (warp ? part[warp - 1] : 0);
}

__global__ void __cluster_dims__(kSelCtas, 1, 1) __launch_bounds__(kSelThreads)
    select_kernel(int C, int N, const unsigned* __restrict__ key, int* __restrict__ out) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned keys[];     // this CTA's keys, where they fit
  __shared__ int hist[kSelBins];
  __shared__ int part[32];
  __shared__ int s_digit, s_above, s_gt, s_eq;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, rank = (int)cl.block_rank();
  const int per = ((C + kSelCtas - 1) / kSelCtas + 31) / 32 * 32;
  const int lo = (int)min((long long)C, (long long)rank * per), hi = (int)min((long long)C, (long long)lo + per);
  const bool cached = per <= kSelCached;
  if (cached)
    for (int i = lo + t; i < hi; i += kSelThreads) keys[i - lo] = key[i];
  auto at = [&](int i) { return cached ? keys[i - lo] : key[i]; };
  unsigned prefix = 0u, mask = 0u;
  int remaining = N;
  for (int pass = 0; pass < 3; ++pass) {
    const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0, bits = pass == 2 ? 10 : 11;
    for (int b = t; b < kSelBins; b += kSelThreads) hist[b] = 0;
    __syncthreads();
    for (int i = lo + t; i < hi; i += kSelThreads) {
      const unsigned k = at(i);
      if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & ((1u << bits) - 1u)], 1);
    }
    cl.sync();
    // this thread's two bins, from the largest digit down, over the cluster
    const int b0 = kSelBins - 1 - 2 * t;
    int n0 = 0, n1 = 0;
    for (int r = 0; r < kSelCtas; ++r) {
      const int* hr = cl.map_shared_rank(hist, r);
      n0 += hr[b0];
      n1 += hr[b0 - 1];
    }
    int total = 0;
    const int incl = block_scan(n0 + n1, part, &total), above = incl - n0 - n1;
    // the digit at which the count from above reaches what remains
    if (above < remaining && remaining <= above + n0) { s_digit = b0; s_above = above; }
    else if (above + n0 < remaining && remaining <= incl) { s_digit = b0 - 1; s_above = above + n0; }
    cl.sync();                         // the digit is known; no CTA reads this pass's histograms any more
    prefix |= (unsigned)s_digit << shift;
    mask |= ((1u << bits) - 1u) << shift;
    remaining -= s_above;
  }
  const unsigned thr = prefix;         // the N-th largest key
  const int need_eq = remaining;       // how many keys equal to it are taken
  // each warp's contiguous part of the range keeps index order
  const int seg = per / 32, rounds = (seg + 31) / 32;
  const int wlo = min(hi, lo + warp * seg), whi = min(hi, wlo + seg);
  int gt = 0, eq = 0;
  for (int i = wlo + lane; i < whi; i += 32) {
    const unsigned k = at(i);
    gt += k > thr;
    eq += k == thr;
  }
  int n_gt = 0, n_eq = 0;
  const int gt_i = block_scan(gt, part, &n_gt), eq_i = block_scan(eq, part, &n_eq);
  if (t == 0) { s_gt = n_gt; s_eq = n_eq; }
  cl.sync();
  int gt_before = 0, eq_before = 0;    // in the CTAs before this one
  for (int r = 0; r < rank; ++r) {
    gt_before += *cl.map_shared_rank(&s_gt, r);
    eq_before += *cl.map_shared_rank(&s_eq, r);
  }
  gt_before += __shfl_sync(0xffffffffu, gt_i - gt, 0);   // and in the warps before this one
  eq_before += __shfl_sync(0xffffffffu, eq_i - eq, 0);
  for (int r = 0; r < rounds; ++r) {
    const int i = wlo + r * 32 + lane;
    const unsigned k = i < whi ? at(i) : 0u;
    const bool g = i < whi && k > thr, e = i < whi && k == thr;
    const unsigned mg = __ballot_sync(0xffffffffu, g), me = __ballot_sync(0xffffffffu, e), below = (1u << lane) - 1u;
    const int eb = eq_before + __popc(me & below);
    if (g || (e && eb < need_eq)) out[gt_before + __popc(mg & below) + min(eb, need_eq)] = i;
    gt_before += __popc(mg);
    eq_before += __popc(me);
  }
  cl.sync();                           // no CTA leaves while its shared memory is read
}

}  // namespace

struct to_ranker_s {
  int n_in = 0;
  float* d_w = nullptr;
  double* d_x = nullptr;
  float* d_score = nullptr;
  unsigned* d_key = nullptr;
  int* d_out = nullptr;
  int cap_c = 0, cap_n = 0;
  int launches = 0;
};

#define RK_CK(x)                                                                                \
  do {                                                                                          \
    cudaError_t e_ = (x);                                                                       \
    if (e_ != cudaSuccess) return to_fail(TO_ERR_CUDA, std::string(#x) + ": " + cudaGetErrorString(e_)); \
  } while (0)

int toranker_create(int n_in, const float* weights, size_t n_weights, to_ranker* out) {
  if (!out || !weights || n_in < 1 || n_in > kMaxIn) return to_fail(TO_ERR_ARG, "toranker_create: bad arguments (1 <= n_in <= 64)");
  *out = nullptr;
  const size_t expect = (size_t)kH * n_in + kH + (size_t)kH * kH + kH + kH + 1;
  if (n_weights != expect) return to_fail(TO_ERR_ARG, "toranker_create: weights must be W1[256 x n_in] b1 W2[256 x 256] b2 W3[1 x 256] b3");
  // every W (out x in, row-major) stored transposed (input-major)
  std::vector<float> t(expect);
  size_t o = 0;
  auto transpose = [&](int rows, int cols) {
    for (int i = 0; i < cols; ++i)
      for (int r = 0; r < rows; ++r) t[o + (size_t)i * rows + r] = weights[o + (size_t)r * cols + i];
    o += (size_t)rows * cols;
  };
  auto copy = [&](int k) {
    std::memcpy(t.data() + o, weights + o, sizeof(float) * k);
    o += k;
  };
  transpose(kH, n_in); copy(kH); transpose(kH, kH); copy(kH); copy(kH); copy(1);
  to_ranker r = new to_ranker_s();
  r->n_in = n_in;
  cudaError_t e = cudaMalloc(&r->d_w, expect * sizeof(float));
  if (e == cudaSuccess) e = cudaMemcpy(r->d_w, t.data(), expect * sizeof(float), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    toranker_destroy(r);
    return to_fail(TO_ERR_CUDA, std::string("toranker_create: ") + cudaGetErrorString(e));
  }
  *out = r;
  return TO_OK;
}

void toranker_destroy(to_ranker r) {
  if (!r) return;
  void* p[] = {r->d_w, r->d_x, r->d_score, r->d_key, r->d_out};
  for (void* q : p)
    if (q) cudaFree(q);
  delete r;
}

int torank_candidates(to_ranker r, int C, const double* x, int N, int* top_idx, float* scores, void* cuda_stream) {
  if (!r || !x || !top_idx || C < 1 || N < 1 || N > C) return to_fail(TO_ERR_ARG, "torank_candidates: bad arguments (1 <= N <= C)");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  if (C > r->cap_c) {
    r->cap_c = 0;                      // (an allocation that fails leaves no capacity behind)
    for (void* q : {(void*)r->d_x, (void*)r->d_score, (void*)r->d_key})
      if (q) cudaFree(q);
    r->d_x = nullptr; r->d_score = nullptr; r->d_key = nullptr;
    RK_CK(cudaMalloc(&r->d_x, sizeof(double) * (size_t)C * r->n_in));
    RK_CK(cudaMalloc(&r->d_score, sizeof(float) * C));
    RK_CK(cudaMalloc(&r->d_key, sizeof(unsigned) * C));
    r->cap_c = C;
  }
  if (N > r->cap_n) {
    r->cap_n = 0;
    if (r->d_out) cudaFree(r->d_out);
    r->d_out = nullptr;
    RK_CK(cudaMalloc(&r->d_out, sizeof(int) * N));
    r->cap_n = N;
  }
  RK_CK(cudaMemcpyAsync(r->d_x, x, sizeof(double) * (size_t)C * r->n_in, cudaMemcpyHostToDevice, s));
  int dev = 0, sms = 0;
  RK_CK(cudaGetDevice(&dev));
  RK_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  switch (pick_q(C, sms)) {
    case 16: RK_CK(launch_std_critic<16>(C, r->n_in, r->d_x, r->d_w, r->d_score, r->d_key, s)); break;
    case 14: RK_CK(launch_std_critic<14>(C, r->n_in, r->d_x, r->d_w, r->d_score, r->d_key, s)); break;
    case 12: RK_CK(launch_std_critic<12>(C, r->n_in, r->d_x, r->d_w, r->d_score, r->d_key, s)); break;
    case 8: RK_CK(launch_std_critic<8>(C, r->n_in, r->d_x, r->d_w, r->d_score, r->d_key, s)); break;
    case 4: RK_CK(launch_std_critic<4>(C, r->n_in, r->d_x, r->d_w, r->d_score, r->d_key, s)); break;
    default: RK_CK(launch_std_critic<2>(C, r->n_in, r->d_x, r->d_w, r->d_score, r->d_key, s));
  }
  const int per = ((C + kSelCtas - 1) / kSelCtas + 31) / 32 * 32;
  const size_t smem = per <= kSelCached ? sizeof(unsigned) * (size_t)per : 0;
  RK_CK(cudaFuncSetAttribute(select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(unsigned) * kSelCached)));
  select_kernel<<<kSelCtas, kSelThreads, smem, s>>>(C, N, r->d_key, r->d_out);
  RK_CK(cudaGetLastError());
  r->launches = 2;
  RK_CK(cudaMemcpyAsync(top_idx, r->d_out, sizeof(int) * N, cudaMemcpyDeviceToHost, s));
  if (scores) RK_CK(cudaMemcpyAsync(scores, r->d_score, sizeof(float) * C, cudaMemcpyDeviceToHost, s));
  RK_CK(cudaStreamSynchronize(s));
  return TO_OK;
}

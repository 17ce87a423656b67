// Log-sum-exp combine of split-KV decode partials.
//
// A branch's decode is split into runs of pages (shared-prefix runs read for
// the whole fork group, and the branch's own runs); each run yields a
// normalised partial O_i with its log-sum-exp lse_i.  Since softmax over the
// union of disjoint key sets is the lse-weighted mixture of the per-set
// softmaxes, lse = log sum_i exp(lse_i) and O = sum_i exp(lse_i - lse) O_i.
#include <math.h>

#include <type_traits>

#include "kernels.cuh"

namespace st {

namespace {

// kWarps warps per row (one layer, branch and query head): lse = log sum_i
// exp(lse_i), O = sum_i exp(lse_i - lse) O_i over the row's ns partials
// (ns <= 32).  Every warp has all the lse values (one per lane) and takes the
// partials [8 w, 8 w + 8), [8 w + 8 kWarps, ...), eight loads in flight; with
// more than one warp their sums meet in shared memory.  One warp moves the
// least for many rows; a launch of few rows is a chain of round trips to L2,
// which four warps make in one (a single agent's step, 28 partials on each of
// 160 rows: from the wait for the decode to the last write 3.1 us with one warp
// and 16 loads in flight, 1.3 with four).  All index arithmetic comes ahead of that wait, in 32 bits.
constexpr int kBatch = 8;
constexpr int kFewRows = 152 * 16;  // rows of a small launch: one block each on the 152 SMs of this part

template <int D, int kWarps>
__global__ void __launch_bounds__(128) combine_kernel(const CombineParams p, const __grid_constant__ InlineSplits inl) {
  constexpr int kPer = D / 32;
  using Vec = std::conditional_t<kPer == 4, float4, float2>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = kWarps == 1 ? blockIdx.x * 4 + warp : blockIdx.x;
  const int part = kWarps == 1 ? 0 : warp;  // this warp's share of the partials
  const bool live = row < p.n_rows;
  const int b = (row / p.Hq) % p.n_br;
  const float* lse_i = p.part_lse + (int64_t)row * p.max_splits;
  const Vec* po = reinterpret_cast<const Vec*>(p.part_o + (int64_t)row * p.max_splits * D) + lane;
  griddep_wait();
  griddep_launch_dependents();
  if (kWarps == 1 && !live) return;
  const int ns = p.n_splits ? p.n_splits[b] : inl.n_splits[b];
  // the first partials are loaded together with the lse values: the loads do
  // not depend on the weights
  auto load = [&](int i, float* x) {
    if (i < ns) {
      const Vec v = __ldcg(po + i * 32);
#pragma unroll
      for (int e = 0; e < kPer; ++e) x[e] = reinterpret_cast<const float*>(&v)[e];
    } else {
#pragma unroll
      for (int e = 0; e < kPer; ++e) x[e] = 0.f;
    }
  };
  const float li = lane < ns ? __ldcg(lse_i + lane) : -INFINITY;
  float x[kBatch][kPer];
#pragma unroll
  for (int u = 0; u < kBatch; ++u) load(part * kBatch + u, x[u]);
  float mx = li;
#pragma unroll
  for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  float w = lane < ns ? expf(li - mx) : 0.f;
  float sum = w;
#pragma unroll
  for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  w *= 1.f / sum;
  float out[kPer];
#pragma unroll
  for (int e = 0; e < kPer; ++e) out[e] = 0.f;
#pragma unroll 1
  for (int i0 = part * kBatch; i0 < ns; i0 += kWarps * kBatch) {
    if (i0 != part * kBatch) {
#pragma unroll
      for (int u = 0; u < kBatch; ++u) load(i0 + u, x[u]);
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const float wv = __shfl_sync(0xffffffffu, w, (i0 + u) & 31);  // 0 past the row's partials
#pragma unroll
      for (int e = 0; e < kPer; ++e) out[e] += wv * x[u][e];
    }
  }
  if constexpr (kWarps > 1) {
    __shared__ Vec sums[kWarps][32];
    Vec v;
#pragma unroll
    for (int e = 0; e < kPer; ++e) reinterpret_cast<float*>(&v)[e] = out[e];
    sums[warp][lane] = v;
    __syncthreads();
    if (warp != 0) return;
#pragma unroll
    for (int k = 1; k < kWarps; ++k) {
      const Vec o = sums[k][lane];
#pragma unroll
      for (int e = 0; e < kPer; ++e) out[e] += reinterpret_cast<const float*>(&o)[e];
    }
  }
  Vec v;
#pragma unroll
  for (int e = 0; e < kPer; ++e) reinterpret_cast<float*>(&v)[e] = out[e];
  reinterpret_cast<Vec*>(p.o + (int64_t)row * D)[lane] = v;
  if (lane == 0) p.lse[row] = mx + logf(sum);
}

}  // namespace

cudaError_t launch_combine(const CombineParams& p, const InlineSplits* inl, int D, cudaStream_t s) {
  static const InlineSplits kNone{};
  const InlineSplits& ip = inl ? *inl : kNone;
  if (p.n_rows == 0) return cudaSuccess;
  // four warps per row while every row's block is resident at once (a block is
  // 128 threads, of which an SM holds 16): fewer round trips; beyond, one warp
  // per row
  const bool wide = p.n_rows <= kFewRows;
  const dim3 grid(wide ? p.n_rows : (p.n_rows + 3) / 4);
  if (D == 128)
    return wide ? launch_chained(combine_kernel<128, 4>, grid, dim3(128), 0, s, p, ip)
                : launch_chained(combine_kernel<128, 1>, grid, dim3(128), 0, s, p, ip);
  if (D == 64)
    return wide ? launch_chained(combine_kernel<64, 4>, grid, dim3(128), 0, s, p, ip)
                : launch_chained(combine_kernel<64, 1>, grid, dim3(128), 0, s, p, ip);
  return cudaErrorInvalidValue;
}

}  // namespace st

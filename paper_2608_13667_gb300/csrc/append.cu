// Block-table refresh and the KV append (scatter + copy-on-write).
//
// The host owns the allocator; the device keeps a copy of every live block
// table.  An append call refreshes the table entries the host changed (in its
// own launch where it is small, else by table_update ahead of it), performs the
// call's copy-on-write page copies and writes its new rows.  A copy fills rows
// [0, off) of a fresh page whose own rows start at row off, so the two need no
// ordering in one launch, except where rows go in place over what is copied
// (below).
#include "kernels.cuh"

namespace st {

namespace {

// runs and values are in the pinned staging slot and read from there: a copy
// to the device first is an operation of another engine, whose hand-overs
// break the chain of dependent launches (with its 2 MiB slot copied whole it
// took 12 us; the update itself takes 2).  A block's loads are in flight
// together, since each is a round trip to the host's memory.
// A run has at most kTableChunk entries (the host cuts longer ranges), one block's
// work: blocks for every run by the longest one's length were nearly all empty
// where one long table was refreshed with thousands of short ones (a table of 8192
// entries beside 4000 of 2: 87 us ahead of a decode, 93 in an append, with this 62
// and 56; 65536 beside 2000: 178 and 59).
__device__ __forceinline__ void table_run(int32_t* __restrict__ table, const TableRun* __restrict__ runs,
                                          const int32_t* __restrict__ values, int r) {
  const TableRun run = runs[r];
  const int i0 = threadIdx.x;
  int32_t v[kTableChunk / kTableThreads];
#pragma unroll
  for (int u = 0; u < kTableChunk / kTableThreads; ++u)
    if (i0 + u * kTableThreads < run.count) v[u] = values[run.src + i0 + u * kTableThreads];
#pragma unroll
  for (int u = 0; u < kTableChunk / kTableThreads; ++u)
    if (i0 + u * kTableThreads < run.count) table[run.dst + i0 + u * kTableThreads] = v[u];
}

__global__ void __launch_bounds__(kTableThreads)
    table_update_kernel(int32_t* __restrict__ table, const TableRun* __restrict__ runs,
                        const int32_t* __restrict__ values) {
  griddep_wait();
  griddep_launch_dependents();
  table_run(table, runs, values, blockIdx.x);
}

// A plan from its pinned staging slot to the device, 16 bytes a thread.  A
// kernel rather than a copy, so that it is one of the chain of dependent
// launches.
__global__ void __launch_bounds__(256) plan_copy_kernel(uint4* __restrict__ dst, const uint4* __restrict__ src, int n) {
  griddep_wait();
  griddep_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = src[i];
}

// One thread moves 16 bytes (8 bf16).  Index space: copy-on-write chunks
// first (n_cow x L x Hkv x 16 rows x D/8, rows past the copy length idle),
// then the appended rows in the input's own order [L][n_rows][Hkv][D/8];
// row r belongs to the branch whose [row0, row0 + n) holds it.  Copies and rows of
// a launch touch different rows of the pool; where a call's would not (the last
// holder of a page, forked from inside it, writes in place over rows that others
// copy), the host launches the copies first and the rows behind them.  A small append
// that also changes the tables (new pages, or a fork's whole table) refreshes
// them in its first blocks and takes its rows' pages from the parameters, one
// launch and one hand-over less in the chain to the attention kernel (a merge
// of 44 rows onto 23040, fork, merge and release: 49.3 us with the refresh in a
// launch of its own, 47.5 without; a prompt of 17 rows 22.2 and 19.4).
template <int D>
__global__ void __launch_bounds__(kTableThreads) append_kernel(const AppendParams p,
                                                     const __grid_constant__ InlineAppendPlan inl) {
  griddep_wait();
  griddep_launch_dependents();
  if ((int)blockIdx.x < p.n_table_blocks) {
    table_run(p.table_out, p.runs, p.values, blockIdx.x);
    return;
  }
  const AppendBranch* branches = p.branches ? p.branches : inl.branches;
  const CowCopy* cows = p.cows ? p.cows : inl.cows;
  constexpr int kChunks = D / 8;
  const int64_t cow_total = (int64_t)p.n_cow * p.L * p.Hkv * kPageTokens * kChunks;
  const int64_t app_total = (int64_t)p.L * p.n_rows * p.Hkv * kChunks;
  const int64_t total = cow_total + app_total;
  const int64_t stride = (int64_t)(gridDim.x - p.n_table_blocks) * blockDim.x;
  for (int64_t i = (int64_t)(blockIdx.x - p.n_table_blocks) * blockDim.x + threadIdx.x; i < total; i += stride) {
    if (i < cow_total) {
      int64_t x = i;
      const int c = (int)(x % kChunks); x /= kChunks;
      const int row = (int)(x % kPageTokens); x /= kPageTokens;
      const int g = (int)(x % p.Hkv); x /= p.Hkv;
      const int l = (int)(x % p.L); x /= p.L;
      const CowCopy cw = cows[x];
      if (row >= cw.rows) continue;
      if ((uint64_t)cw.src_block >= (uint64_t)p.n_blocks ||
          (uint64_t)cw.dst_block >= (uint64_t)p.n_blocks) {
        atomicCAS(p.status, 0, kDevBadIndex);
        continue;
      }
      const int64_t src = ((((int64_t)l * p.n_blocks + cw.src_block) * p.Hkv + g) * kPageTokens + row) * D + c * 8;
      const int64_t dst = ((((int64_t)l * p.n_blocks + cw.dst_block) * p.Hkv + g) * kPageTokens + row) * D + c * 8;
      *reinterpret_cast<uint4*>(p.k_pool + dst) = *reinterpret_cast<const uint4*>(p.k_pool + src);
      *reinterpret_cast<uint4*>(p.v_pool + dst) = *reinterpret_cast<const uint4*>(p.v_pool + src);
    } else {
      const int64_t j = i - cow_total;
      int64_t x = j;
      const int c = (int)(x % kChunks); x /= kChunks;
      const int g = (int)(x % p.Hkv); x /= p.Hkv;
      const int row = (int)(x % p.n_rows); x /= p.n_rows;
      const int l = (int)x;
      int b;
      if (p.ragged) {  // the last branch whose first row is <= row
        int lo = 0, hi = p.n_br - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (branches[mid].row0 <= row) lo = mid;
          else hi = mid - 1;
        }
        b = lo;
      } else {
        b = row / p.n_tok;
      }
      const AppendBranch br = branches[b];
      const int pos = br.start + (row - br.row0);
      const int32_t blk = p.n_table_blocks ? inl.pages[inl.page0[b] + pos / kPageTokens - br.start / kPageTokens]
                                           : p.table[(int64_t)br.slot * p.max_pages + pos / kPageTokens];
      if ((uint64_t)blk >= (uint64_t)p.n_blocks) {
        atomicCAS(p.status, 0, kDevBadIndex);
        continue;
      }
      const int64_t dst = ((((int64_t)l * p.n_blocks + blk) * p.Hkv + g) * kPageTokens + (pos % kPageTokens)) * D + c * 8;
      *reinterpret_cast<uint4*>(p.k_pool + dst) = *reinterpret_cast<const uint4*>(p.k + j * 8);
      *reinterpret_cast<uint4*>(p.v_pool + dst) = *reinterpret_cast<const uint4*>(p.v + j * 8);
    }
  }
}

int grid_for(int64_t total, int threads) {
  static int sms_of[64] = {};
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64) {
    if (!sms_of[dev]) cudaDeviceGetAttribute(&sms_of[dev], cudaDevAttrMultiProcessorCount, dev);
    if (sms_of[dev] > 0) sms = sms_of[dev];
  }
  const int64_t want = (total + threads - 1) / threads;
  const int64_t cap = (int64_t)sms * 16;
  return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

}  // namespace

cudaError_t launch_table_update(int32_t* table, const TableRun* runs, const int32_t* values, int n_runs,
                                cudaStream_t s) {
  if (n_runs <= 0) return cudaSuccess;
  return launch_chained(table_update_kernel, dim3(n_runs), dim3(kTableThreads), 0, s, table, runs, values);
}

cudaError_t launch_plan_copy(void* dst, const void* src, size_t bytes, cudaStream_t s) {
  const int n = (int)((bytes + 15) / 16);
  return launch_chained(plan_copy_kernel, dim3((n + 255) / 256), dim3(256), 0, s, static_cast<uint4*>(dst),
                        static_cast<const uint4*>(src), n);
}

cudaError_t launch_append(const AppendParams& p, const InlineAppendPlan* inl, int D, cudaStream_t s) {
  static const InlineAppendPlan kNone{};
  const InlineAppendPlan& ip = inl ? *inl : kNone;
  const int64_t total = (int64_t)p.n_cow * p.L * p.Hkv * kPageTokens * (D / 8) +
                        (int64_t)p.L * p.n_rows * p.Hkv * (D / 8);
  if (total == 0) return cudaSuccess;
  const int grid = grid_for(total, kTableThreads) + p.n_table_blocks;
  if (D == 128) return launch_chained(append_kernel<128>, dim3(grid), dim3(kTableThreads), 0, s, p, ip);
  if (D == 64) return launch_chained(append_kernel<64>, dim3(grid), dim3(kTableThreads), 0, s, p, ip);
  return cudaErrorInvalidValue;
}

}  // namespace st

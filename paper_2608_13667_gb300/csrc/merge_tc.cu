// Merge prefill on the tcgen05 tensor cores: two 128-row query tiles per CTA
// that share every K/V stage (one CTA per SM), the stages of a row tile split
// over a cluster of CTAs where a launch has few row tiles.
//
// Section 3.5 of the paper: the harvested thoughts are appended after main's
// context and read in order, so thought row i of a merge of T rows attends
// to main's keys [0, L0 + i].  The (thought row, query head) pairs of one KV
// head are stacked G per token; a CTA takes 256 consecutive stacked rows as
// tile A (the first 128) and tile B (the next 128) and walks main's pages up
// to the causal limit of its last row, 128 keys per stage.  Both tiles read
// each K/V stage from shared memory.  A batched prefill (several sequences'
// new rows in one launch) gives each CTA its own (sequence, L0, T, row tile)
// through a work list.
//
// Few rows.  A turn's thoughts are a few dozen rows onto a long context: in
// one layer that is a row tile or three per KV head, 8 to 24 CTAs on 152 SMs,
// each walking the whole context alone.  Two things split that walk:
//   - a cluster of up to 16 CTAs shares a row tile, each taking a range of its
//     stages; the partial results meet in distributed shared memory (no
//     workspace, no second launch).  launch_merge_t picks the size.
//   - a tile of at most 128 rows leaves tile B without rows: then both tiles
//     hold the same rows, A takes the even stages and B the odd ones ("dual"),
//     so the tensor cores do no work for padding and a stage costs half.
// One layer, 32/8 heads, D 128, a context of 23040: 16 rows 350 -> 37 us, 44
// rows 353 -> 47, 133 rows 363 -> 88, 512 rows 363 -> 193; 88 rows onto 8192
// 140 -> 38 us.
//
// CTA layout (384 threads, one CTA per SM, all 512 TMEM columns):
//   warps 0..3  softmax of tile A, warps 4..7 softmax of tile B: thread r of
//               a tile owns its row r = TMEM lane r (warp w reads lanes
//               32 (w % 4) ..).  It stages its Q row in shared memory; per
//               stage it reads its 128 scores, masks keys past the stage's
//               pages and past its causal limit, keeps a running max raised
//               only when a score exceeds it by more than 2^8 (O in TMEM is
//               then rescaled in place), and writes P = 2^(s - m) as two bf16
//               terms (P_hi + P_lo, exact to about 16 bits) into TMEM over its
//               own scores.  At the end it writes O to shared memory, from
//               where its warp writes the rows out, or, where a cluster's CTAs
//               or both tiles share them, the warps put them together.
//   warp 8      K loader, warp 9 V loader: page ids from the block table (32
//               per read, one batch ahead), one 2 KiB TMA copy per (page,
//               64-wide half of D) into separate K and V rings.
//   warp 10     TMEM owner and MMA issuer (the whole warp runs the loop with
//               warp-uniform operands, an elected lane issues), per stage j
//               and tile t = A, B,
//                 O_t += P_t(j-1) V_{j-1}   (A = P_hi, P_lo from TMEM, M 128, N D)
//                 S_t(j) = Q_t K_j^T        (M 128, N 128)
//               so that the softmax of one tile overlaps the MMAs of the
//               other.
//   warp 11     idle: it fills the third warpgroup, for the register split.
//
// What bounds it: at N = 128 a tcgen05.mma takes 65 to 78 cycles here with A in
// tensor memory and some 85 with A in shared memory, against 64; the 48 of a
// stage take 3360 cycles with a trivial softmax in place of this one, which
// makes them 3700 to 3800, by its tensor-memory traffic and by the hand-overs
// (publishing P in quarters, or moving the K and V waits from the MMA warp to
// a softmax warp, cost 4 to 7%).
//
// TMEM columns: tile t (0 = A, 1 = B) has S at 256 t (128 columns; the 16
// columns of keys [16 k, 16 k + 16) then hold P_hi and P_lo of those keys as
// bf16 pairs) and O at 256 t + 128.  S_t(j + 1) overwrites P_t(j)
// only after O_t += P_t(j) V_j, which the same thread issued first; and the
// commit that announces S_t(j) also covers O_t += P_t(j-1) V_{j-1}, so the
// softmax may rescale O_t as soon as it sees S_t(j).
//
// Synchronisation (every wait on these is bounded; one that runs out sets the
// status word and the CTA winds down.  A cluster's CTAs meet at two cluster
// barriers, whose wait has no limit: it ends because every thread of every CTA
// gets there, whatever ran out before):
//   k_full / k_empty, v_full / v_empty   ring slots (TMA bytes / MMA commit)
//   s_full[t]      S_t of the stage is complete                 (MMA commit)
//   p_full[t][h]   P_t of keys [64 h, 64 h + 64) is in TMEM     (128 arrivals)
//   o_final        every MMA of the CTA has completed
// S_t(j + 1) is issued only after p_full[t][1] of stage j, so each barrier is
// at most one phase ahead of its waiters.  The MMAs of the first half of P
// run while the softmax computes the second.
//
// Shared-memory operands use the 128-byte swizzle (8-row x 128-byte atoms):
//   Q_t [D/64][128 rows][64]   K-major A (SBO 1024)
//   K   [D/64][128 keys][64]   K-major B (SBO 1024)
//   V   [D/64][128 keys][64]   MN-major B (LBO = one D-half, SBO 1024)
// V rows of keys that are not valid (past main's end, or in pages a short
// last stage did not load) are zeroed by tile A's threads before P V, so that
// stale shared or pool memory cannot turn 0 * x into NaN in a real row.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <type_traits>
#include <vector>

#include "kernels.cuh"
#include "ptx.cuh"

namespace st {

namespace {

constexpr int kTileRows = 128;
constexpr int kKeys = 128;  // keys per stage
constexpr int kPagesPerStage = kKeys / kPageTokens;
constexpr int kKLoadWarp = 8, kVLoadWarp = 9, kMmaWarp = 10;
constexpr int kThreads = 12 * 32;  // three warpgroups, for the register split
constexpr int kSoftThreads = 8 * 32;
// Where the softmax threads hold a row's 128 scores (kHold), the warpgroups'
// registers are shared out anew, within what the block is launched with (168 a
// thread): 192 + 192 + 120.  setmaxnreg.inc waits without a limit for registers
// that the block does not have, and the launch bounds only cap what the compiler
// assigns, so pair_setup refuses a build with fewer before any launch.
constexpr int kSoftRegs = 192, kOtherRegs = 120;
constexpr bool regs_suffice(int launch_regs) {  // registers a thread at launch
  return launch_regs >= kOtherRegs &&
         kSoftThreads * kSoftRegs + (kThreads - kSoftThreads) * kOtherRegs <= kThreads * launch_regs;
}
template <int D, bool kDecode>
constexpr bool kSharesRegs = D == 128 && !kDecode;
static_assert(regs_suffice(168) && !regs_suffice(167), "registers of a block");
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemTile = 256, kTmemO = 128;  // per-tile column base, O offset within it
constexpr float kRescaleThreshold = 8.f;           // log2 units
constexpr float kLn2 = 0.69314718055994530942f;

// Load 128 consecutive fp32 columns of this thread's TMEM lane with one wait.
__device__ __forceinline__ void tmem_ld128(uint32_t taddr, float* v) {
  uint32_t r[128];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x128.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, "
      "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
      "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63, "
      "%64, %65, %66, %67, %68, %69, %70, %71, %72, %73, %74, %75, %76, %77, %78, %79, "
      "%80, %81, %82, %83, %84, %85, %86, %87, %88, %89, %90, %91, %92, %93, %94, %95, "
      "%96, %97, %98, %99, %100, %101, %102, %103, %104, %105, %106, %107, %108, %109, %110, %111, "
      "%112, %113, %114, %115, %116, %117, %118, %119, %120, %121, %122, %123, %124, %125, %126, %127}, [%128];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
        "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
        "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
        "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
        "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63]),
        "=r"(r[64]), "=r"(r[65]), "=r"(r[66]), "=r"(r[67]), "=r"(r[68]), "=r"(r[69]), "=r"(r[70]), "=r"(r[71]),
        "=r"(r[72]), "=r"(r[73]), "=r"(r[74]), "=r"(r[75]), "=r"(r[76]), "=r"(r[77]), "=r"(r[78]), "=r"(r[79]),
        "=r"(r[80]), "=r"(r[81]), "=r"(r[82]), "=r"(r[83]), "=r"(r[84]), "=r"(r[85]), "=r"(r[86]), "=r"(r[87]),
        "=r"(r[88]), "=r"(r[89]), "=r"(r[90]), "=r"(r[91]), "=r"(r[92]), "=r"(r[93]), "=r"(r[94]), "=r"(r[95]),
        "=r"(r[96]), "=r"(r[97]), "=r"(r[98]), "=r"(r[99]), "=r"(r[100]), "=r"(r[101]), "=r"(r[102]), "=r"(r[103]),
        "=r"(r[104]), "=r"(r[105]), "=r"(r[106]), "=r"(r[107]), "=r"(r[108]), "=r"(r[109]), "=r"(r[110]), "=r"(r[111]),
        "=r"(r[112]), "=r"(r[113]), "=r"(r[114]), "=r"(r[115]), "=r"(r[116]), "=r"(r[117]), "=r"(r[118]), "=r"(r[119]),
        "=r"(r[120]), "=r"(r[121]), "=r"(r[122]), "=r"(r[123]), "=r"(r[124]), "=r"(r[125]), "=r"(r[126]), "=r"(r[127])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 128; ++i) v[i] = __uint_as_float(r[i]);
}

// CTAs of a cluster that share one row tile's keys in a merge, at most (16 is
// the largest cluster of this part).
constexpr int kMaxMergeSplit = 16;
// Stages of 128 keys that a part of a split row tile has, at least.
constexpr int kMinPartStages = 4;

// Parts that a row tile of `all_tiles` stages is split into in a launch of
// clusters of `cluster` CTAs.  It depends on the tile alone where the cluster
// is large enough.
__host__ __device__ constexpr int merge_parts(int all_tiles, int cluster) {
  const int most = all_tiles / kMinPartStages;
  return most < 1 ? 1 : most < cluster ? most : cluster;
}

struct MergeSplitCost {
  int parts;
  float total, longest;  // of its CTAs together, of one of them
};

// Row tiles of a launch that cost the same.
struct MergeTileKind {
  int all_tiles, rows, n;
};

// A decode's run of pages of a fork group, for one KV head of one layer.
struct PairWork {
  AttnItem item;
  int32_t kvh, layer;
  int32_t valid;  // 0: no further one
};

// 16 bytes from global to shared memory, asynchronously; zeros if !valid.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst),
               "l"(__cvta_generic_to_global(src)), "r"(valid ? 16 : 0)
               : "memory");
}

// Registers of this warpgroup's threads from here on.
template <int N>
__device__ __forceinline__ void regs_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void regs_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

// Waits for every copy of this thread.
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int D>
struct PairCfg {
  static constexpr int kHalves = D / 64;
  static constexpr int kQHalfBytes = kTileRows * 128;
  static constexpr int kQTileBytes = kHalves * kQHalfBytes;
  static constexpr int kKVHalfBytes = kKeys * 128;
  static constexpr int kSlotBytes = kHalves * kKVHalfBytes;
  static constexpr int kKStages = D == 128 ? 3 : 4;
  static constexpr int kVStages = D == 128 ? 2 : 4;
  static constexpr int kQOff = 0;
  static constexpr int kKOff = kQOff + 2 * kQTileBytes;
  static constexpr int kVOff = kKOff + kKStages * kSlotBytes;
  static constexpr int kBarOff = kVOff + kVStages * kSlotBytes;
  static constexpr int kSmemBytes = 1024 + kBarOff + 512;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
};

// kMapped: a merge's CTAs (clusters) are not its tiles, heads and layers as the
// grid numbers them.  The layers may start at p.layer_base (a merge's second
// launch), and a last tile of at most 128 rows, whose stages cost half, comes
// behind the other tiles of every head and layer, so that the launch ends on
// the short ones (88 rows onto 8000 in 16 layers: 280 us before, 229).  A form
// of its own, since the arithmetic in every launch cost half a per cent.
//
// kPersist: a decode of more than one wave.  A run of pages is some 30 us here,
// and a CTA of its own for each left its SM idle for 6 more, from the last P V
// to the first of the next one.  So a CTA that is about to load its run's last
// stage asks for a CTA of the grid that has not started (cluster launch
// control) and goes on with its item: the next run's K and V land, its Q goes in
// and its first S is computed while the results come out.  Stage and barrier
// counts run on over a CTA's items; the K loader passes the items on through
// two slots, which every role reads in order.  Two layers of 2 groups of 24
// branches over 65536 tokens 316 -> 300 us, 17 branches in 4 layers 284 -> 263,
// 41 in 4 layers 482 -> 424, D = 64 162 -> 145.
template <int D, bool kDecode, bool kForm>
__global__ void __launch_bounds__(kThreads, 1)
    merge_pair_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                      const AttnParams p, const __grid_constant__ InlineDecodePlan inl) {
  using C = PairCfg<D>;
  constexpr int kKS = C::kKStages, kVS = C::kVStages;
  constexpr bool kMapped = !kDecode && kForm, kPersist = kDecode && kForm;
  constexpr bool kHold = kSharesRegs<D, kDecode>;  // the softmax holds its scores (below)
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_addr(smem_raw);
  uint8_t* base = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + C::kBarOff);
  uint64_t* k_full = bars;
  uint64_t* k_empty = k_full + kKS;
  uint64_t* v_full = k_empty + kKS;
  uint64_t* v_empty = v_full + kVS;
  uint64_t* s_full = v_empty + kVS;  // [2 tiles]
  uint64_t* p_full = s_full + 2;     // [2 tiles][2 key halves]
  uint64_t* o_final = p_full + 4;
  uint64_t* q_ready = o_final + 1;
  uint64_t* work_full = q_ready + 1;     // [2] kPersist: an item taken over is in its slot
  uint64_t* work_empty = work_full + 2;  // [2] every role has read it
  uint64_t* clc_bar = work_empty + 2;    // the answer to a request for one has landed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(clc_bar + 1);
  uint8_t* clc_resp = base + C::kBarOff + 320;  // 16 bytes
  PairWork* work_slots = reinterpret_cast<PairWork*>(base + C::kBarOff + 336);  // [2]
  static_assert(8 * (2 * kKS + 2 * kVS + 14) <= 320 && 336 + 2 * sizeof(PairWork) <= 512, "barrier area");

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int kvh = blockIdx.y, layer = blockIdx.z;
  const int G = p.G;

  // Launched as a programmatic dependent of the kernel before it in the
  // stream; the tensor-memory allocation and the barriers touch no global
  // memory, every global access comes after the wait.
  if (warp == kMmaWarp) tmem_alloc(tmem_slot, kTmemCols);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kKS; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
    }
    for (int s = 0; s < kVS; ++s) {
      mbar_init(&v_full[s], 1);
      mbar_init(&v_empty[s], 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&s_full[t], 1);
      mbar_init(&p_full[2 * t], kTileRows);
      mbar_init(&p_full[2 * t + 1], kTileRows);
    }
    mbar_init(o_final, 1);
    mbar_init(q_ready, kSoftThreads);
    if constexpr (kPersist) {
      for (int b = 0; b < 2; ++b) {
        mbar_init(&work_full[b], 1);
        mbar_init(&work_empty[b], 10);  // the V loader, the MMA warp and the softmax warps
      }
      mbar_init(clc_bar, 1);
    }
    fence_mbar_init();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  griddep_wait();
  if constexpr (kDecode) publish_large_launch(p);
  griddep_launch_dependents();
  // one merge: its row tiles, the last ones (most keys) first; a batch: one
  // work item per cluster (the host orders those longest first); a decode: one
  // run of pages of a fork group (at most 256 stacked rows) per CTA, every
  // row over all of the run's keys
  const int cluster = kDecode ? 1 : p.kv_split;  // CTAs that share a row tile
  const int rank = kDecode ? 0 : (int)blockIdx.x % cluster;
  int slot = p.slot, L0 = p.L0, T = p.T, q_row0 = 0;
  int tile = (int)blockIdx.x / cluster;
  if constexpr (kMapped) {
    const int n = (int)gridDim.x / cluster;
    if (!p.mitems && n > 1 && T * G - (n - 1) * 2 * kTileRows <= kTileRows) {  // tile 0, the last rows, is short
      const int u = tile + n * (int)(blockIdx.y + gridDim.y * blockIdx.z);
      const int full = (n - 1) * (int)(gridDim.y * gridDim.z);  // the other tiles
      const int hl = u < full ? u / (n - 1) : u - full;         // head and layer
      tile = u < full ? 1 + u % (n - 1) : 0;
      kvh = hl % (int)gridDim.y;
      layer = hl / (int)gridDim.y;
    }
    layer += p.layer_base;
  }
  int row_base = ((int)gridDim.x / cluster - 1 - tile) * 2 * kTileRows;
  int page_begin = 0, n_rows, n_pages, n_valid_keys;
  AttnItem item{};
  const int32_t* members = nullptr;
  auto item_at = [&](int x) -> const AttnItem& {
    return p.items ? p.items[p.item_base + x] : inl.items[p.item_base + x];
  };
  auto take_item = [&](const AttnItem& it) {  // a decode's work of this thread's role
    item = it;
    slot = item.slot;
    page_begin = item.page_begin;
    row_base = 0;
    n_rows = min(2 * kTileRows, item.n_members * G);
    n_pages = item.n_pages;
    n_valid_keys = item.n_tokens;
  };
  if constexpr (kDecode) {
    members = p.members ? p.members : inl.members;
    take_item(item_at(blockIdx.x));
  } else {
    if (p.mitems) {
      const MergeItem mi = p.mitems[blockIdx.x / cluster];
      slot = mi.slot;
      L0 = mi.L0;
      T = mi.T;
      q_row0 = mi.q_row0;
      row_base = mi.row_base;
    }
    n_rows = min(2 * kTileRows, T * G - row_base);
    const int t_last = (row_base + n_rows - 1) / G;
    n_pages = (L0 + t_last + 1 + kPageTokens - 1) / kPageTokens;
    n_valid_keys = L0 + T;
  }
  // this CTA's part of the row tile's stages (all of them without a split)
  const int all_tiles = (n_pages + kPagesPerStage - 1) / kPagesPerStage;
  const int n_parts = kDecode ? 1 : merge_parts(all_tiles, cluster);
  if (rank >= n_parts) {  // a tile with fewer parts than the launch's clusters: nothing left for this CTA
    if (warp == kMmaWarp) tmem_dealloc(tmem, kTmemCols);
    if (n_parts > 1) {  // the barriers of the exchange below count every CTA of the cluster
      cluster_sync();
      cluster_sync();
    }
    return;
  }
  // (the longer parts first: the last one has the stages at the causal limit,
  // whose masks cost it another microsecond or two)
  const int j0 = (rank * all_tiles + n_parts - 1) / n_parts, j1 = ((rank + 1) * all_tiles + n_parts - 1) / n_parts;
  int n_tiles = j1 - j0;
  const int key_base = j0 * kKeys;
  page_begin += j0 * kPagesPerStage;
  n_pages = min(n_pages - j0 * kPagesPerStage, n_tiles * kPagesPerStage);
  // at most 128 rows: both tiles hold them, tile A takes the even stages and tile B the odd ones
  const bool dual = !kDecode && n_rows <= kTileRows;
  const bool direct = kDecode || (n_parts == 1 && !dual);  // every row has one source, its thread's

  auto next_item = [&](const PairWork& w) {
    take_item(w.item);
    kvh = w.kvh;
    layer = w.layer;
    n_tiles = (n_pages + kPagesPerStage - 1) / kPagesPerStage;
  };
  // kPersist: the item after a role's n-th, which the K loader writes to slot n % 2.
  // False when there is none (or the wait ran out: *ok).
  auto next_work = [&](int n, PairWork* w, bool* ok) -> bool {
    const int b = n & 1;
    *ok = __all_sync(0xffffffffu, mbar_wait(&work_full[b], (n >> 1) & 1));
    if (!*ok) return false;
    *w = work_slots[b];
    __syncwarp();
    if (lane == 0) mbar_arrive(&work_empty[b]);
    return w->valid != 0;
  };

  if (warp >= kKLoadWarp) {
    if constexpr (kHold) regs_dec<kOtherRegs>();
    // ---- loaders -----------------------------------------------------------------
    // (hold_loads, a test hook: nothing arrives, the other roles' waits run out)
    if ((warp == kKLoadWarp || warp == kVLoadWarp) && !p.hold_loads) {
      const bool is_k = warp == kKLoadWarp;
      const CUtensorMap* map = is_k ? &kmap : &vmap;
      uint64_t* full = is_k ? k_full : v_full;
      uint64_t* empty = is_k ? k_empty : v_empty;
      const int n_st = is_k ? kKS : kVS;
      uint8_t* ring = base + (is_k ? C::kKOff : C::kVOff);
      if (lane == 0) prefetch_tensormap(map);
      int g = 0;  // stages whose copies have been issued, over all items
      bool ok = true;
      for (int n = 0;; ++n) {  // the CTA's items
        // merge: every CTA of one (layer, KV head) walks the same pages, keep them
        // in L2; decode: a page is streamed once, unless a sibling subgroup's CTA
        // reads it too or the whole launch fits in L2
        const uint64_t policy = !kDecode ? l2_policy_evict_last()
                                : (p.keep_l2 || (item.flags & kItemReread)) ? l2_policy_evict_normal()
                                                                             : l2_policy_evict_first();
        const int32_t* ids = p.table + (int64_t)slot * p.max_pages + page_begin;
        int base_id = 0;
        int cur = lane < n_pages ? ids[lane] : 0;
        int nxt = 32 + lane < n_pages ? ids[32 + lane] : 0;
        bool asked = false;
        for (int j = 0; j < n_tiles; ++j, ++g) {
          // ask for the next item no earlier than needed: one taken over sooner
          // waits here while another SM may have run dry
          if (kPersist && is_k && j == n_tiles - 1) {
            asked = true;
            if (lane == 0) {
              mbar_arrive_expect_tx(clc_bar, 16);
              clc_try_cancel(clc_resp, clc_bar);
            }
          }
          const int s = g % n_st;
          if (g >= n_st) {
            int w = 1;
            if (lane == 0) w = mbar_wait(&empty[s], ((g / n_st) - 1) & 1) ? 1 : 0;
            w = __shfl_sync(0xffffffffu, w, 0);
            if (!w) {
              ok = false;
              break;
            }
          }
          const int page0 = j * kPagesPerStage;
          if (page0 >= base_id + 32) {
            base_id += 32;
            cur = nxt;
            nxt = base_id + 32 + lane < n_pages ? ids[base_id + 32 + lane] : 0;
          }
          const int np = min(kPagesPerStage, n_pages - page0);
          uint8_t* dst = ring + s * C::kSlotBytes;
          if (lane == 0) mbar_arrive_expect_tx(&full[s], (uint32_t)(np * C::kHalves * kPageTokens * 128));
          __syncwarp();
          // one copy per lane (lane = D/64 q + h)
          const int q = lane / C::kHalves, h = lane % C::kHalves;
          int b = __shfl_sync(0xffffffffu, cur, (page0 - base_id + (q < kPagesPerStage ? q : 0)) & 31);
          if (lane < C::kHalves * np) {
            if ((uint64_t)b >= (uint64_t)p.n_blocks) {
              atomicCAS(p.status, 0, kDevBadIndex);
              b = 0;
            }
            tma_load_4d(dst + h * C::kKVHalfBytes + q * kPageTokens * 128, map, &full[s], 0, h, kvh * kPageTokens,
                        layer * (int)p.n_blocks + b, policy);
          }
        }
        if constexpr (!kPersist) {
          break;
        } else {
          PairWork w{};
          if (is_k) {
            uint32_t x = 0, y = 0, z = 0;
            const bool answered = asked && __all_sync(0xffffffffu, mbar_wait(clc_bar, n & 1));
            const bool more = answered && clc_answer(clc_resp, &x, &y, &z);
            fence_proxy_async_smem();  // every lane has read the answer before the next one lands
            __syncwarp();
            if (more) w = PairWork{item_at(x), (int)y, (int)z, 1};
            if (ok && answered && n >= 2) {  // the slot's last item has been read by every role
              int e = 1;
              if (lane == 0) e = mbar_wait(&work_empty[n & 1], ((n >> 1) - 1) & 1) ? 1 : 0;
              ok = __shfl_sync(0xffffffffu, e, 0) != 0;
            }
            ok = ok && answered;
            if (!ok) break;
            if (lane == 0) {
              work_slots[n & 1] = w;
              mbar_arrive(&work_full[n & 1]);
            }
          } else if (!ok || !next_work(n, &w, &ok)) {
            break;
          }
          if (!w.valid) break;
          next_item(w);
        }
      }
      if (!ok && lane == 0) {
        atomicCAS(p.status, 0, kDevTimeout);
        for (int t = max(0, g - n_st); t < g; ++t) mbar_wait(&full[t % n_st], (t / n_st) & 1);
      }
    }

    // ---- MMA issuer ----------------------------------------------------------------
    // One warp issues every MMA (two issuing warps interleaving on the tensor
    // pipe measured slower): all its lanes run the loop with warp-uniform
    // operands and an elected lane issues.  The issue rate bounds this kernel
    // (tens of cycles per tcgen05.mma), so the per-MMA work is a constant add:
    // a shared-memory descriptor's start field holds address / 16 (below 2^14
    // here), so the descriptor of an operand shifted by b bytes is the base
    // descriptor + b / 16.
    if (warp == kMmaWarp) {
      {
        constexpr uint32_t idesc_s = tc_idesc_bf16(kTileRows, kKeys, 0, 0);
        constexpr uint32_t idesc_o = tc_idesc_bf16(kTileRows, D, 0, 1);
        const uint64_t q_desc = tc_desc_sw128(smem_addr(base + C::kQOff), 16, 1024);
        const uint64_t k_desc0 = tc_desc_sw128(smem_addr(base + C::kKOff), 16, 1024);
        const uint64_t v_desc0 = tc_desc_sw128(smem_addr(base + C::kVOff), C::kKVHalfBytes, 1024);
        bool ok = true;
        int g0 = 0;  // the item's first stage among the CTA's
        // O_t += P_t(i) V, P_t(i) read from TMEM over S_t(i); each half of P
        // (64 keys) is published on its own, so the first half's MMAs run while
        // the softmax finishes the second
        auto issue_pv = [&](auto tile, int i, uint64_t vd) -> bool {
          constexpr int t = decltype(tile)::value;
          const uint32_t acc0 = i > 0 ? 1u : 0u;
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            if (!__all_sync(0xffffffffu, mbar_wait(&p_full[2 * t + hf], (g0 + i) & 1))) return false;
            tc_fence_after_sync();
#pragma unroll
            for (int kq = 0; kq < kKeys / 32; ++kq) {
              const int ks = hf * (kKeys / 32) + kq;
              const uint64_t vk = vd + (uint64_t)((ks * 16 * 128) >> 4);
              tc_mma_bf16_tmem_a_elect(tmem + t * kTmemTile + kTmemO, tmem + t * kTmemTile + ks * 16, vk, idesc_o,
                                 ks > 0 ? 1u : acc0);                                    // P_hi
              tc_mma_bf16_tmem_a_elect(tmem + t * kTmemTile + kTmemO, tmem + t * kTmemTile + ks * 16 + 8, vk, idesc_o,
                                 1u);                                                     // P_lo
            }
          }
          return true;
        };
        // S_t(i) = Q_t K^T
        auto issue_s = [&](auto tile, uint64_t qd, uint64_t kd) {
          constexpr int t = decltype(tile)::value;
#pragma unroll
          for (int h = 0; h < C::kHalves; ++h)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              tc_mma_bf16_elect(tmem + t * kTmemTile, qd + (uint64_t)((h * C::kQHalfBytes + kk * 32) >> 4),
                                kd + (uint64_t)((h * C::kKVHalfBytes + kk * 32) >> 4), idesc_s, (h | kk) != 0);
          tc_commit_elect(&s_full[t]);
        };
        const std::integral_constant<int, 0> tile_a;
        const std::integral_constant<int, 1> tile_b;
        const uint64_t qd_b = q_desc + (uint64_t)(C::kQTileBytes >> 4);
        for (int n = 0;; ++n) {  // the CTA's items
          ok = __all_sync(0xffffffffu, mbar_wait(q_ready, n & 1));
          tc_fence_after_sync();
          if (!dual) {
            // iteration i of both tiles is stage i
            auto pv = [&](auto tile, int i) -> bool {
              constexpr int t = decltype(tile)::value;
              const int g = g0 + i, s = g % kVS;
              if (t == 0 && !__all_sync(0xffffffffu, mbar_wait(&v_full[s], (g / kVS) & 1))) return false;
              if (!issue_pv(tile, i, v_desc0 + (uint64_t)((s * C::kSlotBytes) >> 4))) return false;
              if (t == 1) tc_commit_elect(&v_empty[s]);
              return true;
            };
            for (int i = 0; ok && i < n_tiles; ++i) {
              const int g = g0 + i, s = g % kKS;
              const uint64_t kd = k_desc0 + (uint64_t)((s * C::kSlotBytes) >> 4);
              ok = (i == 0 || pv(tile_a, i - 1)) && __all_sync(0xffffffffu, mbar_wait(&k_full[s], (g / kKS) & 1));
              if (!ok) break;
              tc_fence_after_sync();
              issue_s(tile_a, q_desc, kd);
              if (i > 0 && !pv(tile_b, i - 1)) {
                ok = false;
                break;
              }
              issue_s(tile_b, qd_b, kd);
              tc_commit_elect(&k_empty[s]);
            }
            if (ok && n_tiles > 0) ok = pv(tile_a, n_tiles - 1) && pv(tile_b, n_tiles - 1);
          } else {
            // iteration i of tile t is stage 2 i + t, its own K and V slot; of an
            // odd number of stages B has one fewer
            auto pv = [&](auto tile, int i) -> bool {
              const int j = 2 * i + decltype(tile)::value, s = j % kVS;
              if (!__all_sync(0xffffffffu, mbar_wait(&v_full[s], (j / kVS) & 1))) return false;
              if (!issue_pv(tile, i, v_desc0 + (uint64_t)((s * C::kSlotBytes) >> 4))) return false;
              tc_commit_elect(&v_empty[s]);
              return true;
            };
            auto qk = [&](auto tile, int i) -> bool {
              const int j = 2 * i + decltype(tile)::value, s = j % kKS;
              if (!__all_sync(0xffffffffu, mbar_wait(&k_full[s], (j / kKS) & 1))) return false;
              tc_fence_after_sync();
              issue_s(tile, q_desc, k_desc0 + (uint64_t)((s * C::kSlotBytes) >> 4));
              tc_commit_elect(&k_empty[s]);
              return true;
            };
            const int n_a = (n_tiles + 1) / 2, n_b = n_tiles / 2;
            for (int i = 0; ok && i < n_a; ++i)
              ok = (i == 0 || pv(tile_a, i - 1)) && qk(tile_a, i) && (i == 0 || pv(tile_b, i - 1)) &&
                   (i >= n_b || qk(tile_b, i));
            if (ok && n_a > 0) ok = pv(tile_a, n_a - 1) && (n_b < n_a || pv(tile_b, n_b - 1));
          }
          tc_commit_elect(o_final);
          if constexpr (!kPersist) {
            break;
          } else {
            g0 += n_tiles;
            PairWork w;
            if (!ok || !next_work(n, &w, &ok)) break;
            next_item(w);
          }
        }
        if (!ok && lane == 0) atomicCAS(p.status, 0, kDevTimeout);
      }
      __syncwarp();
      named_barrier_sync(1, kSoftThreads + 32);
      tc_fence_after_sync();
      tmem_dealloc(tmem, kTmemCols);
    }
    if (n_parts > 1) {  // the softmax warps' exchange
      cluster_sync();
      cluster_sync();
    }
    return;
  }
  if constexpr (kHold) regs_inc<kSoftRegs>();

  // ---- softmax warps ---------------------------------------------------------------
  const int t = warp >> 2;               // tile (of a softmax warp)
  const int r = (warp & 3) * 32 + lane;  // row within the tile = TMEM lane
  const int tile_row0 = row_base + (dual ? 0 : t * kTileRows);
  bool valid;
  int qrow;
  int64_t in_row;  // this row in Q / O / LSE
  auto find_row = [&]() {
    int head = 0;
    valid = tile_row0 - row_base + r < n_rows;
    qrow = 0;
    if (valid) {
      const int gr = tile_row0 + r;
      qrow = kDecode ? members[item.member_base + gr / G] : gr / G;
      head = kvh * G + gr % G;
    }
    in_row = ((int64_t)layer * p.n_rows_q + q_row0 + qrow) * p.Hq + head;
  };
  find_row();
  // Results on their way out, over the K, V and Q buffers once every MMA has
  // completed: xo [2 tiles][128 rows][D/4] float4 of the unnormalised O (xo_at:
  // columns swizzled by the row, so that a warp reads or writes a column of 32
  // rows and a row of 32 columns without bank conflicts); xml [2 tiles][128
  // rows], a row's max and sum; and of the rows that this CTA puts together, at
  // most 256 / parts of them from as many sources: xw and xwt, the sources'
  // maxima, sums and weights, and xrow, their places in the output.
  constexpr int kQuads = D / 4;
  float4* xo = reinterpret_cast<float4*>(base + C::kKOff);
  float2* xml = reinterpret_cast<float2*>(base + C::kQOff);
  float2* xw = xml + 2 * kTileRows;
  float* xwt = reinterpret_cast<float*>(xw + 4 * kTileRows);
  int64_t* xrow = reinterpret_cast<int64_t*>(xw + 8 * kTileRows);
  auto xo_at = [&](int tile, int row, int c) { return (tile * kTileRows + row) * kQuads + (c ^ (row & (kQuads - 1))); };
  static_assert(2 * kTileRows * D * 4 <= C::kBarOff - C::kKOff, "the exchange fits the K and V rings");

  bool ok = true;
  {
    const int tid = threadIdx.x & (kTileRows - 1);
    const uint32_t t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + t * kTmemTile;
    auto load_q = [&]() {
      // D/8 lanes copy a row's D contiguous values, straight to shared memory:
      // all 32 rows of the warp are in flight at once (a thread loading its own
      // row through registers took 4.7 us for the tile, this 1.9)
      constexpr int kChunks = D / 8, kRows = 32 / kChunks;
      const uint32_t q_s = smem_addr(base + C::kQOff + t * C::kQTileBytes);
      const int c = lane % kChunks;
      const int64_t mine = valid ? in_row : -1;
#pragma unroll 4
      for (int i = 0; i < 32 / kRows; ++i) {
        const int x = i * kRows + lane / kChunks, row = (warp & 3) * 32 + x;
        const int64_t from = __shfl_sync(0xffffffffu, mine, x);
        cp_async16(q_s + (c >> 3) * C::kQHalfBytes + row * 128 + (((c & 7) ^ (row & 7)) << 4),
                   p.q + (from >= 0 ? from * D + c * 8 : 0), from >= 0);
      }
      cp_async_wait();
      fence_proxy_async_smem();
    };
    if (!dual || t == 0) load_q();
    mbar_arrive(q_ready);

    const float sl2 = p.scale_log2;
    float m_used, l;
    int n_it, g0 = 0;  // the item's stages of this tile, the first one's number among the CTA's
    for (int n = 0;; ++n) {  // the CTA's items
      // causal limit of this row (a decode row sees the whole run)
      const int limit = kDecode ? n_valid_keys : valid ? L0 + qrow + 1 : n_valid_keys;
      const int min_limit = kDecode ? n_valid_keys : L0 + tile_row0 / G + 1;  // the tile's first row sees the fewest keys
      m_used = -1e30f;
      l = 0.f;
      n_it = dual ? (n_tiles + 1 - t) / 2 : n_tiles;
      for (int it = 0; it < n_it; ++it) {
        const int j = dual ? 2 * it + t : it;  // the stage
        if (!__all_sync(0xffffffffu, mbar_wait(&s_full[t], (g0 + it) & 1))) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        const int key0 = key_base + j * kKeys;
        const int loaded = min(kPagesPerStage, n_pages - j * kPagesPerStage) * kPageTokens;
        const bool edge = key0 + kKeys > min_limit || loaded < kKeys;
        const int n_seen = min(loaded, limit - key0);  // this row's keys of the stage
        // scores of keys [hf * 64, hf * 64 + 64), masked past the stage's pages and
        // past this row's causal limit
        auto load_half = [&](int hf, float* sc) {
          tmem_ld64(t_lane + hf * 64, sc);
          if (edge) {
#pragma unroll
            for (int c = 0; c < 64; ++c)
              if (c >= n_seen - hf * 64) sc[c] = -INFINITY;
          }
        };
        // With kHold the row's scores stay in registers from the maximum to the
        // probabilities: reading them twice takes tensor-memory bandwidth from
        // the MMAs (4 layers of 2048 rows: 1980 us reading twice, 1942 holding;
        // D = 64, whose MMAs leave the softmax the longer chain, and the decode
        // are faster with the shorter code that reads twice).
        float held[kHold ? kKeys : 1];
        float mx;
        if constexpr (kHold) {
          tmem_ld128(t_lane, held);
          if (edge) {
#pragma unroll
            for (int c = 0; c < kKeys; ++c)
              if (c >= n_seen) held[c] = -INFINITY;
          }
          float mx8[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) mx8[i] = fmaxf(held[i], held[8 + i]);
#pragma unroll
          for (int c = 16; c < kKeys; c += 16)
#pragma unroll
            for (int i = 0; i < 8; ++i) mx8[i] = fmax3(mx8[i], held[c + i], held[c + 8 + i]);
          mx = fmax3(fmax3(mx8[0], mx8[1], mx8[2]), fmax3(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7]));
        } else {
          // row max over both halves: independent chains of three-input max
          float mx8[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) mx8[i] = -INFINITY;
#pragma unroll 1  // one half's scores live at a time
          for (int hf = 0; hf < 2; ++hf) {
            float sc[64];
            load_half(hf, sc);
#pragma unroll
            for (int c = 0; c < 64; c += 16)
#pragma unroll
              for (int i = 0; i < 8; ++i) mx8[i] = fmax3(mx8[i], sc[c + i], sc[c + 8 + i]);
          }
          mx = fmax3(fmax3(mx8[0], mx8[1], mx8[2]), fmax3(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7]));
        }
        const float m_new = fmaxf(m_used, mx * sl2);  // sl2 > 0: max commutes with the scale
        const bool need = valid && m_new > m_used + kRescaleThreshold;
        if (__any_sync(0xffffffffu, need)) {
          const float alpha = need ? ex2(m_used - m_new) : 1.f;
          if (it > 0) {
            // the O_t += P_t V before has completed (covered by the commit of this S_t)
#pragma unroll 1
            for (int k = 0; k < D / 32; ++k) {
              float o[32];
              tmem_ld32(t_lane + kTmemO + k * 32, o);
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] *= alpha;
              tmem_st32(t_lane + kTmemO + k * 32, o);
            }
          }
          l *= alpha;
          if (need) m_used = m_new;
        }
        if ((t == 0 || dual) && (key0 + kKeys > n_valid_keys || loaded < kKeys)) {
          // zero the V rows of keys that are not valid once the stage's copies
          // have landed; the P V that read the stage are issued after this tile's
          // first P half
          const int g = g0 + j, s = g % kVS;
          if (!__all_sync(0xffffffffu, mbar_wait(&v_full[s], (g / kVS) & 1))) {
            ok = false;
            break;
          }
          uint8_t* vslot = base + C::kVOff + s * C::kSlotBytes;
          for (int x = tid; x < kKeys * C::kHalves; x += kTileRows) {
            const int c = x % kKeys, h = x / kKeys;
            if (c >= loaded || key0 + c >= n_valid_keys) {
#pragma unroll
              for (int y = 0; y < 8; ++y)
                *reinterpret_cast<uint4*>(vslot + h * C::kKVHalfBytes + c * 128 + y * 16) = make_uint4(0u, 0u, 0u, 0u);
            }
          }
          fence_proxy_async_smem();
        }
        // P = 2^(s sl2 - m) (two keys per packed f32x2 FMA / add) as two bf16
        // terms, P_hi = bf16(P) and P_lo = bf16(P - P_hi), so that P V is exact to
        // about 16 bits whatever the spread of the scores.  The 16 score columns
        // of keys [16 ks, 16 ks + 16) take P_hi of those keys (8 columns of bf16
        // pairs) and then P_lo (8 columns): each store overwrites only scores
        // already read.
        {
          const float2 scale2 = make_float2(sl2, sl2), neg_m2 = make_float2(-m_used, -m_used);
          float2 rs[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
          // one half's P from its scores, published
          auto publish = [&](int hf, const float* sc) {
#pragma unroll
            for (int kq = 0; kq < 4; ++kq) {  // 16 keys per step
              uint32_t pk[16];
#pragma unroll
              for (int c = 0; c < 16; c += 2)
                prob_pair(sc[kq * 16 + c], sc[kq * 16 + c + 1], scale2, neg_m2, &rs[(c >> 1) & 3], &pk[c / 2],
                          &pk[8 + c / 2]);
              tmem_st16u_nowait(t_lane + (hf * 4 + kq) * 16, pk);
            }
            tmem_wait_st();
            tc_fence_before_sync();
            mbar_arrive(&p_full[2 * t + hf]);
          };
          if constexpr (kHold) {
            publish(0, held);
            publish(1, held + 64);
          } else {
#pragma unroll 1
            for (int hf = 0; hf < 2; ++hf) {
              float sc[64];
              load_half(hf, sc);
              publish(hf, sc);
            }
          }
          const float2 s = __fadd2_rn(__fadd2_rn(rs[0], rs[1]), __fadd2_rn(rs[2], rs[3]));
          l += s.x + s.y;
        }
      }
      if constexpr (!kPersist) {
        break;
      } else {
        if (!ok) break;
        // the next item's Q goes in before this one's results come out: its S
        // (every S of this tile has been computed) runs meanwhile.  Its first P V
        // waits for this thread's P, behind the results.
        const int64_t out_row = valid ? in_row * p.max_splits + item.split : -1;
        PairWork next;
        const bool more = next_work(n, &next, &ok);
        if (!ok) break;
        if (more) {
          g0 += n_tiles;
          next_item(next);
          find_row();
          load_q();
          mbar_arrive(q_ready);
        }
        if (!__all_sync(0xffffffffu, mbar_wait(o_final, n & 1))) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        // straight from tensor memory, whole 32-byte sectors: four lanes have 8
        // columns of a row (the next item's stages are landing in the buffers
        // through which a single item's results leave)
        const float inv = 1.f / l;
#pragma unroll 1
        for (int hf = 0; hf < 2; ++hf) {
          const int ra = 16 * hf + lane / 4;  // of the warp's 32 rows; the other one is ra + 8
          const float inv_a = __shfl_sync(0xffffffffu, inv, ra), inv_b = __shfl_sync(0xffffffffu, inv, ra + 8);
          const int64_t to_a = __shfl_sync(0xffffffffu, out_row, ra), to_b = __shfl_sync(0xffffffffu, out_row, ra + 8);
#pragma unroll 1
          for (int k = 0; k < D / 64; ++k) {
            float o[32];
            tmem_ld_16x64(t_lane + ((uint32_t)(16 * hf) << 16) + kTmemO + 64 * k, o);
            const int c = 64 * k + 2 * (lane % 4);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              if (to_a >= 0)
                *reinterpret_cast<float2*>(p.out_o + to_a * D + c + 8 * i) =
                    make_float2(o[4 * i] * inv_a, o[4 * i + 1] * inv_a);
              if (to_b >= 0)
                *reinterpret_cast<float2*>(p.out_o + to_b * D + c + 8 * i) =
                    make_float2(o[4 * i + 2] * inv_b, o[4 * i + 3] * inv_b);
            }
          }
        }
        if (out_row >= 0) p.out_lse[out_row] = (m_used + log2f(l)) * kLn2;
        if (!more) break;
      }
    }
    if constexpr (kPersist) {
      if (!ok && lane == 0) atomicCAS(p.status, 0, kDevTimeout);
      tc_fence_before_sync();
      named_barrier_sync(1, kSoftThreads + 32);
      return;
    }
    if (ok) ok = __all_sync(0xffffffffu, mbar_wait(o_final, 0));
    tc_fence_after_sync();
    if (!ok && lane == 0) atomicCAS(p.status, 0, kDevTimeout);
    // O out of TMEM, a thread its row; final if this tile has the row's only source
    const bool some = ok && n_it > 0;
    if (some) {
      const float scale = direct ? 1.f / l : 1.f;
#pragma unroll 1
      for (int k = 0; k < D / 32; ++k) {
        float o[32];
        tmem_ld32(t_lane + kTmemO + k * 32, o);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          xo[xo_at(t, r, k * 8 + i)] =
              make_float4(o[4 * i] * scale, o[4 * i + 1] * scale, o[4 * i + 2] * scale, o[4 * i + 3] * scale);
      }
    }
    if (!direct) {
      xml[t * kTileRows + r] = make_float2(m_used, some ? l : 0.f);
    } else if (some) {
      // the warp writes its 32 rows, D contiguous values at a time (a thread
      // writing its own row touches 32 rows per store: 6.3 us from the last P V
      // to the end; through the exchange below 5.8; this way 3.1)
      __syncwarp();
      const int64_t out_row = !valid ? -1 : kDecode ? in_row * p.max_splits + item.split : in_row;
      constexpr int kRows = 32 / kQuads < 1 ? 1 : 32 / kQuads;
      const int c = lane % kQuads;
#pragma unroll 4
      for (int i = 0; i < 32 / kRows; ++i) {
        const int x = i * kRows + lane / kQuads;
        const int64_t to = __shfl_sync(0xffffffffu, out_row, x);
        if (to >= 0) reinterpret_cast<float4*>(p.out_o + to * D)[c] = xo[xo_at(t, (warp & 3) * 32 + x, c)];
      }
      if (valid) p.out_lse[out_row] = (m_used + log2f(l)) * kLn2;
    }
    tc_fence_before_sync();
    named_barrier_sync(1, kSoftThreads + 32);
  }

  // ---- results of several sources ------------------------------------------------------
  if (direct) return;
  // A row's sources are the CTAs of its cluster, and in each both tiles when
  // they share their rows: O = sum 2^(m_s - m) O_s / sum 2^(m_s - m) l_s.  The
  // rows are dealt out to the CTAs, and D/4 lanes put together a row: every
  // read of a source's row, through distributed shared memory, and every write
  // of O are D contiguous values.  A source without a key for the row has l = 0,
  // and its O was perhaps never written.
  // This code runs once per CTA, so its time is mostly that of fetching its
  // instructions: loops are kept rolled (a version with 16 loads in flight
  // took 12 us where the same work rolled took 5).
  if (n_parts > 1) cluster_sync();  // (one part: the barrier above has ordered the exchange)
  {
    const int per_cta = dual ? 2 : 1, n_src = n_parts * per_cta;
    // this CTA's rows: x0 + [0, n_own)
    const int x0 = rank * n_rows / n_parts, n_own = (rank + 1) * n_rows / n_parts - x0;
    // source s of row x: CTA s (tile x / 128), or tile s & 1 of CTA s >> 1
    auto src_cta = [&](int s) { return (uint32_t)(dual ? s >> 1 : s); };
    auto src_tile = [&](int s, int x) { return dual ? s & 1 : x >> 7; };
    const int n_pairs = n_own * n_src;
#pragma unroll 1
    for (int i = threadIdx.x; i < n_pairs; i += kSoftThreads) {
      const int x = x0 + i / n_src, s = i % n_src;
      xw[i] = ld_cluster_f2(smem_addr(xml + src_tile(s, x) * kTileRows + (x & (kTileRows - 1))), src_cta(s));
    }
    named_barrier_sync(2, kSoftThreads);
    // each pair's weight, 2^(m_s - m) / sum 2^(m_s - m) l_s
#pragma unroll 1
    for (int i = threadIdx.x; i < n_pairs; i += kSoftThreads) {
      const int k = i / n_src;
      const float2* ml = xw + k * n_src;
      float m = -1e30f, l = 0.f;
#pragma unroll 1
      for (int s = 0; s < n_src; ++s) {
        const float2 x = ml[s];
        if (x.y == 0.f) continue;
        const float m_new = fmaxf(m, x.x);
        l = l * ex2(m - m_new) + x.y * ex2(x.x - m_new);
        m = m_new;
      }
      const float2 mine = xw[i];
      xwt[i] = (mine.y != 0.f ? ex2(mine.x - m) : 0.f) / l;  // (NaN for a row without any weight)
      if (i == k * n_src) {
        const int gr = row_base + x0 + k;
        const int64_t out_row = ((int64_t)layer * p.n_rows_q + q_row0 + gr / G) * p.Hq + kvh * G + gr % G;
        xrow[k] = out_row;
        if (ok) p.out_lse[out_row] = (m + log2f(l)) * kLn2;
      }
    }
    named_barrier_sync(2, kSoftThreads);
    // the pairs of a warp's rows one after another, a few loads in flight
    constexpr int kRows = 32 / kQuads < 1 ? 1 : 32 / kQuads, kStep = kRows * (kSoftThreads / 32), kBatch = 4;
    const int c = lane % kQuads;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    int k = warp * kRows + lane / kQuads, s = 0;  // the next pair to load: row x0 + k, source s
#pragma unroll 1
    while (k < n_own) {
      float4 v[kBatch];
      float w[kBatch];
      int done[kBatch];  // the row that the pair completes, or -1
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        w[u] = 0.f;
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        done[u] = -1;
        if (k < n_own) {
          w[u] = xwt[k * n_src + s];
          if (w[u] != 0.f)
            v[u] = ld_cluster_f4(smem_addr(xo + xo_at(src_tile(s, x0 + k), (x0 + k) & (kTileRows - 1), c)), src_cta(s));
          if (++s == n_src) {
            done[u] = k;
            s = 0;
            k += kStep;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        acc.x += w[u] * v[u].x;
        acc.y += w[u] * v[u].y;
        acc.z += w[u] * v[u].z;
        acc.w += w[u] * v[u].w;
        if (done[u] >= 0) {
          if (ok) reinterpret_cast<float4*>(p.out_o + xrow[done[u]] * D)[c] = acc;
          acc = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
  }
  if (n_parts > 1) cluster_sync();  // a CTA's buffers stay until its peers have read them
}

// Per device: the shared-memory opt-in, and how many CTAs of clusters of n are
// resident at once (a cluster sits inside one GPC, so the SMs that a size
// leaves over stay idle; 0: the size is not available).
struct PairSetup {
  bool done = false;
  int sms = 0;
  int resident[kMaxMergeSplit + 1] = {};
};

template <int D, bool kDecode>
cudaError_t pair_setup(const PairSetup** out) {
  using C = PairCfg<D>;
  static PairSetup setups[64];
  static std::mutex mu;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  PairSetup& ps = setups[dev];
  std::lock_guard<std::mutex> lock(mu);
  if (!ps.done) {
    e = cudaDeviceGetAttribute(&ps.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    auto* kernel = merge_pair_kernel<D, kDecode, false>;
    auto* other = merge_pair_kernel<D, kDecode, true>;
    for (auto* k : {kernel, other}) {
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
      if (e != cudaSuccess) return e;
      if (kSharesRegs<D, kDecode>) {
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, k);
        if (e != cudaSuccess) return e;
        if (!regs_suffice(fa.numRegs)) return cudaErrorInvalidKernelImage;
      }
    }
    if constexpr (!kDecode) {
      for (auto* k : {kernel, other}) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
      }
      for (int n = 1; n <= kMaxMergeSplit; ++n) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(n);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = C::kSmemBytes;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = n;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) {
          cudaGetLastError();  // a size this part does not offer
          clusters = 0;
        }
        ps.resident[n] = clusters * n;
      }
      if (ps.resident[1] < 1) return cudaErrorInvalidConfiguration;
    }
    ps.done = true;
  }
  *out = &ps;
  return cudaSuccess;
}

const InlineDecodePlan kNoInline{};

// Cost of a row tile's CTAs in a launch of clusters of `split`.
MergeSplitCost merge_tile_cost(int all_tiles, int n_rows, int split) {
  // microseconds: a stage of 128 keys for 256 rows and for up to 128 (the tiles
  // taking the stages in turn), a CTA's start and end, the exchange.  The stages
  // and the exchange are as measured at D = 128 (a merge of 183 stages: 344, 182,
  // 99, 58 and 47 us in 1, 2, 4, 8 and 12 parts).  A CTA's start and end take about
  // half of kCta since Q comes in by asynchronous copies and rows with one source
  // leave through their warp; the value stays, because with the measured 5 (and 11
  // for the exchange) the model left tiles of a few stages whole that two parts do
  // faster (9 stages: 31.2 us in the one part it chose, 26.6 in two).  D = 64 has no constants of its own:
  // of 17 shapes the choice was within 7% of the best of 16 sizes in 16, never
  // behind one part, and 15% behind two parts in one (200 rows onto 9000 in 8
  // layers: 262 and 228 us).
  constexpr float kStage = 1.9f, kDualStage = 1.15f, kCta = 10.f, kExchange = 6.f;
  const int parts = merge_parts(all_tiles, split);
  const float stage = n_rows <= kTileRows ? kDualStage : kStage;
  const float fixed = kCta + (parts > 1 ? kExchange : 0.f);
  return {parts, parts * fixed + all_tiles * stage, fixed + (float)((all_tiles + parts - 1) / parts) * stage};
}

template <int D>
cudaError_t launch_merge_t(const CUtensorMap& km, const CUtensorMap& vm, AttnParams p, const MergeItem* host_items,
                           int n_items, cudaStream_t s, int* n_launches) {
  const PairSetup* ps = nullptr;
  cudaError_t e = pair_setup<D, false>(&ps);
  if (e != cudaSuccess) return e;
  // The launch's row tiles, neighbours of equal cost counted together: a batch's
  // come in the order of their keys, and the estimates below go over them up to
  // 32 times (one by one, the call of 600 sequences of a row each took 33 us more, that of
  // 32 of 150 rows 5 of 99).
  std::vector<MergeTileKind> kinds;
  auto list_kinds = [&] {
    for (int i = 0; i < n_items; ++i) {
      const int T = host_items ? host_items[i].T : p.T, L0 = host_items ? host_items[i].L0 : p.L0;
      const int row_base = host_items ? host_items[i].row_base : i * 2 * kTileRows;
      const int rows = std::min(2 * kTileRows, T * p.G - row_base);
      const int keys = L0 + (row_base + rows - 1) / p.G + 1;
      const MergeTileKind k{(keys + kKeys - 1) / kKeys, rows <= kTileRows ? kTileRows : 2 * kTileRows, 1};
      if (!kinds.empty() && kinds.back().all_tiles == k.all_tiles && kinds.back().rows == k.rows) ++kinds.back().n;
      else kinds.push_back(k);
    }
  };
  // Estimated time of `layers` layers in clusters of n: waves of CTAs of average
  // length, or the longest CTA if that is more.
  auto estimate = [&](int n, int layers) {
    int64_t ctas = 0;
    float total = 0.f, longest = 0.f;
    for (const MergeTileKind& k : kinds) {
      const MergeSplitCost c = merge_tile_cost(k.all_tiles, k.rows, n);
      ctas += (int64_t)c.parts * k.n;
      total += c.total * k.n;
      longest = std::max(longest, c.longest);
    }
    const int64_t waves = (ctas * p.Hkv * layers + ps->resident[n] - 1) / ps->resident[n];
    return std::max(longest, waves * total / ctas);
  };
  // CTAs per row tile: the size with the least estimate.  At D = 128 the choice was
  // within 6% of the best of 16 sizes on every shape measured (10 parts for 24 row
  // tiles, say, need two waves and take 105 us, where 5 take 87); D = 64: above.
  auto best_split = [&](int layers, float* time) {
    int split = 1;
    *time = estimate(1, layers);
    for (int n = 2; n <= kMaxMergeSplit; ++n) {
      if (ps->resident[n] < 1) continue;
      const float t = estimate(n, layers);
      if (t < 0.97f * *time) {
        *time = t;
        split = n;
      }
    }
    return split;
  };
  // With 8 waves and more the last one's loss is small and a split only adds
  // CTAs: 4 layers of 256 row tiles took 2.01 ms whole, 2.23 in two parts.
  int split[2] = {1, 1}, layers[2] = {p.L, 0};
  const int64_t sms = ps->resident[1], per_layer = (int64_t)n_items * p.Hkv, total = per_layer * p.L;
  if (total < 8 * sms) {
    list_kinds();
    float time;
    split[0] = best_split(p.L, &time);
    // A few whole waves and a rest: the layers of the whole waves as they are,
    // and the rest in a launch behind them, split so that it fills the SMs
    // (44 rows onto 23040 in 32 layers, 256 row tiles: 755 us in one launch, 712
    // in two).
    const int whole = (int)(total / sms * sms / per_layer);
    if (whole > 0 && whole < p.L) {
      float rest;
      const int rest_split = best_split(p.L - whole, &rest);
      if (estimate(1, whole) + rest < 0.95f * time) {
        split[0] = 1;
        split[1] = rest_split;
        layers[0] = whole;
        layers[1] = p.L - whole;
      }
    }
  }
  const bool short_last = !host_items && n_items > 1 && p.T * p.G - (n_items - 1) * 2 * kTileRows <= kTileRows;
  for (int i = 0; i < 2 && layers[i] > 0; ++i) {
    p.kv_split = split[i];
    p.layer_base = i ? layers[0] : 0;
    auto* kernel = i > 0 || short_last ? merge_pair_kernel<D, false, true> : merge_pair_kernel<D, false, false>;
    e = launch_chained_cluster(kernel, dim3(n_items * split[i], p.Hkv, layers[i]), dim3(kThreads),
                               PairCfg<D>::kSmemBytes, s, split[i], km, vm, p, kNoInline);
    if (e != cudaSuccess) return e;
    *n_launches = i + 1;
  }
  return cudaSuccess;
}

template <int D>
cudaError_t launch_decode_pair_t(const CUtensorMap& km, const CUtensorMap& vm, const AttnParams& p,
                                 const InlineDecodePlan& inl, int n_items, cudaStream_t s) {
  const PairSetup* ps = nullptr;
  cudaError_t e = pair_setup<D, true>(&ps);
  if (e != cudaSuccess) return e;
  // CTAs that take over further items where there is more than one wave of
  // them, one CTA per SM; within one wave there is nothing to take over
  auto* kernel = (int64_t)n_items * p.Hkv * p.L > ps->sms ? merge_pair_kernel<D, true, true>
                                                          : merge_pair_kernel<D, true, false>;
  return launch_chained(kernel, dim3(n_items, p.Hkv, p.L), dim3(kThreads),
                        PairCfg<D>::kSmemBytes, s, km, vm, p, inl);
}

}  // namespace

cudaError_t launch_merge_tc(const CUtensorMap& km, const CUtensorMap& vm, const AttnParams& p,
                            const MergeItem* host_items, int n_items, int D, cudaStream_t s, int* n_launches) {
  *n_launches = 0;
  // one merge: ceil(T G / 256) row tiles; a batch: its work items
  if (!p.mitems) n_items = (p.T * p.G + 2 * kTileRows - 1) / (2 * kTileRows);
  if (n_items <= 0) return cudaSuccess;
  if (D == 128) return launch_merge_t<128>(km, vm, p, host_items, n_items, s, n_launches);
  if (D == 64) return launch_merge_t<64>(km, vm, p, host_items, n_items, s, n_launches);
  return cudaErrorInvalidValue;
}

cudaError_t launch_decode_pair(const CUtensorMap& km, const CUtensorMap& vm, const AttnParams& p,
                               const InlineDecodePlan* inl, int n_items, int D, cudaStream_t s) {
  const InlineDecodePlan& ip = inl ? *inl : kNoInline;
  if (n_items <= 0) return cudaSuccess;
  if (D == 128) return launch_decode_pair_t<128>(km, vm, p, ip, n_items, s);
  if (D == 64) return launch_decode_pair_t<64>(km, vm, p, ip, n_items, s);
  return cudaErrorInvalidValue;
}

}  // namespace st

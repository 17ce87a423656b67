// Fork-group decode partials on the 5th-generation tensor cores (tcgen05,
// accumulators in tensor memory).  The merge prefill is in merge_tc.cu.
//
// Section 3.3 of the paper: every branch receives the snapshot H_t + R_t, so
// the prefix KV is shared by all decoding streams; Section 4.4: branch load
// is dominated by those cached-prefix reads.  A decode CTA owns one run of
// pages of one KV head of one layer and stacks every query row that reads
// it -- for a shared prefix all branches of the fork group x the G query
// heads of the KV head (<= 64 rows) -- so each prefix page crosses HBM once
// per group.
//
// Two tile shapes (Section 3.2 lets the branch count vary, so the stacked
// row count n_b G does):
//   narrow  S at M = 64, up to 64 rows (the paper's 1 + 4 branches at
//           G <= 12); P goes to shared memory over the stage's consumed K
//           slot, its two bf16 terms stacked as the 128 A rows of one P V
//   wide    M = 128, up to 128 rows; P stays in TMEM over its own scores and
//           P V reads it from there (no P in shared memory, so two CTAs still
//           fit an SM).
// A group of 129 to 256 rows runs on the merge kernel's paired tile
// (merge_tc.cu); a larger one is split into paired subgroups whose items over
// the same pages run next to each other, so the second read of a page comes
// from L2.
//
// CTA layout (192 threads, 2 CTAs per SM):
//   warps 0..3  softmax (only those with rows run).  Narrow: row r's scores
//               sit in TMEM lane 32 (r / 16) + r % 16, and threads t and
//               t + 16 of a warp share row t, each with half of the stage's
//               keys (16-lane TMEM loads with a column split); thread t owns
//               the lane of the row's O_hi, thread t + 16 the lane 16 higher,
//               which holds O_lo.  Wide: thread r owns row r = TMEM lane r.
//               A thread loads its part of its Q row into shared memory;
//               per stage it reads its
//               scores from TMEM, masks keys past the run, keeps a running max
//               (narrow: combined with its partner by one shuffle) that is
//               raised only when a score exceeds it by more than 2^8 (O in
//               TMEM is then rescaled in place), and writes P = 2^(s - m) as
//               two bf16 terms.  At the end it normalises O out of TMEM: a
//               split-KV partial with its log-sum-exp.
//   warp 4      loader: page ids from the block table (32 per read, one batch
//               ahead), one 2 KiB TMA copy per (page, 64-wide half of D, K|V)
//               into a ring of stages, per-stage mbarriers with byte counts;
//               a stage's copies are issued by the warp's lanes together.
//               Narrow: one ring of three stages (D = 64: four), a stage's K
//               and V slots freed together after its P V.  Wide: K and V have
//               rings and barriers of their own (two and three slots; D = 64:
//               six and six); a K slot is freed by the commit after S_j, a V
//               slot after P_j V_j.
//               A decode step (st_decode_step): the narrow item that holds a
//               branch's last page first stores the step's new K and V row of
//               its (layer, KV head) into that page, then a proxy fence makes
//               the store visible to the page's TMA copies.  Only that CTA
//               reads the page (a branch's last page is its own), so no
//               separate append launch is needed.
//   warp 5      TMEM owner; lane 0 issues   S = Q K^T  (M, N=64 keys)
//               and O += P V (M = 128, N=D) and commits them to mbarriers.  S is
//               double-buffered in TMEM: S_{j+1} is issued before P_j V_j when
//               its data has landed, so the softmax of stage j+1 overlaps the
//               tensor work of stage j.
//               A rescale of O first waits for the commit of P_{j-1} V_{j-1}.
//
// The kernel is launched as a programmatic dependent of the append before it
// in the stream: the TMEM allocation, and with the plan in the parameters the
// whole set-up, come before griddepcontrol.wait, every global-memory access
// after it (a single agent's step, 5 stages per CTA: the first scores 1.8 us
// after the wait, 2.3 with the set-up behind it).
//
// More than one wave (kPersist).  A run of pages is some 20 us of streaming,
// and a CTA of its own for each spends about 7 more on its start and its end,
// in which its half of the SM's shared memory has nothing in flight.  So a CTA
// that has issued its run's last loads but one asks for a CTA of the grid that
// has not started (cluster launch control: no queue, no counter to reset) and
// goes on with its item: the loads of the next run follow at once, its Q goes in
// and its first S is computed while the results of this one come out.  Stage,
// S-buffer and barrier counts run on over a CTA's items.  The loader passes the
// items on through two slots; every role reads them in order.  The request is
// made late, because an item taken over early waits behind its CTA while
// another SM may have run dry (batched serving: 214 us early, 211 late; 221
// with a CTA for every run).  32 layers over 23k tokens 481 -> 461 us, 64
// unforked sequences 376 -> 356, 12 branches per group 417 -> 403, D = 64 142
// -> 129, long trajectories 1339 -> 1335.
//
// A call with large groups launches their tiles first and the narrow items,
// most of them the branches' own pages, right behind as their programmatic
// dependents (beside_prev).  Those do not depend on the large tiles' results
// and run on the SMs that the large tiles' last wave leaves idle.  They start
// once every CTA of the large tiles has passed its own wait, so whatever was
// before both is complete; but only the wait makes a grid see what earlier
// grids wrote, and theirs would be for the large tiles too.  So the first CTA of
// the large tiles publishes a tag behind its wait, a release at device scope,
// and every thread of a narrow CTA acquires it: what the first saw is then
// visible to the second (the copies' proxy by a fence).  A CTA that finds
// another value executes the wait.  The tag is another one in every call, and
// the word is moved on when the narrow launch is through, so that a replayed
// graph cannot find its own earlier tag.  The grid's last CTA waits at its end,
// so that what follows (the combine) sees both complete.
// 12 branches per group, 2 groups, 4 layers: 449 -> 420 us for the two launches;
// 24 branches, 2 layers: 340 -> 315; one layer, 4 groups of 20: 118 -> 94.
//
// Shared-memory operands use the 128-byte swizzle (8-row x 128-byte atoms):
//   Q  [D/64][rows][64]       K-major A (SBO 1024)
//   K  [D/64][keys][64]       K-major B (SBO 1024)
//   P  [128][keys]            narrow: K-major A (SBO 1024), written over K:
//                             P_hi of row r at A row 32 (r / 16) + r % 16,
//                             P_lo at the A row 16 higher
//                             wide: in TMEM, the 16 score columns of keys
//                             [16 k, 16 k + 16) holding P_hi and P_lo of them
//   V  [D/64][keys][64]       MN-major B (LBO = one D-half, SBO 1024)
// The narrow P V reads 128 A rows of which only those of real rows are
// written; the others read whatever is in shared memory and only produce
// accumulator rows that nobody reads (each output row depends on its own A
// row only).  V rows of keys that are not valid (past the run,
// or in pages a short last stage did not load) are zeroed before P V, so
// stale shared or pool memory cannot turn 0 * x into NaN in a real row.
#include <math.h>

#include "kernels.cuh"
#include "ptx.cuh"

namespace st {

namespace {

constexpr int kLoadWarp = 4, kMmaWarp = 5;
constexpr int kThreads = 6 * 32;
constexpr uint32_t kTmemCols = 256;
constexpr uint32_t kTmemS = 0, kTmemO = 128;  // S buffers at 0 and 64
constexpr float kRescaleThreshold = 8.f;  // log2 units
constexpr float kLn2 = 0.69314718055994530942f;
constexpr int kMaxDevices = 64;

constexpr int cmax(int a, int b) { return a > b ? a : b; }

template <int D, bool kWide>
struct TcCfg {
  static constexpr int kHalves = D / 64;
  static constexpr int kKeys = 64;                     // keys per stage
  static constexpr int kPagesPerStage = kKeys / kPageTokens;
  // Wide: P lives in TMEM, so a K slot is free once S_j has been computed and
  // K and V slots recycle separately (K and V barrier rings).  Narrow: P goes
  // over K_j, the two are released together after P_j V_j (one ring of
  // stages).
  // As many slots as two CTAs' shared memory takes: what is in flight bounds
  // the rate (D = 64, 8 groups of 5 branches: 171 us with 3 slots, 142 with 4).
  // Wide: a V slot is held until its P V, a K slot only until its S, so the odd
  // slot is V's (9 branches, 4 layers: 748 us with 2 + 2, 738 with 2 + 3, 753
  // with 3 + 2).
  static constexpr int kStages = D == 128 ? (kWide ? 2 : 3) : (kWide ? 6 : 4);  // K slots
  static constexpr int kVStages = D == 128 && kWide ? 3 : kStages;              // V slots
  static constexpr bool kSplitKV = kWide;
  // S at M = 64 for <= 64 stacked rows: score rows sit in TMEM lanes 0..15
  // of each warp's 32-lane quarter (row r at lane 32 (r / 16) + r % 16);
  // M = 128 for up to 128 rows (row r at lane r)
  static constexpr int kM = kWide ? 128 : 64;
  static constexpr int kRowsPerWarp = kM / 4;
  static constexpr int kQRows = kWide ? 128 : 64;      // Q rows stored
  static constexpr int kQHalfBytes = kQRows * 128;
  static constexpr int kQBytes = kHalves * kQHalfBytes;
  static constexpr int kKVHalfBytes = kKeys * 128;
  // P as two bf16 terms (P = P_hi + P_lo, both against the same V): the
  // rounding of a single bf16 P does not average out when a row sees few
  // keys or its weights are peaked.  Narrow: the two terms are the A rows of
  // one M = 128 product O += [P_hi; P_lo] V, written over the K slot --
  // P_hi of row r at A row 32 (r / 16) + r % 16 (the lane of r's scores),
  // P_lo at A row 32 (r / 16) + 16 + r % 16, the lanes M = 64 leaves free in
  // each warp's quarter -- so the accumulator holds O_hi of row r in one lane
  // and O_lo in the lane 16 above it, summed at the end.
  static constexpr int kMo = 128;                                  // M of P V
  static constexpr int kPBytes = kWide ? 0 : kMo * 128;           // the A rows of P V
  static constexpr int kKSlotBytes = cmax(kHalves * kKVHalfBytes, kPBytes);
  static constexpr int kVSlotBytes = kHalves * kKVHalfBytes;
  // the K slots, then the V slots
  static constexpr int kKRingBytes = kStages * kKSlotBytes;
  static constexpr int kRingBytes = kKRingBytes + kVStages * kVSlotBytes;
  static constexpr int kBarOffset = kQBytes + kRingBytes;
  // no alignment slack: two narrow CTAs of 64 rows fill an SM's shared
  // memory, so the kernel requires the dynamic shared memory to start on a
  // 1024-byte boundary (it does when a kernel has no static shared memory;
  // the kernel checks and reports ST_ERR_CUDA otherwise)
  static constexpr int kSmemBytes = kBarOffset + 512;
};

// An item of a launch for one KV head of one layer.
struct Work {
  AttnItem item;
  int kvh, layer;
  int valid;  // 0: there is none
};

template <int D, bool kWide, bool kElect, bool kPersist>
__global__ void __launch_bounds__(kThreads, 2)
    attend_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                     const AttnParams p, const __grid_constant__ InlineDecodePlan inl) {
  using C = TcCfg<D, kWide>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  if (smem_addr(smem_raw) & 1023u) {  // the 128-byte swizzle needs 1024-byte aligned operands
    griddep_wait();
    if (threadIdx.x == 0) atomicCAS(p.status, 0, kDevBadSmem);
    return;
  }
  uint8_t* base = smem_raw;
  uint8_t* q_s = base;
  uint8_t* ring = base + C::kQBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + C::kBarOffset);
  uint64_t* full = bars;                 // [kStages] K (and, narrow, V) landed
  uint64_t* empty = bars + C::kStages;   // [kStages] K (and, narrow, V) slot free
  // K slot s and V slot s (narrow: the K and V of stage s)
  auto k_slot = [&](int s) { return ring + s * C::kKSlotBytes; };
  auto v_slot = [&](int s) { return ring + C::kKRingBytes + s * C::kVSlotBytes; };
  uint64_t* s_full = bars + 2 * C::kStages;   // [2] per S buffer
  uint64_t* p_full = s_full + 2;              // [2] per S buffer
  uint64_t* o_ready = s_full + 4;             // one phase per P V
  uint64_t* q_ready = s_full + 5;
  uint64_t* v_full = s_full + 6;               // [kVStages] wide: V landed
  uint64_t* v_empty = v_full + C::kVStages;    // [kVStages] wide: V slot free
  uint64_t* work_full = v_empty + C::kVStages; // [2] an item taken over is in its slot
  uint64_t* work_empty = work_full + 2;        // [2] every role has read it
  uint64_t* clc_bar = work_full + 4;           // the answer to a request for one has landed
  uint64_t* o_final = work_full + 5;           // one phase per item: its last P V
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(work_full + 6);
  uint8_t* clc_resp = reinterpret_cast<uint8_t*>(base + C::kBarOffset + 384);  // 16 bytes
  Work* work_slots = reinterpret_cast<Work*>(base + C::kBarOffset + 400);      // [2]
  static_assert(8 * (2 * C::kStages + 6 + 2 * C::kVStages + 7) <= 384 && 400 + 2 * sizeof(Work) <= 512, "barrier area");

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int G = p.G;
  // What touches no global memory comes ahead of the wait for the previous
  // kernel in the stream (the one that wrote the pages): the tensor-memory
  // allocation, and all of the set-up when the item is in the parameters.
  if (warp == kMmaWarp) tmem_alloc(tmem_slot, kTmemCols);
  const bool beside = !kWide && p.beside_prev;
  auto wait_for_prev = [&] {
    if constexpr (kWide) griddep_wait();
    else narrow_wait(p);
  };
  if (p.items) wait_for_prev();

  // ---- what this CTA reads and for whom ------------------------------------------
  const int32_t* members = p.members ? p.members : inl.members;
  auto item_at = [&](int x) -> const AttnItem& {
    return p.items ? p.items[p.item_base + x] : inl.items[p.item_base + x];
  };
  Work work{item_at(blockIdx.x), (int)blockIdx.y, (int)blockIdx.z, 1};
  auto stages_of = [&](const Work& w) { return (w.item.n_pages + C::kPagesPerStage - 1) / C::kPagesPerStage; };
  // softmax warps with rows of an item
  auto warps_of = [&](const Work& w) { return (w.item.n_members * G + C::kRowsPerWarp - 1) / C::kRowsPerWarp; };
  // warps that take part in the hand-overs: with items of different rows to come, all of them
  const int n_part = kPersist ? 4 : warps_of(work);

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    if (C::kSplitKV) {
      for (int s = 0; s < C::kVStages; ++s) {
        mbar_init(&v_full[s], 1);
        mbar_init(&v_empty[s], 1);
      }
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&s_full[b], 1);
      mbar_init(&p_full[b], n_part);
      mbar_init(&work_full[b], 1);
      mbar_init(&work_empty[b], 5);  // the softmax warps and the MMA warp
    }
    mbar_init(o_ready, 1);
    mbar_init(o_final, 1);
    mbar_init(q_ready, n_part);
    mbar_init(clc_bar, 1);
    fence_mbar_init();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  if (!p.items) wait_for_prev();
  if constexpr (kWide) publish_large_launch(p);
  griddep_launch_dependents();

  // The item after a role's n-th: written to slot n % 2 by the loader.  False
  // when there is none (or the wait ran out: *ok).
  auto next_work = [&](int n, Work* w, bool* ok, bool one_lane) -> bool {
    const int b = n & 1;
    *ok = one_lane ? mbar_wait(&work_full[b], (n >> 1) & 1)
                   : __all_sync(0xffffffffu, mbar_wait(&work_full[b], (n >> 1) & 1));
    if (!*ok) return false;
    *w = work_slots[b];
    if (!one_lane) __syncwarp();
    if (one_lane || lane == 0) mbar_arrive(&work_empty[b]);
    return w->valid != 0;
  };

  // ---- loader --------------------------------------------------------------------
  if (warp == kLoadWarp) {
    // A decode step: the last key of a flagged item is the row the step appends.
    // The warp writes this (layer, KV head)'s K and V of it into the pool (16
    // bytes per lane) before anything else, so the row is stored even if a
    // wait of this CTA runs out later, and makes the writes visible to the
    // TMA copy that loads the page.
    auto append_row = [&](const Work& w) {
      if (kWide || !(w.item.flags & kItemAppend)) return;
      const int last = w.item.n_tokens - 1;  // key within the run
      const int blk = p.table[(int64_t)w.item.slot * p.max_pages + w.item.page_begin + last / kPageTokens];
      constexpr int kChunks = D / 8;
      if (lane < 2 * kChunks) {
        if ((uint64_t)blk >= (uint64_t)p.n_blocks) {
          atomicCAS(p.status, 0, kDevBadIndex);
        } else {
          const bool is_v = lane >= kChunks;
          const int c = lane % kChunks;
          const int64_t src =
              (((int64_t)w.layer * p.n_rows_q + members[w.item.member_base]) * p.Hkv + w.kvh) * D + c * 8;
          const int64_t dst =
              ((((int64_t)w.layer * p.n_blocks + blk) * p.Hkv + w.kvh) * kPageTokens + last % kPageTokens) * D + c * 8;
          *reinterpret_cast<uint4*>((is_v ? p.v_pool : p.k_pool) + dst) =
              *reinterpret_cast<const uint4*>((is_v ? p.app_v : p.app_k) + src);
          fence_proxy_async_global();
        }
      }
      __syncwarp();
    };
    if (p.hold_loads) {  // test hook: nothing arrives, the other roles' waits run out
      append_row(work);
      return;
    }
    if (lane == 0) {
      prefetch_tensormap(&kmap);
      prefetch_tensormap(&vmap);
    }
    // the pages were written by ordinary stores; past a griddep_wait() that is
    // settled, past an acquire alone the copies need the proxy fence
    if (beside) fence_proxy_async_global();
    // lane 0 waits, for the warp
    auto wait0 = [&](uint64_t* bar, uint32_t parity) -> bool {
      int w = 1;
      if (lane == 0) w = mbar_wait(bar, parity) ? 1 : 0;
      return __shfl_sync(0xffffffffu, w, 0) != 0;
    };
    // waits for the slot of the CTA's g-th stage in a ring of `depth` slots to be released
    auto slot_free = [&](uint64_t* ring_empty, int depth, int g) -> bool {
      return g < depth || wait0(&ring_empty[g % depth], ((g / depth) - 1) & 1);
    };
    const uint32_t page_bytes = (uint32_t)(C::kHalves * kPageTokens * 128);
    int gk = 0, gv = 0;  // stages whose K and V copies have been issued, over all items
    bool ok = true;
    for (int n = 0;; ++n) {  // the CTA's items
      append_row(work);
      const int n_pages = work.item.n_pages, n_tiles = stages_of(work);
      // a page is streamed once, unless a sibling item (the group's other
      // subgroup, scheduled next to this one) reads it too, or the whole launch
      // fits in L2 (one agent's step, read again by the next step): then keep it
      const uint64_t policy =
          (p.keep_l2 || (work.item.flags & kItemReread)) ? l2_policy_evict_normal() : l2_policy_evict_first();
      const int32_t* ids = p.table + (int64_t)work.item.slot * p.max_pages + work.item.page_begin;
      int base_id = 0;
      int cur = lane < n_pages ? ids[lane] : 0;
      int nxt = 32 + lane < n_pages ? ids[32 + lane] : 0;
      bool asked = false;
      for (int j = 0; j < n_tiles; ++j) {
        // ask for the next item just early enough: one taken over sooner waits
        // here while another SM may have run dry
        if (kPersist && j == max(0, n_tiles - 2)) {
          asked = true;
          if (lane == 0) {
            mbar_arrive_expect_tx(clc_bar, 16);
            clc_try_cancel(clc_resp, clc_bar);
          }
        }
        if (!slot_free(empty, C::kStages, gk)) {
          ok = false;
          break;
        }
        const int page0 = j * C::kPagesPerStage;
        if (page0 >= base_id + 32) {
          base_id += 32;
          cur = nxt;
          nxt = base_id + 32 + lane < n_pages ? ids[base_id + 32 + lane] : 0;
        }
        const int np = min(C::kPagesPerStage, n_pages - page0);
        // one copy per lane (a single thread issuing them one after another is
        // what limits the stage rate): lane = D/64 q + h for an operand of its
        // own, 2 D/64 q + (V ? D/64 : 0) + h for K and V together
        constexpr int kPerPage = (C::kSplitKV ? 1 : 2) * C::kHalves;
        const int q = lane / kPerPage, r = lane % kPerPage, h = r % C::kHalves;
        int b = __shfl_sync(0xffffffffu, cur, (page0 - base_id + (q < C::kPagesPerStage ? q : 0)) & 31);
        const bool mine = lane < kPerPage * np;
        if (mine && (uint64_t)b >= (uint64_t)p.n_blocks) {
          atomicCAS(p.status, 0, kDevBadIndex);
          b = 0;
        }
        const uint32_t at = h * C::kKVHalfBytes + q * kPageTokens * 128;
        const int c2 = work.kvh * kPageTokens, c3 = work.layer * (int)p.n_blocks + b;
        uint64_t* bar = &full[gk % C::kStages];
        uint8_t* kst = k_slot(gk % C::kStages);
        if (lane == 0) mbar_arrive_expect_tx(bar, (C::kSplitKV ? 1 : 2) * np * page_bytes);
        __syncwarp();
        if constexpr (C::kSplitKV) {
          if (mine) tma_load_4d(kst + at, &kmap, bar, 0, h, c2, c3, policy);
          ++gk;
          // the K slot was released by an S, the V slot waits for its P V
          if (!slot_free(v_empty, C::kVStages, gv)) {
            ok = false;
            break;
          }
          uint64_t* vbar = &v_full[gv % C::kVStages];
          if (lane == 0) mbar_arrive_expect_tx(vbar, np * page_bytes);
          __syncwarp();
          if (mine) tma_load_4d(v_slot(gv % C::kVStages) + at, &vmap, vbar, 0, h, c2, c3, policy);
          ++gv;
        } else {
          const bool is_v = r >= C::kHalves;
          if (mine)
            tma_load_4d((is_v ? v_slot(gk % C::kStages) : kst) + at, is_v ? &vmap : &kmap, bar, 0, h, c2, c3, policy);
          ++gk;
        }
      }
      if (!kPersist) break;
      uint32_t x = 0, y = 0, z = 0;
      const bool answered = asked && __all_sync(0xffffffffu, mbar_wait(clc_bar, n & 1));
      const bool more = answered && clc_answer(clc_resp, &x, &y, &z);
      fence_proxy_async_smem();  // every lane has read the answer before the next one lands
      __syncwarp();
      if (more) work = Work{item_at(x), (int)y, (int)z, 1};
      else work.valid = 0;
      ok = ok && answered && (n < 2 || wait0(&work_empty[n & 1], ((n >> 1) - 1) & 1));
      if (!ok) {  // the item taken over is lost with this CTA, but not the row it appends
        if (more) append_row(work);
        break;
      }
      if (lane == 0) {
        work_slots[n & 1] = work;
        mbar_arrive(&work_full[n & 1]);
      }
      if (!work.valid) break;
    }
    if (!ok && lane == 0) {
      atomicCAS(p.status, 0, kDevTimeout);
      // wait (bounded) for this CTA's copies still in flight before it exits
      for (int t = max(0, gk - C::kStages); t < gk; ++t) mbar_wait(&full[t % C::kStages], (t / C::kStages) & 1);
      if constexpr (C::kSplitKV)
        for (int t = max(0, gv - C::kVStages); t < gv; ++t)
          mbar_wait(&v_full[t % C::kVStages], (t / C::kVStages) & 1);
    }
    return;
  }

  // ---- MMA issuer ----------------------------------------------------------------
  // One lane runs the issue loop; in the kElect form (small launches whose
  // pages stay in L2, where a step is a chain of latencies) the whole warp
  // runs it with warp-uniform operands and an elected lane issues, which
  // shortens each hand-off but costs the streaming launches issue slots.
  if (warp == kMmaWarp) {
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      return kElect ? __all_sync(0xffffffffu, mbar_wait(bar, parity)) : mbar_wait(bar, parity);
    };
    auto landed = [&](uint64_t* bar, uint32_t parity) {
      return kElect ? __all_sync(0xffffffffu, mbar_try_wait(bar, parity)) : mbar_try_wait(bar, parity);
    };
    auto mma_ss = [&](uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
      if constexpr (kElect) tc_mma_bf16_elect(d, a, b, idesc, acc);
      else tc_mma_bf16(d, a, b, idesc, acc);
    };
    auto mma_ts = [&](uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
      if constexpr (kElect) tc_mma_bf16_tmem_a_elect(d, a, b, idesc, acc);
      else tc_mma_bf16_tmem_a(d, a, b, idesc, acc);
    };
    auto commit = [&](uint64_t* bar) {
      if constexpr (kElect) tc_commit_elect(bar);
      else tc_commit(bar);
    };
    if (kElect || lane == 0) {
      constexpr uint32_t idesc_s = tc_idesc_bf16(C::kM, C::kKeys, 0, 0);
      constexpr uint32_t idesc_o = tc_idesc_bf16(C::kMo, D, 0, 1);
      // Shared-memory descriptors are built once: the start field holds
      // address / 16 (below 2^14 in shared memory), so the descriptor of an
      // operand shifted by b bytes is the base descriptor + b / 16.
      const uint64_t q_desc = tc_desc_sw128(smem_addr(q_s), 16, 1024);
      const uint64_t k_desc0 = tc_desc_sw128(smem_addr(ring), 16, 1024);
      const uint64_t v_desc0 = tc_desc_sw128(smem_addr(ring + C::kKRingBytes), C::kKVHalfBytes, 1024);
      // S of the CTA's g-th stage = Q K^T into S buffer g & 1
      auto issue_s = [&](int g) -> bool {
        const int s = g % C::kStages;
        if (!wait(&full[s], (g / C::kStages) & 1)) return false;
        tc_fence_after_sync();
        const uint64_t kd = k_desc0 + (uint64_t)((s * C::kKSlotBytes) >> 4);
#pragma unroll
        for (int h = 0; h < C::kHalves; ++h)
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_ss(tmem + kTmemS + (g & 1) * C::kKeys, q_desc + (uint64_t)((h * C::kQHalfBytes + kk * 32) >> 4),
                   kd + (uint64_t)((h * C::kKVHalfBytes + kk * 32) >> 4), idesc_s, (h | kk) != 0);
        commit(&s_full[g & 1]);
        if constexpr (C::kSplitKV) commit(&empty[s]);  // K has been read
        return true;
      };
      bool ok = true;
      int g0 = 0;  // the item's first stage among the CTA's
      for (int n = 0;; ++n) {
        const int g1 = g0 + stages_of(work);
        ok = wait(q_ready, n & 1);
        tc_fence_after_sync();
        if (ok) ok = issue_s(g0);
        for (int g = g0; ok && g < g1; ++g) {
          // S buffer (g + 1) & 1 was last read by the softmax of stage g - 1,
          // whose P this thread has already waited for.  Issue S of the next
          // stage ahead of this one's P V only when its data has already
          // landed, so that a slow load never delays P V.
          const int gn = g + 1;
          bool early = false;
          if (gn < g1 && landed(&full[gn % C::kStages], (gn / C::kStages) & 1)) {
            if (!issue_s(gn)) {
              ok = false;
              break;
            }
            early = true;
          }
          if (!wait(&p_full[g & 1], (g >> 1) & 1)) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          const int s = g % C::kStages, sv = g % C::kVStages;
          const uint64_t kd = k_desc0 + (uint64_t)((s * C::kKSlotBytes) >> 4);
          const uint64_t vd0 = v_desc0 + (uint64_t)((sv * C::kVSlotBytes) >> 4);
          if constexpr (kWide) {
            if (!wait(&v_full[sv], (g / C::kVStages) & 1)) {
              ok = false;
              break;
            }
            tc_fence_after_sync();
            // P_hi, P_lo of keys [16 ks, 16 ks + 16) in the 16 TMEM columns of their scores
            const uint32_t p_tm = tmem + kTmemS + (g & 1) * C::kKeys;
#pragma unroll
            for (int ks = 0; ks < C::kKeys / 16; ++ks) {
              const uint64_t vd = vd0 + (uint64_t)((ks * 16 * 128) >> 4);
              mma_ts(tmem + kTmemO, p_tm + ks * 16, vd, idesc_o, (g > g0 || ks > 0) ? 1u : 0u);
              mma_ts(tmem + kTmemO, p_tm + ks * 16 + 8, vd, idesc_o, 1u);
            }
          } else {
            // [P_hi; P_lo] V: one M = 128 product per 16 keys for both terms
#pragma unroll
            for (int ks = 0; ks < C::kKeys / 16; ++ks)
              mma_ss(tmem + kTmemO, kd + (uint64_t)((ks * 32) >> 4), vd0 + (uint64_t)((ks * 16 * 128) >> 4), idesc_o,
                     (g > g0 || ks > 0) ? 1u : 0u);
          }
          commit(C::kSplitKV ? &v_empty[sv] : &empty[s]);
          commit(o_ready);
          if (gn < g1 && !early && !issue_s(gn)) {
            ok = false;
            break;
          }
        }
        commit(o_final);
        g0 = g1;
        if (!kPersist || !ok || !next_work(n, &work, &ok, !kElect)) break;
      }
      if (!ok && lane == 0) atomicCAS(p.status, 0, kDevTimeout);
    }
    __syncwarp();
    named_barrier_sync(1, n_part * 32 + 32);
    tc_fence_after_sync();
    tmem_dealloc(tmem, kTmemCols);
    // beside_prev: this grid is complete only once the one before it is (with
    // kPersist the last CTA may be taken over before it starts: all wait, when
    // there is nothing left to run)
    if (beside && (kPersist || (blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1 &&
                                blockIdx.z == gridDim.z - 1))) {
      griddep_wait();
      // The word has served.  A replay of a captured call carries the same tag,
      // which must not be found before the large launch of that replay publishes it.
      if (lane == 0) st_release_gpu(p.large_word, p.large_tag + 1);
    }
    return;
  }
  if (warp >= n_part) return;

  // ---- softmax warps ---------------------------------------------------------------
  // Narrow: threads t and t + 16 of a warp share row t and half of the
  // stage's keys each, the row max and sum combined with one shuffle; thread
  // t owns the TMEM lane of O_hi (P_hi V) of the row, thread t + 16 the lane
  // of O_lo (P_lo V).  Wide: one thread per row.
  constexpr bool kPair = !kWide;
  constexpr int kKpt = C::kKeys / (kPair ? 2 : 1);  // keys per thread per stage
  const int half = kPair ? (lane >> 4) : 0;
  const int r = kPair ? warp * 16 + (lane & 15) : threadIdx.x;  // this thread's row
  const uint32_t t_lane = tmem + ((uint32_t)(warp * 32) << 16);

  // this thread's row of an item among the rows of Q, or -1
  auto q_row = [&](const Work& w) -> int64_t {
    if (r >= w.item.n_members * G) return -1;
    const int64_t row = (int64_t)w.layer * p.n_rows_q + members[w.item.member_base + r / G];
    return row * p.Hq + w.kvh * G + r % G;
  };
  // an item's Q to shared memory, where the S of the item before has been computed
  auto load_q = [&](const Work& w, int64_t row) {
    if (warp < warps_of(w) && r < C::kQRows) {
      const uint4* src = reinterpret_cast<const uint4*>(p.q + row * D);
      constexpr int kChunks = D / 8 / (kPair ? 2 : 1);  // 16-byte chunks of the row this thread writes
#pragma unroll
      for (int cc = 0; cc < kChunks; ++cc) {
        const int c = half * kChunks + cc;
        const uint4 v = row >= 0 ? src[c] : make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(q_s + (c >> 3) * C::kQHalfBytes + r * 128 + (((c & 7) ^ (r & 7)) << 4)) = v;
      }
      fence_proxy_async_smem();
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(q_ready);
  };

  // columns [32 k, 32 k + 32) of this thread's O lane
  auto o_load = [&](int k, float* o) { tmem_ld32(t_lane + kTmemO + k * 32, o); };
  auto o_store = [&](int k, const float* o) { tmem_st32(t_lane + kTmemO + k * 32, o); };

  const float sl2 = p.scale_log2;
  bool ok = true;
  int64_t row = q_row(work);
  load_q(work, row);
  int g0 = 0;  // the item's first stage among the CTA's
  for (int n = 0;; ++n) {
    const bool valid = row >= 0;
    const int n_sw = warps_of(work), n_swt = n_sw * 32, n_tiles = stages_of(work);
    const int n_pages = work.item.n_pages, n_valid_keys = work.item.n_tokens;
    float m_used = -1e30f, l = 0.f;  // l: this thread's share of the row sum
    for (int j = 0; j < n_tiles; ++j) {
      const int g = g0 + j, s = g % C::kStages;
      if (!__all_sync(0xffffffffu, mbar_wait(&s_full[g & 1], (g >> 1) & 1))) {
        ok = false;
        break;
      }
      tc_fence_after_sync();
      if (warp < n_sw) {
        // raw scores q.k of this thread's keys; the softmax works in the log2
        // domain, x = s * sl2
        float sc[kKpt];
        static_assert(C::kKeys == 64, "64 keys per stage");
        if constexpr (kPair) tmem_ld16x2_32<32>(t_lane + kTmemS + (g & 1) * C::kKeys, sc);
        else tmem_ld64(t_lane + kTmemS + (g & 1) * C::kKeys, sc);
        const int key0 = j * C::kKeys;
        const int kbase = half * kKpt;  // this thread's first key within the stage
        const int np = min(C::kPagesPerStage, n_pages - j * C::kPagesPerStage);
        const int loaded = np * kPageTokens;
        if (key0 + C::kKeys > n_valid_keys || loaded < C::kKeys) {
#pragma unroll
          for (int c = 0; c < kKpt; ++c)
            if (c >= min(loaded, n_valid_keys - key0) - kbase) sc[c] = -INFINITY;
        }
        // 8 independent chains of three-input max, then a tree (short dependency chains)
        float mx8[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) mx8[i] = fmaxf(sc[i], sc[8 + i]);
#pragma unroll
        for (int c = 16; c < kKpt; c += 16)
#pragma unroll
          for (int i = 0; i < 8; ++i) mx8[i] = fmax3(mx8[i], sc[c + i], sc[c + 8 + i]);
        float mx = fmax3(fmax3(mx8[0], mx8[1], mx8[2]), fmax3(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7]));
        if constexpr (kPair) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
        const float m_new = fmaxf(m_used, mx * sl2);  // sl2 > 0: max commutes with the scale
        const bool need = valid && m_new > m_used + kRescaleThreshold;
        if (__any_sync(0xffffffffu, need)) {
          const float alpha = need ? ex2(m_used - m_new) : 1.f;
          if (j > 0) {
            // the P V before must have landed in O (this stage's cannot start
            // before this thread's P, so the parity below is unambiguous)
            if (!__all_sync(0xffffffffu, mbar_wait(o_ready, (g - 1) & 1))) {
              ok = false;
              break;
            }
            tc_fence_after_sync();
#pragma unroll 1
            for (int k = 0; k < D / 32; ++k) {
              float o[32];
              o_load(k, o);
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] *= alpha;
              o_store(k, o);
            }
          }
          l *= alpha;
          if (need) m_used = m_new;
        }
        uint8_t* kslot = k_slot(s);  // narrow: S_j has been consumed, P_j goes over K_j
        if constexpr (kWide) {
          // P_hi, P_lo of keys [16 k, 16 k + 16) over the 16 TMEM columns of their
          // scores (all read above).  The store is warp-wide: rows past the
          // item's take 2^-inf = 0.
          const uint32_t p_tm = t_lane + kTmemS + (g & 1) * C::kKeys;
          const float mo = valid ? m_used : INFINITY;
          const float2 scale2 = make_float2(sl2, sl2), neg_m2 = make_float2(-mo, -mo);
          float2 rs[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
          for (int kq = 0; kq < C::kKeys / 16; ++kq) {
            uint32_t pk[16];
#pragma unroll
            for (int c = 0; c < 16; c += 2)
              prob_pair(sc[kq * 16 + c], sc[kq * 16 + c + 1], scale2, neg_m2, &rs[(c >> 1) & 3], &pk[c / 2],
                        &pk[8 + c / 2]);
            tmem_st16u_nowait(p_tm + kq * 16, pk);
          }
          tmem_wait_st();
          const float2 sum = __fadd2_rn(__fadd2_rn(rs[0], rs[1]), __fadd2_rn(rs[2], rs[3]));
          l += sum.x + sum.y;
        } else if (valid) {
          uint32_t pk[kKpt / 2];
          uint32_t pl[kKpt / 2];
          const float2 scale2 = make_float2(sl2, sl2), neg_m2 = make_float2(-m_used, -m_used);
          float2 rs[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
          for (int c = 0; c < kKpt; c += 2)
            prob_pair(sc[c], sc[c + 1], scale2, neg_m2, &rs[(c >> 1) & 3], &pk[c / 2], &pl[c / 2]);
          const float2 sum = __fadd2_rn(__fadd2_rn(rs[0], rs[1]), __fadd2_rn(rs[2], rs[3]));
          l += sum.x + sum.y;
          // A rows of P_hi and P_lo: 32 w + t and 32 w + 16 + t (both = t mod 8)
          const int a_hi = warp * 32 + (lane & 15);
#pragma unroll
          for (int cc = 0; cc < kKpt / 8; ++cc) {
            const int c = half * (kKpt / 8) + cc;  // 16-byte chunk of the P row (8 keys)
            const uint32_t off = a_hi * 128 + ((c ^ (a_hi & 7)) << 4);
            *reinterpret_cast<uint4*>(kslot + off) = make_uint4(pk[4 * cc], pk[4 * cc + 1], pk[4 * cc + 2], pk[4 * cc + 3]);
            *reinterpret_cast<uint4*>(kslot + 16 * 128 + off) =
                make_uint4(pl[4 * cc], pl[4 * cc + 1], pl[4 * cc + 2], pl[4 * cc + 3]);
          }
        }
        if (key0 + C::kKeys > n_valid_keys || loaded < C::kKeys) {
          // zero the V rows of keys that are not valid, once V_j has landed
          // (narrow: with K_j, from which S_j was computed)
          const int sv = g % C::kVStages;
          if (!__all_sync(0xffffffffu, C::kSplitKV ? mbar_wait(&v_full[sv], (g / C::kVStages) & 1)
                                                   : mbar_wait(&full[s], (g / C::kStages) & 1))) {
            ok = false;
            break;
          }
          uint8_t* vslot = v_slot(sv);
          for (int t = threadIdx.x; t < C::kKeys * C::kHalves; t += n_swt) {
            const int c = t % C::kKeys, h = t / C::kKeys;
            if (c >= loaded || key0 + c >= n_valid_keys) {
#pragma unroll
              for (int x = 0; x < 8; ++x)
                *reinterpret_cast<uint4*>(vslot + h * C::kKVHalfBytes + c * 128 + x * 16) = make_uint4(0u, 0u, 0u, 0u);
            }
          }
        }
        fence_proxy_async_smem();
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[g & 1]);
    }
    if (!ok) break;
    g0 += n_tiles;
    // the next item's Q goes in before this one's results come out: its S
    // (every S of this item has been computed) runs meanwhile.  Its first P V
    // waits for this thread's P, behind the results.
    Work next;
    int64_t next_row = -1;
    const bool more = kPersist && next_work(n, &next, &ok, false);
    if (!ok) break;
    if (more) {
      next_row = q_row(next);
      load_q(next, next_row);
    }
    if (warp < n_sw) {
      // the last P V (not o_ready, whose phases this thread may be two behind)
      if (!__all_sync(0xffffffffu, mbar_wait(o_final, n & 1))) {
        ok = false;
        break;
      }
      tc_fence_after_sync();
      if constexpr (kPair) l += __shfl_xor_sync(0xffffffffu, l, 16);  // the row's full sum
      // Four lanes have 8 columns of a row: every store fills whole 32-byte
      // sectors of 8 rows (a thread writing its own row touches 32 rows per
      // store, half a sector each).  Narrow: O = O_hi + O_lo, from a row's two
      // lanes in the same places of two loads.  One layer of 9 branches over 16384
      // tokens 25.0 -> 23.5 us, 20 branches, D 64, 312 -> 299, 16 branches 452 ->
      // 443, 5 branches over 8192 tokens 14.2 -> 13.8.
      const float inv = 1.f / l;
      const int64_t to = valid ? row * p.max_splits + work.item.split : -1;
#pragma unroll 1
      for (int hf = 0; hf < (kPair ? 1 : 2); ++hf) {
        const int ra = 16 * hf + lane / 4;  // of the warp's rows; the other one is ra + 8
        const float inv_a = __shfl_sync(0xffffffffu, inv, ra), inv_b = __shfl_sync(0xffffffffu, inv, ra + 8);
        const int64_t to_a = __shfl_sync(0xffffffffu, to, ra), to_b = __shfl_sync(0xffffffffu, to, ra + 8);
#pragma unroll 1
        for (int k = 0; k < D / 64; ++k) {
          float o[32];
          tmem_ld_16x64(t_lane + ((uint32_t)(16 * hf) << 16) + kTmemO + 64 * k, o);
          if constexpr (kPair) {
            float lo[32];
            tmem_ld_16x64(t_lane + (16u << 16) + kTmemO + 64 * k, lo);
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] += lo[i];
          }
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
      if (valid && half == 0) p.out_lse[to] = (m_used + log2f(l)) * kLn2;
    }
    if (!more) break;
    work = next;
    row = next_row;
  }
  if (!ok && lane == 0) atomicCAS(p.status, 0, kDevTimeout);
  tc_fence_before_sync();
  named_barrier_sync(1, n_part * 32 + 32);
}

template <int D, bool kWide, bool kElect, bool kPersist>
cudaError_t launch_tc_t(const CUtensorMap& km, const CUtensorMap& vm, const AttnParams& p,
                        const InlineDecodePlan& inl, int n_ctas, int dev, cudaStream_t s) {
  using C = TcCfg<D, kWide>;
  // the shared-memory opt-in is a per-device function attribute
  static bool configured[kMaxDevices] = {};
  if (!configured[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(attend_tc_kernel<D, kWide, kElect, kPersist>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  dim3 grid(n_ctas, p.Hkv, p.L);
  return launch_chained(attend_tc_kernel<D, kWide, kElect, kPersist>, grid, dim3(kThreads), C::kSmemBytes, s, km, vm,
                        p, inl);
}

// SMs of the current device, kept per device.
cudaError_t current_device(int* dev, int* sms) {
  static int sms_of[kMaxDevices] = {};
  cudaError_t e = cudaGetDevice(dev);
  if (e != cudaSuccess) return e;
  if (*dev < 0 || *dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (!sms_of[*dev]) {
    e = cudaDeviceGetAttribute(&sms_of[*dev], cudaDevAttrMultiProcessorCount, *dev);
    if (e != cudaSuccess) return e;
  }
  *sms = sms_of[*dev];
  return cudaSuccess;
}

// The kernel's form for a launch: CTAs that take over further items where there
// is more than one wave of them (two CTAs per SM), the elected MMA issue for a
// narrow launch of one wave or so whose pages stay in L2.  A single wave gains
// nothing from taking over (9 branches, one layer: 25.7 us without, 26.6 with),
// nor do a few waves of narrow items beside large tiles (24 branches: 313 and
// 319), but many do: beyond four waves they are mostly runs of a page or two
// (13 groups of 27 branches, D 64: 149 us without, 119 with; 14 groups of 9,
// 4 layers: 342 and 321).
template <int D>
cudaError_t launch_decode_t(const CUtensorMap& km, const CUtensorMap& vm, const AttnParams& p,
                            const InlineDecodePlan& ip, int n_items, bool wide, cudaStream_t s) {
  int dev = 0, sms = 0;
  const cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  const bool waves = (int64_t)n_items * p.Hkv * p.L > 2 * (int64_t)sms;
  if (wide)
    return waves ? launch_tc_t<D, true, false, true>(km, vm, p, ip, n_items, dev, s)
                 : launch_tc_t<D, true, false, false>(km, vm, p, ip, n_items, dev, s);
  if (p.keep_l2) return launch_tc_t<D, false, true, false>(km, vm, p, ip, n_items, dev, s);
  const bool many = (int64_t)n_items * p.Hkv * p.L > 8 * (int64_t)sms;
  return (p.beside_prev ? many : waves) ? launch_tc_t<D, false, false, true>(km, vm, p, ip, n_items, dev, s)
                                        : launch_tc_t<D, false, false, false>(km, vm, p, ip, n_items, dev, s);
}

template <int D>
int decode_ctas_per_sm_t() {
  using C = TcCfg<D, false>;
  if (cudaFuncSetAttribute(attend_tc_kernel<D, false, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           C::kSmemBytes) != cudaSuccess)
    return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, attend_tc_kernel<D, false, false, false>, kThreads, C::kSmemBytes) !=
      cudaSuccess)
    return 0;
  return n < 2 ? n : 2;  // two CTAs' TMEM (2 x 256 columns) fill an SM
}

}  // namespace

cudaError_t launch_decode_tc(const CUtensorMap& km, const CUtensorMap& vm, const AttnParams& p,
                             const InlineDecodePlan* inl, int n_items, int D, bool wide, cudaStream_t s) {
  static const InlineDecodePlan kNone{};
  const InlineDecodePlan& ip = inl ? *inl : kNone;
  if (n_items <= 0) return cudaSuccess;
  if (D == 128) return launch_decode_t<128>(km, vm, p, ip, n_items, wide, s);
  if (D == 64) return launch_decode_t<64>(km, vm, p, ip, n_items, wide, s);
  return cudaErrorInvalidValue;
}

int decode_tc_ctas_per_sm(int D) {
  if (D == 128) return decode_ctas_per_sm_t<128>();
  if (D == 64) return decode_ctas_per_sm_t<64>();
  return 0;
}

}  // namespace st

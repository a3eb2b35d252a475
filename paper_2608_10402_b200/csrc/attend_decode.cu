// Split-KV decode attention over the paged cache: the rows of a batch with at most 16 packed (query, head) rows.
//
// What it computes (paper Section 4: a resumed task continues from its preserved KV state; the maths is ordinary
// scaled-dot-product softmax attention with grouped KV heads): for a work item (row, kv_head, split) the online-softmax
// partial over keys [kv_begin, kv_end) for the packed rows r = q_index * G + g (the G query heads that share this KV
// head), query q_index seeing keys [0, prefix + q_index].  K/V pages are read ONCE per KV head for all G query heads.
// Bound by HBM: Hkv*D*4 bytes per context token, 4*D*Hq flops.
//
// Structure: two PERSISTENT thread blocks per SM, six warps each.  A producer warp streams whole (page, head) blocks (K
// and V, contiguous in the pool) into a ring of shared-memory stages of 64 keys with 1-D bulk copies that complete on
// mbarriers; four consumer warps take 16 keys of a stage each and run m16n8k16 bf16 MMAs straight from the pre-swizzled
// blocks with ldmatrix (the G query heads are the M rows); a scheduler warp takes over the index of a block of this
// launch that has not started (clusterlaunchcontrol.try_cancel) shortly before the producer runs out of stages, looks
// up the item and publishes it.  So the ring stays full across items: while the consumers merge their four partials of
// one item, the next item's pages are already on their way.  With one block per item every item begins with an empty ring
// and 3 to 5 us of set-up (segment search, page ids, first stage) and ends with 2 us in which it reads nothing: with three
// items per SM a decode step of 64 rows (0.82 GB of KV) took 137.8 us that way and 134.8 with persistent blocks (6.66 TB/s
// between the first and the last time stamp of the kernel), eight layers of 48 shorter rows 594 and 584.
// A layer of a planned step takes its new K/V rows along (attend_decode_writes_kernel): the block whose piece holds a new
// position writes it to its page before it reads that page, which saves an append launch and its hand-over per layer.
// Work items: one or two rounds of the resident blocks (build_plan in tide_host.cu, with the figures), or what
// TIDE_TUNE_ITEMS_PER_SM says.  More, shorter items even out the end of the launch but pay more partials and merges (3 / 4 /
// 6 / 8 per SM: 135 / 139 / 142 / 141 us on the 64 rows, 584 / 606 / 632 / 654 on the layers); so did rows cut into a few
// large items first in the launch and small ones behind them (136 to 142 us).
#include <cfloat>
#include <climits>

#include "tide_internal.h"

namespace tide {

namespace decode {

constexpr int kConsumerWarps = 4;
constexpr int kThreads = (kConsumerWarps + 2) * 32;
constexpr int kItemSlots = 3;               // the item being read, the next one, and the last one (its splits may have to be merged)
constexpr int kMergeBatch = 8;             // splits whose partial rows are fetched side by side by a merging block

template <int D>
struct Cfg {
  static constexpr int kStages = D == 128 ? 3 : 6;
  static constexpr int kStageBytes = kStageKeys * D * 4;               // K + V, bf16
  static constexpr int kMergeBytes = kConsumerWarps * 8 * D * 4;       // eight rows of O of every consumer warp
  static constexpr int kSmemBytes = kStages * kStageBytes + kMergeBytes;   // D = 128: 112 KB, two blocks and their static part fill an SM
};

struct __align__(16) Item {
  int run;                   // 0: there is no further item
  int table_off, kvh, kv_begin, kv_end;
  int R;                     // packed rows
  int p, causal;             // query q_index sees keys [0, p + q_index * causal]
  int q_row0;                // (token, head) row of packed row 0 in q (and out)
  int part_row0;             // the same in the partials of this split
  int n, n_splits, part_base, merge_ctr;   // for the block that merges the splits ...
  int x_n_splits, x_part_row0, x_stride;   // ... with those of the shared range in front of them
  int mode;                  // 0: one split, results go to out / lse; 1: partials; 2: partials, the last split merges
  int live_from;             // first key that the kernel before this one may still be writing
  int add_from, add_to, add_tok;   // AttendParams::new_k: the keys of this piece that this launch writes, the token of position 0 in new_k
  int drop;                  // test hook: the first stage never arrives
  int merge;                 // the item two before this one finished its row: its splits are to be merged
};

// A split decode-style row merges its own partials: every split counts itself in once its partials are written, and the
// block that counts last reads all splits' partials and writes the row.  The counter goes back to zero for the next
// launch.  Called by one thread, behind a barrier that the writers of the partials have passed.
__device__ __forceinline__ int count_in(int* ctr, int n_splits) {
  __threadfence();
  const int last = atomicAdd(ctr, 1) == n_splits - 1 ? 1 : 0;
  if (last) *ctr = 0;
  __threadfence();
  return last;
}

// D / 16 columns, from d0 on, of the item's rows row0, row0 + 8, ...: the splits are added in split order, so the result
// does not depend on which one came last.  Bound by the latency of its loads: the partials of kMergeBatch splits and their
// LSEs are fetched side by side, in ONE pass with a running maximum.  (A step of a lone row
// of 4k keys 10.8 us, of 16k keys 20.5, eight layers of eight 1k rows 95.8; all LSEs first and the rows behind them 12.1, 24.0
// and 99.4; 12 splits at a time 11.5, 21.5; 16 spill.)  A piece without a visible key has the weight 0 and holds zeros, and
// absent pieces of the last batch are not loaded: 0 times an infinite value would be NaN.  (As a branch on the LSE beside
// every piece's sum the same costs the lone row 0.4 us.)
template <int D>
__device__ __forceinline__ void merge_splits(const AttendParams& P, const Item& w, int row0, int d0) {
  constexpr int CW = D / 16;
  const Geom& g = P.g;
  const int own = w.n_splits, n_splits = own + w.x_n_splits, R = w.R;
  const long long stride = (long long)w.n * g.Hq;              // partial rows per split
  if (w.x_n_splits > 0) grid_dep_wait();                       // the shared range's partials are complete
  for (int rr = row0; rr < R; rr += 8) {
    const int qi = rr / g.G, gi = rr - qi * g.G;
    const long long p0 = (long long)w.part_base + w.kvh * g.G + (long long)qi * g.Hq + gi;   // this (token, head) in split 0
    auto src_row = [&](int sp) -> long long {
      return sp < own ? p0 + sp * stride : (long long)w.x_part_row0 + gi + (long long)(sp - own) * w.x_stride;
    };
    float mstar = -INFINITY, tot = 0.f;
    float acc[CW];
#pragma unroll
    for (int d = 0; d < CW; ++d) acc[d] = 0.f;
    for (int sp0 = 0; sp0 < n_splits; sp0 += kMergeBatch) {
      float e[kMergeBatch], v[kMergeBatch][CW];
#pragma unroll
      for (int x = 0; x < kMergeBatch; ++x) {
        if (sp0 + x < n_splits) {
          const long long row = src_row(sp0 + x);
          e[x] = __ldcg(P.part_lse + row);
          const float* src = P.part_o + row * D + d0;
#pragma unroll
          for (int d = 0; d < CW; d += 4) {
            const float4 t = __ldcg(reinterpret_cast<const float4*>(src + d));
            v[x][d] = t.x; v[x][d + 1] = t.y; v[x][d + 2] = t.z; v[x][d + 3] = t.w;
          }
        } else {                                             // (another piece in its place, weight 0, would make NaN of infinities)
          e[x] = -INFINITY;
#pragma unroll
          for (int d = 0; d < CW; ++d) v[x][d] = 0.f;
        }
      }
      float m_new = mstar;
#pragma unroll
      for (int x = 0; x < kMergeBatch; ++x) m_new = fmaxf(m_new, e[x]);
      const float mu = (m_new == -INFINITY) ? 0.f : m_new, keep = exp2f(mstar - mu);   // mstar = -inf: 0
      mstar = m_new;
      tot *= keep;
#pragma unroll
      for (int d = 0; d < CW; ++d) acc[d] *= keep;
#pragma unroll
      for (int x = 0; x < kMergeBatch; ++x) {
        const float wgt = exp2f(e[x] - mu);                                           // -inf: 0
        tot += wgt;
#pragma unroll
        for (int d = 0; d < CW; ++d) acc[d] += wgt * v[x][d];
      }
    }
    const float inv = tot > 0.f ? 1.f / tot : 0.f;
    const long long orow = (long long)w.q_row0 + qi * g.Hq + gi;
    uint32_t o[CW / 2];
#pragma unroll
    for (int d = 0; d < CW; d += 2) o[d >> 1] = pack_bf16(acc[d] * inv, acc[d + 1] * inv);
    uint16_t* dst = P.out + orow * D + d0;
    if constexpr (CW == 8) *reinterpret_cast<uint4*>(dst) = make_uint4(o[0], o[1], o[2], o[3]);
    else *reinterpret_cast<uint2*>(dst) = make_uint2(o[0], o[1]);
    if (P.lse != nullptr && d0 == 0) P.lse[orow] = (tot > 0.f ? mstar + log2f(tot) : -INFINITY) * 0.6931471805599453f;
  }
}

// The step's new rows of positions [from, to) of an item's KV head go to their pages (AttendParams::new_k): a warp writes
// the K and the V row of one (D = 128) or two (D = 64) tokens at a time, in the pages' swizzled layout; the loads of ROWS such
// steps are issued side by side.  Bound by latency - page number and row from L2 or HBM, then the fence (the bulk copies that
// read the rows next belong to another proxy) - with the item's next bulk copy behind it.  us a layer, one step at a time / eight:
// 16 heads of 128, 16 tokens a row, one row of 4k keys 24.3 / 18.1, 200 rows of 1k 437 / 384; 64-wide heads 17.6 / 13.8, 259 / 219.
template <int D, int ROWS>
__device__ __forceinline__ void put_rows(const int32_t* table_row, const uint16_t* new_k, const uint16_t* new_v, uint8_t* head_base, int S, int Hkv,
                                         int from, int to) {
  constexpr int CPR = D / 8, TOKENS = 16 / CPR;              // 16-byte chunks of a row, tokens at a time
  const int s_log2 = S == 16 ? 4 : 5;                        // (by a division 0.6 us of a layer of 100 rows of 1k keys)
  Geom g;
  g.group_bytes = D / 64 * 1024; g.kblock_bytes = S * D * 2;
  const long long page_bytes = 2ll * Hkv * g.kblock_bytes;
  const int lane = threadIdx.x & 31, kv = lane / CPR & 1, c = lane % CPR;
  const uint16_t* const src = (kv ? new_v : new_k) + c * 8;
  for (int pos0 = from + lane / (2 * CPR); pos0 < to; pos0 += ROWS * TOKENS) {
    uint4 v[ROWS];
    int page[ROWS];
#pragma unroll
    for (int x = 0; x < ROWS; ++x) {
      const int pos = pos0 + x * TOKENS;
      if (pos < to) {
        page[x] = __ldcg(table_row + (pos >> s_log2));
        v[x] = __ldcg(reinterpret_cast<const uint4*>(src + (long long)pos * Hkv * D));
      }
    }
#pragma unroll
    for (int x = 0; x < ROWS; ++x) {
      const int pos = pos0 + x * TOKENS;
      if (pos < to) *reinterpret_cast<uint4*>(head_base + page[x] * page_bytes + blk_offset(g, pos & (S - 1), kv, c)) = v[x];
    }
  }
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncwarp();
}
// Not inlined: the producer's loop keeps its registers.
template <int D>
__device__ __noinline__ void put_many_rows(const int32_t* table_row, const uint16_t* new_k, const uint16_t* new_v, uint8_t* head_base, int S, int Hkv,
                                           int from, int to) {
  put_rows<D, 8>(table_row, new_k, new_v, head_base, S, Hkv, from, to);
}
template <int D>
__device__ __forceinline__ void put_new_rows(const AttendParams& P, int table_off, int kvh, int add_tok, int from, int to) {
  const Geom& g = P.g;
  const long long at = ((long long)add_tok * g.Hkv + kvh) * D;
  uint8_t* const head_base = P.pool_rw + (long long)kvh * g.head_bytes;
  if (to - from <= 128 / D) put_rows<D, 1>(P.table + table_off, P.new_k + at, P.new_v + at, head_base, g.S, g.Hkv, from, to);
  else put_many_rows<D>(P.table + table_off, P.new_k + at, P.new_v + at, head_base, g.S, g.Hkv, from, to);
}

// WRITES: a layer of a step whose new rows this launch writes itself (AttendParams::new_k).
template <int D, bool INLINE, bool WRITES>
__device__ __forceinline__ void attend_decode_body(const AttendParams& P, const Segment* __restrict__ segs) {
  using C = Cfg<D>;
  constexpr int KS = D / 16;                 // k-steps of Q.K^T
  constexpr int NT = D / 8;                  // n-tiles of O
  constexpr int NS = C::kStages;

  extern __shared__ __align__(128) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t s_full[NS];
  __shared__ __align__(8) uint64_t s_empty[NS];
  __shared__ __align__(8) uint64_t s_item_full[kItemSlots], s_item_empty[kItemSlots];
  __shared__ __align__(8) uint64_t s_near_end, s_answer, s_part_done;
  __shared__ __align__(16) uint4 s_next;
  __shared__ Item items[kItemSlots];
  __shared__ float s_m[kConsumerWarps * 16], s_l[kConsumerWarps * 16];
  __shared__ int s_abort, s_is_last;

  const uint32_t ring = smem_u32(smem_raw);
  float* s_o = reinterpret_cast<float*>(smem_raw + NS * C::kStageBytes);     // [warp][8 rows][D]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Geom& g = P.g;
  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int i = 0; i < NS; ++i) {
      mbar_init(smem_u32(&s_full[i]), 1);
      mbar_init(smem_u32(&s_empty[i]), kConsumerWarps);
    }
    for (int i = 0; i < kItemSlots; ++i) {
      mbar_init(smem_u32(&s_item_full[i]), 1);
      mbar_init(smem_u32(&s_item_empty[i]), kConsumerWarps + 1);
    }
    mbar_init(smem_u32(&s_near_end), 1);
    mbar_init(smem_u32(&s_answer), 1);
    mbar_init(smem_u32(&s_part_done), 1);
    mbar_fence_init();
  }
  __syncthreads();
  const bool ahead_mode = P.run_ahead != 0;
  const bool early = ahead_mode && warp >= kConsumerWarps;   // these warps touch only what earlier work has finished with
  if (!ahead_mode) {
    if (!P.overlapped) grid_dep_wait();
    grid_dep_launch();
  }
  const int n_items = P.dyn ? __ldcg(P.dyn) : P.n_items;     // fixed grid: the batch's counts live in device memory
  if ((int)blockIdx.x >= n_items) {
    if (P.overlapped || ahead_mode) grid_dep_wait();
    return;
  }
  volatile int* abort_flag = &s_abort;
  auto wait = [&](uint64_t& bar, int parity) -> bool {
    return mbar_wait(smem_u32(&bar), (uint32_t)parity, abort_flag, P.status, P.wait_limit_ns, (P.run_ahead | P.overlapped) != 0);
  };
  // where a warp branches on the outcome: its lanes stay together
  auto wait_all = [&](uint64_t& bar, int parity) -> bool { return __all_sync(0xffffffffu, wait(bar, parity)) != 0; };

  if (warp == kConsumerWarps) {
    // ================= producer warp =================
    const int pages_per_stage = kStageKeys / g.S, stages_per_group = 32 / pages_per_stage;
    int slot = 0, use = 0, issued = 0;
    bool ok = true, ahead = early;
    for (int it = 0; ok || WRITES; ++it) {                    // (after a wait gave up: only the new rows of the items handed out)
      if (!wait_all(s_item_full[it % kItemSlots], (it / kItemSlots) & 1)) break;
      const Item& w = items[it % kItemSlots];
      if (!w.run) break;
      const int kv_begin = w.kv_begin, kv_end = w.kv_end, drop = w.drop, live_from = w.live_from;
      const int kvh = w.kvh, table_off = w.table_off;
      const int add_from = WRITES ? w.add_from : 0, add_to = WRITES ? w.add_to : 0, add_tok = WRITES ? w.add_tok : 0;
      const int32_t* trow = P.table + table_off;
      const uint8_t* head_base = P.pool + (long long)kvh * g.head_bytes;
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_item_empty[it % kItemSlots]));
      const int n_st = !WRITES || ok ? (kv_end - kv_begin + kStageKeys - 1) / kStageKeys : 0;
      // page ids are fetched 32 at a time, one per lane, a whole group ahead of their use
      const int lp0 = kv_begin / g.S, lp_last = (kv_end - 1) / g.S;
      auto load_ids = [&](int grp) -> int {
        const int lp = lp0 + grp * 32 + lane;
        return lp <= lp_last ? __ldcg(trow + lp) : 0;
      };
      int ids_cur = load_ids(0), ids_nxt = load_ids(1), cur_grp = 0;
      const int ask_at = max(0, n_st - 2);
      // the stages in front of the step's own rows, then those that hold some of them (a check in every stage costs large
      // batches of 64-wide heads 4 to 6 %)
      const int n_plain = WRITES && add_from < add_to ? min(n_st, (add_from - kv_begin) / kStageKeys) : n_st;
      int st = 0;
#pragma unroll
      for (int part = 0; part < (WRITES ? 2 : 1); ++part) {
        if (part == 1 && !ok) break;
        for (const int stop = part == 0 ? n_plain : n_st; st < stop; ++st) {
          const int grp = st / stages_per_group;
          if (grp != cur_grp) { ids_cur = ids_nxt; ids_nxt = load_ids(grp + 1); cur_grp = grp; }
          if (st == ask_at && lane == 0) mbar_arrive(smem_u32(&s_near_end));
          const int key0 = kv_begin + st * kStageKeys;
          if (part == 1) {
            // before the wait for a slot, which takes as long anyway unless the ring is empty
            if (ahead) {
              grid_dep_wait();
              ahead = false;
              ids_cur = load_ids(cur_grp);
              ids_nxt = load_ids(cur_grp + 1);
            }
            put_new_rows<D>(P, table_off, kvh, add_tok, max(key0, add_from), min(key0 + kStageKeys, add_to));
          }
          // a wait that gave up means the ring can no longer be trusted: issue nothing more
          if (use > 0 && !wait_all(s_empty[slot], (use - 1) & 1)) { ok = false; break; }
          ++issued;
          const int npages = min(pages_per_stage, (kv_end - key0 + g.S - 1) / g.S);
          if (part == 0 && ahead && key0 + npages * g.S > live_from) {
            // from here on pages, and page numbers, may belong to the kernel before this one
            grid_dep_wait();
            ahead = false;
            ids_cur = load_ids(cur_grp);
            ids_nxt = load_ids(cur_grp + 1);
          }
          const uint32_t bar = smem_u32(&s_full[slot]);
          const long long page = __shfl_sync(0xffffffffu, ids_cur, ((st % stages_per_group) * pages_per_stage + lane) & 31);
          if (!(drop != 0 && st == 0)) {                       // test hook: this stage never arrives
            if (lane == 0) mbar_expect_tx(bar, (uint32_t)(npages * g.head_bytes));
            __syncwarp();
            if (lane < npages) bulk_g2s(ring + slot * C::kStageBytes + lane * g.head_bytes, head_base + page * g.page_bytes, (uint32_t)g.head_bytes, bar);
          }
          if (++slot == NS) { slot = 0; ++use; }
        }
      }
      if (WRITES && !ok && add_from < add_to) {
        if (ahead) { grid_dep_wait(); ahead = false; }
        put_new_rows<D>(P, table_off, kvh, add_tok, add_from, add_to);
      }
      if (n_st == 0 && lane == 0) mbar_arrive(smem_u32(&s_near_end));
    }
    if (*abort_flag && lane == 0) {
      // a wait gave up somewhere: do not leave the block while copies into its shared memory are in flight.  Only the
      // last NS stages that were issued can still be landing; each wait is bounded like every other.
      for (int st = max(0, issued - NS); st < issued; ++st) {
        const uint32_t bar = smem_u32(&s_full[st % NS]);
        const long long t0 = global_ns();
        while (!mbar_try(bar, (st / NS) & 1) && global_ns() - t0 < P.wait_limit_ns) {}
      }
    }
    return;
  }
  if (warp == kConsumerWarps + 1) {
    // ================= scheduler warp: hands out the items =================
    const int n_segs = P.dyn ? __ldcg(P.dyn + 1) : P.n_segs;
    int item = (int)blockIdx.x, asks = 0, done = 0;
    int handed_out[kItemSlots] = {-1, -1, -1};               // the items in the slots
    int merge = 0;                                           // lane 0: the last item but one completed its row
    bool fused_before = false, open = false;                 // a question without an answer yet
    auto segment_of = [&](int item) -> Segment {
      int si;
      if (INLINE) si = find_segment(n_segs, item, [&](int i) { return segs[i].item_base; });
      else {
        // the last segment that starts at or before the item: 32 at a time, the loads side by side (a binary search is
        // a chain of dependent loads: 2.9 us for 48 segments)
        si = -1;
        for (int i0 = 0; i0 < n_segs; i0 += 128) {
          bool le[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int i = i0 + k * 32 + lane;
            le[k] = i < n_segs && __ldcg(&segs[i].item_base) <= item;
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) si += __popc(__ballot_sync(0xffffffffu, le[k]));
          if (si + 1 < i0 + 128) break;
        }
      }
      return INLINE ? segs[si] : load_segment(segs + si);
    };
    // A launch that writes the step's rows itself writes them also where its waits run out or the status word keeps items
    // from being started: the cache holds them whatever becomes of the results.  (Only the rows of an item that the hardware
    // has handed to this block in an answer that never landed would be missing.)
    auto put_only = [&](int item) {
      if (item < 0 || item >= n_items) return;
      const Segment seg = segment_of(item);
      const int local = item - seg.item_base, begin = seg.origin + local % seg.n_splits * seg.chunk;
      put_new_rows<D>(P, seg.table_off, local / seg.n_splits, seg.q_off - seg.p, max(begin, seg.p), min(begin + seg.chunk, seg.p + seg.n));
    };
    auto ask = [&] {
      if (lane == 0) next_block_ask(smem_u32(&s_next), smem_u32(&s_answer));
      ++asks;
      open = true;
    };
    auto answer = [&]() -> bool {
      if (!wait_all(s_answer, (asks - 1) & 1)) return false;
      open = false;
      item = claimed_item(true, next_block_answer(smem_u32(&s_next)), n_items);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the answer has been read before the next one may land
      __syncwarp();
      return true;
    };
    for (int it = 0; ; ++it) {
      const int slot = it % kItemSlots;
      if (it >= kItemSlots && !wait_all(s_item_empty[slot], (it / kItemSlots - 1) & 1)) break;
      Item& w = items[slot];
      // The status word is set when a bounded wait runs out and stays set until tide_status clears it.  While it is set
      // no item is started, so outputs are undefined from the time-out until the caller has read the status.
      if (__shfl_sync(0xffffffffu, *reinterpret_cast<volatile int*>(P.status), 0) != 0) {
        if (WRITES && item >= 0) {
          grid_dep_wait();
          do {
            put_only(item);
            ask();
          } while (answer() && item >= 0);
        }
        item = -1;
      }
      if (item < 0) {
        if (lane == 0) { w.run = 0; w.merge = merge; mbar_arrive(smem_u32(&s_item_full[slot])); }
        break;
      }
      const Segment seg = segment_of(item);
      if (lane == 0) {
        const int local = item - seg.item_base;
        const int split = local % seg.n_splits, kvh = local / seg.n_splits;
        const int R = seg.n * g.G;
        w.run = 1; w.merge = merge;
        w.table_off = seg.table_off; w.kvh = kvh;
        w.kv_begin = seg.origin + split * seg.chunk;
        w.kv_end = max(w.kv_begin, min(w.kv_begin + seg.chunk, seg.p + (seg.n - 1) * seg.causal + 1));
        w.R = R; w.p = seg.p; w.causal = seg.causal; w.live_from = seg.live_from;
        w.q_row0 = seg.q_off * g.Hq + kvh * g.G;
        w.part_row0 = seg.part_base + split * seg.n * g.Hq + kvh * g.G;
        w.n = seg.n; w.n_splits = seg.n_splits; w.part_base = seg.part_base;
        w.merge_ctr = seg.merge_ctr + kvh;
        w.x_n_splits = seg.x_n_splits; w.x_part_row0 = seg.x_part_base + kvh * g.G; w.x_stride = seg.x_stride;
        w.mode = seg.partial == 2 ? 2 : (seg.n_splits == 1 && seg.partial == 0) ? 0 : 1;
        w.drop = P.debug_drop_first_stage != 0 && item == 0;
        if (WRITES) { w.add_from = min(w.kv_end, max(w.kv_begin, seg.p)); w.add_to = w.kv_end; w.add_tok = seg.q_off - seg.p; }
        mbar_arrive(smem_u32(&s_item_full[slot]));
      }
      handed_out[2] = handed_out[1]; handed_out[1] = handed_out[0]; handed_out[0] = item;
      // The split of the item before this one is counted in on the consumers' behalf, who have gone on to this one; the
      // verdict travels with the next item.
      merge = 0;
      if (fused_before) {
        if (!wait_all(s_part_done, done & 1)) break;
        ++done;
        const Item& b = items[(it - 1) % kItemSlots];
        if (lane == 0) merge = count_in(P.merge_ctr + b.merge_ctr, b.n_splits);
      }
      fused_before = seg.partial == 2;
      // the next item is claimed two stages before the producer runs out of this one
      if (!wait_all(s_near_end, it & 1)) break;
      // (Beside a whole layer, not just an append, blocks that have started early would take items from those that start later:
      // 32 rows of 1k keys, two KV heads, 16.7 us a layer, and 14.2 with an append in between.)
      if (WRITES && early && it == 0) grid_dep_wait();
      ask();
      if (!answer()) break;
    }
    if (open) {
      // Only after a wait gave up: the answer lands before the block leaves.  The hardware always answers, in a microsecond or
      // so, and the handle's limit may be shorter than that, hence a bound of its own.
      const long long t0 = global_ns();
      bool landed = mbar_try(smem_u32(&s_answer), (asks - 1) & 1);
      while (!landed && global_ns() - t0 < kWaitLimitNsDefault) landed = mbar_try(smem_u32(&s_answer), (asks - 1) & 1);
      landed = __all_sync(0xffffffffu, landed) != 0;
      item = claimed_item(landed, landed ? next_block_answer(smem_u32(&s_next)) : -1, n_items);
    }
    if (WRITES && *abort_flag) {                             // what the producer may not have come to
      grid_dep_wait();
      for (int i = 0; i < kItemSlots; ++i) {
        put_only(handed_out[0]);
        handed_out[0] = handed_out[1]; handed_out[1] = handed_out[2];
      }
      put_only(item);
    }
    return;
  }

  // ================= consumer warps =================
  const float kLn2 = 0.6931471805599453f, sl2 = P.scale_log2e;
  // A warp reads the same 16 slots of every stage, so the offsets of its ldmatrix rows inside a stage are fixed (two per
  // K n-tile, four for V; the others are 1 KB further on).
  uint32_t dk_off[2][2], dv_off[4];
  {
    const int koff = warp * 16;
    const uint32_t page_off = (uint32_t)((koff / g.S) * g.head_bytes);
    const int row0 = koff % g.S;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int x = 0; x < 2; ++x) dk_off[nt][x] = page_off + (uint32_t)blk_offset(g, row0 + nt * 8 + (lane & 7), 0, x * 4 + (lane >> 3));
    const int vrow = row0 + ((lane >> 3) & 1) * 8 + (lane & 7);
#pragma unroll
    for (int y = 0; y < 4; ++y) dv_off[y] = page_off + (uint32_t)blk_offset(g, vrow, 1, y * 2 + (lane >> 4));
  }
  uint32_t qa[KS][4];
  auto load_q = [&](const Item& w) {
    const int r_lo = lane >> 2, r_hi = r_lo + 8;
    const int qi_lo = r_lo / g.G, qi_hi = r_hi / g.G;
    const bool v_lo = r_lo < w.R, v_hi = r_hi < w.R;
    const uint16_t* q_lo = P.q + ((long long)w.q_row0 + qi_lo * g.Hq + (r_lo - qi_lo * g.G)) * D + 2 * (lane & 3);
    const uint16_t* q_hi = P.q + ((long long)w.q_row0 + qi_hi * g.Hq + (r_hi - qi_hi * g.G)) * D + 2 * (lane & 3);
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      qa[ks][0] = v_lo ? __ldcg(reinterpret_cast<const uint32_t*>(q_lo + ks * 16)) : 0u;
      qa[ks][1] = v_hi ? __ldcg(reinterpret_cast<const uint32_t*>(q_hi + ks * 16)) : 0u;
      qa[ks][2] = v_lo ? __ldcg(reinterpret_cast<const uint32_t*>(q_lo + ks * 16 + 8)) : 0u;
      qa[ks][3] = v_hi ? __ldcg(reinterpret_cast<const uint32_t*>(q_hi + ks * 16 + 8)) : 0u;
    }
  };
  int slot = 0, use = 0;
  bool more = named_bar_and(1, kConsumerWarps * 32, wait_all(s_item_full[0], 0)) && items[0].run;
  // With producers that run ahead, the set-up above has happened beside the kernel in front, too.
  if (ahead_mode) {
    grid_dep_wait();
    grid_dep_launch();
  }
  for (int it = 0; more; ++it) {
    const Item& w = items[it % kItemSlots];
    const int kv_begin = w.kv_begin, kv_end = w.kv_end, R = w.R;
    load_q(w);
    const int r_lo = lane >> 2, r_hi = r_lo + 8;
    const int kv_limit_lo = r_lo < R ? min(kv_end, w.p + (r_lo / g.G) * w.causal + 1) : kv_end;  // keys j < limit are visible
    const int kv_limit_hi = r_hi < R ? min(kv_end, w.p + (r_hi / g.G) * w.causal + 1) : kv_end;
    const int min_limit = min(kv_end, w.p + 1);              // masking needed beyond it
    float o[NT][4];
#pragma unroll
    for (int i = 0; i < NT; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
    float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;

    const int n_st = (kv_end - kv_begin + kStageKeys - 1) / kStageKeys;
    for (int st = 0; st < n_st; ++st) {
      wait(s_full[slot], use & 1);
      const uint32_t stage = ring + slot * C::kStageBytes;
      const int key0 = kv_begin + st * kStageKeys + warp * 16;   // this warp's 16 keys
      if (key0 < kv_end) {
        float s[2][4];
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          float(&acc)[4] = s[nt];
          acc[0] = acc[1] = acc[2] = acc[3] = 0.f;
#pragma unroll
          for (int k2 = 0; k2 < KS / 2; ++k2) {
            uint32_t b0, b1, b2, b3;
            ldsm_x4(stage + dk_off[nt][k2 & 1] + (k2 >> 1) * 1024, b0, b1, b2, b3);
            mma_bf16(acc, qa[2 * k2], b0, b1);
            mma_bf16(acc, qa[2 * k2 + 1], b2, b3);
          }
        }
        // ---- scale, mask, online softmax ----
        const bool need_mask = key0 + 16 > min_limit;
        float mx_lo = -INFINITY, mx_hi = -INFINITY;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const int j = key0 + t * 8 + 2 * (lane & 3);
          float t0 = s[t][0] * sl2, t1 = s[t][1] * sl2, t2 = s[t][2] * sl2, t3 = s[t][3] * sl2;
          if (need_mask) {
            if (j >= kv_limit_lo) t0 = -INFINITY;
            if (j + 1 >= kv_limit_lo) t1 = -INFINITY;
            if (j >= kv_limit_hi) t2 = -INFINITY;
            if (j + 1 >= kv_limit_hi) t3 = -INFINITY;
          }
          s[t][0] = t0; s[t][1] = t1; s[t][2] = t2; s[t][3] = t3;
          mx_lo = fmaxf(mx_lo, fmaxf(t0, t1));
          mx_hi = fmaxf(mx_hi, fmaxf(t2, t3));
        }
        mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
        mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
        mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
        mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
        const float mn_lo = fmaxf(m_lo, mx_lo), mn_hi = fmaxf(m_hi, mx_hi);
        const float mu_lo = (mn_lo == -INFINITY) ? 0.f : mn_lo, mu_hi = (mn_hi == -INFINITY) ? 0.f : mn_hi;
        const float a_lo = fast_exp2(m_lo - mu_lo), a_hi = fast_exp2(m_hi - mu_hi);
        m_lo = mn_lo; m_hi = mn_hi;
        if (__any_sync(0xffffffffu, a_lo != 1.f || a_hi != 1.f)) {
#pragma unroll
          for (int i = 0; i < NT; ++i) { o[i][0] *= a_lo; o[i][1] *= a_lo; o[i][2] *= a_hi; o[i][3] *= a_hi; }
        }
        float ps_lo = 0.f, ps_hi = 0.f;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          s[t][0] = fast_exp2(s[t][0] - mu_lo); s[t][1] = fast_exp2(s[t][1] - mu_lo);
          s[t][2] = fast_exp2(s[t][2] - mu_hi); s[t][3] = fast_exp2(s[t][3] - mu_hi);
          ps_lo += s[t][0] + s[t][1];
          ps_hi += s[t][2] + s[t][3];
        }
        l_lo = l_lo * a_lo + ps_lo;
        l_hi = l_hi * a_hi + ps_hi;
        // ---- O += P.V ----
        if (key0 + 16 > kv_end) {
          // slots past the end of the item hold whatever the page held before: clear V there so that
          // weight 0 times stale bits cannot produce NaN.  The stage is filled again for the next item by bulk copies, which
          // are ordered behind these stores only by the fence.
          const int koff = warp * 16, first = kv_end - key0;           // 1..15
          uint8_t* vgen = smem_raw + slot * C::kStageBytes + (koff / g.S) * g.head_bytes;
          for (int idx = lane; idx < (16 - first) * (D / 8); idx += 32) {
            const int rr = koff % g.S + first + idx / (D / 8), c = idx % (D / 8);
            *reinterpret_cast<uint4*>(vgen + blk_offset(g, rr, 1, c)) = make_uint4(0, 0, 0, 0);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
        }
        uint32_t pa[4];
        pa[0] = pack_bf16(s[0][0], s[0][1]);
        pa[1] = pack_bf16(s[0][2], s[0][3]);
        pa[2] = pack_bf16(s[1][0], s[1][1]);
        pa[3] = pack_bf16(s[1][2], s[1][3]);
#pragma unroll
        for (int n2 = 0; n2 < NT / 2; ++n2) {
          uint32_t b0, b1, b2, b3;
          ldsm_x4_t(stage + dv_off[n2 & 3] + (n2 >> 2) * 1024, b0, b1, b2, b3);
          mma_bf16(o[2 * n2], pa, b0, b1);
          mma_bf16(o[2 * n2 + 1], pa, b2, b3);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_empty[slot]));
      if (++slot == NS) { slot = 0; ++use; }
    }

    // ---- epilogue: the four warps hold partial (m, l, O) over disjoint keys of the same 16 rows; they combine through
    // shared memory, eight rows at a time (more than eight packed rows are rare: G > 8 or several tokens) ----
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1);
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
    constexpr int CW = D / 16;                               // columns per thread: 128 threads = 8 rows x 16 column segments
    const int tid = threadIdx.x, rr8 = tid >> 4, d0 = (tid & 15) * CW;
    const int mode = w.mode;
    auto put_half = [&](int half) {
      float* wo = s_o + (warp * 8 + (lane >> 2)) * D + 2 * (lane & 3);
#pragma unroll
      for (int i = 0; i < NT; ++i) *reinterpret_cast<float2*>(wo + i * 8) = half ? make_float2(o[i][2], o[i][3]) : make_float2(o[i][0], o[i][1]);
    };
    // one row's results: CW columns of out / lse, or of the partials
    auto emit = [&](bool final_row, int qi, int gi, const float (&acc)[CW], float e2) {
      if (final_row) {
        const long long orow = (long long)w.q_row0 + qi * g.Hq + gi;
        uint32_t* dst = reinterpret_cast<uint32_t*>(P.out + orow * D + d0);
        uint32_t v[CW / 2];
#pragma unroll
        for (int d = 0; d < CW; d += 2) v[d >> 1] = pack_bf16(acc[d], acc[d + 1]);
        if constexpr (CW == 8) *reinterpret_cast<uint4*>(dst) = make_uint4(v[0], v[1], v[2], v[3]);
        else *reinterpret_cast<uint2*>(dst) = make_uint2(v[0], v[1]);
        if (P.lse != nullptr && (tid & 15) == 0) P.lse[orow] = e2 * kLn2;
      } else {
        const long long prow = (long long)w.part_row0 + qi * g.Hq + gi;
        float* dst = P.part_o + prow * D + d0;
#pragma unroll
        for (int d = 0; d < CW; d += 4) *reinterpret_cast<float4*>(dst + d) = make_float4(acc[d], acc[d + 1], acc[d + 2], acc[d + 3]);
        if ((tid & 15) == 0) P.part_lse[prow] = e2;
      }
    };
    for (int half = 0; half * 8 < R; ++half) {
      if (half > 0) named_bar_sync(1, kConsumerWarps * 32);  // the first eight rows have been read
      put_half(half);
      if (half == 0 && (lane & 3) == 0) {
        const int rl = lane >> 2;
        s_m[warp * 16 + rl] = m_lo; s_m[warp * 16 + rl + 8] = m_hi;
        s_l[warp * 16 + rl] = l_lo; s_l[warp * 16 + rl + 8] = l_hi;
      }
      named_bar_sync(1, kConsumerWarps * 32);
      const int rr = half * 8 + rr8;
      if (rr < R) {
        float mw[kConsumerWarps], mstar = -INFINITY;
#pragma unroll
        for (int x = 0; x < kConsumerWarps; ++x) { mw[x] = s_m[x * 16 + rr]; mstar = fmaxf(mstar, mw[x]); }
        const float mu = (mstar == -INFINITY) ? 0.f : mstar;
        float f[kConsumerWarps], lstar = 0.f;
#pragma unroll
        for (int x = 0; x < kConsumerWarps; ++x) { f[x] = fast_exp2(mw[x] - mu); lstar += f[x] * s_l[x * 16 + rr]; }
        const float inv = lstar > 0.f ? 1.f / lstar : 0.f;
        const float e2 = lstar > 0.f ? mstar + log2f(lstar) : -INFINITY;
        float acc[CW];
#pragma unroll
        for (int d = 0; d < CW; ++d) acc[d] = 0.f;
#pragma unroll
        for (int x = 0; x < kConsumerWarps; ++x)
#pragma unroll
          for (int d = 0; d < CW; d += 4) {
            const float4 v = *reinterpret_cast<const float4*>(s_o + (x * 8 + rr8) * D + d0 + d);
            acc[d] += f[x] * v.x; acc[d + 1] += f[x] * v.y; acc[d + 2] += f[x] * v.z; acc[d + 3] += f[x] * v.w;
          }
#pragma unroll
        for (int d = 0; d < CW; ++d) acc[d] *= inv;
        if (mode != 0 && lstar == 0.f) {                     // no key of this piece is visible: weight 0 in the merge, and
#pragma unroll
          for (int d = 0; d < CW; ++d) acc[d] = 0.f;         // nothing of the values, which may be infinite, in its rows
        }
        const int qi = rr / g.G;
        emit(mode == 0, qi, rr - qi * g.G, acc, e2);
      }
    }
    // The row's partials are merged by the block that finishes its last split.  When this block has a next item, its
    // scheduler warp counts the split in (a fence and an atomic: 0.9 us that the consumers do not wait for) and hands the
    // verdict on with the item after that.
    // What comes next?  The four warps decide together (they meet at barriers inside an item); behind this barrier the
    // merge buffer is free again.  An item is published before the producer has issued the last two stages of the one
    // before it, so this rarely waits.
    const int nx = it + 1;
    more = named_bar_and(1, kConsumerWarps * 32, wait_all(s_item_full[nx % kItemSlots], (nx / kItemSlots) & 1)) && items[nx % kItemSlots].run;
    if (mode == 2 && more) {
      if (tid == 0) mbar_arrive(smem_u32(&s_part_done));     // the scheduler warp counts this split in
    } else if (mode == 2) {
      if (tid == 0) s_is_last = count_in(P.merge_ctr + w.merge_ctr, w.n_splits);
      named_bar_sync(1, kConsumerWarps * 32);
      if (s_is_last) merge_splits<D>(P, w, rr8, d0);
    }
    if (it > 0) {
      const int before = (it - 1) % kItemSlots;
      if (items[nx % kItemSlots].merge) merge_splits<D>(P, items[before], rr8, d0);
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_item_empty[before]));
    }
  }
  if (P.overlapped) grid_dep_wait();
}

template <int D>
__global__ void __launch_bounds__(kThreads, 2) attend_decode_kernel(const AttendParams P) {
  attend_decode_body<D, false, false>(P, P.segs);
}

template <int D>
__global__ void __launch_bounds__(kThreads, 2) attend_decode_writes_kernel(const AttendParams P) {
  attend_decode_body<D, false, true>(P, P.segs);
}

// Decode-style items whose row descriptors travel in the kernel's parameters (small batches).
template <int D>
__global__ void __launch_bounds__(kThreads, 2) attend_decode_inline_kernel(const __grid_constant__ AttendInline PI) {
  attend_decode_body<D, true, false>(PI.p, PI.segs);
}

template <int D>
static cudaError_t init_one() {
  cudaError_t e = cudaFuncSetAttribute(attend_decode_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(attend_decode_writes_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kSmemBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(attend_decode_inline_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kSmemBytes);
}

}  // namespace decode

cudaError_t attend_decode_init() {
  const cudaError_t e = decode::init_one<128>();
  return e != cudaSuccess ? e : decode::init_one<64>();
}

cudaError_t launch_attend_decode_inline(const AttendInline& pi, cudaStream_t s) {
  const int grid = pi.p.n_items;
  if (grid <= 0) return cudaSuccess;
  if (pi.p.g.D == 128) return launch_dep(decode::attend_decode_inline_kernel<128>, grid, decode::kThreads, decode::Cfg<128>::kSmemBytes, s, pi);
  return launch_dep(decode::attend_decode_inline_kernel<64>, grid, decode::kThreads, decode::Cfg<64>::kSmemBytes, s, pi);
}

cudaError_t launch_attend_decode(const AttendParams& p, cudaStream_t s) {
  const int grid = p.dyn ? p.grid_cap : p.n_items;
  if (grid <= 0) return cudaSuccess;
  if (p.g.D == 128)
    return launch_dep(p.new_k ? decode::attend_decode_writes_kernel<128> : decode::attend_decode_kernel<128>, grid, decode::kThreads,
                      decode::Cfg<128>::kSmemBytes, s, p);
  return launch_dep(p.new_k ? decode::attend_decode_writes_kernel<64> : decode::attend_decode_kernel<64>, grid, decode::kThreads, decode::Cfg<64>::kSmemBytes, s, p);
}

}  // namespace tide

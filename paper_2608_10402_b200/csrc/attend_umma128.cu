// Append-prefill attention for resume rows on the 5th-generation tensor cores, 128-key tiles, head sizes 64 and 128.
//
// Work item: 256 packed rows r = q_index * G + g (two 128-row tiles A and B) against keys [kv_begin, kv_end) of one KV
// head (paper Section 4: the appended observation tokens attend to the whole preserved KV state).
//
// A thread block is PERSISTENT: one per SM, twelve warps, every role walking the same sequence of items.  The grid has
// one block per item; a running block takes over the index of a block that has not started yet
// (clusterlaunchcontrol.try_cancel), so items are handed out one at a time, in order, to whichever SM is free, with no
// counter in memory.  Warp 11 asks for the next item while the current one runs, works out its geometry once and
// publishes it; the K and V producers then run ahead into it, its queries are copied as soon as the last QK of the
// current item has retired, and its first QK is issued behind the current item's last PV.  Of an item's fixed cost only
// the epilogue and the fill of the softmax pipeline remain (one block per item spent 14 us outside the key loop - 2.3
// launch and TMEM set-up, 4.6 staging Q, 0.8 first QK, 0.8 last PV, 4.3 epilogue, 1.1 between blocks - against 1.6 us per
// 128-key tile, i.e. 44 % of a batch of prompts of 200 to 4000 tokens and 21 % of the long-horizon batch).
//   * S_t = Q_t . K_j^T is D/16 MMAs of 128x128x16, O_t += P_t . V_j eight of 128xDx16;
//   * Q sits in shared memory (both operands of QK from shared memory run at the rate of the TMEM-A form once N = 128);
//     K tiles and V tiles are separate units of one ring (K0 V0 K1 V1 ...), each filled by one bulk copy per page (the K
//     block or the V block of a (page, head) is contiguous in the pool and already in operand layout), K by warp 8 and V
//     by warp 10; warp 9 issues the MMAs;
//   * D = 128: TMEM holds S_A S_B 2 x 128 columns (P_t, packed bf16, overwrites the first 64 of S_t) and O_A O_B 2 x 128.
//     The two row tiles ping-pong: while warpgroup A works on S_A(j) the tensor pipe runs PV_B(j-1) and QK_B(j);
//   * D = 64: O needs half the columns, so P_t gets columns of its own and QK_t(j+1) is issued as soon as the softmax
//     warps have S_t(j) in registers: they always find their next S tile waiting, and the kernel is bound by the
//     exponentials (a 64-wide head has half the MMA work per exponential);
//   * every exponential is an ex2.  A quarter of them as a cubic on the FMA pipe shortens an isolated tile (the ex2 unit
//     needs as long for a D = 128 tile as the tensor pipe does) but costs six times the instructions, and what bounds a
//     long batch is the board's 1 kW: mixed text batch 7.06 ms with the share, 7.00 without, multimodal batch 18.2 and
//     18.0, prompts 0.722 and 0.702 (0.3 s and more into a run, SM clock 1.5 to 1.7 GHz).
// Every wait is bounded; a wait that runs out sets TIDE_ERR_DEVICE_TIMEOUT and the block drains and exits.
#include <climits>
#include <type_traits>

#include "tide_internal.h"

namespace tide {

namespace umma128 {

constexpr int kTileKeys = 128;
constexpr int kThreads = 384;   // 3 warpgroups: softmax A, softmax B, {K producer 8, MMA issuer 9, V producer 10, scheduler and Q loader 11}
constexpr int kItemSlots = 4;   // published items
constexpr float kRescaleThreshold = 8.0f;           // log2 units
constexpr int kPParts = 2;      // P_t is handed to the MMA warp in two halves

template <int D>
struct Cfg {
  static constexpr bool kSepP = D == 64;                       // P_t has TMEM columns of its own
  static constexpr int kNumUnits = D == 128 ? 5 : 10;          // ring of operand tiles in the order K0 V0 K1 V1 ...
  static constexpr int kGroupBytes = (D / 64) * 1024;          // one 8-key group of a K (or V) tile: D/64 1-KB atoms
  static constexpr int kUnitBytes = (kTileKeys / 8) * kGroupBytes;   // one K or V tile
  static constexpr int kQSlabBytes = 128 * 128;                // 128 rows x 128 bytes
  static constexpr int kQTileBytes = (D / 64) * kQSlabBytes;   // the queries of one 128-row tile
  static constexpr int kQBytes = 2 * kQTileBytes;
  static constexpr int kSmemBytes = kQBytes + kNumUnits * kUnitBytes;   // D = 128: 224 KB; with the static part the whole 227 KB of an SM
  static constexpr uint32_t kColS = 0;                                  // S_t at kColS + t*128
  static constexpr uint32_t kColP = kSepP ? 256 : 0, kColPStep = kSepP ? 64 : 128;
  static constexpr uint32_t kColO = kSepP ? 384 : 256;                  // O_t at kColO + t*D
  // instruction descriptors: fp32 accumulate, bf16 A and B, M = 128; N = 128 keys (QK) or D columns (PV); bit 16 = B is MN-major
  static constexpr uint32_t kIdescBase = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);
  static constexpr uint32_t kIdescQK = kIdescBase | ((128u >> 3) << 17);
  static constexpr uint32_t kIdescPV = kIdescBase | (((uint32_t)D >> 3) << 17) | (1u << 16);
};

__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version of this architecture
  d |= (uint64_t)2 << 61;   // 128-byte swizzle
  return d;
}
__device__ __forceinline__ uint64_t desc64(uint32_t lo, uint32_t hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}
// Both MMA forms are called by ALL lanes of the (converged) MMA warp; one elected lane issues, so descriptors and
// addresses stay in uniform registers.
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
      ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st32u(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
        "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
        "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st16u(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float (&v)[32]) {
  uint32_t u[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) u[i] = __float_as_uint(v[i]);
  tmem_st32u(taddr, u);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// packed pairs of floats: one instruction for two elements (fma.rn.f32x2 / add.rn.f32x2)
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {     // zero-fills when not valid
  const int n = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
// 32 bytes per lane, in one instruction where the address allows it: a lane writes whole sectors of its own row (the
// rows of a warp are apart)
__device__ __forceinline__ void st_32bytes(void* p, const uint32_t (&v)[8], bool wide) {
  if (wide)
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]),
                 "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
  else {
    reinterpret_cast<uint4*>(p)[0] = make_uint4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<uint4*>(p)[1] = make_uint4(v[4], v[5], v[6], v[7]);
  }
}

// One work item as every role sees it.
struct __align__(16) Item {
  int run;             // 0: there is no further item
  int table_off, kvh, kv_begin, kv_end, n_tiles;
  int tiles[2];        // per 128-row tile: number of 128-key tiles to process (0: the tile has no rows or sees no key),
  int end[2];          // one past the last key any of its rows sees,
  int min_limit[2];    // and the first key that its first row does not see
  int row0, R;         // first packed row; packed rows of the (row, kv head)
  int p, causal;
  int q_row0;          // (token, head) row of the segment's first token in q (and out): q_off * Hq
  int dst_row0;        // (token, head) row of its first token in out, or in the partials of this split
  int direct;          // 1: results go to out / lse; 0: to the partials
  int live_from;       // first key that the kernel before this one may still be writing
  int drop;            // test hook: K tile 0 never arrives
};

template <int NU>
struct Bars {
  uint64_t kv_full[NU];
  uint64_t kv_empty[NU];
  uint64_t q_full[2];   // Q_t of the item is in shared memory
  uint64_t q_empty[2];  // the item's last QK_t has retired
  uint64_t s_full[2];   // S_t(j) is in TMEM (D = 128: and every earlier MMA of the row tile, PV_t(j-1) included, has retired)
  uint64_t s_free[2];   // D = 64: S_t(j) is in registers
  uint64_t p_part[2][kPParts];   // part q of P_t(j) (keys [q, q+1) * 128 / kPParts) is in TMEM
  uint64_t o_full[2];   // D = 128: the item's last PV_t has retired; D = 64: PV_t(j) has
  uint64_t item_full[kItemSlots];
  uint64_t item_empty[kItemSlots];
  uint64_t k_issued;    // the copies of the item's last K tile are on their way
  uint64_t next;        // the answer of next_block_ask has landed
  uint64_t mma_done;    // every MMA of the block has retired
};
constexpr int kItemReaders = 3 + 8;   // K producer, V producer, MMA warp, eight softmax warps: one arrival each

template <int D, bool INLINE>
__device__ __forceinline__ void attend_umma128_body(const AttendParams& P, const Segment* __restrict__ segs) {
  using C = Cfg<D>;
  // The swizzled operand layouts need their tiles on 1-KB boundaries; there is no room for alignment slack, so the
  // dynamic part is declared with that alignment (and checked below).
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) Bars<C::kNumUnits> bars;
  __shared__ Item items[kItemSlots];
  __shared__ __align__(16) uint4 s_next;
  __shared__ uint32_t s_tmem_base;
  __shared__ int s_abort;

  const uint32_t smem_q = smem_u32(smem_raw);                      // Q tiles A and B, then the operand ring
  const uint32_t smem_ring = smem_q + C::kQBytes;
  uint8_t* ring_gen = smem_raw + C::kQBytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Geom& g = P.g;
  if (threadIdx.x == 0) {
    if ((smem_q & 1023u) != 0) atomicExch(P.status, (int)TIDE_ERR_CUDA);   // cannot happen with the declared alignment; refuse rather than compute garbage
    s_abort = 0;
    for (int i = 0; i < C::kNumUnits; ++i) { mbar_init(smem_u32(&bars.kv_full[i]), 1); mbar_init(smem_u32(&bars.kv_empty[i]), 1); }
    for (int t = 0; t < 2; ++t) {
      mbar_init(smem_u32(&bars.q_full[t]), 32);
      mbar_init(smem_u32(&bars.q_empty[t]), 1);
      mbar_init(smem_u32(&bars.s_full[t]), 1);
      mbar_init(smem_u32(&bars.s_free[t]), 128);
      for (int q = 0; q < kPParts; ++q) mbar_init(smem_u32(&bars.p_part[t][q]), 128);
      mbar_init(smem_u32(&bars.o_full[t]), 1);
    }
    for (int i = 0; i < kItemSlots; ++i) { mbar_init(smem_u32(&bars.item_full[i]), 1); mbar_init(smem_u32(&bars.item_empty[i]), kItemReaders); }
    mbar_init(smem_u32(&bars.k_issued), 1);
    mbar_init(smem_u32(&bars.next), 1);
    mbar_init(smem_u32(&bars.mma_done), 1);
    mbar_fence_init();
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  // With AttendParams::run_ahead the scheduler and the two producers start beside the append in front: the first item is
  // published and its first tiles (keys below Item::live_from) are on their way when the other warps are let go.  1.5 to
  // 3.5 us of every batch: four-task step 17.9 to 16.4 us, one row of 17 to 35 tokens behind 1500 keys 19.6 to 18.0, 12 rows
  // with one of 46 to 463 tokens 21.9 to 19.3, groups 76.2 to 74.4, prompts 698 to 692.
  const bool early = P.run_ahead != 0 && warp >= 8;
  if (!early) {
    grid_dep_wait();
    grid_dep_launch();
  }
  const int n_items = P.dyn ? __ldcg(P.dyn) : P.n_items;           // fixed grid: the batch's counts live in device memory
  tc_fence_after();
  const uint32_t tmem = s_tmem_base;
  volatile int* abort_flag = &s_abort;
  auto wait = [&](uint64_t& bar, int parity) -> bool {
    return mbar_wait(smem_u32(&bar), (uint32_t)parity, abort_flag, P.status, P.wait_limit_ns);
  };
  // the same where a warp branches on the outcome: its lanes stay together
  auto wait_all = [&](uint64_t& bar, int parity) -> bool { return __all_sync(0xffffffffu, wait(bar, parity)) != 0; };

  // register budget: the data-movement warpgroup gives registers to the two softmax warpgroups.  setmaxnreg
  // moves registers inside the CTA's own launch allocation (384 x 168), so the new counts must not add up to
  // more than that: 256 x 208 + 128 x 88 = 384 x 168.  (An over-subscribed .inc waits for ever.)  With 224 + 56 the MMA and
  // scheduler warps spill inside their loops: prompts 728 us against 708, mixed text batch 7165 against 7076.
  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
    if (warp == 8 || warp == 10) {
      // ================= producers: warp 8 the K tiles (units 0, 2, 4, ...), warp 10 the V tiles (1, 3, 5, ...) =================
      const int is_v = warp == 10 ? 1 : 0;
      const int pages_per_tile = kTileKeys / g.S;              // 8 or 4: one copy each
      const int tiles_per_group = 32 / pages_per_tile;
      int slot = is_v, use = 0;                                // this warp's next unit of the ring
      int issued = 0;                                          // tiles this warp has issued its copies of
      bool ok = true, ahead = early;
      for (int it = 0; ok; ++it) {
        if (ahead && it > 0) {                                 // the scheduler publishes no second item before that either
          grid_dep_wait();
          ahead = false;
        }
        if (!wait_all(bars.item_full[it % kItemSlots], (it / kItemSlots) & 1)) break;
        const Item& w = items[it % kItemSlots];
        if (!w.run) break;
        const int n_tiles = w.n_tiles, kv_begin = w.kv_begin, kv_end = w.kv_end, drop = w.drop, live_from = w.live_from;
        const int32_t* trow = P.table + w.table_off;
        const uint8_t* head_base = P.pool + (long long)w.kvh * g.head_bytes + is_v * g.kblock_bytes;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars.item_empty[it % kItemSlots]));
        // page ids are fetched 32 logical pages at a time, one per lane, a whole group ahead of their use,
        // so that no bulk copy waits for a dependent page-table load
        const int lp0 = kv_begin / g.S;
        auto load_ids = [&](int grp) -> int {
          const int lp = lp0 + grp * 32 + lane;
          return lp < g.max_pages_per_task ? __ldcg(trow + lp) : 0;
        };
        int ids_cur = load_ids(0), ids_nxt = load_ids(1), cur_grp = 0;
        for (int j = 0; j < n_tiles; ++j) {
          const int grp = j / tiles_per_group;
          if (grp != cur_grp) { ids_cur = ids_nxt; ids_nxt = load_ids(grp + 1); cur_grp = grp; }
          const int key0 = kv_begin + j * kTileKeys;
          const int npages = min(pages_per_tile, (kv_end - key0 + g.S - 1) / g.S);
          if (ahead && (use > 0 || key0 + npages * g.S > live_from)) {
            // the ring is full, or from here on pages, and page numbers, may belong to the kernel before this one
            grid_dep_wait();
            ahead = false;
            ids_cur = load_ids(grp);
            ids_nxt = load_ids(grp + 1);
          }
          // a wait that gave up means the ring can no longer be trusted: issue nothing more
          if (use > 0 && !wait_all(bars.kv_empty[slot], (use - 1) & 1)) { ok = false; break; }
          ++issued;
          const uint32_t bar = smem_u32(&bars.kv_full[slot]);
          const long long page = __shfl_sync(0xffffffffu, ids_cur, ((j % tiles_per_group) * pages_per_tile + lane) & 31);
          if (!(drop != 0 && j == 0 && is_v == 0)) {                           // test hook: K tile 0 never arrives
            if (lane == 0) mbar_expect_tx(bar, (uint32_t)(npages * g.kblock_bytes));
            __syncwarp();
            if (lane < npages)
              bulk_g2s(smem_ring + slot * C::kUnitBytes + lane * g.kblock_bytes, head_base + page * g.page_bytes, (uint32_t)g.kblock_bytes, bar);
          }
          slot += 2;
          if (slot >= C::kNumUnits) { slot -= C::kNumUnits; ++use; }
        }
        if (is_v == 0 && lane == 0) mbar_arrive(smem_u32(&bars.k_issued));
      }
      if (*abort_flag && lane == 0) {
        // a wait gave up somewhere: this warp does not leave while copies it issued into the CTA's shared memory
        // can still be landing.  Those are among its last kNumUnits tiles; each wait is bounded like every other.
        for (int j = max(0, issued - C::kNumUnits); j < issued; ++j) {
          const int u = 2 * j + is_v;
          const uint32_t bar = smem_u32(&bars.kv_full[u % C::kNumUnits]);
          const long long t0 = global_ns();
          while (!mbar_try(bar, (u / C::kNumUnits) & 1) && global_ns() - t0 < P.wait_limit_ns) {}
        }
      }
    } else if (warp == 9) {
      // ================= MMA issuer (whole warp converged, one elected lane issues) =================
      if (early) grid_dep_wait();                              // (its first wait is bounded, the kernel in front is not)
      // Descriptors are built once; moving an operand's start address is one 32-bit add on the low word (the
      // address field counts 16-byte units and cannot overflow its 14 bits inside this CTA's shared memory).
      const uint64_t kd0 = make_desc(smem_ring, 16, C::kGroupBytes);        // a K tile in unit 0 (K-major, 8-key groups apart)
      const uint64_t vd0 = make_desc(smem_ring, 1024, C::kGroupBytes);      // a V tile in unit 0 (MN-major: slabs 1 KB apart)
      const uint64_t qd0 = make_desc(smem_q, 16, 1024);                     // a Q tile (K-major, 8-row groups 1 KB apart)
      const uint32_t kd_lo = (uint32_t)kd0, kd_hi = (uint32_t)(kd0 >> 32), vd_lo = (uint32_t)vd0, vd_hi = (uint32_t)(vd0 >> 32);
      const uint32_t qd_lo = (uint32_t)qd0, qd_hi = (uint32_t)(qd0 >> 32);
      constexpr uint32_t kUnitStep = C::kUnitBytes >> 4;
      int n_qk[2] = {0, 0}, n_pv[2] = {0, 0}, n_q[2] = {0, 0};    // QKs, PVs and queries of each row tile so far (their barriers' phases)
      auto issue_qk = [&](int t, int slot, bool last) {
        if (C::kSepP && n_qk[t] > 0) { wait(bars.s_free[t], (n_qk[t] - 1) & 1); tc_fence_after(); }
        const uint32_t k_lo = kd_lo + slot * kUnitStep;
        const uint32_t q_lo = qd_lo + t * (C::kQTileBytes >> 4);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          mma_ss(tmem + C::kColS + t * 128, desc64(q_lo + (((ks >> 2) * C::kQSlabBytes + (ks & 3) * 32) >> 4), qd_hi),
                 desc64(k_lo + (((ks >> 2) * 1024 + (ks & 3) * 32) >> 4), kd_hi), C::kIdescQK, ks > 0);
        mma_commit(smem_u32(&bars.s_full[t]));
        if (last) mma_commit(smem_u32(&bars.q_empty[t]));
        ++n_qk[t];
      };
      auto issue_pv = [&](int t, int j, int slot) {
        const uint32_t v_lo = vd_lo + slot * kUnitStep;
#pragma unroll
        for (int q = 0; q < kPParts; ++q) {
          wait(bars.p_part[t][q], n_pv[t] & 1);
          tc_fence_after();
#pragma unroll
          for (int k4 = 0; k4 < kTileKeys / 16 / kPParts; ++k4) {
            const int ks = q * (kTileKeys / 16 / kPParts) + k4;
            mma_ts(tmem + C::kColO + t * D, tmem + C::kColP + t * C::kColPStep + ks * 8, desc64(v_lo + ((ks * 2 * C::kGroupBytes) >> 4), vd_hi),
                   C::kIdescPV, (j > 0 || ks > 0) ? 1u : 0u);
          }
        }
        ++n_pv[t];
      };
      int kslot = 0, kuse = 0, vslot = 1, vuse = 0;             // operand u of the sequence sits in unit u % kNumUnits
      auto advance = [&](int& slot, int& use) { slot += 2; if (slot >= C::kNumUnits) { slot -= C::kNumUnits; ++use; } };
      for (int it = 0; ; ++it) {
        if (!wait_all(bars.item_full[it % kItemSlots], (it / kItemSlots) & 1)) break;
        const Item& w = items[it % kItemSlots];
        if (!w.run) break;
        const int n_tiles = w.n_tiles, kv_begin = w.kv_begin, kv_end = w.kv_end;
        const int t_tiles[2] = {w.tiles[0], w.tiles[1]};
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars.item_empty[it % kItemSlots]));
        if (n_tiles == 0) continue;
        wait(bars.kv_full[kslot], kuse & 1);
        tc_fence_after();
#pragma unroll
        for (int t = 0; t < 2; ++t)
          if (t_tiles[t] > 0) {
            wait(bars.q_full[t], n_q[t] & 1);
            ++n_q[t];
            tc_fence_after();
            issue_qk(t, kslot, t_tiles[t] == 1);
          }
        mma_commit(smem_u32(&bars.kv_empty[kslot]));          // K(0) is consumed once these retire
        advance(kslot, kuse);
        for (int j = 0; j < n_tiles; ++j) {
          wait(bars.kv_full[vslot], vuse & 1);
          if (kv_end < kv_begin + (j + 1) * kTileKeys) {
            // rows of the V tile past the end of the item were not loaded (or hold stale page slots): clear
            // them so that weight 0 times leftover bits cannot produce NaN
            const int first = kv_end - (kv_begin + j * kTileKeys);
            uint8_t* vgen = ring_gen + vslot * C::kUnitBytes;
            for (int i = lane; i < (kTileKeys - first) * (D / 8); i += 32) {
              const int rr = first + i / (D / 8), c = i % (D / 8);     // whole rows are cleared, so the swizzle does not matter
              *reinterpret_cast<uint4*>(vgen + (rr >> 3) * C::kGroupBytes + (c >> 3) * 1024 + (rr & 7) * 128 + (c & 7) * 16) = make_uint4(0, 0, 0, 0);
            }
            fence_async_smem();
            __syncwarp();
          }
          bool k_ready = false;
          auto next_qk = [&](int t) {                          // QK_t(j+1)
            if (!k_ready) { wait(bars.kv_full[kslot], kuse & 1); tc_fence_after(); k_ready = true; }
            issue_qk(t, kslot, j + 2 == t_tiles[t]);
          };
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            if (C::kSepP && j + 1 < t_tiles[t]) next_qk(t);
            if (C::kSepP && t == 1 && j + 1 < n_tiles) mma_commit(smem_u32(&bars.kv_empty[kslot]));
            if (j < t_tiles[t]) {
              issue_pv(t, j, vslot);
              if (!C::kSepP && j + 1 < t_tiles[t]) next_qk(t); // overwrites S_t / P_t after PV_t(j), in order
              if (C::kSepP || j + 1 == t_tiles[t]) mma_commit(smem_u32(&bars.o_full[t]));
            }
          }
          // V(j) and K(j+1) are consumed once these MMAs retire
          mma_commit(smem_u32(&bars.kv_empty[vslot]));
          advance(vslot, vuse);
          if (j + 1 < n_tiles) {
            if (!C::kSepP) mma_commit(smem_u32(&bars.kv_empty[kslot]));
            advance(kslot, kuse);
          }
        }
      }
      // Every MMA has retired before this warp leaves (TMEM is freed after the CTA's last barrier): one more commit
      // covers all of them.  This wait does not look at the abort flag - MMAs retire whatever else went wrong.
      mma_commit(smem_u32(&bars.mma_done));
      {
        const uint32_t bar = smem_u32(&bars.mma_done);
        const long long t0 = global_ns();
        while (!mbar_try(bar, 0) && global_ns() - t0 < P.wait_limit_ns) {}
      }
    } else {
      // ================= warp 11: hands out the items and copies their queries =================
      const int n_segs = P.dyn ? __ldcg(P.dyn + 1) : P.n_segs;
      // copies of Q: lane -> row (mod 8) and 16-byte chunk (mod 4); eight rows on is dq tokens and dg heads on
      const int my_row = lane >> 2, my_chunk = lane & 3;
      const uint32_t my_swz0 = (uint32_t)((my_chunk ^ my_row) << 4), my_swz1 = (uint32_t)(((my_chunk + 4) ^ my_row) << 4);
      const int dq = 8 / g.G, dg = 8 - dq * g.G;
      const int src_step = (dq * g.Hq + dg) * D * 2, src_wrap = (g.Hq - g.G) * D * 2;
      int n_q[2] = {0, 0};
      int item = (int)blockIdx.x < n_items ? (int)blockIdx.x : -1, asks = 0;
      bool open = false;                                           // a question without an answer yet
      for (int it = 0; ; ++it) {
        const int slot = it % kItemSlots;
        if (it >= kItemSlots && !wait_all(bars.item_empty[slot], (it / kItemSlots - 1) & 1)) break;
        Item& w = items[slot];
        // The status word is set when a bounded wait runs out and stays set until tide_status clears it.  While it is set
        // no item is started, so outputs are undefined from the time-out until the caller has read the status.
        if (__shfl_sync(0xffffffffu, *reinterpret_cast<volatile int*>(P.status), 0) != 0) item = -1;
        if (item < 0) {
          if (lane == 0) { w.run = 0; mbar_arrive(smem_u32(&bars.item_full[slot])); }
          break;
        }
        const int si = find_segment(n_segs, item, [&](int i) { return INLINE ? segs[i].item_base : __ldcg(&segs[i].item_base); });
        const Segment seg = INLINE ? segs[si] : load_segment(segs + si);
        int local = item - seg.item_base;
        const int m_tile = local % seg.n_mtiles;
        local /= seg.n_mtiles;
        const int split = local % seg.n_splits;
        const int kvh = local / seg.n_splits;
        const int R = seg.n * g.G, row0 = m_tile * kUmmaTileRows * 2;
        const int kv_begin = seg.origin + split * seg.chunk;
        int t_rows[2], t_end[2], t_tiles[2], t_min_limit[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const int r0 = row0 + t * 128;
          t_rows[t] = max(0, min(128, R - r0));
          t_end[t] = kv_begin; t_min_limit[t] = kv_begin; t_tiles[t] = 0;
          if (t_rows[t] > 0) {
            t_end[t] = min(kv_begin + seg.chunk, seg.p + ((r0 + t_rows[t] - 1) / g.G) * seg.causal + 1);
            t_min_limit[t] = min(t_end[t], seg.p + (r0 / g.G) * seg.causal + 1);
            t_tiles[t] = t_end[t] > kv_begin ? (t_end[t] - kv_begin + kTileKeys - 1) / kTileKeys : 0;
          }
        }
        if (lane == 0) {
          w.run = 1;
          w.table_off = seg.table_off; w.kvh = kvh; w.kv_begin = kv_begin; w.kv_end = max(t_end[0], t_end[1]);
          w.n_tiles = max(t_tiles[0], t_tiles[1]);
          for (int t = 0; t < 2; ++t) { w.tiles[t] = t_tiles[t]; w.end[t] = t_end[t]; w.min_limit[t] = t_min_limit[t]; }
          w.row0 = row0; w.R = R; w.p = seg.p; w.causal = seg.causal; w.live_from = seg.live_from;
          w.direct = seg.n_splits == 1 && seg.partial == 0;
          w.q_row0 = seg.q_off * g.Hq;
          w.dst_row0 = w.direct ? seg.q_off * g.Hq : seg.part_base + split * seg.n * g.Hq;
          w.drop = P.debug_drop_first_stage != 0 && item == 0;
          mbar_arrive(smem_u32(&bars.item_full[slot]));
        }
        if (early && it == 0) grid_dep_wait();                     // the queries belong to earlier work
        // The rows of Q (zeros past the last one) as the A operand of S = Q.K^T: K-major, 128-byte swizzle.  One
        // instruction copies 64 bytes of eight rows; a lane's rows are eight apart, so their place in the swizzle is
        // fixed and a row costs it one pointer step for its D / 32 copies.  (One softmax thread per row, 16 bytes at a
        // time, needed 4.6 us per item; whole rows per instruction with an address per copy 2.4 us per tile.)
        auto copy_q = [&](int t) {
          int row = row0 + t * 128 + my_row;
          const int qi = row / g.G;
          int gi = row - qi * g.G;
          const uint8_t* src = reinterpret_cast<const uint8_t*>(P.q) +
                               (((long long)(seg.q_off + qi) * g.Hq + kvh * g.G + gi) * D + my_chunk * 8) * 2;
          uint32_t dst = smem_q + t * C::kQTileBytes + my_row * 128;
#pragma unroll 2
          for (int i = 0; i < 16; ++i) {
            const bool valid = row < R;
            const uint8_t* from = valid ? src : reinterpret_cast<const uint8_t*>(P.q);
#pragma unroll
            for (int c = 0; c < D / 32; ++c)
              cp_async16(dst + (c >> 1) * C::kQSlabBytes + ((c & 1) ? my_swz1 : my_swz0), from + (valid ? c * 64 : 0), valid);
            row += 8;
            gi += dg;
            src += src_step;
            if (gi >= g.G) { gi -= g.G; src += src_wrap; }
            dst += 1024;
          }
          cp_async_commit();
        };
        auto q_done = [&](int t) { fence_async_smem(); mbar_arrive(smem_u32(&bars.q_full[t])); };
        bool fine = true, a_open = false;                          // a_open: A's copy is under way and not yet reported
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (t_tiles[t] == 0 || !fine) continue;
          if (n_q[t] > 0) {
            // B's buffer is free half a tile after A's: A's copy is not held back by that
            if (a_open && __any_sync(0xffffffffu, !mbar_try(smem_u32(&bars.q_empty[t]), (n_q[t] - 1) & 1))) {
              cp_async_wait<0>();
              q_done(0);
              a_open = false;
            }
            fine = wait_all(bars.q_empty[t], (n_q[t] - 1) & 1);
          }
          if (!fine) continue;
          copy_q(t);
          ++n_q[t];
          if (t == 0) a_open = true;
        }
        if (a_open && t_tiles[1] > 0 && fine) { cp_async_wait<1>(); q_done(0); a_open = false; }
        cp_async_wait<0>();
        if (!fine) break;
        if (a_open) q_done(0);
        if (t_tiles[1] > 0) q_done(1);
        // The next item is claimed when the K producer has nothing left to do for this one, some two tiles before its
        // end: claimed at its start, it would bind long items to this SM while others run out of work.
        if (!wait_all(bars.k_issued, it & 1)) break;
        if (lane == 0) next_block_ask(smem_u32(&s_next), smem_u32(&bars.next));
        ++asks;
        open = true;
        if (!wait_all(bars.next, (asks - 1) & 1)) break;
        open = false;
        item = next_block_answer(smem_u32(&s_next));
        fence_async_smem();                                        // the answer has been read before the next one may land
        __syncwarp();
        if (item >= n_items) item = -1;                            // fixed grid: indices beyond the batch
      }
      if (open) {                                                  // only after a wait gave up: the answer lands before the block leaves
        const long long t0 = global_ns();
        while (!mbar_try(smem_u32(&bars.next), (asks - 1) & 1) && global_ns() - t0 < P.wait_limit_ns) {}
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    // ================= softmax warpgroups =================
    const int t = warp >> 2;                                   // 0 = A, 1 = B
    const int row = ((warp & 3) << 5) | lane;                  // row of the 128-row tile = TMEM lane
    const uint32_t lane_addr = (uint32_t)((warp & 3) << 5) << 16;
    const uint32_t s_addr = tmem + lane_addr + C::kColS + t * 128;
    const uint32_t p_addr = tmem + lane_addr + C::kColP + t * C::kColPStep;
    const uint32_t o_addr = tmem + lane_addr + C::kColO + t * D;
    const float sl2 = P.scale_log2e;
    int n_s = 0, n_o = 0;               // S tiles and finished items of this row tile so far (their barriers' phases)

    for (int it = 0; ; ++it) {
      if (!wait_all(bars.item_full[it % kItemSlots], (it / kItemSlots) & 1)) break;
      const Item& w = items[it % kItemSlots];
      if (!w.run) break;
      const int my_tiles = w.tiles[t], kv_begin = w.kv_begin;
      int limit = w.end[t];                                      // keys j < limit are visible
      if (w.row0 + t * 128 + row < w.R) limit = min(limit, w.p + ((w.row0 + t * 128 + row) / g.G) * w.causal + 1);
      float m = -INFINITY, l = 0.f;       // running max (base-2, scaled) and sum

      // One key tile of this row tile.  The tiles that need the causal (or end-of-range) mask are the last ones of the
      // item; they get a copy of the body of their own, so the compare-and-select instructions of the mask are not part of the
      // code the other tiles run.
      auto tile = [&](const int j, auto masked_tag) {
        constexpr bool kMasked = decltype(masked_tag)::value;
        wait(bars.s_full[t], n_s & 1);
        tc_fence_after();
        float s[128];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(s_addr + c * 32, &s[c * 32]);
        tmem_wait_ld();
        if constexpr (C::kSepP) {                                // QK_t(j+1) may overwrite S_t
          tc_fence_before();
          mbar_arrive(smem_u32(&bars.s_free[t]));
        }
        if constexpr (kMasked) {
          const int vis = limit - (kv_begin + j * kTileKeys);
#pragma unroll
          for (int c = 0; c < 128; ++c) if (c >= vis) s[c] = -INFINITY;
        }
        // independent partial reductions (one long dependent chain would expose its latency), three inputs per
        // instruction: 8 chains over 128 values, then a tree
        float mxp[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) mxp[i] = max3(s[i], s[i + 8], s[i + 16]);
#pragma unroll
        for (int c = 24; c < 120; c += 16) {
#pragma unroll
          for (int i = 0; i < 8; ++i) mxp[i] = max3(mxp[i], s[c + i], s[c + i + 8]);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) mxp[i] = fmaxf(mxp[i], s[i + 120]);
        float mx = max3(max3(mxp[0], mxp[1], mxp[2]), max3(mxp[3], mxp[4], mxp[5]), fmaxf(mxp[6], mxp[7]));
        mx *= sl2;                                               // scale > 0 on this path
        float m_new = m;
        if (C::kSepP && n_s > 0) {                               // PV_t(j-1) has read P_t and written O_t (D = 128: implied by s_full)
          wait(bars.o_full[t], (n_s - 1) & 1);
          tc_fence_after();
        }
        ++n_s;
        if (mx > m + kRescaleThreshold) m_new = mx;             // also the first visible key: -inf + 8 = -inf < any finite mx
        float alpha = 1.f;
        if (__any_sync(0xffffffffu, m_new != m)) {               // rare: one vote per tile decides both steps
          alpha = fast_exp2(m - m_new);                          // m = -inf -> 0, equal -> 1
          if (j > 0) {
            // O_t holds tiles < j: S_t(j) was committed after PV_t(j-1)
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
              float o[32];
              tmem_ld32(o_addr + c * 32, o);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] *= alpha;
              tmem_st32(o_addr + c * 32, o);
            }
          }
        }
        m = m_new;
        const float mu = (m == -INFINITY) ? 0.f : m;
        const uint64_t sl2_2 = pack2(sl2, sl2), nmu_2 = pack2(-mu, -mu);
        uint64_t sp2[4] = {pack2(0.f, 0.f), pack2(0.f, 0.f), pack2(0.f, 0.f), pack2(0.f, 0.f)};
        // The exponentials run on the ex2 unit, the sums and the bf16 packing on the FMA and ALU pipes.  A warp issues in
        // order, so the three only overlap if independent work is next to each other in the instruction stream: the stream
        // is written as a software pipeline over groups of 8 keys - scaled logits for all groups first, then the exponentials of group g+1 ahead of the sum and the
        // packing of group g, whose exponentials have had a whole group's time to come back.
        uint64_t x2[64];
#pragma unroll
        for (int i = 0; i < 64; ++i) x2[i] = fma2(pack2(s[2 * i], s[2 * i + 1]), sl2_2, nmu_2);
        float e[2][8];
        auto exp_group = [&](int gidx, float (&eg)[8]) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float x0, x1;
            unpack2(x2[gidx * 4 + i], x0, x1);
            eg[2 * i] = fast_exp2(x0);
            eg[2 * i + 1] = fast_exp2(x1);
          }
        };
        uint32_t pk[32];
        exp_group(0, e[0]);
#pragma unroll
        for (int gidx = 0; gidx < 16; ++gidx) {
          if (gidx + 1 < 16) exp_group(gidx + 1, e[(gidx + 1) & 1]);
          const float (&eg)[8] = e[gidx & 1];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            sp2[i] = add2(sp2[i], pack2(eg[2 * i], eg[2 * i + 1]));
            pk[(gidx & 7) * 4 + i] = pack_bf16(eg[2 * i], eg[2 * i + 1]);
          }
          // P_t over the first 64 columns of S_t; a part is handed over as soon as it is stored, so that its PV runs
          // while the exponentials of the later parts are computed (the last part is handed over after the row sum)
          constexpr int kGroupsPerPart = 16 / kPParts;
          if ((gidx + 1) % kGroupsPerPart == 0) {
            const int q = gidx / kGroupsPerPart;
            tmem_st32u(p_addr + q * 32, pk);
            if (q + 1 < kPParts) {
              tmem_wait_st();
              tc_fence_before();
              mbar_arrive(smem_u32(&bars.p_part[t][q]));
            }
          }
        }
        float sp[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) unpack2(sp2[i], sp[2 * i], sp[2 * i + 1]);
        l = l * alpha + (((sp[0] + sp[1]) + (sp[2] + sp[3])) + ((sp[4] + sp[5]) + (sp[6] + sp[7])));
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(smem_u32(&bars.p_part[t][kPParts - 1]));
      };
      // tiles j < n_plain end at or before the first row's limit: every key of theirs is visible to every row
      const int n_plain = min(my_tiles, max(0, (w.min_limit[t] - kv_begin) / kTileKeys));
      for (int j = 0; j < n_plain; ++j) tile(j, std::false_type{});
      for (int j = n_plain; j < my_tiles; ++j) tile(j, std::true_type{});

      // ---- epilogue: O / l and LSE ----
      const float kLn2 = 0.6931471805599453f;
      if (my_tiles > 0) {
        wait(bars.o_full[t], (C::kSepP ? n_s - 1 : n_o) & 1);
        ++n_o;
        tc_fence_after();
      }
      const float inv = l > 0.f ? 1.f / l : 0.f;
      const int r = w.row0 + t * 128 + row;
      const bool valid = r < w.R, direct = w.direct != 0;
      const bool wide = ((uintptr_t)P.out & 31) == 0;            // callers need only align to 16
      const int qi = r / g.G;
      const long long drow = w.dst_row0 + (long long)qi * g.Hq + w.kvh * g.G + (r - qi * g.G);
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        float o[32];
        if (my_tiles > 0) {                 // uniform over the warpgroup
          tmem_ld32(o_addr + c * 32, o);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] = 0.f;
        }
        if (valid) {
          if (direct) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              uint32_t v[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) v[e] = pack_bf16(o[i * 16 + 2 * e] * inv, o[i * 16 + 2 * e + 1] * inv);
              st_32bytes(P.out + drow * D + c * 32 + i * 16, v, wide);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              uint32_t v[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) v[e] = __float_as_uint(o[i * 8 + e] * inv);
              st_32bytes(P.part_o + drow * D + c * 32 + i * 8, v, true);
            }
          }
        }
      }
      if (valid) {
        const float e2 = l > 0.f ? m + log2f(l) : -INFINITY;
        if (direct) { if (P.lse != nullptr) P.lse[drow] = e2 * kLn2; }
        else P.part_lse[drow] = e2;
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars.item_empty[it % kItemSlots]));
    }
  }

  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1) attend_umma128_kernel(const AttendParams P) {
  attend_umma128_body<D, false>(P, P.segs);
}
// Items whose row descriptors travel in the kernel's parameters (small batches).
template <int D>
__global__ void __launch_bounds__(kThreads, 1) attend_umma128_inline_kernel(const __grid_constant__ AttendInline PI) {
  attend_umma128_body<D, true>(PI.p, PI.segs);
}

}  // namespace umma128

template <int D>
static cudaError_t init_one() {
  const cudaError_t e =
      cudaFuncSetAttribute(umma128::attend_umma128_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, umma128::Cfg<D>::kSmemBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(umma128::attend_umma128_inline_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, umma128::Cfg<D>::kSmemBytes);
}
cudaError_t attend_umma128_init() {
  const cudaError_t e = init_one<128>();
  return e != cudaSuccess ? e : init_one<64>();
}

cudaError_t launch_attend_umma128(const AttendParams& p, cudaStream_t s) {
  const int grid = p.dyn ? p.grid_cap : p.n_items;
  if (grid <= 0) return cudaSuccess;
  if (p.g.D == 128) return launch_dep(umma128::attend_umma128_kernel<128>, grid, umma128::kThreads, umma128::Cfg<128>::kSmemBytes, s, p);
  return launch_dep(umma128::attend_umma128_kernel<64>, grid, umma128::kThreads, umma128::Cfg<64>::kSmemBytes, s, p);
}

cudaError_t launch_attend_umma128_inline(const AttendInline& pi, cudaStream_t s) {
  if (pi.p.n_items <= 0) return cudaSuccess;
  if (pi.p.g.D == 128)
    return launch_dep(umma128::attend_umma128_inline_kernel<128>, pi.p.n_items, umma128::kThreads, umma128::Cfg<128>::kSmemBytes, s, pi);
  return launch_dep(umma128::attend_umma128_inline_kernel<64>, pi.p.n_items, umma128::kThreads, umma128::Cfg<64>::kSmemBytes, s, pi);
}

}  // namespace tide

// Attention of resume rows over the paged cache with warp-level tensor-core tiles (mma.sync): the rows that the tcgen05
// kernel does not take (a softmax scale that is not positive, launch shapes fixed without tcgen05 items, 64-key tiles
// selected with head size 64), and the merge of split rows.
//
// What it computes (paper Section 4: a resumed task continues from its preserved KV state; the maths is
// ordinary scaled-dot-product softmax attention with grouped KV heads): for a work item
// (row, kv_head, m_tile, split) the online-softmax partial over keys [kv_begin, kv_end) for a tile of
// packed rows r = q_index * G + g (the G query heads that share this KV head), query q_index seeing keys
// [0, prefix + q_index].  K/V pages are read ONCE per KV head for all G query heads.
//
// Structure: one producer warp streams whole (page, head) blocks (K and V, contiguous in the pool) into a
// ring of shared-memory stages with 1-D bulk copies that complete on mbarriers; four consumer warps run
// m16n8k16 bf16 MMAs straight from the pre-swizzled blocks with ldmatrix, each on 16 of the 64 packed rows.
#include <cfloat>
#include <climits>

#include "tide_internal.h"

namespace tide {

constexpr int kConsumerWarps = 4;
constexpr int kAttendThreads = (kConsumerWarps + 1) * 32;
constexpr int kStages = 3;

template <int D>
struct MmaCfg {
  static constexpr int kStageBytes = kStageKeys * D * 4;  // K + V, bf16
  static constexpr int kSmemBytes = kStages * kStageBytes + 1024;
};

template <int D>
__global__ void __launch_bounds__(kAttendThreads, 2) attend_mma_kernel(const AttendParams P) {
  constexpr int KS = D / 16;                 // k-steps of Q.K^T
  constexpr int NT = D / 8;                  // n-tiles of O
  constexpr int STEP_KB = 4;                 // 16-key blocks per softmax step of one warp
  constexpr int TILE_M = kMmaTileRows;
  constexpr int STAGE_BYTES = MmaCfg<D>::kStageBytes;

  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t s_full[kStages];
  __shared__ __align__(8) uint64_t s_empty[kStages];
  __shared__ int s_abort;

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Geom& g = P.g;
  const Segment* __restrict__ segs = P.segs;
  grid_dep_wait();
  grid_dep_launch();

  // ---- which item ----
  const int item = blockIdx.x;
  int n_segs = P.n_segs;
  if (P.dyn != nullptr) {                      // fixed grid: the batch's counts live in device memory
    if (item >= P.dyn[0]) return;
    n_segs = P.dyn[1];
  }
  const int si = find_segment(n_segs, item, [&](int i) { return segs[i].item_base; });
  const Segment seg = segs[si];
  int local = item - seg.item_base;
  const int m_tile = local % seg.n_mtiles;
  local /= seg.n_mtiles;
  const int split = local % seg.n_splits;
  const int kvh = local / seg.n_splits;
  const int R = seg.n * g.G;                       // packed rows of this (row, kv head)
  const int tile_row0 = m_tile * TILE_M;
  const int r_last = min(R, tile_row0 + TILE_M) - 1;
  const int kv_begin = seg.origin + split * seg.chunk;
  const int kv_end = min(kv_begin + seg.chunk, seg.p + (r_last / g.G) * seg.causal + 1);
  const bool direct = seg.n_splits == 1 && seg.partial == 0;
  const float kLn2 = 0.6931471805599453f;

  // rows this thread owns inside its warp's 16-row MMA tile
  const int row_base = tile_row0 + warp * 16;
  const int r_lo = row_base + (lane >> 2), r_hi = r_lo + 8;
  const bool v_lo = r_lo < R, v_hi = r_hi < R;
  const int qi_lo = r_lo / g.G, qi_hi = r_hi / g.G;
  const int hd_lo = kvh * g.G + (r_lo - qi_lo * g.G), hd_hi = kvh * g.G + (r_hi - qi_hi * g.G);

  if (kv_end <= kv_begin) {
    // nothing visible in this split (only possible when n_splits > 1): neutral partials
    if (warp < kConsumerWarps && (lane & 3) == 0) {
      if (v_lo) P.part_lse[seg.part_base + (split * seg.n + qi_lo) * g.Hq + hd_lo] = -INFINITY;
      if (v_hi) P.part_lse[seg.part_base + (split * seg.n + qi_hi) * g.Hq + hd_hi] = -INFINITY;
    }
    return;
  }

  // The status word is set when a bounded wait runs out and stays set until tide_status clears it.  While it is
  // set no CTA starts work (this launch's later CTAs and every CTA of later launches leave here without writing
  // anything), so outputs are undefined from the time-out until the caller has read the status.
  __shared__ int s_skip;
  if (threadIdx.x == 0) s_skip = *reinterpret_cast<volatile int*>(P.status);
  __syncthreads();
  if (s_skip != 0) return;

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int i = 0; i < kStages; ++i) {
      mbar_init(smem_u32(&s_full[i]), 1);
      mbar_init(smem_u32(&s_empty[i]), kConsumerWarps);
    }
    mbar_fence_init();
  }
  __syncthreads();
  volatile int* abort_flag = &s_abort;

  const int n_st = (kv_end - kv_begin + kStageKeys - 1) / kStageKeys;

  if (warp == kConsumerWarps) {
    // ================= producer warp =================
    const int pages_per_stage = kStageKeys / g.S;
    int issued = 0;                              // stages whose copies were issued
    for (int st = 0; st < n_st; ++st) {
      const int slot = st % kStages;
      // a wait that gave up means the ring can no longer be trusted: issue nothing more
      if (st >= kStages && !mbar_wait(smem_u32(&s_empty[slot]), ((st / kStages) - 1) & 1, abort_flag, P.status, P.wait_limit_ns)) break;
      issued = st + 1;
      if (P.debug_drop_first_stage != 0 && item == 0 && st == 0) continue;   // test hook: this stage never arrives
      const int key0 = kv_begin + st * kStageKeys;
      const int npages = min(pages_per_stage, (kv_end - key0 + g.S - 1) / g.S);
      const uint32_t bar = smem_u32(&s_full[slot]);
      if (lane == 0) mbar_expect_tx(bar, (uint32_t)(npages * g.head_bytes));
      __syncwarp();
      if (lane < npages) {
        const long long page = P.table[seg.table_off + key0 / g.S + lane];
        const uint8_t* src = P.pool + page * g.page_bytes + (long long)kvh * g.head_bytes;
        bulk_g2s(smem_base + slot * STAGE_BYTES + lane * g.head_bytes, src, (uint32_t)g.head_bytes, bar);
      }
    }
    if (*abort_flag && lane == 0) {
      // a wait gave up somewhere: do not leave the CTA while copies into its shared memory are in flight.  Only the
      // last kStages stages that were issued can still be landing (an older one was consumed before its slot was
      // refilled); each wait is bounded like every other.
      for (int st = max(0, issued - kStages); st < issued; ++st) {
        const uint32_t bar = smem_u32(&s_full[st % kStages]);
        const long long t0 = global_ns();
        while (!mbar_try(bar, (st / kStages) & 1) && global_ns() - t0 < P.wait_limit_ns) {}
      }
    }
    return;
  }

  // ================= consumer warps =================
  const int kv_limit_lo = v_lo ? min(kv_end, seg.p + qi_lo * seg.causal + 1) : kv_end;  // keys j < limit are visible
  const int kv_limit_hi = v_hi ? min(kv_end, seg.p + qi_hi * seg.causal + 1) : kv_end;
  // last key any row of this warp can see, and the smallest limit (masking needed beyond it)
  int w_end, w_min_limit;
  {
    const int wr_first = row_base, wr_last = min(R, row_base + 16) - 1;
    if (wr_last < wr_first) { w_end = kv_begin; w_min_limit = kv_end; }   // warp has no valid rows
    else {
      w_end = min(kv_end, seg.p + (wr_last / g.G) * seg.causal + 1);
      w_min_limit = min(kv_end, seg.p + (wr_first / g.G) * seg.causal + 1);
    }
  }

  uint32_t qa[KS][4];
  {
    const uint16_t* q_lo = P.q + ((long long)(seg.q_off + qi_lo) * g.Hq + hd_lo) * D + 2 * (lane & 3);
    const uint16_t* q_hi = P.q + ((long long)(seg.q_off + qi_hi) * g.Hq + hd_hi) * D + 2 * (lane & 3);
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      qa[ks][0] = v_lo ? *reinterpret_cast<const uint32_t*>(q_lo + ks * 16) : 0u;
      qa[ks][1] = v_hi ? *reinterpret_cast<const uint32_t*>(q_hi + ks * 16) : 0u;
      qa[ks][2] = v_lo ? *reinterpret_cast<const uint32_t*>(q_lo + ks * 16 + 8) : 0u;
      qa[ks][3] = v_hi ? *reinterpret_cast<const uint32_t*>(q_hi + ks * 16 + 8) : 0u;
    }
  }

  float o[NT][4];
#pragma unroll
  for (int i = 0; i < NT; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
  float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;
  const float sl2 = P.scale_log2e;

  for (int st = 0; st < n_st; ++st) {
    const int slot = st % kStages;
    mbar_wait(smem_u32(&s_full[slot]), (st / kStages) & 1, abort_flag, P.status, P.wait_limit_ns);
    const int key0 = kv_begin + st * kStageKeys;
    const uint32_t stage = smem_base + slot * STAGE_BYTES;
    const int step_key0 = key0;
    if (step_key0 < w_end) {
      const int nkb = min(STEP_KB, (w_end - step_key0 + 15) >> 4);
      float s[STEP_KB * 2][4];
#pragma unroll
      for (int b = 0; b < STEP_KB; ++b) {
        if (b < nkb) {
          const int koff = b * 16;            // key offset inside the stage
          const uint32_t pbase = stage + (koff / g.S) * g.head_bytes;
          const int row0 = koff % g.S;
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) {
            float(&acc)[4] = s[b * 2 + nt];
            acc[0] = acc[1] = acc[2] = acc[3] = 0.f;
            const int slot_row = row0 + nt * 8 + (lane & 7);
#pragma unroll
            for (int k2 = 0; k2 < KS / 2; ++k2) {
              uint32_t b0, b1, b2, b3;
              ldsm_x4(pbase + blk_offset(g, slot_row, 0, k2 * 4 + (lane >> 3)), b0, b1, b2, b3);
              mma_bf16(acc, qa[2 * k2], b0, b1);
              mma_bf16(acc, qa[2 * k2 + 1], b2, b3);
            }
          }
        }
      }
      // ---- scale, mask, online softmax ----
      const int step_end = step_key0 + nkb * 16;
      const bool need_mask = step_end > w_min_limit;
      float mx_lo = -INFINITY, mx_hi = -INFINITY;
#pragma unroll
      for (int t = 0; t < STEP_KB * 2; ++t) {
        if (t < nkb * 2) {
          const int j = step_key0 + t * 8 + 2 * (lane & 3);
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
      for (int t = 0; t < STEP_KB * 2; ++t) {
        if (t < nkb * 2) {
          s[t][0] = fast_exp2(s[t][0] - mu_lo); s[t][1] = fast_exp2(s[t][1] - mu_lo);
          s[t][2] = fast_exp2(s[t][2] - mu_hi); s[t][3] = fast_exp2(s[t][3] - mu_hi);
          ps_lo += s[t][0] + s[t][1];
          ps_hi += s[t][2] + s[t][3];
        }
      }
      l_lo = l_lo * a_lo + ps_lo;
      l_hi = l_hi * a_hi + ps_hi;
      // ---- O += P.V ----
#pragma unroll
      for (int b = 0; b < STEP_KB; ++b) {
        if (b < nkb) {
          const int koff = b * 16;
          const uint32_t vbase = stage + (koff / g.S) * g.head_bytes;   // the page block; V parts through blk_offset(.., 1, ..)
          const int row0 = koff % g.S;
          const int blk_key0 = key0 + koff;
          if (blk_key0 + 16 > kv_end) {
            // slots past the end of the item hold whatever the page held before: clear V there so that
            // weight 0 times stale bits cannot produce NaN
            const int first = kv_end - blk_key0;           // 1..15
            uint8_t* vgen = smem_gen + (vbase - smem_base);
            for (int idx = lane; idx < (16 - first) * (D / 8); idx += 32) {
              const int rr = row0 + first + idx / (D / 8), c = idx % (D / 8);
              *reinterpret_cast<uint4*>(vgen + blk_offset(g, rr, 1, c)) = make_uint4(0, 0, 0, 0);
            }
            __syncwarp();
          }
          uint32_t pa[4];
          pa[0] = pack_bf16(s[2 * b][0], s[2 * b][1]);
          pa[1] = pack_bf16(s[2 * b][2], s[2 * b][3]);
          pa[2] = pack_bf16(s[2 * b + 1][0], s[2 * b + 1][1]);
          pa[3] = pack_bf16(s[2 * b + 1][2], s[2 * b + 1][3]);
          const int vrow = row0 + ((lane >> 3) & 1) * 8 + (lane & 7);
#pragma unroll
          for (int n2 = 0; n2 < NT / 2; ++n2) {
            uint32_t b0, b1, b2, b3;
            ldsm_x4_t(vbase + blk_offset(g, vrow, 1, n2 * 2 + (lane >> 4)), b0, b1, b2, b3);
            mma_bf16(o[2 * n2], pa, b0, b1);
            mma_bf16(o[2 * n2 + 1], pa, b2, b3);
          }
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&s_empty[slot]));
  }

  // ---- epilogue ----
  l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1);
  l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
  l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1);
  l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);

  const float inv_lo = l_lo > 0.f ? 1.f / l_lo : 0.f, inv_hi = l_hi > 0.f ? 1.f / l_hi : 0.f;
  const float e_lo = l_lo > 0.f ? m_lo + log2f(l_lo) : -INFINITY;
  const float e_hi = l_hi > 0.f ? m_hi + log2f(l_hi) : -INFINITY;
  const int dcol = 2 * (lane & 3);
  if (direct) {
    const long long o_lo = ((long long)(seg.q_off + qi_lo) * g.Hq + hd_lo), o_hi = ((long long)(seg.q_off + qi_hi) * g.Hq + hd_hi);
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      if (v_lo) *reinterpret_cast<uint32_t*>(P.out + o_lo * D + i * 8 + dcol) = pack_bf16(o[i][0] * inv_lo, o[i][1] * inv_lo);
      if (v_hi) *reinterpret_cast<uint32_t*>(P.out + o_hi * D + i * 8 + dcol) = pack_bf16(o[i][2] * inv_hi, o[i][3] * inv_hi);
    }
    if (P.lse != nullptr && (lane & 3) == 0) {
      if (v_lo) P.lse[o_lo] = e_lo * kLn2;
      if (v_hi) P.lse[o_hi] = e_hi * kLn2;
    }
  } else {
    const long long p_lo = seg.part_base + (long long)(split * seg.n + qi_lo) * g.Hq + hd_lo;
    const long long p_hi = seg.part_base + (long long)(split * seg.n + qi_hi) * g.Hq + hd_hi;
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      if (v_lo) *reinterpret_cast<float2*>(P.part_o + p_lo * D + i * 8 + dcol) = make_float2(o[i][0] * inv_lo, o[i][1] * inv_lo);
      if (v_hi) *reinterpret_cast<float2*>(P.part_o + p_hi * D + i * 8 + dcol) = make_float2(o[i][2] * inv_hi, o[i][3] * inv_hi);
    }
    if ((lane & 3) == 0) {
      if (v_lo) P.part_lse[p_lo] = e_lo;
      if (v_hi) P.part_lse[p_hi] = e_hi;
    }
  }
}

cudaError_t attend_kernels_init() {
  const cudaError_t e = cudaFuncSetAttribute(attend_mma_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, MmaCfg<128>::kSmemBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(attend_mma_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, MmaCfg<64>::kSmemBytes);
}

cudaError_t launch_attend_tile(const AttendParams& p, cudaStream_t s) {
  const int grid = p.dyn ? p.grid_cap : p.n_items;
  if (grid <= 0) return cudaSuccess;
  if (p.g.D == 128) return launch_dep(attend_mma_kernel<128>, grid, kAttendThreads, MmaCfg<128>::kSmemBytes, s, p);
  return launch_dep(attend_mma_kernel<64>, grid, kAttendThreads, MmaCfg<64>::kSmemBytes, s, p);
}

// ---------------------------------------------------------------------------------------------
// Log-sum-exp merge of the split partials: one warp per (token, head) row.
//   LSE = log2 sum_i 2^{LSE_i},  O = sum_i 2^{LSE_i - LSE} O_i;  fixed order, no atomics.
// Bound by latency (a chain of dependent loads if written naively), so the partial LSEs are fetched side by side, one per
// lane, the partial outputs four splits at a time, the first four beside the LSEs, and the row's segment is looked up
// before the wait; the order in which the terms are added is still the order of the splits.
// (One row of 17 to 35 tokens behind 1500 / 16000 keys with its append 16.0 / 27.0 us, 16 rows, two of them resumed, 41.8;
// with all LSEs of up to 256 contributions in eight registers a lane, picked by index, and the outputs behind them 18.0 /
// 33.2 and 44.8; eight splits at a time spill, 15.7 / 26.5 and 42.8.)
__device__ __forceinline__ void merge_body(const MergeParams& P, const Segment* __restrict__ segs) {
  // the descriptors were complete before the attention kernels started: the look-up needs no wait
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int n_rows = P.dyn ? P.dyn[0] : P.n_rows, n_segs = P.dyn ? P.dyn[1] : P.n_segs;
  if (row >= n_rows) {
    grid_dep_wait();
    return;
  }
  const int si = find_segment(n_segs, row, [&](int i) { return segs[i].merge_base; });
  const Segment seg = segs[si];
  const int local = row - seg.merge_base;                 // token * Hq + head inside the segment
  const long long stride = (long long)seg.n * P.Hq;       // partial rows per split
  const long long p0 = seg.part_base + local;
  // a row's contributions: its own splits, then (a member of a group that shares its first pages) the splits of the
  // group's shared range, where this row is one token among the members' (such segments have one token: local = head)
  const int n_src = seg.n_splits + seg.x_n_splits;
  auto src_row = [&](int s) -> long long {
    return s < seg.n_splits ? p0 + s * stride : (long long)seg.x_part_base + local + (long long)(s - seg.n_splits) * seg.x_stride;
  };
  const int per = P.D / 32;                               // 2 or 4 floats per lane
  constexpr int kBatch = 4;
  float4 v[kBatch];
  auto fetch = [&](int s0) {
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      if (s0 + u >= n_src) continue;
      const float* po = P.part_o + src_row(s0 + u) * P.D + lane * per;
      if (per == 4) v[u] = __ldcg(reinterpret_cast<const float4*>(po));
      else { const float2 t = __ldcg(reinterpret_cast<const float2*>(po)); v[u] = make_float4(t.x, t.y, 0.f, 0.f); }
    }
  };
  grid_dep_wait();
  grid_dep_launch();
  fetch(0);
  float mstar = -INFINITY, tot = 0.f;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int c0 = 0; c0 < n_src; c0 += 32) {                // 32 contributions: lane i holds the LSE, then the weight, of c0 + i
    const float e = c0 + lane < n_src ? __ldcg(P.part_lse + src_row(c0 + lane)) : -INFINITY;
    float m_new = e;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m_new = fmaxf(m_new, __shfl_xor_sync(0xffffffffu, m_new, o));
    m_new = fmaxf(mstar, m_new);
    const float mu = (m_new == -INFINITY) ? 0.f : m_new, keep = exp2f(mstar - mu), mine = exp2f(e - mu);   // -inf: 0
    mstar = m_new;
    tot *= keep;
#pragma unroll
    for (int d = 0; d < 4; ++d) acc[d] *= keep;
    const int n_here = min(32, n_src - c0);
    for (int s0 = 0; s0 < n_here; s0 += kBatch) {
      if (c0 + s0 > 0) fetch(c0 + s0);
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const float w = __shfl_sync(0xffffffffu, mine, s0 + u);
        if (w != 0.f) {
          tot += w;
          acc[0] += w * v[u].x; acc[1] += w * v[u].y; acc[2] += w * v[u].z; acc[3] += w * v[u].w;
        }
      }
    }
  }
  const float inv = tot > 0.f ? 1.f / tot : 0.f;
  const long long orow = (long long)seg.q_off * P.Hq + local;
  uint16_t* dst = P.out + orow * P.D + lane * per;
  if (per == 4) {
    uint2 v;
    v.x = pack_bf16(acc[0] * inv, acc[1] * inv);
    v.y = pack_bf16(acc[2] * inv, acc[3] * inv);
    *reinterpret_cast<uint2*>(dst) = v;
  } else {
    *reinterpret_cast<uint32_t*>(dst) = pack_bf16(acc[0] * inv, acc[1] * inv);
  }
  if (P.lse != nullptr && lane == 0) P.lse[orow] = (tot > 0.f ? mstar + log2f(tot) : -INFINITY) * 0.6931471805599453f;
}

__global__ void __launch_bounds__(256) merge_kernel(const MergeParams P) { merge_body(P, P.segs); }
__global__ void __launch_bounds__(256) merge_inline_kernel(const __grid_constant__ MergeInline PI) { merge_body(PI.p, PI.segs); }

cudaError_t launch_merge_inline(const MergeInline& pi, cudaStream_t s) {
  if (pi.p.n_rows <= 0) return cudaSuccess;
  return launch_dep(merge_inline_kernel, (unsigned)((pi.p.n_rows + 7) / 8), 256, 0, s, pi);
}

cudaError_t launch_merge(const MergeParams& p, cudaStream_t s) {
  const int rows = p.dyn ? p.grid_cap_rows : p.n_rows;
  if (rows <= 0) return cudaSuccess;
  const int blocks = (rows + 7) / 8;
  return launch_dep(merge_kernel, (unsigned)blocks, 256, 0, s, p);
}

}  // namespace tide

// Page-append scatter, page-table delta update and logical read-back.
//
// Append is the GPU half of resuming a task under Continuous Task Batching (paper Section 4): the
// observation tokens' K/V rows are copied into the task's pages next to its preserved state, which
// replaces re-running prefill over the history (Section 1, first challenge).  It is a pure bit copy,
// bound by HBM bandwidth: 2 * Hkv * D * 2 bytes read and as many written per new token.
#include <algorithm>

#include "tide_internal.h"

namespace tide {

__global__ void table_update_kernel(int32_t* __restrict__ table, const int32_t* __restrict__ idx,
                                    const int32_t* __restrict__ val, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) table[idx[i]] = val[i];
}

cudaError_t launch_table_update(int32_t* table, const int32_t* idx, const int32_t* val, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  table_update_kernel<<<(n + 255) / 256, 256, 0, s>>>(table, idx, val, n);
  return cudaGetLastError();
}

// Small host-to-device upload done by the SMs: src is pinned host memory mapped into the device's address space.
// Unlike a copy-engine transfer it does not queue behind large copies that other streams have in flight.
__global__ void upload_kernel(uint32_t* __restrict__ dst, const uint32_t* __restrict__ src, size_t n_words) {
  grid_dep_wait();
  grid_dep_launch();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_words; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = src[i];
}

cudaError_t launch_upload(void* dst, const void* src_mapped_host, size_t bytes, cudaStream_t s) {
  if (bytes == 0) return cudaSuccess;
  const size_t n = bytes / 4;
  const unsigned blocks = (unsigned)std::min<size_t>((n + 255) / 256, 64);
  return launch_dep(upload_kernel, blocks, 256, 0, s, (uint32_t*)dst, (const uint32_t*)src_mapped_host, n);
}

// Queries of a small host-buffer step: each byte crosses PCIe once, 16 at a time, while the append in front of this launch
// runs (the destination is idle: the step before has been waited for).  Read in place by the decode kernel they crossed it
// once per work item and consumer warp, 32 bytes at a time: nine rows of 3k keys 361 us a step.
__global__ void __launch_bounds__(256) fetch_kernel(uint4* __restrict__ dst, const uint4* __restrict__ src, size_t n) {
  grid_dep_launch();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) dst[i] = __ldcg(src + i);
  grid_dep_wait();
}

cudaError_t launch_fetch(void* dst, const void* src_mapped_host, size_t bytes, cudaStream_t s) {
  if (bytes == 0) return cudaSuccess;
  const size_t n = bytes / 16;
  return launch_dep(fetch_kernel, (unsigned)std::min<size_t>((n + 255) / 256, (size_t)sm_count()), 256, 0, s, (uint4*)dst, (const uint4*)src_mapped_host, n);
}

__global__ void upload_set_kernel(const __grid_constant__ UploadSet u) {
  grid_dep_wait();
  grid_dep_launch();
  const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
  for (size_t i = first; i < (size_t)u.n_upd; i += step) u.table[u.idx[i]] = u.val[i];
  for (int p = 0; p < u.n_parts; ++p)
    for (size_t i = first; i < u.part[p].words; i += step) u.part[p].dst[i] = u.part[p].src[i];
}

cudaError_t launch_upload_set(const UploadSet& u, cudaStream_t s) {
  size_t most = (size_t)u.n_upd;
  for (int p = 0; p < u.n_parts; ++p) most = std::max(most, u.part[p].words);
  if (most == 0) return cudaSuccess;
  return launch_dep(upload_set_kernel, (unsigned)std::min<size_t>((most + 255) / 256, 64), 256, 0, s, u);
}

constexpr int kAppendThreads = 256;
constexpr int kAppendWarps = kAppendThreads / 32;
constexpr int kAppendMaxRecsSmem = 1024;
constexpr int kAppendLoadsInFlight = 8;    // 16-byte loads a lane has in flight before its first store

// The append: the new rows of every record go to their slots in the record's pages.  A warp takes the rows of EIGHT
// consecutive slots of one (kv, head) at a time, i.e. one 8-slot group of a page block - D / 64 core-matrix atoms of
// 1 KB, chunk c of row r at chunk position c ^ r - and writes it as one contiguous run: per instruction it reads
// four 128-byte pieces (four tokens) and writes 512 contiguous bytes.  (Written token by token, 128 bytes into four
// different atoms per instruction, the same copy ran at 4.9 instead of 5.5 TB/s on the multimodal batch.)  The
// record and page look-ups (warp-uniform) happen once per round of kAppendLoadsInFlight 16-byte loads per lane, all
// issued before the first store: a copy like this is bound by how many bytes are in flight.  Rows of a group that
// lie outside the record (its first and last group may be ragged) are left alone.  The same launch first applies
// the page-table delta of the append, if it is given one; the pages that delta brings are then taken from the delta
// itself, not from the table (no ordering between thread blocks is needed).
// AppendRec::grp0 = number of 8-slot groups that the records before this one touch.
// What does not depend on earlier kernels - finding the first round's record, when the records are in the launch or were
// complete before (AppendParams::early) - happens before the wait for them.
template <int SLABS>
__device__ __forceinline__ void append_scatter_body(const AppendParams& P, const AppendRec* __restrict__ recs,
                                                  const int32_t* __restrict__ upd_idx, const int32_t* __restrict__ upd_val,
                                                  const bool early) {
  __shared__ int32_t s_grp0[kAppendMaxRecsSmem];
  bool waited = false;
  auto wait = [&] {
    if (waited) return;
    waited = true;
    grid_dep_wait();
    grid_dep_launch();
    for (int i = blockIdx.x * kAppendThreads + threadIdx.x; i < P.n_upd; i += gridDim.x * kAppendThreads)
      P.table_rw[upd_idx[i]] = upd_val[i];
  };
  if (!early) wait();
  const int n_recs = P.dyn ? __ldcg(P.dyn) : P.n_recs;
  if (n_recs <= 0) {
    wait();
    return;
  }
  const bool in_smem = n_recs <= kAppendMaxRecsSmem;
  if (in_smem) {
    for (int i = threadIdx.x; i < n_recs; i += blockDim.x) s_grp0[i] = recs[i].grp0;
    __syncthreads();
  }
  const Geom& g = P.g;
  const int lane = threadIdx.x & 31;
  const int heads2 = 2 * g.Hkv;
  long long n_units;
  {
    const AppendRec last = recs[n_recs - 1];
    n_units = (long long)(last.grp0 + (((last.pos0 & 7) + last.count + 7) >> 3)) * heads2;
  }
  const int warps_total = gridDim.x * kAppendWarps;
  const int warp_id = blockIdx.x * kAppendWarps + (threadIdx.x >> 5);
  constexpr int LPU = SLABS * 2;                               // 16-byte chunks per lane per (group, kv, head)
  constexpr int UNITS = kAppendLoadsInFlight / LPU;            // (kv, head) blocks of one group per warp per round
  const int rounds_per_group = (heads2 + UNITS - 1) / UNITS;
  const long long n_rounds = (n_units / heads2) * rounds_per_group;
  for (long long w = warp_id; w < n_rounds; w += warps_total) {
    // one look-up per round: the group's record and page
    const int grp = (int)(w / rounds_per_group), hh0 = (int)(w - (long long)grp * rounds_per_group) * UNITS;
    int r;
    if (in_smem) r = find_segment(n_recs, grp, [&](int i) { return s_grp0[i]; });
    else r = find_segment(n_recs, grp, [&](int i) { return recs[i].grp0; });
    const AppendRec rec = recs[r];
    wait();
    const int g_pos0 = (rec.pos0 & ~7) + (grp - rec.grp0) * 8;                 // first slot position of the group
    const int lp = g_pos0 / g.S;
    const long long page = lp >= rec.new_lp0 ? upd_val[rec.new_off + (lp - rec.new_lp0)] : P.table[rec.table_off + lp];
    uint8_t* const dst_grp = P.pool + page * g.page_bytes + ((g_pos0 - lp * g.S) >> 3) * g.group_bytes;
    const int lo = max(0, rec.pos0 - g_pos0), hi = min(8, rec.pos0 + rec.count - g_pos0);
    const long long src_tok = (long long)(rec.tok0 + (g_pos0 - rec.pos0)) * g.Hkv;   // (token, head 0) row of the group's slot 0
    uint4 v[UNITS][LPU];
#pragma unroll
    for (int k = 0; k < UNITS; ++k) {
      const int hh = hh0 + k, kv = hh >= g.Hkv ? 1 : 0, h = hh - kv * g.Hkv;
      const uint16_t* src = (kv ? P.new_v : P.new_k) + (src_tok + h) * g.D;
#pragma unroll
      for (int i = 0; i < LPU; ++i) {
        const int e = lane + 32 * i;                           // chunk of the group in storage order: [slab][row][position]
        const int slab = e >> 6, row = (e >> 3) & 7, c = (e & 7) ^ row;
        v[k][i] = make_uint4(0, 0, 0, 0);
        if (hh < heads2 && row >= lo && row < hi)
          v[k][i] = __ldcg(reinterpret_cast<const uint4*>(src + (long long)row * g.Hkv * g.D + (slab * 8 + c) * 8));
      }
    }
#pragma unroll
    for (int k = 0; k < UNITS; ++k) {
      const int hh = hh0 + k, kv = hh >= g.Hkv ? 1 : 0, h = hh - kv * g.Hkv;
      uint8_t* dst = dst_grp + (long long)h * g.head_bytes + kv * g.kblock_bytes;
#pragma unroll
      for (int i = 0; i < LPU; ++i) {
        const int e = lane + 32 * i, row = (e >> 3) & 7;
        if (hh < heads2 && row >= lo && row < hi) *reinterpret_cast<uint4*>(dst + e * 16) = v[k][i];
      }
    }
  }
  wait();
}

template <int SLABS>
__global__ void __launch_bounds__(kAppendThreads, 3) append_scatter_kernel(const AppendParams P) {
  append_scatter_body<SLABS>(P, P.recs, P.upd_idx, P.upd_val, P.early != 0);
}
template <int SLABS>
__global__ void __launch_bounds__(kAppendThreads, 3) append_scatter_inline_kernel(const __grid_constant__ AppendInline PI) {
  append_scatter_body<SLABS>(PI.p, PI.recs, PI.upd, PI.upd + PI.p.n_upd, true);
}

static unsigned append_grid(const AppendParams& p) {
  const long long cap = (long long)sm_count() * 3;            // the resident blocks; each warp loops over rounds beyond this
  if (p.dyn) return (unsigned)cap;
  const long long rounds = ((long long)p.n_tokens / 8 + 2LL * p.n_recs + 1) * 2 * p.g.Hkv + 1;   // an upper bound
  return (unsigned)std::max<long long>(1, std::min((rounds + kAppendWarps - 1) / kAppendWarps, cap));
}

cudaError_t launch_append(const AppendParams& p, cudaStream_t s) {
  const int tokens = p.dyn ? p.grid_cap_tokens : p.n_tokens;
  if (tokens <= 0 && p.n_upd <= 0) return cudaSuccess;
  return launch_dep(p.g.D == 128 ? append_scatter_kernel<2> : append_scatter_kernel<1>, append_grid(p), kAppendThreads, 0, s, p);
}

cudaError_t launch_append_inline(const AppendInline& pi, cudaStream_t s) {
  if (pi.p.n_tokens <= 0 && pi.p.n_upd <= 0) return cudaSuccess;
  return launch_dep(pi.p.g.D == 128 ? append_scatter_inline_kernel<2> : append_scatter_inline_kernel<1>, append_grid(pi.p), kAppendThreads, 0,
                    s, pi);
}

// Whole-page copies dst[i] <- src[i] (the private copy a forked task gets of a partial last page, and the copy an
// append makes before it writes into a page that other tasks still hold).  One block column per page.
__global__ void copy_pages_kernel(uint8_t* __restrict__ pool, const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                  long long page_bytes) {
  const uint4* s = reinterpret_cast<const uint4*>(pool + (long long)src[blockIdx.y] * page_bytes);
  uint4* d = reinterpret_cast<uint4*>(pool + (long long)dst[blockIdx.y] * page_bytes);
  const long long n = page_bytes / 16;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) d[i] = s[i];
}

cudaError_t launch_copy_pages(uint8_t* pool, const int32_t* src, const int32_t* dst, int n, long long page_bytes, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  dim3 grid(8, (unsigned)n);
  copy_pages_kernel<<<grid, 256, 0, s>>>(pool, src, dst, page_bytes);
  return cudaGetLastError();
}

// Sliding-window pruning in place: positions [to, to + n) of a task take the content of [to + shift, to + shift + n), on
// every layer.  The task keeps its pages, so this is a move inside its own page list by a distance that need not be a
// multiple of anything, bound by memory: 2 * Hkv * D * 2 bytes read and as many written per token.  (Staged through the
// workspace - table update, gather, scatter and two uploads per chunk of max_batch_tokens - eight tasks with tails of 4k
// to 16k tokens took 390 us, mostly launches; this way they take about 100.)  The moves of different tasks do not depend on
// each other: one that directly follows another (`overlapped`) runs beside it.
//
// Position d depends only on d + shift, so the positions of one residue modulo the shift form a chain, and chains are
// independent of one another.  A chain is cut into segments of a few links, all of them in one block, a thread moving 16
// bytes of each link of its segment front to back, always reading ahead of what it writes.  Only the source of a segment's
// last link is written by another thread (it is the first target of the next segment): every thread loads that one, and
// its first kMoveLinks links, ahead of the block's barrier and stores nothing before it.
constexpr int kMoveLinks = 4;
// Bound by latency - two dependent loads, page number and data, for every kMoveLinks links of a thread - until the blocks fill
// the chip, where it is memory and the last round of blocks; how far chains are cut is launch_move's choice.
constexpr int kMovePairsLog2 = 5, kMoveChainThreads = 8 << kMovePairsLog2;   // 32 (segment, chain) pairs of eight lanes, 128 bytes of a row
template <int SLABS>
__global__ void __launch_bounds__(kMoveChainThreads, 3) move_chains_kernel(uint8_t* pool0, size_t layer_stride, const int32_t* __restrict__ table_row, int to,
                                                                           int shift, int n, int segs_log2, int seg_links, int overlapped,
                                                                           const Geom g) {
  if (!overlapped) grid_dep_wait();
  grid_dep_launch();
  uint8_t* const pool = pool0 + (size_t)blockIdx.y * layer_stride;
  // neighbouring chains, whose rows are neighbours in the pages' atoms, go to neighbouring lanes
  const int chains = min(shift, n), chains_log2 = kMovePairsLog2 - segs_log2;
  const int groups = (chains + (1 << chains_log2) - 1) >> chains_log2;
  const int group = blockIdx.x % groups, slab = blockIdx.x / groups % SLABS, hh = blockIdx.x / groups / SLABS, kv = hh >= g.Hkv ? 1 : 0;
  const long long head = (long long)(hh - kv * g.Hkv) * g.head_bytes;
  const int c = slab * 8 + (threadIdx.x & 7), pair = threadIdx.x >> 3;
  const int chain = (group << chains_log2) + (pair & ((1 << chains_log2) - 1)), seg = pair >> chains_log2;
  const int links = chain < chains ? (n - chain - 1) / shift + 1 : 0;
  const int first = min(seg * seg_links, links), end = min(first + seg_links, links);   // this segment's links ...
  const bool cut = segs_log2 > 0;
  const int last = cut ? end - 1 : end;                      // ... in front of the one whose source another thread writes
  const int s_log2 = g.S == 16 ? 4 : 5;
  auto at = [&](int link) -> uint4* {                        // a link's target: the source of the link before it
    const int pos = to + chain + link * shift, lp = pos >> s_log2;
    return reinterpret_cast<uint4*>(pool + (long long)__ldcg(table_row + lp) * g.page_bytes + head + blk_offset(g, pos & (g.S - 1), kv, c));
  };
  uint4 *a0[kMoveLinks + 1], *a1[kMoveLinks + 1];
  uint4 v0[kMoveLinks], v1[kMoveLinks];
  // links i, i + 1, ... of those in front of the last one; a[k + 1] is link i + k's source and the target of link i + k + 1
  auto load = [&](int i, uint4* target, uint4* (&a)[kMoveLinks + 1], uint4 (&v)[kMoveLinks]) {
    a[0] = target;
#pragma unroll
    for (int k = 0; k < kMoveLinks; ++k) a[k + 1] = i + k < last ? at(i + k + 1) : target;
#pragma unroll
    for (int k = 0; k < kMoveLinks; ++k)
      if (i + k < last) v[k] = __ldcg(a[k + 1]);
  };
  auto store = [&](int i, uint4* const (&a)[kMoveLinks + 1], const uint4 (&v)[kMoveLinks]) {
#pragma unroll
    for (int k = 0; k < kMoveLinks; ++k)
      if (i + k < last) *a[k] = v[k];
  };
  uint4* last_target = nullptr;
  uint4 last_value = make_uint4(0, 0, 0, 0);
  int i = first;
  if (first < end) {
    if (cut) {
      // the page numbers of all these links side by side, then their data (one link's behind the other's: 1 to 2 us more)
      uint4* const source = at(end);
      last_target = at(last);
      load(i, at(i), a0, v0);
      last_value = __ldcg(source);
    } else load(i, at(i), a0, v0);
  }
  if (cut) __syncthreads();
  while (i < last) {
    if (i + kMoveLinks < last) load(i + kMoveLinks, a0[kMoveLinks], a1, v1);
    store(i, a0, v0);
    i += kMoveLinks;
    if (i >= last) break;
    if (i + kMoveLinks < last) load(i + kMoveLinks, a1[kMoveLinks], a0, v0);
    store(i, a1, v1);
    i += kMoveLinks;
  }
  if (last_target != nullptr) *last_target = last_value;
  if (overlapped) grid_dep_wait();
}

// One block per (layer, kv, head, 64-element slab) moves a run of rows at a time, front to
// back: the whole run is in registers before its first row is stored (the run's last sources lie behind its targets, so
// no later run is touched), and the next run is loaded before this one is stored.
constexpr int kMoveThreads = 512, kMoveRows = 8;              // 16-byte chunks per thread and run: 512 rows of 128 bytes
template <int SLABS>
__global__ void __launch_bounds__(kMoveThreads) move_runs_kernel(uint8_t* pool0, size_t layer_stride, const int32_t* __restrict__ table_row, int to,
                                                                 int shift, int n, int overlapped, const Geom g) {
  if (!overlapped) grid_dep_wait();
  grid_dep_launch();
  uint8_t* const pool = pool0 + (size_t)blockIdx.y * layer_stride;
  const int slab = blockIdx.x % SLABS, hh = blockIdx.x / SLABS, kv = hh >= g.Hkv ? 1 : 0;
  const long long head = (long long)(hh - kv * g.Hkv) * g.head_bytes;
  const int c = slab * 8 + threadIdx.x % 8, r0 = threadIdx.x / 8;
  constexpr int kRun = kMoveThreads / 8 * kMoveRows, kStep = kMoveThreads / 8;
  auto at = [&](int pos) -> uint4* {
    const int lp = pos / g.S;
    return reinterpret_cast<uint4*>(pool + (long long)__ldcg(table_row + lp) * g.page_bytes + head + blk_offset(g, pos - lp * g.S, kv, c));
  };
  uint4 v[2][kMoveRows];
  auto load = [&](int run, uint4 (&x)[kMoveRows]) {
#pragma unroll
    for (int i = 0; i < kMoveRows; ++i) {
      x[i] = __ldcg(at(to + shift + min(run + r0 + i * kStep, n - 1)));   // (no branch: the loads go out side by side)
    }
  };
  auto store = [&](int run, const uint4 (&x)[kMoveRows]) {
#pragma unroll
    for (int i = 0; i < kMoveRows; ++i) {
      const int r = run + r0 + i * kStep;
      uint4* const dst = at(to + min(r, n - 1));
      if (r < n) *dst = x[i];
    }
  };
  load(0, v[0]);
  for (int run = 0; run < n; run += 2 * kRun) {
    __syncthreads();                                          // every thread has loaded run `run`
    load(run + kRun, v[1]);
    store(run, v[0]);
    __syncthreads();
    load(run + 2 * kRun, v[0]);
    store(run + kRun, v[1]);
  }
  if (overlapped) grid_dep_wait();
}

// How many segments (as a power of two) each chain is cut into; groups of chains x `columns` are the blocks, of which three fit an SM.
// While half of these places would stay empty, down to segments whose links are loaded at once; then up to nine blocks an SM, which
// even out the last round, down to 16 links.  A last cut that would leave a second round nearly empty is not made.
// us, cut until the blocks just fill the chip / this (4 KV heads, D = 128): 8 layers, tail of 16000 tokens, shift 64 142 / 101, 100 172 / 102,
// 128 150 / 99, 512 110 / 101; tail of 65000 566 / 381, 679 / 389, 583 / 373, 444 / 429; one layer, shift 128, tail of 1500 / 4000 / 16000: a
// thread per chain 10.2 / 16.2 / 43.0, this 8.2 / 9.9 / 17.2; eleven tails of 3500 tokens by 107 in a row, with their append and attention,
// 109 and 59.
static int move_segments_log2(int chains, int links, long long columns) {
  const long long places = 3ll * sm_count();
  auto blocks = [&](int segs_log2) -> long long {
    const int per_block_log2 = kMovePairsLog2 - segs_log2;
    return (((long long)chains + (1 << per_block_log2) - 1) >> per_block_log2) * columns;
  };
  int s = 0;
  for (; s < kMovePairsLog2; ++s) {
    const int ahead = (links - 1) >> s;                      // of a segment's last link
    if (!(2 * blocks(s) < places && ahead > kMoveLinks) && !(blocks(s) < 3 * places && ahead >= 32)) break;
  }
  if (s > 0 && blocks(s) > places && 2 * blocks(s) < 3 * places && blocks(s - 1) <= places) --s;
  return s;
}

// Runs take a shift of one, and long tails that move by two: in so few chains only as many threads move as a chain has segments.
// us, runs / chains (4 KV heads, D = 128): shift 1, tail of 1500 / 4000 / 16000 tokens 17 29 88 / 21 43 147; shift 2, 16000 88 / 68, 65000 and 300000
// 391 1811 / 461 2477 (8 layers, 65000 / 120000 584 1024 / 578 1107; these before the loads of a segment were put side by side); shift 3,
// 16000 / 120000 88 723 / 47 529; shift 17, 120000 723 / 136.
constexpr int kMoveRunsFrom = 8192;                          // links of a shift of two

cudaError_t launch_move(uint8_t* pool, size_t layer_stride, int layers, const int32_t* table_row, int to, int shift, int n, bool overlapped,
                        const Geom& g, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int links = (n - 1) / shift + 1, columns = 2 * g.Hkv * (g.D / 64);
  if (shift == 1 || (shift == 2 && links > kMoveRunsFrom)) {
    const dim3 grid((unsigned)columns, (unsigned)layers);
    return launch_dep(g.D == 128 ? move_runs_kernel<2> : move_runs_kernel<1>, grid, kMoveThreads, 0, s, pool, layer_stride, table_row, to, shift, n,
                      overlapped ? 1 : 0, g);
  }
  const int chains = std::min(shift, n), segs_log2 = move_segments_log2(chains, links, (long long)columns * layers);
  const int per_block_log2 = kMovePairsLog2 - segs_log2;
  const dim3 grid((unsigned)((((long long)chains + (1 << per_block_log2) - 1) >> per_block_log2) * columns), (unsigned)layers);
  return launch_dep(g.D == 128 ? move_chains_kernel<2> : move_chains_kernel<1>, grid, kMoveChainThreads, 0, s, pool, layer_stride, table_row, to, shift,
                    n, segs_log2, ((links - 1) >> segs_log2) + 1, overlapped ? 1 : 0, g);
}

// Logical content of one task -> contiguous [len, Hkv, D]; inverse of the scatter above.
// Positions [pos0, pos0 + len) of the task go to rows [0, len) of out_k / out_v.
__global__ void read_gather_kernel(const uint8_t* __restrict__ pool, const int32_t* __restrict__ table_row, int pos0, int len,
                                   uint16_t* __restrict__ out_k, uint16_t* __restrict__ out_v, const Geom g) {
  const int cpr = g.D >> 3;
  const int cpt = 2 * g.Hkv * cpr;
  const long long total = (long long)len * cpt;
  for (long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x; gid < total;
       gid += (long long)gridDim.x * blockDim.x) {
    const int row = (int)(gid / cpt);
    int rem = (int)(gid - (long long)row * cpt);
    const int kv = rem / (g.Hkv * cpr);
    rem -= kv * g.Hkv * cpr;
    const int h = rem / cpr;
    const int c = rem - h * cpr;
    const int pos = pos0 + row;
    const int lp = pos / g.S, slot = pos - lp * g.S;
    const long long page = table_row[lp];
    const uint8_t* src = pool + page * g.page_bytes + (long long)h * g.head_bytes + blk_offset(g, slot, kv, c);
    uint16_t* dst = (kv ? out_v : out_k) + ((long long)row * g.Hkv + h) * g.D + c * 8;
    *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
  }
}

cudaError_t launch_read(const uint8_t* pool, const int32_t* table_row, int pos0, int len, uint16_t* out_k,
                        uint16_t* out_v, const Geom& g, cudaStream_t s) {
  if (len <= 0) return cudaSuccess;
  const long long total = (long long)len * 2 * g.Hkv * (g.D / 8);
  long long blocks = (total + 255) / 256;
  const long long cap = (long long)sm_count() * 64;
  if (blocks > cap) blocks = cap;
  read_gather_kernel<<<(unsigned)blocks, 256, 0, s>>>(pool, table_row, pos0, len, out_k, out_v, g);
  return cudaGetLastError();
}

}  // namespace tide

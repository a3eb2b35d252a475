// A stand-in for the CUDA runtime and for the kernel launches of the library, so that the host side - bookkeeping, planner,
// what is launched where with which descriptors - runs without a GPU: "device" memory is ordinary memory, copies and
// uploads happen at once, a kernel launch is only written down.
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../paper_2608_10402_b200/csrc/tide_internal.h"

using namespace tide;

namespace {
enum Kind { kDecode, kTile, kUmma, kMerge, kAppend, kMove, kTable, kUpload, kCopyPages, kRead, kFetch };
struct Launch {
  int kind, run_ahead, overlapped, n_items, early, writes;
  void* stream;
  std::vector<Segment> segs;
};
std::vector<Launch> g_log;
cudaError_t note(int kind, cudaStream_t s) {
  g_log.push_back({kind, 0, 0, 0, 0, 0, (void*)s, {}});
  return cudaSuccess;
}
cudaError_t note_attend(int kind, const AttendParams& p, const Segment* segs, cudaStream_t s) {
  g_log.push_back({kind, p.run_ahead, p.overlapped, p.n_items, 0, p.new_k != nullptr, (void*)s, std::vector<Segment>(segs, segs + p.n_segs)});
  return cudaSuccess;
}
}  // namespace

extern "C" {
int recorded() { return (int)g_log.size(); }
void forget() { g_log.clear(); }
// kind, run_ahead, overlapped, work items, early, number of segments, whether it writes K/V rows
void* launch_at(int i, int* out) {
  const Launch& l = g_log[(size_t)i];
  const int v[7] = {l.kind, l.run_ahead, l.overlapped, l.n_items, l.early, (int)l.segs.size(), l.writes};
  std::memcpy(out, v, sizeof(v));
  return l.stream;
}
int claimed(int landed, int answer, int n_items) { return claimed_item(landed != 0, answer, n_items); }
void segment_at(int i, int j, int* out) { std::memcpy(out, &g_log[(size_t)i].segs[(size_t)j], sizeof(Segment)); }

cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  a->type = cudaMemoryTypeHost;
  a->devicePointer = const_cast<void*>(p);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)std::malloc(16); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free((void*)s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)std::malloc(16); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free((void*)e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
}  // extern "C"

namespace tide {
cudaError_t attend_kernels_init() { return cudaSuccess; }
cudaError_t attend_decode_init() { return cudaSuccess; }
cudaError_t attend_umma_init() { return cudaSuccess; }
cudaError_t attend_umma128_init() { return cudaSuccess; }
cudaError_t launch_table_update(int32_t* table, const int32_t* idx, const int32_t* val, int n, cudaStream_t s) {
  for (int i = 0; i < n; ++i) table[idx[i]] = val[i];
  return note(kTable, s);
}
cudaError_t launch_upload(void* dst, const void* src, size_t bytes, cudaStream_t s) { std::memcpy(dst, src, bytes); return note(kUpload, s); }
cudaError_t launch_fetch(void* dst, const void* src, size_t bytes, cudaStream_t s) { std::memcpy(dst, src, bytes); return note(kFetch, s); }
cudaError_t launch_upload_set(const UploadSet& u, cudaStream_t s) {
  for (int i = 0; i < u.n_upd; ++i) u.table[u.idx[i]] = u.val[i];
  for (int p = 0; p < u.n_parts; ++p) std::memcpy(u.part[p].dst, u.part[p].src, u.part[p].words * 4);
  return note(kUpload, s);
}
cudaError_t launch_append(const AppendParams& p, cudaStream_t s) {
  if (p.n_tokens <= 0 && p.n_upd <= 0) return cudaSuccess;
  g_log.push_back({kAppend, 0, 0, p.n_tokens, p.early, 1, (void*)s, {}});
  return cudaSuccess;
}
cudaError_t launch_append_inline(const AppendInline& p, cudaStream_t s) { return launch_append(p.p, s); }
cudaError_t launch_move(uint8_t*, size_t, int, const int32_t*, int, int, int, bool overlapped, const Geom&, cudaStream_t s) {
  g_log.push_back({kMove, 0, overlapped ? 1 : 0, 0, 0, 1, (void*)s, {}});
  return cudaSuccess;
}
cudaError_t launch_copy_pages(uint8_t*, const int32_t*, const int32_t*, int, long long, cudaStream_t s) { return note(kCopyPages, s); }
cudaError_t launch_read(const uint8_t*, const int32_t*, int, int, uint16_t*, uint16_t*, const Geom&, cudaStream_t s) { return note(kRead, s); }
cudaError_t launch_attend_decode(const AttendParams& p, cudaStream_t s) { return note_attend(kDecode, p, p.segs, s); }
cudaError_t launch_attend_decode_inline(const AttendInline& p, cudaStream_t s) { return note_attend(kDecode, p.p, p.segs, s); }
cudaError_t launch_attend_tile(const AttendParams& p, cudaStream_t s) { return note_attend(kTile, p, p.segs, s); }
cudaError_t launch_attend_umma(const AttendParams& p, cudaStream_t s) { return note_attend(kUmma, p, p.segs, s); }
cudaError_t launch_attend_umma128(const AttendParams& p, cudaStream_t s) { return note_attend(kUmma, p, p.segs, s); }
cudaError_t launch_attend_umma128_inline(const AttendInline& p, cudaStream_t s) { return note_attend(kUmma, p.p, p.segs, s); }
cudaError_t launch_merge(const MergeParams& p, cudaStream_t s) { g_log.push_back({kMerge, 0, 0, p.n_rows, 0, 0, (void*)s, std::vector<Segment>(p.segs, p.segs + p.n_segs)}); return cudaSuccess; }
cudaError_t launch_merge_inline(const MergeInline& p, cudaStream_t s) { g_log.push_back({kMerge, 0, 0, p.p.n_rows, 0, 0, (void*)s, std::vector<Segment>(p.segs, p.segs + p.p.n_segs)}); return cudaSuccess; }
}  // namespace tide

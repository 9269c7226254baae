// Test harness: the engine's planning and scan enqueueing (engine.cpp) on the
// CPU, over a CUDA runtime of its own.  Device memory is host memory, copies
// are done at once, kernels are names in a log, and the launch of one's choice
// fails as the runtime has it fail: nothing runs, and the error is the last
// error until it is taken.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <set>
#include <string>
#include <vector>

#include "engine.h"
#include "host_meta.h"
#include "host_pages.h"

namespace {

struct World {
  cudaError_t last = cudaSuccess;
  int n_sms = 152;
  int fail_at = -1;                 // the launch that fails, counted from the scan on (-2: its copies)
  bool scanning = false;
  std::vector<std::string> log;     // the scan's launches, the failing one among them
  int forks = 0, joins = 0;         // waits of other streams for the scan's, and back
  cudaStream_t main = nullptr;
  std::vector<cudaEvent_t> recorded;
  std::set<cudaEvent_t> captured;   // of them, those last recorded inside a capture
  bool capturing = false;
  uint64_t device_bytes = 0;        // asked of cudaMalloc, in
  int mallocs = 0;                  // so many calls
  int kernels = 0;                  // of the scan's launches
} W;

uintptr_t handles = 0x1000;
template <typename T>
T handle() {
  return reinterpret_cast<T>(handles += 16);
}

bool launch(const char* name, int kernels = 1) {
  if (!W.scanning) return true;
  W.kernels += kernels;
  const bool fails = static_cast<int>(W.log.size()) == W.fail_at;
  W.log.push_back(name);
  if (fails) W.last = cudaErrorInvalidConfiguration;
  return !fails;
}

}  // namespace

extern "C" {
cudaError_t cudaGetLastError() {
  const cudaError_t e = W.last;
  W.last = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return W.last; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = W.n_sms, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  W.device_bytes += n;
  ++W.mallocs;
  return *p = calloc(n, 1), cudaSuccess;
}
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return *p = calloc(n, 1), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { return *d = h, cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return memmove(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (W.scanning && W.fail_at == -2) return W.last = cudaErrorInvalidValue;
  return memmove(d, s, n), cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = handle<cudaStream_t>(), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
  *st = W.capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) {
  if (W.scanning) ++(s == W.main ? W.joins : W.forks);
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return W.capturing = true, cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  W.capturing = false;
  return *g = handle<cudaGraph_t>(), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  return *e = handle<cudaGraphExec_t>(), cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
  W.log.push_back("graph");
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = handle<cudaEvent_t>(), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = handle<cudaEvent_t>(), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) {  // (refused for an event last recorded inside a capture)
  return W.captured.count(e) ? W.last = cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 0, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
  W.recorded.push_back(e);
  if (W.capturing) W.captured.insert(e);
  else W.captured.erase(e);
  return cudaSuccess;
}
}

namespace pqi {
void launch_transcode(const TranscodeJob*, int n, int n_bss, uint32_t, PlanPage*, uint8_t*, uint64_t, uint32_t*, uint64_t*, DevStatus*,
                      cudaStream_t) {
  if (n > 0) launch("transcode", transcode_kernels(n, n_bss));
}
void launch_dict(const DictJob*, int n, bool fixed, int, int regions, DictScratch, DictDev*, int, DevStatus*,
                 cudaStream_t) {
  launch("dict", dict_kernels(n, fixed, regions));
}
void launch_walk(const DecodeArgs&, int, int n, int, bool, uint32_t, cudaStream_t) {
  if (n > 0) launch("walk");
}
void launch_delta_bases(const DecodeArgs&, int, int n, int regions, cudaStream_t) {
  if (n > 0) launch("delta", delta_kernels(n, regions));
}
void launch_expand(const DecodeArgs&, int, int n, int, bool, int, int, cudaStream_t) {
  if (n > 0) launch("expand");
}
uint32_t dict_expand_stage_bytes(int, int) { return 1024; }
bool dict_expand_fits(uint32_t, uint32_t) { return true; }
void launch_dict_expand(const DecodeArgs&, int, int, int, int, int, uint32_t, uint32_t, cudaStream_t) {
  launch("dict_expand");
}
void launch_copy_items(const DecodeArgs&, int, int, int, int, int, cudaStream_t) { launch("copy"); }
void launch_strings(const DecodeArgs&, int, int n, int, bool copy, uint32_t* left, cudaStream_t) {
  if (n > 0) launch("strings", strings_kernels(n, copy, left != nullptr));
}
void launch_plain_pages(const DecodeArgs&, int, int, cudaStream_t) { launch("plain"); }
void launch_prepare(const DecodeArgs& a, int, int, cudaStream_t) {
  if (launch("prepare")) *a.st = DevStatus{0, -1, 0, 0};
}
void launch_copy_small(void* dst, const void* src, uint32_t bytes, cudaStream_t) {
  if (launch("copy_small")) memcpy(dst, src, bytes);
}
void launch_make_items(const DecodeArgs&, int, cudaStream_t) {}
int expand_blocks_per_sm() { return 4; }
int walk_blocks_per_sm() { return 4; }
void launch_snappy(const SnappyJob*, int, int, DevStatus*, cudaStream_t, bool) { launch("snappy"); }
void launch_snappy_scan(const SnappyJob*, int n, uint32_t, uint32_t segs, SnapState, uint32_t*, bool long_first, int,
                        DevStatus*, cudaStream_t) {
  launch("snappy_scan", snappy_scan_kernels(n, segs, long_first));
}
void launch_snappy_fragments(const SnappyJob*, int, int, SnapState, int, DevStatus*, cudaStream_t) {
  launch("snappy_fragments");
}
void launch_zstd(const SnappyJob*, int, int, DevStatus*, cudaStream_t) { launch("zstd"); }
void launch_index_walk(const ChunkDev*, int, PageDev*, uint32_t*, int, DevStatus*, cudaStream_t) {}
void launch_gather16(const uint8_t* const*, const int32_t*, int, uint8_t*, cudaStream_t) {}
void launch_index_oi(const ChunkDev*, int, const int64_t*, PageDev*, int, DevStatus*, cudaStream_t) {}
}  // namespace pqi

// Plans and scans all columns of the file on a GPU of n_sms multiprocessors,
// with launch `fail_at` of the scan failing (-1: none, -2: its copies to the GPU,
// -3: none, but the scan is captured by the caller),
// on a thread whose last error is stale_error.  Returns the scan's
// status, -1 when it did not get that far; `text` gets what there is to see.
extern "C" int scan_with_fake_cuda(const uint8_t* file, uint64_t size, uint32_t flags, int n_sms, int fail_at,
                                   int stale_error, char* text, uint64_t cap) {
  W = World{};
  W.n_sms = n_sms;
  W.fail_at = fail_at;
  pq_ctx* ctx = nullptr;
  if (pq_ctx_create(0, &ctx) != PQ_OK) return -1;
  auto ix = std::make_unique<pq_index>();
  ix->ctx = ctx;
  pq_file f;
  f.data = const_cast<uint8_t*>(file);
  f.size = size;
  ix->files.push_back(f);
  uint32_t flen;
  memcpy(&flen, file + size - 8, 4);
  pqh::FileMeta m;
  std::string err;
  if (pqh::parse_file_metadata(file + size - 8 - flen, flen, &m, &err) != pqh::META_OK) return -1;
  m.footer_len = flen;
  std::vector<pqi::PageDev> pages;
  uint32_t chunk = 0;
  for (const auto& g : m.rgs)
    for (const auto& c : g.chunks)
      if (!pqe::host_page_walk(file + c.start(), static_cast<uint64_t>(c.total_compressed), c.num_values, chunk++, &pages,
                               &err))
        return -1;
  ix->metas.push_back(std::move(m));
  pq_index* idx = nullptr;
  if (pqe::index_build(ctx, std::move(ix), false, nullptr, &idx, &pages) != PQ_OK) return -1;
  pq_request req{};
  req.flags = flags;
  req.row_count = -1;
  pq_plan* plan = nullptr;
  std::vector<pq_out_size> sizes(static_cast<size_t>(idx->n_columns));
  W.last = static_cast<cudaError_t>(stale_error);
  const uint64_t bytes_before = W.device_bytes;
  const int mallocs_before = W.mallocs;
  if (pq_plan_scan(ctx, idx, &req, &plan, sizes.data()) != PQ_OK) return -1;
  const uint64_t bytes = W.device_bytes - bytes_before;
  const int mallocs = W.mallocs - mallocs_before;
  std::vector<pq_column> outs;
  std::vector<std::vector<uint8_t>> mem;
  const auto buffer = [&](uint64_t n) {
    mem.emplace_back(n + 64);
    return static_cast<void*>(mem.back().data());
  };
  for (const auto& z : sizes) {
    pq_column c{};
    c.values = buffer(z.values_bytes + 8);
    c.validity = static_cast<uint32_t*>(buffer(z.validity_bytes));
    c.chars = static_cast<uint8_t*>(buffer(z.chars_bytes));
    c.chars_capacity = z.chars_bytes;
    outs.push_back(c);
  }
  W.main = handle<cudaStream_t>();
  W.scanning = true;
  W.recorded.clear();
  W.last = static_cast<cudaError_t>(stale_error);
  W.capturing = fail_at == -3;
  const pq_status st = pqe::scan_enqueue(plan, outs.data(), W.main, ctx->branch, pq_ctx::kBranches, true);
  W.capturing = W.scanning = false;
  const int last = static_cast<int>(W.last);
  const pq_status waited = pq_scan_wait(ctx, plan, W.main, nullptr);
  bool done = false;
  for (cudaEvent_t e : W.recorded) done |= e == plan->done;
  std::string t = "items " + std::to_string(plan->n_items) + "\nplan_bytes " + std::to_string(bytes) + "\nplan_mallocs " + std::to_string(mallocs) + "\nbudget " +
                  std::to_string(plan->device_bytes) + "\nplanned_kernels " + std::to_string(plan->launches) + "\nkernels " + std::to_string(W.kernels) + "\ndone " + std::to_string(done) + "\nforks " + std::to_string(W.forks) + "\njoins " +
                  std::to_string(W.joins) + "\nwait " + std::to_string(static_cast<int>(waited)) + "\nlast_error " + std::to_string(last) + "\nlaunches";
  for (const auto& l : W.log) t += " " + l;
  pq_free_plan(plan);
  // another plan, with the first one's events, that is never scanned
  W.last = cudaSuccess;
  pq_plan* unscanned = nullptr;
  if (pq_plan_scan(ctx, idx, &req, &unscanned, sizes.data()) != PQ_OK) return -1;
  pq_free_plan(unscanned);
  t += "\nlast_error_unscanned " + std::to_string(static_cast<int>(W.last));
  snprintf(text, cap, "%s", t.c_str());
  pq_free_index(idx);
  pq_ctx_destroy(ctx);
  return st;
}

// The host runtime (plans, user calls, arena, staging) on a CUDA that is not there:
// device memory is host memory, every copy and launch happens at once and is noted.
// Each scenario prints one line per fact for tests/test_host_runtime.py.
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <string>

#include "zmc_udf.cpp"  // struct zmc_udf is defined there

// ---------------------------------------------------------------- the CUDA that is not there
namespace {
struct Range {
  uintptr_t begin, end;
  bool meets(const Range &o) const { return begin < o.end && o.begin < end; }
};
std::vector<Range> g_uploads;       // host-to-device copies
std::vector<std::string> g_events;  // launches and counter resets, in order
bool g_sync_fails = false;
bool g_capturing = false;  // a caller's capture

void note(const char *fmt, ...) {
  char buf[256];
  va_list ap;
  va_start(ap, fmt);
  std::vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_events.push_back(buf);
}
uint32_t splits(const LaunchHdr *h) { return h->split[0] + h->split[1] + h->split[2] + h->split[3]; }
}  // namespace

extern "C" {
cudaError_t cudaGetDeviceCount(int *n) { return *n = 1, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
  std::memset(p, 0, sizeof *p);
  std::strcpy(p->name, "none");
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  return *s = reinterpret_cast<cudaStream_t>(std::malloc(1)), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  return g_sync_fails ? cudaErrorLaunchFailure : cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  return *e = reinterpret_cast<cudaEvent_t>(std::malloc(1)), cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) {
  return *p = std::aligned_alloc(256, (n + 255) & ~size_t{255}), cudaSuccess;
}
cudaError_t cudaFree(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *to, const void *from, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  if (kind == cudaMemcpyHostToDevice)
    g_uploads.push_back({reinterpret_cast<uintptr_t>(to), reinterpret_cast<uintptr_t>(to) + n});
  std::memmove(to, from, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *to, int v, size_t n, cudaStream_t) {
  note("memset");
  std::memset(to, v, n);
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  note("device sync");
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
  *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) {
  return *x = reinterpret_cast<cudaGraphExec_t>(std::malloc(1)), cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return std::free(x), cudaSuccess; }
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **args, size_t, cudaStream_t) {
  note("udf split %u", splits(*static_cast<LaunchHdr **>(args[1])));
  return cudaSuccess;
}
cudaError_t cudaLibraryLoadData(cudaLibrary_t *, const void *, cudaJitOption *, void **, unsigned,
                                cudaLibraryOption *, void **, unsigned) {
  return cudaErrorNotSupported;
}
cudaError_t cudaLibraryUnload(cudaLibrary_t) { return cudaSuccess; }
cudaError_t cudaLibraryGetKernel(cudaKernel_t *, cudaLibrary_t, const char *) {
  return cudaErrorNotSupported;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
  return *n = 2, cudaSuccess;
}
}  // extern "C"

zmc_status serving_start(zmc_ctx *) { return ZMC_OK; }
void serving_stop(zmc_ctx *) {}

namespace zmc {
cudaError_t launch_batched(int f, const Entry *, LaunchHdr *h, unsigned, unsigned, cudaStream_t, int) {
  note("batched %d split %u", f, h->split[f]);
  h->counter[f] = h->item_end[f] - h->item_begin[f];
  return cudaSuccess;
}
cudaError_t launch_merge(const FnDev *const *, LaunchHdr *h, unsigned, cudaStream_t, bool reset) {
  note("merge");
  if (reset) std::memset(h->counter, 0, sizeof h->counter);
  return cudaSuccess;
}
cudaError_t launch_finish(const Entry *, LaunchHdr *h, uint64_t, int, cudaStream_t, bool merge) {
  note("%s split %u", merge ? "finish" : "records", splits(h));
  std::memset(h->counter, 0, sizeof h->counter);
  return cudaSuccess;
}
cudaError_t launch_plain(const PlainFn &, double *, unsigned, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_plain_merge(const PlainJob *, uint32_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_philox(const uint32_t *, const uint32_t *, uint32_t *, size_t, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_eval(int, const FnDev *, uint64_t, uint32_t, float *, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_philox_rate(uint32_t, unsigned, uint32_t *, cudaStream_t) { return cudaSuccess; }
int batched_max_blocks_per_sm(int, int, int) { return 2; }
int batched_regs_per_thread(int, int) { return 128; }
unsigned plain_grid(const PlainFn &, int) { return 1; }
}  // namespace zmc

// ---------------------------------------------------------------- scenarios
namespace {

zmc_ctx *context(size_t bytes, uint32_t quints) {
  zmc_options o;
  zmc_default_options(&o);
  o.mem_budget_bytes = bytes;
  o.quints_per_lane = quints;
  zmc_ctx *c = nullptr;
  if (zmc_create(&o, &c) != ZMC_OK) std::abort();
  return c;
}

std::vector<zmc_desc> gauss_rows(size_t n, uint32_t dim, uint64_t samples) {
  zmc_desc d;
  std::memset(&d, 0, sizeof d);
  d.family = ZMC_GAUSS;
  d.dim = dim;
  d.n_samples = samples;
  d.p[0] = 1.0;
  d.p[1] = 0.1;
  for (uint32_t k = 0; k < dim; ++k) {
    d.hi[k] = 1.0;
    d.p[2 + k] = 0.5;
  }
  return std::vector<zmc_desc>(n, d);
}

zmc_udf *user(uint32_t precision) {
  auto *u = new zmc_udf;
  u->dims = {1};
  u->scales = {1.0};
  u->precision = precision;
  u->max_blocks = 2;
  u->lib = reinterpret_cast<cudaLibrary_t>(1);
  return u;
}

zmc_plan *plan(zmc_ctx *c, const std::vector<zmc_desc> &rows) {
  zmc_plan *p = nullptr;
  return zmc_plan_create(c, rows.data(), rows.size(), &p) == ZMC_OK ? p : nullptr;
}

// Parts whose staging slots and device blocks are as far apart, with room in between
// that is not theirs.
void upload_gap() {
  char dev[4096], stage[4096];
  const UploadPart parts[] = {{dev, 0, 160}, {dev + 2048, 2048, 300}, {dev + 2560, 2560, 10}};
  upload_parts(parts, 3, stage, nullptr);
  for (const Range &r : g_uploads)
    std::printf("%zu %zu\n", r.begin - reinterpret_cast<uintptr_t>(dev), r.end - r.begin);
}

// A kept plan between the header and the parameters of an FP64 user call that splits
// nothing: 1 when any of the call's copies meets one of the plan's.
void udf_next_to_plan() {
  zmc_ctx *c = context(8 << 20, 13);
  std::vector<zmc_desc> rows = gauss_rows(400, 1, 1);
  for (size_t i = 0; i < 264; ++i) rows[i].n_samples = 2 * 2080 + 1;  // 928 chunks in all
  zmc_plan *hole = plan(c, rows);
  g_uploads.clear();
  zmc_plan *kept = plan(c, gauss_rows(1, 1, 1));
  const std::vector<Range> mine = g_uploads;
  zmc_plan_destroy(hole);
  g_uploads.clear();
  std::vector<zmc_desc> user_rows = gauss_rows(440, 1, 1);
  std::vector<UdfRow> ur(user_rows.size());
  for (size_t i = 0; i < ur.size(); ++i) ur[i] = row_of(user_rows[i]);
  std::vector<zmc_result> out(ur.size());
  const zmc_status st = udf_run(c, user(ZMC_UDF_F64), ur.data(), ur.size(), out.data());
  int met = 0;
  for (const Range &a : g_uploads)
    for (const Range &b : mine) met += a.meets(b);
  std::printf("%d %d\n", st, met > 0);
  zmc_plan_destroy(kept);
  zmc_destroy(c);
}

// Two tables that exactly fill the arena, the first with chunks to split: 1 when the
// second is taken as well.
std::vector<zmc_desc> unlike_rows(size_t n) {
  std::vector<zmc_desc> rows = gauss_rows(n, 1, 1);
  for (size_t i = 0; i < n; i += 2) rows[i] = gauss_rows(1, 7, 1)[0];
  return rows;
}
size_t table_bytes(size_t n) {  // records, results, descriptors, entries, merge list, header
  return round256(n * 8) + round256(n * sizeof(zmc_result)) + round256(n * sizeof(FnDev)) +
         round256(n * sizeof(Entry)) + round256(n * 8) + 256;
}
void two_tables(bool serving) {
  zmc_options o;
  zmc_default_options(&o);
  o.mem_budget_bytes = 2 * table_bytes(1000);
  o.quints_per_lane = 104;
  o.serving = serving;
  zmc_ctx *c = nullptr;
  if (zmc_create(&o, &c) != ZMC_OK) std::abort();
  zmc_plan *a = plan(c, unlike_rows(1000)), *b = plan(c, unlike_rows(1000));
  std::printf("%d %d\n", a != nullptr, b != nullptr);
  zmc_plan_destroy(a);
  zmc_plan_destroy(b);
  zmc_destroy(c);
}

// A sampled plan whose scratch a later table takes: what was launched for it.
void scratch_taken_after_sampling() {
  zmc_ctx *c = context(table_bytes(1000) + split_bytes(1000, 1000, 104) + 4096, 104);
  zmc_plan *a = plan(c, unlike_rows(1000));
  zmc_plan_run(a, ZMC_STAGE_SAMPLE);
  g_events.clear();
  zmc_plan *b = plan(c, unlike_rows(1000));
  std::printf("%d\n", b != nullptr);
  for (const std::string &e : g_events) std::printf("%s\n", e.c_str());
  zmc_plan_destroy(a);
  zmc_plan_destroy(b);
  zmc_destroy(c);
}

// Split chunks that a plan's next sampling hands out.
unsigned split_of(zmc_plan *p) {
  g_events.clear();
  zmc_plan_run(p, ZMC_STAGE_SAMPLE);
  unsigned n = 0, f = 0, k = 0;
  for (const std::string &e : g_events)
    if (std::sscanf(e.c_str(), "batched %u split %u", &f, &k) == 2) n += k;
  return n;
}

// Three plans with scratch, and a table that has room after one of them gave its back
// (rows) or that has no room whatever they give.
void scratch_taken_from(size_t rows) {
  const size_t one = table_bytes(1000) + split_bytes(1000, 1000, 104);
  zmc_ctx *c = context(3 * one + 4096, 104);
  zmc_plan *a[3], *b;
  for (zmc_plan *&p : a) p = plan(c, unlike_rows(1000));
  b = plan(c, unlike_rows(rows));
  std::printf("%d\n", b != nullptr);
  unsigned whole = 0;
  for (zmc_plan *p : a) whole += split_of(p) == 0;
  std::printf("%u\n", whole);
  for (zmc_plan *p : a) zmc_plan_destroy(p);
  zmc_plan_destroy(b);
  zmc_destroy(c);
}

// The wait for a plan's last launches fails while its scratch is taken back.
void scratch_cannot_be_taken() {
  zmc_ctx *c = context(table_bytes(1000) + split_bytes(1000, 1000, 104) + 4096, 104);
  zmc_plan *a = plan(c, unlike_rows(1000)), *b = nullptr;
  const std::vector<zmc_desc> rows = unlike_rows(1000);
  g_sync_fails = true;
  std::printf("%d\n", zmc_plan_create(c, rows.data(), rows.size(), &b));
  g_sync_fails = false;
  std::printf("%d\n", zmc_plan_run(a, ZMC_STAGE_ALL));
  zmc_plan_destroy(a);
  zmc_destroy(c);
}

// Split chunks of a plan at first, with its scratch taken, and run again after the table
// that took it has gone.
void scratch_comes_back() {
  zmc_ctx *c = context(table_bytes(1000) + split_bytes(1000, 1000, 104) + 4096, 104);
  zmc_plan *a = plan(c, unlike_rows(1000));
  std::printf("%u", split_of(a));
  zmc_plan *b = plan(c, unlike_rows(1000));
  zmc_plan_run(a, ZMC_STAGE_ALL);
  std::printf(" %u", split_of(a));
  zmc_plan_destroy(b);
  zmc_plan_run(a, ZMC_STAGE_ALL);
  std::printf(" %u\n", split_of(a));
  zmc_plan_destroy(a);
  zmc_destroy(c);
}

// What a caller's graph of the sampling stage holds, what a run holds after that graph
// may have been replayed, and what taking the scratch back then does.
void captured_by_a_caller() {
  zmc_ctx *c = context(table_bytes(1000) + split_bytes(1000, 1000, 104) + 4096, 104);
  zmc_plan *a = plan(c, unlike_rows(1000)), *b;
  const auto run = [&](uint32_t stages) {
    g_events.clear();
    zmc_plan_run(a, stages);
    for (const std::string &e : g_events) std::printf("%s; ", e.c_str());
    std::printf("\n");
  };
  g_capturing = true;
  run(ZMC_STAGE_SAMPLE);
  g_capturing = false;
  run(ZMC_STAGE_MERGE);
  run(ZMC_STAGE_SAMPLE);
  zmc_plan_run(a, ZMC_STAGE_MERGE);
  g_events.clear();
  b = plan(c, unlike_rows(1000));
  for (const std::string &e : g_events) std::printf("%s; ", e.c_str());
  std::printf("\n");
  zmc_plan_destroy(a);
  zmc_plan_destroy(b);
  zmc_destroy(c);
}

// With the geometry tuner: what it times for a table of 3000 chunks, and the launch of
// one row after it.
void tuned_geometry() {
  zmc_options o;
  zmc_default_options(&o);
  o.mem_budget_bytes = 64 << 20;
  o.quints_per_lane = 104;
  o.autotune = ZMC_TUNE_GEOMETRY;
  zmc_ctx *c = nullptr;
  if (zmc_create(&o, &c) != ZMC_OK) std::abort();
  zmc_plan *a = plan(c, unlike_rows(3000));
  std::printf("%s\n", g_events.empty() ? "nothing" : g_events[0].c_str());
  g_events.clear();
  zmc_plan *b = plan(c, gauss_rows(1, 1, 100000));
  zmc_plan_info i;
  zmc_plan_info_get(b, &i);
  std::printf("%zu %u %u %d\n", g_events.size(), i.family_grid[2], i.family_block[2],
              i.tune_source[2]);
  zmc_plan_destroy(a);
  zmc_plan_destroy(b);
  zmc_destroy(c);
}

// Of each table the chunks that its plan splits.
void split_rule() {
  zmc_ctx *c = context(64 << 20, 104);
  const auto of = [&](const std::vector<zmc_desc> &rows) {
    zmc_plan *p = plan(c, rows);
    zmc_plan_info i;
    zmc_plan_info_get(p, &i);
    zmc_plan_destroy(p);
    return i.split_chunks;
  };
  const auto alike = [&](uint32_t dim, std::initializer_list<int> counts) {
    for (int n : counts) std::printf("%u ", of(gauss_rows(n, dim, 1)));
    std::printf("\n");
  };
  alike(1, {1, 851, 852, 1216, 1217, 1629, 1630, 2432, 2433, 9000});
  alike(3, {1, 972, 973, 1216, 1217, 1945, 1946, 2432, 2433, 9000});
  for (int n : {2433, 3404, 3405, 3648, 3649, 4864, 4865})  // whole chunks: 1 to 2 waves
    std::printf("%u ", of(gauss_rows(n, 3, 16640)));
  // 2800 chunks of 0.99 and 0.79 waves of work
  std::printf("%u %u\n", of(gauss_rows(400, 3, 100000)), of(gauss_rows(2800, 3, 11400)));
  std::vector<zmc_desc> rows = gauss_rows(3000, 2, 1);  // two and three dimensions: alike
  for (size_t i = 0; i < rows.size(); i += 2) rows[i] = gauss_rows(1, 3, 1)[0];
  std::printf("%u %u %u ", of(rows), of(unlike_rows(2000)), of(unlike_rows(3000)));
  for (zmc_desc &d : rows) {  // constants
    d.family = ZMC_POLY;
    d.deg = 0;
  }
  std::printf("%u\n", of(rows));
  zmc_destroy(c);
}

}  // namespace

int main(int, char **argv) {
  const std::string what = argv[1];
  if (what == "upload_gap") upload_gap();
  if (what == "udf_next_to_plan") udf_next_to_plan();
  if (what == "two_tables") two_tables(false);
  if (what == "two_serving_tables") two_tables(true);
  if (what == "scratch_taken_after_sampling") scratch_taken_after_sampling();
  if (what == "scratch_taken_from") scratch_taken_from(std::strtoul(argv[2], nullptr, 10));
  if (what == "scratch_cannot_be_taken") scratch_cannot_be_taken();
  if (what == "scratch_comes_back") scratch_comes_back();
  if (what == "captured_by_a_caller") captured_by_a_caller();
  if (what == "tuned_geometry") tuned_geometry();
  if (what == "split_rule") split_rule();
  return 0;
}

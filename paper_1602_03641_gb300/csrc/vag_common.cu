// Shared device utilities: budget-checked allocation, exclusive scan, status.
#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "vag_internal.cuh"

namespace vag {

static std::atomic<unsigned long long> g_launches{0};
static thread_local bool t_capturing = false;
void set_capturing(bool on) { t_capturing = on; }
void note_launches(unsigned long long n) {
  if (!t_capturing) g_launches.fetch_add(n, std::memory_order_relaxed);
}
unsigned long long launches_so_far() { return g_launches.load(std::memory_order_relaxed); }

// ------------------------------------------------------------------ trace ---
// With the environment variable VAG_TRACE set, the phases of each API call
// are marked with a device event and a host clock reading on the call's
// stream, and printed to stderr when the call ends (device time between
// consecutive marks, and host time spent issuing them).  Off by default;
// marks are skipped while a graph is being captured.
namespace {
struct TraceMark {
  const char *label;
  cudaEvent_t ev;
  std::chrono::steady_clock::time_point host;
};
thread_local std::vector<TraceMark> t_marks;
bool trace_on() {
  static const bool on = std::getenv("VAG_TRACE") != nullptr;
  return on;
}
}  // namespace

bool trace_enabled() { return trace_on(); }

void trace_mark(cudaStream_t st, const char *label) {
  if (!trace_on() || t_capturing) return;
  cudaEvent_t e;
  if (cudaEventCreate(&e) != cudaSuccess) return;
  cudaEventRecord(e, st);
  t_marks.push_back({label, e, std::chrono::steady_clock::now()});
}

void trace_report(const char *call) {
  if (!trace_on() || t_marks.empty()) return;
  cudaEventSynchronize(t_marks.back().ev);
  std::fprintf(stderr, "[vag trace] %s\n", call);
  for (size_t i = 1; i < t_marks.size(); ++i) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, t_marks[i - 1].ev, t_marks[i].ev);
    const double host = std::chrono::duration<double, std::milli>(t_marks[i].host - t_marks[i - 1].host).count();
    std::fprintf(stderr, "  %-34s device %9.3f ms   host %9.3f ms\n", t_marks[i].label, ms, host);
  }
  for (auto &m : t_marks) cudaEventDestroy(m.ev);
  t_marks.clear();
}

void loop_destroy(LoopGraph &g) {
  if (g.exec) cudaGraphExecDestroy(g.exec);
  g = LoopGraph{};
}

void loop_build(LoopGraph &g, cudaStream_t st, const std::function<void(cudaGraphConditionalHandle)> &body) {
  loop_destroy(g);
  struct Graph {   // released on every path
    cudaGraph_t g = nullptr;
    ~Graph() {
      if (g) cudaGraphDestroy(g);
    }
  } top;
  VAG_CUDA(cudaGraphCreate(&top.g, 0));
  cudaGraphConditionalHandle h;
  VAG_CUDA(cudaGraphConditionalHandleCreate(&h, top.g, 1, cudaGraphCondAssignDefault));
  cudaGraphNodeParams p{};
  p.type = cudaGraphNodeTypeConditional;
  p.conditional.handle = h;
  p.conditional.type = cudaGraphCondTypeWhile;
  p.conditional.size = 1;
  cudaGraphNode_t node;
  VAG_CUDA(cudaGraphAddNode(&node, top.g, nullptr, nullptr, 0, &p));
  cudaGraph_t inner = p.conditional.phGraph_out[0];   // owned by the conditional node
  VAG_CUDA(cudaStreamBeginCaptureToGraph(st, inner, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
  set_capturing(true);
  try {
    body(h);
  } catch (...) {
    set_capturing(false);
    cudaStreamEndCapture(st, &inner);
    throw;
  }
  set_capturing(false);
  VAG_CUDA(cudaStreamEndCapture(st, &inner));
  VAG_CUDA(cudaGraphGetNodes(inner, nullptr, &g.nodes));
  VAG_CUDA(cudaGraphInstantiate(&g.exec, top.g, 0));
}

void *ctx_alloc(Ctx *c, size_t bytes) {
  void *p = nullptr;
  cudaError_t e = c->pool ? cudaMallocFromPoolAsync(&p, bytes, c->pool, c->stream) : cudaMalloc(&p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    fail(VAG_ENOMEM, "device allocation of " + std::to_string(bytes) + " bytes failed");
  }
  return p;
}

void ctx_free(Ctx *c, void *p) {
  if (!p) return;
  if (c->pool) cudaFreeAsync(p, c->stream);
  else cudaFree(p);
}

int *ctx_pin(Ctx *c) {
  if (!c->pin) VAG_CUDA(cudaMallocHost(&c->pin, kPinWords * sizeof(int)));
  return c->pin;
}

void *ctx_stage(Ctx *c, size_t bytes) {
  if (bytes > c->stage_bytes) {
    if (c->stage) VAG_CUDA(cudaFreeHost(c->stage));
    c->stage = nullptr;
    c->stage_bytes = 0;
    bytes = std::max<size_t>(2 * bytes, 16384);
    VAG_CUDA(cudaMallocHost(&c->stage, bytes));
    c->stage_bytes = bytes;
  }
  return c->stage;
}

void *sys_alloc_bytes(System *s, size_t bytes) {
  Ctx *c = s->ctx;
  bytes = (std::max<size_t>(bytes, 1) + 255) & ~size_t(255);   // a zero-size array still gets a valid pointer
  if (c->budget && c->in_use + bytes > c->budget)
    fail(VAG_EBUDGET, "device memory budget exceeded (" + std::to_string(c->in_use + bytes) +
                          " > " + std::to_string(c->budget) + " bytes)");
  void *p = ctx_alloc(c, bytes);
  s->allocs.push_back({p, bytes});
  s->bytes += bytes;
  c->in_use += bytes;
  return p;
}

void sys_free_all(System *s) {
  for (auto &a : s->allocs) ctx_free(s->ctx, a.ptr);
  if (s->ctx) s->ctx->in_use -= s->bytes;
  s->allocs.clear();
  s->bytes = 0;
}

int num_sms() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

int grid_for(int64_t n, int block) {
  int64_t g = (n + block - 1) / block;
  if (g < 1) g = 1;
  if (g > 0x7fffffff) g = 0x7fffffff;
  return (int)g;
}

int read_status(System *s) {
  int *pin = ctx_pin(s->ctx);
  VAG_CUDA(cudaMemcpyAsync(pin, s->status, sizeof(int), cudaMemcpyDeviceToHost, s->ctx->stream));
  VAG_CUDA(cudaStreamSynchronize(s->ctx->stream));
  return *pin;
}

// ------------------------------------------------------------------ scan ----
// Tiles of 4096 values: one kernel sums the tiles, a second one scans them,
// each block first adding the sums of the tiles before its own (a few
// thousand values from L2 even for 10^7 inputs).  Two launches whatever the
// length, one up to 4096 values; the scans of the setup phases are short and
// many, so that launches are what they cost (tiles of 1024 with a recursive
// scan of their sums took two to seven).
namespace {
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

// exclusive prefix of v over the block's threads; *total in every thread
__device__ __forceinline__ int block_exclusive_sum(int v, int *total) {
  __shared__ int warp_tot[kScanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();   // warp_tot may still be read from a previous call
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  int before = 0, sum = 0;
#pragma unroll
  for (int w = 0; w < kScanThreads / 32; ++w) {
    if (w < warp) before += warp_tot[w];
    sum += warp_tot[w];
  }
  *total = sum;
  return incl - v + before;
}

__global__ void __launch_bounds__(kScanThreads) scan_sums(const int *__restrict__ in, int *__restrict__ sums, int n) {
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  int v = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const int64_t k = base + i * kScanThreads + threadIdx.x;
    v += k < n ? in[k] : 0;
  }
  int tot;
  block_exclusive_sum(v, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanThreads) scan_write(const int *__restrict__ in, const int *__restrict__ sums,
                                                           int *__restrict__ out, int n) {
  int before = 0;
  for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanThreads) before += sums[b];
  int offset, tot;
  block_exclusive_sum(before, &offset);
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  int v[kScanItems];
  int sum = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = base + i < n ? in[base + i] : 0;
    sum += v[i];
  }
  int run = offset + block_exclusive_sum(sum, &tot);
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < n) out[base + i] = run;
    run += v[i];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = offset + tot;
}
}  // namespace

int scan_exclusive(Ctx *c, const int *in, int *out, int n, bool want_total) {
  cudaStream_t st = c->stream;
  if (n == 0) {
    VAG_CUDA(cudaMemsetAsync(out, 0, sizeof(int), st));
    return 0;
  }
  const int ntiles = (int)(((int64_t)n + kScanTile - 1) / kScanTile);
  Scratch scratch(c);
  int *sums = ntiles > 1 ? scratch.get<int>(ntiles) : nullptr;
  if (ntiles > 1) scan_sums<<<ntiles, kScanThreads, 0, st>>>(in, sums, n);
  scan_write<<<ntiles, kScanThreads, 0, st>>>(in, sums, out, n);
  VAG_CHECK_LAUNCH();
  note_launches(ntiles > 1 ? 2 : 1);
  if (!want_total) return -1;
  int *pin = ctx_pin(c);
  VAG_CUDA(cudaMemcpyAsync(pin, out + n, sizeof(int), cudaMemcpyDeviceToHost, st));
  VAG_CUDA(cudaStreamSynchronize(st));
  return *pin;
}

}  // namespace vag

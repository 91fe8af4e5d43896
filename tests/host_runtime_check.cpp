// The host runtime (snn_host.cpp) on a fake CUDA runtime: device memory is host
// memory, copies are memcpy, streams do nothing, and the kernels' launchers note
// what they were given.  Built and run by test_host_runtime.py, one check per run.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <set>

#include "snn_host.cpp"

#define CHECK(c)                                                       \
  do {                                                                 \
    if (!(c)) {                                                        \
      std::printf("%s:%d: %s (%s)\n", __FILE__, __LINE__, #c, g_last_error.c_str()); \
      std::exit(1);                                                    \
    }                                                                  \
  } while (0)

// ---- fake CUDA runtime
static std::vector<cudaStream_t> g_graph_streams;   // of every graph launched
static uintptr_t g_next_id = 16;
template <class T>
static cudaError_t new_handle(T *out) {
  *out = reinterpret_cast<T>(g_next_id += 16);
  return cudaSuccess;
}
extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return (*p = std::aligned_alloc(256, (n + 255) / 256 * 256)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetLimit(size_t *v, cudaLimit) { *v = 0; return cudaSuccess; }
cudaError_t cudaDeviceSetLimit(cudaLimit, size_t) { return cudaSuccess; }
cudaError_t cudaCtxResetPersistingL2Cache() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return new_handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return new_handle(g); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { return new_handle(x); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphUpload(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return new_handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return new_handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { g_graph_streams.push_back(s); return cudaSuccess; }
}

// ---- fake kernels
static uint32_t g_fit = 0xFFFFFFFFu;           // tiles of one launch of the persistent kernel
static int g_fail_at = -1;                     // its launch that reports a barrier that was not met,
static bool g_fail_launch = false;             // or fails itself
static std::vector<std::vector<std::pair<uint32_t, uint32_t>>> g_runs;   // windows of every launch's networks
namespace snn {
int device_sm_count() { return 152; }
cudaError_t prepare_kernels() { return cudaSuccess; }
cudaError_t prepare_run_kernels() { return cudaSuccess; }
cudaError_t launch_build_rows(const NetDev &, const BuildDev &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_init_state(const NetDev &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_update(const NetDev &, uint32_t, StepMod, int, int, const L2Window &, bool, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_deliver(const NetDev &, uint32_t, StepMod, uint32_t, int, int, const L2Window &, bool, cudaStream_t) { return cudaSuccess; }
RunShape run_shape(uint32_t n_tiles, uint32_t, int threads, uint32_t, bool) {
  RunShape s;
  s.blocks = n_tiles <= g_fit ? 1 : 0;
  s.threads = threads;
  return s;
}
cudaError_t launch_run(const RunArgs &a, const RunShape &, const L2Window &, cudaStream_t) {
  std::vector<std::pair<uint32_t, uint32_t>> w;
  for (uint32_t i = 0; i < a.n_nets; ++i) {
    const NetWin &x = a.n_nets > 1u ? a.wins[i] : a.win;
    w.emplace_back(x.t0, x.t_end);
    // the exchange period is counted from one phase for all networks that advance
    if (x.t_end > x.t0) CHECK(a.phase == x.t0 % a.kmin);
  }
  const int at = (int)g_runs.size();
  g_runs.push_back(w);
  if (at == g_fail_at && g_fail_launch) return cudaErrorLaunchOutOfResources;
  if (at == g_fail_at) *a.status |= kStatusBarrier;
  return cudaSuccess;
}
}  // namespace snn

// ---- networks
static snn_params params(int gx, int n_delay, int min_delay) {
  snn_params p{};
  p.gx = gx;
  p.gy = 1;
  p.lambda = 1.0f;
  p.p_local = 0.8f;
  p.out_degree = 8;
  p.n_delay = n_delay;
  p.min_delay = min_delay;
  p.dt_ms = 0.1f;
  p.bin_steps = 50;
  for (int q = 0; q < 3; ++q) {
    p.tau_m[q] = 20.0f;
    p.C_m[q] = 1.0f;
    p.V_th[q] = 20.0f;
    p.V_r[q] = 15.0f;
    p.tau_arp[q] = 2.0f;
    p.tau_c[q] = 1000.0f;
    p.J_ext[q] = 0.8f;
  }
  return p;
}
static std::vector<snn_handle> networks(int n, int n_delay, int min_delay, int window, int gx = 1) {
  std::vector<snn_handle> hs(n);
  for (int i = 0; i < n; ++i) {
    const snn_params p = params(gx, n_delay, min_delay);
    CHECK(snn_build_network(&p, 5 + i, reinterpret_cast<void *>(uintptr_t(i + 1)), &hs[i]) == SNN_OK);
    snn_launch c;
    CHECK(snn_get_launch(hs[i], &c) == SNN_OK);
    c.window_steps = window;
    CHECK(snn_set_launch(hs[i], &c) == SNN_OK);
  }
  return hs;
}
static void free_all(std::vector<snn_handle> &hs) {
  for (auto h : hs) snn_free(h);
}

// Every network that advances in a launch has the phase the launch counts its
// exchange periods from, also after others have stopped (launch_run checks).
static void check_phase() {
  for (int kmin : {2, 10, 33}) {
    auto hs = networks(4, 40, kmin, 12);
    uint32_t x = 1;
    std::vector<uint64_t> t(hs.size());
    for (int call = 0; call < 40; ++call) {
      std::vector<uint64_t> steps(hs.size());
      for (size_t i = 0; i < hs.size(); ++i) {
        x = x * 1664525u + 1013904223u;
        steps[i] = x >> 16 & 1u ? (x >> 17) % 90u : 0u;
        t[i] += steps[i];
      }
      CHECK(snn_run_batch(hs.data(), steps.data(), (int)hs.size()) == SNN_OK);
    }
    for (size_t i = 0; i < hs.size(); ++i) CHECK(hs[i]->t == t[i]);
    free_all(hs);
  }
}

// A launch that fails: of its networks, those whose windows it (or one still in
// flight) was to advance answer SNN_ERR_STATE from then on; the others go on.
static void check_failure() {
  const uint64_t one[1] = {1};
  for (bool launch : {false, true})
    for (int at : {0, 1, 2, 3}) {
      auto hs = networks(4, 20, 1, 10);
      const std::vector<uint64_t> steps = {15, 200, 0, 200};
      g_runs.clear();
      g_fail_at = at;
      g_fail_launch = launch;
      CHECK(snn_run_batch(hs.data(), steps.data(), 4) == SNN_ERR_CUDA);
      g_fail_at = -1;
      for (int i = 0; i < 4; ++i) {
        const uint64_t undrained = launch ? (uint64_t)(10 * at) : (uint64_t)(10 * at + 20);   // issued: two in flight
        const uint64_t drained = launch ? (uint64_t)(10 * std::max(0, at - 1)) : (uint64_t)(10 * at);
        const bool lost = std::min(steps[i], undrained) > std::min(steps[i], drained);
        CHECK(hs[i]->t == std::min(steps[i], drained));
        CHECK(snn_run_batch(&hs[i], one, 1) == (lost ? SNN_ERR_STATE : SNN_OK));
      }
      free_all(hs);
    }
  // the same of a single network
  auto hs = networks(1, 20, 1, 10);
  g_runs.clear();
  g_fail_at = 1;
  g_fail_launch = true;
  CHECK(snn_run(hs[0], 100) == SNN_ERR_CUDA);
  CHECK(snn_run(hs[0], 1) == SNN_ERR_STATE);
  free_all(hs);
  g_fail_at = -1;
  g_fail_launch = false;
}

// Networks too large for a launch of the persistent kernel advance side by side
// on streams of their own, also when the caller gave them one stream.
static void check_large() {
  g_fit = 12;   // a network of one module has 10 tiles, one of two 20
  for (bool one_stream : {false, true}) {
    std::vector<snn_handle> hs;
    for (int gx : {2, 1, 2, 2}) hs.push_back(networks(1, 20, 3, 10, gx)[0]);
    for (size_t i = 0; i < hs.size(); ++i) hs[i]->stream = reinterpret_cast<cudaStream_t>(uintptr_t(one_stream ? 1 : i + 1));
    const std::vector<uint64_t> steps = {25, 25, 0, 40};
    g_runs.clear();
    g_graph_streams.clear();
    CHECK(snn_run_batch(hs.data(), steps.data(), 4) == SNN_OK);
    for (size_t i = 0; i < hs.size(); ++i) CHECK(hs[i]->t == steps[i]);
    CHECK(g_runs.size() == 3 && g_graph_streams.size() == 3 + 4);
    // the second network's first window is launched before the first network's third
    std::set<cudaStream_t> first(g_graph_streams.begin(), g_graph_streams.begin() + 4);
    CHECK(first.size() == 2);
    free_all(hs);
  }
}

// Only grids that the persistent kernel can take hold its further input buffers.
static void check_footprint() {
  for (int kmin : {1, 4})
    for (int gx : {2, 1900, 2000}) {   // 2.375M and 2.5M neurons, around 128 tiles on each of 152 SMs
      const Layout L = make_layout(params(gx, 20, kmin));
      CHECK(L.off_rows - L.off_more == (gx < 2000 ? (size_t)kMaxVisit * L.N_pad * 4 : 0u));
      CHECK(L.off_more == L.off_hist + (size_t)L.D * L.N_pad * 4);
    }
}

// What a set costs does not depend on the sets before it: its windows' tables
// hold its own networks only.
static void check_tables() {
  const auto copied = [](std::vector<snn_handle> &hs) {
    std::vector<uint64_t> steps(hs.size(), 30);
    uint64_t bytes[2];
    for (uint64_t &b : bytes) {
      snn_stats st;
      CHECK(snn_get_stats(hs[0], &st) == SNN_OK);
      b = st.h2d_bytes;
      if (&b == bytes) CHECK(snn_run_batch(hs.data(), steps.data(), (int)hs.size()) == SNN_OK);
    }
    return bytes[1] - bytes[0];
  };
  auto two = networks(2, 20, 1, 10), many = networks(100, 20, 1, 10);
  const uint64_t before = copied(two);
  CHECK(copied(many) > 20 * before);
  CHECK(copied(two) == before);
  free_all(two);
  free_all(many);
}

// Which pairs run as two kernels per step on their own streams.
static void check_pairs() {
  const struct {
    int a, b;
    bool apart;
  } pairs[] = {{400, 399, false}, {400, 400, true}, {400, 600, true}, {400, 601, false}, {559, 839, false}, {560, 841, true}};
  for (const auto &p : pairs) {
    std::vector<snn_handle> hs = {networks(1, 20, 1, 10, p.a)[0], networks(1, 20, 1, 10, p.b)[0]};
    for (int i = 0; i < 2; ++i) hs[i]->stream = reinterpret_cast<cudaStream_t>(uintptr_t(i + 1));
    const uint64_t steps[2] = {20, 20};
    g_graph_streams.clear();
    CHECK(snn_run_concurrent(hs.data(), steps, 2) == SNN_OK);
    CHECK(!g_graph_streams.empty() == p.apart);
    free_all(hs);
  }
}

int main(int argc, char **argv) {
  const std::map<std::string, void (*)()> checks = {{"phase", check_phase}, {"failure", check_failure}, {"large", check_large}, {"footprint", check_footprint}, {"tables", check_tables}, {"pairs", check_pairs}};
  if (argc != 2 || !checks.count(argv[1])) return 2;
  checks.at(argv[1])();
  std::puts("ok");
  return 0;
}

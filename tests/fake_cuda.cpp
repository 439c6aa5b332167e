// A CUDA runtime and kernels of host memory, to run the host side of the library (dd_tv.cu,
// compiled as C++) without a GPU: device memory is malloc'ed, a stream executes at once,
// stream capture records what a graph launch then executes.  Every kernel launch leaves a
// line in a log; of the kernels' work only as much is done as tells one state from another:
// an inner iteration of the full-dimension path adds 1 to the first pixel of u.
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <string>
#include <vector>

#include "../paper_1901_00682_gb300/csrc/internal.cuh"

using namespace ddtv;

namespace {

using Work = std::vector<std::function<void()>>;
Work* g_capture = nullptr;   // the capture under way
std::string g_log;
size_t g_fail_bytes = 0;     // an allocation of at least this size fails (0: none does)
int g_operations = 0;        // put on the stream (copies, memsets, launches)
bool g_chain = false;        // the local solves make the multiplier update
int g_allocations = 0;
int g_fail_at = 0;           // the allocation that fails, counted from here (0: none does)
cudaError_t g_prepare_error = cudaSuccess;

cudaError_t enqueue(std::function<void()> f) {
  ++g_operations;
  if (g_capture) g_capture->push_back(std::move(f));
  else f();
  return cudaSuccess;
}

cudaError_t launch(std::string line, std::function<void()> f = [] {}) {
  return enqueue([line, f] {
    g_log += line + "\n";
    f();
  });
}

std::string masked(const uint8_t* mask) { return mask ? " masked" : ""; }

}  // namespace

extern "C" {

const char* fake_log() { return g_log.c_str(); }
void fake_clear_log() { g_log.clear(); }
void fake_fail_allocations(size_t at_least_bytes) { g_fail_bytes = at_least_bytes; }
int fake_allocations() { return g_allocations; }
int fake_operations() { return g_operations; }
void fake_chain(int on) { g_chain = on; }
void fake_fail_allocation(int k) { g_fail_at = k; }
void fake_fail_prepare(int error) { g_prepare_error = (cudaError_t)error; }

cudaError_t cudaMalloc(void** p, size_t n) {
  ++g_allocations;
  if ((g_fail_bytes && n >= g_fail_bytes) || (g_fail_at && --g_fail_at == 0)) return cudaErrorMemoryAllocation;
  *p = std::calloc(n, 1);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  return enqueue([=] { std::memcpy(d, s, n); });
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  return enqueue([=] { std::memset(d, v, n); });
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  if (g_capture) return cudaErrorIllegalState;
  g_capture = new Work;
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = g_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = (cudaGraph_t)g_capture;
  g_capture = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long) {
  *x = (cudaGraphExec_t) new Work(*(Work*)g);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
  if (g_capture) return cudaErrorStreamCaptureUnsupported;
  for (auto& f : *(Work*)x) f();
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  delete (Work*)g;
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
  delete (Work*)x;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = nullptr;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}
cudaError_t cudaStreamCreate(cudaStream_t* s) {
  *s = nullptr;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }

}  // extern "C"

namespace ddtv {

// ---- local solves (one launch each), multiplier updates
bool fused_chains(const Grid&, int, int, double) { return g_chain; }
cudaError_t fused_prepare(const Grid&, int, int, double) { return g_prepare_error; }
bool fused_out_of_place(const Grid&, int) { return true; }
void fused_max_tile(int* r, int* c) { *r = *c = 128; }
int fused_num_variants() { return 4; }
cudaError_t launch_fused_local(const LocalArgs& a, int, int, cudaStream_t) { return launch("local" + masked(a.mask)); }
cudaError_t launch_interface(const Grid&, float, Strips, Strips, float*, float*, cudaStream_t) {
  return launch("interface");
}
cudaError_t launch_extract_strips(const Grid&, const float*, const float*, Strips, const float*, const float*, Strips,
                                  cudaStream_t) {
  return launch("extract");
}
cudaError_t launch_scatter_strips(const Grid&, Strips, float*, float*, cudaStream_t) { return launch("scatter"); }
cudaError_t launch_chain_rebuild(int, int, const float*, const float*, float*, const float*, const float*, float*,
                                 cudaStream_t) {
  return launch("rebuild");
}
cudaError_t launch_init_u(const Grid& g, int, const float* f, const uint8_t*, float* u, cudaStream_t) {
  return launch("init", [=] { std::memcpy(u, f, sizeof(float) * g.H * g.W); });
}

// ---- full-dimension and plain paths
cudaError_t full_prepare(int) { return g_prepare_error; }
int full_max_steps() { return 10; }
cudaError_t launch_full(const FullArgs& a, int, int n, cudaStream_t) {
  const float* in = a.in.u;
  float* out = a.out.u;
  const size_t px = (size_t)a.H * a.W;
  return launch("full" + masked(a.mask), [=] {
    std::memcpy(out, in, px * sizeof(float));
    out[0] += n;
  });
}
cudaError_t launch_plain_phat(const LocalArgs&, float*, float*, float*, float*, cudaStream_t) { return launch("phat"); }
cudaError_t launch_plain_ustep(const LocalArgs& a, const float*, const float*, const Coef*, int, cudaStream_t) {
  return launch("ustep" + masked(a.mask));
}
cudaError_t launch_plain_pstep(const LocalArgs& a, const float*, const float*, float*, float*, const Coef*, bool,
                               cudaStream_t) {
  float* u = a.u;
  return launch("pstep", [=] { u[0] += 1; });
}

// ---- reductions
int reduce_partials_count() { return 1; }
int sum_f64_partials_count() { return 1; }
cudaError_t launch_energy(const Grid&, int, float, float, float, const float*, const float*, const uint8_t*,
                          const float*, const float*, double*, unsigned int*, double*, cudaStream_t) {
  return launch("energy");
}
cudaError_t launch_row_tv(const float*, const float*, int, double*, cudaStream_t) { return launch("row_tv"); }
cudaError_t launch_sum_f64(const double*, long long, double*, unsigned int*, double*, cudaStream_t) {
  return launch("sum");
}
cudaError_t launch_wait_probe(int*, unsigned long long*, cudaStream_t) { return launch("probe"); }

// ---- reverse pass
long long adj_alpha_slots(const Grid&) { return 1; }
long long adj_alpha_slots_fused(const Grid&) { return 1; }
size_t adj_fused_tape_floats(const Grid&, int) { return 1; }
cudaError_t adj_fused_prepare(const Grid&) { return cudaSuccess; }
cudaError_t launch_adj_fused(const LocalArgs&, const AdjArgs&, int, cudaStream_t) { return launch("reverse"); }
cudaError_t launch_adj_inner(const AdjArgs&, const Coef*, const float*, const uint8_t*, const uint8_t*, bool, bool,
                             cudaStream_t) {
  return launch("reverse inner");
}
cudaError_t launch_adj_interface(const AdjArgs&, float, float, cudaStream_t) { return launch("reverse interface"); }
cudaError_t launch_adj_initial(const AdjArgs&, cudaStream_t) { return launch("reverse initial"); }
cudaError_t launch_ustep_tape(const LocalArgs&, const int4*, const int4*, const float*, const float*, const Coef*, int,
                              float*, cudaStream_t) {
  return launch("ustep tape");
}
cudaError_t launch_pstep_tape(const LocalArgs&, const int4*, const int4*, const float*, const float*, float*, float*,
                              const Coef*, uint8_t*, uint8_t*, cudaStream_t) {
  return launch("pstep tape");
}

}  // namespace ddtv

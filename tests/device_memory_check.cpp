// Host check of what the library does when device memory runs out: test code, built
// by tests/test_device_memory.py from the library's host objects and the fake CUDA
// runtime below (a byte budget, no GPU; the kernel launches only count).  For a
// growing budget it compresses a matrix, multiplies a few right-hand sides, makes the
// first adjoint product and a product on host buffers.  The buffers of batch passes
// are optional: once a budget suffices, no larger one may fail, the smallest that
// suffices runs single products and the largest runs batches.  Everything allocated
// is freed.
// Two to eight right-hand sides run as batches in every format when the buffers are there.
// usage: device_memory_check <points file> n eps codec leaf format
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "program.h"

using namespace hm;

static int g_fails = 0;
#define CHECK(cond)                                                         \
  do {                                                                      \
    if (!(cond) && g_fails++ < 20) std::printf("FAIL line %d: %s\n", __LINE__, #cond); \
  } while (0)

static size_t g_budget = 0, g_used = 0;
static std::map<void*, size_t> g_mem;
static std::map<std::string, int> g_calls;

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = nullptr;
  if (n > g_budget - g_used) return cudaErrorMemoryAllocation;
  *p = std::malloc(n ? n : 1);
  g_mem[*p] = n;
  g_used += n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  CHECK(g_mem.count(p) == 1);
  g_used -= g_mem[p];
  g_mem.erase(p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
  *f = g_budget - g_used;
  *t = g_budget;
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void* d, int v, size_t n) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) { return std::memset(p, 0, sizeof *p), cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* g, cudaGraph_t, unsigned long long) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}

namespace hm {
#define LAUNCH(name, ...) \
  cudaError_t name(__VA_ARGS__) { return ++g_calls[#name], cudaSuccess; }
using I = const int32_t*;
using S = cudaStream_t;
LAUNCH(kernels_init)
LAUNCH(batch_init)
LAUNCH(mr_init)
LAUNCH(tc_init)
LAUNCH(launch_gather, const double*, I, int, float2*, S)
LAUNCH(launch_cdot, int, int, const ItemCopy*, I, int, const uint8_t*, const float2*, F2, F2*, float2*, int*, S)
LAUNCH(launch_fanout, I, int, float2*, const float2*, S)
LAUNCH(launch_gsum, const GsumOut*, int, const F2*, const F2*, F2, float2*, I, I, I, int, S)
LAUNCH(launch_rgemv, int, int, int, const PieceCopy*, I, int, const uint8_t*, const float2*, double, F2, double, double*,
       I, float2*, const F2*, F2*, int32_t*, const Split*, int*, S)
LAUNCH(launch_rseq, int, int, const SeqPhase*, int, const PieceCopy*, I, const uint8_t*, float2*, double, F2, double,
       double*, I, const F2*, F2*, int32_t*, const Split*, const SeqDep*, unsigned*, int, int*, S)
LAUNCH(launch_prog, int, int, const ProgPhase*, int, const double*, const ItemCopy*, const GsumOut*, const F2*, F2*, I,
       const PieceCopy*, I, const SeqPhase*, const SeqDep*, unsigned*, int, const uint8_t*, float2*, double, double,
       double*, I, const F2*, F2*, int32_t*, const Split*, I, I, I, int*, S)
LAUNCH(launch_cdot_tc, const ItemCopy*, I, int, const uint8_t*, const float*, F2, float*, float*, int*, S)
LAUNCH(launch_cdot_ws, const ItemCopy*, I, int, const uint8_t*, const float*, F2, float*, float*, int*, S)
LAUNCH(launch_gather_mr, const double*, int64_t, int, I, int, float*, S)
LAUNCH(launch_gsum_mr, const GsumOut*, int, int64_t, const F2*, const float*, F2, float*, S)
LAUNCH(launch_rgemv_tc, int, const PieceCopy*, I, int, const uint8_t*, const float*, double, F2, double, double*, int64_t,
       int, I, float*, const F2*, F2*, int32_t*, const Split*, I, int32_t, int*, S)
LAUNCH(launch_rgemv_ms, int, const PieceCopy*, I, int, const uint8_t*, const float*, double, F2, double, double*, int64_t,
       int, I, float*, const F2*, F2*, int32_t*, const Split*, I, int32_t, int*, S)
LAUNCH(launch_gather_b, int, const double*, int64_t, int, I, int, float2*, S)
LAUNCH(launch_gsum_b, int, const GsumOut*, int, const F2*, const float2*, F2, float2*, S)
LAUNCH(launch_cdot_b, int, int, const ItemCopy*, I, int, const uint8_t*, const float2*, F2, float2*, float2*, int*, S)
LAUNCH(launch_rgemv_b, int, int, int, const PieceCopy*, I, int, const uint8_t*, float2*, F2, double, double*, int64_t, int,
       I, const F2*, F2*, int64_t, int32_t*, int, const Split*, I, int32_t, int*, S)
LAUNCH(launch_decode, const uint8_t*, int64_t, int, int, int, int, double, double*, S)
LAUNCH(launch_decode_debug, int, const DbgTask*, int64_t, const uint8_t*, float2*, int*, S)
int rseq_max_blocks() { return 152; }
int prog_max_blocks() { return 152; }
int batch_shape(int, int) { return 1; }
}  // namespace hm

int main(int argc, char** argv) {
  if (argc != 7) return 2;
  const int64_t n = std::atoll(argv[2]);
  std::vector<double> pts(3 * n), x(64 * n, 1.0), y(64 * n, 0.0);
  FILE* f = std::fopen(argv[1], "rb");
  if (!f || std::fread(pts.data(), 8, 3 * n, f) != (size_t)(3 * n)) return 2;
  std::fclose(f);
  hm_build_params prm{};
  prm.kernel = HM_KERNEL_LAPLACE;
  prm.eta = 2.0;
  prm.eps_build = std::atof(argv[3]);
  prm.leaf_size = std::atoi(argv[5]);
  prm.format = std::atoi(argv[6]);
  prm.nthreads = 4;
  struct Result {
    hm_status s;
    bool batch;
    size_t used;
  };
  auto attempt = [&](size_t budget) {
    g_budget = budget;
    g_calls.clear();
    hm_matrix* M = nullptr;
    Result r{hm_build(&prm, pts.data(), n, &M), false, 0};
    if (r.s == HM_OK) r.s = hm_compress(M, prm.eps_build, std::atoi(argv[4]), 1);
    if (r.s == HM_OK) r.s = hm_matvec(M, 1.0, x.data(), n, 0.0, y.data(), n, 3, nullptr);
    r.batch = g_calls["launch_gather_b"] > 0;
    if (r.s == HM_OK) CHECK(g_calls["launch_gather_b"] + g_calls["launch_gather"] >= 1);
    if (r.s == HM_OK) r.s = hm_matvec_adjoint(M, 1.0, x.data(), n, 0.0, y.data(), n, 1, nullptr);
    if (r.s == HM_OK) r.s = hm_matvec_host(M, 1.0, x.data(), 0.0, y.data(), 64, nullptr);
    r.used = g_used;
    hm_free(M);
    CHECK(g_used == 0 && g_mem.empty());
    return r;
  };
  g_budget = size_t(1) << 40;
  for (int r = 2; r <= 8; ++r) {
    hm_matrix* M = nullptr;
    CHECK(hm_build(&prm, pts.data(), n, &M) == HM_OK && hm_compress(M, prm.eps_build, std::atoi(argv[4]), 1) == HM_OK);
    g_calls.clear();
    CHECK(hm_matvec(M, 1.0, x.data(), n, 0.0, y.data(), n, r, nullptr) == HM_OK);
    CHECK(g_calls["launch_gather_b"] >= 1 && g_calls["launch_gather"] <= (r == 5));
    hm_free(M);
  }
  const Result all = attempt(size_t(1) << 40);
  CHECK(all.s == HM_OK && all.batch);
  // budgets up to that use and the room that batches ask for, in steps finer than any of their buffers' sum
  size_t first = 0;
  int seen = 0;
  const size_t top = 4 * all.used + (size_t(256) << 20);
  for (size_t b = all.used / 16; b < top; b += b < 2 * all.used ? all.used / 64 : top / 32) {
    const Result r = attempt(b);
    if (r.s == HM_OK && !first) {
      first = b;
      CHECK(!r.batch);
    }
    CHECK(r.s == HM_OK || (!first && r.s == HM_ERR_OOM));
    seen += r.batch;
  }
  CHECK(first > 0 && seen > 0);
  std::printf("used %zu, first %zu\n", all.used, first);
  std::printf(g_fails ? "FAILED %d\n" : "ok\n", g_fails);
  return g_fails != 0;
}

// Which kernels a call launches, without a GPU: the library's own objects linked
// against a stand-in for the CUDA runtime.  Device memory is host memory, a
// launch only records the kernel's name, and a cooperative launch of a kernel
// whose name contains `refused` fails the way the runtime refuses one whose
// CTAs do not fit the SMs a context may use.  Built and run by
// tests/test_launch_routes.py.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "grom.h"

static std::map<const void*, std::string> g_names;
static std::vector<std::string> g_launched;
static std::string g_refused;
static cudaError_t g_last = cudaSuccess;

static cudaError_t launched(const void* f) {
  g_launched.push_back(g_names[f]);
  return cudaSuccess;
}
static CUresult fake_encode() { return CUDA_SUCCESS; }

extern "C" {
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = *b = dim3(1);
  *s = 0;
  *static_cast<void**>(st) = nullptr;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t) {
  return launched(reinterpret_cast<const void*>(k));
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void**) { return launched(f); }
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t) {
  if (!g_refused.empty() && g_names[f].find(g_refused) != std::string::npos)
    return g_last = cudaErrorCooperativeLaunchTooLarge;
  return launched(f);
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "refused"; }
cudaError_t cudaMalloc(void** p, size_t n) {
  n = (n + 255) / 256 * 256 + 256;
  *p = aligned_alloc(256, n);
  if (*p) memset(*p, 0, n);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
  for (size_t y = 0; y < h; ++y) memcpy(static_cast<char*>(d) + y * dp, static_cast<const char*>(s) + y * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  *a = cudaPointerAttributes{};
  a->type = cudaMemoryTypeDevice;
  a->devicePointer = const_cast<void*>(p);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return cudaMalloc(p, 2 << 20); }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = 1, cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { return *n = 76, cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *f = reinterpret_cast<void*>(fake_encode);
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
static int g_handle;
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = reinterpret_cast<cudaEvent_t>(&g_handle), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  return *s = reinterpret_cast<cudaStream_t>(&g_handle), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamGetDevice(cudaStream_t, int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
  return *st = cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  return *g = reinterpret_cast<cudaGraph_t>(&g_handle), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  return *x = reinterpret_cast<cudaGraphExec_t>(&g_handle), cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t*, size_t* n) { return *n = 0, cudaSuccess; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType*) { return cudaSuccess; }
cudaError_t cudaGraphEventRecordNodeGetEvent(cudaGraphNode_t, cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaGraphExecEventRecordNodeSetEvent(cudaGraphExec_t, cudaGraphNode_t, cudaEvent_t) { return cudaSuccess; }
}

static long bad = 0, checks = 0;
static void check(bool ok, const char* what) {
  ++checks;
  if (ok) return;
  ++bad;
  std::printf("FAIL %s; launched:", what);
  for (const std::string& k : g_launched) std::printf(" %s", k.c_str());
  std::printf("; %s\n", grom_last_error());
}
static bool ran(const char* kernel) {
  for (const std::string& k : g_launched)
    if (k.find(kernel) != std::string::npos) return true;
  return false;
}

// An FP64 CP ROM (skew, n = 64, r = 48).
static grom_rom* cp_rom(std::vector<double>& data, int batch) {
  const int n = 64, r = 48;
  data.assign((size_t)3 * n * r + n, 0.25);
  grom_desc d{};
  d.n = n;
  d.rank = r;
  d.form = GROM_FORM_CP_SKEW;
  d.storage = GROM_F64;
  d.fa = data.data();
  d.fb = d.fa + n * r;
  d.fc = d.fb + n * r;
  d.stiffness_diag = d.fc + n * r;
  d.nu = 1e-2;
  d.dt = 1e-3;
  d.order = 3;
  d.max_batch = batch;
  grom_rom* rom = nullptr;
  check(grom_create(&d, nullptr, &rom) == GROM_OK, "create");
  return rom;
}

// A cooperative launch that cannot be placed: the evaluation takes the two
// plain kernels, the steps the next path, and no call fails for it.
static void refused_launches() {
  std::vector<double> data, u(64 * 4, 0.5), c(64 * 4);
  grom_rom* rom = cp_rom(data, 4);
  grom_traj* t = nullptr;
  check(grom_traj_create(rom, 1, u.data(), &t) == GROM_OK, "trajectory");
  for (int batch : {1, 4}) {
    for (const char* refused : {"", "k3x"}) {
      g_refused = refused;
      g_launched.clear();
      check(grom_nonlinear(rom, batch, u.data(), c.data()) == GROM_OK, "evaluation succeeds");
      check(ran("k3x_eval") == g_refused.empty() && (g_launched.size() == 2) == !g_refused.empty(), "evaluation's kernels");
      check(g_last == cudaSuccess, "no error left behind by the evaluation");
    }
  }
  const struct {
    const char *refused, *kernel;
  } steps[] = {{"", "k3x_kernel"}, {"k3x", "k3p_kernel"}, {"k3", "project"}};
  for (const auto& s : steps) {
    g_refused = s.refused;
    g_launched.clear();
    check(grom_step(t, 8, nullptr, nullptr) == GROM_OK, "steps succeed");
    check(ran(s.kernel), s.kernel);
    check(g_last == cudaSuccess, "no error left behind by the steps");
  }
  g_refused.clear();
  grom_traj_destroy(t);
  grom_destroy(rom);
}

// A dense full ROM with a CTA per test index: one kernel an evaluation, two
// where c is u (a CTA of the one-kernel form writes c while others read u).
static void whole_test_indices() {
  for (int storage : {GROM_F64, GROM_F32X2, GROM_F32, GROM_BF16}) {
    const int n = 64;
    std::vector<double> C((size_t)n * n * n, 0.125), a(n, 1.0), u(8 * n, 0.5), c(8 * n);
    grom_desc d{};
    d.n = n;
    d.form = GROM_FORM_FULL;
    d.storage = storage;
    d.tensor = C.data();
    d.stiffness_diag = a.data();
    d.nu = 1e-2;
    d.dt = 1e-3;
    d.order = 3;
    d.max_batch = 8;
    grom_rom* rom = nullptr;
    check(grom_create(&d, nullptr, &rom) == GROM_OK, "create");
    for (int batch : {1, 8}) {
      g_launched.clear();
      check(grom_nonlinear(rom, batch, u.data(), c.data()) == GROM_OK, "evaluation");
      const size_t apart = g_launched.size();
      check(!ran("k1_finalize"), "no second kernel");
      g_launched.clear();
      check(grom_nonlinear(rom, batch, u.data(), u.data()) == GROM_OK, "evaluation in place");
      check(ran("k1_finalize") && g_launched.size() == 2 * apart, "the sums in a second kernel where c is u");
    }
    grom_destroy(rom);
  }
}

int main() {
  refused_launches();
  whole_test_indices();
  std::printf("%ld checks, %ld failed\n", checks, bad);
  return bad ? 1 : 0;
}

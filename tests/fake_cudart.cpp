// fake_cudart.cpp -- a stand-in for the CUDA runtime on the host, for tests of the library's host code and error
// paths without a GPU: device memory is host memory, kernels do nothing but call a hook, and the n-th allocation
// (or any named call) can be made to fail.  Linked with the library's objects; no CUDA header is needed.
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

struct dim3 {
  unsigned x, y, z;
};
typedef void (*Hook)(const char* kernel, unsigned gx, unsigned gy, unsigned gz, size_t smem, void** args);

typedef std::map<char*, size_t> Blocks;
static Blocks& live() {  // device memory
  static Blocks m;
  return m;
}
static Blocks& pinned() {
  static Blocks m;
  return m;
}
static std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}
static std::map<std::string, int>& limits() {  // dynamic shared memory allowed per kernel
  static std::map<std::string, int> m;
  return m;
}
static Hook hook = nullptr;
static long fail_at = -1;          // allocations until one fails (-1: none)
static std::string fail_call;      // a call that fails
static int last_error = 0, blocks_per_sm = 4;
static dim3 cfg_grid, cfg_block;
static size_t cfg_smem;
static void* cfg_stream;

static int ret(int e) {
  if (e) last_error = e;
  return e;
}
static int alloc(Blocks& m, void** p, size_t n) {
  if (fail_at >= 0 && fail_at-- == 0) return ret(2);
  *p = std::calloc(n ? n : 1, 1);
  m[(char*)*p] = n;
  return 0;
}
static int release(Blocks& m, void* p) {
  if (!p) return 0;
  if (!m.erase((char*)p)) return ret(1);
  std::free(p);
  return 0;
}
static int run(const void* k, dim3 g, size_t smem, void** args) {
  const std::string& n = names()[k];
  if (fail_call == n) return ret(1);
  const auto it = limits().find(n);
  if (smem > 48 * 1024 && (it == limits().end() || (size_t)it->second < smem)) return ret(1);
  if (hook) hook(n.c_str(), g.x, g.y, g.z, smem, args);
  return 0;
}

extern "C" {
// ---- for the tests ----
void fake_hook(Hook h) { hook = h; }
void fake_fail_alloc(long n) { fail_at = n; }
long fake_fail_alloc_left() { return fail_at; }  // -1: it has failed
void fake_forget_limits() { limits().clear(); }
void fake_fail_call(const char* name) { fail_call = name; }
void fake_blocks_per_sm(int n) { blocks_per_sm = n; }
int fake_pending_error() { return last_error; }
int fake_limit(const char* kernel) {
  const auto it = limits().find(kernel);
  return it == limits().end() ? 0 : it->second;
}
size_t fake_allocations() { return live().size() + pinned().size(); }
size_t fake_room(const void* p) {  // bytes from p to the end of its live allocation (0: in none)
  auto it = live().upper_bound((char*)p);
  if (it == live().begin()) return 0;
  --it;
  const char* end = it->first + it->second;
  return (const char*)p < end ? end - (const char*)p : 0;
}
void* fake_find(size_t bytes) {  // the device allocation of this size
  for (auto& a : live())
    if (a.second == bytes) return a.first;
  return nullptr;
}

// ---- the runtime ----
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
  names()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void* st) {
  cfg_grid = g, cfg_block = b, cfg_smem = smem, cfg_stream = st;
  return 0;
}
int __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void** st) {
  *g = cfg_grid, *b = cfg_block, *smem = cfg_smem, *st = cfg_stream;
  return 0;
}
int __cudaGetKernel(const void** k, const void* host) {
  *k = host;
  return 0;
}
int __cudaLaunchKernel(const void* k, dim3 g, dim3, void** args, size_t smem, void*) { return run(k, g, smem, args); }
int cudaLaunchKernel(const void* k, dim3 g, dim3, void** args, size_t smem, void*) { return run(k, g, smem, args); }
int cudaLaunchCooperativeKernel(const void* k, dim3 g, dim3, void** args, size_t smem, void*) {
  return run(k, g, smem, args);
}
int cudaFuncSetAttribute(const void* k, int attr, int v) {
  if (fail_call == "cudaFuncSetAttribute") return ret(1);
  if (attr == 8) limits()[names()[k]] = v;  // cudaFuncAttributeMaxDynamicSharedMemorySize
  return 0;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  if (fail_call == "cudaOccupancy") return ret(1);
  *n = blocks_per_sm;
  return 0;
}
int cudaGetLastError() {
  const int e = last_error;
  last_error = 0;
  return e;
}
int cudaGetDevice(int* d) {
  *d = 0;
  return 0;
}
int cudaDeviceGetAttribute(int* v, int attr, int) {
  *v = attr == 16 ? 152 : 1;  // cudaDevAttrMultiProcessorCount
  return 0;
}
int cudaDeviceSynchronize() { return 0; }
int cudaMalloc(void** p, size_t n) { return alloc(live(), p, n); }
int cudaHostAlloc(void** p, size_t n, unsigned) { return alloc(pinned(), p, n); }
int cudaMallocHost(void** p, size_t n) { return alloc(pinned(), p, n); }
int cudaFree(void* p) { return release(live(), p); }
int cudaFreeHost(void* p) { return release(pinned(), p); }
int cudaMemset(void* p, int v, size_t n) {
  if (v || n < 1 << 20) std::memset(p, v, n);  // large allocations stay untouched, as they came: zero
  return 0;
}
int cudaMemsetAsync(void* p, int v, size_t n, void*) { return cudaMemset(p, v, n); }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) {
  std::memmove(d, s, n);
  return 0;
}
int cudaStreamSynchronize(void*) { return 0; }
int cudaEventCreate(void** e) {
  *e = nullptr;
  return 0;
}
int cudaEventDestroy(void*) { return 0; }
int cudaEventRecord(void*, void*) { return 0; }
int cudaEventSynchronize(void*) { return 0; }
int cudaEventElapsedTime(float* ms, void*, void*) {
  *ms = 1.f;
  return 0;
}
// not reached by the tests
#define UNUSED(f) \
  int f() { return ret(801); }
UNUSED(cudaStreamUpdateCaptureDependencies)
UNUSED(cudaStreamIsCapturing)
UNUSED(cudaStreamGetCaptureInfo)
UNUSED(cudaStreamEndCapture)
UNUSED(cudaStreamDestroy)
UNUSED(cudaStreamCreateWithFlags)
UNUSED(cudaStreamBeginCaptureToGraph)
UNUSED(cudaStreamBeginCapture)
UNUSED(cudaGraphLaunch)
UNUSED(cudaGraphInstantiate)
UNUSED(cudaGraphExecDestroy)
UNUSED(cudaGraphDestroy)
UNUSED(cudaGraphConditionalHandleCreate)
UNUSED(cudaGraphAddNode)
UNUSED(cudaGetSymbolAddress)
UNUSED(cudaGetDriverEntryPointByVersion)
}

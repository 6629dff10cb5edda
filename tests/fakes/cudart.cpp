// A CUDA runtime without a GPU, for tests of the library's host code: device
// memory is host memory, kernels do not run, and any call can be made to fail.
// It has the entry points that the library's objects refer to.
#include <cstddef>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
struct Dim {
  unsigned x, y, z;
};
struct Config {  // the start of cudaLaunchConfig_t
  Dim grid, block;
  size_t smem;
  void* stream;
};
std::map<const void*, std::string> names;
std::map<std::string, int> limits;  // cudaFuncAttributeMaxDynamicSharedMemorySize per kernel
std::string launches;                // "name gx gy gz threads smem limit\n" per launch
constexpr int kOk = 0, kMalloc = 2, kUnknown = 999, kDefaultSmem = 48 * 1024;
int last = kOk;

}  // namespace

extern "C" {
long fake_calls, fake_fail_at, fake_live, fake_ones;  // ones: device-to-host copies deliver 32-bit ones

const char* fake_launches() { return launches.c_str(); }
void fake_reset(long fail_at, long ones) {
  fake_calls = 0;
  fake_fail_at = fail_at;
  fake_ones = ones;
  last = kOk;
  launches.clear();
}

static int step(int error) {
  if (++fake_calls != fake_fail_at) return kOk;
  return last = error;
}

static int launch(const void* f, Dim g, Dim b, size_t smem) {
  const std::string& n = names[f];
  const int limit = limits.count(n) ? limits[n] : kDefaultSmem;
  launches += n + " " + std::to_string(g.x) + " " + std::to_string(g.y) + " " + std::to_string(g.z) + " " +
              std::to_string(b.x * b.y * b.z) + " " + std::to_string(smem) + " " + std::to_string(limit) + "\n";
  return step(kUnknown);
}

int cudaMalloc(void** p, size_t n) {
  if (int e = step(kMalloc)) return e;
  *p = calloc(1, n ? n : 1);
  ++fake_live;
  return kOk;
}
int cudaFree(void* p) {
  if (p) --fake_live;
  free(p);
  return kOk;
}
int cudaMemcpy(void* d, const void* s, size_t n, int kind) {
  if (int e = step(kUnknown)) return e;
  memcpy(d, s, n);
  if (kind == 2 && fake_ones)
    for (size_t i = 0; i + 4 <= n; i += 4) *reinterpret_cast<int*>(static_cast<char*>(d) + i) = 1;
  return kOk;
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void*) { return cudaMemcpy(d, s, n, kind); }
int cudaMemset(void* d, int v, size_t n) {
  if (int e = step(kUnknown)) return e;
  memset(d, v, n);
  return kOk;
}
int cudaMemsetAsync(void* d, int v, size_t n, void*) { return cudaMemset(d, v, n); }
int cudaStreamSynchronize(void*) { return step(kUnknown); }
int cudaDeviceSynchronize() { return step(kUnknown); }
int cudaEventRecord(void*, void*) { return step(kUnknown); }
int cudaGetDevice(int* d) {
  *d = 0;
  return kOk;
}
int cudaDeviceGetAttribute(int* v, int, int) {
  *v = 152;
  return kOk;
}
int cudaFuncSetAttribute(const void* f, int, int v) {
  if (int e = step(kUnknown)) return e;
  limits[names[f]] = v;
  return kOk;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t smem, unsigned) {
  if (int e = step(kUnknown)) return e;
  *n = (int)(228 * 1024 / (smem + 39 * 1024));  // (as for k_row)
  return kOk;
}
int cudaGetSymbolAddress(void** p, const void* s) {
  *p = const_cast<void*>(s);
  return kOk;
}
const char* cudaGetErrorString(int) { return "injected"; }
int cudaGetLastError() {
  const int e = last;
  last = kOk;
  return e;
}

// what nvcc's host code calls to register and launch kernels
static Config pushed;
void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
  names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(Dim g, Dim b, size_t smem, void* st) {
  pushed = Config{g, b, smem, st};
  return 0;
}
int __cudaPopCallConfiguration(Dim* g, Dim* b, size_t* smem, void* st) {
  *g = pushed.grid;
  *b = pushed.block;
  *smem = pushed.smem;
  *static_cast<void**>(st) = pushed.stream;
  return kOk;
}
int __cudaGetKernel(const void** k, const void* f) {
  *k = f;
  return kOk;
}
int __cudaLaunchKernel(const void* k, Dim g, Dim b, void**, size_t smem, void*) { return launch(k, g, b, smem); }
int cudaLaunchKernelExC(const Config* c, const void* f, void**) { return launch(f, c->grid, c->block, c->smem); }
}

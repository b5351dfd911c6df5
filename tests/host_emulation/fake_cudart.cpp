// fake_cudart.cpp -- the CUDA runtime calls that the library's host code makes, on
// host memory: copies and memsets are done, kernel launches only counted. The
// launch or memset chosen by fake_fail returns an error, as the runtime would for
// one that it refuses, and records it as the thread's last one until
// cudaGetLastError takes it (test infrastructure: no kernel runs, no GPU is used).
#include <cstddef>
#include <cstdlib>
#include <cstring>

namespace {
int g_launch = 0, g_fail_launch = -1, g_last = 0, g_memsets = 0;
bool g_fail_memsets = false;
alignas(256) unsigned char g_symbol[64 << 20];
constexpr int kInvalid = 1;

int launch() {
  const int e = g_launch++ == g_fail_launch ? kInvalid : 0;
  if (e) g_last = e;
  return e;
}
}  // namespace

extern "C" {
// the fail-th launch from now on fails (-1: none), and every memset if memsets
void fake_fail(int fail, int memsets) {
  g_launch = 0;
  g_fail_launch = fail;
  g_fail_memsets = memsets != 0;
  g_memsets = 0;
}
int fake_launches() { return g_launch; }
int fake_pending_error() { return g_last; }
int fake_memsets() { return g_memsets; }

int __cudaLaunchKernel() { return launch(); }
int cudaLaunchKernelExC() { return launch(); }
int __cudaGetKernel() { return 0; }
unsigned __cudaPushCallConfiguration() { return 0; }
int __cudaPopCallConfiguration() { return 0; }
void** __cudaRegisterFatBinary() { return nullptr; }
void __cudaRegisterFatBinaryEnd() {}
void __cudaRegisterFunction() {}
void __cudaRegisterVar() {}
void __cudaUnregisterFatBinary() {}

int cudaGetLastError() {
  const int e = g_last;
  g_last = 0;
  return e;
}
int cudaMemsetAsync(void* p, int v, size_t n) {
  ++g_memsets;
  if (g_fail_memsets) return g_last = kInvalid;
  std::memset(p, v, n);
  return 0;
}
int cudaMemset(void* p, int v, size_t n) { return cudaMemsetAsync(p, v, n); }
int cudaMemcpyAsync(void* d, const void* s, size_t n) {
  std::memcpy(d, s, n);
  return 0;
}
int cudaMemcpy(void* d, const void* s, size_t n) { return cudaMemcpyAsync(d, s, n); }
int cudaMemcpyToSymbol() { return 0; }
int cudaGetSymbolAddress(void** p) {
  *p = g_symbol;
  return 0;
}
int cudaMalloc(void** p, size_t n) { return (*p = std::malloc(n)) ? 0 : 2; }
int cudaFree(void* p) {
  std::free(p);
  return 0;
}
int cudaGetDevice(int* d) {
  *d = 0;
  return 0;
}
int cudaDeviceGetAttribute(int* v) {
  *v = 152;
  return 0;
}
int cudaSetDevice() { return 0; }
int cudaFuncSetAttribute() { return 0; }
int cudaStreamSynchronize() { return 0; }
int cudaEventCreate(void** e) {
  *e = g_symbol;
  return 0;
}
int cudaEventRecord() { return 0; }
int cudaEventSynchronize() { return 0; }
int cudaEventDestroy() { return 0; }
int cudaEventElapsedTime(float* t) {
  *t = 0.f;
  return 0;
}
int cufftCreate() { return 1; }
int cufftDestroy() { return 0; }
int cufftMakePlan3d() { return 1; }
int cufftExecD2Z() { return 1; }
int cufftSetAutoAllocation() { return 1; }
int cufftSetStream() { return 1; }
int cufftSetWorkArea() { return 1; }
}

// A CUDA runtime for host tests: memory is the host's, launches and copies are
// counted and nothing runs. The test sets the current device and an error left
// behind by an earlier call. The remaining entry points, which the test
// generates, do nothing and succeed.
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

static std::map<const void*, std::string> names;  // kernels by their host functions
static std::string launched;

extern "C" {

int fake_device = 0, fake_last_error = 0, fake_launch_error = 0;
int fake_launches = 0, fake_copies = 0, fake_waits = 0;

int cudaGetDevice(int* d) { *d = fake_device; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return 0; }
int cudaMalloc(void** p, size_t n) { *p = std::calloc(1, n); return 0; }
int cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
int cudaFree(void* p) { std::free(p); return 0; }
int cudaFreeHost(void* p) { std::free(p); return 0; }
int cudaMemsetAsync(void* p, int v, size_t n, void*) { std::memset(p, v, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) {
  std::memcpy(d, s, n);
  ++fake_copies;
  return 0;
}
int cudaStreamSynchronize(void*) { ++fake_waits; return 0; }
int cudaGetLastError() {
  const int e = fake_last_error;
  fake_last_error = 0;
  return e;
}

struct Dim3 { unsigned x, y, z; };
// the names of the kernels launched since the last call, one a line
const char* fake_launched() {
  static std::string out;
  out = launched;
  launched.clear();
  return out.c_str();
}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*,
                            void*, void*, int*) {
  names[host] = name;
}
static int launch(const void* f) {
  ++fake_launches;
  launched += names[f] + "\n";
  if (fake_launch_error) fake_last_error = fake_launch_error;
  return fake_launch_error;
}
int cudaLaunchKernel(const void* f, Dim3, Dim3, void**, size_t, void*) { return launch(f); }
int __cudaLaunchKernel(void* k, Dim3, Dim3, void**, size_t, void*) { return launch(k); }
int __cudaGetKernel(void** k, const void* f) { *k = const_cast<void*>(f); return 0; }
int __cudaPushCallConfiguration(Dim3, Dim3, size_t, void*) { return 0; }
int __cudaPopCallConfiguration(Dim3* g, Dim3* b, size_t* n, void* s) {
  *g = *b = {1, 1, 1};
  *n = 0;
  *static_cast<void**>(s) = nullptr;
  return 0;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }

}

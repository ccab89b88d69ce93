// A CUDA runtime with no device behind it: linked to the library's own objects
// in place of the real one, it records what the host side asks for (each launch's
// kernel, grid and block) so that the launchers can be tested without a GPU.
// Nothing runs; copies and fills act on host memory.
#include <chrono>
#include <cstddef>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

namespace {

struct Dim {
  unsigned x, y, z;
};
struct Launch {
  std::string kernel;
  Dim grid, block;
};
struct Config {
  Dim grid, block;
  size_t shared;
  void* stream;
};

std::mutex mu;
std::map<const void*, std::string> kernels;
std::vector<Launch> launches;
int occupancy_delay_ms = 0;
thread_local Config config;
thread_local int last_error = 0;
constexpr int kInvalidConfiguration = 9, kNotSupported = 801;

}  // namespace

extern "C" {

void** __cudaRegisterFatBinary(void* p) { return new void*(p); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void** h) { delete h; }
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
  std::lock_guard<std::mutex> g(mu);
  kernels[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(Dim grid, Dim block, size_t shared, void* stream) {
  config = {grid, block, shared, stream};
  return 0;
}
int __cudaPopCallConfiguration(Dim* grid, Dim* block, size_t* shared, void** stream) {
  *grid = config.grid;
  *block = config.block;
  *shared = config.shared;
  *stream = config.stream;
  return 0;
}
int __cudaGetKernel(const void** kernel, const void* host) {
  *kernel = host;
  return 0;
}
int __cudaLaunchKernel(const void* kernel, Dim grid, Dim block, void**, size_t, void*) {
  if (grid.x == 0 || grid.x > 0x7FFFFFFFu || block.x == 0) return last_error = kInvalidConfiguration;
  std::lock_guard<std::mutex> g(mu);
  launches.push_back({kernels[kernel], grid, block});
  return 0;
}
int cudaGetLastError() {
  const int e = last_error;
  last_error = 0;
  return e;
}
const char* cudaGetErrorString(int e) { return e == kInvalidConfiguration ? "invalid configuration" : "error"; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* blocks, const void*, int, size_t, unsigned) {
  std::this_thread::sleep_for(std::chrono::milliseconds(occupancy_delay_ms));
  *blocks = 4;
  return 0;
}
int cudaGetDevice(int* d) { return *d = 0; }
int cudaDeviceGetAttribute(int* v, int, int) {
  *v = 152;
  return 0;
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) {
  std::memcpy(d, s, n);
  return 0;
}
int cudaMemsetAsync(void* d, int v, size_t n, void*) {
  std::memset(d, v, n);
  return 0;
}
int cudaStreamSynchronize(void*) { return 0; }
// not used by the launchers under test
int cudaEventCreate(void**) { return kNotSupported; }
int cudaEventCreateWithFlags(void**, unsigned) { return kNotSupported; }
int cudaEventDestroy(void*) { return 0; }
int cudaEventElapsedTime(float*, void*, void*) { return kNotSupported; }
int cudaEventRecord(void*, void*) { return kNotSupported; }
int cudaEventSynchronize(void*) { return kNotSupported; }
int cudaFreeHost(void*) { return 0; }
int cudaGetSymbolAddress(void**, const void*) { return kNotSupported; }
int cudaHostAlloc(void**, size_t, unsigned) { return kNotSupported; }
int cudaLaunchHostFunc(void*, void (*)(void*), void*) { return kNotSupported; }
int cudaStreamCreateWithFlags(void**, unsigned) { return kNotSupported; }
int cudaStreamDestroy(void*) { return 0; }
int cudaStreamWaitEvent(void*, void*, unsigned) { return kNotSupported; }

// what a test reads and sets
__attribute__((visibility("default"))) void fake_occupancy_delay(int ms) { occupancy_delay_ms = ms; }
__attribute__((visibility("default"))) int fake_launches() {
  std::lock_guard<std::mutex> g(mu);
  return (int)launches.size();
}
__attribute__((visibility("default"))) unsigned fake_launch(int i, char* name, int cap) {
  std::lock_guard<std::mutex> g(mu);
  std::strncpy(name, launches[i].kernel.c_str(), cap - 1);
  return launches[i].grid.x;
}

}  // extern "C"

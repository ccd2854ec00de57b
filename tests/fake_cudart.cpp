// A stand-in for the CUDA runtime's host side, for CPU tests of launch code
// (preloaded in front of libcudart): device memory is host memory, kernels do
// nothing, and
// * asynchronous copies run when the runtime may run them at the latest: behind
//   the work queued before them, when something waits for them (FAKE_DEFER=1), or
//   at the call, as from a staging buffer. Their bytes go to the file FAKE_LOG;
// * the shared-memory limit of a kernel is 48 KB until it is raised, on the
//   device that is current (fake_device); a launch above it is an error;
// * with FAKE_MEMORY the device holds that many bytes.
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <map>
#include <utility>

namespace {
struct Op {
  void* dst;
  const void* src;  // null: a memset
  int value;
  size_t n;
};
std::deque<Op> queue;
uint64_t queued = 0, done = 0;
int device = 0, last_error = 0;
std::map<std::pair<int, const void*>, size_t> limit;
std::map<void*, size_t> sizes;
size_t held = 0;
struct Dim3 {
  unsigned x, y, z;
};

void run_to(uint64_t upto) {
  static FILE* log = std::getenv("FAKE_LOG") ? std::fopen(std::getenv("FAKE_LOG"), "wb") : nullptr;
  for (; done < upto; ++done) {
    const Op o = queue.front();
    queue.pop_front();
    if (o.src) std::memcpy(o.dst, o.src, o.n);
    else std::memset(o.dst, o.value, o.n);
    if (o.src && log) {
      std::fwrite(o.src, 1, o.n, log);
      std::fflush(log);
    }
  }
}
int push(const Op& o) {
  static const bool defer = std::getenv("FAKE_DEFER") && std::getenv("FAKE_DEFER")[0] == '1';
  queue.push_back(o);
  ++queued;
  if (!defer) run_to(queued);
  return 0;
}
int launch(const void* f, size_t smem) {
  const auto it = limit.find({device, f});
  if (smem > (it == limit.end() ? 48u * 1024u : it->second)) return last_error = 1;  // invalid value
  return 0;
}
}  // namespace

extern "C" {
void fake_device(int d) { device = d; }
int cudaGetDevice(int* d) { return *d = device, 0; }
int cudaDeviceGetAttribute(int* v, int, int) { return *v = 152, 0; }
int cudaGetLastError() { return std::exchange(last_error, 0); }
int cudaMalloc(void** p, size_t n) {
  static const size_t all = std::getenv("FAKE_MEMORY") ? std::strtoull(std::getenv("FAKE_MEMORY"), nullptr, 10) : ~0ull;
  if (n > all - held || !(*p = std::calloc(n ? n : 1, 1))) return 2;
  held += sizes[*p] = n;
  return 0;
}
int cudaFree(void* p) {
  run_to(queued);
  held -= sizes[p];
  sizes.erase(p);
  std::free(p);
  return 0;
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) { return push(Op{d, s, 0, n}); }
int cudaMemsetAsync(void* d, int v, size_t n, void*) { return push(Op{d, nullptr, v, n}); }
int cudaMemcpy(void* d, const void* s, size_t n, int) {
  run_to(queued);
  std::memcpy(d, s, n);
  return 0;
}
int cudaMemset(void* d, int v, size_t n) { return std::memset(d, v, n), 0; }
int cudaMemcpyToSymbol(const void*, const void*, size_t, size_t, int) { return 0; }
int cudaStreamSynchronize(void*) { return run_to(queued), 0; }
int cudaDeviceSynchronize() { return run_to(queued), 0; }
int cudaEventCreate(uint64_t** e) { return *e = new uint64_t(0), 0; }
int cudaEventCreateWithFlags(uint64_t** e, unsigned) { return cudaEventCreate(e); }
int cudaEventRecord(uint64_t* e, void*) { return *e = queued, 0; }
int cudaEventSynchronize(uint64_t* e) { return run_to(*e), 0; }
int cudaEventElapsedTime(float* ms, uint64_t*, uint64_t*) { return *ms = 0.f, 0; }
int cudaEventDestroy(uint64_t* e) { return delete e, 0; }
int cudaFuncSetAttribute(const void* f, int attr, int v) {
  if (attr == 8) limit[{device, f}] = (size_t)v;  // cudaFuncAttributeMaxDynamicSharedMemorySize
  return 0;
}
int cudaLaunchKernel(const void* f, Dim3, Dim3, void**, size_t smem, void*) { return launch(f, smem); }
int __cudaGetKernel(const void** k, const void* f) { return *k = f, 0; }
int __cudaLaunchKernel(const void* f, Dim3, Dim3, void**, size_t smem, void*) { return launch(f, smem); }
}

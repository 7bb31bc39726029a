// A stand-in for the CUDA runtime, linked with compiled objects of the library
// in place of libcudart so that their host code runs without a device.  Device
// memory is host memory.  Copies and kernels queue up and are carried out at
// the next synchronisation, the latest moment that stream semantics allow; an
// asynchronous copy reads its host source then.  Kernels compute nothing: the
// batch order that k_mlp_grad is given is recorded when the launch is carried out.
// A launch with more dynamic shared memory than its kernel's limit is refused.
// CTAs, threads and shared memory of every launch of the patch kernels are
// recorded.  Device 0 has 152 multiprocessors, device n has n.  While a stream is captured nothing is queued.  A double copied to the host
// asynchronously (a dot product) reads as one.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cstdint>
#include <cstdlib>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <mutex>
#include <numeric>
#include <random>
#include <string>
#include <thread>
#include <vector>

namespace {

std::mutex mtx;
std::deque<std::function<void()>> queue;
size_t done = 0;                                  // operations carried out so far
std::map<const void*, std::string> names;
std::map<std::string, int> calls, fail_at;        // calls of a function so far; the call of it that fails
thread_local cudaError_t last_error = cudaSuccess;
std::vector<int> orders;                          // every k_mlp_grad launch: b, perm[0..b)

std::vector<int> patch;                           // every patch kernel launch: CTAs, threads, dynamic shared memory
thread_local int device = 0;
bool capturing = false;
std::map<const void*, size_t> smem_limit;         // of a kernel; 48 KB until raised
size_t overtake = 0;                              // fake_overtake
int overtaken = 0;
std::condition_variable limit_set;

thread_local struct { dim3 grid, block; size_t smem; void* stream; } config;

bool fails(const char* f) {
  std::lock_guard<std::mutex> g(mtx);
  const int n = ++calls[f];
  return fail_at.count(f) && fail_at[f] == n;
}
cudaError_t later(std::function<void()> op) {
  std::lock_guard<std::mutex> g(mtx);
  if (!capturing) queue.push_back(std::move(op));
  return cudaSuccess;
}
// carries out what was queued before operation number `end`
cudaError_t drain(size_t end = SIZE_MAX) {
  std::lock_guard<std::mutex> g(mtx);
  for (; !queue.empty() && done < end; ++done, queue.pop_front()) queue.front()();
  return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- control
void fake_reset() {
  drain();
  std::lock_guard<std::mutex> g(mtx);
  orders.clear();
  patch.clear();
  calls.clear();
  fail_at.clear();
  last_error = cudaSuccess;
}
void fake_fail(const char* function, int call) { fail_at[function] = call; }
// the next limit below `bytes` takes effect only after one of at least `bytes`
// has, and the call that set that one returns last (each waits a second at most)
void fake_overtake(size_t bytes) {
  overtake = bytes;
  overtaken = 0;
}
int fake_patch_launches(int* out, int capacity) {
  if ((int)patch.size() <= capacity) std::copy(patch.begin(), patch.end(), out);
  const int n = (int)patch.size();
  patch.clear();
  return n;
}
int fake_calls(const char* function) { return calls[function]; }
int fake_orders(int* out, int capacity) {
  if ((int)orders.size() <= capacity) std::copy(orders.begin(), orders.end(), out);
  return (int)orders.size();
}
// the order of epochs 0 .. epochs - 1: one shuffle of the previous order each
void fake_expected_orders(unsigned long long seed, int n, int epochs, int* out) {
  std::vector<int> v(n);
  std::iota(v.begin(), v.end(), 0);
  std::mt19937_64 rng(seed);
  for (int e = 0; e < epochs; ++e) {
    std::shuffle(v.begin(), v.end(), rng);
    std::copy(v.begin(), v.end(), out + (size_t)e * n);
  }
}

// ---- runtime
cudaError_t cudaGetDevice(int* d) { return *d = device, cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return device = d, cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = std::calloc(n ? n : 1, 1);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  drain();
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  if (fails("cudaMemcpyAsync")) return last_error = cudaErrorInvalidValue;
  if (kind == cudaMemcpyDeviceToHost && n == sizeof(double)) return later([=] { *(double*)d = 1.0; });
  return later([=] { std::memcpy(d, s, n); });
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  drain();
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  if (fails("cudaMemsetAsync")) return last_error = cudaErrorInvalidValue;
  return later([=] { std::memset(d, v, n); });
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return drain(); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = (cudaEvent_t) new size_t(0), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
  std::lock_guard<std::mutex> g(mtx);
  *(size_t*)e = done + queue.size();
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return drain(*(size_t*)e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete (size_t*)e, cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return last_error; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}

cudaError_t cudaFuncSetAttribute(const void* host, cudaFuncAttribute, int value) {
  const auto second = std::chrono::seconds(1);
  std::unique_lock<std::mutex> g(mtx);
  const bool cross = overtake > 0, small = cross && (size_t)value < overtake;
  if (small) limit_set.wait_for(g, second, [] { return overtaken > 0; });
  smem_limit[host] = value;
  if (cross) ++overtaken, limit_set.notify_all();
  if (cross && !small) {
    limit_set.wait_for(g, second, [] { return overtaken > 1; });
    g.unlock();
    std::this_thread::sleep_for(second / 4);      // the other call's caller goes first
  }
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }

cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemset(void* d, int v, size_t n) { return drain(), std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return drain(); }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int dev) { return *v = dev ? dev : 152, cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return drain(); }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) { return *p = (void*)symbol, cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = 1, cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  drain();
  capturing = true;
  return fails("cudaStreamBeginCapture") ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  capturing = false;
  return *g = (cudaGraph_t)std::malloc(1), cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  return *e = (cudaGraphExec_t)std::malloc(1), cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return fails("cudaGraphLaunch"), cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return std::free((void*)g), cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return std::free((void*)e), cudaSuccess; }

// ---- cuSOLVER: every factorisation succeeds
int cusolverDnCreate(void** h) { return *h = nullptr, 0; }
int cusolverDnDestroy(void*) { return 0; }
int cusolverDnSetStream(void*, void*) { return 0; }
int cusolverDnDpotrf_bufferSize(void*, int, int, double*, int, int* n) { return *n = 1, 0; }
int cusolverDnDpotri_bufferSize(void*, int, int, double*, int, int* n) { return *n = 1, 0; }
int cusolverDnDpotrf(void*, int, int, double*, int, double*, int, int*) { return 0; }
int cusolverDnDpotri(void*, int, int, double*, int, double*, int, int*) { return 0; }

// ---- what compiled launches call
char __cudaInitModule(void**) { return 1; }
void** __cudaRegisterFatBinary(void*) {
  static void* handle[1];
  return handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*,
                            int*) {
  names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, struct CUstream_st* s) {
  config = {g, b, sm, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* s) {
  *g = config.grid;
  *b = config.block;
  *sm = config.smem;
  *(void**)s = config.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) { return *k = (cudaKernel_t)host, cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* host, void** args) {
  if (fails("launch")) return last_error = cudaErrorInvalidConfiguration;
  {
    std::lock_guard<std::mutex> g(mtx);
    const size_t limit = smem_limit.count(host) ? smem_limit[host] : 48 * 1024;
    if (cfg->dynamicSmemBytes > limit) return last_error = cudaErrorInvalidValue;
  }
  for (const char* k : {"k_upatch", "k_patch"})
    if (names[host].find(k) != std::string::npos)
      patch.insert(patch.end(), {(int)cfg->gridDim.x, (int)cfg->blockDim.x, (int)cfg->dynamicSmemBytes});
  if (names[host].find("k_mlp_grad") == std::string::npos) return cudaSuccess;
  const int* perm = *(const int**)args[4];
  const int b = *(const int*)args[5];
  return later([=] {
    orders.push_back(b);
    if (perm) orders.insert(orders.end(), perm, perm + b);
  });
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** args, size_t sm, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = g;
  cfg.blockDim = b;
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  return cudaLaunchKernelExC(&cfg, (const void*)k, args);
}

}  // extern "C"

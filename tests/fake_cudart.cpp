// A CUDA runtime without a device: the host code of the library is linked against it (tests/fake_cuda.py), so that what
// a call asks of the runtime and what it enqueues, by which thread and in which order, can be looked at on the CPU.
// No kernel runs.
#include <cuda_runtime_api.h>
#include <string.h>

#include <chrono>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

namespace {
struct Launch {
  int caller, grid, threads, cluster;
  std::string name;
};
std::mutex mutex;
std::map<const void*, std::string> names;   // host function of a kernel -> its mangled name
std::vector<Launch> launches;
int launch_pause_us = 0, device = 0, major = 10, sms = 148, query_error = 0, ask_error = 0;
int resident[17];                           // clusters of n CTAs at once
thread_local int caller = 0, last_error = 0;
cudaError_t result(const int e) {
  if (e) last_error = e;
  return (cudaError_t)e;
}
unsigned char symbol[16];
// A thread has no context until a call of the runtime that needs one binds it; the driver's functions want one.
thread_local bool bound = false;
int encode() { return bound ? 0 : 201; }
}  // namespace

extern "C" {
// ---- what the tests set and read
// query_error: of every question about a kernel; ask_error: of those about clusters
void fake_reset(int device_, int sms_, int major_, int query_error_, int ask_error_, int pause_us) {
  device = device_, sms = sms_, major = major_, query_error = query_error_, ask_error = ask_error_, launch_pause_us = pause_us;
  for (int n = 1; n <= 16; ++n) resident[n] = sms_ / n;
  launches.clear();
  last_error = 0;
}
void fake_resident(int size, int clusters) { resident[size] = clusters; }
void fake_caller(int id) { caller = id; }   // of the launches of this thread
int fake_launches() { return (int)launches.size(); }
const char* fake_launch(int i, int* caller_, int* grid, int* threads, int* cluster) {
  const Launch& l = launches[i];
  *caller_ = l.caller, *grid = l.grid, *threads = l.threads, *cluster = l.cluster;
  return l.name.c_str();
}

// ---- the runtime
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
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 1; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return result(cudaErrorNotSupported); }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return result(cudaErrorNotSupported); }
cudaError_t cudaGetDevice(int* dev) {
  if (device < 0) return result(cudaErrorNoDevice);
  *dev = device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* value, cudaDeviceAttr attr, int) {
  *value = attr == cudaDevAttrComputeCapabilityMajor ? major : attr == cudaDevAttrMultiProcessorCount ? sms : 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const int e = last_error;
  last_error = 0;
  return (cudaError_t)e;
}
cudaError_t cudaPeekAtLastError() { return (cudaError_t)last_error; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
  bound = device >= 0;
  return result(device < 0 ? cudaErrorNoDevice : query_error);
}
cudaError_t cudaSetDevice(int dev) {
  if (device < 0 || dev != device) return result(cudaErrorInvalidDevice);
  bound = true;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  bound = true;
  return *p = symbol, cudaSuccess;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void** p, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&encode);
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* cfg) {
  if (device < 0) return result(cudaErrorNoDevice);
  bound = true;
  if (query_error || ask_error) return result(query_error ? query_error : ask_error);
  *n = resident[cfg->attrs[0].val.clusterDim.x] * (cfg->blockDim.x <= 512 ? 2 : 1);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* f, void**) {
  bound = true;
  int cluster = 1;
  for (unsigned i = 0; i < cfg->numAttrs; ++i)
    if (cfg->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = (int)cfg->attrs[i].val.clusterDim.x;
  {
    std::lock_guard<std::mutex> lock(mutex);
    launches.push_back({caller, (int)cfg->gridDim.x, (int)cfg->blockDim.x, cluster, names[f]});
  }
  if (launch_pause_us) std::this_thread::sleep_for(std::chrono::microseconds(launch_pause_us));
  // a cluster that no group of SMs holds does not start
  return result(cluster > 1 && resident[cluster] == 0 ? (int)cudaErrorInvalidClusterSize : 0);
}
}

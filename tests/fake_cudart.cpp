// The CUDA runtime calls that libsbi makes, on host memory: no kernel runs, and
// the asynchronous copies and fills of a stream happen when that stream is
// synchronised (pageable sources are read at the call, as the real runtime
// does).  The library's host code linked against it shows what it orders itself
// and what it leaves to chance.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <vector>

namespace {
std::map<cudaStream_t, std::vector<std::function<void()>>> queue;
std::map<void*, size_t> live;                 // device allocations
std::vector<std::pair<void*, size_t>> made;   // the same in order, freed ones too
int launches = 0;          // kernels, those of graphs not among them
int captured = 0;          // kernels of the last capture
int overtaken = 0;         // kernels started beside unfinished work of the library's own stream
cudaStream_t capturing = nullptr, own = nullptr;   // own: the stream that captures
int cluster_size = 0;      // of the last launch that has one
std::map<unsigned, int> max_clusters;
dim3 cfg_grid, cfg_block;
size_t cfg_smem;
cudaStream_t cfg_stream;
long next_handle = 16;
std::map<cudaEvent_t, cudaStream_t> recorded;

void drain(cudaStream_t s) {
  std::vector<std::function<void()>> q;
  q.swap(queue[s]);
  for (auto& f : q) f();
}
void drain_all() {
  for (auto& s : queue) drain(s.first);
}
template <typename T>
cudaError_t handle(T* out) {
  *out = (T)(next_handle += 16);
  return cudaSuccess;
}
bool on_device(const void* p) {
  for (auto& m : live)
    if (p >= m.first && p < (char*)m.first + m.second) return true;
  return false;
}
cudaError_t launch(cudaStream_t s) {
  if (capturing) {
    ++captured;
    return cudaSuccess;
  }
  ++launches;
  if (s != own && !queue[own].empty()) ++overtaken;
  queue[s].push_back([] {});
  return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_drain() { drain_all(); }
int fake_made() { return (int)made.size(); }
void* fake_made_at(int i, size_t* bytes) {
  *bytes = made[i].second;
  return made[i].first;
}
size_t fake_live_bytes() {
  size_t n = 0;
  for (auto& a : live) n += a.second;
  return n;
}
int fake_launches() { return launches; }
int fake_captured() { return captured; }
int fake_overtaken() { return overtaken; }
int fake_cluster_size() { return cluster_size; }
void fake_max_clusters(int size, int most) { max_clusters[size] = most; }

cudaError_t cudaMalloc(void** p, size_t n) {
  *p = malloc(n);
  memset(*p, 0x5a, n);
  live[*p] = n;
  made.push_back({*p, n});
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  drain_all();
  live.erase(p);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
  if (s == capturing && s) return cudaErrorStreamCaptureUnsupported;
  queue[s].push_back([=] { memset(p, v, n); });
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* p, size_t n, cudaMemcpyKind k, cudaStream_t s) {
  if (s == capturing && s) return cudaErrorStreamCaptureUnsupported;
  if (k == cudaMemcpyHostToDevice || (k == cudaMemcpyDefault && !on_device(p))) {
    std::vector<char> staged((const char*)p, (const char*)p + n);
    queue[s].push_back([=] { memcpy(d, staged.data(), n); });
  } else {
    queue[s].push_back([=] { memcpy(d, p, n); });
  }
  return cudaSuccess;
}
// the legacy stream: not ordered with the library's non-blocking ones
cudaError_t cudaMemcpy(void* d, const void* p, size_t n, cudaMemcpyKind) {
  memcpy(d, p, n);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (s == capturing && s) return cudaErrorStreamCaptureUnsupported;
  drain(s);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle(s); }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { drain(s); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  const cudaStream_t from = recorded[e];
  if (!capturing && from != s) queue[s].push_back([=] { drain(from); });
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  capturing = own = s;
  captured = 0;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { capturing = nullptr; return handle(g); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { return handle(e); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  recorded[e] = s;
  return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { drain_all(); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) { *least = *greatest = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof(*a));
  a->type = on_device(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  a->devicePointer = const_cast<void*>(p);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static char room[1 << 20];
  *p = room;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster_size = (int)c->attrs[i].val.clusterDim.x;
  return launch(c->stream);
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
  const unsigned k = c->attrs[0].val.clusterDim.x;
  *n = max_clusters.count(k) ? max_clusters[k] : 152 / (int)k;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t s) { return launch(s); }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t s) { return launch(s); }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void*) { return handle(k); }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, struct CUstream_st* s) {
  cfg_grid = g;
  cfg_block = b;
  cfg_smem = m;
  cfg_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
  *g = cfg_grid;
  *b = cfg_block;
  *m = cfg_smem;
  *(cudaStream_t*)s = cfg_stream;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}

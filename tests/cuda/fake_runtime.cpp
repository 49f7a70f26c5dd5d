// A CUDA runtime without a GPU, for tests of the library's host code: device memory is host memory, copies
// happen at once, kernels do nothing.  It keeps account of what the host code is answerable for:
//   - work that has been launched and that no synchronisation has waited for yet, and memory that is given back
//     while such work is not ordered before it;
//   - memory that the library's pool holds, with the rules of a stream-ordered pool (a block whose free is still
//     pending cannot be trimmed; a synchronisation gives back what is above the release threshold);
//   - an error that stays pending until cudaGetLastError reads it.
// Calls can be made to fail (fake_fail), and the bytes of a kernel's argument kept (fake_watch).
// Only one host thread at a time.
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <set>
#include <string>
#include <vector>

namespace {

using Items = std::set<long>;
struct Block {
  size_t bytes;
  bool pooled;
};
struct State {
  long next = 0, bad_frees = 0;
  Items unfinished;
  std::map<cudaStream_t, Items> before{{nullptr, {}}};    // what each stream's next item comes after
  std::set<cudaStream_t> non_blocking;
  std::map<cudaEvent_t, Items> events;
  std::map<void*, Block> blocks;
  std::map<long, size_t> pending;                          // free of a pool's block, not observed complete
  size_t reserved = 0, used = 0, threshold = 0, plain = 0;
  cudaStream_t capturing = reinterpret_cast<cudaStream_t>(-1);
  cudaError_t last = cudaSuccess;
  std::string fail_call;
  int fail_skip = 0;
  cudaError_t fail_with = cudaSuccess;
  std::map<const void*, std::string> kernels;
  std::string watch;
  int watch_arg = 0;
  size_t watch_bytes = 0;
  std::vector<std::string> seen;
  long launches = 0;
  struct {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
  } config;
};
State& st() {
  static State* s = new State;      // (outlives every static destructor)
  return *s;
}

cudaError_t give(cudaError_t e) {
  if (e != cudaSuccess) st().last = e;
  return e;
}
bool injected(const char* call) {
  State& s = st();
  if (s.fail_call != call) return false;
  if (s.fail_skip-- > 0) return false;
  s.fail_call.clear();
  return true;
}
#define FAKE_ENTRY() \
  if (injected(__func__)) return give(st().fail_with)

long put(cudaStream_t stream) {
  State& s = st();
  if (stream == s.capturing) return -1;
  const long id = s.next++;
  s.before[stream].insert(id);
  s.unfinished.insert(id);
  return id;
}
// what the legacy stream comes after
Items legacy() {
  Items all;
  for (auto& b : st().before)
    if (!st().non_blocking.count(b.first)) all.insert(b.second.begin(), b.second.end());
  return all;
}
Items ordered(cudaStream_t stream) { return stream == nullptr ? legacy() : st().before[stream]; }
void finish(const Items& done) {
  State& s = st();
  for (long id : done) {
    s.unfinished.erase(id);
    s.pending.erase(id);
  }
  size_t busy = s.used;
  for (auto& p : s.pending) busy += p.second;
  s.reserved = std::max(busy, std::min(s.reserved, std::max(busy, s.threshold)));
}
void check_free(const Items& first) {
  State& s = st();
  for (long id : s.unfinished)
    if (!first.count(id) && !s.pending.count(id)) {
      ++s.bad_frees;
      return;
    }
}
void* block(size_t bytes, bool pooled) {
  State& s = st();
  void* p = nullptr;
  if (posix_memalign(&p, 256, bytes ? bytes : 1)) return nullptr;
  s.blocks[p] = {bytes, pooled};
  if (pooled) {
    size_t busy = s.used;
    for (auto& q : s.pending) busy += q.second;
    s.used += bytes;
    s.reserved = std::max(s.reserved, busy + bytes);
  } else {
    s.plain += bytes;
  }
  return p;
}

}  // namespace

// An allocation of host memory of `refuse_from` bytes or more is refused.
static size_t refuse_from = ~(size_t)0;
void* operator new(size_t n) {
  void* p = n >= refuse_from ? nullptr : std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }

extern "C" {

// ---- the tests' side ----
// The call `call` fails with `error` once, after `skip` more of them have gone through.
void fake_fail(const char* call, int skip, int error) {
  st().fail_call = call;
  st().fail_skip = skip;
  st().fail_with = (cudaError_t)error;
}
int fake_failed() { return st().fail_call.empty(); }
long fake_bad_frees() { return st().bad_frees; }
long fake_unfinished() { return (long)st().unfinished.size(); }
size_t fake_pool_reserved() { return st().reserved; }
size_t fake_pool_used() { return st().used; }
size_t fake_plain_bytes() { return st().plain; }
long fake_launches() { return st().launches; }
void fake_refuse_from(size_t bytes) { refuse_from = bytes; }
// Keep the first `bytes` bytes of argument `arg` of every launch of a kernel whose name contains `name`.
void fake_watch(const char* name, int arg, size_t bytes) {
  st().watch = name;
  st().watch_arg = arg;
  st().watch_bytes = bytes;
  st().seen.clear();
}
int fake_seen(int i, void* out) {
  if (i >= 0 && i < (int)st().seen.size()) std::memcpy(out, st().seen[i].data(), st().seen[i].size());
  return (int)st().seen.size();
}
// Work on `stream` that the library knows nothing of.
void fake_work(void* stream) { put((cudaStream_t)stream); }
void* fake_stream(int non_blocking) {
  cudaStream_t s = nullptr;
  cudaStreamCreateWithFlags(&s, non_blocking ? cudaStreamNonBlocking : 0);
  return s;
}

// ---- kernels ----
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* fn, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  st().kernels[fn] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block_, size_t smem, struct CUstream_st* stream) {
  st().config = {grid, block_, smem, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block_, size_t* smem, void* stream) {
  auto& c = st().config;
  *grid = c.grid;
  *block_ = c.block;
  *smem = c.smem;
  *(cudaStream_t*)stream = c.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) {
  *k = (cudaKernel_t)fn;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t stream) {
  FAKE_ENTRY();
  State& s = st();
  ++s.launches;
  if (s.watch_bytes && s.kernels[(const void*)k].find(s.watch) != std::string::npos)
    s.seen.emplace_back((const char*)args[s.watch_arg], s.watch_bytes);
  put(stream);
  return cudaSuccess;
}

// ---- device ----
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) { return d == 0 ? cudaSuccess : give(cudaErrorInvalidDevice); }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  FAKE_ENTRY();
  finish(Items(st().unfinished));
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "an error that a test asked for"; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = st().last;
  st().last = cudaSuccess;
  return e;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static void* scratch = std::calloc(1, 8 << 20);
  *p = scratch;
  return cudaSuccess;
}

// ---- streams, events, graphs ----
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned flags) {
  FAKE_ENTRY();
  *s = (cudaStream_t)std::malloc(1);
  st().before[*s] = {};
  if (flags & cudaStreamNonBlocking) st().non_blocking.insert(*s);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  FAKE_ENTRY();
  finish(ordered(s));
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  FAKE_ENTRY();
  st().before[s].insert(st().events[e].begin(), st().events[e].end());
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  FAKE_ENTRY();
  *e = (cudaEvent_t)std::malloc(1);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  FAKE_ENTRY();
  st().events[e] = ordered(s);
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  FAKE_ENTRY();
  finish(Items(st().events[e]));
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.0f;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  FAKE_ENTRY();
  st().capturing = s;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  st().capturing = reinterpret_cast<cudaStream_t>(-1);
  FAKE_ENTRY();
  *g = (cudaGraph_t)std::malloc(1);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  FAKE_ENTRY();
  *x = (cudaGraphExec_t)std::malloc(1);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) {
  FAKE_ENTRY();
  put(s);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

// ---- memory ----
cudaError_t cudaMalloc(void** p, size_t n) {
  FAKE_ENTRY();
  *p = block(n, false);
  return *p ? cudaSuccess : give(cudaErrorMemoryAllocation);
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
  FAKE_ENTRY();
  *p = block(n, true);
  return *p ? cudaSuccess : give(cudaErrorMemoryAllocation);
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
// of a pool's block: at once, and the caller answers for everything having finished; else after all work
cudaError_t cudaFree(void* p) {
  FAKE_ENTRY();
  State& s = st();
  if (!p) return cudaSuccess;
  if (!s.blocks.count(p)) return give(cudaErrorInvalidValue);
  const Block b = s.blocks[p];
  if (b.pooled) {
    check_free({});
    s.used -= b.bytes;
    finish({});
  } else {
    finish(Items(s.unfinished));
    s.plain -= b.bytes;
  }
  s.blocks.erase(p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t stream) {
  FAKE_ENTRY();
  State& s = st();
  if (!s.blocks.count(p)) return give(cudaErrorInvalidValue);
  check_free(ordered(stream));
  const Block b = s.blocks[p];
  if (b.pooled) {
    s.used -= b.bytes;
    s.pending[put(stream)] = b.bytes;
  } else {
    s.plain -= b.bytes;
  }
  s.blocks.erase(p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  FAKE_ENTRY();
  finish(legacy());
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  FAKE_ENTRY();
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  FAKE_ENTRY();
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
  FAKE_ENTRY();
  *p = (cudaMemPool_t)std::malloc(1);
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr a, void* v) {
  if (a == cudaMemPoolAttrReleaseThreshold) st().threshold = *(unsigned long long*)v;
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t keep) {
  State& s = st();
  size_t busy = s.used;
  for (auto& p : s.pending) busy += p.second;
  s.reserved = std::max(busy, std::min(s.reserved, keep));
  return cudaSuccess;
}

}  // extern "C"

// A CUDA runtime over host memory, for tests of the library's host code: linked with the library's
// object files in place of libcudart.  Device memory is host memory from a bounded pool,
// allocations (device or host) can be made to fail, and a launch runs nothing on a GPU: the few
// kernels whose results the host code reads are done here, the operands of the packed float
// product's kernels are checked against the live allocations, and every launch is counted by
// the kernel's name.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>

namespace {

std::map<uintptr_t, size_t>& live() {
  static auto* m = new std::map<uintptr_t, size_t>();
  return *m;
}
std::map<const void*, std::string>& names() {
  static auto* m = new std::map<const void*, std::string>();
  return *m;
}
std::map<std::string, int64_t>& launches() {
  static auto* m = new std::map<std::string, int64_t>();
  return *m;
}
size_t g_total = (size_t)1 << 40, g_used = 0;
int64_t g_dev_fail = -1, g_host_fail = -1, g_dev_calls = 0, g_host_calls = 0;
float g_event_ms = 1.0f;
int64_t g_bad = 0;  // launches whose operands are not in live memory
cudaError_t g_last = cudaSuccess;
int g_own = 0;  // > 0: an allocation of this file's own
struct Own {
  Own() { ++g_own; }
  ~Own() { --g_own; }
};

cudaError_t note(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}

bool inside(const void* p, size_t bytes) {
  const uintptr_t a = (uintptr_t)p;
  auto it = live().upper_bound(a);
  if (it == live().begin()) return false;
  --it;
  return a + bytes <= it->first + it->second;
}

// Argument layouts of the packed float product's kernels.
struct Side {
  const int64_t* ptr;
  const int32_t* idx;
  const int32_t* blk;
  const int64_t* off;
};
struct Pack {
  int64_t nb;
  const int32_t *bsize, *brow, *bcol;
  const int64_t *voff, *poff;
  int trans;
  const float* src;
  float* dst;
};
struct Args {
  const float *X, *Y;
  const void* ent;
  int64_t base;
  const void* tiles;
  uint32_t ntiles;
  unsigned int* counter;
  float* C;
};

template <typename T>
T arg(void** args, int i) {
  return *(T*)args[i];
}

void check(bool ok) { g_bad += ok ? 0 : 1; }

bool pack_ok(const Pack& p) {
  return p.nb == 0 || (inside(p.poff, 8 * (size_t)p.nb) && inside(p.dst, 4) && inside(p.src, 4));
}

void run(const std::string& n, void** a) {
  auto is = [&](const char* s) { return n.find(s) != std::string::npos; };
  if (is("tile_count_kernel")) {
    const int32_t *bs = arg<const int32_t*>(a, 0), *br = arg<const int32_t*>(a, 1), *bc = arg<const int32_t*>(a, 2);
    const int64_t nb = arg<int64_t>(a, 3);
    const int edge = arg<int>(a, 4);
    int32_t* out = arg<int32_t*>(a, 5);
    for (int64_t k = 0; k < nb; ++k) out[k] = ((bs[br[k]] + edge - 1) / edge) * ((bs[bc[k]] + edge - 1) / edge);
  } else if (is("nt_list_kernelILb0E")) {
    // one entry per matching lambda block and piece of 20 (padded) values of t
    const Side x = arg<Side>(a, 0), y = arg<Side>(a, 1);
    const int32_t *bs = arg<const int32_t*>(a, 2), *br = arg<const int32_t*>(a, 3), *bc = arg<const int32_t*>(a, 4);
    int32_t* cnt = arg<int32_t*>(a, 7);
    for (int64_t k = arg<int64_t>(a, 5); k < arg<int64_t>(a, 6); ++k) {
      int32_t c = 0;
      int64_t i = x.ptr[br[k]], j = y.ptr[bc[k]];
      while (i < x.ptr[br[k] + 1] && j < y.ptr[bc[k] + 1]) {
        if (x.idx[i] < y.idx[j]) ++i;
        else if (y.idx[j] < x.idx[i]) ++j;
        else {
          c += (((bs[x.idx[i]] + 1) & ~1) + 19) / 20;
          ++i;
          ++j;
        }
      }
      cnt[k] = c;
    }
  } else if (is("nt_list_kernelILb1E")) {
    const int64_t k1 = arg<int64_t>(a, 6), base = arg<int64_t>(a, 9);
    const int64_t* eptr = arg<const int64_t*>(a, 8);
    check(inside(eptr + k1, 8) && eptr[arg<int64_t>(a, 5)] == base &&
          (eptr[k1] == base || inside(arg<void*>(a, 10), 16 * (size_t)(eptr[k1] - base))));
  } else if (is("nt_prepare_kernel")) {
    check(pack_ok(arg<Pack>(a, 0)) && pack_ok(arg<Pack>(a, 1)));
  } else if (is("mul_f32_nt_kernel")) {
    const Args p = arg<Args>(a, 0);
    check(inside(p.X, 4) && inside(p.Y, 4) && inside(p.ent, 16) && inside(p.tiles, 32 * (size_t)p.ntiles) && inside(p.C, 4));
  }
}

cudaError_t launch(const void* f, void** args) {
  Own own;
  const std::string& n = names()[f];
  ++launches()[n];
  run(n, args);
  return cudaSuccess;
}

struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} g_cfg;

}  // namespace

// Host allocations of the library (its references bind to these, the rest of the process keeps its own).
void* operator new(size_t n) {
  if (!g_own && g_host_fail >= 0 && g_host_calls++ == g_host_fail) throw std::bad_alloc();
  if (void* p = std::malloc(n ? n : 1)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }

extern "C" {

// ---- control ----------------------------------------------------------------------------
void fake_pool(int64_t bytes) { g_total = (size_t)bytes; }
int64_t fake_used(void) { return (int64_t)g_used; }
int64_t fake_bad(void) { return g_bad; }
// The i-th device (host) allocation from now fails; -1: none.
void fake_fail_device(int64_t i) { g_dev_fail = i, g_dev_calls = 0; }
void fake_fail_host(int64_t i) { g_host_fail = i, g_host_calls = 0; }
void fake_event_ms(float ms) { g_event_ms = ms; }
int64_t fake_device_calls(void) { return g_dev_calls; }
int64_t fake_host_calls(void) { return g_host_calls; }
void fake_reset_launches(void) { launches().clear(); }
int64_t fake_launches(const char* part) {
  int64_t n = 0;
  for (const auto& kv : launches())
    if (kv.first.find(part) != std::string::npos) n += kv.second;
  return n;
}

// ---- memory -----------------------------------------------------------------------------
cudaError_t cudaMalloc(void** p, size_t n) {
  Own own;
  *p = nullptr;
  const bool fail = g_dev_fail >= 0 && g_dev_calls == g_dev_fail;
  ++g_dev_calls;
  if (fail || n > g_total - g_used) return note(cudaErrorMemoryAllocation);
  *p = std::calloc(1, n ? n : 1);
  if (!*p) return note(cudaErrorMemoryAllocation);
  live()[(uintptr_t)*p] = n;
  g_used += n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  auto it = live().find((uintptr_t)p);
  if (it != live().end()) {
    g_used -= it->second;
    live().erase(it);
    std::free(p);
  } else if (p) {
    ++g_bad;  // freed twice, or not the pool's
  }
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
  *f = g_total - g_used;
  *t = g_total;
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned int) { return (*p = std::calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned int) { return *d = h, cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { return *p = (void*)s, cudaSuccess; }

// ---- device, errors, streams, events, graphs ------------------------------------------------
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned int) { return *n = 4, cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned int) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = g_event_ms, cudaSuccess; }

// ---- registration and launches --------------------------------------------------------------
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { names()[host] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t stream) { return g_cfg = Config{grid, block, smem, stream}, 0u; }
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = g_cfg.grid;
  *block = g_cfg.block;
  *smem = g_cfg.smem;
  *(cudaStream_t*)stream = g_cfg.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { return *k = (cudaKernel_t)f, cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t) { return launch((const void*)k, args); }
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void** args, size_t, cudaStream_t) { return launch(f, args); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void** args) { return launch(f, args); }
}

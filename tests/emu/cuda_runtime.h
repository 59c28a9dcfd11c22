// Enough of the CUDA language and run time to compile the library's sources
// with a host compiler and run its kernels on the CPU: a block at a time, each
// thread a fibre, warp collectives and barriers as rendezvous (emu.cpp).
// Kernels run in the order they are enqueued; streams are all the same.
//
// emu::Shared<T> stands in for a shared-memory variable that is watched: it
// reports accesses that CUDA does not order -- two threads of a warp with no
// __syncwarp (votes, shuffles and reductions order no memory), two warps with
// no __syncthreads, one of the accesses a write -- and reads of what the block
// has not written.
#pragma once
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __shared__ static
#define __launch_bounds__(...)
#define __maxnreg__(...)
#define __align__(x) __attribute__((aligned(x)))

using std::max;
using std::min;

struct alignas(8) int2 { int x, y; };
struct alignas(16) int4 { int x, y, z, w; };
struct alignas(16) uint4 { unsigned x, y, z, w; };
struct alignas(16) float4 { float x, y, z, w; };
inline int2 make_int2(int a, int b) { return {a, b}; }
inline int4 make_int4(int a, int b, int c, int d) { return {a, b, c, d}; }
inline uint4 make_uint4(unsigned a, unsigned b, unsigned c, unsigned d) { return {a, b, c, d}; }
struct dim3 {
  unsigned x, y, z;
  dim3(unsigned a = 1, unsigned b = 1, unsigned c = 1) : x(a), y(b), z(c) {}
};

namespace emu {
extern int tid;                  // the running thread
extern dim3 bdim, bidx, gdim;
extern char* dyn;                // dynamic shared memory of the running block
extern uint64_t slot[1024];      // what each thread brings to a collective
extern uint64_t block_serial;    // blocks begun
extern uint64_t block_epoch;     // block barriers passed, over all blocks
extern uint64_t warp_epoch[32];  // __syncwarp and block barriers passed, by warp
struct T3 { int x, y, z; };
inline T3 tidx() { return {tid, 0, 0}; }
void wait_warp(bool orders_memory);
void wait_block();
void nap();
void report(const char* what);
void launch(dim3 g, dim3 b, size_t smem, std::function<void()> kernel);
void enqueue(std::function<void()> work);
void* device_alloc(size_t n);
void device_free(void* p);

template <class F>
inline auto collective(uint64_t v, F f) {
  slot[tid] = v;
  wait_warp(false);
  auto r = f(slot + (tid & ~31), tid & 31);
  wait_warp(false);
  return r;
}

template <class T>
class Shared {
 public:
  operator T() const { read(); return v_; }
  Shared& operator=(T v) { write(); v_ = v; return *this; }
  Shared& operator=(const Shared& o) { return *this = (T)o; }
  Shared& operator+=(T v) { return *this = (T)(*this) + v; }
  Shared& operator++() { return *this = (T)(*this) + 1; }
  T operator++(int) { const T v = *this; *this = v + 1; return v; }

 private:
  struct Reads { uint64_t epoch; uint32_t lanes; };  // by lanes of one warp since its last __syncwarp
  void read() const {
    const int w = tid >> 5;
    if (serial_ != block_serial) return report("read of shared memory that the block has not written");
    if (wtid_ != tid && (wtid_ >> 5 == w ? wwarp_ == warp_epoch[w] : wblock_ == block_epoch))
      report("read not ordered after another thread's write");
    if (rblock_ != block_epoch) {
      rblock_ = block_epoch;
      rwarps_ = 0;
    }
    if (!(rwarps_ >> w & 1) || reads_[w].epoch != warp_epoch[w]) reads_[w] = {warp_epoch[w], 0};
    rwarps_ |= 1u << w;
    reads_[w].lanes |= 1u << (tid & 31);
  }
  void write() {
    const int w = tid >> 5;
    if (serial_ == block_serial) {
      if (wtid_ != tid && (wtid_ >> 5 == w ? wwarp_ == warp_epoch[w] : wblock_ == block_epoch))
        report("write not ordered after another thread's write");
      if (rblock_ == block_epoch) {
        const bool mine = rwarps_ >> w & 1 && reads_[w].epoch == warp_epoch[w];
        if (rwarps_ & ~(1u << w) || (mine && reads_[w].lanes & ~(1u << (tid & 31))))
          report("write not ordered after another thread's read");
      }
    }
    serial_ = block_serial;
    wtid_ = tid;
    wwarp_ = warp_epoch[w];
    wblock_ = block_epoch;
  }
  T v_;
  uint64_t serial_, wwarp_, wblock_;
  int wtid_;
  mutable uint64_t rblock_;
  mutable uint32_t rwarps_;  // warps with reads since the last block barrier
  mutable Reads reads_[32];
};
}  // namespace emu
template <class T>
inline T max(T a, const emu::Shared<T>& b) { return max(a, (T)b); }

#define threadIdx (emu::tidx())
#define blockDim (emu::bdim)
#define blockIdx (emu::bidx)
#define gridDim (emu::gdim)

// ---- warp and block collectives (full warps only) ---------------------------
inline void __syncwarp() { emu::wait_warp(true); }
inline void __syncthreads() { emu::wait_block(); }
inline unsigned __ballot_sync(unsigned, int p) {
  return emu::collective(p != 0, [](uint64_t* s, int) {
    unsigned b = 0;
    for (int i = 0; i < 32; ++i) b |= s[i] ? 1u << i : 0u;
    return b;
  });
}
inline int __any_sync(unsigned m, int p) { return __ballot_sync(m, p) != 0; }
template <class T, class L>
inline T emu_shuffle(T v, L from) {
  uint64_t u = 0;
  memcpy(&u, &v, sizeof(T));
  const uint64_t r = emu::collective(u, [&](uint64_t* s, int l) { return s[from(l)]; });
  memcpy(&v, &r, sizeof(T));
  return v;
}
template <class T>
inline T __shfl_sync(unsigned, T v, int src) { return emu_shuffle(v, [=](int) { return src & 31; }); }
template <class T>
inline T __shfl_up_sync(unsigned, T v, int d) { return emu_shuffle(v, [=](int l) { return l >= d ? l - d : l; }); }
template <class T>
inline T __shfl_xor_sync(unsigned, T v, int d) { return emu_shuffle(v, [=](int l) { return l ^ d; }); }
inline unsigned __match_any_sync(unsigned, int v) {
  return emu::collective((uint32_t)v, [](uint64_t* s, int l) {
    unsigned b = 0;
    for (int i = 0; i < 32; ++i) b |= s[i] == s[l] ? 1u << i : 0u;
    return b;
  });
}
template <class T, class F>
inline T emu_reduce(T v, F f) {
  return emu::collective((uint64_t)(int64_t)v, [&](uint64_t* s, int) {
    T r = (T)(int64_t)s[0];
    for (int i = 1; i < 32; ++i) r = f(r, (T)(int64_t)s[i]);
    return r;
  });
}
template <class T>
inline T __reduce_max_sync(unsigned, T v) { return emu_reduce(v, [](T a, T b) { return max(a, b); }); }
template <class T>
inline T __reduce_min_sync(unsigned, T v) { return emu_reduce(v, [](T a, T b) { return min(a, b); }); }
inline unsigned __reduce_add_sync(unsigned, unsigned v) {
  return emu_reduce(v, [](unsigned a, unsigned b) { return a + b; });
}

// ---- arithmetic and atomics ---------------------------------------------------
inline int __ffs(unsigned v) { return __builtin_ffs((int)v); }
inline int __clz(unsigned v) { return v ? __builtin_clz(v) : 32; }
inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((uint64_t)a * b) >> 32); }
inline float __uint2float_rn(unsigned v) { return (float)v; }
inline float __ull2float_rn(uint64_t v) { return (float)v; }
inline float __double2float_rn(double v) { return (float)v; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fdiv_rn(float a, float b) { return a / b; }
inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
inline float rsqrtf(float x) { return 1.0f / sqrtf(x); }
inline float __int_as_float(int v) { float f; memcpy(&f, &v, 4); return f; }
inline int __float_as_int(float v) { int i; memcpy(&i, &v, 4); return i; }
template <class T, class U>
inline T atomicAdd(T* p, U v) { const T o = *p; *p = o + (T)v; return o; }
template <class T, class U>
inline T atomicMin(T* p, U v) { const T o = *p; *p = min(o, (T)v); return o; }
template <class T, class U>
inline T atomicMax(T* p, U v) { const T o = *p; *p = max(o, (T)v); return o; }
template <class T, class U>
inline T atomicOr(T* p, U v) { const T o = *p; *p = o | (T)v; return o; }
namespace emu {
// An entry for a list whose entries are worked on side by side.
template <class T>
inline void append_once(T* list, int* count, T e) {
  for (int i = 0; i < *count; ++i)
    if (!memcmp(&list[i], &e, sizeof(T))) return report("second entry for the same work in a list");
  list[(*count)++] = e;
}
}  // namespace emu
inline void __nanosleep(unsigned) { emu::nap(); }

// ---- run time -------------------------------------------------------------------
typedef int cudaError_t;
typedef struct emuStream* cudaStream_t;
typedef struct emuEvent* cudaEvent_t;
typedef std::vector<std::function<void()>>*cudaGraph_t, *cudaGraphExec_t;
enum { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorMemoryAllocation = 2, cudaErrorNotReady = 600 };
enum cudaMemcpyKind { cudaMemcpyHostToDevice, cudaMemcpyDeviceToHost, cudaMemcpyDeviceToDevice };
enum { cudaStreamNonBlocking = 1, cudaEventDisableTiming = 2, cudaStreamCaptureModeThreadLocal = 1,
       cudaHostAllocDefault = 0 };
enum cudaDeviceAttr {
  cudaDevAttrMaxSharedMemoryPerBlockOptin,
  cudaDevAttrMultiProcessorCount,
  cudaDevAttrMaxSharedMemoryPerMultiprocessor,
  cudaDevAttrReservedSharedMemoryPerBlock,
  cudaDevAttrMaxRegistersPerMultiprocessor,
};
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize };
struct cudaFuncAttributes { size_t sharedSizeBytes; int numRegs; };
inline cudaError_t cudaGetDevice(int* d) { *d = 0; return 0; }
inline cudaError_t cudaSetDevice(int) { return 0; }
inline cudaError_t cudaGetDeviceCount(int* d) { *d = 1; return 0; }
inline cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  const char* sm_shared = getenv("EMU_SM_SHARED");  // a device with less of it: smaller tables in a batch
  *v = a == cudaDevAttrMaxSharedMemoryPerBlockOptin       ? 232448
       : a == cudaDevAttrMultiProcessorCount              ? 152
       : a == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? (sm_shared ? atoi(sm_shared) : 233472)
       : a == cudaDevAttrReservedSharedMemoryPerBlock     ? 1024
                                                          : 65536;
  return 0;
}
inline cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* f, const void*) { *f = {2560, 80}; return 0; }
inline cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return 0; }
template <class F>
inline cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, F, int threads, size_t) {
  *n = 65536 / 80 / threads;
  return 0;
}
inline cudaError_t cudaGetLastError() { return 0; }
template <class T>
inline cudaError_t cudaMalloc(T** p, size_t n) { *p = static_cast<T*>(emu::device_alloc(n)); return 0; }
inline cudaError_t cudaFree(void* p) { emu::device_free(p); return 0; }
inline cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = malloc(n); return 0; }
inline cudaError_t cudaFreeHost(void* p) { free(p); return 0; }
inline cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return 0; }
inline cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t = nullptr) {
  emu::enqueue([=] { memcpy(d, s, n); });
  return 0;
}
inline cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t = nullptr) {
  emu::enqueue([=] { memset(d, v, n); });
  return 0;
}
inline cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return 0; }
inline cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(8); return 0; }
inline cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return 0; }
inline cudaError_t cudaStreamSynchronize(cudaStream_t) { return 0; }
inline cudaError_t cudaDeviceSynchronize() { return 0; }
inline cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return 0; }
inline cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)malloc(8); return 0; }
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
inline cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return 0; }
inline cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t = nullptr) { return 0; }
inline cudaError_t cudaEventSynchronize(cudaEvent_t) { return 0; }
inline cudaError_t cudaEventQuery(cudaEvent_t) { return 0; }
inline cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1; return 0; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, int);
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g);
inline cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, int) {
  *e = new std::vector<std::function<void()>>(*g);
  return 0;
}
inline cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete g; return 0; }
inline cudaError_t cudaGraphExecDestroy(cudaGraphExec_t g) { delete g; return 0; }
inline cudaError_t cudaGraphLaunch(cudaGraphExec_t g, cudaStream_t) {
  for (auto& f : *g) f();
  return 0;
}
template <class T>
inline cudaError_t cudaGetSymbolAddress(void** p, T& s) { *p = (void*)&s; return 0; }

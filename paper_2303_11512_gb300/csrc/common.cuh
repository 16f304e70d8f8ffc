// Internal definitions shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <cstring>
#include <mutex>
#include <set>
#include <stdexcept>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/mgmlmc.h"

namespace mg {

// ---------------------------------------------------------------- errors
struct Error : public std::runtime_error {
  int code;
  Error(int c, const std::string& m) : std::runtime_error(m), code(c) {}
};

#define MG_CUDA(call)                                                              \
  do {                                                                             \
    cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess) {                                                       \
      throw ::mg::Error(e_ == cudaErrorMemoryAllocation ? MGMLMC_ERR_OOM            \
                                                          : MGMLMC_ERR_CUDA,       \
                        std::string(#call) + ": " + cudaGetErrorString(e_));       \
    }                                                                              \
  } while (0)

// Raise a kernel's dynamic shared-memory limit once per (kernel, device, size): the attribute belongs to the
// device's context, so a process that drives several GPUs needs it set on each.
inline void ensure_max_smem(const void* kernel, int bytes) {
  static std::mutex mu;
  static std::set<std::tuple<const void*, int, int>> done;
  int dev = 0;
  MG_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  if (done.count(std::make_tuple(kernel, dev, bytes))) return;
  MG_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  done.insert(std::make_tuple(kernel, dev, bytes));
}

#define MG_CHECK_ARG(cond, msg)                                                    \
  do {                                                                             \
    if (!(cond)) throw ::mg::Error(MGMLMC_ERR_INVALID_ARG, msg);                   \
  } while (0)

// launch bookkeeping: every kernel launch of the library goes through MG_LAUNCH
// (counted per context) or MG_LAUNCH_W, which also carries the launch's
// algorithmic bytes and flops for the optional per-kernel event timer.
extern thread_local int64_t* g_launch_counter;
// Per-kernel CUDA-event timer (enabled per context for kernels whose name
// contains a filter string); records are resolved when the report is read.
struct KTimer {
  bool on = false;
  std::string filter;
  struct Rec {
    const char* name;
    const char* where;  // launching function (its template arguments name the precision)
    double bytes, flops;
    cudaEvent_t a, b;
  };
  std::vector<Rec> recs;
  std::vector<cudaEvent_t> pool;
  cudaEvent_t get() {
    if (!pool.empty()) {
      cudaEvent_t e = pool.back();
      pool.pop_back();
      return e;
    }
    cudaEvent_t e;
    MG_CUDA(cudaEventCreate(&e));
    return e;
  }
  bool want(const char* name) const { return on && (filter.empty() || std::strstr(name, filter.c_str())); }
};
extern thread_local KTimer* g_timer;
// number of right-hand sides still iterating (host hint for byte accounting), -1 = all
extern thread_local int g_nact_hint;
inline double act_rhs(int nrhs) { return (g_nact_hint >= 0 && g_nact_hint < nrhs) ? g_nact_hint : nrhs; }

#define MG_LAUNCH_W(bytes, flops, kernel, grid, block, smem, stream, ...)          \
  do {                                                                             \
    ::mg::KTimer* t_ = ::mg::g_timer;                                              \
    if (t_ && t_->want(#kernel)) {                                                 \
      cudaEvent_t a_ = t_->get(), b_ = t_->get();                                  \
      MG_CUDA(cudaEventRecord(a_, (stream)));                                      \
      kernel<<<(grid), (block), (smem), (stream)>>>(__VA_ARGS__);                  \
      MG_CUDA(cudaGetLastError());                                                 \
      MG_CUDA(cudaEventRecord(b_, (stream)));                                      \
      t_->recs.push_back({#kernel, __PRETTY_FUNCTION__, (double)(bytes), (double)(flops), a_, b_}); \
    } else {                                                                       \
      kernel<<<(grid), (block), (smem), (stream)>>>(__VA_ARGS__);                  \
      MG_CUDA(cudaGetLastError());                                                 \
    }                                                                              \
    if (::mg::g_launch_counter) ++*::mg::g_launch_counter;                         \
  } while (0)
#define MG_LAUNCH(kernel, grid, block, smem, stream, ...) \
  MG_LAUNCH_W(0, 0, kernel, grid, block, smem, stream, __VA_ARGS__)

// 16 bytes from global to shared memory, in flight until their group is waited for
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
// one complex number
template <typename C>
__device__ __forceinline__ void cp_async_elem(C* dst, const C* src) {
  if constexpr (sizeof(C) == 16)
    cp_async16(dst, src);
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Programmatic dependent launch: a kernel that begins with pdl_begin() may be launched with MG_LAUNCH_P, and the GPU
// then places its blocks while the last blocks of the kernel before it still run.  pdl_begin() waits until that
// kernel has completed and its writes are visible, so nothing may be read or written before it (and what an earlier
// kernel wrote is not read through __restrict__ const pointers or __ldg, whose loads need not stay behind it); it
// also lets the next kernel be placed.  Used by the kernels of a V-cycle, where a launch below PDL_BYTES takes 5 to
// 12 us of which this hides about 2 (V(1,1) at L = 128 with 5 right-hand sides: 157 -> 129 us).  Larger launches lose
// by it (V(2,2) at L = 512 with 32: 1.82 -> 1.93 ms with every launch, 1.79 with those below 24 MB, 1.81 below 8 MB).
// A stream capture, the library's own or a caller's, gets plain launches: in a graph there is nothing left to hide, and
// some of these kernels follow a memset node, which a programmatic edge cannot start from.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
constexpr double PDL_BYTES = 24e6;
// FP64 kernels that keep their units busy for more than some 14 us are launched plainly: blocks placed beside the last
// ones of the kernel before come to lie unevenly on the SMs, and the fullest SM decides.
constexpr double PDL_FLOPS64 = 1.7e7;
template <typename R>
inline bool early_launch(double bytes, double flops) {
  return bytes < PDL_BYTES && (sizeof(R) == 4 || flops < PDL_FLOPS64);
}
// Launches of this call go into a graph: 1 yes, 0 no, -1 not looked up yet.  Looked up where it matters and at most once
// a call (200 ns), because the smallest calls take 5 us.
extern thread_local int g_capturing;
inline bool in_capture(cudaStream_t stream) {
  if (g_capturing < 0) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool known = cudaStreamIsCapturing(stream, &cap) == cudaSuccess;
    if (!known) cudaGetLastError();  // the legacy stream beside another capture
    g_capturing = !known || cap != cudaStreamCaptureStatusNone;
  }
  return g_capturing != 0;
}
template <typename... Par, typename... Arg>
inline void launch_pdl(bool early, void (*kernel)(Par...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                       Arg&&... arg) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &at;
  cfg.numAttrs = early ? 1 : 0;
  MG_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<Par>(arg)...));
}
#define MG_LAUNCH_PE(early, bytes, flops, kernel, grid, block, smem, stream, ...)  \
  do {                                                                             \
    ::mg::KTimer* t_ = ::mg::g_timer;                                              \
    cudaEvent_t a_ = nullptr, b_ = nullptr;                                        \
    if (t_ && t_->want(#kernel)) {                                                 \
      a_ = t_->get();                                                              \
      b_ = t_->get();                                                              \
      MG_CUDA(cudaEventRecord(a_, (stream)));                                      \
    }                                                                              \
    ::mg::launch_pdl((early) && !::mg::in_capture(stream), kernel, (grid), (block), (smem), (stream), __VA_ARGS__); \
    if (a_) {                                                                      \
      MG_CUDA(cudaEventRecord(b_, (stream)));                                      \
      t_->recs.push_back({#kernel, __PRETTY_FUNCTION__, (double)(bytes), (double)(flops), a_, b_}); \
    }                                                                              \
    if (::mg::g_launch_counter) ++*::mg::g_launch_counter;                         \
  } while (0)
#define MG_LAUNCH_P(bytes, flops, kernel, grid, block, smem, stream, ...) \
  MG_LAUNCH_PE((bytes) < ::mg::PDL_BYTES, bytes, flops, kernel, grid, block, smem, stream, __VA_ARGS__)

// ---------------------------------------------------------------- complex
template <typename R> struct CT;
template <> struct CT<float> { typedef float2 T; };
template <> struct CT<double> { typedef double2 T; };

__host__ __device__ __forceinline__ float2 cmake(float a, float b) { return make_float2(a, b); }
__host__ __device__ __forceinline__ double2 cmake(double a, double b) { return make_double2(a, b); }
template <typename C> __host__ __device__ __forceinline__ C czero() { C z; z.x = 0; z.y = 0; return z; }
template <typename C> __host__ __device__ __forceinline__ C cadd(C a, C b) { a.x += b.x; a.y += b.y; return a; }
template <typename C> __host__ __device__ __forceinline__ C csub(C a, C b) { a.x -= b.x; a.y -= b.y; return a; }
template <typename C> __host__ __device__ __forceinline__ C cneg(C a) { a.x = -a.x; a.y = -a.y; return a; }
template <typename C> __host__ __device__ __forceinline__ C cconj(C a) { a.y = -a.y; return a; }
template <typename C> __host__ __device__ __forceinline__ C cmul(C a, C b) {
  C r; r.x = a.x * b.x - a.y * b.y; r.y = a.x * b.y + a.y * b.x; return r;
}
// conj(a) * b
template <typename C> __host__ __device__ __forceinline__ C cmulc(C a, C b) {
  C r; r.x = a.x * b.x + a.y * b.y; r.y = a.x * b.y - a.y * b.x; return r;
}
// acc + a * b
template <typename C> __host__ __device__ __forceinline__ C cfma(C a, C b, C acc) {
  acc.x = fma(a.x, b.x, acc.x); acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y); acc.y = fma(a.y, b.x, acc.y);
  return acc;
}
// acc + conj(a) * b
template <typename C> __host__ __device__ __forceinline__ C cfmac(C a, C b, C acc) {
  acc.x = fma(a.x, b.x, acc.x); acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y); acc.y = fma(-a.y, b.x, acc.y);
  return acc;
}
template <typename C, typename R> __host__ __device__ __forceinline__ C cscale(C a, R s) { a.x *= s; a.y *= s; return a; }
// i * a and -i * a
template <typename C> __host__ __device__ __forceinline__ C cmuli(C a) { C r; r.x = -a.y; r.y = a.x; return r; }
template <typename C> __host__ __device__ __forceinline__ C cmulmi(C a) { C r; r.x = a.y; r.y = -a.x; return r; }

template <typename Cdst, typename Csrc> __host__ __device__ __forceinline__ Cdst cconv(Csrc a) {
  Cdst r; r.x = a.x; r.y = a.y; return r;
}

// ---------------------------------------------------------------- RNG
// SplitMix64 output finaliser (Steele, Lea & Flood 2014).
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z ^= z >> 30; z *= 0xBF58476D1CE4E5B9ull;
  z ^= z >> 27; z *= 0x94D049BB133111EBull;
  z ^= z >> 31; return z;
}
__host__ __device__ __forceinline__ uint64_t stream_key(uint64_t seed, int level, int phase, uint64_t sample) {
  uint64_t ctr = ((uint64_t)level << 56) | ((uint64_t)phase << 48) | sample;
  return mix64(seed ^ mix64(ctr));
}
__host__ __device__ __forceinline__ double rad_sign(uint64_t key, uint64_t i) {
  return (mix64(key + 0x9E3779B97F4A7C15ull * (i + 1)) >> 63) ? -1.0 : 1.0;
}

// ---------------------------------------------------------------- device memory
// RAII device buffer (stream-ordered allocation).
struct DBuf {
  void* p = nullptr;
  size_t bytes = 0;
  cudaStream_t st = 0;
  DBuf() {}
  DBuf(size_t b, cudaStream_t s) { alloc(b, s); }
  DBuf(const DBuf&) = delete;
  DBuf& operator=(const DBuf&) = delete;
  DBuf(DBuf&& o) noexcept { p = o.p; bytes = o.bytes; st = o.st; o.p = nullptr; o.bytes = 0; }
  DBuf& operator=(DBuf&& o) noexcept {
    if (this != &o) { release(); p = o.p; bytes = o.bytes; st = o.st; o.p = nullptr; o.bytes = 0; }
    return *this;
  }
  void alloc(size_t b, cudaStream_t s) {
    release();
    st = s;
    if (b) {
      const cudaError_t e = cudaMallocAsync(&p, b, s);
      if (e != cudaSuccess) p = nullptr;  // a buffer that is kept stays empty, and the next call asks again
      MG_CUDA(e);
    }
    bytes = b;
  }
  void ensure(size_t b, cudaStream_t s) { if (b > bytes) alloc(b, s); }
  void release() {
    if (p) cudaFreeAsync(p, st);
    p = nullptr;
    bytes = 0;
  }
  ~DBuf() { release(); }
  template <typename T> T* as() const { return reinterpret_cast<T*>(p); }
};

inline unsigned cdiv(long a, long b) { return (unsigned)((a + b - 1) / b); }
// SMs of the device of this thread's current call (a thread's variable that every call sets, because the smallest calls
// take 5 us); looked up outside of any
extern thread_local int g_sms;
inline int sm_count() {
  if (g_sms > 0) return g_sms;
  int dev = 0, n = 0;
  MG_CUDA(cudaGetDevice(&dev));
  MG_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
  return n;
}

}  // namespace mg

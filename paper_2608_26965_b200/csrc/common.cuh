// Shared host/device helpers of libclusterattn (sm_100a only).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/cluster_attention.h"

namespace ca {

// Status block at the start of every workspace: word 0 is the status code (CA_OK or the first
// error a kernel recorded), word kTileWord the counter that hands out tiles of the attention kernel;
// every call clears the first kStatusClearBytes on its stream, by a memset or in its first kernel (which saves
// 3 us: 4 heads of 512 rows in fp32 212 -> 208.5 us, 8 heads of 1,531 x 23,117 rows 328.5 -> 324).  The last word is a counter that calls
// only add to (query clusters recomputed by the second attention pass).
constexpr size_t kStatusBytes = 256;
constexpr size_t kStatusClearBytes = 252;
constexpr int kTileWord = 1;
constexpr int kRecomputedWord = 63;

extern std::atomic<unsigned long long> g_kernel_launches;   // kernels enqueued since the library was loaded

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

#define CA_RETURN_IF_CUDA(expr)                    \
  do {                                             \
    cudaError_t _e = (expr);                       \
    if (_e != cudaSuccess) return CA_ERR_CUDA;     \
  } while (0)

// Follows every kernel launch: counts it and turns a launch error into CA_ERR_CUDA.
#define CA_LAUNCH_CHECK()                                   \
  do {                                                      \
    ++::ca::g_kernel_launches;                              \
    if (cudaPeekAtLastError() != cudaSuccess) {             \
      (void)cudaGetLastError();                             \
      return CA_ERR_CUDA;                                   \
    }                                                       \
  } while (0)

// A stream and whether the launches on it overlap (launch_chained).
struct LaunchStream {
  cudaStream_t stream;
  bool chained;
  LaunchStream(cudaStream_t s, bool c = true) : stream(s), chained(c) {}
  operator cudaStream_t() const { return stream; }
};

// Launches that overlap: a kernel of a chain announces near its end (let_next_start) that the next one on
// the stream may be brought onto the SMs; that one waits at its very top (wait_for_previous) until the
// kernels before it have finished and their results are visible, before it reads or writes anything.  It hides
// the start of a launch, about 1.3 us of each of the sixteen in a row that a small call consists of (12 heads
// of 1,370 rows: 218 -> 196 us).  The announcement stands near the end, because a waiting CTA holds its shared
// memory and registers against kernels of other streams.  Every kernel that is launched this way
// waits, in every CTA, so that its completion implies that of the kernels before.
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Params, typename... Args>
inline void launch_chained(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, LaunchStream st,
                           const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = st.chained ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, kernel, Params(args)...);      // CA_LAUNCH_CHECK picks up an error
}

// Per-kernel-group device times (ca_profile / ca_profile_read of the public header).  A scope
// records a pair of CUDA events around the launches it encloses when profiling is on.
enum ProfGroup {
  kProfGram = 0, kProfFactor, kProfPca, kProfTransform, kProfSplitLevels, kProfSplitTail, kProfPermute,
  kProfSelect, kProfAttnPrep, kProfAttn, kProfAttnSecond, kProfGroups
};
bool prof_enabled();
void prof_mark(int group, cudaStream_t st, bool begin);
struct ProfScope {
  int group;
  cudaStream_t st;
  bool on;
  ProfScope(int g, cudaStream_t s) : group(g), st(s), on(prof_enabled()) { if (on) prof_mark(group, st, true); }
  ~ProfScope() { if (on) prof_mark(group, st, false); }
};

template <typename T>
__device__ __forceinline__ float to_f32(T x);
template <>
__device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename T>
__device__ __forceinline__ T from_f32(float x);
template <>
__device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// four consecutive elements as floats
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&u.x), b = *reinterpret_cast<const __nv_bfloat162*>(&u.y);
  const float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
  return make_float4(fa.x, fa.y, fb.x, fb.y);
}
__device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v) {
  uint2 u;
  *reinterpret_cast<__nv_bfloat162*>(&u.x) = __floats2bfloat162_rn(v.x, v.y);
  *reinterpret_cast<__nv_bfloat162*>(&u.y) = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = u;
}

// Carves aligned sub-buffers out of a workspace (host side).
struct Carver {
  char* base;
  size_t off;
  explicit Carver(void* p) : base(static_cast<char*>(p)), off(0) {}
  template <typename T>
  T* take(size_t n) {
    off = align_up(off, 256);
    T* r = reinterpret_cast<T*>(base + off);
    off += n * sizeof(T);
    return r;
  }
  size_t used() const { return align_up(off, 256); }
};

}  // namespace ca

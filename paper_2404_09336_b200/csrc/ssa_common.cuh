// Shared device/host helpers of libssa (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "ssa.h"

namespace ssa {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// Per-thread bookkeeping shared by the entry points (defined in ssa_api.cu).
void note_launches(int n);
void take_kernel_events(cudaEvent_t* begin, cudaEvent_t* end);
int sm_count();   // multiprocessors of the current device (cached; no synchronisation)
// Bytes from p to the end of the allocation it lies in, as far as that is device memory mapped as a whole; else 0.  Reading
// these is safe whatever offsets said that they are a list.  `known`: an allocation asked for before, which may hold p too.
struct Allocation { uintptr_t begin, end; };
size_t readable_bytes(const void* p, Allocation* known);
template <typename Entry>
inline int32_t readable_entries(const void* p, Allocation* known) {
  const size_t n = readable_bytes(p, known) / sizeof(Entry);
  return n < 0x7fffffff ? (int32_t)n : 0x7fffffff;
}

// Programmatic dependent launch.  Every kernel of the library is launched
// with the programmatic-serialization attribute: its blocks may become
// resident while the preceding kernel of the stream is still draining, and
// they call grid_dependency_wait(), which returns once that kernel has
// completed and its writes are visible, before they write anything or rely
// on anything they read (see load_early).
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Before that wait a block may only read, and what it reads may be about to change: an input that the kernel in front is
// still writing.  It is good for guesses alone: which cache rows to prefetch, or work that is checked against the
// inputs after the wait.  (relaxed.gpu: from L2, so that no stale line is left in L1.)
__device__ __forceinline__ int32_t load_early(const int32_t* p) {
  int32_t v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int2 load_early(const int2* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return make_int2((int32_t)(uint32_t)v, (int32_t)(v >> 32));
}
// The same after the wait, for what a guess is compared with: an ordinary load, but volatile, so that it stays behind the wait
// whatever the compiler makes of read-only memory.
__device__ __forceinline__ int32_t load_now(const int32_t* p) {
  int32_t v;
  asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ int2 load_now(const int2* p) {
  int2 v;
  asm volatile("ld.global.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
// The 32 bytes around p into L2.
__device__ __forceinline__ void prefetch_sector(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// A launch takes the host 1.9 us where a kernel's parameters are 17 to 32 bytes more than a multiple of 64, and 2.2..2.3 us where
// they are not (measured over 8..512 bytes, driver 580): kernels with other needs take some more bytes.  Another driver may have
// other sizes, and no kernel depends on them.
template <int kBytes> struct Spare { char unused[kBytes]; };

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_smem(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t dynamic_smem,
                                   cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = dynamic_smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
#ifdef SSA_NO_PDL
  cfg.numAttrs = 0;
#else
  cfg.numAttrs = 1;
#endif
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t stream, Args... args) {
  return launch_pdl_smem(kernel, grid, block, 0, stream, args...);
}

__device__ __forceinline__ float neg_inf() { return __int_as_float(0xff800000); }

// 16-byte read-only load that does not allocate in L1: every K/V row is used once.
__device__ __forceinline__ uint4 ld_stream_16B(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// A K/V cache stored as 8-bit e4m3 values (1 sign, 4 exponent, 3 mantissa bits; outside the paper).  Queries and
// outputs that go with such a cache are bf16.
struct Fp8E4M3 { uint8_t bits; };
template <typename T> struct Storage { using Query = T; };
template <> struct Storage<Fp8E4M3> { using Query = __nv_bfloat16; };
template <typename T> constexpr bool kIsFp8 = false;
template <> constexpr bool kIsFp8<Fp8E4M3> = true;

// Two e4m3 values (the low 16 bits of `pair`) -> two floats (exact: every e4m3 value is an fp16 value).
__device__ __forceinline__ float2 e4m3x2_to_float2(uint32_t pair) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((unsigned short)pair));
  return __half22float2(*reinterpret_cast<const __half2*>(&h2));
}

// Two packed 16-bit storage values -> two floats (exact).
template <typename T>
__device__ __forceinline__ float2 unpack2(uint32_t u);
template <>
__device__ __forceinline__ float2 unpack2<__nv_bfloat16>(uint32_t u) {
  return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}
template <>
__device__ __forceinline__ float2 unpack2<__half>(uint32_t u) {
  return __half22float2(*reinterpret_cast<const __half2*>(&u));
}

template <typename T>
__device__ __forceinline__ void unpack8(const uint4& r, float (&f)[8]) {
  float2 a = unpack2<T>(r.x), b = unpack2<T>(r.y), c = unpack2<T>(r.z), d = unpack2<T>(r.w);
  f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y;
  f[4] = c.x; f[5] = c.y; f[6] = d.x; f[7] = d.y;
}

template <typename T>
__device__ __forceinline__ T from_float(float x);
template <>
__device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }
template <>
__device__ __forceinline__ __half from_float<__half>(float x) { return __float2half_rn(x); }

__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ float to_float(__half x) { return __half2float(x); }

// Packed fp32 multiply-add on both halves: a * b + c.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(*reinterpret_cast<unsigned long long*>(&d))
      : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)),
        "l"(*reinterpret_cast<unsigned long long*>(&c)));
  return d;
}

// 2^x; 2^-inf = +0.
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The larger of two values, NaN if one of them is.
__device__ __forceinline__ float max_or_nan(float a, float b) {
  float y;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
  return y;
}

}  // namespace ssa

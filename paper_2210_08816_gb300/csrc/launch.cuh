// Launches with programmatic stream serialisation: a kernel may start (block scheduling, barrier and tensor-memory
// set-up, metrics) while its predecessor on the stream drains, and waits for the predecessor's results where it first
// needs them.  Chains of short kernels are what this is for: a 64^3 J.v + projection is nine launches of 4-9 us.
//
// A kernel launched this way calls pdl_begin() first and pdl_wait() before its first access to anything a predecessor
// writes or reads; every thread waits, so that a kernel never completes before its predecessor.  Read-only loads may
// be moved by the compiler across a memory barrier, so pdl_wait() returns a zero that the compiler cannot know, to be
// added to each pointer to such data: the addresses then depend on the wait.  (Passing the pointers themselves through
// an asm statement loses their address space and __restrict__: 32^3 FP64 products 71 -> 101 us.)  Data written once at
// grid creation (metrics, matrices) may be read before.
//
// What a predecessor wrote is read by ordinary loads: not by __ldg, nor through a kernel's `const __restrict__` pointer,
// which the compiler may turn into the same.  The read-only path is defined for data that nobody writes while the kernel is
// resident, and such a kernel is resident while its predecessor still writes.
#pragma once
#include <cuda_runtime.h>

namespace fv {

__device__ __forceinline__ void pdl_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ unsigned pdl_wait() {
  unsigned zero;
  asm volatile("griddepcontrol.wait;\n mov.u32 %0, 0;" : "=r"(zero)::"memory");
  return zero;
}

// An ordinary load that the compiler may move past stores, as it could __ldg (the kernel does not write what it reads; the
// address holds pdl_wait()'s zero).
__device__ __forceinline__ float load_global(const float* p) {
  float v;
  asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ double load_global(const double* p) {
  double v;
  asm("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ unsigned load_global(const unsigned* p) {
  unsigned v;
  asm("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ float2 load_global(const float2* p) {
  float2 v;
  asm("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ double2 load_global(const double2* p) {
  double2 v;
  asm("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ float4 load_global(const float4* p) {
  float4 v;
  asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(__cvta_generic_to_global(p)));
  return v;
}

template <typename T>
struct same_type {
  using type = T;
};

template <typename... P>
inline void launch(bool overlap, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                   typename same_type<P>::type... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = stream;
  c.attrs = &at;
  c.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, args...);
}
template <typename... P>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                   typename same_type<P>::type... args) {
  launch(true, kernel, grid, block, smem, stream, args...);
}
// With the overlap, in clusters of C blocks along x.
template <typename... P>
inline void launch_cluster(int C, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                           typename same_type<P>::type... args) {
  cudaLaunchAttribute at[2] = {};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)C;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = stream;
  c.attrs = at;
  c.numAttrs = 2;
  cudaLaunchKernelEx(&c, kernel, args...);
}
// Dynamic shared memory of a launch of `blocks` blocks, `most` of which (by registers and the `smem` they need) fit on a
// multiprocessor: padded so that no more of them fit there than an even spread puts there.  Blocks placed early, beside the
// predecessor's last ones, would pile up on the multiprocessors that are free first (see launch_spread): 33 products of
// 32^3 FP32, 132 stencil blocks, took 164 us and 128 so.  No more than that takes, since a launch waits for what it asks
// for (8^3, a block of eight: 41.4 us with all of an SM's memory for one block, 38.9 with half).  kSpreadSmem: what the
// kernel's limit has to allow.
constexpr size_t kSpreadSmem = 115 * 1024;
inline size_t spread_smem(size_t smem, long long blocks, int sms, int most) {
  const long long per = (blocks + sms - 1) / sms;
  if (per >= most) return smem;
  const size_t pad = (size_t)(228 * 1024 / (per + 1) + 1024);  // one block more does not fit
  return pad > smem ? pad : smem;
}
// Without the overlap, for kernels bound by the FP64 pipe (two operations per clock and SM): blocks placed while the
// predecessor still occupies most SMs pile up on the others, and the busiest SM sets the time (32^3 FP64 J.v +
// projection 101 us with the overlap, 71 without).  A kernel whose registers or shared memory let one block on an SM
// is spread evenly either way.
template <typename... P>
inline void launch_spread(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                          typename same_type<P>::type... args) {
  launch(false, kernel, grid, block, smem, stream, args...);
}

}  // namespace fv

// common.cuh -- shared device helpers of libbigint (sm_103a).
//
// Digits: every kernel works on 32-bit digits.  A little-endian array of
// 64-bit limbs is, byte for byte, a little-endian array of 32-bit digits
// (limb i = digit 2i + 2^32 * digit 2i+1), so device code may reinterpret a
// limb pointer as a digit pointer.
#pragma once

#include <atomic>
#include <cstdint>
#include <cuda_runtime.h>

#include "bigint.h"

namespace bigint {

constexpr unsigned FULL = 0xffffffffu;

// ---------------------------------------------------------------------------
// Carry resolution over 32 lanes with two ballots.
//
// Each lane holds a (generate, propagate) pair for its digits: g = the lane's
// digits produce a carry by themselves, p = they pass an incoming carry
// through (all result digits are at their maximum).  g and p are never both
// set.  With G and P the warp's ballots and X = G | P, the binary sum
// X + G + cin carries into bit i exactly when the digit-level carry reaches
// lane i: a generate lane has X_i = G_i = 1 (always carries out), a propagate
// lane has X_i = 1, G_i = 0 (carries out iff a carry comes in), any other
// lane has X_i = G_i = 0 (never carries out).  So the carry INTO every lane
// is bit i of (X + G + cin) ^ X ^ G, and the carry out of the warp is bit 32.
// This evaluates the exclusive scan with the operator of Fig. 3,
//   (g1,p1) o (g2,p2) = (g2 | (g1 & p2), p1 & p2),
// in a handful of integer instructions.
// ---------------------------------------------------------------------------
struct WarpCarry {
  uint32_t G, X;
};

__device__ __forceinline__ WarpCarry warp_gp(uint32_t g, uint32_t p) {
  WarpCarry w;
  w.G = __ballot_sync(FULL, g);
  w.X = w.G | __ballot_sync(FULL, p);
  return w;
}

// 64-bit word whose bit i (i < 32) is the carry into lane i and whose bit 32
// is the carry out of lane 31.
__device__ __forceinline__ uint64_t warp_carries(WarpCarry w, uint32_t cin) {
  const uint64_t s = (uint64_t)w.X + w.G + cin;
  return s ^ w.X ^ w.G;
}

// Carry out of the whole warp for a given carry in.
__device__ __forceinline__ uint32_t warp_carry_out(WarpCarry w, uint32_t cin) {
  return (uint32_t)(((uint64_t)w.X + w.G + cin) >> 32);
}

// (g, p) of a whole warp: generate = carry out with carry-in 0,
// propagate = every lane propagates.
__device__ __forceinline__ uint32_t warp_all_propagate(WarpCarry w) {
  return (w.X == FULL) && (w.G == 0);
}

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31; }

// Streaming global accesses (each limb is touched once).
__device__ __forceinline__ ulonglong2 ld_stream2(const uint64_t *p) {
  return __ldcs(reinterpret_cast<const ulonglong2 *>(p));
}
__device__ __forceinline__ void st_stream2(uint64_t *p, ulonglong2 v) {
  __stcs(reinterpret_cast<ulonglong2 *>(p), v);
}

// Programmatic dependent launch: pdl_trigger lets a dependent kernel (one
// launched by chain_launch right behind this one) be scheduled as SM resources
// allow, pdl_wait holds a kernel until the kernel before it has completed and
// its writes are visible.  A kernel calls pdl_wait before it touches global
// memory, and does not declare what it reads __restrict__: loads through such
// pointers are taken to be of memory that nothing writes while the kernel runs,
// which the kernel before it may do, and could move above the wait.  Both do
// nothing in kernels launched the ordinary way.
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace bigint

// Host-side helpers --------------------------------------------------------
// BIGINT_ECUDA for a CUDA call that failed; takes the error off the calling
// thread, whose later calls would report it as theirs.
static inline int bigint_cuda_error() {
  cudaGetLastError();
  return BIGINT_ECUDA;
}

#define BIGINT_CUDA_TRY(expr)                          \
  do {                                                 \
    cudaError_t e__ = (expr);                          \
    if (e__ != cudaSuccess) return bigint_cuda_error(); \
  } while (0)

namespace bigint {
// Counts the kernel launches the library enqueues (bigint_kernel_launches).
void count_launch();

// SMs of the current device (0: a CUDA error).
inline int sm_count() {
  static std::atomic<int> sms{0};
  int n = sms.load(std::memory_order_relaxed);
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 0;
    sms.store(n, std::memory_order_relaxed);
  }
  return n;
}

// Column sums of a chain of split-K products: two buffers of `bytes`, all
// zero at the start; a product takes buf[cur], and its finish clears what the
// product before left in the other (`used` bytes of each instance's `used`).
struct SkBuffers {
  void *buf[2] = {nullptr, nullptr};
  size_t bytes = 0;
  int cur = 0;
  size_t used = 0;  // bytes the last product dirtied in buf[cur ^ 1]
};

// Shapes the tensor-core product can be forced to (the autotuner's
// candidates; 0 = chosen by the cost model): 128-digit x blocks with the
// 64-, 128- or 256-column tile, or narrow x blocks of 64 or 32 digits.
constexpr int TC_FORCE_64 = 64, TC_FORCE_128 = 128, TC_FORCE_256 = 256;
constexpr int TC_FORCE_N64 = 1064, TC_FORCE_N32 = 1032;
}  // namespace bigint

// Called right after every kernel launch of the library: counts it and
// reports a launch error, which it takes off the thread.
static inline int bigint_launch_status() {
  bigint::count_launch();
  return cudaGetLastError() == cudaSuccess ? BIGINT_OK : BIGINT_ECUDA;
}

namespace bigint {
// Launches a kernel of a chain of dependent launches and counts it.  overlap:
// it may start its prologue (block setup, tensor-memory allocation) while the
// kernel before it in the stream finishes (see pdl_wait).  For launches that
// put at most one CTA on an SM: with several, those that start early crowd on
// the SMs that empty first and queue there for tensor memory (4096 divisions
// of 1024 by 512 limbs 810 -> 874 us), while a chain of small launches gains
// (one division of 16384 by 8192 limbs 470 -> 359 us).  CLUSTER: CTAs per
// thread-block cluster (grid a multiple of it).
template <int CLUSTER = 1, class... P, class... A>
inline int chain_launch(bool overlap, void (*kern)(P...), unsigned grid, unsigned threads,
                        size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at[2];
  c.attrs = at;
  if (CLUSTER > 1) {
    at[c.numAttrs].id = cudaLaunchAttributeClusterDimension;
    at[c.numAttrs].val.clusterDim.x = CLUSTER;
    at[c.numAttrs].val.clusterDim.y = at[c.numAttrs].val.clusterDim.z = 1;
    c.numAttrs++;
  }
  if (overlap) {
    at[c.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[c.numAttrs].val.programmaticStreamSerializationAllowed = 1;
    c.numAttrs++;
  }
  if (cudaLaunchKernelEx(&c, kern, static_cast<P>(args)...) != cudaSuccess)
    return bigint_cuda_error();
  return bigint_launch_status();
}
}  // namespace bigint

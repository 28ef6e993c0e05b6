// Shared device helpers for the JAB kernels (sm_103a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/jab.h"

namespace jab {

using half_t = __half;
using bf16_t = __nv_bfloat16;

// Records the first device-side problem in the per-device status word (0 = OK).
__device__ __forceinline__ void report(int* status, int code) {
  if (status != nullptr) atomicCAS(status, 0, code);
}

// Checked build (nvcc -DJAB_CHECKED=1, libjab_checked.so): the kernels test the last index of each
// computed global access against its buffer's extent before making it; a failed test reports
// JAB_ERR_DEVICE_ASSERT and the caller skips the access (no trap, no fault). Compiled out otherwise.
#ifndef JAB_CHECKED
#define JAB_CHECKED 0
#endif
__device__ __forceinline__ bool in_bounds(int64_t last, int64_t extent, int* status) {
#if JAB_CHECKED
  if (last < 0 || last >= extent) {
    report(status, JAB_ERR_DEVICE_ASSERT);
    return false;
  }
#else
  (void)last;
  (void)extent;
  (void)status;
#endif
  return true;
}

__host__ __device__ __forceinline__ int qmax_of(int bits) { return (1 << (bits - 1)) - 1; }

// Eq. 2 with reading R1: v = fl32(w / s) (IEEE round-to-nearest division), q = clip(rint(v)).
__device__ __forceinline__ float quant_code(float w, float s, int qmax, float* v_out) {
  const float v = __fdiv_rn(w, s);
  float q = rintf(v);  // round half to even
  q = fminf(fmaxf(q, -(float)qmax), (float)qmax);
  if (v_out) *v_out = v;
  return q;
}

// Eq. 13: d w_hat / d s = q - v if |v| <= qmax, else sign(v) * qmax.
__device__ __forceinline__ float lsq_factor(float w, float s, int qmax) {
  float v;
  const float q = quant_code(w, s, qmax, &v);
  return (fabsf(v) <= (float)qmax) ? (q - v) : copysignf((float)qmax, v);
}

// fl32(w / s) of several bf16 weights with one scale: with r = fl32(1 / s) and v0 = fl32(w r), the
// remainder w - v0 s is exact in one fused operation and v0 + r (w - v0 s) rounds to the IEEE quotient
// (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990).
// Equal to w / s for every pair of a bf16 and an fp32 mantissa (2^7 x 2^23, one by one in
// tests/test_quotient_cpu.py), and so wherever no intermediate leaves the normal range: s within 2^-60 .. 2^60, |w| within 2^-90 ..
// 2^60 or 0 (below 2^-90 the quotient is less than 2^-30 and its code 0 either way). Other values take
// the division. Three operations a weight, in packed pairs, where the division takes about ten.
__device__ __forceinline__ bool quot_window(float s) { return s >= 8.6736174e-19f && s <= 1.1529215e18f; }
// Largest magnitude bits of packed 16-bit floats seen so far, per half: one AND and one 16x2 maximum.
__device__ __forceinline__ uint32_t max_abs_f16x2(uint32_t acc, uint32_t v2) {
  return __vmaxu2(acc, v2 & 0x7fff7fffu);
}
// Whether either half of such a maximum is at or above `limit`.
__device__ __forceinline__ bool either_at_least(uint32_t m2, uint32_t limit) {
  return (m2 & 0xffffu) >= limit || (m2 >> 16) >= limit;
}
constexpr uint32_t kBf16Inf = 0x7f80u, kHalfInf = 0x7c00u;
constexpr uint32_t kBf16TwoTo60 = 187u << 7, kBf16TwoToM60 = 67u << 7;

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// a + b = s + e exactly (Knuth).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// Adds the unevaluated pair (h, l) to (hi, lo): about 2^-46 of the sum is lost.
__device__ __forceinline__ void pair_add(float& hi, float& lo, float h, float l) {
  float s, e;
  two_sum(hi, h, s, e);
  hi = s;
  lo = __fadd_rn(__fadd_rn(lo, l), e);
}

// Value of a sum kept as a pair (the low part of an infinite one is NaN).
__device__ __forceinline__ double pair_value(float hi, float lo) {
  return fabsf(hi) < INFINITY ? (double)hi + (double)lo : (double)hi;
}

// Sum of a warp's pairs (hi, lo), in every lane. (The chip runs two FP64 operations a clock and SM: an fp64
// warp_sum holds a role that others wait for ten times as long.)
__device__ __forceinline__ void warp_pair_sum(float& hi, float& lo) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h = __shfl_xor_sync(0xffffffffu, hi, o), l = __shfl_xor_sync(0xffffffffu, lo, o);
    pair_add(hi, lo, h, l);
  }
}

// Block-wide sum in a fixed order (deterministic); every thread gets the result.
template <int NT>
__device__ __forceinline__ double block_sum(double x, double* smem /* >= NT/32 */) {
  x = warp_sum(x);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) smem[w] = x;
  __syncthreads();
  double t = 0.0;
#pragma unroll
  for (int i = 0; i < NT / 32; ++i) t += smem[i];
  return t;
}

// Division of 0 <= n < 2^30 by a constant of the launch, 1 <= d < 2^30: one wide multiplication by
// floor(2^k / d) + 1, k = 30 + ceil(log2 d), exact as n (that d - 2^k) < 2^k. A tile's indices take
// four or five quotients, each some 200 clocks of dependent instructions as plain integer divisions, at a
// point where every role of a persistent kernel waits for them.
struct FastDiv {
  uint64_t m;
  int d, k;
  FastDiv() = default;
  explicit FastDiv(int div) : d(div) {
    k = 30;
    while ((1ll << (k - 30)) < div) ++k;
    m = ((uint64_t)1 << k) / (uint64_t)div + 1;
  }
  __device__ __forceinline__ int quot(int n) const { return (int)(((uint64_t)(uint32_t)n * m) >> k); }
  __device__ __forceinline__ void divmod(int n, int& q, int& r) const {
    q = quot(n);
    r = n - q * d;
  }
};

// Programmatic dependent launch: a kernel started by launch_after may begin while its predecessor on the
// stream still runs, sets up what needs no memory of the predecessor's (barriers, tensor memory, descriptors)
// and then calls stream_order() in every thread. From there on the predecessor is complete, its writes are
// visible, and whatever it read may be overwritten; only then is the successor let in, so that at most one
// kernel waits behind the running one and, with all of a grid's tensor memory allocated before, none can take
// what a block still to be set up needs. The seven kernels of a small fitting step (GPT-2 block, 4 x 128 tokens)
// take 40.9 us this way; one after the other, each with its launch and its set-up in the open, 56.5 us.
__device__ __forceinline__ void stream_order() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... P, class... A>
cudaError_t launch_after(void (*kern)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st,
                         const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
  if (e != cudaSuccess) cudaGetLastError();  // reported here, not again by a later query
  return e;
}

// Static schedule of a persistent kernel: the tile a CTA takes in round i when `ntiles` tiles,
// ordered from the most work to the least, are dealt to `grid` CTAs. Rounds alternate direction
// (CTA x takes position x, then grid - 1 - x, ...), so every CTA gets a similar total; the tile
// index grows with i, so a CTA is done at its first index >= ntiles.
__device__ __forceinline__ int sched_tile(int i, int grid, int cta) {
  return i * grid + ((i & 1) ? grid - 1 - cta : cta);
}

}  // namespace jab

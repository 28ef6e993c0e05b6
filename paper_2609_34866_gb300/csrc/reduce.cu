// Loss reduction (Eq. 3, MSE term): per-tile fp64 partials -> SSE per (candidate, sequence, head)
// and L = SSE / (B T Hq d_h). Fixed summation order, so repeated calls give identical bits.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "workspace.h"

namespace jab {

// One warp, `blk` of `nblk`: sum of its share of the rows ((sequence, head) pairs, nP partials each; a lane
// per row, the partials in order). A warp and no more per SM: fp64 additions go at about two a clock there,
// 16 clocks an instruction of a warp.
__device__ __forceinline__ double loss_slice(const double* __restrict__ part, int nbh, int nP, int blk,
                                             int nblk, double* __restrict__ parts_out) {
  double acc = 0.0;
  for (int i = blk * 32 + (threadIdx.x & 31); i < nbh; i += nblk * 32) {
    const double* p = part + (int64_t)i * nP;
    double s = 0.0;
#pragma unroll 8
    for (int k = 0; k < nP; ++k) s += p[k];
    if (parts_out) parts_out[i] = s;
    acc += s;
  }
  return warp_sum(acc);
}

// Counts a warp's partial, published by its lane 0 (of `total`); true, in all its lanes, in the one that comes
// last, with every partial visible: lane 0's fences order its count against the partials, and __syncwarp the
// other lanes' reads behind it (a shuffle orders no memory). The counter (0 before the launch) is left at 0.
__device__ __forceinline__ bool last_warp(int* counter, int total) {
  int last = 0;
  if ((threadIdx.x & 31) == 0) {
    __threadfence();
    last = atomicAdd(counter, 1) == total - 1;
    if (last) {
      *counter = 0;
      __threadfence();
    }
  }
  __syncwarp();
  return __shfl_sync(0xffffffffu, last, 0) != 0;
}

// Sum of n published partials by one warp, lane-strided and then a fixed tree.
__device__ __forceinline__ double sum_published(const double* part, int n) {
  double acc = 0.0;
  for (int k = threadIdx.x & 31; k < n; k += 32) acc += __ldcg(part + k);
  return warp_sum(acc);
}

// nblk one-warp blocks per candidate, the last block of the grid adds their sums (one block per candidate
// took 88 us for 4096 x 32 partials, 24 us for 5 x 1024 x 32; now 11 us).
__global__ void __launch_bounds__(32) loss_reduce_kernel(const double* __restrict__ part, int C, int nbh,
                                                         int nP, int nblk, double inv_n,
                                                         double* __restrict__ out,
                                                         double* __restrict__ parts_out,
                                                         double* __restrict__ red, int* counter,
                                                         int* status) {
  stream_order();
  const int c = blockIdx.x / nblk, blk = blockIdx.x - c * nblk;
  const double t = loss_slice(part + (int64_t)c * nbh * nP, nbh, nP, blk, nblk,
                              parts_out ? parts_out + (int64_t)c * nbh : nullptr);
  if (threadIdx.x == 0) red[c * kRedBlocks + blk] = t;
  if (!last_warp(counter, gridDim.x)) return;
  for (int k = 0; k < C; ++k) {
    const double tot = sum_published(red + k * kRedBlocks, nblk);
    if (threadIdx.x == 0) {
      out[k] = tot * inv_n;
      if (!isfinite(tot)) report(status, JAB_ERR_NONFINITE);
    }
  }
}

__global__ void loss_combine_kernel(const double* __restrict__ a, const double* __restrict__ b,
                                    double lam, int C, double* __restrict__ out) {
  stream_order();
  for (int c = threadIdx.x; c < C; c += blockDim.x) out[c] = a[c] + lam * b[c];
}

// Omega of Eq. 6, one block per candidate: c1[c] = Tr(H) * sum of the candidate's quantisation-error
// partials (strided per thread, then a fixed tree; one thread adding 1024 of them took 48 us),
// c2[c] = layers_after * c1[c].
__global__ void __launch_bounds__(256) omega_finish_kernel(const double* __restrict__ part,
                                                           int nblocks,
                                                           const double* __restrict__ trace,
                                                           double layers_after,
                                                           double* __restrict__ c1,
                                                           double* __restrict__ c2) {
  __shared__ double red[8];
  const int c = blockIdx.x;
  double e = 0.0;
  for (int k = threadIdx.x; k < nblocks; k += 256) e += part[(int64_t)c * nblocks + k];
  const double tot = block_sum<256>(e, red);
  if (threadIdx.x == 0) {
    const double v = *trace * tot;
    c1[c] = v;
    if (c2) c2[c] = layers_after * v;
  }
}

__global__ void check_finite_kernel(const float* __restrict__ x, int64_t n, int* status) {
  bool bad = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    bad |= !isfinite(x[i]);
  if (__syncthreads_or(bad) && threadIdx.x == 0) report(status, JAB_ERR_NONFINITE);
}

// Sum of squares: block b sums its contiguous chunk (fixed per-thread order, fixed tree), one block then
// adds the kRedBlocks partials. The chip runs about two FP64 operations per clock and SM, and a
// conversion and a multiply-add per value bounded the kernel (101 us for 25M values, now 27; 43 with eight
// values at a time): up to sixteen squares are added in floats with every rounding error carried along, and only
// that goes to the fp64 accumulator. (Eight blocks to an SM: all kRedBlocks are resident at once.)
// The products' low parts are a pair of their own: their last bits do not round evenly (an odd
// square is 1 modulo 8), and with all errors in one float the sum came out 1.1e-15 small. Values whose
// largest is outside 2^-40 .. 2^60 are squared in fp64. With `status` a non-finite value is reported.
template <int N>
__device__ __forceinline__ double sum_squares(const float (&v)[N]) {
  float big = 0.f;
#pragma unroll
  for (int k = 0; k < N; ++k) big = fmaxf(big, fabsf(v[k]));
  if (!(big >= 9.0949470e-13f && big <= 1.1529215e18f)) {
    double acc = 0.0;
    for (int k = 0; k < N; ++k) acc += (double)v[k] * (double)v[k];
    return acc;
  }
  float sh = 0.f, se = 0.f, sl = 0.f, s3 = 0.f;  // products and their sums' errors, low parts and theirs
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const float h = __fmul_rn(v[k], v[k]), l = __fmaf_rn(v[k], v[k], -h);
    float t, e;
    two_sum(sh, h, t, e);
    sh = t;
    se = __fadd_rn(se, e);
    two_sum(sl, l, t, e);
    sl = t;
    s3 = __fadd_rn(s3, e);
  }
  float a, b;
  two_sum(se, sl, a, b);
  return (double)sh + ((double)a + (double)__fadd_rn(b, s3));
}

__global__ void __launch_bounds__(256, 8) sumsq_partial_kernel(const float* __restrict__ x, int64_t n,
                                                            double* __restrict__ part, int* status) {
  __shared__ double red[8];
  const int64_t n8 = n / 8;  // n is a multiple of 64 (rows of a weight)
  const int64_t chunk = (n8 + gridDim.x - 1) / gridDim.x;
  const int64_t lo = blockIdx.x * chunk, hi = lo + chunk < n8 ? lo + chunk : n8;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  double acc = 0.0;
  int64_t i = lo + threadIdx.x;
  for (; i + blockDim.x < hi; i += 2 * blockDim.x) {
    const float4 a = x4[2 * i], b = x4[2 * i + 1];
    const float4 c = x4[2 * (i + blockDim.x)], d = x4[2 * (i + blockDim.x) + 1];
    const float v[16] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w, d.x, d.y, d.z, d.w};
    acc += sum_squares(v);
  }
  if (i < hi) {
    const float4 a = x4[2 * i], b = x4[2 * i + 1];
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    acc += sum_squares(v);
  }
  const double t = block_sum<256>(acc, red);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = t;
    if (status != nullptr && !isfinite(t)) report(status, JAB_ERR_NONFINITE);
  }
}

// One block: thread t adds its contiguous chunk in order, then a fixed tree (block_sum), so the
// result is the same on every call.
__global__ void __launch_bounds__(256) sum_scaled_kernel(const double* __restrict__ part, int n,
                                                         double scale, double* __restrict__ out) {
  __shared__ double red[8];
  const int chunk = (n + blockDim.x - 1) / blockDim.x;
  const int lo = threadIdx.x * chunk, hi = min(lo + chunk, n);
  double t = 0.0;
  for (int i = lo; i < hi; ++i) t += part[i];
  const double tot = block_sum<256>(t, red);
  if (threadIdx.x == 0) *out = scale * tot;
}

// Natural-log log-sum-exp rows [BH, T] to log2 units with the row pitch of the backward workspace.
__global__ void lse_to_log2_kernel(const float* __restrict__ in, int BH, int T, int pitch,
                                   float* __restrict__ out) {
  stream_order();
  const int64_t n = (int64_t)BH * T;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / T, t = i - r * T;
    out[r * pitch + t] = in[i] * 1.4426950408889634f;
  }
}

// The end of a scale-gradient call in one launch: every gradient element as the sum of its K-split partials
// in the order of the splits (a non-finite sum is reported), and in the first blocks' first warps the loss from its partials
// and, with KL partials, the KL value and loss + lambda KL. (Three to five launches before; 4 x 128 fit 68.7 ->
// 64 us a call.)
__global__ void __launch_bounds__(256) finish_kernel(const __grid_constant__ FinishArgs p) {
  stream_order();
  bool bad = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < p.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double t = 0.0;
    for (int s = 0; s < p.splits; ++s) t += p.gpart[(int64_t)s * p.n + i];
    const float v = (float)t;
    p.grad[i] = v;
    bad |= !isfinite(v);
  }
  if (bad) report(p.status, JAB_ERR_NONFINITE);
  if ((int)blockIdx.x >= p.nblk || threadIdx.x >= 32) return;
  const double l = loss_slice(p.part, p.nbh, p.nP, blockIdx.x, p.nblk, nullptr);
  double kl = 0.0;
  if (p.klpart != nullptr) {
    for (int i = blockIdx.x * 32 + threadIdx.x; i < p.nkl; i += p.nblk * 32) kl += p.klpart[i];
    kl = warp_sum(kl);
  }
  if (threadIdx.x == 0) {
    p.red[blockIdx.x] = l;
    p.red[kRedBlocks / 2 + blockIdx.x] = kl;
  }
  if (!last_warp(p.counter, p.nblk)) return;
  const double tot = sum_published(p.red, p.nblk);
  const double ktot = p.klpart != nullptr ? sum_published(p.red + kRedBlocks / 2, p.nblk) : 0.0;
  if (threadIdx.x == 0) {
    if (!isfinite(tot)) report(p.status, JAB_ERR_NONFINITE);
    const double klv = ktot * p.kl_scale;
    *p.loss = p.klpart != nullptr ? tot * p.inv_n + p.lambda * klv : tot * p.inv_n;
    if (p.kl_out) *p.kl_out = klv;
  }
}

// Blocks that a sum over nbh rows is worth (at most half of the kRedBlocks slots).
static int loss_blocks(int nbh) { return std::min(kRedBlocks / 2, std::max(1, (nbh + 31) / 32)); }

cudaError_t launch_loss_reduce(const double* part, int C, int B, int Hq, int nP, double inv_n,
                               double* out, double* parts_out, double* red, int* counter, int* status,
                               cudaStream_t st) {
  const int nbh = B * Hq, nblk = loss_blocks(nbh);
  return launch_after(loss_reduce_kernel, (unsigned)(C * nblk), 32, 0, st, part, C, nbh, nP, nblk, inv_n, out, parts_out,
                      red, counter, status);
}

cudaError_t launch_finish(FinishArgs a, cudaStream_t st) {
  a.nblk = loss_blocks(std::max(a.nbh, a.klpart != nullptr ? a.nkl : 0));
  const int64_t blocks = std::min<int64_t>(4096, std::max<int64_t>((a.n + 255) / 256, a.nblk));
  return launch_after(finish_kernel, (unsigned)blocks, 256, 0, st, a);
}

cudaError_t launch_loss_combine(const double* a, const double* b, double lam, int C, double* out,
                                cudaStream_t st) {
  return launch_after(loss_combine_kernel, 1, 128, 0, st, a, b, lam, C, out);
}

cudaError_t launch_omega_finish(const double* part, int nblocks, int C, const double* trace,
                                double layers_after, double* c1, double* c2, cudaStream_t st) {
  omega_finish_kernel<<<C, 256, 0, st>>>(part, nblocks, trace, layers_after, c1, c2);
  return cudaGetLastError();
}

cudaError_t launch_sumsq(const float* x, int64_t n, double* part, double* out, int* status,
                         cudaStream_t st) {
  sumsq_partial_kernel<<<kRedBlocks, 256, 0, st>>>(x, n, part, status);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_sum_scaled(part, kRedBlocks, 1.0, out, st);
}

cudaError_t launch_sum_scaled(const double* part, int n, double scale, double* out, cudaStream_t st) {
  sum_scaled_kernel<<<1, 256, 0, st>>>(part, n, scale, out);
  return cudaGetLastError();
}

cudaError_t launch_lse_to_log2(const float* in, int BH, int T, int pitch, float* out,
                               cudaStream_t st) {
  int64_t blocks = ((int64_t)BH * T + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  return launch_after(lse_to_log2_kernel, (unsigned)blocks, 256, 0, st, in, BH, T, pitch, out);
}

cudaError_t launch_check_finite(const float* x, int64_t n, int* status, cudaStream_t st) {
  int64_t blocks = (n + 255) / 256;
  if (blocks > 1024) blocks = 1024;
  check_finite_kernel<<<(unsigned)blocks, 256, 0, st>>>(x, n, status);
  return cudaGetLastError();
}

}  // namespace jab

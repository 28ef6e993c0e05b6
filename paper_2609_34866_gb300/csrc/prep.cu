// Elementwise and small kernels of the L_JAB path: X conversion, the quantiser (Eq. 2), scale
// initialisation, the RoPE table. All are HBM-bound: 16-byte vector loads and stores, grids sized
// in multiples of the SM count.
#include "common.cuh"
#include "kernels.h"
#include "tc.cuh"

namespace jab {

// ---------------------------------------------------------------- X: bf16 -> fp16 (+ range check)
__global__ void convert_x_kernel(const uint4* __restrict__ x, uint4* __restrict__ xh, int64_t n8,
                                 int* status) {
  int bad = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n8;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint4 v = __ldg(x + i);
    const bf16_t* b = reinterpret_cast<const bf16_t*>(&v);
    uint4 o;
    half_t* h = reinterpret_cast<half_t*>(&o);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float f = __bfloat162float(b[k]);
      h[k] = __float2half_rn(f);
      if (!isfinite(f)) bad |= 2;
      else if (__hisinf(h[k])) bad |= 1;
    }
    xh[i] = o;
  }
  if (bad & 2) report(status, JAB_ERR_NONFINITE);
  else if (bad & 1) report(status, JAB_ERR_RANGE);
}

// ---------------------------------------------------------------- quantiser (Section 2.1, Eq. 2)
// bits == 0: plain bf16 -> fp16 conversion of W (the teacher's weights).
__global__ void quantize_kernel(const uint4* __restrict__ w, const float* __restrict__ s, int D,
                                int d, int G, int bits, uint4* __restrict__ w16,
                                int8_t* __restrict__ codes, float* __restrict__ w_hat32,
                                int* status) {
  const int64_t n8 = (int64_t)D * d / 8;
  const int qmax = bits > 0 ? qmax_of(bits) : 0;
  const int ng = d / G;
  int bad = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n8;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint4 v = __ldg(w + i);
    const bf16_t* b = reinterpret_cast<const bf16_t*>(&v);
    const int64_t e0 = i * 8;
    const int64_t row = e0 / d;
    const int col = (int)(e0 - row * d);
    float out[8];
    if (bits == 0) {
#pragma unroll
      for (int k = 0; k < 8; ++k) out[k] = __bfloat162float(b[k]);
    } else {
      float sc = __ldg(s + row * ng + col / G);
      if (!(sc > 0.f) || !isfinite(sc)) {  // reading: scales must be finite and > 0
        bad = 1;
        sc = 1.f;
      }
      char cq[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float q = quant_code(__bfloat162float(b[k]), sc, qmax, nullptr);
        cq[k] = (char)(int)q;
        out[k] = __fmul_rn(q, sc);
      }
      if (codes) *reinterpret_cast<uint2*>(codes + e0) = *reinterpret_cast<uint2*>(cq);
      if (w_hat32) {
        reinterpret_cast<float4*>(w_hat32 + e0)[0] = make_float4(out[0], out[1], out[2], out[3]);
        reinterpret_cast<float4*>(w_hat32 + e0)[1] = make_float4(out[4], out[5], out[6], out[7]);
      }
    }
    if (w16) {
      uint4 o;
      half_t* h = reinterpret_cast<half_t*>(&o);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        h[k] = __float2half_rn(out[k]);
        if (__hisinf(h[k]) || __hisnan(h[k])) bad |= 2;  // not representable as an fp16 operand
      }
      w16[i] = o;
    }
  }
  if (bad & 1) report(status, JAB_ERR_NONFINITE);
  else if (bad & 2) report(status, JAB_ERR_RANGE);
}

// ---------------------------------------------------------------- Rademacher probes (Section 2.4)
// SplitMix64 (Steele, Lea and Flood, "Fast splittable pseudorandom number generators", 2014) used as
// a counter-based generator: entry n of the probe sequence (n = probe * D * d + flat index) takes
// the (n + 1)-th output of the stream seeded with `seed`; its top bit selects -1, else +1.
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t n) {
  uint64_t z = seed + (n + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Entries are written as +-2^-k (fp16: exponent field 15 - k, zero mantissa), an exact scaling.
__global__ void rademacher_probe_kernel(uint64_t seed, uint64_t first, int64_t n8, int k2,
                                        uint4* __restrict__ out) {
  const uint16_t pos = (uint16_t)((15 - k2) << 10), neg = (uint16_t)(0x8000u | pos);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n8;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint4 o;
    uint16_t* h = reinterpret_cast<uint16_t*>(&o);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      h[k] = (splitmix64_at(seed, first + (uint64_t)(i * 8 + k)) >> 63) ? neg : pos;
    out[i] = o;
  }
}

// ---------------------------------------------------------------- quantisation error (Eq. 6)
// Partial sums of (Q_b(w) - w)^2 over a grid-stride range, one per block, reduced in fixed order by
// omega_finish_kernel. Each term is the oracle's (q s - w in double, squared), but the chip runs only
// about two FP64 operations per clock and SM, and five of them per weight bounded the kernel (199 us
// for 6144 x 4096). So a term is formed as an unevaluated pair of floats: q s - w exactly (product and
// difference with their rounding errors), its square to about 2^-46 of itself, eight of them added
// with the errors carried along, and only that sum goes to the fp64 accumulator: 52 us. Weights and
// scale are first multiplied by the power of two that brings the scale to [1, 2) (exact), so that no
// square under- or overflows; a chunk whose values leave that window takes the fp64 form.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Sum of (q s - w)^2 over the 8 weights of a chunk.
__device__ __forceinline__ double qerr_chunk(const bf16_t* b, float sc, int qmax) {
  const int ex = (__float_as_int(sc) >> 23) & 0xff;  // exponent field of the scale
  const float up = __int_as_float((254 - ex) << 23);  // 2^(127 - ex): the scale times this is in [1, 2)
  const float ss = sc * up;
  bool fast = ex > 27 && ex < 227;
#pragma unroll
  for (int k = 0; k < 8; ++k) fast &= fabsf(__bfloat162float(b[k]) * up) < 1.09951163e12f;  // 2^40
  if (!fast) {
    double acc = 0.0;
    for (int k = 0; k < 8; ++k) {
      const float wv = __bfloat162float(b[k]);
      const double e = (double)quant_code(wv, sc, qmax, nullptr) * (double)sc - (double)wv;
      acc += e * e;
    }
    return acc;
  }
  float sh = 0.f, sl = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float wv = __bfloat162float(b[k]);
    const float q = quant_code(wv, sc, qmax, nullptr);
    const float ph = __fmul_rn(q, ss), pl = __fmaf_rn(q, ss, -ph);  // q s = ph + pl
    float dh, dl;
    two_sum(ph, -(wv * up), dh, dl);
    const float lo = __fadd_rn(dl, pl);
    const float eh = __fadd_rn(dh, lo), el = __fsub_rn(lo, __fsub_rn(eh, dh));  // q s - w = eh + el
    const float h = __fmul_rn(eh, eh);
    const float l = __fmaf_rn(2.f * eh, el, __fmaf_rn(eh, eh, -h));
    float t, err;
    two_sum(sh, h, t, err);
    sh = t;
    sl = __fadd_rn(sl, __fadd_rn(err, l));
  }
  const double down = __hiloint2double((2 * (ex - 127) + 1023) << 20, 0);  // 2^(2 (ex - 127))
  return ((double)sh + (double)sl) * down;
}

__global__ void __launch_bounds__(256) qerr_partial_kernel(const uint4* __restrict__ w,
                                                           const float* __restrict__ s, int D,
                                                           int d, int G, int bits,
                                                           double* __restrict__ part, int* status) {
  __shared__ double red[8];
  const int64_t n8 = (int64_t)D * d / 8;
  const int qmax = qmax_of(bits);
  const int ng = d / G, d8 = d / 8, g8 = G / 8;
  double acc = 0.0;
  int bad = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n8;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint4 v = __ldg(w + i);
    int64_t row;
    int c8;
    if (n8 <= INT32_MAX) {  // (a 64-bit division costs more than the rest of the addressing)
      row = (int)i / d8;
      c8 = (int)i - (int)row * d8;
    } else {
      row = i / d8;
      c8 = (int)(i - row * d8);
    }
    float sc = __ldg(s + row * ng + c8 / g8);
    if (!(sc > 0.f) || !isfinite(sc)) {
      bad = 1;
      sc = 1.f;
    }
    acc += qerr_chunk(reinterpret_cast<const bf16_t*>(&v), sc, qmax);
  }
  const double t = block_sum<256>(acc, red);
  if (threadIdx.x == 0) part[blockIdx.x] = t;
  if (bad) report(status, JAB_ERR_NONFINITE);
}

// ---------------------------------------------------------------- flip count (App. B, Eq. 15)
// Number of positions where two int8 code arrays differ; 16 bytes per thread and step, one 64-bit
// atomic per block (integer sums: the result does not depend on the order).
__global__ void __launch_bounds__(256) flip_count_kernel(const uint4* __restrict__ a,
                                                         const uint4* __restrict__ b, int64_t n16,
                                                         const int8_t* __restrict__ a_tail,
                                                         const int8_t* __restrict__ b_tail,
                                                         int tail,
                                                         unsigned long long* __restrict__ count) {
  __shared__ unsigned long long red[8];
  unsigned long long c = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n16;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint4 x = __ldg(a + i), y = __ldg(b + i);
    // __vcmpne4: 0xff in each byte that differs
    c += __popc(__vcmpne4(x.x, y.x)) + __popc(__vcmpne4(x.y, y.y)) + __popc(__vcmpne4(x.z, y.z)) +
         __popc(__vcmpne4(x.w, y.w));
  }
  c >>= 3;  // eight set bits per differing byte
  if (blockIdx.x == 0 && (int)threadIdx.x < tail) c += a_tail[threadIdx.x] != b_tail[threadIdx.x];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < 8; ++w) t += red[w];
    atomicAdd(count, t);
  }
}

// ---------------------------------------------------------------- starting scales
// mode 0: absmax / qmax, one warp per (row, group).
__global__ void init_scales_kernel(const bf16_t* __restrict__ w, int D, int d, int G, int bits,
                                   float* __restrict__ s_out) {
  const int ng = d / G;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= (int64_t)D * ng) return;
  const int64_t row = warp / ng;
  const int g = (int)(warp - row * ng);
  const bf16_t* wp = w + row * d + (int64_t)g * G;
  float amax = 0.f;
  for (int i = lane; i < G; i += 32) amax = fmaxf(amax, fabsf(__bfloat162float(wp[i])));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if (lane == 0) s_out[warp] = (amax > 0.f) ? __fdiv_rn(amax, (float)qmax_of(bits)) : 1.f;
}

// mode 1: the trial scale s_k = fl32(s0 (100 - k) / 100), k < 80, with the least sum of
// (Q(w; s_k) - w)^2, the sums in fp64 and ties to the smallest k.
constexpr int kTrials = 80;
__device__ __forceinline__ float trial_scale(float s0, int k) {
  return (float)((double)s0 * (double)(100 - k) / 100.0);
}
// The same value from fp32 operations (an fp64 division per trial and group would cost more than the
// whole search): the product s0 (100 - k) exactly as ph + pl, its hundredth r, and one correction of r
// by the remainder, which is exact. The true quotient is either exactly between two floats or at
// least a hundredth of an ulp away from there, and the correction is good to 2^-22 ulp: only the
// exact ties need the second look, which takes the even neighbour.
__device__ __forceinline__ float trial_scale_f32(float s0, int k) {
  const float m = (float)(100 - k);
  const float ph = __fmul_rn(s0, m), pl = __fmaf_rn(s0, m, -ph);
  const float r = __fmul_rn(ph, 0.01f);
  const float rem = __fadd_rn(__fmaf_rn(-r, 100.f, ph), pl);
  const float y = __fmaf_rn(rem, 0.01f, r);
  const float left = __fmaf_rn(-100.f, __fsub_rn(y, r), rem);  // 100 (quotient - y), exact
  const float other = __int_as_float(__float_as_int(y) + (left > 0.f ? 1 : -1));
  const bool tie = __fmul_rn(50.f, fabsf(__fsub_rn(other, y))) == fabsf(left);
  return tie && (__float_as_int(y) & 1) ? other : y;
}

// Bound: FP64. A sum per trial in fp64 took 47.9 ms for 6144 x 4096 weights in groups of 64 (about two
// FP64 operations per clock and SM). Two stages instead, 0.40 ms:
//   1. all trials in fp32 with a bounded relative error: half a warp per group, five trials per lane,
//      the group's weights read from shared memory as broadcasts, packed pairs, no cross-lane sums.
//      The quotient is w * (1 / s_k) here, so a code can be off by one where the quotient is within
//      (qmax + 1) 2^-21 of a rounding boundary: both codes then have almost the same error.
//   2. where more than one trial lies within twice that bound of the least, exactly those are summed
//      in fp64 (the codes by the true quotient) by the whole warp, in the order of k.
// The choice is therefore that of the fp64 search. Groups whose scale is outside 2^-100 .. 2^100
// go through stage 2 with every trial.
__global__ void __launch_bounds__(256) init_scales_minmse_kernel(const bf16_t* __restrict__ w,
                                                                 int64_t ngroups, int G, int bits,
                                                                 float* __restrict__ s_out) {
  constexpr int kChunk = 64;               // weights of a group staged at a time (G is a multiple)
  constexpr int kSlots = kTrials / 16;     // trials per lane: k = 16 slot + lane % 16
  __shared__ float4 stage[8][2][kChunk / 4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int half = lane >> 4, l16 = lane & 15;
  const int64_t first = ((int64_t)blockIdx.x * 8 + warp) * 2;  // this warp's two groups
  if (first >= ngroups) return;
  const int64_t grp = first + half;
  const bool live = grp < ngroups;
  const bf16_t* wp = w + (live ? grp : first) * G;  // groups are consecutive: d is a multiple of G
  const int qmax = qmax_of(bits);
  const float qm = (float)qmax;
  float amax = 0.f;
  for (int i = l16; i < G; i += 16) amax = fmaxf(amax, fabsf(__bfloat162float(wp[i])));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  const float s0 = (amax > 0.f) ? __fdiv_rn(amax, qm) : 1.f;
  const bool window = s0 >= 7.8886091e-31f && s0 <= 1.2676506e30f;  // 2^-100, 2^100
  // weights and scales times 2^-exponent(s0), exactly: the squares neither under- nor overflow
  const float up = window ? __int_as_float((254 - ((__float_as_int(s0) >> 23) & 0xff)) << 23) : 0.f;
  float2 ns[kSlots], inv[kSlots], acc[kSlots];
#pragma unroll
  for (int j = 0; j < kSlots; ++j) {
    const float sk = window ? trial_scale_f32(s0, 16 * j + l16) * up : 1.f;
    const float r = __frcp_rn(sk);
    ns[j] = make_float2(-sk, -sk);
    inv[j] = make_float2(r, r);
    acc[j] = make_float2(0.f, 0.f);
  }
  const float2 magic = make_float2(12582912.f, 12582912.f);  // 1.5 * 2^23: adding it rounds to even
  for (int c = 0; c < G; c += kChunk) {
    __syncwarp();
    // (scalar loads: the weights need no more than their own alignment here)
    float* st = reinterpret_cast<float*>(stage[warp][half]);
#pragma unroll
    for (int e = 0; e < kChunk / 16; ++e)
      st[l16 + 16 * e] = __bfloat162float(wp[c + l16 + 16 * e]) * up;
    __syncwarp();
#pragma unroll 4
    for (int i = 0; i < kChunk / 4; ++i) {
      const float4 x4 = stage[warp][half][i];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float2 x = e ? make_float2(x4.z, x4.w) : make_float2(x4.x, x4.y);
#pragma unroll
        for (int j = 0; j < kSlots; ++j) {
          float2 v = tc::mul2(x, inv[j]);
          v.x = fminf(fmaxf(v.x, -qm), qm);
          v.y = fminf(fmaxf(v.y, -qm), qm);
          const float2 q = tc::sub2(tc::add2(v, magic), magic);
          const float2 err = tc::fma2(q, ns[j], x);
          acc[j] = tc::fma2(err, err, acc[j]);
        }
      }
    }
  }
  // Relative bound of stage 1: 8 (qmax + 1) 2^-21 from the codes, (G / 2 + 8) 2^-24 from the sums;
  // twice that on both sides, and an absolute term for sums lost below the smallest float.
  float least = INFINITY;
  float sum[kSlots];
#pragma unroll
  for (int j = 0; j < kSlots; ++j) {
    sum[j] = window ? acc[j].x + acc[j].y : 0.f;
    least = fminf(least, sum[j]);
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) least = fminf(least, __shfl_xor_sync(0xffffffffu, least, o));
  const float rel = (qm + 1.f) * 1.6e-5f + (float)G * 1.2e-7f + 2e-6f;
  const float limit = fmaf(least, rel, least) + 1e-30f;
  uint32_t cand[kSlots];  // bit l of each half: trial 16 slot + l is within the bound
  int count = 0;
#pragma unroll
  for (int j = 0; j < kSlots; ++j) {
    cand[j] = __ballot_sync(0xffffffffu, amax > 0.f && sum[j] <= limit);
    count += __popc((cand[j] >> (16 * half)) & 0xffffu);
  }
  int best = -1;  // index of the chosen trial; -1: keep s0 (an all-zero group, or NaN sums)
  if (count == 1) {
#pragma unroll
    for (int j = 0; j < kSlots; ++j) {
      const uint32_t m = (cand[j] >> (16 * half)) & 0xffffu;
      if (m) best = 16 * j + __ffs((int)m) - 1;
    }
  }
  const uint32_t several = __ballot_sync(0xffffffffu, count > 1);
  for (int hh = 0; hh < 2; ++hh) {  // stage 2: the whole warp on one group
    if (!((several >> (16 * hh)) & 1u)) continue;
    const float t0 = __shfl_sync(0xffffffffu, s0, 16 * hh);
    const bf16_t* gp = w + (first + hh) * G;
    double best_err = INFINITY;
    int pick = -1;
    for (int j = 0; j < kSlots; ++j) {
      uint32_t m = 0;
#pragma unroll
      for (int jj = 0; jj < kSlots; ++jj)
        if (jj == j) m = (cand[jj] >> (16 * hh)) & 0xffffu;
      for (; m; m &= m - 1) {
        const int k = 16 * j + __ffs((int)m) - 1;
        const float sk = trial_scale(t0, k);
        double err = 0.0;
        for (int i = lane; i < G; i += 32) {
          const float wv = __bfloat162float(gp[i]);
          const float q = quant_code(wv, sk, qmax, nullptr);
          const double e = (double)q * (double)sk - (double)wv;
          err += e * e;
        }
        err = warp_sum(err);
        if (err < best_err) {
          best_err = err;
          pick = k;
        }
      }
    }
    if (half == hh) best = pick;
  }
  if (live && l16 == 0) s_out[grp] = best >= 0 ? trial_scale(s0, best) : s0;
}

// ---------------------------------------------------------------- RoPE table (reading R7)
__global__ void rope_table_kernel(int T, int dh, double theta, float* __restrict__ cos_t,
                                  float* __restrict__ sin_t) {
  const int half = dh / 2;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)T * half) return;
  const int t = (int)(i / half), j = (int)(i % half);
  const double inv_freq = pow(theta, -2.0 * (double)j / (double)dh);
  const double phi = (double)t * inv_freq;
  double sn, cs;
  sincos(phi, &sn, &cs);
  cos_t[i] = (float)cs;
  sin_t[i] = (float)sn;
}

// ---------------------------------------------------------------- host launchers
static int grid_for(int64_t n, int threads, int sms) {
  int64_t g = (n + threads - 1) / threads;
  const int64_t cap = (int64_t)sms * 8;
  return (int)(g < cap ? (g < 1 ? 1 : g) : cap);
}

cudaError_t launch_convert_x(const void* x, void* xh, int64_t n, int* status, int sms,
                             cudaStream_t st) {
  const int64_t n8 = n / 8;
  convert_x_kernel<<<grid_for(n8, 256, sms), 256, 0, st>>>((const uint4*)x, (uint4*)xh, n8, status);
  return cudaGetLastError();
}

cudaError_t launch_quantize(const void* w, const float* s, int D, int d, int G, int bits,
                            void* w16, int8_t* codes, float* w_hat32, int* status, int sms,
                            cudaStream_t st) {
  const int64_t n8 = (int64_t)D * d / 8;
  quantize_kernel<<<grid_for(n8, 256, sms), 256, 0, st>>>(
      (const uint4*)w, s, D, d, G, bits, (uint4*)w16, codes, w_hat32, status);
  return cudaGetLastError();
}

cudaError_t launch_flip_count(const int8_t* a, const int8_t* b, int64_t n, int64_t* count,
                              int sms, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int64_t), st);
  if (e != cudaSuccess) return e;
  const int64_t n16 = n / 16;
  const int tail = (int)(n - n16 * 16);
  flip_count_kernel<<<grid_for(n16 > 0 ? n16 : 1, 256, sms), 256, 0, st>>>(
      (const uint4*)a, (const uint4*)b, n16, a + n16 * 16, b + n16 * 16, tail,
      reinterpret_cast<unsigned long long*>(count));
  return cudaGetLastError();
}

cudaError_t launch_rademacher_probe(uint64_t seed, uint64_t first, int64_t n, int log2_scale,
                                    void* out, int sms, cudaStream_t st) {
  const int64_t n8 = n / 8;
  if (log2_scale < 0 || log2_scale > 14) return cudaErrorInvalidValue;
  rademacher_probe_kernel<<<grid_for(n8, 256, sms), 256, 0, st>>>(seed, first, n8, log2_scale,
                                                                 (uint4*)out);
  return cudaGetLastError();
}

cudaError_t launch_qerr_partial(const void* w, const float* s, int D, int d, int G, int bits,
                                double* part, int nblocks, int* status, cudaStream_t st) {
  qerr_partial_kernel<<<nblocks, 256, 0, st>>>((const uint4*)w, s, D, d, G, bits, part, status);
  return cudaGetLastError();
}

cudaError_t launch_init_scales(const void* w, int D, int d, int G, int bits, int mode,
                               float* s_out, cudaStream_t st) {
  const int64_t groups = (int64_t)D * (d / G);
  if (mode == 0)
    init_scales_kernel<<<(unsigned)((groups + 7) / 8), 256, 0, st>>>((const bf16_t*)w, D, d, G, bits,
                                                                     s_out);
  else
    init_scales_minmse_kernel<<<(unsigned)((groups + 15) / 16), 256, 0, st>>>((const bf16_t*)w, groups,
                                                                              G, bits, s_out);
  return cudaGetLastError();
}

cudaError_t launch_rope_table(int T, int dh, double theta, float* cos_t, float* sin_t,
                              cudaStream_t st) {
  const int64_t n = (int64_t)T * (dh / 2);
  rope_table_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(T, dh, theta, cos_t, sin_t);
  return cudaGetLastError();
}

}  // namespace jab

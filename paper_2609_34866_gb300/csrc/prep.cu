// Elementwise and small kernels of the L_JAB path: X conversion, the quantiser (Eq. 2) and the RoPE
// table in one launch, the quantiser alone, scale initialisation, probes, sums over the weights.
// 16-byte vector loads and stores, grids sized in multiples of the SM count.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "tc.cuh"

namespace jab {

// Arguments of prep_kernel (a part that is not wanted has no blocks).
struct PrepArgs {
  static constexpr int kMaxCand = 8;  // candidates of one launch
  int nrope, nw, nx;                  // blocks of the RoPE table, the weights and X
  const uint4* x;
  uint4* xh;
  int64_t n8x;
  const uint4* w;
  uint4* w16;  // [ncand, D, d] fp16
  const float* s[kMaxCand];
  int bits[kMaxCand];
  int ncand, D, d, G;
  float *cos_t, *sin_t;
  int T, half;
  double freq_pi[64];  // theta^(-j / half) / pi
  int* status;
  int* counter;  // zeroed for the call's reductions
};

// ---------------------------------------------------------------- X: bf16 -> fp16 (+ range check)
// 8 bf16 as fp16; the largest magnitudes before and after, for the finiteness and range checks.
__device__ __forceinline__ uint4 convert8(const uint4& v, uint32_t& in, uint32_t& out) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  uint4 o;
  uint32_t* u = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    u[k] = tc::pack_half2(__uint_as_float(w[k] << 16), __uint_as_float(w[k] & 0xffff0000u));
    in = max_abs_f16x2(in, w[k]);
    out = max_abs_f16x2(out, u[k]);
  }
  return o;
}

// Block `blk` of `nblk`: four 16-byte loads of a thread in flight at a time.
__device__ __forceinline__ void convert_x_role(const uint4* __restrict__ x, uint4* __restrict__ xh,
                                               int64_t n8, int blk, int nblk, int* status) {
  uint32_t in = 0, out = 0;
  const int64_t step = (int64_t)nblk * blockDim.x;
  int64_t i = (int64_t)blk * blockDim.x + threadIdx.x;
  for (; i + 3 * step < n8; i += 4 * step) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = __ldg(x + i + u * step);
#pragma unroll
    for (int u = 0; u < 4; ++u) xh[i + u * step] = convert8(v[u], in, out);
  }
  for (; i < n8; i += step) xh[i] = convert8(__ldg(x + i), in, out);
  if (either_at_least(in, kBf16Inf)) report(status, JAB_ERR_NONFINITE);
  else if (either_at_least(out, kHalfInf)) report(status, JAB_ERR_RANGE);
}

// ---------------------------------------------------------------- quantiser (Section 2.1, Eq. 2)
// Codes of 8 weights that share a scale, as floats: clip(rint(fl32(w / s))), a zero of either sign.
__device__ __forceinline__ void quant_codes8(const uint4& v, float sc, int qmax, float (&q)[8]) {
  const uint32_t w2[4] = {v.x, v.y, v.z, v.w};
  const bf16_t* b = reinterpret_cast<const bf16_t*>(&v);
  uint32_t big = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) big = max_abs_f16x2(big, w2[k]);
  if (quot_window(sc) && !either_at_least(big, kBf16TwoTo60)) {
    const float r = __frcp_rn(sc), qm = (float)qmax;
    const float2 r2 = make_float2(r, r), ns2 = make_float2(-sc, -sc);
    const float2 magic = make_float2(12582912.f, 12582912.f);  // 1.5 * 2^23: rounds half to even
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 w = make_float2(__uint_as_float(w2[k] << 16), __uint_as_float(w2[k] & 0xffff0000u));
      const float2 v0 = tc::mul2(w, r2);
      float2 t = tc::fma2(tc::fma2(v0, ns2, w), r2, v0);
      t.x = fminf(fmaxf(t.x, -qm), qm);  // qmax is whole: clipping before rounding is the same
      t.y = fminf(fmaxf(t.y, -qm), qm);
      const float2 c = tc::sub2(tc::add2(t, magic), magic);
      q[2 * k] = c.x;
      q[2 * k + 1] = c.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) q[k] = quant_code(__bfloat162float(b[k]), sc, qmax, nullptr);
  }
}

// The scale of 8-weight chunk i is number i / (G / 8), as G divides the row length. Walks that quotient
// along a grid-stride loop by additions: an integer division per chunk costs as much as its codes.
struct GroupWalk {
  int64_t g;       // quotient
  int r;           // remainder
  int64_t dg;      // steps of both
  int dr, g8;
  __device__ __forceinline__ GroupWalk(int64_t i, int64_t step, int g8_) : g8(g8_) {
    g = i / g8;
    r = (int)(i - g * g8);
    dg = step / g8;
    dr = (int)(step - dg * g8);
  }
  __device__ __forceinline__ int64_t next() {  // the quotient at i, then on to i + step
    const int64_t now = g;
    g += dg;
    r += dr;
    if (r >= g8) {
      r -= g8;
      ++g;
    }
    return now;
  }
};

// w_hat = q s of 8 weights as fp16 operands; the largest magnitude, for the range check.
__device__ __forceinline__ uint4 pack_w16(const float (&f)[8], uint32_t& out) {
  uint4 o;
  uint32_t* u = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    u[k] = tc::pack_half2(f[2 * k], f[2 * k + 1]);
    out = max_abs_f16x2(out, u[k]);
  }
  return o;
}

// A scale as the quantiser uses it: finite and > 0 (else flagged, and 1 in its place).
__device__ __forceinline__ float checked_scale(float sc, int& bad) {
  if (sc > 0.f && isfinite(sc)) return sc;
  bad |= 1;
  return 1.f;
}

// jab_quantize: int8 codes and / or fp32 w_hat.
__global__ void __launch_bounds__(256) quantize_kernel(const uint4* __restrict__ w,
                                                       const float* __restrict__ s, int D, int d,
                                                       int G, int bits, int8_t* __restrict__ codes,
                                                       float* __restrict__ w_hat32, int* status) {
  const int64_t n8 = (int64_t)D * d / 8, step = (int64_t)gridDim.x * blockDim.x;
  const int qmax = qmax_of(bits);
  int bad = 0;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  GroupWalk at(i, step, G / 8);
  auto put = [&](const uint4& v, float sc, int64_t i) {
    float q[8];
    quant_codes8(v, sc, qmax, q);
    if (codes) {
      uint32_t c[2];
#pragma unroll
      for (int h = 0; h < 2; ++h)
        c[h] = (uint32_t)((int)q[4 * h] & 0xff) | (uint32_t)((int)q[4 * h + 1] & 0xff) << 8 |
               (uint32_t)((int)q[4 * h + 2] & 0xff) << 16 | (uint32_t)(int)q[4 * h + 3] << 24;
      *reinterpret_cast<uint2*>(codes + i * 8) = make_uint2(c[0], c[1]);
    }
    if (w_hat32) {
      const uint32_t w2[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 8; ++k)  // with the weight's sign, which rint keeps in a code of 0 and quant_codes8 does not
        q[k] = __uint_as_float(__float_as_uint(__fmul_rn(q[k], sc)) |
                               ((k & 1 ? w2[k / 2] : w2[k / 2] << 16) & 0x80000000u));
      reinterpret_cast<float4*>(w_hat32 + i * 8)[0] = make_float4(q[0], q[1], q[2], q[3]);
      reinterpret_cast<float4*>(w_hat32 + i * 8)[1] = make_float4(q[4], q[5], q[6], q[7]);
    }
  };
  for (; i + step < n8; i += 2 * step) {
    const uint4 v0 = __ldg(w + i), v1 = __ldg(w + i + step);
    const float s0 = __ldg(s + at.next()), s1 = __ldg(s + at.next());
    put(v0, checked_scale(s0, bad), i);
    put(v1, checked_scale(s1, bad), i + step);
  }
  if (i < n8) put(__ldg(w + i), checked_scale(__ldg(s + at.next()), bad), i);
  if (bad) report(status, JAB_ERR_NONFINITE);
}

// Block `blk` of `nblk`: the fp16 operand of every candidate (or of W itself, ncand = 0). W is read
// once for all candidates; the outputs are what moves.
__device__ __forceinline__ void quantize_role(const PrepArgs& p, int blk, int nblk) {
  const int64_t n8 = (int64_t)p.D * p.d / 8, step = (int64_t)nblk * blockDim.x;
  int bad = 0;
  uint32_t in = 0, out = 0;
  int64_t i = (int64_t)blk * blockDim.x + threadIdx.x;
  if (p.ncand == 0) {
    for (; i + step < n8; i += 2 * step) {
      const uint4 v0 = __ldg(p.w + i), v1 = __ldg(p.w + i + step);
      p.w16[i] = convert8(v0, in, out);
      p.w16[i + step] = convert8(v1, in, out);
    }
    if (i < n8) p.w16[i] = convert8(__ldg(p.w + i), in, out);
  } else {
    GroupWalk at(i, step, p.G / 8);
    auto put = [&](const uint4& v, float sc, int c, int64_t i) {
      float q[8];
      sc = checked_scale(sc, bad);
      quant_codes8(v, sc, qmax_of(p.bits[c]), q);
#pragma unroll
      for (int k = 0; k < 8; ++k) q[k] = __fmul_rn(q[k], sc);
      p.w16[c * n8 + i] = pack_w16(q, out);
    };
    for (; i < n8; i += 2 * step) {
      const bool two = i + step < n8;
      const uint4 v0 = __ldg(p.w + i);
      uint4 v1 = make_uint4(0u, 0u, 0u, 0u);
      if (two) v1 = __ldg(p.w + i + step);
      const int64_t g0 = at.next(), g1 = two ? at.next() : g0;
      float s0 = __ldg(p.s[0] + g0), s1 = __ldg(p.s[0] + g1);
      for (int c = 0; c < p.ncand; ++c) {
        const int cn = c + 1 < p.ncand ? c + 1 : c;  // the next candidate's scales, ahead
        const float n0 = __ldg(p.s[cn] + g0), n1 = __ldg(p.s[cn] + g1);
        put(v0, s0, c, i);
        if (two) put(v1, s1, c, i + step);
        s0 = n0;
        s1 = n1;
      }
    }
  }
  if (bad) report(p.status, JAB_ERR_NONFINITE);
  else if (either_at_least(out, kHalfInf)) report(p.status, JAB_ERR_RANGE);  // not an fp16 operand
}

// ---------------------------------------------------------------- RoPE table (reading R7)
// fp64: a pow and a sincos per entry took 48 us for 2048 x 64, as an SM issues an fp64 instruction of a
// warp in about 16 clocks. The frequencies come with the launch; a thread takes the sincos of its
// first row and of one step and rotates on through kRopeRun rows (an fp64 rotation adds 1e-16, the
// table keeps 6e-8); a block has one run of rows only, so that the work spreads over all SMs.
constexpr int kRopeRun = 16;
__device__ __forceinline__ void rope_role(const PrepArgs& p, int blk) {
  const int j = threadIdx.x, t0 = blk * kRopeRun;
  if (j >= p.half) return;
  const double f = p.freq_pi[j];  // (the pi forms need no long argument reduction)
  double sn, cs, sd, cd;
  sincospi((double)t0 * f, &sn, &cs);
  sincospi(f, &sd, &cd);
  const int n = min(kRopeRun, p.T - t0);
  int64_t i = (int64_t)t0 * p.half + j;
  for (int k = 0; k < n; ++k, i += p.half) {
    p.cos_t[i] = (float)cs;
    p.sin_t[i] = (float)sn;
    const double c2 = cs * cd - sn * sd;
    sn = sn * cd + cs * sd;
    cs = c2;
  }
}

// Everything the projection reads that is not there yet, in one launch: blocks [0, nrope) the RoPE
// table, then nw blocks the weights, then nx blocks X. As launches of their own, and with a 64-bit index
// division per chunk and a quotient division per weight, they took 38 us for one candidate's 6144 x
// 4096 weights and 30-85 us for the table (1337-4096 rows), now 31 us together at 1337 rows; for five
// candidates, 2048 rows and 65536 x 4096 of X 462 us, now 248 us (1.37 GB: 202 us at the copy rate).
__global__ void __launch_bounds__(256, 4) prep_kernel(const __grid_constant__ PrepArgs p) {
  stream_order();
  const int blk = blockIdx.x;
  if (blk == 0 && threadIdx.x == 0 && p.counter != nullptr) *p.counter = 0;
  if (blk < p.nrope)
    rope_role(p, blk);
  else if (blk < p.nrope + p.nw)
    quantize_role(p, blk - p.nrope, p.nw);
  else
    convert_x_role(p.x, p.xh, p.n8x, blk - p.nrope - p.nw, p.nx, p.status);
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
// with the errors carried along, and only that sum goes to the fp64 accumulator: 42 us. Weights and
// scale are first multiplied by the power of two that brings the scale to [1, 2) (exact), so that no
// square under- or overflows; a chunk whose values leave that window takes the fp64 form.
// Sum of (q s - w)^2 over the 8 weights of a chunk.
__device__ __forceinline__ double qerr_chunk(const uint4& v, float sc, int qmax) {
  const bf16_t* b = reinterpret_cast<const bf16_t*>(&v);
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
  float sh = 0.f, sl = 0.f, code[8];
  quant_codes8(v, sc, qmax, code);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float wv = __bfloat162float(b[k]), q = code[k];
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
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  double acc = 0.0;
  int bad = 0;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (GroupWalk at(i, step, G / 8); i < n8; i += step) {
    const uint4 v = __ldg(w + i);
    const float sc = checked_scale(__ldg(s + at.next()), bad);
    acc += qerr_chunk(v, sc, qmax);
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

// ---------------------------------------------------------------- host launchers
static int grid_for(int64_t n, int threads, int sms) {
  int64_t g = (n + threads - 1) / threads;
  const int64_t cap = (int64_t)sms * 8;
  return (int)(g < cap ? (g < 1 ? 1 : g) : cap);
}

cudaError_t launch_prep(const PrepInputs& in, int* status, int sms, cudaStream_t st) {
  const int64_t n8 = (int64_t)in.D * in.d / 8;
  for (int c0 = 0; c0 == 0 || c0 < in.ncand; c0 += PrepArgs::kMaxCand) {
    PrepArgs p{};
    p.status = status;
    p.counter = in.counter;
    p.D = in.D;
    p.d = in.d;
    p.G = in.G;
    if (in.w != nullptr) {
      p.w = static_cast<const uint4*>(in.w);
      p.w16 = static_cast<uint4*>(in.w16) + c0 * n8;
      p.ncand = std::min(in.ncand - c0, (int)PrepArgs::kMaxCand);
      for (int c = 0; c < p.ncand; ++c) {
        p.s[c] = in.s[c0 + c];
        p.bits[c] = in.bits[c0 + c];
      }
      p.nw = std::min(grid_for(n8, 256, sms), 4 * sms);  // what is resident at once
    }
    if (c0 == 0 && in.x != nullptr) {
      p.x = static_cast<const uint4*>(in.x);
      p.xh = static_cast<uint4*>(in.xh);
      p.n8x = in.nx / 8;
      p.nx = std::min(grid_for((p.n8x + 3) / 4, 256, sms), 4 * sms);
    }
    if (c0 == 0 && in.cos_t != nullptr) {
      p.cos_t = in.cos_t;
      p.sin_t = in.sin_t;
      p.T = in.T;
      p.half = in.dh / 2;
      // by squares of the first ratio: one pow a call, each frequency a product of at most six powers
      // (long double: the rounding to double is the only one that counts)
      long double pw[6];
      pw[0] = powl((long double)in.theta, -1.0L / p.half);
      for (int b = 1; b < 6; ++b) pw[b] = pw[b - 1] * pw[b - 1];
      for (int j = 0; j < p.half; ++j) {
        long double f = 0.318309886183790671537767526745028724L;  // 1 / pi
        for (int b = 0; b < 6; ++b)
          if ((j >> b) & 1) f *= pw[b];
        p.freq_pi[j] = (double)f;
      }
      p.nrope = (in.T + kRopeRun - 1) / kRopeRun;
    }
    const int grid = p.nrope + p.nw + p.nx;
    if (grid == 0) return cudaSuccess;
    const cudaError_t e = launch_after(prep_kernel, (unsigned)grid, 256, 0, st, p);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_quantize(const void* w, const float* s, int D, int d, int G, int bits,
                            int8_t* codes, float* w_hat32, int* status, int sms, cudaStream_t st) {
  const int64_t n8 = (int64_t)D * d / 8;
  quantize_kernel<<<grid_for(n8, 256, sms), 256, 0, st>>>((const uint4*)w, s, D, d, G, bits, codes,
                                                          w_hat32, status);
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

}  // namespace jab

// Tensor-core (tcgen05) GEMMs of the L_JAB path on sm_103a.
//
//   C[m, n] = sum_k A[m, k] B[n, k]        A K-major 16-bit, fp32 accumulation in TMEM; B K-major
//                                          (stored [n][k]) or MN-major (stored [k][n])
//
// Persistent, warp-specialised kernel on CTA pairs (clusters of two CTAs on two SMs, cta_group::2):
// a pair computes a 256 x 256 tile with M256 N256 K16 UMMAs issued by its even CTA; each CTA holds
// 128 rows of A, half of the B tile and 128 lanes of the accumulator (details above the kernel).
//   warp 0      TMA producer: the CTA's 128x64 A tile and 128x64 half of B per stage, 6-stage ring
//   warp 1      TMEM owner (two accumulators, allocated by the pair) and, in the even CTA, UMMA issuer
//   warps 2..5  epilogue: tcgen05.ld of the CTA's 128 x 256 fp32 accumulator, one lane per thread;
//               the projection's fp16 results leave by TMA through two boxes per warp
// Two accumulators (2 x 256 TMEM columns) let the epilogue of one tile overlap the next mainloop.
// With few tiles a pair takes 256 x 128 of C instead (tile_cols).
//
// Epilogues:
//   projection  [Q|K|V] = X w_hat^T: rotate-half RoPE on the Q and K heads (partner column +-d_h/2
//               lives in the same thread's row), fp16 store.
//   wgrad       G = dQKV^T X (K = tokens, split-K): ds[o, g] += coef * sum_{i in g} G[o,i] r[o,i]
//               with the LSQ factor r of Eq. 13 recomputed from w and s; G is never stored. X is
//               read as it is stored, [tokens, features], as the MN-major B operand (two 64-feature
//               TMA boxes per CTA and stage), so no transposed copy of X is needed.
//   store       coef * dQKV^T X as fp32 dW (STE weight gradient) and / or its squared norm; with a
//               split K the partial tiles are added into a zeroed dW with vector atomics and the
//               norm is reduced from dW afterwards in fixed order.
#include <cudaTypedefs.h>

#include "kernels.h"
#include "tc.cuh"

namespace jab {
namespace {

constexpr int BM = 128, BK = 64;  // BM: rows of one CTA (an epilogue's 128 TMEM lanes); BN: 256 or 128 (tile_cols)
constexpr int A_BYTES = BM * BK * 2;
constexpr int NUM_THREADS = 192;

enum EpiKind { kEpiRope = 0, kEpiLsq = 1, kEpiStore = 2 };

struct GemmParams {
  int64_t M;
  int Nn, K;
  int num_m, num_n, splits, k_blocks, group_m;
  int* status;
  // projection epilogue
  int D, n_rot, dh, T;
  const float* cos_t;
  const float* sin_t;
  // LSQ epilogue
  const bf16_t* w;
  const float* s;
  int d, G, bits;
  float coef;
  int parts;      // tiles that a group may touch (lsq_group_parts)
  float* dspart;  // fp32 [splits, parts, M, d/G]: each unit's partials, summed in order afterwards
  // weight-gradient store epilogue (a split K adds partial tiles into a zeroed dw)
  float* dw;
};

__device__ __forceinline__ void decode_unit(const GemmParams& p, int unit, int& mb, int& nb,
                                            int& ks) {
  const int tiles = p.num_m * p.num_n;
  ks = unit / tiles;
  const int t = unit - ks * tiles;
  const int span = p.group_m * p.num_n;
  const int grp = t / span;
  const int first_m = grp * p.group_m;
  const int gm = min(p.group_m, p.num_m - first_m);
  const int local = t - grp * span;
  mb = first_m + local % gm;
  nb = local / gm;
}

__device__ __forceinline__ void k_range(const GemmParams& p, int ks, int& kb0, int& kb1) {
  kb0 = (int)((int64_t)p.k_blocks * ks / p.splits);
  kb1 = (int)((int64_t)p.k_blocks * (ks + 1) / p.splits);
}

// Waits for a barrier phase while draining at exit: time-bounded, ignores the abort flag.
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = tc::globaltimer();
  while (!tc::mbar_test(bar, parity)) {
    if (tc::globaltimer() - t0 > tc::kWaitLimitNs) break;
  }
}

// The projection's 128 rows x 256 columns of one CTA, RoPE applied, to fp16 C. A thread has one row, so
// storing its registers directly is 16 bytes of 32 different rows per instruction; at K = 768 (12 K
// blocks) that took 11.5k clocks a tile where the products take 6.1k (65536 x 9216: 735 us, now 526). The
// warp's 32 rows x 64 columns go through a swizzled box in shared memory and leave by TMA (rows past M
// are clipped by the tensor map). buf: the warp's two boxes.
template <int BN>
__device__ __forceinline__ void epi_rope(const GemmParams& p, const CUtensorMap* tmC, uint32_t taddr,
                                         int mb, int nb, int row, uint8_t* buf) {
  const int lane = row & 31;
  const int64_t m = (int64_t)mb * BM + row;
  const int64_t y = m - lane;  // the warp's first row
  const bool row_ok = m < p.M;
  const int t = row_ok ? (int)(m % p.T) : 0;
  const int half = p.dh >> 1;
  uint32_t big = 0;  // largest magnitude bits of the row's fp16 results
#pragma unroll 1
  for (int pr = 0; pr < BN / 64; ++pr) {
    const int c1 = (p.dh == 128) ? (pr >> 1) * 4 + (pr & 1) : pr * 2;
    const int c2 = c1 + half / 32;
    const int col1 = nb * BN + c1 * 32;
    if (col1 >= p.Nn) continue;  // uniform over the warp
    uint32_t ra[32], rb[32];
    __syncwarp();  // tcgen05.ld is warp-collective (.sync.aligned)
    tc::tmem_ld32(taddr + c1 * 32, ra);
    tc::tmem_ld32(taddr + c2 * 32, rb);
    tc::tmem_ld_wait();
    float a[32], b[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      a[i] = __uint_as_float(ra[i]);
      b[i] = __uint_as_float(rb[i]);
    }
    const int o = col1 % p.D;
    if (p.n_rot > 0 && o < p.n_rot &&
        in_bounds((int64_t)t * half + o % p.dh + 31, (int64_t)p.T * half, p.status)) {
      const int jj0 = o % p.dh;
      const float4* cp = reinterpret_cast<const float4*>(p.cos_t + (int64_t)t * half + jj0);
      const float4* sp = reinterpret_cast<const float4*>(p.sin_t + (int64_t)t * half + jj0);
      // Packed FP32 pairs: this epilogue overlaps the next tile's UMMAs, which scalar FP32
      // instructions at a high rate slow down.
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        const float4 c4 = __ldg(cp + v), s4 = __ldg(sp + v);
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
          const int i = v * 4 + e;
          const float2 cs = e ? make_float2(c4.z, c4.w) : make_float2(c4.x, c4.y);
          const float2 sn = e ? make_float2(s4.z, s4.w) : make_float2(s4.x, s4.y);
          const float2 nsn = make_float2(tc::neg_bits(sn.x), tc::neg_bits(sn.y));
          const float2 x1 = make_float2(a[i], a[i + 1]), x2 = make_float2(b[i], b[i + 1]);
          const float2 ra = tc::fma2(x2, nsn, tc::mul2(x1, cs));  // x1 cos - x2 sin
          const float2 rb = tc::fma2(x1, sn, tc::mul2(x2, cs));   // x2 cos + x1 sin
          a[i] = ra.x;
          a[i + 1] = ra.y;
          b[i] = rb.x;
          b[i + 1] = rb.y;
        }
      }
    }
    // Boxes of 64 columns. d_h = 64: a and b are the halves of one box, the two boxes in turn. d_h = 128:
    // columns c1 are in the head's first box, c2 in its second; two rounds fill both.
    const bool wide = p.dh == 128;
    if (tc::elect_one()) {  // (the same lane that issues the stores) the box has been read
      if (!wide)
        tc::bulk_wait_group_read<1>();
      else if ((pr & 1) == 0)
        tc::bulk_wait_group_read<0>();
    }
    __syncwarp();
    uint8_t* box_a = buf + (wide ? 0 : (pr & 1) * 4096) + lane * 128;
    uint8_t* box_b = wide ? box_a + 4096 : box_a;
    const int ua = wide ? (pr & 1) * 4 : 0, ub = wide ? ua : 4;  // 16-byte units of the box row
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      uint32_t u1[4], u2[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        u1[e] = tc::pack_half2(a[v * 8 + 2 * e], a[v * 8 + 2 * e + 1]);
        u2[e] = tc::pack_half2(b[v * 8 + 2 * e], b[v * 8 + 2 * e + 1]);
        big = max_abs_f16x2(max_abs_f16x2(big, u1[e]), u2[e]);
      }
      *reinterpret_cast<uint4*>(box_a + (((ua + v) ^ (lane & 7)) << 4)) = make_uint4(u1[0], u1[1], u1[2], u1[3]);
      *reinterpret_cast<uint4*>(box_b + (((ub + v) ^ (lane & 7)) << 4)) = make_uint4(u2[0], u2[1], u2[2], u2[3]);
    }
    if (!wide || (pr & 1)) {
      tc::fence_proxy_async_smem();
      __syncwarp();
      if (tc::elect_one()) {
        if (y < p.M) {
          const int x0 = wide ? col1 - 32 : col1;
          tc::tma_store_2d(tmC, buf + (wide ? 0 : (pr & 1) * 4096), x0, (int32_t)y);
          if (wide) tc::tma_store_2d(tmC, buf + 4096, x0 + 64, (int32_t)y);
        }
        tc::bulk_commit_group();
      }
      __syncwarp();
    }
  }
  // a half with all exponent bits set: inf (out of fp16 range) or NaN
  if (row_ok && either_at_least(big, kHalfInf)) report(p.status, JAB_ERR_RANGE);
}

// STE weight gradient (App. B: d w_hat / d w = 1, so dL/dW = dL/dw_hat = coef * dQKV^T X): the
// tile times coef stored as fp32 rows of dw (with a split K each unit's partial tile is added with
// vector atomics). Packed FP32 pairs, as this runs beside the next tile's UMMAs.
template <int BN>
__device__ __forceinline__ void epi_store(const GemmParams& p, uint32_t taddr, int mb, int nb,
                                          int row) {
  const int64_t o = (int64_t)mb * BM + row;  // M = D is a multiple of 128: every row is valid
  const float2 c2 = make_float2(p.coef, p.coef);
#pragma unroll 1
  for (int c = 0; c < BN / 32; ++c) {
    const int i0 = nb * BN + c * 32;
    if (i0 >= p.Nn) break;  // uniform over the warp
    uint32_t r[32];
    __syncwarp();
    tc::tmem_ld32(taddr + c * 32, r);
    tc::tmem_ld_wait();
    float g[32];
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
      const float2 v = tc::mul2(make_float2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), c2);
      g[i] = v.x;
      g[i + 1] = v.y;
    }
    if (p.dw != nullptr && in_bounds(o * p.Nn + i0 + 31, p.M * (int64_t)p.Nn, p.status)) {
      float4* d = reinterpret_cast<float4*>(p.dw + o * p.Nn + i0);
      if (p.splits > 1) {  // a K range: add the partial tile into the zeroed dw
#pragma unroll
        for (int v = 0; v < 8; ++v)
          atomicAdd(d + v, make_float4(g[4 * v], g[4 * v + 1], g[4 * v + 2], g[4 * v + 3]));
      } else {
#pragma unroll
        for (int v = 0; v < 8; ++v) d[v] = make_float4(g[4 * v], g[4 * v + 1], g[4 * v + 2], g[4 * v + 3]);
      }
    }
  }
}

// Sum over 32 columns of G[o, i] r(w_i, sc) with the LSQ factor of Eq. 13. g: this row's columns of G, w: the
// 32 bf16 weights. The quotient in packed pairs from a corrected reciprocal where that is the IEEE one
// (see quot_window), by division elsewhere: with 32 divisions a chunk took 3k clocks, and small
// batches waited for the epilogue (512 tokens x 2304 x 768: 20.6 us).
__device__ __forceinline__ float lsq_chunk(const uint32_t (&g)[32], const uint4 (&w)[4], float sc, int qmax) {
  uint32_t big = 0, small = 0xffffffffu;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const uint32_t x[4] = {w[v].x, w[v].y, w[v].z, w[v].w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t m = x[e] & 0x7fff7fffu;
      big = __vmaxu2(big, m);
      small = __vminu2(small, m);  // (a zero weight takes the division too)
    }
  }
  const bool fast = quot_window(sc) && !either_at_least(big, kBf16TwoTo60) &&
                    (small & 0xffffu) >= kBf16TwoToM60 && (small >> 16) >= kBf16TwoToM60;
  float2 acc = make_float2(0.f, 0.f);
  if (fast) {
    const float r = __frcp_rn(sc), qm = (float)qmax;
    const float2 r2 = make_float2(r, r), ns2 = make_float2(-sc, -sc);
    const float2 magic = make_float2(12582912.f, 12582912.f);  // 1.5 * 2^23: rounds half to even
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const uint32_t x[4] = {w[v].x, w[v].y, w[v].z, w[v].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 wv = make_float2(__uint_as_float(x[e] << 16), __uint_as_float(x[e] & 0xffff0000u));
        const float2 v0 = tc::mul2(wv, r2);
        const float2 q = tc::fma2(tc::fma2(v0, ns2, wv), r2, v0);  // fl32(w / s)
        // q clipped to +-qmax (whole); inside, its rounding error is the factor, else the bound itself
        const float2 c = make_float2(fminf(fmaxf(q.x, -qm), qm), fminf(fmaxf(q.y, -qm), qm));
        const float2 d = tc::sub2(tc::sub2(tc::add2(c, magic), magic), q);
        const float2 f = make_float2(c.x == q.x ? d.x : c.x, c.y == q.y ? d.y : c.y);
        const int i = 8 * v + 2 * e;
        acc = tc::fma2(make_float2(__uint_as_float(g[i]), __uint_as_float(g[i + 1])), f, acc);
      }
    }
  } else {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const bf16_t* wb = reinterpret_cast<const bf16_t*>(&w[v]);
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        acc.x = fmaf(__uint_as_float(g[v * 8 + e]), lsq_factor(__bfloat162float(wb[e]), sc, qmax), acc.x);
        acc.y = fmaf(__uint_as_float(g[v * 8 + e + 1]), lsq_factor(__bfloat162float(wb[e + 1]), sc, qmax), acc.y);
      }
    }
  }
  return acc.x + acc.y;
}

template <int BN>
__device__ __forceinline__ void epi_lsq(const GemmParams& p, uint32_t taddr, int mb, int nb,
                                        int ks, int row) {
  const int o = mb * BM + row;  // M = D is a multiple of 128: every row is valid
  const int qmax = qmax_of(p.bits);
  const int ng = p.d / p.G;
  // One value per (split, part, row, group): with parts = 1 this unit's tile covers whole groups (BN is a
  // multiple of G); otherwise the tile is the group's part nb - (its first tile), and the one in which the
  // group ends writes zeros for the parts it does not have.
  const int64_t part_extent = (int64_t)p.splits * p.parts * p.M * ng;
  float* part_out = p.dspart + ((int64_t)ks * p.parts * p.M + o) * ng;
  const int64_t at0 = ((int64_t)ks * p.parts * p.M + o) * ng;
  auto put = [&](int g, float v) {
    if (p.parts == 1) {
      if (in_bounds(at0 + g, part_extent, p.status)) part_out[g] = v;
      return;
    }
    const int q0 = nb - (int)((int64_t)g * p.G / BN);
    const int q1 = (int64_t)(g + 1) * p.G > (int64_t)(nb + 1) * BN ? q0 : p.parts - 1;
    for (int q = q0; q <= q1; ++q) {
      const int64_t at = (int64_t)q * p.M * ng + g;
      if (in_bounds(at0 + at, part_extent, p.status)) part_out[at] = q == q0 ? v : 0.f;
    }
  };
  float part = 0.f;
  int cur = -1;
  // The weights and scale of a chunk are loaded while the one before it is summed.
  uint4 wn[4];
  float sn = 0.f;
  auto load = [&](int c) {
    const int i0 = nb * BN + c * 32;
    if (c < BN / 32 && i0 < p.Nn && in_bounds((int64_t)o * p.d + i0 + 31, (int64_t)p.M * p.d, p.status) &&
        in_bounds((int64_t)o * ng + i0 / p.G, (int64_t)p.M * ng, p.status)) {
      const uint4* wp = reinterpret_cast<const uint4*>(p.w + (int64_t)o * p.d + i0);
#pragma unroll
      for (int v = 0; v < 4; ++v) wn[v] = __ldg(wp + v);
      sn = __ldg(p.s + (int64_t)o * ng + i0 / p.G);
    }
  };
#pragma unroll
  for (int v = 0; v < 4; ++v) wn[v] = make_uint4(0u, 0u, 0u, 0u);
  load(0);
#pragma unroll 1
  for (int c = 0; c < BN / 32; ++c) {
    const int i0 = nb * BN + c * 32;
    if (i0 >= p.Nn) break;  // uniform over the warp
    uint32_t r[32];
    __syncwarp();
    tc::tmem_ld32(taddr + c * 32, r);
    const uint4 w[4] = {wn[0], wn[1], wn[2], wn[3]};
    const float sc = sn;
    load(c + 1);
    tc::tmem_ld_wait();
    const int g = i0 / p.G;
    if (g != cur) {
      if (cur >= 0) put(cur, p.coef * part);
      part = 0.f;
      cur = g;
    }
    part += lsq_chunk(r, w, sc, qmax);
  }
  if (cur >= 0) put(cur, p.coef * part);
}

// ------------------------------------------------------------------ CTA-pair variant (cta_group::2)
// Two CTAs of a cluster on two SMs share one 256 x 256 tile: CTA r holds rows 128 r .. 128 r + 127
// of A and rows 128 r .. of the B tile (the N half it loads), and its 128 accumulator lanes. One
// M256 N256 K16 UMMA per 16-deep K step, issued by the even CTA, reads A and B from both CTAs' shared
// memory. Each SM then stages 16 KB of A and 16 KB of B per K block instead of the 16 + 32 KB of a
// one-CTA 128 x 256 tile, so six stages fit where four did and the operand loads have 1.7x the
// look-ahead (the one-CTA layout was bound by it: three stages instead of four cost it 10-26 %).
//   warp 0      TMA producer (both CTAs): its rows of A and its half of B, completion counted on the
//               even CTA's stage barrier, which expects both CTAs' bytes
//   warp 1      TMEM owner (both CTAs, allocated collectively); UMMA issuer (even CTA, one thread);
//               each stage's commit releases the stage in both CTAs, each tile's commit wakes both
//               CTAs' epilogues
//   warps 2..5  epilogue (both CTAs): this CTA's 128 rows, as in the single-CTA kernel; the
//               accumulator is free again once all eight epilogue warps of the pair have arrived on
//               the even CTA's barrier
constexpr int STAGES2 = 6;
constexpr int BM2 = 2 * BM;                 // rows of A per pair tile
template <int BN>
constexpr int B2_ROWS = BN / 2;  // rows (K-major) or columns (MN-major) of B per CTA
template <int BN>
constexpr int STAGE2_BYTES = A_BYTES + B2_ROWS<BN> * BK * 2;
constexpr int EPI2_BYTES = 4 * 2 * 4096;  // two output boxes per epilogue warp
template <int BN>
constexpr int SMEM2_BYTES = STAGES2 * STAGE2_BYTES<BN> + EPI2_BYTES + 1024 + 256;

struct Bars2 {
  uint64_t full[STAGES2], empty[STAGES2], tfull[2], tempty[2], drain;
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(Bars2) <= 256, "barrier block");
static_assert(SMEM2_BYTES<256> <= 227 * 1024, "shared memory budget");

template <int EPI, bool BF16, bool B_MN, int BN>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    gemm2_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmC, const GemmParams p) {
  constexpr int SB = STAGE2_BYTES<BN>, BR = B2_ROWS<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  Bars2* bars = reinterpret_cast<Bars2*>(smem + STAGES2 * SB + EPI2_BYTES);
  const int warp = tc::warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = tc::cluster_ctarank();  // 0: issues the pair's UMMAs
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int total = p.num_m * p.num_n * p.splits;  // num_m counts 256-row blocks here
  volatile int* abort = &bars->abort;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES2; ++s) {
      tc::mbar_init(&bars->full[s], 1);
      tc::mbar_init(&bars->empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      tc::mbar_init(&bars->tfull[a], 1);
      tc::mbar_init(&bars->tempty[a], 2 * 4);  // the epilogue warps of both CTAs
    }
    tc::mbar_init(&bars->drain, 1);
    bars->abort = 0;
    tc::fence_mbar_init();
    tc::prefetch_tmap(&tmA);
    tc::prefetch_tmap(&tmB);
    if (EPI == kEpiRope) tc::prefetch_tmap(&tmC);
  }
  if (warp == 1) {
    tc::tmem_alloc2(&bars->tmem_base, 2 * BN);
    tc::tmem_relinquish2();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  // both CTAs' barriers are initialised and their tensor memory allocated before any signal crosses
  tc::cluster_sync();
  const uint32_t tmem = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  stream_order();
  const uint32_t full_lead = tc::mapa_shared(tc::smem_u32(&bars->full[0]), 0);
  const uint32_t tempty_lead = tc::mapa_shared(tc::smem_u32(&bars->tempty[0]), 0);

  if (warp == 0) {
    if (tc::elect_one()) {  // ---------------- TMA producer
      int stage = 0;
      uint32_t phase = 0;
      uint32_t issued = 0, last_parity = 0;  // per-stage bitmasks for the exit drain (even CTA)
      for (int unit = pair; unit < total && !*abort; unit += npairs) {
        int mb, nb, ks, kb0, kb1;
        decode_unit(p, unit, mb, nb, ks);
        k_range(p, ks, kb0, kb1);
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!tc::mbar_wait(&bars->empty[stage], phase ^ 1, abort, p.status)) break;
          uint8_t* sa = smem + stage * SB;
          const uint32_t bar = full_lead + stage * 8;
          if (leader) tc::mbar_expect_tx(&bars->full[stage], 2 * SB);
          tc::tma_load_2d_pair(sa, &tmA, bar, kb * BK, mb * BM2 + (int)rank * BM);
          if (B_MN)  // B stored [k][n]: this CTA's two boxes of BK rows x 64 columns
            for (int c = 0; c < BR / 64; ++c)
              tc::tma_load_2d_pair(sa + A_BYTES + c * (BK * 128), &tmB, bar,
                                   nb * BN + (int)rank * BR + c * 64, kb * BK);
          else
            tc::tma_load_2d_pair(sa + A_BYTES, &tmB, bar, kb * BK, nb * BN + (int)rank * BR);
          issued |= 1u << stage;
          last_parity = (last_parity & ~(1u << stage)) | (phase << stage);
          if (++stage == STAGES2) {
            stage = 0;
            phase ^= 1;
          }
        }
      }
      if (*abort && leader)  // let every issued copy of the pair land before shared memory goes
        for (int s = 0; s < STAGES2; ++s)
          if (issued & (1u << s)) drain_wait(&bars->full[s], (last_parity >> s) & 1);
    }
  } else if (warp == 1) {
    if (leader && tc::elect_one()) {  // ---------------- UMMA issuer of the pair
      constexpr uint32_t IDESC = tc::idesc_f16(BF16, BM2, BN) | (B_MN ? (1u << 16) : 0u);
      int stage = 0, it = 0;
      uint32_t phase = 0;
      for (int unit = pair; unit < total && !*abort; unit += npairs, ++it) {
        int mb, nb, ks, kb0, kb1;
        decode_unit(p, unit, mb, nb, ks);
        k_range(p, ks, kb0, kb1);
        const int acc = it & 1;
        const uint32_t aphase = (it >> 1) & 1;
        if (!tc::mbar_wait_cluster(&bars->tempty[acc], aphase ^ 1, abort, p.status)) break;
        tc::fence_after_sync();
        const uint32_t d_tmem = tmem + acc * BN;
        bool ok = true;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!tc::mbar_wait(&bars->full[stage], phase, abort, p.status)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint32_t a0 = tc::smem_u32(smem + stage * SB);
          const uint32_t b0 = a0 + A_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            tc::umma2_f16(d_tmem, tc::sdesc_kmajor_sw128(a0 + k * 32),
                          B_MN ? tc::sdesc_mnmajor_sw128(b0 + k * 16 * 128, BK * 128, 1024)
                               : tc::sdesc_kmajor_sw128(b0 + k * 32),
                          IDESC, (kb > kb0 || k > 0) ? 1u : 0u);
          tc::umma2_commit_mc(&bars->empty[stage], 0x3);
          if (++stage == STAGES2) {
            stage = 0;
            phase ^= 1;
          }
        }
        if (!ok) break;
        tc::umma2_commit_mc(&bars->tfull[acc], 0x3);
      }
      tc::umma2_commit_mc(&bars->drain, 0x1);  // every UMMA of the pair has completed once this flips
      drain_wait(&bars->drain, 0);
    }
  } else {  // ---------------- epilogue warps 2..5 (both CTAs)
    const int q = warp & 3;
    const int row = q * 32 + lane;
    int it = 0;
    for (int unit = pair; unit < total && !*abort; unit += npairs, ++it) {
      int mb, nb, ks;
      decode_unit(p, unit, mb, nb, ks);
      const int acc = it & 1;
      const uint32_t aphase = (it >> 1) & 1;
      if (!tc::mbar_wait(&bars->tfull[acc], aphase, abort, p.status)) break;
      tc::fence_after_sync();
      const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + acc * BN;
      const int mb128 = 2 * mb + (int)rank;  // this CTA's 128-row block
      if (EPI == kEpiRope)
        epi_rope<BN>(p, &tmC, taddr, mb128, nb, row,  // rows past M are masked there
                 smem + STAGES2 * SB + q * 8192);
      else if ((int64_t)mb128 * BM < p.M) {  // M is a multiple of 128: whole halves are valid or not
        if (EPI == kEpiLsq)
          epi_lsq<BN>(p, taddr, mb128, nb, ks, row);
        else
          epi_store<BN>(p, taddr, mb128, nb, row);
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        if (leader)
          tc::mbar_arrive(&bars->tempty[acc]);
        else
          tc::mbar_arrive_cluster(tempty_lead + acc * 8);
      }
    }
    if (EPI == kEpiRope && tc::elect_one()) tc::bulk_wait_group<0>();  // the stores have read their boxes
  }
  tc::fence_before_sync();
  __syncthreads();
  // the pair's UMMAs have completed (the issuer drained) and no arrival is in flight to the other
  // CTA before either frees its tensor memory or exits
  tc::cluster_sync();
  tc::fence_after_sync();
  if (warp == 1) {
    __syncwarp();
    tc::tmem_dealloc2(tmem, 2 * BN);
  }
}

// ------------------------------------------------------------------ host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return (PFN_cuTensorMapEncodeTiled_v12000) nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  }();
  return fn;
}

// Row-major [outer, inner] 16-bit matrix with row pitch `pitch` elements; box = box_outer rows of
// 64 elements (128 B, the swizzle span).
bool make_tmap(CUtensorMap* m, const void* base, bool bf16, uint64_t inner, uint64_t outer,
               uint64_t pitch, uint32_t box_outer) {
  auto fn = encode_fn();
  if (fn == nullptr) return false;
  if ((reinterpret_cast<uintptr_t>(base) & 15u) || (pitch * 2) % 16) return false;
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {pitch * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, box_outer};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
            const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int sm_count() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

// Columns of a pair's tile. 256 is the better tile (a 128 one reads A and B from shared memory as often for
// half the products), but with few tiles a narrow one puts twice as many SMs to work, each with half the
// products and half the epilogue: taken when its rounds over the pairs, each reckoned 15 % dearer than half a
// round of wide tiles, take less. GPT-2 block, fitting step 4 x 128 (18 and 27 wide tiles on 76 pairs):
// 45.3 -> 40.3 us; a teacher pass of 16 x 1024 (576 wide tiles, 8 rounds against 16) keeps the wide tile.
int tile_cols(int num_m, int n, int splits) {
  const int64_t pairs = std::max(sm_count() / 2, 1), u = (int64_t)num_m * splits;
  const int64_t wide = (u * ((n + 255) / 256) + pairs - 1) / pairs, narrow = (u * ((n + 127) / 128) + pairs - 1) / pairs;
  return 0.575 * (double)narrow < (double)wide ? 128 : 256;
}

// CTA-pair launch: clusters of two, one pair per two SMs (as many pairs as fit at once).
template <int EPI, bool BF16, bool B_MN, int BN>
cudaError_t launch_gemm2(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& tcm,
                         GemmParams& p, cudaStream_t st) {
  auto kern = gemm2_tc_kernel<EPI, BF16, B_MN, BN>;
  p.num_n = (p.Nn + BN - 1) / BN;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM2_BYTES<BN>);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = SMEM2_BYTES<BN>;
  cfg.stream = st;
  const int sms = sm_count();
  // The pairs that fit at once depend only on the kernel and the device: asked once, so that a
  // launch makes no occupancy query (a launch-bound loop pays for every host call).
  static int clusters = 0;
  if (clusters < 1) {
    cfg.gridDim = dim3((unsigned)(sms / 2 * 2));
    if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess || clusters < 1)
      clusters = sms / 2;
  }
  const int64_t total = (int64_t)p.num_m * p.num_n * p.splits;
  const int pairs = (int)std::min<int64_t>(total, std::min(clusters, sms / 2));
  cfg.gridDim = dim3((unsigned)(2 * pairs));
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // stream_order() in the kernel
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, ta, tb, tcm, p);
}

}  // namespace

cudaError_t launch_proj_gemm_tc(const void* A, const void* Bw, void* C, int64_t M, int Nn, int K,
                                int D, int n_rot, int dh, int T, const float* cos_t,
                                const float* sin_t, int* status, cudaStream_t st) {
  CUtensorMap ta, tb, tcm;
  const int bn = tile_cols((int)((M + BM2 - 1) / BM2), Nn, 1);
  if (!make_tmap(&ta, A, false, K, M, K, BM) || !make_tmap(&tb, Bw, false, K, Nn, K, bn / 2) ||
      !make_tmap(&tcm, C, false, Nn, M, Nn, 32))
    return cudaErrorInvalidValue;
  GemmParams p{};
  p.M = M;
  p.Nn = Nn;
  p.K = K;
  p.num_m = (int)((M + BM2 - 1) / BM2);  // 256-row blocks: CTA pairs
  p.splits = 1;
  p.k_blocks = K / BK;
  p.group_m = 16;  // 16 pair rows = 4096 rows of X and all of W in L2 while the N tiles pass
  p.status = status;
  p.D = D;
  p.n_rot = n_rot;
  p.dh = dh;
  p.T = T;
  p.cos_t = cos_t;
  p.sin_t = sin_t;
  return bn == 128 ? launch_gemm2<kEpiRope, false, false, 128>(ta, tb, tcm, p, st)
                   : launch_gemm2<kEpiRope, false, false, 256>(ta, tb, tcm, p, st);
}

// Split K so that the units (tile x K range) fill whole waves of the persistent grid: the makespan
// in k-blocks is ceil(tiles * s / sms) * (k_blocks / s + kFill), kFill standing for a unit's pipeline
// fill and drain. (768 tiles on 152 SMs without a split leave 8 SMs a sixth full-K unit while the
// others idle.) Each unit keeps at least 16 k-blocks; near-ties go to fewer splits (fewer atomics
// and unit boundaries).
int choose_splits(int tiles, int k_blocks, int sms) {
  constexpr double kFill = 8.0;
  int splits = 1;
  double best = (double)((tiles + sms - 1) / sms) * ((double)k_blocks + kFill);
  for (int s = 2; s <= 32 && k_blocks / s >= 16; ++s) {
    const double t = (double)(((int64_t)tiles * s + sms - 1) / sms) * ((double)k_blocks / s + kFill);
    if (t < best * 0.995) {
      best = t;
      splits = s;
    }
  }
  return splits;
}

int lsq_group_parts(int G) {
  return 256 % G == 0 ? 1 : G % 256 == 0 ? G / 256 : (G - 1) / 256 + 2;
}

cudaError_t launch_wgrad_lsq_tc(const void* dqkvt, int64_t ldt, const void* x, const void* w,
                                const float* s, int64_t N, int D, int d, int G, int bits,
                                float coef, float* dspart, int* splits, int* status, cudaStream_t st) {
  CUtensorMap ta, tb;
  if (!make_tmap(&ta, dqkvt, true, N, D, ldt, BM) || !make_tmap(&tb, x, true, d, N, d, BK))
    return cudaErrorInvalidValue;
  GemmParams p{};
  p.M = D;
  p.Nn = d;
  p.K = (int)std::min<int64_t>(N, INT32_MAX);
  p.num_m = (D + BM2 - 1) / BM2;  // 256-row blocks: CTA pairs
  p.k_blocks = (int)((N + BK - 1) / BK);
  p.splits = choose_splits(p.num_m * ((d + 255) / 256), p.k_blocks, sm_count() / 2);
  p.group_m = 8;
  p.status = status;
  p.w = static_cast<const bf16_t*>(w);
  p.s = s;
  p.d = d;
  p.G = G;
  p.bits = bits;
  p.coef = coef;
  p.dspart = dspart;
  // every (split, part, row, group) partial is written once; they are summed in order by the caller's
  // last launch: the scale gradient is bit-identical between calls
  p.parts = lsq_group_parts(G);
  *splits = p.splits * p.parts;
  // a tile covers whole groups: the narrow one only those that divide it
  return 128 % G == 0 && tile_cols(p.num_m, d, p.splits) == 128 ? launch_gemm2<kEpiLsq, true, true, 128>(ta, tb, ta, p, st)
                                                                : launch_gemm2<kEpiLsq, true, true, 256>(ta, tb, ta, p, st);
}

cudaError_t launch_wgrad_store_tc(const void* dqkvt, int64_t ldt, const void* x, int64_t N, int D,
                                  int d, float coef, float* dw, double* sqnorm, float* scratch,
                                  double* red, bool deterministic, int* status, cudaStream_t st) {
  CUtensorMap ta, tb;
  if (!make_tmap(&ta, dqkvt, true, N, D, ldt, BM) || !make_tmap(&tb, x, true, d, N, d, BK))
    return cudaErrorInvalidValue;
  GemmParams p{};
  p.M = D;
  p.Nn = d;
  p.K = (int)std::min<int64_t>(N, INT32_MAX);
  p.num_m = (D + BM2 - 1) / BM2;  // 256-row blocks: CTA pairs
  p.k_blocks = (int)((N + BK - 1) / BK);
  p.group_m = 8;
  p.status = status;
  p.coef = coef;
  // dW goes to the caller's buffer, or to the scratch when only the norm is asked for. A split K
  // adds the partial tiles into a zeroed dW with atomics (the last bits depend on their order);
  // the deterministic mode keeps one unit per tile.
  const int64_t n_w = (int64_t)D * d;
  float* target = dw != nullptr ? dw : scratch;
  p.splits = deterministic ? 1 : choose_splits(p.num_m * ((d + 255) / 256), p.k_blocks, sm_count() / 2);
  p.dw = target;
  cudaError_t e;
  if (p.splits > 1) {
    e = cudaMemsetAsync(target, 0, (size_t)n_w * sizeof(float), st);
    if (e != cudaSuccess) return e;
  }
  e = tile_cols(p.num_m, d, p.splits) == 128 ? launch_gemm2<kEpiStore, true, true, 128>(ta, tb, ta, p, st)
                                             : launch_gemm2<kEpiStore, true, true, 256>(ta, tb, ta, p, st);
  if (e != cudaSuccess) return e;
  // a dW that the caller gets is checked, in the pass over it for its norm where there is one
  if (sqnorm != nullptr) return launch_sumsq(target, n_w, red, sqnorm, dw != nullptr ? status : nullptr, st);
  return launch_check_finite(target, n_w, status, st);
}

}  // namespace jab

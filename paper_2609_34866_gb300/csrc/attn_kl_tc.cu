// Tensor-core (tcgen05) KL attention-map term of L_JAB (Eq. 3, second term), sm_103a.
//
// For every query row i of every (candidate, sequence, query head), with the teacher's map P (float
// weights) and the student's map Q (quantised weights) over the causally visible keys j:
//
//     KL_i = sum_j P_ij (log P_ij - log Q_ij)
//          = sum_j P_ij (s^T_ij - s^S_ij) + lse^S_i - lse^T_i          (s = scaled scores)
//
// Persistent; a tile is 128 query rows of one (candidate, sequence, head), keys in blocks of 128. Both score
// blocks come from TS-form UMMAs whose A operand (the 128 query rows, teacher or student) was copied into
// tensor memory once:
//   S^S_j = Q^S K^S_j^T,  S^T_j = Q^T K^T_j^T            M128 N128 K = d_h
// The elementwise warps read the scores into registers at once and release them, so that the products of the
// next block, of the next tile too (Q is double-buffered in tensor memory), run under the exponentials of
// this one. Every thread keeps, for its 16 keys of two rows in each block, two online softmaxes of its own in
// the log2 domain (running maxima m, sums l, lazy rescaling when a maximum grows by more than 2^8) and
// a = sum_j p^T_j (s^T_j - s^S_j) with p^T_j = 2^(y^T_j - m^T), y = s log2(e) scale; the eight threads of a row
// (four lanes x two key halves) meet once a tile. The row result is formed from differences only,
//     KL_i / ln 2 = scale log2(e) a / l^T + (m^S - m^T) + log2(l^S / l^T),
// so no absolute log-sum-exp (of the size of the scores) is ever subtracted from another: the
// terms are of the size of the score perturbation and the KL, which is second order in it, keeps
// its relative precision.
//   warp 0       TMA: Q^S and Q^T of a tile, then K^S_j and K^T_j (ring)
//   warp 1       TMEM owner, tcgen05.cp of Q^S / Q^T, UMMA issuer (one thread)
//   warps 2..17  elementwise, 16 rows x 64 keys each (16x256b TMEM shape)
//   warp 18      row results of the tile before, from the states of its two key halves in shared memory
// Bound by the exponentials, 2 x 128 x 128 a block at 32 a clock and SM = 1024 clocks, next to 896 of packed
// fp32 work and 512 (d_h 64) of products; 16 x 12 heads of 777 x 64 with three candidates take 133 us,
// about 1700 clocks a block and 2700 a tile (one CTA a tile with eight elementwise warps: 227 us; with the rows'
// results in those warps, 4000 clocks more a tile: 173 us).
// Outputs: per-row KL (optional) and one fp64 partial per tile, summed in fixed order afterwards.
#include <cudaTypedefs.h>

#include <algorithm>

#include "kernels.h"
#include "tc.cuh"

namespace jab {
namespace {

constexpr int BQ = 128, BK = 128;
constexpr int EW_WARPS = 16;
constexpr int NUM_THREADS = (2 + EW_WARPS + 1) * 32;  // warp 0 TMA, warp 1 UMMA, warps 2..17 elementwise, 18 rows
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleLog2 = 8.f;
// Score of a hidden key: finite, so that the difference of two is 0. Products of fp16 rows stay below 2^40, so
// with the running maximum before the first visible key at no_key = -(2^41 sl2 + 2^10) every visible
// score is above it and a hidden one, times sl2, more than 2^10 below, for every sl2 from kMinSl2 on.
constexpr float kMasked = -3e38f;
constexpr float kMinSl2 = 1e-34f;

template <int DH>
struct KlLayout {
  static constexpr int TILE = 128 * DH * 2;  // 128 rows of fp16
  static constexpr int CHUNK = 128 * 128;    // 64 columns of a 128-row tile (128-byte swizzle)
  static constexpr int QS_OFF = 0, QT_OFF = TILE;
  static constexpr int K_OFF = 2 * TILE;     // stage st: K^S at K_OFF + 2 st TILE, K^T after it
  static constexpr int STAGES = DH == 64 ? 4 : 2;
  static constexpr int BAR_OFF = K_OFF + STAGES * 2 * TILE;
  static constexpr int USED = BAR_OFF + 12288;  // base alignment checked in the kernel
  static constexpr int SMEM = USED > 118 * 1024 ? USED : 118 * 1024;
  // tile parity t: Q^S at Q_COL + t DH, Q^T DH / 2 after it
  static constexpr uint32_t SS_COL = 0, ST_COL = 128, Q_COL = 256;
  static_assert(Q_COL + 2 * DH <= 512, "TMEM budget");
  static_assert(USED <= 227 * 1024, "shared memory budget");
};

// Running state of one row: maxima (log2 domain), sums of 2^(y - m) and a.
struct RowState {
  float mt, ms, lt, ls, a;
};

struct KlBars {
  uint64_t q_full, stg_free, k_full[4], k_empty[4], s_full, s_empty, st_full[2], st_free[2], drain;
  uint32_t tmem_base;
  int abort;
  RowState state[2][2][128];  // [tile parity][key half][row]
};
static_assert(sizeof(KlBars) <= 12288, "barrier block");

struct KlParams {
  int T, B, C, Hq, Hkv, D, nqb, nP, ntiles, balanced;
  FastDiv outer, by_ratio, by_hkv, by_b;  // by the tiles of one length (balanced) or of one group; Hq / Hkv; Hkv; B
  float sl2;           // softmax scale * log2(e)
  float no_key;        // running maximum before the first visible key (log2 units)
  double* part;        // [C, B, Hq, nP]  sum of KL_i over the tile's rows
  float* kl_rows;      // [C, B, Hq, T] or null
  int* status;
};

__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = tc::globaltimer();
  while (!tc::mbar_test(bar, parity))
    if (tc::globaltimer() - t0 > tc::kWaitLimitNs) break;
}

struct KlTile {
  int c, b, g, h, qb;  // candidate, sequence, KV head, query head, 128-row block (qb + 1 key blocks)
};
// Tile k: row blocks from the last (most keys) to the first, grouped by (candidate, sequence, KV head) so
// that the tiles which stream the K blocks of one KV head run close together (read from HBM about once);
// with `balanced` all tiles of a length come before the next shorter ones.
__device__ __forceinline__ KlTile kl_tile(const KlParams& p, int k) {
  KlTile t;
  int grp, hu, q, rem, bc;
  if (p.balanced) {
    p.outer.divmod(k, q, rem);
    p.by_ratio.divmod(rem, grp, hu);
  } else {
    p.outer.divmod(k, grp, rem);
    p.by_ratio.divmod(rem, q, hu);
  }
  t.qb = p.nqb - 1 - q;
  p.by_hkv.divmod(grp, bc, t.g);
  p.by_b.divmod(bc, t.c, t.b);
  t.h = t.g * p.by_ratio.d + hu;
  return t;
}

// Maximum of this thread's 16 scores of row A (x[4n + 0, 1]) and of row B (x[4n + 2, 3]).
__device__ __forceinline__ void thread_max(const float (&x)[32], float& ma, float& mb) {
  ma = fmaxf(x[0], x[1]);
  mb = fmaxf(x[2], x[3]);
#pragma unroll
  for (int n = 1; n < 8; ++n) {
    ma = tc::fmax3(ma, x[4 * n], x[4 * n + 1]);
    mb = tc::fmax3(mb, x[4 * n + 2], x[4 * n + 3]);
  }
}

// 2^d for an integer d <= 0, exactly (0 below the normal range).
__device__ __forceinline__ float exp2_int(float d) {
  return __int_as_float(((int)fmaxf(d, -127.f) + 127) << 23);
}

// Moves the running maxima to the block maxima (raw scores bt, bs) when they grow by more than 2^8,
// rescaling the sums accordingly. The maxima are whole numbers, so that every rescaling is exact, and the
// student's is the teacher's where they are near, so that log2(l^S / l^T) is near 0: a KL of 1e-5 is left
// of three terms, and factors rounded separately for student and teacher took 1 % of it.
__device__ __forceinline__ void advance_max(RowState& r, float bt, float bs, float sl2) {
  const float nt = ceilf(bt * sl2), ns = ceilf(bs * sl2);
  if (nt > r.mt + kRescaleLog2) {
    const float al = exp2_int(r.mt - nt);  // 0 for the first visible key
    r.lt *= al;
    r.a *= al;
    r.mt = nt;
  }
  if (ns > r.ms + kRescaleLog2) {
    const float m = fabsf(ns - r.mt) <= kRescaleLog2 && r.mt > r.ms ? r.mt : ns;
    r.ls *= exp2_int(r.ms - m);
    r.ms = m;
  }
}

// The state over both sets of keys. Its maxima are the larger ones, the factors powers of two.
__device__ __forceinline__ RowState merge(const RowState& x, const RowState& y) {
  RowState r;
  r.mt = fmaxf(x.mt, y.mt);
  r.ms = fmaxf(x.ms, y.ms);
  const float fx = exp2_int(x.mt - r.mt), fy = exp2_int(y.mt - r.mt);
  const float gx = exp2_int(x.ms - r.ms), gy = exp2_int(y.ms - r.ms);
  r.lt = x.lt * fx + y.lt * fy;
  r.a = x.a * fx + y.a * fy;
  r.ls = x.ls * gx + y.ls * gy;
  return r;
}
// The state over the keys of the four lanes of a row, in all of them: the maxima first, then one rescaling.
__device__ __forceinline__ void merge_lanes(RowState& r) {
  float mt = r.mt, ms = r.ms;
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1) {
    mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, o));
    ms = fmaxf(ms, __shfl_xor_sync(0xffffffffu, ms, o));
  }
  const float ft = exp2_int(r.mt - mt), fs = exp2_int(r.ms - ms);
  r.mt = mt;
  r.ms = ms;
  r.lt *= ft;
  r.a *= ft;
  r.ls *= fs;
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1) {
    r.lt += __shfl_xor_sync(0xffffffffu, r.lt, o);
    r.a += __shfl_xor_sync(0xffffffffu, r.a, o);
    r.ls += __shfl_xor_sync(0xffffffffu, r.ls, o);
  }
}

template <int DH>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    attn_kl_tc_kernel(const __grid_constant__ CUtensorMap tm_s,
                      const __grid_constant__ CUtensorMap tm_t, const KlParams p) {
  using L = KlLayout<DH>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  if (tc::smem_u32(smem_raw) & 1023u) {  // the swizzled TMA tiles need a 1024-byte aligned base
    if (threadIdx.x == 0) report(p.status, JAB_ERR_INTERNAL);
    return;
  }
  uint8_t* smem = smem_raw;
  KlBars* bars = reinterpret_cast<KlBars*>(smem + L::BAR_OFF);
  const int warp = tc::warp_index(), lane = threadIdx.x & 31;
  volatile int* abort = &bars->abort;

  if (threadIdx.x == 0) {
    tc::mbar_init(&bars->q_full, 1);
    tc::mbar_init(&bars->stg_free, 1);
    for (int i = 0; i < L::STAGES; ++i) {
      tc::mbar_init(&bars->k_full[i], 1);
      tc::mbar_init(&bars->k_empty[i], 1);
    }
    tc::mbar_init(&bars->s_full, 1);
    tc::mbar_init(&bars->s_empty, EW_WARPS);
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&bars->st_full[i], EW_WARPS);
      tc::mbar_init(&bars->st_free[i], 1);
    }
    tc::mbar_init(&bars->drain, 1);
    bars->abort = 0;
    tc::fence_mbar_init();
    tc::prefetch_tmap(&tm_s);
    tc::prefetch_tmap(&tm_t);
  }
  if (warp == 1) {
    tc::tmem_alloc(&bars->tmem_base, 512);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  stream_order();
  const int grid = gridDim.x, cta = blockIdx.x;

  if (warp == 0) {
    if (tc::elect_one()) {  // ---------------------------------------------------------------- TMA
      uint32_t g = 0, q_n = 0;  // K blocks and Q loads so far
      bool ok = true;
      // The student's tile at column cs and the teacher's at ct into dst and the tile after it.
      auto load_pair = [&](uint8_t* dst, uint64_t* bar, int cs, int ct, int row) {
        tc::mbar_expect_tx(bar, 2 * L::TILE);
        for (int ch = 0; ch < DH / 64; ++ch) {
          tc::tma_load_2d(dst + ch * L::CHUNK, &tm_s, bar, cs + ch * 64, row);
          tc::tma_load_2d(dst + L::TILE + ch * L::CHUNK, &tm_t, bar, ct + ch * 64, row);
        }
      };
      for (int it = 0, k = sched_tile(0, grid, cta); ok && k < p.ntiles; k = sched_tile(++it, grid, cta)) {
        const KlTile tl = kl_tile(p, k);
        const int row0 = tl.b * p.T, nkb = tl.qb + 1;
        if (it > 0 && !tc::mbar_wait(&bars->stg_free, (it - 1) & 1, abort, p.status)) break;
        load_pair(smem + L::QS_OFF, &bars->q_full, tl.c * p.D + tl.h * DH, tl.h * DH, row0 + tl.qb * BQ);
        ++q_n;
        const int kcol = (p.Hq + tl.g) * DH;
        for (int j = 0; j < nkb; ++j, ++g) {
          const uint32_t st = g % L::STAGES, ph = (g / L::STAGES) & 1;
          ok = tc::mbar_wait(&bars->k_empty[st], ph ^ 1, abort, p.status);
          if (!ok) break;
          load_pair(smem + L::K_OFF + st * 2 * L::TILE, &bars->k_full[st], tl.c * p.D + kcol, kcol, row0 + j * BK);
        }
      }
      if (*abort) {  // every copy issued lands before shared memory goes
        if (q_n > 0) drain_wait(&bars->q_full, (q_n - 1) & 1);
        for (uint32_t i = g > L::STAGES ? g - L::STAGES : 0; i < g; ++i)
          drain_wait(&bars->k_full[i % L::STAGES], (i / L::STAGES) & 1);
      }
    }
  } else if (warp == 1) {
    if (tc::elect_one()) {  // ---------------------------------------------------------------- UMMA
      constexpr uint32_t ID_S = tc::idesc_f16(false, BQ, BK);
      const uint32_t qs = tc::smem_u32(smem + L::QS_OFF), qt = tc::smem_u32(smem + L::QT_OFF);
      const uint64_t kd0 = tc::sdesc_kmajor_sw128(tc::smem_u32(smem + L::K_OFF));
      // Q of the CTA's tile `it` into its half of the tensor-memory columns, last read by the products of
      // tile it - 2; those were complete when the elementwise warps released a score block of tile it - 1.
      auto copy_q = [&](int it) {
        if (!tc::mbar_wait(&bars->q_full, it & 1, abort, p.status)) return false;
        tc::fence_after_sync();
        const uint32_t col = tmem + L::Q_COL + (it & 1) * DH;
#pragma unroll
        for (int kk = 0; kk < DH / 16; ++kk) {
          const uint32_t off = (kk >> 2) * L::CHUNK + (kk & 3) * 32;
          tc::tmem_cp_128x256b(col + kk * 8, tc::sdesc_kmajor_sw128(qs + off));
          tc::tmem_cp_128x256b(col + DH / 2 + kk * 8, tc::sdesc_kmajor_sw128(qt + off));
        }
        tc::umma_commit(&bars->stg_free);
        return true;
      };
      uint32_t g = 0;
      int it = 0, k = sched_tile(0, grid, cta);
      bool ok = k < p.ntiles && copy_q(0);
      while (ok && k < p.ntiles) {
        const int nkb = kl_tile(p, k).qb + 1;
        const uint32_t qc = tmem + L::Q_COL + (it & 1) * DH;
        for (int j = 0; j < nkb; ++j, ++g) {
          const uint32_t st = g % L::STAGES;
          if (!tc::mbar_wait(&bars->k_full[st], (g / L::STAGES) & 1, abort, p.status) ||
              !tc::mbar_wait(&bars->s_empty, (g & 1) ^ 1, abort, p.status)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint64_t kd_s = tc::sdesc_advance(kd0, st * 2 * L::TILE), kd_t = tc::sdesc_advance(kd_s, L::TILE);
#pragma unroll
          for (int kk = 0; kk < DH / 16; ++kk) {
            const uint32_t off = (kk >> 2) * L::CHUNK + (kk & 3) * 32;
            tc::umma_f16_ts(tmem + L::SS_COL, qc + kk * 8, tc::sdesc_advance(kd_s, off), ID_S, kk > 0 ? 1u : 0u);
            tc::umma_f16_ts(tmem + L::ST_COL, qc + DH / 2 + kk * 8, tc::sdesc_advance(kd_t, off), ID_S,
                            kk > 0 ? 1u : 0u);
          }
          tc::umma_commit(&bars->s_full);
          tc::umma_commit(&bars->k_empty[st]);
        }
        k = sched_tile(++it, grid, cta);
        if (ok && k < p.ntiles) ok = copy_q(it);
      }
      tc::umma_commit(&bars->drain);
      drain_wait(&bars->drain, 0);
    }
  } else if (warp < 2 + EW_WARPS) {  // -------------------------------------------- elementwise
    // Warp w (2..17) may access TMEM lane quarter w % 4; the four warps of a quarter take its two 16-row
    // groups x the block's two 64-key halves.
    const int quarter = warp & 3;
    const int idx = (warp - 2) >> 2;
    const int half = idx & 1, khalf = idx >> 1;
    const int grp = quarter * 2 + half;
    const int cq = lane & 3;
    const int rA = grp * 16 + (lane >> 2), rB = rA + 8;
    const uint32_t lane16 = (uint32_t)(grp * 16) << 16;
    const float2 sl2 = make_float2(p.sl2, p.sl2);
    uint32_t g = 0;
    bool ok = true;
    for (int it = 0, k = sched_tile(0, grid, cta); ok && k < p.ntiles; k = sched_tile(++it, grid, cta)) {
      const KlTile tl = kl_tile(p, k);
      const int q0 = tl.qb * BQ, nkb = tl.qb + 1;
      RowState ra{p.no_key, p.no_key, 0.f, 0.f, 0.f}, rb = ra;
      for (int j = 0; j < nkb; ++j, ++g) {
        if (!tc::mbar_wait(&bars->s_full, g & 1, abort, p.status)) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        // xs / xt[4n + e]: e < 2 row A, key 128 j + 64 khalf + 8n + 2 cq + e; e = 2, 3 row B.
        float xs[32], xt[32];
        {
          uint32_t r0[32], r1[32];
          __syncwarp();
          tc::tmem_ld_16x256b_x8(tmem + lane16 + L::ST_COL + 64 * khalf, r0);
          tc::tmem_ld_16x256b_x8(tmem + lane16 + L::SS_COL + 64 * khalf, r1);
          tc::tmem_ld_wait();
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&bars->s_empty);  // the next block's scores may overwrite
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            xt[i] = __uint_as_float(r0[i]);
            xs[i] = __uint_as_float(r1[i]);
          }
        }
        const bool masked = j == nkb - 1;  // the diagonal block (ragged or not)
        if (masked) {
          // rows past T have no result, so the causal mask alone hides the keys past T
          const int kl = j * BK + 64 * khalf - q0;  // first key of this warp, counted from the tile's first row
          if (kl > grp * 16 + 15) continue;         // no key of this half is visible to these 16 rows
          const uint32_t va = tc::columns_upto(rA - kl - 2 * cq), vb = tc::columns_upto(rB - kl - 2 * cq);
          // (a finite score: no weight either, and the difference of two is 0)
#pragma unroll
          for (int n = 0; n < 8; ++n)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int bit = 2 * n + e;
              xs[4 * n + e] = (va >> bit) & 1 ? xs[4 * n + e] : kMasked;
              xt[4 * n + e] = (va >> bit) & 1 ? xt[4 * n + e] : kMasked;
              xs[4 * n + 2 + e] = (vb >> bit) & 1 ? xs[4 * n + 2 + e] : kMasked;
              xt[4 * n + 2 + e] = (vb >> bit) & 1 ? xt[4 * n + 2 + e] : kMasked;
            }
        }
        float btA, btB, bsA, bsB;
        thread_max(xt, btA, btB);
        thread_max(xs, bsA, bsB);
        advance_max(ra, btA, bsA, p.sl2);
        advance_max(rb, btB, bsB, p.sl2);
        const float2 nmtA = make_float2(tc::neg_bits(ra.mt), tc::neg_bits(ra.mt));
        const float2 nmsA = make_float2(tc::neg_bits(ra.ms), tc::neg_bits(ra.ms));
        const float2 nmtB = make_float2(tc::neg_bits(rb.mt), tc::neg_bits(rb.mt));
        const float2 nmsB = make_float2(tc::neg_bits(rb.ms), tc::neg_bits(rb.ms));
        float2 ltA = make_float2(0.f, 0.f), lsA = ltA, aA = ltA, ltB = ltA, lsB = ltA, aB = ltA;
#pragma unroll
        for (int n = 0; n < 8; ++n) {
          const float2 tA2 = make_float2(xt[4 * n], xt[4 * n + 1]);
          const float2 sA2 = make_float2(xs[4 * n], xs[4 * n + 1]);
          const float2 tB2 = make_float2(xt[4 * n + 2], xt[4 * n + 3]);
          const float2 sB2 = make_float2(xs[4 * n + 2], xs[4 * n + 3]);
          const float2 etA = tc::fma2(tA2, sl2, nmtA), esA = tc::fma2(sA2, sl2, nmsA);
          const float2 etB = tc::fma2(tB2, sl2, nmtB), esB = tc::fma2(sB2, sl2, nmsB);
          const float2 ptA = make_float2(tc::fast_exp2(etA.x), tc::fast_exp2(etA.y));
          const float2 psA = make_float2(tc::fast_exp2(esA.x), tc::fast_exp2(esA.y));
          const float2 ptB = make_float2(tc::fast_exp2(etB.x), tc::fast_exp2(etB.y));
          const float2 psB = make_float2(tc::fast_exp2(esB.x), tc::fast_exp2(esB.y));
          const float2 dA = tc::sub2(tA2, sA2), dB = tc::sub2(tB2, sB2);
          ltA = tc::add2(ltA, ptA);
          lsA = tc::add2(lsA, psA);
          aA = tc::fma2(ptA, dA, aA);
          ltB = tc::add2(ltB, ptB);
          lsB = tc::add2(lsB, psB);
          aB = tc::fma2(ptB, dB, aB);
        }
        ra.lt += ltA.x + ltA.y;
        ra.ls += lsA.x + lsA.y;
        ra.a += aA.x + aA.y;
        rb.lt += ltB.x + ltB.y;
        rb.ls += lsB.x + lsB.y;
        rb.a += aB.x + aB.y;
      }
      if (!ok) break;
      // The four lanes of a row here; its two key halves and the row's result are left to the last warp, so
      // that these go on with the next tile (done by the lower half, 3k clocks a tile).
      merge_lanes(ra);
      merge_lanes(rb);
      const int pb = it & 1;
      ok = it < 2 || tc::mbar_wait(&bars->st_free[pb], ((it >> 1) - 1) & 1, abort, p.status);
      if (!ok) break;
      if (cq < 2) bars->state[pb][khalf][cq == 0 ? rA : rB] = cq == 0 ? ra : rb;
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bars->st_full[pb]);
    }
  } else {  // --------------------------------------------------------------------- row results
    for (int it = 0, k = sched_tile(0, grid, cta); k < p.ntiles; k = sched_tile(++it, grid, cta)) {
      const KlTile tl = kl_tile(p, k);
      const int pb = it & 1, q0 = tl.qb * BQ;
      if (!tc::mbar_wait(&bars->st_full[pb], (it >> 1) & 1, abort, p.status)) break;
      RowState r[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        r[i] = merge(bars->state[pb][0][32 * i + lane], bars->state[pb][1][32 * i + lane]);
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bars->st_free[pb]);
      float sum = 0.f, sum_lo = 0.f;  // KL over the tile's rows and the rounding of its additions
      const int64_t head = ((int64_t)tl.c * p.B + tl.b) * p.Hq + tl.h;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float kl =
            kLn2 * (p.sl2 * __fdiv_rn(r[i].a, r[i].lt) + (r[i].ms - r[i].mt) + log2f(__fdiv_rn(r[i].ls, r[i].lt)));
        const int t = q0 + 32 * i + lane;
        if (t < p.T) {
          pair_add(sum, sum_lo, kl, 0.f);
          if (p.kl_rows && in_bounds(head * p.T + t, (int64_t)p.C * p.B * p.Hq * p.T, p.status))
            p.kl_rows[head * p.T + t] = kl;
        }
      }
      warp_pair_sum(sum, sum_lo);
      const int64_t pi = head * p.nP + tl.qb;
      if (lane == 0 && in_bounds(pi, (int64_t)p.C * p.B * p.Hq * p.nP, p.status)) p.part[pi] = pair_value(sum, sum_lo);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 1) {
    __syncwarp();
    tc::tmem_dealloc(tmem, 512);
  }
}

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

// fp16 [rows, cols] row-major, 64 x 128 boxes with the 128-byte swizzle.
bool tmap_fp16(CUtensorMap* m, const void* base, uint64_t cols, uint64_t rows) {
  auto fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, 128};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int DH>
cudaError_t launch_kl(const CUtensorMap& ts, const CUtensorMap& tt, const KlParams& p, int sms,
                      cudaStream_t st) {
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(attn_kl_tc_kernel<DH>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         KlLayout<DH>::SMEM);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  return launch_after(attn_kl_tc_kernel<DH>, (unsigned)std::min(p.ntiles, sms), NUM_THREADS, KlLayout<DH>::SMEM, st,
                      ts, tt, p);
}

}  // namespace

int attn_kl_tc_rows() { return BQ; }

cudaError_t launch_attn_kl_tc(const void* qkv_s, int64_t ldq, const void* qkv_t, int B, int T,
                              int C, int Hq, int Hkv, int dh, float scale, double* part, int nP,
                              float* kl_rows, int* status, cudaStream_t st) {
  const int D = (Hq + 2 * Hkv) * dh;
  const int64_t N = (int64_t)B * T;
  CUtensorMap ts, tt;
  if (!tmap_fp16(&ts, qkv_s, (uint64_t)ldq, (uint64_t)N) ||
      !tmap_fp16(&tt, qkv_t, (uint64_t)D, (uint64_t)N))
    return cudaErrorInvalidValue;
  KlParams p{};
  p.T = T;
  p.B = B;
  p.C = C;
  p.Hq = Hq;
  p.Hkv = Hkv;
  p.D = D;
  p.nqb = (T + BQ - 1) / BQ;
  p.nP = nP;
  p.sl2 = std::max(scale * kLog2e, kMinSl2);  // (far above it already every map is uniform)
  p.no_key = -std::min(2199023255552.f * p.sl2 + 1024.f, 3e38f);
  p.part = part;
  p.kl_rows = kl_rows;
  p.status = status;
  if (p.nqb > nP) return cudaErrorInvalidValue;
  const int64_t ntiles = (int64_t)Hq * B * C * p.nqb;
  if (ntiles >= (1ll << 30)) return cudaErrorInvalidValue;
  p.ntiles = (int)ntiles;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms <= 0) sms = 1;
  // with few tiles per CTA their lengths decide the makespan, and all their K is in L2 anyway
  p.balanced = ntiles < 24 * (int64_t)sms;
  p.outer = FastDiv(p.balanced ? p.ntiles / p.nqb : Hq / Hkv * p.nqb);
  p.by_ratio = FastDiv(Hq / Hkv);
  p.by_hkv = FastDiv(Hkv);
  p.by_b = FastDiv(B);
  return dh == 128 ? launch_kl<128>(ts, tt, p, sms, st) : launch_kl<64>(ts, tt, p, sms, st);
}

}  // namespace jab

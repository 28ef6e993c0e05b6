// Tensor-core (tcgen05) forward-mode product of causal GQA attention, sm_103a: ||J_A v||^2 for the
// Hutchinson estimate of Tr(H) (Section 2.4, Eq. 5). At the float weights w* the Hessian of the MSE
// term is H = 2 J_A^T J_A / n, so a probe v gives v^T H v = 2 ||J_A v||^2 / n, and only the
// forward-mode derivative of the block output along v is needed, not a second backward pass.
//
// With the primal projections Q, K, V, the tangent projections dQ, dK, dV (the same projection and
// RoPE applied to the probe), S = scale Q K^T, P = softmax(S) and O = P V:
//     dS = scale (dQ K^T + Q dK^T)               (visible keys)
//     dO = (P o dS) V + P dV - rowsum(P o dS) O
// The teacher pass already has the row log-sum-exp and O (= A_ref), so P = exp(S - lse) is exact
// tile by tile and one pass over the keys suffices (no online rescaling).
//
// Persistent; a tile is 128 query rows of one (sequence, query head), keys in blocks of 128. Tensor
// memory: one score buffer X (columns 0 .. 127) that S = Q K^T and T = dQ K^T + Q dK^T use in turn, P and
// U = P o dS as packed fp16 (64 columns each), Z = U V + P dV (d_h), Q and dQ (d_h / 2 each, copied in by
// tcgen05.cp). All products are TS form. The elementwise warps read X out into registers at once:
//   S_j read -> T_j issued, while P_j is computed;   T_j read -> S_{j+1} issued, while U_j is
// A block takes about 4000 clocks, 2560 of them products: 529 us a probe for 8 x 32 heads of 2048 x 128, 73 %
// of the measured bf16 rate over all products. With S and T side by side and P and U written over them,
// S_{j+1} waited for Z_j, nothing overlapped and a block took 6570 clocks: 792 us (881 us before the issuing
// threads were elected). The rest is the chain S read -> P -> T read -> U of one tile, as tensor memory
// has no room for a second.
//   warp 0       TMA: ring of three slots that K_j and dK_j take in turn (K_j is read by S_j and T_j, dK_j
//                by T_j only), V/dV ring of two stages, through which a tile's Q and dQ come first. With two
//                K/dK stages and one V/dV slot, V_{j+1} was asked for only when Z_j was done: 594 us against 544
//   warp 1       TMEM owner, tcgen05.cp, issue of S and T;   warp 18  issue of Z (one thread each)
//   warps 2..17  elementwise, 16 rows x 64 keys each (16x256b TMEM shape), then the epilogue dO = Z - r O
//                with O read from A_ref, and its squared norm
// Output: one fp64 partial per tile, summed in fixed order afterwards.
#include <cudaTypedefs.h>

#include <algorithm>

#include "kernels.h"
#include "tc.cuh"

namespace jab {
namespace {

constexpr int BQ = 128, BK = 128;
constexpr int EW_WARPS = 16;
constexpr int NUM_THREADS = (2 + EW_WARPS + 1) * 32;
constexpr int Z_WARP = 2 + EW_WARPS;
constexpr float kLog2e = 1.4426950408889634f;

template <int DH>
struct JvpLayout {
  static constexpr int TILE = 128 * DH * 2;  // 128 rows of fp16
  static constexpr int CHUNK = 128 * 128;    // 64 columns of a 128-row tile (128-byte swizzle)
  static constexpr int KST = 3, VST = 2;
  static constexpr int VD_OFF = 0;                    // stage st: V at VD_OFF + 2 st TILE, dV after it
  static constexpr int KD_OFF = VST * 2 * TILE;       // slot u: K or dK
  static constexpr int BAR_OFF = KD_OFF + KST * TILE;
  static constexpr int USED = BAR_OFF + 2048;  // base alignment checked in the kernel
  static constexpr int SMEM = USED > 118 * 1024 ? USED : 118 * 1024;
  static constexpr uint32_t X_COL = 0, P_COL = 128, U_COL = 192, Z_COL = 256, Q_COL = 384, DQ_COL = 448;
  static_assert(Z_COL + DH <= Q_COL && Q_COL + DH / 2 <= DQ_COL && DQ_COL + DH / 2 <= 512, "TMEM budget");
  static_assert(USED <= 227 * 1024, "shared memory budget");
};

struct JvpBars {
  uint64_t q_full, stg_free, k_full[3], k_empty[3], vd_full[2], vd_empty[2], s_full, s_read, t_full;
  uint64_t t_read, pu_full, z_done, o_full, drain, drain_z;
  uint32_t tmem_base;
  int abort, fail[2];       // fail[tile parity]: an elementwise warp gave a wait up
  float2 red[2][EW_WARPS];  // [tile parity][warp]: sum of squares, high and low part
  float rsum[2][128];       // [key half][row] rowsum(P o dS)
};
static_assert(sizeof(JvpBars) <= 2048, "barrier block");

struct JvpParams {
  int T, B, Hq, Hkv, D, nqb, nP, lse_pitch, ntiles, balanced;
  FastDiv outer, by_ratio, by_hkv;  // by the tiles of one length (balanced) or of one group; by Hq / Hkv; by Hkv
  float scale, sl2;     // softmax scale; scale * log2(e)
  const float* lse;     // [B, Hq, lse_pitch] natural log (teacher)
  const float* a_ref;   // [B*T, Hq*DH] fp32: O of the teacher
  double* part;         // [B, Hq, nP]
  int* status;
};

__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = tc::globaltimer();
  while (!tc::mbar_test(bar, parity))
    if (tc::globaltimer() - t0 > tc::kWaitLimitNs) break;
}

struct JvpTile {
  int b, g, h, qb;  // sequence, KV head, query head, 128-row block (qb + 1 key blocks)
};
// Tile k: row blocks from the last (most keys) to the first, grouped by (sequence, KV head) so that the
// tiles which stream the blocks of one KV head run close together (read from HBM about once); with
// `balanced` all tiles of a length come before the next shorter ones.
__device__ __forceinline__ JvpTile jvp_tile(const JvpParams& p, int k) {
  JvpTile t;
  int grp, hu, q, rem;
  if (p.balanced) {
    p.outer.divmod(k, q, rem);
    p.by_ratio.divmod(rem, grp, hu);
  } else {
    p.outer.divmod(k, grp, rem);
    p.by_ratio.divmod(rem, q, hu);
  }
  t.qb = p.nqb - 1 - q;
  p.by_hkv.divmod(grp, t.b, t.g);
  t.h = t.g * p.by_ratio.d + hu;
  return t;
}

template <int DH>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    attn_jvp_tc_kernel(const __grid_constant__ CUtensorMap tm_p,
                       const __grid_constant__ CUtensorMap tm_t, const JvpParams p) {
  using L = JvpLayout<DH>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  if (tc::smem_u32(smem_raw) & 1023u) {  // the swizzled TMA tiles need a 1024-byte aligned base
    if (threadIdx.x == 0) report(p.status, JAB_ERR_INTERNAL);
    return;
  }
  uint8_t* smem = smem_raw;
  JvpBars* bars = reinterpret_cast<JvpBars*>(smem + L::BAR_OFF);
  const int warp = tc::warp_index(), lane = threadIdx.x & 31;
  volatile int* abort = &bars->abort;

  if (threadIdx.x == 0) {
    tc::mbar_init(&bars->q_full, 1);
    tc::mbar_init(&bars->stg_free, 1);
    for (int i = 0; i < L::KST; ++i) {
      tc::mbar_init(&bars->k_full[i], 1);
      tc::mbar_init(&bars->k_empty[i], 1);
    }
    for (int i = 0; i < L::VST; ++i) {
      tc::mbar_init(&bars->vd_full[i], 1);
      tc::mbar_init(&bars->vd_empty[i], 1);
    }
    tc::mbar_init(&bars->s_full, 1);
    tc::mbar_init(&bars->s_read, EW_WARPS);
    tc::mbar_init(&bars->t_full, 1);
    tc::mbar_init(&bars->t_read, EW_WARPS);
    tc::mbar_init(&bars->pu_full, EW_WARPS);
    tc::mbar_init(&bars->z_done, 1);
    tc::mbar_init(&bars->o_full, 1);
    tc::mbar_init(&bars->drain, 1);
    tc::mbar_init(&bars->drain_z, 1);
    bars->abort = bars->fail[0] = bars->fail[1] = 0;
    tc::fence_mbar_init();
    tc::prefetch_tmap(&tm_p);
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
    if (tc::elect_one()) {  // -------------------------------------------------------------- TMA
      uint32_t g = 0, u = 0, q_n = 0, v_n = 0;  // blocks, K / dK slots, Q loads and V loads so far
      bool ok = true;
      // K (tangent = false) or dK of a block into the ring's next slot.
      auto load_k = [&](bool tangent, int col, int row) {
        const uint32_t sl = u % L::KST, ph = (u / L::KST) & 1;
        if (!tc::mbar_wait(&bars->k_empty[sl], ph ^ 1, abort, p.status)) return false;
        tc::mbar_expect_tx(&bars->k_full[sl], L::TILE);
        for (int ch = 0; ch < DH / 64; ++ch)
          tc::tma_load_2d(smem + L::KD_OFF + sl * L::TILE + ch * L::CHUNK, tangent ? &tm_t : &tm_p,
                          &bars->k_full[sl], col + ch * 64, row);
        ++u;
        return true;
      };
      // Primal and tangent tiles into a V/dV stage.
      auto load_pair = [&](uint32_t st, uint64_t* bar, int col, int row) {
        uint8_t* dst = smem + L::VD_OFF + st * 2 * L::TILE;
        tc::mbar_expect_tx(bar, 2 * L::TILE);
        for (int ch = 0; ch < DH / 64; ++ch) {
          tc::tma_load_2d(dst + ch * L::CHUNK, &tm_p, bar, col + ch * 64, row);
          tc::tma_load_2d(dst + L::TILE + ch * L::CHUNK, &tm_t, bar, col + ch * 64, row);
        }
      };
      for (int it = 0, k = sched_tile(0, grid, cta); ok && k < p.ntiles; k = sched_tile(++it, grid, cta)) {
        const JvpTile tl = jvp_tile(p, k);
        const int row0 = tl.b * p.T, nkb = tl.qb + 1;
        const int qcol = tl.h * DH, kcol = (p.Hq + tl.g) * DH, vcol = (p.Hq + p.Hkv + tl.g) * DH;
        for (int j = 0; ok && j < nkb; ++j, ++g) {
          const uint32_t st = g & 1;
          ok = load_k(false, kcol, row0 + j * BK);
          if (j > 0) ok = ok && load_k(true, kcol, row0 + j * BK);
          ok = ok && tc::mbar_wait(&bars->vd_empty[st], ((g >> 1) & 1) ^ 1, abort, p.status);
          if (!ok) break;
          if (j == 0) {  // Q and dQ through the stage first
            load_pair(st, &bars->q_full, qcol, row0 + tl.qb * BQ);
            ++q_n;
            ok = load_k(true, kcol, row0) && tc::mbar_wait(&bars->stg_free, it & 1, abort, p.status);
            if (!ok) break;
          }
          load_pair(st, &bars->vd_full[st], vcol, row0 + j * BK);
          ++v_n;
        }
      }
      if (*abort) {  // every copy issued lands before shared memory goes
        if (q_n > 0) drain_wait(&bars->q_full, (q_n - 1) & 1);
        for (uint32_t i = u > L::KST ? u - L::KST : 0; i < u; ++i)
          drain_wait(&bars->k_full[i % L::KST], (i / L::KST) & 1);
        for (uint32_t i = v_n > 2 ? v_n - 2 : 0; i < v_n; ++i) drain_wait(&bars->vd_full[i & 1], (i >> 1) & 1);
      }
    }
  } else if (warp == 1) {
    if (tc::elect_one()) {  // ------------------------------------------------------- UMMA: S, T
      constexpr uint32_t ID_S = tc::idesc_f16(false, BQ, BK);
      const uint32_t vd_base = tc::smem_u32(smem + L::VD_OFF);
      const uint64_t kd0 = tc::sdesc_kmajor_sw128(tc::smem_u32(smem + L::KD_OFF));
      uint32_t g = 0;
      bool ok = true;
      for (int it = 0, k = sched_tile(0, grid, cta); ok && k < p.ntiles; k = sched_tile(++it, grid, cta)) {
        const int nkb = jvp_tile(p, k).qb + 1;
        // Q and dQ into tensor memory, once the previous tile's last T, which reads the old ones, is done
        if (!tc::mbar_wait(&bars->q_full, it & 1, abort, p.status) ||
            (g > 0 && !tc::mbar_wait(&bars->t_full, (g - 1) & 1, abort, p.status)))
          break;
        tc::fence_after_sync();
        const uint32_t qs = vd_base + (g & 1) * 2 * L::TILE, dqs = qs + L::TILE;
#pragma unroll
        for (int kk = 0; kk < DH / 16; ++kk) {
          const uint32_t off = (kk >> 2) * L::CHUNK + (kk & 3) * 32;
          tc::tmem_cp_128x256b(tmem + L::Q_COL + kk * 8, tc::sdesc_kmajor_sw128(qs + off));
          tc::tmem_cp_128x256b(tmem + L::DQ_COL + kk * 8, tc::sdesc_kmajor_sw128(dqs + off));
        }
        tc::umma_commit(&bars->stg_free);  // the slot may take V / dV of the tile's first block
        for (int j = 0; j < nkb; ++j, ++g) {
          const uint32_t u0 = 2 * g, u1 = u0 + 1, sl0 = u0 % L::KST, sl1 = u1 % L::KST;
          // S_j once K_j has landed and T_{j-1} has been read out of X
          if (!tc::mbar_wait(&bars->k_full[sl0], (u0 / L::KST) & 1, abort, p.status) ||
              (g > 0 && !tc::mbar_wait(&bars->t_read, (g - 1) & 1, abort, p.status))) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint64_t kd = tc::sdesc_advance(kd0, sl0 * L::TILE);
          const uint64_t dkd = tc::sdesc_advance(kd0, sl1 * L::TILE);
#pragma unroll
          for (int kk = 0; kk < DH / 16; ++kk)
            tc::umma_f16_ts(tmem + L::X_COL, tmem + L::Q_COL + kk * 8,
                            tc::sdesc_advance(kd, (kk >> 2) * L::CHUNK + (kk & 3) * 32), ID_S,
                            kk > 0 ? 1u : 0u);
          tc::umma_commit(&bars->s_full);
          // T_j once S_j has been read out and dK_j has landed
          if (!tc::mbar_wait(&bars->k_full[sl1], (u1 / L::KST) & 1, abort, p.status) ||
              !tc::mbar_wait(&bars->s_read, g & 1, abort, p.status)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
#pragma unroll
          for (int kk = 0; kk < DH / 16; ++kk)
            tc::umma_f16_ts(tmem + L::X_COL, tmem + L::DQ_COL + kk * 8,
                            tc::sdesc_advance(kd, (kk >> 2) * L::CHUNK + (kk & 3) * 32), ID_S,
                            kk > 0 ? 1u : 0u);
#pragma unroll
          for (int kk = 0; kk < DH / 16; ++kk)
            tc::umma_f16_ts(tmem + L::X_COL, tmem + L::Q_COL + kk * 8,
                            tc::sdesc_advance(dkd, (kk >> 2) * L::CHUNK + (kk & 3) * 32), ID_S, 1u);
          tc::umma_commit(&bars->t_full);
          tc::umma_commit(&bars->k_empty[sl0]);
          tc::umma_commit(&bars->k_empty[sl1]);
        }
      }
      tc::umma_commit(&bars->drain);
      drain_wait(&bars->drain, 0);
    }
  } else if (warp == Z_WARP) {
    if (tc::elect_one()) {  // ---------------------------------------------------------- UMMA: Z
      constexpr uint32_t ID_Z = tc::idesc_f16(false, BQ, DH) | (1u << 16);  // B = V / dV, MN-major
      const uint64_t vd0 = tc::sdesc_mnmajor_sw128(tc::smem_u32(smem + L::VD_OFF), L::CHUNK, 1024);
      uint32_t g = 0;
      bool ok = true;
      for (int it = 0, k = sched_tile(0, grid, cta); ok && k < p.ntiles; k = sched_tile(++it, grid, cta)) {
        const int nkb = jvp_tile(p, k).qb + 1;
        for (int j = 0; j < nkb; ++j, ++g) {
          // Z += U_j V_j + P_j dV_j (a tile's first one comes after the elementwise warps' epilogue of the
          // previous tile, which precedes their P)
          const uint32_t st = g & 1;
          if (!tc::mbar_wait(&bars->vd_full[st], (g >> 1) & 1, abort, p.status) ||
              !tc::mbar_wait(&bars->pu_full, g & 1, abort, p.status)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint64_t vd = tc::sdesc_advance(vd0, st * 2 * L::TILE);
          const uint64_t dvd = tc::sdesc_advance(vd, L::TILE);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            tc::umma_f16_ts(tmem + L::Z_COL, tmem + L::U_COL + kk * 8,
                            tc::sdesc_advance(vd, kk * 16 * 128), ID_Z, (j > 0 || kk > 0) ? 1u : 0u);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            tc::umma_f16_ts(tmem + L::Z_COL, tmem + L::P_COL + kk * 8,
                            tc::sdesc_advance(dvd, kk * 16 * 128), ID_Z, 1u);
          tc::umma_commit(&bars->z_done);
          tc::umma_commit(&bars->vd_empty[st]);
          if (j == nkb - 1) tc::umma_commit(&bars->o_full);
        }
      }
      tc::umma_commit(&bars->drain_z);
      drain_wait(&bars->drain_z, 0);
    }
  } else {  // -------------------------------------------------------------------- elementwise
    // Warp w (2..17) may access TMEM lane quarter w % 4; the four warps of a quarter take its two 16-row
    // groups x the block's two 64-key halves.
    const int quarter = warp & 3;
    const int idx = (warp - 2) >> 2;
    const int half = idx & 1, chalf = idx >> 1;
    const int cq = lane & 3;
    const int rA = quarter * 32 + half * 16 + (lane >> 2), rB = rA + 8;
    const uint32_t lane16 = (uint32_t)(quarter * 32 + half * 16) << 16;
    const float2 sl2 = make_float2(p.sl2, p.sl2), sc = make_float2(p.scale, p.scale);
    uint32_t g = 0, range_bits = 0;
    float lA = INFINITY, lB = INFINITY;  // row log-sum-exp; rows past T: P = 0 (+inf)
    auto load_lse = [&](const JvpTile& t) {
      const int a = t.qb * BQ + rA, b = a + 8;
      const float* l = p.lse + ((int64_t)t.b * p.Hq + t.h) * p.lse_pitch;
      lA = a < p.T ? l[a] : INFINITY;
      lB = b < p.T ? l[b] : INFINITY;
    };
    const int k_first = sched_tile(0, grid, cta);
    JvpTile tl = jvp_tile(p, k_first < p.ntiles ? k_first : 0);
    load_lse(tl);
    for (int it = 0, k = sched_tile(0, grid, cta); k < p.ntiles; k = sched_tile(++it, grid, cta)) {
      const int q0 = tl.qb * BQ, nkb = tl.qb + 1, row0 = tl.b * p.T;
      const int tA = q0 + rA, tB = q0 + rB;
      const float2 nlA = make_float2(tc::neg_bits(lA * kLog2e), tc::neg_bits(lA * kLog2e));
      const float2 nlB = make_float2(tc::neg_bits(lB * kLog2e), tc::neg_bits(lB * kLog2e));
      // The rows of O that the epilogue reads, DH / 2 columns of 16 rows, into L2 (its loads otherwise
      // waited for HBM, 11k clocks a tile against 3k).
      constexpr int W = DH / 2;  // columns of this warp
      const int64_t pitch = (int64_t)p.Hq * DH;
      const float* o_rows = p.a_ref + (int64_t)row0 * pitch + tl.h * DH + W * chalf;
      {
        const int t = q0 + rA - (lane >> 2) + (lane & 15);
        if (t < p.T && (lane >> 4) * 32 < W) tc::prefetch_line_l2(o_rows + t * pitch + (lane >> 4) * 32);
      }
      float rsA = 0.f, rsB = 0.f;  // this thread's share of rowsum(P o dS)
      bool ok = true;
      for (int j = 0; j < nkb; ++j, ++g) {
        if (!tc::mbar_wait(&bars->s_full, g & 1, abort, p.status)) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        // x[4n + e]: e < 2 row A, key 128 j + 64 chalf + 8n + 2 cq + e; e = 2, 3 row B
        float x[32];
        {
          uint32_t r0[32];
          __syncwarp();
          tc::tmem_ld_16x256b_x8(tmem + lane16 + L::X_COL + 64 * chalf, r0);
          tc::tmem_ld_wait();
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&bars->s_read);  // T_j may overwrite X
#pragma unroll
          for (int c = 0; c < 32; ++c) x[c] = __uint_as_float(r0[c]);
        }
        const int k0 = j * BK + 64 * chalf + 2 * cq;
        const bool masked = j == nkb - 1;  // the diagonal block (ragged or not)
        uint32_t pw[16];  // packed: pw[2n] row A, pw[2n + 1] row B, packed column 32 chalf + 4n + cq
#pragma unroll
        for (int n = 0; n < 8; ++n) {
          const float2 ea = tc::fma2(make_float2(x[4 * n], x[4 * n + 1]), sl2, nlA);
          const float2 eb = tc::fma2(make_float2(x[4 * n + 2], x[4 * n + 3]), sl2, nlB);
          float2 pa = make_float2(tc::fast_exp2(ea.x), tc::fast_exp2(ea.y));
          float2 pb = make_float2(tc::fast_exp2(eb.x), tc::fast_exp2(eb.y));
          if (masked) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int key = k0 + 8 * n + e;
              if (key > tA || key >= p.T) (e ? pa.y : pa.x) = 0.f;
              if (key > tB || key >= p.T) (e ? pb.y : pb.x) = 0.f;
            }
          }
          x[4 * n] = pa.x;
          x[4 * n + 1] = pa.y;
          x[4 * n + 2] = pb.x;
          x[4 * n + 3] = pb.y;
          pw[2 * n] = tc::pack_half2(pa.x, pa.y);
          pw[2 * n + 1] = tc::pack_half2(pb.x, pb.y);
        }
        // Z_{j-1} has read P_{j-1} and U_{j-1}
        if (g > 0 && !tc::mbar_wait(&bars->z_done, (g - 1) & 1, abort, p.status)) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        __syncwarp();
        tc::tmem_st_16x128b_x8(tmem + lane16 + L::P_COL + 32 * chalf, pw);
        if (!tc::mbar_wait(&bars->t_full, g & 1, abort, p.status)) {
          tc::tmem_st_wait();
          ok = false;
          break;
        }
        tc::fence_after_sync();
        uint32_t rt[32];
        __syncwarp();
        tc::tmem_ld_16x256b_x8(tmem + lane16 + L::X_COL + 64 * chalf, rt);
        tc::tmem_ld_wait();
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bars->t_read);  // S_{j+1} may overwrite X
        float2 uA = make_float2(0.f, 0.f), uB = uA;
        uint32_t uw[16];
#pragma unroll
        for (int n = 0; n < 8; ++n) {
          const float2 ta = make_float2(__uint_as_float(rt[4 * n]), __uint_as_float(rt[4 * n + 1]));
          const float2 tb = make_float2(__uint_as_float(rt[4 * n + 2]), __uint_as_float(rt[4 * n + 3]));
          const float2 ua = tc::mul2(make_float2(x[4 * n], x[4 * n + 1]), tc::mul2(ta, sc));
          const float2 ub = tc::mul2(make_float2(x[4 * n + 2], x[4 * n + 3]), tc::mul2(tb, sc));
          uA = tc::add2(uA, ua);
          uB = tc::add2(uB, ub);
          uw[2 * n] = tc::pack_half2(ua.x, ua.y);
          uw[2 * n + 1] = tc::pack_half2(ub.x, ub.y);
          range_bits = max_abs_f16x2(max_abs_f16x2(range_bits, uw[2 * n]), uw[2 * n + 1]);
        }
        __syncwarp();
        tc::tmem_st_16x128b_x8(tmem + lane16 + L::U_COL + 32 * chalf, uw);
        tc::tmem_st_wait();
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bars->pu_full);
        rsA += uA.x + uA.y;
        rsB += uB.x + uB.y;
      }
      const int64_t part_at = ((int64_t)tl.b * p.Hq + tl.h) * p.nP + tl.qb;
      {  // on to the next tile, its log-sum-exp loaded while the epilogue runs
        const int kn = sched_tile(it + 1, grid, cta);
        if (kn < p.ntiles) {
          tl = jvp_tile(p, kn);
          load_lse(tl);
        }
      }
      // ---------------------------------------------------------------- epilogue: dO = Z - r O
      float sq = 0.f, sq_lo = 0.f;  // this thread's squares and the rounding of their additions
      rsA += __shfl_xor_sync(0xffffffffu, rsA, 1);
      rsB += __shfl_xor_sync(0xffffffffu, rsB, 1);
      rsA += __shfl_xor_sync(0xffffffffu, rsA, 2);
      rsB += __shfl_xor_sync(0xffffffffu, rsB, 2);
      if (cq == 0) {
        bars->rsum[chalf][rA] = rsA;
        bars->rsum[chalf][rB] = rsB;
      }
      // the two key halves of these 16 rows: warps of the same quarter and half
      tc::named_bar_sync(2 + quarter * 2 + half, 64);
      const float* oA = o_rows + (tA < p.T ? tA : 0) * pitch;
      const float* oB = o_rows + (tB < p.T ? tB : 0) * pitch;
      float2 a[4], bb[4];
      auto load_o = [&](int c) {
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          a[n] = __ldg(reinterpret_cast<const float2*>(oA + 32 * c + 8 * n + 2 * cq));
          bb[n] = __ldg(reinterpret_cast<const float2*>(oB + 32 * c + 8 * n + 2 * cq));
        }
      };
      load_o(0);  // ahead of the waits
      const float nra = tc::neg_bits(bars->rsum[0][rA] + bars->rsum[1][rA]);
      const float nrb = tc::neg_bits(bars->rsum[0][rB] + bars->rsum[1][rB]);
      if (ok && tc::mbar_wait(&bars->o_full, it & 1, abort, p.status)) {
        tc::fence_after_sync();
        float2 qA = make_float2(0.f, 0.f), qB = qA;
        const float2 nrA = make_float2(nra, nra), nrB = make_float2(nrb, nrb);
#pragma unroll 1
        for (int c = 0; c < W / 32; ++c) {
          uint32_t z[16];
          __syncwarp();
          tc::tmem_ld_16x256b_x4(tmem + lane16 + L::Z_COL + W * chalf + 32 * c, z);
          tc::tmem_ld_wait();
#pragma unroll
          for (int n = 0; n < 4; ++n) {
            const float2 dA = tc::fma2(nrA, a[n], make_float2(__uint_as_float(z[4 * n]), __uint_as_float(z[4 * n + 1])));
            const float2 dB = tc::fma2(nrB, bb[n], make_float2(__uint_as_float(z[4 * n + 2]), __uint_as_float(z[4 * n + 3])));
            qA = tc::fma2(dA, dA, qA);
            qB = tc::fma2(dB, dB, qB);
          }
          if (c + 1 < W / 32) load_o(c + 1);
        }
        tc::fence_before_sync();  // Z is read out before this warp's next arrival on pu_full
        // Sums as pairs of floats with the additions' rounding carried along, and fp64 only for the 16
        // warps' totals: an fp64 addition in every thread of every warp took 3k clocks a tile.
        if (tA < p.T) {
          two_sum(qA.x, qA.y, sq, sq_lo);
        }
        if (tB < p.T) {
          pair_add(sq, sq_lo, qB.x, 0.f);
          pair_add(sq, sq_lo, qB.y, 0.f);
        }
      } else {
        ok = false;
      }
      warp_pair_sum(sq, sq_lo);
      float2* red = bars->red[it & 1];
      if (lane == 0) red[warp - 2] = make_float2(sq, sq_lo);
      // All elementwise warps leave after the same tile: one that stayed would wait on the next tile's barriers.
      if (!ok) reinterpret_cast<volatile int*>(bars->fail)[it & 1] = 1;
      tc::named_bar_sync(1, EW_WARPS * 32);  // every elementwise warp reaches this once per tile
      if (warp == 2 && ok) {
        const float2 r = red[lane & (EW_WARPS - 1)];
        double tot = (double)r.x + (double)r.y;
#pragma unroll
        for (int o = EW_WARPS / 2; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
        if (lane == 0 && in_bounds(part_at, (int64_t)p.B * p.Hq * p.nP, p.status)) p.part[part_at] = tot;
      }
      if (reinterpret_cast<volatile int*>(bars->fail)[it & 1]) break;
    }
    if (either_at_least(range_bits, kHalfInf)) report(p.status, JAB_ERR_RANGE);  // U out of the fp16 range
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
cudaError_t launch_jvp(const CUtensorMap& tp, const CUtensorMap& tt, const JvpParams& p, int sms,
                       cudaStream_t st) {
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(attn_jvp_tc_kernel<DH>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         JvpLayout<DH>::SMEM);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  return launch_after(attn_jvp_tc_kernel<DH>, (unsigned)std::min(p.ntiles, sms), NUM_THREADS, JvpLayout<DH>::SMEM, st,
                      tp, tt, p);
}

}  // namespace

int attn_jvp_tc_rows() { return BQ; }

cudaError_t launch_attn_jvp_tc(const void* qkv, const void* tqkv, const float* lse, int lse_pitch,
                               const float* a_ref, int B, int T, int Hq, int Hkv, int dh,
                               float scale, double* part, int nP, int* status, cudaStream_t st) {
  const int D = (Hq + 2 * Hkv) * dh;
  const int64_t N = (int64_t)B * T;
  CUtensorMap tp, tt;
  if (!tmap_fp16(&tp, qkv, (uint64_t)D, (uint64_t)N) || !tmap_fp16(&tt, tqkv, (uint64_t)D, (uint64_t)N))
    return cudaErrorInvalidValue;
  JvpParams p{};
  p.T = T;
  p.B = B;
  p.Hq = Hq;
  p.Hkv = Hkv;
  p.D = D;
  p.nqb = (T + BQ - 1) / BQ;
  p.nP = nP;
  p.lse_pitch = lse_pitch;
  p.scale = scale;
  p.sl2 = scale * kLog2e;
  p.lse = lse;
  p.a_ref = a_ref;
  p.part = part;
  p.status = status;
  if (p.nqb > nP) return cudaErrorInvalidValue;
  const int64_t ntiles = (int64_t)Hq * B * p.nqb;
  if (ntiles >= (1ll << 30)) return cudaErrorInvalidValue;
  p.ntiles = (int)ntiles;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms <= 0) sms = 1;
  // with few tiles per CTA their lengths decide the makespan, and all their K and V are in L2 anyway
  p.balanced = ntiles < 24 * (int64_t)sms;
  p.outer = FastDiv(p.balanced ? p.ntiles / p.nqb : Hq / Hkv * p.nqb);
  p.by_ratio = FastDiv(Hq / Hkv);
  p.by_hkv = FastDiv(Hkv);
  return dh == 128 ? launch_jvp<128>(tp, tt, p, sms, st) : launch_jvp<64>(tp, tt, p, sms, st);
}

}  // namespace jab

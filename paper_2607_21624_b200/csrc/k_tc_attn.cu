// Fused attention on tcgen05 tensor cores, operands in R-Tile order fetched by TMA.
//
// Forward: one block per (128-query tile, head, batch).  S = Q K^T goes to TMEM (two buffers, so the
// tensor pipe computes the next score tile while the softmax warps work on the current one); the
// softmax warps own one query row per thread, keep the running max / sum, and hand P (bf16) to the
// tensor pipe in tensor memory, over the score columns it was computed from; O accumulates in TMEM and is
// rescaled in place only when a row's running max moved.  K/V tiles of the group's KV head are addressed by the head map
// g = h / G; the head split of Q, K, V and the merge of O are column-panel coordinates of the TMA
// boxes and of the output rows, no data is rearranged.
#include <string.h>

#include <type_traits>

#include "attn_common.cuh"
#include "fbl_internal.h"
#include "launch_memo.h"
#include "pdl.cuh"
#include "tc_common.cuh"

namespace {

constexpr int BQ = 128, BKV = 128;
constexpr float LOG2E = 1.4426950408889634f;

struct alignas(64) AttnFwdParams {
  CUtensorMap tq, tk, tv;
  __nv_bfloat16* a;      // merged-head output [n_pad, dq] in R-Tile order
  float* lse;            // [B, Hq, t_pad]
  long long n_pad;
  int seq, t_pad, hq, group, causal;
  int seq_k, t_pad_k;    // key-side sequence length and padded length (those of the query side in self-attention)
  int pair;              // 1: each block owns two adjacent query tiles, one per softmax warp group
  int batch, n_slots, chunk;   // grid = n_slots * hq * batch blocks, see decode_block
  float scale;
  int32_t* status;
};

// Two values as packed bf16, and what the rounding leaves of them likewise.
__device__ __forceinline__ void split_bf16(float x, float y, uint32_t& hi, uint32_t& lo) {
  hi = tc::pack_bf16(x, y);
  lo = tc::pack_bf16(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
}

template <int HD, int TILES>
struct FwdSmem {
  static constexpr uint32_t PANELS = HD / 64;
  static constexpr uint32_t TILE = PANELS * 16384;          // 128 rows x HD bf16
  static constexpr uint32_t Q_OFF = 0;                      // TILES query tiles
  static constexpr uint32_t K_OFF = TILES * TILE;           // 2 stages
  static constexpr uint32_t V_OFF = (TILES + 2) * TILE;     // 2 stages
  static constexpr uint32_t BAR_OFF = (TILES + 4) * TILE;
  static constexpr uint32_t N_BARS = 18;
  static constexpr uint32_t TOTAL = BAR_OFF + 8 * N_BARS + 16;
};

enum { B_QFULL = 0, B_KFULL = 1, B_KEMPTY = 3, B_VFULL = 5, B_VEMPTY = 7, B_SFULL = 9, B_PFULL = 12, B_PVDONE = 15 };   // SFULL, PFULL: one per score buffer (up to 3)

// warp 0 TMA, warp 1 MMA, then one softmax warp group (4 warps) per query tile of the block.  TILES = 2: two
// adjacent query tiles share the K/V tiles, one block per SM.  TILES = 1 (head_dim 64 only: its tiles leave room): a
// block of 192 threads with one query tile, half the tensor memory and at most 128 registers per thread, so that two
// blocks share an SM and one's set-up and epilogue overlap the other's key loop (short sequences are mostly that).

// A row's running max is only raised (and O rescaled) when the new max exceeds it by more than this many
// powers of two; until then the probabilities are computed against the stale max and stay below 2^8.
constexpr float RESCALE_LOG2 = 8.f;

// SPLIT (attn_fp32): P goes to the tensor pipe as two bf16 values, its rounding and what that leaves, 16 bits and more in all:
// A is off by 1.6414e-3 of its norm, the final rounding, as with P in fp32 (1.8e-3 with P in bf16; 60 layers of 1 to 120 rows
// against 64 bits), for a second P V product: 19.2 -> 19.3 us a 50-token forward, 28.7 -> 30.2 us one of 120 tokens with heads
// of 128 (on the FP32 pipe 24.3 and 47.7).
template <int HD, int TILES, bool SPLIT>
__global__ void __launch_bounds__(64 + 128 * TILES, TILES == 1 ? 2 : 1) attn_fwd_tc_kernel(const __grid_constant__ AttnFwdParams P) {
  using SM = FwdSmem<HD, TILES>;
  constexpr uint32_t PANELS = SM::PANELS;
  // Score buffers in tensor memory.  HD = 128 (and one-tile blocks): one per query tile, P written over S, so the
  // next S of a tile follows its P V product.  HD = 64 with two tiles leaves room for a third buffer (3 x 128 score
  // columns + 2 x 64 output columns = 512): the block's work items (tile, key tile), in issue order, then take the
  // buffers in rotation, item n using buffer n % 3, and the S product of item n + 3 is issued right after the P V
  // product of item n.  Every warp group then finds its next scores computed when it finishes a tile, instead of
  // waiting for P V and S behind its own P.
  constexpr bool ROT = TILES == 2 && HD == 64;
  constexpr int NBUF = ROT ? 3 : TILES;
  constexpr uint32_t O_COL = 128 * NBUF, TMEM_COLS = 256 * TILES;   // score buffer i at 128 i, O of tile g at O_COL + HD g
  static_assert(O_COL + TILES * HD <= TMEM_COLS, "tensor memory columns");
  // the remainders: behind the packed P where a thread holds all its scores, else in columns of their own
  constexpr uint32_t LO_COL = TILES == 1 ? O_COL + HD : 64;
  static_assert(!SPLIT || (!ROT && LO_COL + 64 <= (TILES == 1 ? TMEM_COLS : 128)), "tensor memory columns");
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = tc::smem_u32(smem_raw);
  const uint32_t bars = base + SM::BAR_OFF;
  const uint32_t slot = bars + 8 * SM::N_BARS;
  auto bar = [&](int i) { return bars + 8u * i; };
  const int warp = (int)tc::uniform(threadIdx.x / 32), lane = threadIdx.x % 32;
  const int n_qt = (P.seq + BQ - 1) / BQ;
  int slot_i, hb;
  decode_block((int)blockIdx.x, P.n_slots, P.hq * P.batch, P.chunk, &slot_i, &hb);
  const int h = hb % P.hq, b = hb / P.hq, g = h / P.group;
  const int row0 = b * P.t_pad;                            // first row of this sequence
  int32_t* status = P.status;
  // with pairing a block owns two adjacent tiles, whose key ranges differ by one tile, so both warp groups stay
  // busy for the whole loop
  const int slot_x = P.n_slots - 1 - slot_i;                 // heaviest (latest) causal tiles first
  const bool pair = TILES == 2 && P.pair;
  const int qt0 = pair ? min(2 * slot_x + 1, n_qt - 1) : slot_x;
  const int qt1 = (pair && 2 * slot_x + 1 < n_qt) ? 2 * slot_x : -1;   // odd tile count: the last block has one tile
  auto kv_tiles = [&](int t) {
    const int kv_end = t < 0 ? 0 : (P.causal ? min(P.seq_k, (t + 1) * BQ) : P.seq_k);
    return (kv_end + BKV - 1) / BKV;
  };
  const int n_kv0 = kv_tiles(qt0), n_kv1 = kv_tiles(qt1);
  const int n_kv_max = max(n_kv0, n_kv1);
  if ((base & 1023u) != 0) {
    if (threadIdx.x == 0) atomicCAS(status, 0, 299);
    return;
  }

  if (threadIdx.x == 0) {
    tc::mbar_init(bar(B_QFULL), 1);
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(bar(B_KFULL + s), 1);
      tc::mbar_init(bar(B_KEMPTY + s), 1);
      tc::mbar_init(bar(B_VFULL + s), 1);
      tc::mbar_init(bar(B_VEMPTY + s), 1);
      tc::mbar_init(bar(B_PVDONE + s), 1);
    }
    for (int s = 0; s < 3; ++s) {
      tc::mbar_init(bar(B_SFULL + s), 1);
      tc::mbar_init(bar(B_PFULL + s), 128);
    }
    tc::fence_barrier_init();
    // This thread is the TMA producer: once the kernel before this one (which writes Q, K, V) is complete, the
    // query tiles and the first K / V tiles are requested right here, so that their latency overlaps the
    // tensor-memory allocation and the block-wide barrier below.
    tc::tma_prefetch_desc(&P.tq);
    tc::tma_prefetch_desc(&P.tk);
    tc::tma_prefetch_desc(&P.tv);
    pdl_wait();
    tc::mbar_expect_tx(bar(B_QFULL), (qt1 >= 0 ? 2u : 1u) * SM::TILE);
    tc::tma_load_4d(base + SM::Q_OFF, &P.tq, bar(B_QFULL), 0, qt0 * BQ, b, h * (int)PANELS);
    if (qt1 >= 0) tc::tma_load_4d(base + SM::Q_OFF + SM::TILE, &P.tq, bar(B_QFULL), 0, qt1 * BQ, b, h * (int)PANELS);
    if (n_kv_max > 0) {
      tc::mbar_expect_tx(bar(B_KFULL), SM::TILE);
      tc::tma_load_4d(base + SM::K_OFF, &P.tk, bar(B_KFULL), 0, 0, b, g * (int)PANELS);
      tc::mbar_expect_tx(bar(B_VFULL), SM::TILE);
      tc::tma_load_4d(base + SM::V_OFF, &P.tv, bar(B_VFULL), 0, 0, b, g * (int)PANELS);
    }
  }
  if (warp == 1) {
    tc::tmem_alloc(slot, TMEM_COLS);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  uint32_t tmem_base;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(slot));
  tmem_base = tc::uniform(tmem_base);
  pdl_launch_dependents();

  if (warp == 0 && lane == 0) {
    // ---- TMA producer (the query tiles and key tile 0 were requested during set-up) ---------------
    for (int j = 1; j < n_kv_max; ++j) {
      const int s = j & 1;
      const uint32_t ph = (j >> 1) & 1;
      if (!tc::mbar_wait(bar(B_KEMPTY + s), ph ^ 1, status, 201)) break;
      tc::mbar_expect_tx(bar(B_KFULL + s), SM::TILE);
      tc::tma_load_4d(base + SM::K_OFF + s * SM::TILE, &P.tk, bar(B_KFULL + s), 0, j * BKV, b, g * (int)PANELS);
      if (!tc::mbar_wait(bar(B_VEMPTY + s), ph ^ 1, status, 202)) break;
      tc::mbar_expect_tx(bar(B_VFULL + s), SM::TILE);
      tc::tma_load_4d(base + SM::V_OFF + s * SM::TILE, &P.tv, bar(B_VFULL + s), 0, j * BKV, b, g * (int)PANELS);
    }
  } else if (warp == 1) {
    const bool leader = tc::elect_one();
    // ---- MMA issuer --------------------------------------------------------------------------
    // Per key tile j: [P0(j) ready] PV0(j), S0(j+1), [P1(j) ready] PV1(j), S1(j+1): while one warp group works
    // on its scores the tensor pipe serves the other one.  S and P of a query tile share TMEM columns, so
    // S(j+1) is issued after PV(j), which reads P(j) (the tensor pipe executes in issue order).
    const uint32_t idesc_s = tc::idesc_bf16(BQ, BKV, 0, 0);          // Q K-major, K K-major
    const uint32_t idesc_o = tc::idesc_bf16(BQ, HD, 0, 1);           // P from TMEM, V MN-major (rows are keys)
    // Descriptor words are formed once; per instruction only the start-address field of the low word moves.
    const uint32_t hi = tc::smem_desc_hi(1024);
    const uint32_t q_lo = tc::smem_desc_lo(base + SM::Q_OFF, 16), k_lo = tc::smem_desc_lo(base + SM::K_OFF, 16);
    const uint32_t v_lo = tc::smem_desc_lo(base + SM::V_OFF, 16384);
    auto issue_s = [&](int w, int j) {
      if (!leader) return;
      const uint32_t ql = q_lo + w * (SM::TILE >> 4), kl = k_lo + (j & 1) * (SM::TILE >> 4);
#pragma unroll
      for (uint32_t kk = 0; kk < HD / 16; ++kk) {
        const uint32_t o = (kk / 4) * 1024 + (kk % 4) * 2;            // 16-byte units: 64-column panel, 16-element step
        tc::mma_bf16_ss_w(tmem_base + w * 128, ql + o, hi, kl + o, hi, idesc_s, kk > 0);
      }
      tc::mma_commit(bar(B_SFULL + w));
    };
    auto issue_pv = [&](int w, int j) {
      if (!leader) return;
      const uint32_t vl = v_lo + (j & 1) * (SM::TILE >> 4);
#pragma unroll
      for (uint32_t kk = 0; kk < BKV / 16; ++kk) {
        // A operand from tensor memory: the packed bf16 P row of each lane, 16 keys = 8 columns per step
        tc::mma_bf16_ts_w(tmem_base + O_COL + w * HD, tmem_base + w * 128 + kk * 8, vl + kk * 128, hi, idesc_o,
                          (j > 0 || kk > 0) ? 1u : 0u);
        if constexpr (SPLIT) tc::mma_bf16_ts_w(tmem_base + O_COL + w * HD, tmem_base + w * 128 + LO_COL + kk * 8, vl + kk * 128, hi, idesc_o, 1u);
      }
      tc::mma_commit(bar(B_PVDONE + w));
    };
    if constexpr (ROT) {
      // Work items in issue order: (tile 0, j), (tile 1, j) while tile 1 has key tiles, then tile 0's remaining
      // ones (n_kv0 >= n_kv1: tile 0 is the later query tile).  Barriers of a score buffer are used once per
      // rotation, so neither side can run more than one phase ahead on any of them.
      struct Item { int w, j, buf; uint32_t ph; };          // tile, key tile, score buffer and its phase
      auto next = [&](Item& i) {
        if (i.w == 0 && i.j < n_kv1) i.w = 1; else { i.w = 0; ++i.j; }
        if (++i.buf == 3) { i.buf = 0; i.ph ^= 1; }
      };
      const int n_items = n_kv0 + n_kv1;
      auto issue_s_item = [&](const Item& i) -> bool {
        // tile 0 is the first user of every key tile, and the last one where tile 1 has none
        if (i.w == 0 && !tc::mbar_wait_warp(bar(B_KFULL + (i.j & 1)), (i.j >> 1) & 1, status, 205)) return false;
        const uint32_t ql = q_lo + i.w * (SM::TILE >> 4), kl = k_lo + (i.j & 1) * (SM::TILE >> 4);
        const uint32_t d = tmem_base + (uint32_t)i.buf * 128;
        if (leader) {
#pragma unroll
          for (uint32_t kk = 0; kk < HD / 16; ++kk) {
            const uint32_t o = (kk / 4) * 1024 + (kk % 4) * 2;
            tc::mma_bf16_ss_w(d, ql + o, hi, kl + o, hi, idesc_s, kk > 0);
          }
          tc::mma_commit(bar(B_SFULL + i.buf));
          if (i.w == 1 || i.j >= n_kv1) tc::mma_commit(bar(B_KEMPTY + (i.j & 1)));
        }
        __syncwarp();
        return true;
      };
      bool ok = tc::mbar_wait_warp(bar(B_QFULL), 0, status, 203);
      if (ok) tc::tc_fence_after();
      Item now{0, 0, 0, 0}, ahead = now;
      for (int n = 0; n < 3 && n < n_items && ok; ++n) { ok = issue_s_item(ahead); next(ahead); }
      for (int n = 0; n < n_items && ok; ++n) {
        if (now.w == 0 && !tc::mbar_wait_warp(bar(B_VFULL + (now.j & 1)), (now.j >> 1) & 1, status, 207)) break;
        if (!tc::mbar_wait_warp(bar(B_PFULL + now.buf), now.ph, status, 206)) break;
        tc::tc_fence_after();
        const uint32_t vl = v_lo + (now.j & 1) * (SM::TILE >> 4);
        const uint32_t pa = tmem_base + (uint32_t)now.buf * 128, od = tmem_base + O_COL + now.w * HD;
        if (leader) {
#pragma unroll
          for (uint32_t kk = 0; kk < BKV / 16; ++kk)
            tc::mma_bf16_ts_w(od, pa + kk * 8, vl + kk * 128, hi, idesc_o, (now.j > 0 || kk > 0) ? 1u : 0u);
          tc::mma_commit(bar(B_PVDONE + now.w));
          if (now.w == 1 || now.j >= n_kv1) tc::mma_commit(bar(B_VEMPTY + (now.j & 1)));
        }
        __syncwarp();
        next(now);
        if (n + 3 < n_items) { ok = issue_s_item(ahead); next(ahead); }     // into the buffer whose P the product above has just read
      }
    } else {
    bool ok = tc::mbar_wait_warp(bar(B_QFULL), 0, status, 203) && tc::mbar_wait_warp(bar(B_KFULL), 0, status, 204);
    if (ok) {
      tc::tc_fence_after();
      if (n_kv0 > 0) issue_s(0, 0);
      if (TILES == 2 && n_kv1 > 0) issue_s(1, 0);
    }
    for (int j = 0; j < n_kv_max && ok; ++j) {
      const bool next = j + 1 < n_kv_max;
      if (!tc::mbar_wait_warp(bar(B_VFULL + (j & 1)), (j >> 1) & 1, status, 207)) { ok = false; break; }
      if (next && !tc::mbar_wait_warp(bar(B_KFULL + ((j + 1) & 1)), ((j + 1) >> 1) & 1, status, 205)) { ok = false; break; }
#pragma unroll
      for (int w = 0; w < TILES; ++w) {
        const int nk = w ? n_kv1 : n_kv0;
        if (ok && j < nk) {
          if (!tc::mbar_wait_warp(bar(B_PFULL + w), j & 1, status, 206)) { ok = false; }
          else { tc::tc_fence_after(); issue_pv(w, j); }
        }
        if (ok && j + 1 < nk) issue_s(w, j + 1);
      }
      if (!ok) break;
      if (leader) {
        tc::mma_commit(bar(B_VEMPTY + (j & 1)));            // both P V products of this stage are behind us
        if (next) tc::mma_commit(bar(B_KEMPTY + ((j + 1) & 1)));   // ... and both score products of the next stage
        if (j == 0) tc::mma_commit(bar(B_KEMPTY));          // stage 0 scores were issued before the loop
      }
    }
    }
  } else if (warp >= 2) {
    // ---- softmax warp groups: group w owns query tile qt[w], one query row per thread --------------
    const int w = (warp - 2) / 4;
    const int q = warp % 4;
    const int r = q * 32 + lane;
    const int n_kvw = w ? n_kv1 : n_kv0;
    const int i0 = (w ? qt1 : qt0) * BQ;
    const int gi = i0 + r;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    const uint32_t o_addr = lane_addr + O_COL + w * HD;
    const float c = P.scale * LOG2E;
    const float tau = RESCALE_LOG2 / c;              // the same threshold in raw score units
    pdl_wait();                                      // before this role writes anything
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int j = 0; j < n_kvw && ok; ++j) {
      const int j0 = j * BKV;
      // score buffer and barrier phase of this (tile, key tile): see the MMA issuer
      const int n_item = ROT ? (w ? 2 * j + 1 : j + min(j, n_kv1)) : j;
      const int sbuf = ROT ? n_item % 3 : w;
      const uint32_t sph = ROT ? (uint32_t)(n_item / 3) & 1u : (uint32_t)j & 1u;
      const uint32_t s_addr = lane_addr + (uint32_t)sbuf * 128;
      if (!tc::mbar_wait(bar(B_SFULL + sbuf), sph, status, 208)) { ok = false; break; }
      tc::tc_fence_after();
      const bool need_mask = (j0 + BKV > P.seq_k) || (P.causal && j0 + BKV - 1 > i0);
      float mx, alpha, mc;
      float2 sum01 = make_float2(0.f, 0.f), sum23 = sum01;
      const float2 c2 = make_float2(c, c);
      bool moved;
      if constexpr (TILES == 2) {
        // The row's 128 scores come into registers with one wait (one block per SM: a thread may hold them all):
        // the maximum, the exponentials and the packing then run without touching tensor memory again until
        // the packed P row is stored over the score columns.
        uint32_t sr[128];
  #pragma unroll
        for (int cc = 0; cc < 4; ++cc) tc::tmem_ld32(s_addr + cc * 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[cc * 32]));
        tc::tmem_ld_wait();
        float* sv = reinterpret_cast<float*>(sr);
        if (need_mask) {
  #pragma unroll
          for (int k = 0; k < 128; ++k) {
            const int gj = j0 + k;
            if (gj >= P.seq_k || (P.causal && gj > gi)) sv[k] = -INFINITY;
          }
        }
        float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
  #pragma unroll
        for (int k = 0; k < 128; k += 8) {               // three-input maxima: one instruction per two scores
          mx0 = tc::fmax3(mx0, sv[k], sv[k + 1]); mx1 = tc::fmax3(mx1, sv[k + 2], sv[k + 3]);
          mx2 = tc::fmax3(mx2, sv[k + 4], sv[k + 5]); mx3 = tc::fmax3(mx3, sv[k + 6], sv[k + 7]);
        }
        mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
        // lazy running max: move it only when the tile's max beats it by more than the threshold
        moved = mx > m + tau;                       // (a first finite maximum always does)
        const float m_new = moved ? fmaxf(m, mx) : m;
        alpha = (m == -INFINITY) ? 0.f : tc::fast_exp2((m - m_new) * c);
        mc = (m_new == -INFINITY) ? 0.f : m_new * c;
        m = m_new;
        if (j > 0 && __any_sync(0xffffffffu, moved)) {
          // O is rescaled in place: the previous P V product must have finished
          if (!tc::mbar_wait(bar(B_PVDONE + w), (j - 1) & 1, status, 209)) { ok = false; break; }
          tc::tc_fence_after();
          const float a = moved ? alpha : 1.f;
  #pragma unroll 1
          for (int cc = 0; cc < HD / 32; ++cc) {
            uint32_t o[32];
            tc::tmem_ld32(o_addr + cc * 32, o);
            tc::tmem_ld_wait();
  #pragma unroll
            for (int k = 0; k < 32; k += 2) {
              const float2 v = __fmul2_rn(make_float2(__uint_as_float(o[k]), __uint_as_float(o[k + 1])), make_float2(a, a));
              o[k] = __float_as_uint(v.x); o[k + 1] = __float_as_uint(v.y);
            }
            tc::tmem_st32(o_addr + cc * 32, o);
          }
        }
        // P = exp2(S c - m c), its row sum, and P packed to bf16 (128 scores become 64 packed columns)
        const float2 nmc2 = make_float2(-mc, -mc);
  #pragma unroll
        for (int k = 0; k < 128; k += 4) {
          const float2 x01 = __ffma2_rn(make_float2(sv[k], sv[k + 1]), c2, nmc2);       // two-wide fp32 operations
          const float2 x23 = __ffma2_rn(make_float2(sv[k + 2], sv[k + 3]), c2, nmc2);
          const float p0 = tc::fast_exp2(x01.x), p1 = tc::fast_exp2(x01.y), p2 = tc::fast_exp2(x23.x), p3 = tc::fast_exp2(x23.y);
          sum01 = __fadd2_rn(sum01, make_float2(p0, p1)); sum23 = __fadd2_rn(sum23, make_float2(p2, p3));
          if constexpr (SPLIT) {
            split_bf16(p0, p1, sr[k], sr[k + 1]);
            split_bf16(p2, p3, sr[k + 2], sr[k + 3]);
          } else {
            sr[k / 2] = tc::pack_bf16(p0, p1);
            sr[k / 2 + 1] = tc::pack_bf16(p2, p3);
          }
        }
        if constexpr (SPLIT) {
#pragma unroll
          for (int x = 0; x < 4; ++x) {                // P's columns, first and second half, then the remainders'
            uint32_t v[32];
#pragma unroll
            for (int k = 0; k < 32; ++k) v[k] = sr[(x & 1) * 64 + 2 * k + x / 2];
            tc::tmem_st32(s_addr + 32 * x, v);
          }
        } else {
          tc::tmem_st32(s_addr, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
          tc::tmem_st32(s_addr + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
        }
      } else {
        // At most 128 registers here (two blocks per SM): two passes over the scores in tensor memory in 32-column
        // loads instead of holding the row, and only as many as the warp attends to.
        // 32-key chunks of this tile that any row of the warp attends to (the rest: beyond the keys, above the diagonal;
        // none for a warp of padding rows).  P is zero in the others, and their scores are not looked at.
        const int gw = gi - lane, key_end = gw >= P.seq ? 0 : P.causal ? min(P.seq_k, gw + 32) : P.seq_k;
        const int n_ch = min(4, max(0, key_end - j0 + 31) / 32);
        auto mask_chunk = [&](float* sc, int cc) {
          if (j0 + cc * 32 + 32 <= P.seq_k && (!P.causal || j0 + cc * 32 + 31 <= gw)) return;
#pragma unroll
          for (int k = 0; k < 32; ++k) {
            const int gj = j0 + cc * 32 + k;
            if (gj >= P.seq_k || (P.causal && gj > gi)) sc[k] = -INFINITY;
          }
        };
        float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll 1
        for (int cc = 0; cc < n_ch; ++cc) {
          uint32_t sr[32];
          tc::tmem_ld32(s_addr + cc * 32, sr);
          tc::tmem_ld_wait();
          float* sc = reinterpret_cast<float*>(sr);
          if (need_mask) mask_chunk(sc, cc);
#pragma unroll
          for (int k = 0; k < 32; k += 8) {
            mx0 = tc::fmax3(mx0, sc[k], sc[k + 1]); mx1 = tc::fmax3(mx1, sc[k + 2], sc[k + 3]);
            mx2 = tc::fmax3(mx2, sc[k + 4], sc[k + 5]); mx3 = tc::fmax3(mx3, sc[k + 6], sc[k + 7]);
          }
        }
        mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
        moved = mx > m + tau;                       // (a first finite maximum always does)
        const float m_new = moved ? fmaxf(m, mx) : m;
        alpha = (m == -INFINITY) ? 0.f : tc::fast_exp2((m - m_new) * c);
        mc = (m_new == -INFINITY) ? 0.f : m_new * c;
        m = m_new;
        if (j > 0 && __any_sync(0xffffffffu, moved)) {
          if (!tc::mbar_wait(bar(B_PVDONE + w), (j - 1) & 1, status, 209)) { ok = false; break; }
          tc::tc_fence_after();
          const float a = moved ? alpha : 1.f;
#pragma unroll 1
          for (int cc = 0; cc < HD / 32; ++cc) {
            uint32_t o[32];
            tc::tmem_ld32(o_addr + cc * 32, o);
            tc::tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 32; k += 2) {
              const float2 v = __fmul2_rn(make_float2(__uint_as_float(o[k]), __uint_as_float(o[k + 1])), make_float2(a, a));
              o[k] = __float_as_uint(v.x); o[k + 1] = __float_as_uint(v.y);
            }
            tc::tmem_st32(o_addr + cc * 32, o);
          }
        }
        const float2 nmc2 = make_float2(-mc, -mc);
        // pass 2: P packed to bf16 over the score columns already consumed (32 scores become 16 packed columns;
        // the thread owns the lane, so nobody else's data is overwritten)
#pragma unroll 1
        for (int cc = 0; cc < n_ch; ++cc) {
          uint32_t sr[32];
          tc::tmem_ld32(s_addr + cc * 32, sr);
          tc::tmem_ld_wait();
          float* sc = reinterpret_cast<float*>(sr);
          if (need_mask) mask_chunk(sc, cc);
          uint32_t pk[16], lo[SPLIT ? 16 : 1];
#pragma unroll
          for (int k = 0; k < 32; k += 4) {
            const float2 x01 = __ffma2_rn(make_float2(sc[k], sc[k + 1]), c2, nmc2);
            const float2 x23 = __ffma2_rn(make_float2(sc[k + 2], sc[k + 3]), c2, nmc2);
            const float p0 = tc::fast_exp2(x01.x), p1 = tc::fast_exp2(x01.y), p2 = tc::fast_exp2(x23.x), p3 = tc::fast_exp2(x23.y);
            sum01 = __fadd2_rn(sum01, make_float2(p0, p1)); sum23 = __fadd2_rn(sum23, make_float2(p2, p3));
            if constexpr (SPLIT) {
              split_bf16(p0, p1, pk[k / 2], lo[k / 2]);
              split_bf16(p2, p3, pk[k / 2 + 1], lo[k / 2 + 1]);
            } else {
              pk[k / 2] = tc::pack_bf16(p0, p1);
              pk[k / 2 + 1] = tc::pack_bf16(p2, p3);
            }
          }
          tc::tmem_st16(s_addr + cc * 16, pk);
          if constexpr (SPLIT) tc::tmem_st16(s_addr + LO_COL + cc * 16, lo);
        }
        const uint32_t zero[16] = {};
#pragma unroll 1
        for (int cc = n_ch; cc < 4; ++cc) {
          tc::tmem_st16(s_addr + cc * 16, zero);
          if constexpr (SPLIT) tc::tmem_st16(s_addr + LO_COL + cc * 16, zero);
        }
      }
      if (moved) l *= alpha;
      l += (sum01.x + sum01.y) + (sum23.x + sum23.y);
      tc::tmem_st_wait();
      tc::tc_fence_before();
      // With rotating buffers a tile's scores say nothing about its last P V product, and a wait that has let a phase of
      // that barrier pass unseen would take an older one for it: see every phase before the next one can complete.
      if (ROT && j > 0 && !tc::mbar_wait(bar(B_PVDONE + w), (j - 1) & 1, status, 211)) { ok = false; break; }
      tc::mbar_arrive(bar(B_PFULL + sbuf));
    }
    if (ok && n_kvw > 0) ok = tc::mbar_wait(bar(B_PVDONE + w), (n_kvw - 1) & 1, status, 210);
    tc::tc_fence_after();
    if (ok && n_kvw > 0) {
      const bool live = gi < P.seq;
      const float inv = live ? 1.f / l : 0.f;
#pragma unroll
      for (int cc = 0; cc < HD / 32; ++cc) {
        uint32_t o[32];
        tc::tmem_ld32(o_addr + cc * 32, o);
        tc::tmem_ld_wait();
        if (gi < P.t_pad) {
          const int col = h * HD + cc * 32;
          __nv_bfloat16* dst = P.a + ((long long)(col / 64) * P.n_pad + row0 + gi) * 64 + (col % 64);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            uint4 v;
            v.x = tc::pack_bf16(__uint_as_float(o[k * 8 + 0]) * inv, __uint_as_float(o[k * 8 + 1]) * inv);
            v.y = tc::pack_bf16(__uint_as_float(o[k * 8 + 2]) * inv, __uint_as_float(o[k * 8 + 3]) * inv);
            v.z = tc::pack_bf16(__uint_as_float(o[k * 8 + 4]) * inv, __uint_as_float(o[k * 8 + 5]) * inv);
            v.w = tc::pack_bf16(__uint_as_float(o[k * 8 + 6]) * inv, __uint_as_float(o[k * 8 + 7]) * inv);
            *reinterpret_cast<uint4*>(dst + 8 * k) = v;
          }
        }
      }
      if (gi < P.t_pad) P.lse[((long long)b * P.hq + h) * P.t_pad + gi] = live ? m * P.scale + logf(l) : 0.f;
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem_base, TMEM_COLS);
}

// A launch made ready but for its addresses: what the launchers keep.
template <typename Params>
struct AttnLaunch {
  Params P;
  void (*kernel)(const Params);
  int grid, threads, cluster;                              // cluster: blocks of one where the launch has any, else 0
  size_t smem;
  cudaError_t set(void (*k)(const Params), int g, int t, size_t s, int c = 0) {
    kernel = k; grid = g; threads = t; smem = s; cluster = c;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s);
  }
};

template <int HD, int TILES, bool SPLIT = false>
cudaError_t fwd_make_t(AttnLaunch<AttnFwdParams>& L, const fbl_plan* p, int n_qt) {
  AttnFwdParams& P = L.P;
  if (TILES == 1) P.pair = 0;
  P.batch = p->d.batch;
  P.n_slots = P.pair ? (n_qt + 1) / 2 : n_qt;
  P.chunk = chunk_for((long long)p->seq_kv * HD * 4, p->d.n_q_heads * p->d.batch, 96ll << 20);   // K and V of one head
  return L.set(attn_fwd_tc_kernel<HD, TILES, SPLIT>, P.n_slots * p->d.n_q_heads * p->d.batch, 64 + 128 * TILES, FwdSmem<HD, TILES>::TOTAL);
}

// head_dim 64: one query tile a block and two blocks per SM, or two tiles (a single one where `pair` is 0) and one block per SM.
// A block of two tiles takes 0.93 of the time of two blocks of one (it looks at a score once, and three score buffers rotate), a
// tile alone on its SM 0.8 of what it takes in a block of one; blocks of one start and end faster and fill the SMs in
// finer steps.  So, from forward passes of 200 to 2048 tokens, 8 to 128 heads and sequences (one / two tiles, us):
//   short: one (5 x 16 heads of 384: 37.5 / 41.8; 1500 queries over 200 keys: 77.0 / 82.7);
//   less than an SM's worth of pairs: a tile alone where all tiles fit at once (12 heads of 500: 25.3 / 23.2, of 1500 causal 41.8 /
//   36.0), else one (2 x 20 heads of 830: 49.5 / 59.2), but for long causal chains (16 heads of 1536: 49.6 / 40.2);
//   causal pairs: an odd count leaves a tile alone in its block, so odd counts change over later.  One up to six tiles (4 x 32 heads of
//   760: 63.8 / 63.3, 16 x 32 219 / 234), two from eight on where the count is even (4 x 32 of 960: 84.6 / 82.0, 8 x 16 of 1020 93.2 /
//   91.0, 3 x 40 83.5 / 84.5; 8 x 16 of 1260 124.7 / 120.9, of 1500 153.8 / 148.1), past nine where it is odd (16 x 12 of 890: 117 /
//   124, 4 x 32 of 890 79.0 / 77.5; of 1150 96.5 / 100, 3 x 40 94.0 / 98.8; 11 and 13 tiles within 2 %);
//   else rounds: one where the pairs' last round costs more (3 x 32 heads of 1150: 134 / 140, of 1500: 180 / 168); five rounds and more even out.
bool fwd_one_tile(const fbl_plan* p, int n_qt, int pair) {
  const int n_kt = (p->seq_kv + BKV - 1) / BKV;
  if (n_qt <= 2 || n_kt <= 2) return true;
  const long long sm = p->sm_count, heads = (long long)p->d.n_q_heads * p->d.batch, blocks = n_qt * heads, pairs = (n_qt + 1) / 2 * heads;
  if (!pair) return blocks > sm && (!p->d.causal || n_qt <= 6);
  if (n_qt <= 4 || n_kt <= 4) return true;
  if (p->d.causal) return n_qt <= (n_qt % 2 ? 9 : 6);
  return pairs <= 5 * sm && 1.08 * ((blocks + 2 * sm - 1) / (2 * sm)) < (pairs + sm - 1) / sm;
}

template <int HD>
cudaError_t fwd_make(AttnLaunch<AttnFwdParams>& L, const fbl_plan* p, const void* Q, const void* K, const void* V) {
  AttnFwdParams& P = L.P;
  memset(&P, 0, sizeof(P));
  const int panels = HD / 64;
  if (!fbl_encode_seq_map(&P.tq, false, Q, p->t_pad, p->d.batch, p->dq / 64, BQ, panels)) return cudaErrorInvalidValue;
  if (!fbl_encode_seq_map(&P.tk, false, K, p->t_pad_kv, p->d.batch, p->dkv / 64, BKV, panels)) return cudaErrorInvalidValue;
  if (!fbl_encode_seq_map(&P.tv, false, V, p->t_pad_kv, p->d.batch, p->dkv / 64, BKV, panels)) return cudaErrorInvalidValue;
  P.n_pad = p->n_pad;
  P.seq = p->d.seq; P.t_pad = p->t_pad; P.hq = p->d.n_q_heads; P.group = p->group; P.causal = p->d.causal;
  P.seq_k = p->seq_kv; P.t_pad_k = p->t_pad_kv;
  P.scale = p->scale;
  const int n_qt = (p->d.seq + BQ - 1) / BQ;
  // two query tiles per block when that still leaves at least one block per SM
  P.pair = (n_qt >= 2 && (long long)((n_qt + 1) / 2) * p->d.n_q_heads * p->d.batch >= p->sm_count) ? 1 : 0;
  if (attn_fp32(p)) return fwd_make_t<HD, HD == 64 ? 1 : 2, true>(L, p, n_qt);
  if (HD == 64) {
    // tuning knob: 1 = one query tile per block and two blocks per SM, 2 = two tiles per block; default by shape
    const int mode = p->knob_fwd_tiles;
    if (mode == 1 || (mode == 0 && fwd_one_tile(p, n_qt, P.pair))) return fwd_make_t<64, 1>(L, p, n_qt);
  }
  return fwd_make_t<HD, 2>(L, p, n_qt);
}

// ---------------------------------------------------------------------------------------------------
// Backward: one block per (128-key tile, KV head, batch).  For every query head of the group and every
// query tile it recomputes the transposed scores S^T = K Q^T and dP^T = V dO^T on the tensor pipe (so
// the rows a thread owns are keys), forms P^T = exp(S^T - LSE) and dS^T = P^T * (dP^T - D) in registers,
// and writes both once to swizzled shared memory.  Those two tiles then feed three products:
//   dV += P^T dO  and  dK += dS^T Q   (sequence-axis reductions; accumulators stay in TMEM over the
//                                      whole query loop and over the G heads of the group), and
//   dQ  = dS K    (the same dS^T bytes read MN-major, i.e. transposed by descriptor), a key-axis
//                  reduction across blocks, added to an fp32 buffer with vector red operations.
// ---------------------------------------------------------------------------------------------------
struct alignas(64) AttnBwdParams {
  CUtensorMap tq, tk, tv, tdo, tdq;   // tdq: fp32 dQ accumulator, target of the bulk reductions
  const float* lse;      // [B, Hq, t_pad]
  const float* dvec;     // [B, Hq, t_pad]   D = rowsum(dO * O)
  float* dqacc;          // fp32 [n_pad, dq] in the bf16 tile order
  __nv_bfloat16* dq;     // where dQ goes at once when a block sees all keys of its queries
  __nv_bfloat16* dk;
  __nv_bfloat16* dv;
  long long n_pad, n_pad_k;          // rows of the query-side (Q, dO, dQ) and key-side (K, V, dK, dV) buffers
  int seq, t_pad, hq, group, causal, dkv;
  int seq_k, t_pad_k;                // key-side sequence length and padded length
  int batch, chunk;      // grid = key tiles * KV heads * batch blocks, see decode_block
  int slices;            // SLICED: blocks of a cluster, which share a key tile's items
  float scale;
  int32_t* status;
};

// P^T never touches shared memory: the softmax warps store it (bf16, two per column) over the S^T columns
// in tensor memory once every warp has read them, and dV += P^T dO takes its A operand from there.  HD = 64
// has spare TMEM columns for dQ and shared memory to double-buffer Q/dO and dS^T, so the tensor pipe computes
// the next tile's S^T / dP^T and this tile's dK, dQ while the softmax warps are busy.  HD = 128 fills TMEM
// (S^T, dP^T, dV, dK = 512 columns): dQ reuses the dP^T columns, so only the next S^T can be issued before dQ
// has been drained.  Both keep a separate staging area for the asynchronous dQ reduction.
template <int HD>
struct BwdSmem {
  static constexpr bool PIPE = HD == 64;
  // stages: Q (needed first, for the next S^T, and freed last, by dK) three deep, dO and dS^T two deep, one dQ
  // staging tile; everything single at HD = 128
  static constexpr uint32_t NQQ = PIPE ? 3 : 1, NDO = PIPE ? 2 : 1, NP = PIPE ? 2 : 1, NS = 1;
  static constexpr uint32_t PANELS = HD / 64;
  static constexpr uint32_t TILE = PANELS * 16384;
  static constexpr uint32_t STAGE_BYTES = 128 * HD * 4;               // one fp32 dQ tile
  static constexpr uint32_t K_OFF = 0, V_OFF = TILE, Q_OFF = 2 * TILE, DO_OFF = Q_OFF + NQQ * TILE;
  static constexpr uint32_t DS_OFF = DO_OFF + NDO * TILE, STAGE_OFF = DS_OFF + NP * 32768;
  static constexpr uint32_t LSE_OFF = STAGE_OFF + NS * STAGE_BYTES;    // 128 floats of LSE per Q stage, then 128 of D per dO stage
  static constexpr uint32_t D_OFF = LSE_OFF + NQQ * 512;
  static constexpr uint32_t BAR_OFF = D_OFF + NDO * 512;
  static constexpr uint32_t N_BARS = 24;          // BB_* below: 22 in use
  static constexpr uint32_t TOTAL = BAR_OFF + 8 * N_BARS + 16;
};

enum { BB_KVFULL = 0, BB_QFULL = 1, BB_QEMPTY = 4, BB_DOFULL = 7, BB_DOEMPTY = 9, BB_SFULL = 11, BB_PDSFULL, BB_DQFULL, BB_DQDRAINED, BB_DQSTAGED, BB_STAGEFREE = BB_DQSTAGED + 2, BB_SREAD = BB_STAGEFREE + 2, BB_DVDONE, BB_DPFULL };

// No (query, key) pair of nq queries from i and the 32 keys from j takes part.
__device__ __forceinline__ bool warp_masked(int i, int nq, int j, const AttnBwdParams& P) {
  return i >= P.seq || j >= P.seq_k || (P.causal && i + nq - 1 < j);
}

// NC accumulator columns of one row, scaled and rounded, to columns col .. of row `row` of an R-Tile matrix.
template <int NC>
__device__ __forceinline__ void store_cols(__nv_bfloat16* m, long long rows, long long row, int col, const uint32_t (&o)[NC], float f) {
  __nv_bfloat16* dst = m + ((long long)(col / 64) * rows + row) * 64 + (col % 64);
#pragma unroll
  for (int k = 0; k < NC / 8; ++k) {
    uint4 v;
    v.x = tc::pack_bf16(__uint_as_float(o[k * 8 + 0]) * f, __uint_as_float(o[k * 8 + 1]) * f);
    v.y = tc::pack_bf16(__uint_as_float(o[k * 8 + 2]) * f, __uint_as_float(o[k * 8 + 3]) * f);
    v.z = tc::pack_bf16(__uint_as_float(o[k * 8 + 4]) * f, __uint_as_float(o[k * 8 + 5]) * f);
    v.w = tc::pack_bf16(__uint_as_float(o[k * 8 + 6]) * f, __uint_as_float(o[k * 8 + 7]) * f);
    *reinterpret_cast<uint4*>(dst + 8 * k) = v;
  }
}

constexpr int BWD_THREADS = 608;     // warp 0 TMA loads, warp 1 MMA, warps 2-17 softmax (four per TMEM lane quarter), warp 18 dQ reductions
constexpr int BWD_SM_THREADS = 512;

// DIRECT: the sequence has a single key tile, so a block's dQ tile is complete and goes out rounded, without the fp32
// accumulator, its zero-fill and the rounding pass.
// SLICED: a cluster of `slices` blocks shares a key tile's (query head, query tile) items, in contiguous runs, and adds its
// fp32 dK and dV through distributed shared memory in a fixed order.  For grouped heads whose key tiles, KV heads and
// sequences make a fraction of 148 blocks: the bound is then the items' chain.
template <int HD, bool DIRECT, bool SLICED>
__global__ void __launch_bounds__(BWD_THREADS, 1) attn_bwd_tc_kernel(const __grid_constant__ AttnBwdParams P) {
  using SM = BwdSmem<HD>;
  constexpr bool PIPE = SM::PIPE;
  constexpr uint32_t PANELS = SM::PANELS, NQQ = SM::NQQ, NDO = SM::NDO, NP = SM::NP, NS = SM::NS;
  constexpr uint32_t S_COL = 0, DP_COL = 128, DV_COL = 256, DK_COL = 256 + HD;
  constexpr uint32_t DQ_COL = PIPE ? 384 : DP_COL;   // HD = 128: dQ reuses the dP^T columns
  constexpr uint32_t P_COL = PIPE ? 448 : S_COL;     // HD = 64: own columns; HD = 128: P^T overwrites S^T in place
  constexpr uint32_t TMEM_COLS = 512;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = tc::smem_u32(smem_raw);
  const uint32_t bars = base + SM::BAR_OFF;
  const uint32_t slot = bars + 8 * SM::N_BARS;
  auto bar = [&](int i) { return bars + 8u * i; };
  const int warp = (int)tc::uniform(threadIdx.x / 32), lane = threadIdx.x % 32;
  // under a causal mask key tile 0 has the most query tiles: it is slot 0
  const int n_kvh = P.hq / P.group;
  int slot_i, gb;
  const int slices = SLICED ? P.slices : 1, slice = SLICED ? (int)blockIdx.x % slices : 0;
  decode_block((int)blockIdx.x / slices, (P.t_pad_k + BKV - 1) / BKV, n_kvh * P.batch, P.chunk, &slot_i, &gb);
  const int j0 = slot_i * BKV, g = gb % n_kvh, b = gb / n_kvh;
  const int row0 = b * P.t_pad, row0k = b * P.t_pad_k;
  const int n_qt = (P.seq + BQ - 1) / BQ;
  const int qt_begin = P.causal ? j0 / BQ : 0;
  const int per_head = n_qt - qt_begin;
  const int share = SLICED ? (P.group * per_head + slices - 1) / slices : P.group * per_head;
  const int it0 = SLICED ? slice * share : 0, n_it = SLICED ? min(share, P.group * per_head - it0) : share;     // none: n_it <= 0
  const int h0 = g * P.group + (SLICED && n_it > 0 ? it0 / per_head : 0), c0_q = SLICED && n_it > 0 ? it0 % per_head : 0;   // first item
  int32_t* status = P.status;
  if ((base & 1023u) != 0) {                    // the swizzled tiles need a 1024-byte aligned window
    if (threadIdx.x == 0) atomicCAS(status, 0, 399);
    return;
  }

  if (threadIdx.x == 0) {
    tc::mbar_init(bar(BB_KVFULL), 1);
    for (int s = 0; s < 3; ++s) {
      tc::mbar_init(bar(BB_QFULL + s), 1);
      tc::mbar_init(bar(BB_QEMPTY + s), 1);
    }
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(bar(BB_DOFULL + s), 1);
      tc::mbar_init(bar(BB_DOEMPTY + s), 1);
    }
    tc::mbar_init(bar(BB_SFULL), 1);
    tc::mbar_init(bar(BB_PDSFULL), BWD_SM_THREADS);
    tc::mbar_init(bar(BB_DQFULL), 1);
    tc::mbar_init(bar(BB_DQDRAINED), BWD_SM_THREADS);
    tc::mbar_init(bar(BB_DQSTAGED), BWD_SM_THREADS);
    tc::mbar_init(bar(BB_DQSTAGED + 1), BWD_SM_THREADS);
    tc::mbar_init(bar(BB_STAGEFREE), 1);
    tc::mbar_init(bar(BB_STAGEFREE + 1), 1);
    tc::mbar_init(bar(BB_SREAD), BWD_SM_THREADS);
    tc::mbar_init(bar(BB_DVDONE), 1);
    tc::mbar_init(bar(BB_DPFULL), 1);
    tc::fence_barrier_init();
    // This thread is the TMA producer: K, V and the first Q tile (forward-pass data) are requested right here, so
    // that their latency overlaps the tensor-memory allocation and the block-wide barrier below.
    tc::tma_prefetch_desc(&P.tk); tc::tma_prefetch_desc(&P.tv); tc::tma_prefetch_desc(&P.tq);
    tc::tma_prefetch_desc(&P.tdo);
    if (!DIRECT) tc::tma_prefetch_desc(&P.tdq);
    tc::mbar_expect_tx(bar(BB_KVFULL), 2 * SM::TILE);
    tc::tma_load_3d(base + SM::K_OFF, &P.tk, bar(BB_KVFULL), 0, row0k + j0, g * (int)PANELS);
    tc::tma_load_3d(base + SM::V_OFF, &P.tv, bar(BB_KVFULL), 0, row0k + j0, g * (int)PANELS);
    if (n_it > 0) {
      // LSE travels with Q and D with dO: 128 floats each, into the iteration's staging buffer
      tc::mbar_expect_tx(bar(BB_QFULL), SM::TILE + 512);
      tc::tma_load_3d(base + SM::Q_OFF, &P.tq, bar(BB_QFULL), 0, row0 + (qt_begin + c0_q) * BQ, h0 * (int)PANELS);
      tc::bulk_load(base + SM::LSE_OFF, P.lse + ((long long)b * P.hq + h0) * P.t_pad + (qt_begin + c0_q) * BQ, 512, bar(BB_QFULL));
    }
  }
  if (warp == 1) {
    tc::tmem_alloc(slot, TMEM_COLS);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  uint32_t tmem_base;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(slot));
  tmem_base = tc::uniform(tmem_base);
  pdl_launch_dependents();
  // Where a block's dQ tiles are staged for the bulk reduction: one staging tile; with the pipelined variant the
  // last tile goes to the dS^T buffer that the last iteration does not use (its readers, the dK and dQ products of
  // the tile before, are complete by then), so the block's final drain does not wait for the previous reduction.
  auto stage_is_alt = [&](int dit) { return PIPE && dit == n_it - 1 && n_it >= 2; };
  auto stage_addr = [&](int dit) -> uint32_t {
    return stage_is_alt(dit) ? base + SM::DS_OFF + (uint32_t)(n_it % (int)NP) * 32768u
                             : base + SM::STAGE_OFF + (uint32_t)(dit % (int)NS) * SM::STAGE_BYTES;
  };
  // Of this kernel's inputs only dO (and D) come from the kernel before it (the dA GEMM); K, V, Q and LSE are the
  // forward pass's.  Each role therefore waits for that kernel where it first needs it: the producer has K, V
  // and the first Q tile on their way before it does.
  if (warp == 0 && lane == 0) {
    // ---- TMA producer ------------------------------------------------------------------------
    // (K, V and Q of the first tile were requested during set-up)
    bool waited = false;
    for (int it = 0; it < n_it; ++it) {
      const int h = g * P.group + (it0 + it) / per_head, qt = qt_begin + (it0 + it) % per_head;
      // LSE travels with Q and D with dO, 128 floats each.  A stage's previous readers (the products, and for
      // LSE / D the softmax warps, which finish a tile before its dK and dV products are issued) are behind the
      // barrier that frees it.  Rows past the sequence end may hold anything: the softmax warps mask them.
      const long long stat_off = ((long long)b * P.hq + h) * P.t_pad + qt * BQ;
      const uint32_t sq = it % NQQ, sd = it % NDO;
      if (it > 0) {
        if (!tc::mbar_wait(bar(BB_QEMPTY + sq), ((it / NQQ) & 1) ^ 1, status, 301)) break;
        tc::mbar_expect_tx(bar(BB_QFULL + sq), SM::TILE + 512);
        tc::tma_load_3d(base + SM::Q_OFF + sq * SM::TILE, &P.tq, bar(BB_QFULL + sq), 0, row0 + qt * BQ, h * (int)PANELS);
        tc::bulk_load(base + SM::LSE_OFF + sq * 512, P.lse + stat_off, 512, bar(BB_QFULL + sq));
      }
      if (!tc::mbar_wait(bar(BB_DOEMPTY + sd), ((it / NDO) & 1) ^ 1, status, 313)) break;
      if (!waited) { pdl_wait(); waited = true; }
      tc::mbar_expect_tx(bar(BB_DOFULL + sd), SM::TILE + 512);
      tc::tma_load_3d(base + SM::DO_OFF + sd * SM::TILE, &P.tdo, bar(BB_DOFULL + sd), 0, row0 + qt * BQ, h * (int)PANELS);
      tc::bulk_load(base + SM::D_OFF + sd * 512, P.dvec + stat_off, 512, bar(BB_DOFULL + sd));
    }
  } else if (warp == 1) {
    const bool leader = tc::elect_one();
    // ---- MMA issuer --------------------------------------------------------------------------
    const uint32_t idesc_s = tc::idesc_bf16(BKV, BQ, 0, 0);
    const uint32_t idesc_kv = tc::idesc_bf16(BKV, HD, 0, 1);
    const uint32_t idesc_dq = tc::idesc_bf16(BQ, HD, 1, 1);
    // Descriptor words are formed once; per instruction only the start-address field of the low word moves
    // (offsets below are in 16-byte units: a 64-column panel is 1024, a 16-element step along a row 2, 16 rows 128).
    const uint32_t hi = tc::smem_desc_hi(1024);
    const uint32_t k_km = tc::smem_desc_lo(base + SM::K_OFF, 16), k_mn = tc::smem_desc_lo(base + SM::K_OFF, 16384);
    const uint32_t v_km = tc::smem_desc_lo(base + SM::V_OFF, 16);
    const uint32_t q_km = tc::smem_desc_lo(base + SM::Q_OFF, 16), q_mn = tc::smem_desc_lo(base + SM::Q_OFF, 16384);
    const uint32_t do_km = tc::smem_desc_lo(base + SM::DO_OFF, 16), do_mn = tc::smem_desc_lo(base + SM::DO_OFF, 16384);
    const uint32_t ds_km = tc::smem_desc_lo(base + SM::DS_OFF, 16), ds_mn = tc::smem_desc_lo(base + SM::DS_OFF, 16384);
    auto issue_s = [&](int it) {              // S^T = K Q^T of tile `it`
      if (!leader) return;
      const uint32_t qs = q_km + (it % NQQ) * (SM::TILE >> 4);
#pragma unroll
      for (uint32_t kk = 0; kk < HD / 16; ++kk) {
        const uint32_t o = (kk / 4) * 1024 + (kk % 4) * 2;
        tc::mma_bf16_ss_w(tmem_base + S_COL, k_km + o, hi, qs + o, hi, idesc_s, kk > 0);
      }
      if (!PIPE) tc::mma_commit(bar(BB_SFULL));     // HD = 128: the softmax warps start on the scores while dP^T is
    };                                              // still to come (it waits for the previous tile's dQ drain)
    auto issue_dp = [&](int it) {             // dP^T = V dO^T of tile `it`, announced on its own barrier
      if (!leader) return;
      const uint32_t dos = do_km + (it % NDO) * (SM::TILE >> 4);
#pragma unroll
      for (uint32_t kk = 0; kk < HD / 16; ++kk) {
        const uint32_t o = (kk / 4) * 1024 + (kk % 4) * 2;
        tc::mma_bf16_ss_w(tmem_base + DP_COL, v_km + o, hi, dos + o, hi, idesc_s, kk > 0);
      }
      tc::mma_commit(bar(PIPE ? BB_SFULL : BB_DPFULL));      // HD = 64: one announcement for both score tiles
    };
    auto issue_dv = [&](int it) {             // dV += P^T dO, P^T read from tensor memory
      if (!leader) return;
      const uint32_t dos = do_mn + (it % NDO) * (SM::TILE >> 4);
#pragma unroll
      for (uint32_t kk = 0; kk < BQ / 16; ++kk)                      // dO: MN-major, 16 query rows per step;
        tc::mma_bf16_ts_w(tmem_base + DV_COL, tmem_base + P_COL + kk * 8,   // 16 queries = 8 packed columns
                          dos + kk * 128, hi, idesc_kv, (it > 0 || kk > 0) ? 1u : 0u);
    };
    auto issue_dk = [&](int it) {             // dK += dS^T Q
      if (!leader) return;
      const uint32_t qs = q_mn + (it % NQQ) * (SM::TILE >> 4);
      const uint32_t dss = ds_km + (it % NP) * 2048;
#pragma unroll
      for (uint32_t kk = 0; kk < BQ / 16; ++kk) {
        const uint32_t ao = (kk / 4) * 1024 + (kk % 4) * 2;        // dS^T: K-major, reduction over queries
        tc::mma_bf16_ss_w(tmem_base + DK_COL, dss + ao, hi, qs + kk * 128, hi, idesc_kv,   // Q: MN-major, 16 query rows
                          (it > 0 || kk > 0) ? 1u : 0u);
      }
    };
    auto issue_dq = [&](int it) {             // dQ = dS K: the dS^T tile read MN-major, i.e. transposed by descriptor
      if (!leader) return;
      const uint32_t dss = ds_mn + (it % NP) * 2048;
#pragma unroll
      for (uint32_t kk = 0; kk < BKV / 16; ++kk)                     // both operands MN-major: 16 key rows per step
        tc::mma_bf16_ss_w(tmem_base + DQ_COL, dss + kk * 128, hi, k_mn + kk * 128, hi, idesc_dq, kk > 0);
      tc::mma_commit(bar(BB_DQFULL));
    };
    bool ok = tc::mbar_wait_warp(bar(BB_KVFULL), 0, status, 302);
    if (ok && n_it > 0) {
      ok = tc::mbar_wait_warp(bar(BB_QFULL), 0, status, 303) && tc::mbar_wait_warp(bar(BB_DOFULL), 0, status, 314);
      if (ok) { tc::tc_fence_after(); issue_s(0); issue_dp(0); }
    }
    if (PIPE) {
      // P^T has its own columns here, so the next tile's products come first and the softmax warps start on
      // tile it + 1 while the tensor pipe works on dV, dK, dQ of tile it
      for (int it = 0; it < n_it && ok; ++it) {
        if (it + 1 < n_it) {
          // S^T(it+1) as soon as every softmax warp has copied S^T(it) to registers: it is computed while
          // they work on tile it
          if (!tc::mbar_wait_warp(bar(BB_SREAD), it & 1, status, 311)) { ok = false; break; }
          if (!tc::mbar_wait_warp(bar(BB_QFULL + ((it + 1) % NQQ)), ((it + 1) / NQQ) & 1, status, 303)) { ok = false; break; }
          tc::tc_fence_after();
          issue_s(it + 1);
        }
        if (!tc::mbar_wait_warp(bar(BB_PDSFULL), it & 1, status, 305)) { ok = false; break; }
        tc::tc_fence_after();
        if (it + 1 < n_it) {
          if (!tc::mbar_wait_warp(bar(BB_DOFULL + ((it + 1) % NDO)), ((it + 1) / NDO) & 1, status, 314)) { ok = false; break; }
          issue_dp(it + 1);                             // dP^T(it) has been read as well: announce tile it + 1
        }
        issue_dv(it);
        if (leader) tc::mma_commit(bar(BB_DVDONE));                 // P^T(it) has been read: P^T(it+1) may be stored
        if (leader) tc::mma_commit(bar(BB_DOEMPTY + (it % NDO)));   // ... and dO of this tile is not read again
        issue_dk(it);
        if (leader) tc::mma_commit(bar(BB_QEMPTY + (it % NQQ)));    // nor is Q
        if (it > 0 && !tc::mbar_wait_warp(bar(BB_DQDRAINED), (it - 1) & 1, status, 304)) { ok = false; break; }
        tc::tc_fence_after();
        issue_dq(it);
      }
    } else {
      for (int it = 0; it < n_it && ok; ++it) {
        if (!tc::mbar_wait_warp(bar(BB_PDSFULL), it & 1, status, 305)) { ok = false; break; }
        tc::tc_fence_after();
        // dQ first: its drain to shared memory (which frees the dP^T columns for the next tile) then overlaps
        // the dV and dK products
        issue_dq(it);
        issue_dk(it);
        if (leader) tc::mma_commit(bar(BB_QEMPTY));                 // Q of this tile is not read again: the next one is fetched
        issue_dv(it);                                   // while dV runs
        if (leader) tc::mma_commit(bar(BB_DOEMPTY));                // ... and dO
        if (it + 1 < n_it) {
          if (!tc::mbar_wait_warp(bar(BB_QFULL), (it + 1) & 1, status, 303)) { ok = false; break; }
          tc::tc_fence_after();
          issue_s(it + 1);                   // the S^T columns (P^T by now) were last read by dV above
          if (!tc::mbar_wait_warp(bar(BB_DQDRAINED), it & 1, status, 304)) { ok = false; break; }
          if (!tc::mbar_wait_warp(bar(BB_DOFULL), (it + 1) & 1, status, 314)) { ok = false; break; }
          tc::tc_fence_after();
          issue_dp(it + 1);                  // the dP^T columns held dQ until it was drained
        }
      }
      // dQ is issued first here, so its barrier does not cover the last tile's dK and dV products: one more
      // arrival, on the barrier the pipelined variant uses for dV, tells the epilogue that they are complete
      if (ok && n_it > 0 && leader) tc::mma_commit(bar(BB_DVDONE));
    }
  } else if (!DIRECT && warp == 18) {
    // ---- dQ reduction warp: adds each staged dQ tile to the fp32 accumulator with bulk tensor reductions ----
    if (lane == 0) {
      pdl_wait();                                    // the accumulator's zero-fill precedes the kernel before this one
      for (int dit = 0; dit < n_it; ++dit) {
        const int h = g * P.group + (it0 + dit) / per_head, i0 = (qt_begin + (it0 + dit) % per_head) * BQ;
        if (!tc::mbar_wait(bar(BB_DQSTAGED + (dit % NS)), (dit / (int)NS) & 1, status, 309)) break;   // one per buffer, like STAGEFREE
        const uint32_t stage = stage_addr(dit);
#pragma unroll
        for (int pn = 0; pn < (int)PANELS; ++pn)
          tc::tma_reduce_add_4d(&P.tdq, stage + pn * 32768, 0, 0, row0 + i0, h * (int)PANELS + pn);
        tc::bulk_commit_group();
        tc::bulk_wait_group_read0();                 // the staging tile has been read: it may be overwritten
        tc::mbar_arrive(bar(BB_STAGEFREE + (dit % NS)));     // one barrier per staging buffer: a waiter is never
                                                             // more than one phase behind
      }
      tc::bulk_wait_group0();                        // all sums are in global memory before the block exits, as in the products
    }
  } else if (warp >= 2 && warp < 18) {
    // ---- softmax warps: thread = (key row, one quarter of the 128 query columns) -----------------------
    const int q = warp % 4;                         // TMEM lane quarter
    const int part = (warp - 2) / 4;                // which 32 query columns (and which quarter of HD later)
    const int r = q * 32 + lane;
    const int t = threadIdx.x - 64;                 // 0..511
    const int gj = j0 + r;
    pdl_wait();                                     // D is written by the kernel before this one; dK, dV may still be read by it
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    const float c = P.scale * LOG2E;
    float* s_stage = reinterpret_cast<float*>(smem_raw + SM::LSE_OFF);
    bool ok = true;

    // dQ tile of iteration `dit` (row = query i0 + row): each thread copies its TMEM row segment, scaled, to a
    // staging tile in shared memory in the 128-byte-swizzled box layout of the accumulator's tensor map; the
    // reduction warp then adds the whole tile to global memory asynchronously, off the critical path.
    auto drain_dq = [&](int dit) -> bool {
      const uint32_t stage = stage_addr(dit);
      if (!tc::mbar_wait(bar(BB_DQFULL), dit & 1, status, 307)) return false;
      tc::tc_fence_after();
      // this thread's HD / 4 accumulator columns in one go; the tensor pipe gets the columns back (at HD = 128 the
      // next tile's dP^T waits for them) as soon as they are in registers, before the stores to the staging tile
      constexpr int NC = HD / 4;                     // 16 or 32 columns
      const int c0 = part * NC;
      uint32_t o[NC];
      if constexpr (NC == 32) tc::tmem_ld32(lane_addr + DQ_COL + c0, o);
      else tc::tmem_ld16(lane_addr + DQ_COL + c0, o);
      tc::tmem_ld_wait();
      tc::tc_fence_before();
      tc::mbar_arrive(bar(BB_DQDRAINED));            // TMEM side done: the tensor pipe may reuse the columns
      if constexpr (DIRECT) {
        const int h = g * P.group + (it0 + dit) / per_head, gi = (qt_begin + (it0 + dit) % per_head) * BQ + r;
        if (gi < P.t_pad) store_cols<NC>(P.dq, P.n_pad, row0 + gi, h * HD + c0, o, P.scale);
        return true;
      }
      // Only now wait for the staging buffer (its previous tile must have been read by its bulk reduction, which
      // takes a few thousand cycles): the values sit in registers meanwhile and the columns are already free.
      if (dit >= (int)NS && !stage_is_alt(dit) && !tc::mbar_wait(bar(BB_STAGEFREE + (dit % NS)), (dit / (int)NS - 1) & 1, status, 310)) return false;
#pragma unroll
      for (int u = 0; u < NC / 16; ++u) {            // 16 columns = half of a 128-byte unit of the box
        const int cu = c0 + u * 16;
        const uint32_t unit = (uint32_t)(r * 2 + (cu % 64) / 32);
        const uint32_t rowaddr = stage + (cu / 64) * 32768 + unit * 128;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t chk = (uint32_t)((cu % 32) / 4 + k);
          const uint32_t addr = rowaddr + ((chk ^ (unit & 7)) * 16);
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(__uint_as_float(o[u * 16 + 4 * k]) * P.scale),
                       "f"(__uint_as_float(o[u * 16 + 4 * k + 1]) * P.scale), "f"(__uint_as_float(o[u * 16 + 4 * k + 2]) * P.scale),
                       "f"(__uint_as_float(o[u * 16 + 4 * k + 3]) * P.scale) : "memory");
        }
      }
      tc::fence_proxy_async();
      tc::mbar_arrive(bar(BB_DQSTAGED + (dit % NS)));     // staging side done: the reduction warp takes over
      return true;
    };

    int c_q = c0_q;                                 // query tile within the head of the tile being processed
    for (int it = 0; it < n_it && ok; ++it) {
      const int i0 = (qt_begin + c_q) * BQ;
      if (++c_q == per_head) c_q = 0;
      // LSE and D of this query tile were copied to shared memory by the producer (a buffer per Q / dO stage)
      // and arrived before the score products awaited below were issued
      const float* s_lse = s_stage + (it % NQQ) * 128;
      const float* s_d = s_stage + NQQ * 128 + (it % NDO) * 128;
      if (!tc::mbar_wait(bar(BB_SFULL), it & 1, status, 306)) { ok = false; break; }
      tc::tc_fence_after();
      // element masks are needed only on the diagonal tile and on tiles with keys or queries beyond the sequence
      const bool need_mask = (P.causal && (i0 < j0 + BKV - 1)) || (j0 + BKV > P.seq_k) || (i0 + BQ > P.seq);
      const uint32_t dsrow = base + SM::DS_OFF + (it % NP) * 32768 + (part / 2) * 16384 + r * 128;
      // this thread's 32 score columns first: with HD = 128 the packed P^T overwrites S^T columns that belong to
      // other warps of the same lane quarter, so every warp must have read its scores before any P^T store
      uint32_t sv[32];
      tc::tmem_ld32(lane_addr + S_COL + part * 32, sv);
      tc::tmem_ld_wait();
      tc::tc_fence_before();
      tc::mbar_arrive(bar(BB_SREAD));                   // this thread's scores are in registers
      if (!PIPE) {
        if (!tc::mbar_wait(bar(BB_SREAD), it & 1, status, 311)) { ok = false; break; }
        tc::tc_fence_after();
      }
      if constexpr (PIPE) {
      // One 16-column chunk: P^T = exp2(S^T c - LSE) to tensor memory, dS^T = P^T (dP^T - D) to the swizzled
      // shared-memory operand tile, both rounded to bf16.  MASKED is the rare path (diagonal / ragged tiles).
      auto chunk = [&](int cc, auto masked_tag) {
        constexpr bool MASKED = decltype(masked_tag)::value;
        const int c0 = part * 32 + cc * 16;
        uint32_t pp[8], dd[8];
        // a warp whose 32 keys x 16 queries are all masked (beyond a sequence, above the diagonal) only writes zeros
        if (MASKED && warp_masked(i0 + c0, 16, j0 + q * 32, P)) {
#pragma unroll
          for (int k = 0; k < 8; ++k) pp[k] = dd[k] = 0u;
        } else {
        uint32_t dpv[16];
        tc::tmem_ld16(lane_addr + DP_COL + c0, dpv);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
          const float4 l4 = *reinterpret_cast<const float4*>(&s_lse[c0 + k]);
          const float4 d4 = *reinterpret_cast<const float4*>(&s_d[c0 + k]);
          // two-wide fp32 operations (one instruction per pair): x = S^T c - LSE log2e, then dS^T = P^T (dP^T - D)
          const float2 c2 = make_float2(c, c);
          const float2 nl2e = make_float2(-LOG2E, -LOG2E), neg1 = make_float2(-1.f, -1.f);
          const float2 x01 = __ffma2_rn(make_float2(__uint_as_float(sv[cc * 16 + k]), __uint_as_float(sv[cc * 16 + k + 1])), c2, __fmul2_rn(make_float2(l4.x, l4.y), nl2e));
          const float2 x23 = __ffma2_rn(make_float2(__uint_as_float(sv[cc * 16 + k + 2]), __uint_as_float(sv[cc * 16 + k + 3])), c2, __fmul2_rn(make_float2(l4.z, l4.w), nl2e));
          float pv[4] = {tc::fast_exp2(x01.x), tc::fast_exp2(x01.y), tc::fast_exp2(x23.x), tc::fast_exp2(x23.y)};
          if (MASKED) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int gi = i0 + c0 + k + u;
              if (gj >= P.seq_k || gi >= P.seq || (P.causal && gi < gj)) pv[u] = 0.f;
            }
          }
          const float2 g01 = __fmul2_rn(make_float2(pv[0], pv[1]), __ffma2_rn(make_float2(d4.x, d4.y), neg1, make_float2(__uint_as_float(dpv[k]), __uint_as_float(dpv[k + 1]))));
          const float2 g23 = __fmul2_rn(make_float2(pv[2], pv[3]), __ffma2_rn(make_float2(d4.z, d4.w), neg1, make_float2(__uint_as_float(dpv[k + 2]), __uint_as_float(dpv[k + 3]))));
          float gv[4] = {g01.x, g01.y, g23.x, g23.y};
          if (MASKED) {                              // LSE / D of rows past the sequence end are not defined
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int gi = i0 + c0 + k + u;
              if (gj >= P.seq_k || gi >= P.seq || (P.causal && gi < gj)) gv[u] = 0.f;
            }
          }
          pp[k / 2] = tc::pack_bf16(pv[0], pv[1]);
          pp[k / 2 + 1] = tc::pack_bf16(pv[2], pv[3]);
          dd[k / 2] = tc::pack_bf16(gv[0], gv[1]);
          dd[k / 2 + 1] = tc::pack_bf16(gv[2], gv[3]);
        }
        }
        if (PIPE && cc == 0 && it > 0) {
          // P^T has its own columns, single-buffered: the dV product of the previous tile must have read them.
          // The wait sits here, behind the first chunk's arithmetic, which needs only S^T and dP^T.
          if (!tc::mbar_wait(bar(BB_DVDONE), (it - 1) & 1, status, 312)) { ok = false; return; }
          tc::tc_fence_after();
        }
        tc::tmem_st8(lane_addr + P_COL + c0 / 2, pp);
        // 16 query columns = 2 swizzled 16-byte chunks of this key row inside its 64-query panel
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          const uint32_t chk = (uint32_t)((part % 2) * 4 + cc * 2 + ch);
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dsrow + ((chk ^ (uint32_t)(r & 7)) * 16)),
                       "r"(dd[ch * 4]), "r"(dd[ch * 4 + 1]), "r"(dd[ch * 4 + 2]), "r"(dd[ch * 4 + 3]) : "memory");
        }
      };
      if (need_mask) {
        chunk(0, std::true_type{});
        if (ok) chunk(1, std::true_type{});
      } else {
        chunk(0, std::false_type{});
        if (ok) chunk(1, std::false_type{});
      }
      } else {
      // Phase A needs only S^T: P^T = exp2(S^T c - LSE) for this thread's 32 query columns, kept in the score
      // registers as fp32 and stored to tensor memory as bf16.  It runs while the tensor pipe is still busy with
      // dP^T of this tile (which at HD = 128 also waits for the previous tile's dQ to be drained).
      auto phase_a = [&](auto masked_tag) {
        constexpr bool MASKED = decltype(masked_tag)::value;
        const float2 c2 = make_float2(c, c), nl2e = make_float2(-LOG2E, -LOG2E);
#pragma unroll
        for (int k = 0; k < 32; k += 4) {
          const float4 l4 = *reinterpret_cast<const float4*>(&s_lse[part * 32 + k]);
          const float2 x01 = __ffma2_rn(make_float2(__uint_as_float(sv[k]), __uint_as_float(sv[k + 1])), c2, __fmul2_rn(make_float2(l4.x, l4.y), nl2e));
          const float2 x23 = __ffma2_rn(make_float2(__uint_as_float(sv[k + 2]), __uint_as_float(sv[k + 3])), c2, __fmul2_rn(make_float2(l4.z, l4.w), nl2e));
          float pv[4] = {tc::fast_exp2(x01.x), tc::fast_exp2(x01.y), tc::fast_exp2(x23.x), tc::fast_exp2(x23.y)};
          if (MASKED) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int gi = i0 + part * 32 + k + u;
              if (gj >= P.seq_k || gi >= P.seq || (P.causal && gi < gj)) pv[u] = 0.f;
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) sv[k + u] = __float_as_uint(pv[u]);
        }
      };
      if (need_mask) phase_a(std::true_type{}); else phase_a(std::false_type{});
      {
        uint32_t pp[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) pp[k] = tc::pack_bf16(__uint_as_float(sv[2 * k]), __uint_as_float(sv[2 * k + 1]));
        if (PIPE && it > 0) {
          // P^T has its own columns, single-buffered: the dV product of the previous tile must have read them
          if (!tc::mbar_wait(bar(BB_DVDONE), (it - 1) & 1, status, 312)) { ok = false; break; }
          tc::tc_fence_after();
        }
        tc::tmem_st16(lane_addr + P_COL + part * 16, pp);
      }
      // Phase B: dS^T = P^T (dP^T - D), rounded to bf16, to the swizzled shared-memory operand tile, in two
      // 16-column chunks.  MASKED is the rare path (diagonal / ragged tiles).
      if (!tc::mbar_wait(bar(BB_DPFULL), it & 1, status, 316)) { ok = false; break; }
      tc::tc_fence_after();
      auto phase_b = [&](int cc, auto masked_tag) {
        constexpr bool MASKED = decltype(masked_tag)::value;
        const int c0 = part * 32 + cc * 16;
        uint32_t dpv[16];
        tc::tmem_ld16(lane_addr + DP_COL + c0, dpv);
        tc::tmem_ld_wait();
        uint32_t dd[8];
        const float2 neg1 = make_float2(-1.f, -1.f);
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
          const float4 d4 = *reinterpret_cast<const float4*>(&s_d[c0 + k]);
          const float* pv = reinterpret_cast<const float*>(&sv[cc * 16 + k]);
          const float2 g01 = __fmul2_rn(make_float2(pv[0], pv[1]), __ffma2_rn(make_float2(d4.x, d4.y), neg1, make_float2(__uint_as_float(dpv[k]), __uint_as_float(dpv[k + 1]))));
          const float2 g23 = __fmul2_rn(make_float2(pv[2], pv[3]), __ffma2_rn(make_float2(d4.z, d4.w), neg1, make_float2(__uint_as_float(dpv[k + 2]), __uint_as_float(dpv[k + 3]))));
          float gv[4] = {g01.x, g01.y, g23.x, g23.y};
          if (MASKED) {                              // LSE / D of rows past the sequence end are not defined
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int gi = i0 + c0 + k + u;
              if (gj >= P.seq_k || gi >= P.seq || (P.causal && gi < gj)) gv[u] = 0.f;
            }
          }
          dd[k / 2] = tc::pack_bf16(gv[0], gv[1]);
          dd[k / 2 + 1] = tc::pack_bf16(gv[2], gv[3]);
        }
        // 16 query columns = 2 swizzled 16-byte chunks of this key row inside its 64-query panel
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          const uint32_t chk = (uint32_t)((part % 2) * 4 + cc * 2 + ch);
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dsrow + ((chk ^ (uint32_t)(r & 7)) * 16)),
                       "r"(dd[ch * 4]), "r"(dd[ch * 4 + 1]), "r"(dd[ch * 4 + 2]), "r"(dd[ch * 4 + 3]) : "memory");
        }
      };
      if (need_mask) { phase_b(0, std::true_type{}); phase_b(1, std::true_type{}); }
      else { phase_b(0, std::false_type{}); phase_b(1, std::false_type{}); }
      }
      if (!ok) break;
      tc::tmem_st_wait();
      tc::fence_proxy_async();
      tc::tc_fence_before();
      tc::mbar_arrive(bar(BB_PDSFULL));
      if (PIPE) {
        if (it > 0) ok = drain_dq(it - 1);
      } else {
        ok = drain_dq(it);
      }
    }
    if (PIPE && ok && n_it > 0) ok = drain_dq(n_it - 1);
    // dK, dV of this key tile: every MMA has completed (HD = 64: dQ is the last product issued, and the wait for
    // it is behind us; HD = 128: the extra arrival above)
    if (!PIPE && ok && n_it > 0) ok = tc::mbar_wait(bar(BB_DVDONE), 0, status, 315);
    tc::tc_fence_after();
    if constexpr (SLICED) {
      // fp32 rows of dV, then of dK, over the operand tiles, which no product reads any more (without items: which have come)
      if (n_it <= 0) ok = tc::mbar_wait(bar(BB_KVFULL), 0, status, 316);
#pragma unroll 1
      for (int which = 0; which < 2; ++which) {
#pragma unroll 1
        for (int cc = 0; cc < HD / 64; ++cc) {
          const int c0 = part * (HD / 4) + cc * 16;
          const uint32_t at = base + ((which * BKV + r) * (HD + 4) + c0) * 4;
          if (n_it > 0) {
            uint32_t o[16];
            tc::tmem_ld16(lane_addr + (which ? DK_COL : DV_COL) + c0, o);
            tc::tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 16; k += 4)
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + k * 4), "r"(o[k]), "r"(o[k + 1]), "r"(o[k + 2]), "r"(o[k + 3]) : "memory");
          } else {
#pragma unroll
            for (int k = 0; k < 16; k += 4)
              asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(at + k * 4), "r"(0u) : "memory");
          }
        }
      }
    } else if (ok && n_it > 0) {
      const bool live = gj < P.seq_k;
#pragma unroll 1
      for (int which = 0; which < 2; ++which) {
        __nv_bfloat16* out = which ? P.dk : P.dv;
        const float f = live ? (which ? P.scale : 1.f) : 0.f;
#pragma unroll 1
        for (int cc = 0; cc < HD / 64; ++cc) {
          const int c0 = part * (HD / 4) + cc * 16;
          uint32_t o[16];
          tc::tmem_ld16(lane_addr + (which ? DK_COL : DV_COL) + c0, o);   // warp-collective: no lane may skip it
          tc::tmem_ld_wait();
          if (gj < P.t_pad_k) {
            store_cols<16>(out, P.n_pad_k, row0k + gj, g * HD + c0, o, f);
          }
        }
      }
    }
  }
  if constexpr (SLICED) {
    __syncwarp();
    tc::cluster_sync_all();
    const int rows = BKV / slices;                        // of either matrix, that this block finishes
    for (int e = threadIdx.x; e < 2 * rows * (HD / 8); e += BWD_THREADS) {
      const bool is_k = e >= rows * (HD / 8);
      const int row = slice * rows + e / (HD / 8) % rows, col = e % (HD / 8) * 8;
      const uint32_t at = base + (((is_k ? BKV : 0) + row) * (HD + 4) + col) * 4;
      float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int c = 0; c < slices; ++c) {
        const uint32_t from = tc::map_to_cta(at, c);
        float4 x, y;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(from) : "memory");
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(y.x), "=f"(y.y), "=f"(y.z), "=f"(y.w) : "r"(from + 16) : "memory");
        sum[0] += x.x; sum[1] += x.y; sum[2] += x.z; sum[3] += x.w;
        sum[4] += y.x; sum[5] += y.y; sum[6] += y.z; sum[7] += y.w;
      }
      if (j0 + row >= P.t_pad_k) continue;
      const float f = j0 + row < P.seq_k ? (is_k ? P.scale : 1.f) : 0.f;
      uint4 v;
      v.x = tc::pack_bf16(sum[0] * f, sum[1] * f); v.y = tc::pack_bf16(sum[2] * f, sum[3] * f);
      v.z = tc::pack_bf16(sum[4] * f, sum[5] * f); v.w = tc::pack_bf16(sum[6] * f, sum[7] * f);
      const int cg = g * HD + col;
      *reinterpret_cast<uint4*>((is_k ? P.dk : P.dv) + ((long long)(cg / 64) * P.n_pad_k + row0k + j0 + row) * 64 + cg % 64) = v;
    }
    __syncwarp();
    tc::cluster_sync_all();                               // no block leaves while another may still read its sums
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem_base, TMEM_COLS);
}

// ---------------------------------------------------------------------------------------------------
// Backward of short sequences (two key tiles, at most two query tiles, head_dim 64, a KV head per query head): one block
// per (head, sequence) takes all their tile pairs.  K, V, Q and dO are loaded once and stay in shared memory; dQ of both
// query tiles accumulates in tensor memory over the key tiles and goes out rounded, so there is no fp32 accumulator, no
// zero-fill and no rounding pass; dV and dK of a key tile are copied out while the next key tile's scores are at work.
// The roles and the per-tile schedule are those of the pipelined variant above, except that P^T goes through shared
// memory like dS^T: tensor memory is full (S^T, dP^T, dV, dK and two dQ tiles are 512 columns).
// Bound: start-up and drain of a block against its three or four tiles of softmax arithmetic; one block does both key
// tiles' with one start-up, half the loads and no bulk reductions.
// ---------------------------------------------------------------------------------------------------
struct ShortSmem {
  static constexpr uint32_t TILE = 16384;                                // 128 rows x 64 bf16
  static constexpr uint32_t K_OFF = 0, V_OFF = 2 * TILE, Q_OFF = 4 * TILE, DO_OFF = 6 * TILE;
  static constexpr uint32_t DS_OFF = 8 * TILE, P_OFF = DS_OFF + 2 * 32768;
  static constexpr uint32_t LSE_OFF = P_OFF + 32768, D_OFF = LSE_OFF + 2 * 512, BAR_OFF = D_OFF + 2 * 512;
  static constexpr uint32_t N_BARS = 16, TOTAL = BAR_OFF + 8 * N_BARS + 16;
};
enum { SB_KVFULL = 0, SB_QFULL = 2, SB_DOFULL = 4, SB_SFULL = 6, SB_SREAD, SB_PDSFULL, SB_DVDONE, SB_DQDONE, SB_DKDONE, SB_KVDRAINED, SB_FINAL };
constexpr int SHORT_THREADS = 576;       // warp 0 TMA loads, warp 1 MMA, warps 2-17 softmax

__global__ void __launch_bounds__(SHORT_THREADS, 1) attn_bwd_short_kernel(const __grid_constant__ AttnBwdParams P) {
  using SM = ShortSmem;
  constexpr int HD = 64;
  constexpr uint32_t S_COL = 0, DP_COL = 128, DV_COL = 256, DK_COL = 320, DQ_COL = 384, TMEM_COLS = 512;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = tc::smem_u32(smem_raw);
  const uint32_t bars = base + SM::BAR_OFF, slot = bars + 8 * SM::N_BARS;
  auto bar = [&](int i) { return bars + 8u * i; };
  const int warp = (int)tc::uniform(threadIdx.x / 32), lane = threadIdx.x % 32;
  const int h = blockIdx.x % P.hq, b = blockIdx.x / P.hq;
  const int row0 = b * P.t_pad, row0k = b * P.t_pad_k;
  const int n_qt = (P.seq + BQ - 1) / BQ, n_kt = (P.seq_k + BKV - 1) / BKV;
  const int i1 = P.causal ? 1 : 0;                                       // first query tile of key tile 1
  const int n0 = n_qt, n_it = n0 + (n_kt > 1 ? n_qt - i1 : 0);           // tile pairs: key tile 0's, then key tile 1's
  auto key_tile = [&](int it) { return it < n0 ? 0 : 1; };
  auto query_tile = [&](int it) { return it < n0 ? it : it - n0 + i1; };
  int32_t* status = P.status;
  if ((base & 1023u) != 0) {
    if (threadIdx.x == 0) atomicCAS(status, 0, 398);
    return;
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(bar(SB_KVFULL + s), 1);
      tc::mbar_init(bar(SB_QFULL + s), 1);
      tc::mbar_init(bar(SB_DOFULL + s), 1);
    }
    tc::mbar_init(bar(SB_SFULL), 1);
    tc::mbar_init(bar(SB_SREAD), BWD_SM_THREADS);
    tc::mbar_init(bar(SB_PDSFULL), BWD_SM_THREADS);
    tc::mbar_init(bar(SB_DVDONE), 1);
    tc::mbar_init(bar(SB_DQDONE), 1);
    tc::mbar_init(bar(SB_DKDONE), 1);
    tc::mbar_init(bar(SB_KVDRAINED), BWD_SM_THREADS);
    tc::mbar_init(bar(SB_FINAL), 1);
    tc::fence_barrier_init();
    // forward-pass data: requested before the allocation, the block barrier and the wait for the kernel in front
    tc::tma_prefetch_desc(&P.tk); tc::tma_prefetch_desc(&P.tv); tc::tma_prefetch_desc(&P.tq); tc::tma_prefetch_desc(&P.tdo);
    for (int t = 0; t < 2; ++t) {
      if (t < n_kt) {
        tc::mbar_expect_tx(bar(SB_KVFULL + t), 2 * SM::TILE);
        tc::tma_load_3d(base + SM::K_OFF + t * SM::TILE, &P.tk, bar(SB_KVFULL + t), 0, row0k + t * BKV, h);
        tc::tma_load_3d(base + SM::V_OFF + t * SM::TILE, &P.tv, bar(SB_KVFULL + t), 0, row0k + t * BKV, h);
      }
      if (t < n_qt) {
        tc::mbar_expect_tx(bar(SB_QFULL + t), SM::TILE + 512);
        tc::tma_load_3d(base + SM::Q_OFF + t * SM::TILE, &P.tq, bar(SB_QFULL + t), 0, row0 + t * BQ, h);
        tc::bulk_load(base + SM::LSE_OFF + t * 512, P.lse + ((long long)b * P.hq + h) * P.t_pad + t * BQ, 512, bar(SB_QFULL + t));
      }
    }
  }
  if (warp == 1) {
    tc::tmem_alloc(slot, TMEM_COLS);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  uint32_t tmem_base;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(slot));
  tmem_base = tc::uniform(tmem_base);
  pdl_launch_dependents();

  if (warp == 0 && lane == 0) {
    pdl_wait();                                          // dO and D come from the kernel in front
    for (int t = 0; t < n_qt; ++t) {
      tc::mbar_expect_tx(bar(SB_DOFULL + t), SM::TILE + 512);
      tc::tma_load_3d(base + SM::DO_OFF + t * SM::TILE, &P.tdo, bar(SB_DOFULL + t), 0, row0 + t * BQ, h);
      tc::bulk_load(base + SM::D_OFF + t * 512, P.dvec + ((long long)b * P.hq + h) * P.t_pad + t * BQ, 512, bar(SB_DOFULL + t));
    }
  } else if (warp == 1) {
    const bool leader = tc::elect_one();
    // ---- MMA issuer ----
    const uint32_t idesc_s = tc::idesc_bf16(BKV, BQ, 0, 0), idesc_kv = tc::idesc_bf16(BKV, HD, 0, 1), idesc_dq = tc::idesc_bf16(BQ, HD, 1, 1);
    const uint32_t hi = tc::smem_desc_hi(1024), TW = SM::TILE >> 4;
    const uint32_t k_km = tc::smem_desc_lo(base + SM::K_OFF, 16), k_mn = tc::smem_desc_lo(base + SM::K_OFF, 16384);
    const uint32_t v_km = tc::smem_desc_lo(base + SM::V_OFF, 16);
    const uint32_t q_km = tc::smem_desc_lo(base + SM::Q_OFF, 16), q_mn = tc::smem_desc_lo(base + SM::Q_OFF, 16384);
    const uint32_t do_km = tc::smem_desc_lo(base + SM::DO_OFF, 16), do_mn = tc::smem_desc_lo(base + SM::DO_OFF, 16384);
    const uint32_t ds_km = tc::smem_desc_lo(base + SM::DS_OFF, 16), ds_mn = tc::smem_desc_lo(base + SM::DS_OFF, 16384);
    const uint32_t p_km = tc::smem_desc_lo(base + SM::P_OFF, 16);
    auto scores = [&](uint32_t col, uint32_t a, uint32_t q) {            // S^T = K Q^T, dP^T = V dO^T
      if (!leader) return;
#pragma unroll
      for (uint32_t kk = 0; kk < 4; ++kk) tc::mma_bf16_ss_w(tmem_base + col, a + kk * 2, hi, q + kk * 2, hi, idesc_s, kk > 0);
    };
    auto product = [&](uint32_t col, uint32_t a, uint32_t q, bool more) {  // dV += P^T dO, dK += dS^T Q
      if (!leader) return;
#pragma unroll
      for (uint32_t kk = 0; kk < 8; ++kk)
        tc::mma_bf16_ss_w(tmem_base + col, a + (kk / 4) * 1024 + (kk % 4) * 2, hi, q + kk * 128, hi, idesc_kv, more || kk > 0);
    };
    bool ok = tc::mbar_wait_warp(bar(SB_KVFULL), 0, status, 321) && tc::mbar_wait_warp(bar(SB_QFULL), 0, status, 322) &&
              tc::mbar_wait_warp(bar(SB_DOFULL), 0, status, 323);
    if (ok) {
      tc::tc_fence_after();
      scores(S_COL, k_km, q_km);
      scores(DP_COL, v_km, do_km);
      if (leader) tc::mma_commit(bar(SB_SFULL));
    }
    for (int it = 0; it < n_it && ok; ++it) {
      const int j = key_tile(it), i = query_tile(it);
      const bool next = it + 1 < n_it;
      const int jn = next ? key_tile(it + 1) : 0, in = next ? query_tile(it + 1) : 0;
      if (next) {                                        // S^T of the next pair once every warp holds this one's scores
        if (!tc::mbar_wait_warp(bar(SB_SREAD), it & 1, status, 324)) break;
        if (!tc::mbar_wait_warp(bar(SB_QFULL + in), 0, status, 322) || !tc::mbar_wait_warp(bar(SB_KVFULL + jn), 0, status, 321)) break;
        tc::tc_fence_after();
        scores(S_COL, k_km + jn * TW, q_km + in * TW);
      }
      if (!tc::mbar_wait_warp(bar(SB_PDSFULL), it & 1, status, 325)) break;
      tc::tc_fence_after();
      if (next) {
        if (!tc::mbar_wait_warp(bar(SB_DOFULL + in), 0, status, 323)) break;
        tc::tc_fence_after();
        scores(DP_COL, v_km + jn * TW, do_km + in * TW);
        if (leader) tc::mma_commit(bar(SB_SFULL));
      }
      if (it == n0 && !tc::mbar_wait_warp(bar(SB_KVDRAINED), 0, status, 326)) break;   // key tile 0's dV, dK are copied out
      tc::tc_fence_after();
      const bool more = it != 0 && it != n0;
      product(DV_COL, p_km, do_mn + i * TW, more);
      if (leader) tc::mma_commit(bar(SB_DVDONE));
      product(DK_COL, ds_km + (it & 1) * 2048, q_mn + i * TW, more);
      if (it + 1 == n0 && leader) tc::mma_commit(bar(SB_DKDONE));
#pragma unroll
      for (uint32_t kk = 0; kk < 8 && leader; ++kk)      // dQ += dS K: the dS^T tile read MN-major
        tc::mma_bf16_ss_w(tmem_base + DQ_COL + i * 64, ds_mn + (it & 1) * 2048 + kk * 128, hi, k_mn + j * TW + kk * 128, hi, idesc_dq,
                          (j > 0 || kk > 0) ? 1u : 0u);
      if (leader) tc::mma_commit(bar(SB_DQDONE));
      if (!next && leader) tc::mma_commit(bar(SB_FINAL));
    }
  } else if (warp >= 2) {
    // ---- softmax warps: thread = (key row, one quarter of the 128 query columns) ----
    const int q = warp % 4, part = (warp - 2) / 4, r = q * 32 + lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    const float c = P.scale * LOG2E;
    const float* s_lse = reinterpret_cast<const float*>(smem_raw + SM::LSE_OFF);
    const float* s_d = reinterpret_cast<const float*>(smem_raw + SM::D_OFF);
    pdl_wait();                                          // before this role writes anything
    bool ok = true;
    auto copy_kv = [&](int j) {                          // dV, dK of key tile j: 16 columns each per thread
      const int gj = j * BKV + r;
      const bool live = gj < P.seq_k;
#pragma unroll 1
      for (int which = 0; which < 2; ++which) {
        uint32_t o[16];
        tc::tmem_ld16(lane_addr + (which ? DK_COL : DV_COL) + part * 16, o);
        tc::tmem_ld_wait();
        if (gj < P.t_pad_k) store_cols<16>(which ? P.dk : P.dv, P.n_pad_k, row0k + gj, h * HD + part * 16, o, live ? (which ? P.scale : 1.f) : 0.f);
      }
    };
    for (int it = 0; it < n_it && ok; ++it) {
      const int j0 = key_tile(it) * BKV, i = query_tile(it), i0 = i * BQ, gj = j0 + r;
      if (!tc::mbar_wait(bar(SB_SFULL), it & 1, status, 327)) { ok = false; break; }
      tc::tc_fence_after();
      const bool need_mask = (P.causal && i0 < j0 + BKV - 1) || j0 + BKV > P.seq_k || i0 + BQ > P.seq;
      uint32_t sv[32];
      tc::tmem_ld32(lane_addr + S_COL + part * 32, sv);
      tc::tmem_ld_wait();
      tc::tc_fence_before();
      tc::mbar_arrive(bar(SB_SREAD));
      const uint32_t row_off = (uint32_t)(part / 2) * 16384 + r * 128;
      auto chunk = [&](int cc, auto masked_tag) {
        constexpr bool MASKED = decltype(masked_tag)::value;
        const int c0 = part * 32 + cc * 16;
        uint32_t pp[8], dd[8];
        if (MASKED && warp_masked(i0 + c0, 16, j0 + q * 32, P)) {
#pragma unroll
          for (int k = 0; k < 8; ++k) pp[k] = dd[k] = 0u;
        } else {
          uint32_t dpv[16];
          tc::tmem_ld16(lane_addr + DP_COL + c0, dpv);
          tc::tmem_ld_wait();
          const float2 c2 = make_float2(c, c), nl2e = make_float2(-LOG2E, -LOG2E), neg1 = make_float2(-1.f, -1.f);
#pragma unroll
          for (int k = 0; k < 16; k += 2) {
            const float2 l = *reinterpret_cast<const float2*>(&s_lse[i * 128 + c0 + k]);
            const float2 d = *reinterpret_cast<const float2*>(&s_d[i * 128 + c0 + k]);
            const float2 x = __ffma2_rn(make_float2(__uint_as_float(sv[cc * 16 + k]), __uint_as_float(sv[cc * 16 + k + 1])), c2, __fmul2_rn(l, nl2e));
            float pv[2] = {tc::fast_exp2(x.x), tc::fast_exp2(x.y)};
            const float2 gd = __ffma2_rn(d, neg1, make_float2(__uint_as_float(dpv[k]), __uint_as_float(dpv[k + 1])));
            float gv[2] = {pv[0] * gd.x, pv[1] * gd.y};
            if (MASKED) {                                // LSE / D of rows past the sequence end are not defined
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const int gi = i0 + c0 + k + u;
                if (gj >= P.seq_k || gi >= P.seq || (P.causal && gi < gj)) pv[u] = gv[u] = 0.f;
              }
            }
            pp[k / 2] = tc::pack_bf16(pv[0], pv[1]);
            dd[k / 2] = tc::pack_bf16(gv[0], gv[1]);
          }
        }
        if (cc == 0 && it > 0) {                         // dV of the pair before has read P^T
          if (!tc::mbar_wait(bar(SB_DVDONE), (it - 1) & 1, status, 328)) { ok = false; return; }
        }
        const uint32_t ds = base + SM::DS_OFF + (it & 1) * 32768 + row_off, pt = base + SM::P_OFF + row_off;
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          const uint32_t at = (((uint32_t)((part % 2) * 4 + cc * 2 + ch) ^ (uint32_t)(r & 7)) * 16);
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(pt + at), "r"(pp[ch * 4]), "r"(pp[ch * 4 + 1]), "r"(pp[ch * 4 + 2]), "r"(pp[ch * 4 + 3]) : "memory");
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ds + at), "r"(dd[ch * 4]), "r"(dd[ch * 4 + 1]), "r"(dd[ch * 4 + 2]), "r"(dd[ch * 4 + 3]) : "memory");
        }
      };
      if (need_mask) {
        chunk(0, std::true_type{});
        if (ok) chunk(1, std::true_type{});
      } else {
        chunk(0, std::false_type{});
        if (ok) chunk(1, std::false_type{});
      }
      if (!ok) break;
      // dK and dQ of the pair before are complete before this pair's products can be issued: the dS^T buffer of the pair
      // after this one is free, and no warp falls a phase behind on this barrier
      if (it > 0 && !tc::mbar_wait(bar(SB_DQDONE), (it - 1) & 1, status, 329)) { ok = false; break; }
      tc::fence_proxy_async();
      tc::tc_fence_before();
      tc::mbar_arrive(bar(SB_PDSFULL));
      if (it == n0) {                                    // key tile 0's sums, while the tensor pipe has the next scores to do
        if (!tc::mbar_wait(bar(SB_DKDONE), 0, status, 330)) { ok = false; break; }
        tc::tc_fence_after();
        copy_kv(0);
        tc::tc_fence_before();
        tc::mbar_arrive(bar(SB_KVDRAINED));
      }
    }
    if (ok) ok = tc::mbar_wait(bar(SB_FINAL), 0, status, 331);
    tc::tc_fence_after();
    if (ok) {
      copy_kv(n_kt - 1);
      for (int i = 0; i < n_qt; ++i) {
        const int gi = i * BQ + r;
        uint32_t o[16];
        tc::tmem_ld16(lane_addr + DQ_COL + i * 64 + part * 16, o);
        tc::tmem_ld_wait();
        if (gi < P.t_pad) store_cols<16>(P.dq, P.n_pad, row0 + gi, h * HD + part * 16, o, P.scale);
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem_base, TMEM_COLS);
}


template <int HD, bool DIRECT>
cudaError_t bwd_make_t(AttnLaunch<AttnBwdParams>& L, const fbl_plan* p) {
  // Q, dO (bf16) and the fp32 dQ accumulator of the query heads of one KV head.  The HD = 128 variant waits for
  // its single-buffered Q / dO tiles on the critical path, so it keeps the blocks that share those tiles close
  // together (small chunks: L2 hits); the pipelined HD = 64 variant hides that latency and prefers balance.
  L.P.chunk = chunk_for((long long)p->group * p->d.seq * HD * 8, p->d.n_kv_heads * p->d.batch,
                        BwdSmem<HD>::PIPE ? (96ll << 20) : (8ll << 20));
  // slices of a key tile's items: at least two items each, and no more blocks than seven eighths of the SMs, on which all
  // clusters still find room at once
  const int blocks = ((p->t_pad_kv + BKV - 1) / BKV) * p->d.n_kv_heads * p->d.batch, items = (p->d.seq + BQ - 1) / BQ * p->group;
  int slices = 1;
  while (slices < 8 && 4 * slices <= items && 16ll * blocks * slices <= 7 * p->sm_count) slices *= 2;
  if (slices == 1) return L.set(attn_bwd_tc_kernel<HD, DIRECT, false>, blocks, BWD_THREADS, BwdSmem<HD>::TOTAL);
  L.P.slices = slices;
  return L.set(attn_bwd_tc_kernel<HD, DIRECT, true>, blocks * slices, BWD_THREADS, BwdSmem<HD>::TOTAL, slices);
}

template <int HD>
cudaError_t bwd_make(AttnLaunch<AttnBwdParams>& L, const fbl_plan* p, const void* Q, const void* K, const void* V, const void* dA,
                     float* dqacc) {
  AttnBwdParams& P = L.P;
  memset(&P, 0, sizeof(P));
  const int panels = HD / 64;
  if (!fbl_encode_rtile_map(&P.tq, Q, p->n_pad, p->dq / 64, BQ, panels)) return cudaErrorInvalidValue;
  if (!fbl_encode_rtile_map(&P.tdo, dA, p->n_pad, p->dq / 64, BQ, panels)) return cudaErrorInvalidValue;
  if (!fbl_encode_rtile_map(&P.tk, K, p->n_pad_kv, p->dkv / 64, BKV, panels)) return cudaErrorInvalidValue;
  if (!fbl_encode_rtile_map(&P.tv, V, p->n_pad_kv, p->dkv / 64, BKV, panels)) return cudaErrorInvalidValue;
  const bool direct = attn_bwd_tc_direct(p);
  if (!direct && !fbl_encode_f32_panel_map(&P.tdq, dqacc, p->n_pad, p->dq / 64, BQ)) return cudaErrorInvalidValue;
  P.n_pad = p->n_pad; P.seq = p->d.seq; P.t_pad = p->t_pad; P.hq = p->d.n_q_heads; P.group = p->group;
  P.causal = p->d.causal; P.dkv = p->dkv; P.scale = p->scale;
  P.n_pad_k = p->n_pad_kv; P.seq_k = p->seq_kv; P.t_pad_k = p->t_pad_kv;
  P.batch = p->d.batch;
  if (!direct) return bwd_make_t<HD, false>(L, p);
  if (p->t_pad_kv <= BKV) return bwd_make_t<HD, true>(L, p);
  return L.set(attn_bwd_short_kernel, P.hq * P.batch, SHORT_THREADS, ShortSmem::TOTAL);
}

}  // namespace

// Every block of the backward sees all keys of its queries, and writes dQ itself: sequences of one key tile, or of two key
// and at most two query tiles where every query head has its own keys and head_dim is 64 (attn_bwd_short_kernel).
bool attn_bwd_tc_direct(const fbl_plan* p) {
  if (p->t_pad_kv <= BKV) return true;
  return p->d.head_dim == 64 && p->group == 1 && p->t_pad_kv <= 2 * BKV && p->t_pad <= 2 * BQ;
}

cudaError_t launch_attn_fwd_tc(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse,
                               int32_t* status, cudaStream_t st) {
  typedef AttnLaunch<AttnFwdParams> Launch;
  return LaunchMemo<Launch, 2>::run(p, FBL_MEMO_TC_FWD, LaunchKey(),                // its shape is the plan's
      [&](Launch& L) { return p->d.head_dim == 64 ? fwd_make<64>(L, p, Q, K, V) : fwd_make<128>(L, p, Q, K, V); },
      [&](Launch& L) {
        L.P.a = (__nv_bfloat16*)A; L.P.lse = lse; L.P.status = status;
        return fbl_map_set_base(&L.P.tq, Q) && fbl_map_set_base(&L.P.tk, K) && fbl_map_set_base(&L.P.tv, V);
      },
      [&](const Launch& L) { return launch_pdl(L.kernel, dim3(L.grid), dim3(L.threads), L.smem, st, L.P); });
}

cudaError_t launch_attn_bwd_tc(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* A,
                               const void* dA, const float* lse, float* dvec, float* dqacc, void* dQ, void* dK,
                               void* dV, bool dvec_ready, int32_t* status, cudaStream_t st, const float2* rope) {
  // D = rowsum(dO * O) unless the dA GEMM's epilogue already produced it
  cudaError_t e = launch_attn_bwd_pre(p, A, dA, dvec, dvec_ready, st);
  if (e != cudaSuccess) return e;
  typedef AttnLaunch<AttnBwdParams> Launch;
  e = LaunchMemo<Launch, 2>::run(p, FBL_MEMO_TC_BWD, LaunchKey(),
      [&](Launch& L) { return p->d.head_dim == 64 ? bwd_make<64>(L, p, Q, K, V, dA, dqacc) : bwd_make<128>(L, p, Q, K, V, dA, dqacc); },
      [&](Launch& L) {
        AttnBwdParams& P = L.P;
        P.lse = lse; P.dvec = dvec; P.dqacc = dqacc; P.dq = (__nv_bfloat16*)dQ; P.dk = (__nv_bfloat16*)dK; P.dv = (__nv_bfloat16*)dV;
        P.status = status;
        return fbl_map_set_base(&P.tq, Q) && fbl_map_set_base(&P.tdo, dA) && fbl_map_set_base(&P.tk, K) && fbl_map_set_base(&P.tv, V) &&
               (attn_bwd_tc_direct(p) || fbl_map_set_base(&P.tdq, dqacc));
      },
      [&](const Launch& L) {
        return L.cluster ? launch_cluster(L.kernel, dim3(L.grid), dim3(L.threads), L.smem, st, L.cluster, true, L.P)
                         : launch_pdl(L.kernel, dim3(L.grid), dim3(L.threads), L.smem, st, L.P);
      });
  if (e != cudaSuccess) return e;
  // dQ: fp32 accumulator -> storage dtype where the kernel has not written it; with the rotary embedding (`rope`: the
  // forward's table) dQ and dK are turned back by the opposite angle on the way
  if (attn_bwd_tc_direct(p)) return rope ? launch_rope(p, dQ, p->d.n_q_heads, dK, p->d.n_kv_heads, 1, st) : cudaSuccess;
  if (rope) return launch_rope_bwd_round(p, dqacc, dQ, dK, rope, st);
  return launch_attn_bwd_post(p, dqacc, dQ, st);
}

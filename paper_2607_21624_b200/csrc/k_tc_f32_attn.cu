// fp32 attention on the tensor cores, with the accuracy of fp32 arithmetic: every operand of a product goes in as three bf16
// parts and six tcgen05 products take the multiply-adds' place, as in k_tc_f32.cu (see there for what is lost and what is not).
// An accumulator holds one 64-key tile's product, or half of a score's, and is then added to sums in registers, so that no value
// passes more than four (two) accumulations at its full size before it is rounded to nearest.  Forward and backward form the same
// scores in the same order: P = exp(S - LSE) depends on it.  Softmax is fp32.  Heads of 128 stay on the FP32 pipe
// (k_ffma_attn.cu): their scores would take eight, and the backward there forms P from its own scores and this kernel's LSE
// (dQ, dK, dV off by 1.0e-6 of their norm instead of 6e-7 where scores are large).
#include <float.h>
#include <string.h>

#include "fbl_internal.h"
#include "launch_memo.h"
#include "pdl.cuh"
#include "tc_common.cuh"

namespace {

// What each operand is raised by (tc::split3).  A score is summed over half of head_dim (one or two full-size additions), P V, dV and
// dK over 64 rows, dQ over 32: Q + K = the scores' loss, V (backward) + dO = the same, P + dO = dS + Q = that of 64, dS + K = that
// of 32.
template <int HD>
struct Lift {
  static constexpr float S = HD == 64 ? tc::LIFT_2 : tc::LIFT_1;
  static constexpr float Q = 0.5f * (tc::LIFT_4 + S - tc::LIFT_2), K = S - Q, V = S, P = tc::LIFT_4, DS = tc::LIFT_4 - Q;
};

struct alignas(64) F32FwdParams {
  CUtensorMap tq, tk, tv;
  const float *q, *k, *v;       // the same operands, for blocks that are worked through by plain arithmetic
  float* a;                     // merged-head output [n_pad, dq]
  float* lse;                   // [B, Hq, t_pad]
  long long n_pad, n_pad_k;
  int seq, t_pad, seq_k, t_pad_k, hq, group, causal;
  float scale;
  int32_t* status;
};

// ------------------------------------------------------------------------------------------
// Forward: one block per (128 queries, head, batch), 64 keys at a time.  14 warps: one loads fp32 tiles by TMA, one issues the
// products, eight have two threads to a query row (half of the keys' scores and of the output's columns each; they meet for the
// row maximum) and four turn K and V into bf16 parts in shared memory (K-major and MN-major as they lie).  Q's and P's parts are
// operands in tensor memory.  The scores of the next tile and the output of this one are products under way while the softmax
// works; the products alone, 24 + 24 instructions a tile at head_dim 64, are some 2300 clk (counted on short chains, 48 heads of 197
// tokens: tensor pipe active for 23 % of active cycles, the start and the conversions the rest).
// ------------------------------------------------------------------------------------------
constexpr int QT = 128, KT = 64;
constexpr int SOFT_WARPS = 8, CONV_WARPS = 4, FWD_THREADS = 32 * (2 + SOFT_WARPS + CONV_WARPS);

template <int HD>
struct FwdSmem {
  static constexpr int NB = 2, NS = 2;                       // K and V tiles, fp32 and parts; score accumulators
  static constexpr uint32_t RAW = KT * HD * 4, PART = KT * 128, PARTS = 3 * PART;
  static constexpr uint32_t Q_OFF = 0, K_OFF = QT * HD * 4, V_OFF = K_OFF + NB * RAW;
  static constexpr uint32_t KP_OFF = V_OFF + NB * RAW, VP_OFF = KP_OFF + NB * PARTS;
  static constexpr uint32_t MAX_OFF = Q_OFF;                 // [2 tiles][2 halves][128 rows] of row maxima (the sums at the end), over Q,
                                                             // which is in parts before there is a score
  static constexpr uint32_t BAR_OFF = VP_OFF + NB * PARTS, N_BARS = 8 * NB + 2 * NS + 8;
  static constexpr uint32_t TOTAL = BAR_OFF + 8 * N_BARS + 16 + 1024;      // + tensor memory slot, flag, alignment slack
  // tensor memory: score accumulators (two to a tile, for the halves of head_dim), Q's parts, P's parts, the output accumulator
  static constexpr uint32_t S_COL = 0, QP_COL = 2 * NS * KT, P_COL = QP_COL + 3 * HD / 2, O_COL = P_COL + 96;
  static_assert(O_COL + HD <= 512, "tensor memory columns");
};

// A block's rows by plain arithmetic, where an operand is out of range (tc::probe_range), so that a score is never more than the
// products can form: the threads that are left when the others' work is
// done, two to a query row (half of the keys' scores and of the output's columns each), tiles of 64 keys in shared memory.  A key
// that the mask leaves out takes no part, whatever it holds.
template <int HD>
__device__ __noinline__ void plain_rows(const F32FwdParams& P, uint32_t base, int i0, int h, int b) {
  constexpr int LD = HD + 4, LDP = KT + 1, N = HD / 4, HC = HD / 2;      // row pitches that keep a warp's rows on different banks
  const uint32_t sq = base, sk = sq + QT * LD * 4, sv = sk + KT * HD * 4, sp = sv + KT * HD * 4, sm = sp + QT * LDP * 4;
  static_assert((QT * LD + 2 * KT * HD + QT * LDP + 2 * QT) * 4 <= (int)FwdSmem<HD>::BAR_OFF, "shared memory");
  const int r = threadIdx.x % QT, half = threadIdx.x / QT, gi = i0 + r, g = h / P.group;
  const bool work = threadIdx.x < 2 * QT;
  auto fill = [&](uint32_t to, int ld, int rows, const float* m, long long n_pad, int t_pad, int row0, int end, int col) {
    for (int e = threadIdx.x; e < rows * N; e += FWD_THREADS) {
      const int row = e / N, c = e % N * 4;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row0 + row < end) x = *reinterpret_cast<const float4*>(m + rt_off<32>(n_pad, (long long)b * t_pad + row0 + row, col + c));
      asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(to + (row * ld + c) * 4), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w) : "memory");
    }
  };
  fill(sq, LD, QT, P.q, P.n_pad, P.t_pad, i0, P.seq, h * HD);
  const int j_end = P.causal ? min(P.seq_k, i0 + QT) : P.seq_k, mine_end = P.causal ? min(P.seq_k, gi + 1) : P.seq_k;
  float m = -INFINITY, l = 0.f, o[HC];
#pragma unroll
  for (int c = 0; c < HC; ++c) o[c] = 0.f;
#pragma unroll 1
  for (int j0 = 0; j0 < j_end; j0 += KT) {
    __syncthreads();
    fill(sk, HD, KT, P.k, P.n_pad_k, P.t_pad_k, j0, P.seq_k, g * HD);
    fill(sv, HD, KT, P.v, P.n_pad_k, P.t_pad_k, j0, P.seq_k, g * HD);
    __syncthreads();
    float s[KT / 2], mx = -INFINITY;
    if (work) {
#pragma unroll
      for (int k = 0; k < KT / 2; ++k) s[k] = 0.f;
#pragma unroll 1
      for (int d = 0; d < HD; d += 4) {
        const float4 q = tc::lds4(sq + (r * LD + d) * 4);
#pragma unroll
        for (int k = 0; k < KT / 2; ++k) {
          const float4 x = tc::lds4(sk + ((half * 32 + k) * HD + d) * 4);
          s[k] = fmaf(q.x, x.x, fmaf(q.y, x.y, fmaf(q.z, x.z, fmaf(q.w, x.w, s[k]))));
        }
      }
#pragma unroll
      for (int k = 0; k < KT / 2; ++k) {
        s[k] = j0 + half * 32 + k < mine_end ? s[k] * P.scale : -INFINITY;
        mx = fmaxf(mx, s[k]);
      }
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(sm + threadIdx.x * 4), "f"(mx) : "memory");
    }
    __syncthreads();
    float alpha = 1.f;
    if (work) {
      float mo;
      asm volatile("ld.shared.f32 %0, [%1];" : "=f"(mo) : "r"(sm + ((half ^ 1) * QT + r) * 4) : "memory");
      const float m_new = fmaxf(m, fmaxf(mx, mo));
      alpha = m_new == -INFINITY ? 1.f : expf(m - m_new);
      m = m_new;
      float sum = 0.f;
#pragma unroll
      for (int k = 0; k < KT / 2; ++k) {
        const float p = m == -INFINITY || j0 + half * 32 + k >= mine_end ? 0.f : expf(s[k] - m);
        sum += p;
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(sp + (r * LDP + half * 32 + k) * 4), "f"(p) : "memory");
      }
      l = l * alpha + sum;
    }
    __syncthreads();
    if (work) {
#pragma unroll
      for (int c = 0; c < HC; ++c) o[c] *= alpha;
#pragma unroll 1
      for (int k = 0; k < min(KT, mine_end - j0); ++k) {
        float p;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(p) : "r"(sp + (r * LDP + k) * 4) : "memory");
#pragma unroll
        for (int c = 0; c < HC; c += 4) {
          const float4 v = tc::lds4(sv + (k * HD + half * HC + c) * 4);
          o[c] = fmaf(p, v.x, o[c]); o[c + 1] = fmaf(p, v.y, o[c + 1]); o[c + 2] = fmaf(p, v.z, o[c + 2]); o[c + 3] = fmaf(p, v.w, o[c + 3]);
        }
      }
    }
  }
  __syncthreads();
  if (work) asm volatile("st.shared.f32 [%0], %1;" ::"r"(sm + threadIdx.x * 4), "f"(l) : "memory");
  __syncthreads();
  if (!work || gi >= P.seq) return;
  float lo;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(lo) : "r"(sm + ((half ^ 1) * QT + r) * 4) : "memory");
  l = half ? lo + l : l + lo;
  const float inv = 1.f / l;
#pragma unroll
  for (int c = 0; c < HC; c += 4)
    *reinterpret_cast<float4*>(P.a + rt_off<32>(P.n_pad, (long long)b * P.t_pad + gi, h * HD + half * HC + c)) =
        make_float4(o[c] * inv, o[c + 1] * inv, o[c + 2] * inv, o[c + 3] * inv);
  if (half == 0) P.lse[((long long)b * P.hq + h) * P.t_pad + gi] = m + logf(l);
}

// One 16-value piece of a row of an fp32 tile as TMA leaves it (`rows` rows to a 32-column panel) -> three parts, each a bf16
// tile of 64-column panels in the canonical 128-byte-swizzled layout.
__device__ __forceinline__ void convert_piece(uint32_t src, uint32_t dst, uint32_t part, int rows, int r, int piece, float lift, float2& probe) {
  const uint32_t from = src + (piece / 2) * (rows * 128) + r * 128, to = dst + (piece / 4) * (rows * 128) + r * 128;
  float x[16];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float4 v = tc::lds4(from + (((piece % 2 * 4 + c) ^ (r & 7)) << 4));
    x[4 * c] = v.x; x[4 * c + 1] = v.y; x[4 * c + 2] = v.z; x[4 * c + 3] = v.w;
  }
  uint32_t p[3][8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    tc::split3(x[2 * k], x[2 * k + 1], lift, p[0][k], p[1][k], p[2][k]);
    tc::probe_range(x[2 * k], x[2 * k + 1], probe);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int c = 0; c < 2; ++c) tc::sts4(to + i * part + (((piece % 4 * 2 + c) ^ (r & 7)) << 4), &p[i][4 * c]);
}

template <int HD>
__global__ void __launch_bounds__(FWD_THREADS, 1) attn_fwd_tc_f32_kernel(const __grid_constant__ F32FwdParams P) {
  using SM = FwdSmem<HD>;
  constexpr int NB = SM::NB, NS = SM::NS, PN = HD / 32, HC = HD / 2;      // HC: output columns of a thread
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + SM::BAR_OFF, slot = bars + 8 * SM::N_BARS, flag = slot + 8;
  auto bar = [&](int i) { return bars + 8u * i; };
  enum { KFULL = 0, KEMPTY = NB, VFULL = 2 * NB, VEMPTY = 3 * NB, KPARTS = 4 * NB, KFREE = 5 * NB, VPARTS = 6 * NB, VFREE = 7 * NB,
         SFULL = 8 * NB, SREAD = SFULL + NS, QFULL = SREAD + NS, QPARTS, PFULL, PVDONE, MEET };
  const int warp = (int)tc::uniform(threadIdx.x / 32), lane = threadIdx.x % 32;
  // later queries first: under a causal mask they have the most keys
  const int i0 = ((int)gridDim.x - 1 - (int)blockIdx.x) * QT, h = blockIdx.y, b = blockIdx.z, g = h / P.group;
  const int j_end = P.causal ? min(P.seq_k, i0 + QT) : P.seq_k, n_tiles = (j_end + KT - 1) / KT;
  int32_t* status = P.status;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NB; ++s) {
      tc::mbar_init(bar(KFULL + s), 1); tc::mbar_init(bar(VFULL + s), 1);
      tc::mbar_init(bar(KEMPTY + s), CONV_WARPS); tc::mbar_init(bar(VEMPTY + s), CONV_WARPS);
      tc::mbar_init(bar(KPARTS + s), CONV_WARPS); tc::mbar_init(bar(VPARTS + s), CONV_WARPS);
      tc::mbar_init(bar(KFREE + s), 1); tc::mbar_init(bar(VFREE + s), 1);
    }
    for (int s = 0; s < NS; ++s) { tc::mbar_init(bar(SFULL + s), 1); tc::mbar_init(bar(SREAD + s), SOFT_WARPS); }
    tc::mbar_init(bar(QFULL), 1);
    tc::mbar_init(bar(QPARTS), SOFT_WARPS);
    tc::mbar_init(bar(PFULL), SOFT_WARPS);
    tc::mbar_init(bar(PVDONE), 1);
    for (int s = 0; s < 4; ++s) tc::mbar_init(bar(MEET + s), 2);
    tc::fence_barrier_init();
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag), "r"(0u) : "memory");
    tc::tma_prefetch_desc(&P.tq); tc::tma_prefetch_desc(&P.tk); tc::tma_prefetch_desc(&P.tv);
    pdl_wait();
    tc::mbar_expect_tx(bar(QFULL), QT * HD * 4);
    tc::tma_load_4d(base + SM::Q_OFF, &P.tq, bar(QFULL), 0, i0, b, h * PN);
    tc::mbar_expect_tx(bar(KFULL), SM::RAW);
    tc::tma_load_4d(base + SM::K_OFF, &P.tk, bar(KFULL), 0, 0, b, g * PN);
    tc::mbar_expect_tx(bar(VFULL), SM::RAW);
    tc::tma_load_4d(base + SM::V_OFF, &P.tv, bar(VFULL), 0, 0, b, g * PN);
  }
  if (warp == 1) {
    tc::tmem_alloc(slot, 512);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  uint32_t tmem_base;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(slot));
  tmem_base = tc::uniform(tmem_base);
  pdl_launch_dependents();

  if (warp == 0) {
    if (lane == 0) {
      // ---- loads (the first tiles are on their way) ----
      for (int j = 1; j < n_tiles; ++j) {
        const int s = j % NB;
        const uint32_t ph = ((j / NB) & 1) ^ 1;
        if (!tc::mbar_wait(bar(KEMPTY + s), ph, status, 401)) break;
        tc::mbar_expect_tx(bar(KFULL + s), SM::RAW);
        tc::tma_load_4d(base + SM::K_OFF + s * SM::RAW, &P.tk, bar(KFULL + s), 0, j * KT, b, g * PN);
        if (!tc::mbar_wait(bar(VEMPTY + s), ph, status, 402)) break;
        tc::mbar_expect_tx(bar(VFULL + s), SM::RAW);
        tc::tma_load_4d(base + SM::V_OFF + s * SM::RAW, &P.tv, bar(VFULL + s), 0, j * KT, b, g * PN);
      }
    }
  } else if (warp == 1) {
    const bool leader = tc::elect_one();
    // ---- products, the small ones first ----
    const uint32_t hi = tc::smem_desc_hi(1024), idesc_s = tc::idesc_bf16(QT, KT, 0, 0), idesc_o = tc::idesc_bf16(QT, HD, 0, 1);
    const uint32_t k_lo = tc::smem_desc_lo(base + SM::KP_OFF, 16), v_lo = tc::smem_desc_lo(base + SM::VP_OFF, 8192);
    auto issue_s = [&](int j) -> bool {
      const int s = j % NB, sb = j % NS;
      if (!tc::mbar_wait_warp(bar(KPARTS + s), (j / NB) & 1, status, 403) || !tc::mbar_wait_warp(bar(SREAD + sb), ((j / NS) & 1) ^ 1, status, 404)) return false;
      tc::tc_fence_after();
      const uint32_t kl = k_lo + s * (SM::PARTS >> 4);
#pragma unroll
      for (uint32_t first = 0; first < HD / 16; first += HD / 32) {
        const uint32_t d = tmem_base + SM::S_COL + sb * (2 * KT) + (first ? KT : 0);
        uint32_t acc = 0;
        auto product = [&](int pa, int pb) {
          if (!leader) return;
#pragma unroll
          for (uint32_t kk = first; kk < first + HD / 32; ++kk) {
            tc::mma_bf16_ts_w(d, tmem_base + SM::QP_COL + pa * (HD / 2) + kk * 8, kl + pb * (SM::PART >> 4) + kk * 2, hi, idesc_s, acc);
            acc = 1;
          }
        };
        product(2, 0); product(0, 2); product(1, 1); product(1, 0); product(0, 1); product(0, 0);
      }
      if (leader) tc::mma_commit(bar(SFULL + sb));
      if (leader) tc::mma_commit(bar(KFREE + s));
      return true;
    };
    bool ok = tc::mbar_wait_warp(bar(QPARTS), 0, status, 405) && issue_s(0);
    for (int j = 0; j < n_tiles && ok; ++j) {
      if (j + 1 < n_tiles && !issue_s(j + 1)) break;
      const int s = j % NB;
      if (!tc::mbar_wait_warp(bar(VPARTS + s), (j / NB) & 1, status, 406) || !tc::mbar_wait_warp(bar(PFULL), j & 1, status, 407)) break;
      tc::tc_fence_after();
      const uint32_t vl = v_lo + s * (SM::PARTS >> 4);
      uint32_t acc = 0;
      auto product = [&](int pa, int pb) {
        if (!leader) return;
#pragma unroll
        for (uint32_t kk = 0; kk < KT / 16; ++kk) {
          tc::mma_bf16_ts_w(tmem_base + SM::O_COL, tmem_base + SM::P_COL + pa * 32 + kk * 8, vl + pb * (SM::PART >> 4) + kk * 128, hi, idesc_o, acc);
          acc = 1;
        }
      };
      product(2, 0); product(0, 2); product(1, 1); product(1, 0); product(0, 1); product(0, 0);
      if (leader) tc::mma_commit(bar(PVDONE));
      if (leader) tc::mma_commit(bar(VFREE + s));
    }
  } else if (warp >= 2 + SOFT_WARPS) {
    // ---- K and V into parts ----
    const int tid = threadIdx.x - 32 * (2 + SOFT_WARPS);
    float2 probe = make_float2(0.f, 0.f);
    for (int j = 0; j < n_tiles; ++j) {
      const int s = j % NB;
      bool ok = true;
#pragma unroll 1
      for (int which = 0; which < 2 && ok; ++which) {
        ok = tc::mbar_wait(bar((which ? VFULL : KFULL) + s), (j / NB) & 1, status, 408) &&
             tc::mbar_wait(bar((which ? VFREE : KFREE) + s), ((j / NB) & 1) ^ 1, status, 409);
        if (!ok) break;
        const uint32_t src = base + (which ? SM::V_OFF : SM::K_OFF) + s * SM::RAW, dst = base + (which ? SM::VP_OFF : SM::KP_OFF) + s * SM::PARTS;
#pragma unroll
        for (int u = 0; u < KT * HD / 16 / (32 * CONV_WARPS); ++u) {
          const int unit = u * 32 * CONV_WARPS + tid;
          convert_piece(src, dst, SM::PART, KT, unit % KT, unit / KT, which ? 0.f : Lift<HD>::K, probe);
        }
        // the flag before anything that depends on these parts
        if (tc::probe_failed(probe)) asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag), "r"(1u) : "memory");
        tc::fence_proxy_async();
        __syncwarp();
        if (lane == 0) { tc::mbar_arrive(bar((which ? VEMPTY : KEMPTY) + s)); tc::mbar_arrive(bar((which ? VPARTS : KPARTS) + s)); }
      }
      if (!ok) break;
    }
  } else {
    // ---- softmax: thread = (query row, half) ----
    const int q = warp % 4, half = (warp - 2) / 4, r = q * 32 + lane, gi = i0 + r;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    const float scale = P.scale * tc::PARTS_BACK;             // of scores as they come out of the products
    const uint32_t mine = base + SM::MAX_OFF + (half * QT + r) * 4, other = base + SM::MAX_OFF + ((half ^ 1) * QT + r) * 4;
    uint32_t met = 0;
    auto meet = [&]() -> bool {                              // the two warps of these rows
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(bar(MEET + q));
      return tc::mbar_wait(bar(MEET + q), met++ & 1, status, 413);
    };
    bool ok = tc::mbar_wait(bar(QFULL), 0, status, 410);
    if (ok) {
      float2 probe = make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < HC / 16; ++u) {
        const int piece = half * (HC / 16) + u;
        const uint32_t row = base + SM::Q_OFF + (piece / 2) * (QT * 128) + r * 128;
        uint32_t p[3][8];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4 v = tc::lds4(row + (((piece % 2 * 4 + c) ^ (r & 7)) << 4));
          tc::split3(v.x, v.y, Lift<HD>::Q, p[0][2 * c], p[1][2 * c], p[2][2 * c]);
          tc::split3(v.z, v.w, Lift<HD>::Q, p[0][2 * c + 1], p[1][2 * c + 1], p[2][2 * c + 1]);
          tc::probe_range(v.x, v.y, probe);
          tc::probe_range(v.z, v.w, probe);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) tc::tmem_st8(lane_addr + SM::QP_COL + i * (HD / 2) + piece * 8, p[i]);
      }
      if (tc::probe_failed(probe)) asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag), "r"(1u) : "memory");
      tc::tmem_st_wait();
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(bar(QPARTS));
    }
    pdl_wait();                                              // before this role writes anything to global memory
    float m = -INFINITY, l = 0.f;
    float2 o[HC / 2];
#pragma unroll
    for (int c = 0; c < HC / 2; ++c) o[c] = make_float2(0.f, 0.f);
    auto add_output = [&](int j) -> bool {                   // the product of tile j, in the scale of the maximum then
      if (!tc::mbar_wait(bar(PVDONE), j & 1, status, 411)) return false;
      tc::tc_fence_after();
#pragma unroll
      for (int c = 0; c < HC / 16; ++c) {
        uint32_t v[16];
        tc::tmem_ld16(lane_addr + SM::O_COL + half * HC + 16 * c, v);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 8; ++k) o[8 * c + k] = __fadd2_rn(o[8 * c + k], make_float2(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1])));
      }
      return true;
    };
    for (int j = 0; j < n_tiles && ok; ++j) {
      const int j0 = j * KT + half * 32, sb = j % NS;
      if (!tc::mbar_wait(bar(SFULL + sb), (j / NS) & 1, status, 412)) { ok = false; break; }
      tc::tc_fence_after();
      uint32_t raw[32];
      tc::tmem_ld32(lane_addr + SM::S_COL + sb * (2 * KT) + half * 32, raw);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t more[16];
        tc::tmem_ld16(lane_addr + SM::S_COL + sb * (2 * KT) + KT + half * 32 + 16 * c, more);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 16; ++k) raw[16 * c + k] = __float_as_uint(__uint_as_float(raw[16 * c + k]) + __uint_as_float(more[k]));
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(bar(SREAD + sb));
      float* s = reinterpret_cast<float*>(raw);
      const bool need_mask = j0 + 32 > P.seq_k || (P.causal && j0 + 31 > i0);
      float mx = -INFINITY;
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        s[k] *= scale;
        if (need_mask && (j0 + k >= P.seq_k || (P.causal && j0 + k > gi))) s[k] = -INFINITY;
        mx = fmaxf(mx, s[k]);
      }
      const uint32_t slot_j = (j & 1) * (2 * QT * 4);
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(mine + slot_j), "f"(mx) : "memory");
      if (!meet()) { ok = false; break; }
      float mo;
      asm volatile("ld.shared.f32 %0, [%1];" : "=f"(mo) : "r"(other + slot_j) : "memory");
      const float m_new = fmaxf(m, fmaxf(mx, mo));
      const float alpha = m_new == -INFINITY ? 1.f : expf(m - m_new);
      m = m_new;
      uint32_t p[3][16];
      float sum = 0.f;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const float p0 = m == -INFINITY ? 0.f : expf(s[2 * k] - m), p1 = m == -INFINITY ? 0.f : expf(s[2 * k + 1] - m);
        sum += p0 + p1;
        tc::split3(p0, p1, Lift<HD>::P, p[0][k], p[1][k], p[2][k]);
      }
      l = l * alpha + sum;
      // P's columns and the output accumulator are free once the product of the tile before has been added
      if (j > 0 && !add_output(j - 1)) { ok = false; break; }
#pragma unroll
      for (int c = 0; c < HC / 2; ++c) o[c] = __fmul2_rn(o[c], make_float2(alpha, alpha));
#pragma unroll
      for (int i = 0; i < 3; ++i) tc::tmem_st16(lane_addr + SM::P_COL + i * 32 + half * 16, p[i]);
      tc::tmem_st_wait();
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(bar(PFULL));
    }
    if (ok && n_tiles > 0) ok = add_output(n_tiles - 1);
    // the row's sum: both halves', where the next tile's maxima would go
    const uint32_t slot_l = (n_tiles & 1) * (2 * QT * 4);
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(mine + slot_l), "f"(l) : "memory");
    ok = ok && meet();
    float lo;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(lo) : "r"(other + slot_l) : "memory");
    l = half ? lo + l : l + lo;
    if (ok && gi < P.t_pad) {
      const bool live = gi < P.seq;
      const float inv = live ? 1.f / l * tc::PARTS_BACK : 0.f;
#pragma unroll
      for (int c = 0; c < HC / 4; ++c) {
        const float4 v = live ? make_float4(o[2 * c].x * inv, o[2 * c].y * inv, o[2 * c + 1].x * inv, o[2 * c + 1].y * inv) : make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(P.a + rt_off<32>(P.n_pad, (long long)b * P.t_pad + gi, h * HD + half * HC + 4 * c)) = v;
      }
      if (half == 0) P.lse[((long long)b * P.hq + h) * P.t_pad + gi] = live ? m + logf(l) : 0.f;
    }
  }
  __syncwarp();
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem_base, 512);
  uint32_t again;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(again) : "r"(flag) : "memory");
  if (again) plain_rows<HD>(P, base, i0, h, b);
}

template <int HD>
cudaError_t fwd_launch(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse, int32_t* status, cudaStream_t st) {
  auto k = attn_fwd_tc_f32_kernel<HD>;
  const dim3 grid((p->t_pad + QT - 1) / QT, p->d.n_q_heads, p->d.batch);
  auto make = [&](F32FwdParams& P) {
    memset(&P, 0, sizeof(P));
    P.n_pad = p->n_pad; P.n_pad_k = p->n_pad_kv; P.seq = p->d.seq; P.t_pad = p->t_pad; P.seq_k = p->seq_kv; P.t_pad_k = p->t_pad_kv;
    P.hq = p->d.n_q_heads; P.group = p->group; P.causal = p->d.causal; P.scale = p->scale;
    if (!fbl_encode_seq_map(&P.tq, true, Q, p->t_pad, p->d.batch, p->dq / 32, QT, HD / 32) ||
        !fbl_encode_seq_map(&P.tk, true, K, p->t_pad_kv, p->d.batch, p->dkv / 32, KT, HD / 32) ||
        !fbl_encode_seq_map(&P.tv, true, V, p->t_pad_kv, p->d.batch, p->dkv / 32, KT, HD / 32))
      return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FwdSmem<HD>::TOTAL);
  };
  auto point = [&](F32FwdParams& P) {
    P.q = (const float*)Q; P.k = (const float*)K; P.v = (const float*)V;
    P.a = (float*)A; P.lse = lse; P.status = status;
    return fbl_map_set_base(&P.tq, Q) && fbl_map_set_base(&P.tk, K) && fbl_map_set_base(&P.tv, V);
  };
  LaunchKey key;
  key.add(0, 0);
  return LaunchMemo<F32FwdParams, 4>::run(p, FBL_MEMO_TC_F32_FWD, key, make, point, [&](const F32FwdParams& P) {
    return launch_pdl(k, grid, dim3(FWD_THREADS), FwdSmem<HD>::TOTAL, st, P);
  });
}

// ------------------------------------------------------------------------------------------
// Backward, heads of 32 and 64: one block per (128 keys, KV head, batch), 64 queries of a head at a time; the rows a thread owns
// are keys.  S^T = K Q^T and dP^T = V dO^T, then P^T and dS^T in fp32, whose parts (tensor memory) make dV += P^T dO and
// dK += dS^T Q, added up in registers; dS^T's parts in shared memory, read with the axes swapped, make dQ = dS K (M = 64: a warp's
// rows lie in the first 16 of its lanes), 32 keys to an accumulator, whose sum goes to memory by 16-byte reductions.  18 warps: one
// loads, one issues, 16 work (four threads to a key row): softmax, then the next queries' parts while this tile's products run.
// Where that makes fewer blocks than SMs, a cluster of 2 to 8 blocks takes a key tile's items in turn and adds dK and dV through
// distributed shared memory in a fixed order.  The products alone, 144 instructions an item, are some 7000 clk (48 heads of 197
// tokens: tensor pipe active for 36 % of active cycles).
// ------------------------------------------------------------------------------------------
constexpr int BKT = 128, BQT = 64, WORK_WARPS = 16, BWD_THREADS = 32 * (2 + WORK_WARPS);

struct alignas(64) F32BwdParams {
  CUtensorMap tq, tk, tv, tdo;
  const float *q, *k, *v, *dO;
  const float* lse;
  const float* dvec;
  float* dq;                    // zeroed; added into
  float *dk, *dv;
  long long n_pad, n_pad_k;
  int seq, t_pad, seq_k, t_pad_k, hq, group, causal;
  int slices;
  float scale;
  int32_t* status;
};

struct BwdSmem {                                             // the same for both head widths: rows of 128 bytes, half used at 32
  static constexpr uint32_t KV_PART = BKT * 128, Q_PART = BQT * 128;
  static constexpr uint32_t K_OFF = 0, V_OFF = 3 * KV_PART, Q_OFF = 6 * KV_PART, DO_OFF = Q_OFF + 3 * Q_PART, DS_OFF = DO_OFF + 3 * Q_PART;
  static constexpr uint32_t RAW_OFF = DS_OFF + 3 * KV_PART, RAW = BQT * 256;      // fp32 Q, then dO; K's and V's over dS^T and over Q's and dO's parts
  static constexpr uint32_t STAT_OFF = RAW_OFF + 2 * RAW;    // two items' LSE and D, 64 floats each
  static constexpr uint32_t BAR_OFF = STAT_OFF + 4 * 256, N_BARS = 16, TOTAL = BAR_OFF + 8 * N_BARS + 32 + 1024;
  static_assert(TOTAL <= 232448, "shared memory of a block");
  // tensor memory
  static constexpr uint32_t S_COL = 0, DP_COL = 64, DV_COL = 128, DK_COL = 192, DQ_COL = 256, P_COL = 320, DS_COL = 416;
};

// A block's items by plain arithmetic, where an operand or a dS is out of range (tc::probe_range): dK and dV of all of them, left where the kernel leaves
// its own, and dQ of those whose own was not added (even and odd items from the two numbers at `from_at` on).  16 warps, four threads to a key row (a quarter of
// the queries, then of the columns of dK and dV), eight to a query row for dQ.  Pairs that the mask leaves out take no part.
template <int HD>
__device__ __noinline__ void plain_items(const F32BwdParams& P, uint32_t base, uint32_t from_at, int n_it, int t0, int per_head) {
  constexpr int LD = HD + 4, LDP = BQT + 1, N = HD / 4, HC = HD / 4, HQ = HD / 8;
  const uint32_t sk = base, sv = sk + BKT * LD * 4, sq = sv + BKT * LD * 4, so = sq + BQT * HD * 4, sp = so + BQT * HD * 4, sd = sp + BKT * LDP * 4;
  static_assert((2 * BKT * LD + 2 * BQT * HD + 2 * BKT * LDP) * 4 <= (int)BwdSmem::STAT_OFF, "shared memory");
  const bool work = threadIdx.x < 4 * BKT;
  const int slice = blockIdx.x % P.slices, j0 = blockIdx.x / P.slices * BKT, g = blockIdx.y, b = blockIdx.z;
  int from[2];
  for (int i = 0; i < 2; ++i) asm volatile("ld.shared.s32 %0, [%1];" : "=r"(from[i]) : "r"(from_at + 4 * i) : "memory");
  const int r = threadIdx.x % BKT, quarter = threadIdx.x / BKT % 4, gj = j0 + r, i = threadIdx.x % BQT, eighth = threadIdx.x / BQT % 8;
  auto fill = [&](uint32_t to, int ld, int rows, const float* m, long long n_pad, int t_pad, int row0, int end, int col) {
    for (int e = threadIdx.x; e < rows * N; e += BWD_THREADS) {
      const int row = e / N, c = e % N * 4;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row0 + row < end) x = *reinterpret_cast<const float4*>(m + rt_off<32>(n_pad, (long long)b * t_pad + row0 + row, col + c));
      asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(to + (row * ld + c) * 4), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w) : "memory");
    }
  };
  fill(sk, LD, BKT, P.k, P.n_pad_k, P.t_pad_k, j0, P.seq_k, g * HD);
  fill(sv, LD, BKT, P.v, P.n_pad_k, P.t_pad_k, j0, P.seq_k, g * HD);
  float dk[HC], dv[HC];
#pragma unroll
  for (int c = 0; c < HC; ++c) dk[c] = dv[c] = 0.f;
#pragma unroll 1
  for (int n = 0; n < n_it; ++n) {
    const int item = slice + n * P.slices, h = g * P.group + item / per_head, i0 = (t0 + item % per_head) * BQT, gi = i0 + i;
    const long long at = ((long long)b * P.hq + h) * P.t_pad;
    __syncthreads();
    fill(sq, HD, BQT, P.q, P.n_pad, P.t_pad, i0, P.seq, h * HD);
    fill(so, HD, BQT, P.dO, P.n_pad, P.t_pad, i0, P.seq, h * HD);
    __syncthreads();
    // queries of this item that take part with this thread's key: first .. last - 1
    const int first = P.causal ? max(0, gj - i0) : 0, last = gj < P.seq_k ? min(BQT, P.seq - i0) : 0;
    if (work) {
      float s[16], dp[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) s[k] = dp[k] = 0.f;
#pragma unroll 1
      for (int d = 0; d < HD; d += 4) {
        const float4 k4 = tc::lds4(sk + (r * LD + d) * 4), v4 = tc::lds4(sv + (r * LD + d) * 4);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float4 q4 = tc::lds4(sq + ((quarter * 16 + k) * HD + d) * 4), o4 = tc::lds4(so + ((quarter * 16 + k) * HD + d) * 4);
          s[k] = fmaf(k4.x, q4.x, fmaf(k4.y, q4.y, fmaf(k4.z, q4.z, fmaf(k4.w, q4.w, s[k]))));
          dp[k] = fmaf(v4.x, o4.x, fmaf(v4.y, o4.y, fmaf(v4.z, o4.z, fmaf(v4.w, o4.w, dp[k]))));
        }
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int c = quarter * 16 + k;
        float p = 0.f, ds = 0.f;
        if (c >= first && c < last) {
          p = expf(s[k] * P.scale - P.lse[at + i0 + c]);
          ds = p * (dp[k] - P.dvec[at + i0 + c]);
        }
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(sp + (r * LDP + c) * 4), "f"(p) : "memory");
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(sd + (r * LDP + c) * 4), "f"(ds) : "memory");
      }
    }
    __syncthreads();
    if (!work) continue;
#pragma unroll 1
    for (int c = first; c < last; ++c) {
      float p, ds;
      asm volatile("ld.shared.f32 %0, [%1];" : "=f"(p) : "r"(sp + (r * LDP + c) * 4) : "memory");
      asm volatile("ld.shared.f32 %0, [%1];" : "=f"(ds) : "r"(sd + (r * LDP + c) * 4) : "memory");
#pragma unroll
      for (int x = 0; x < HC; x += 4) {
        const float4 o4 = tc::lds4(so + (c * HD + quarter * HC + x) * 4), q4 = tc::lds4(sq + (c * HD + quarter * HC + x) * 4);
        dv[x] = fmaf(p, o4.x, dv[x]); dv[x + 1] = fmaf(p, o4.y, dv[x + 1]); dv[x + 2] = fmaf(p, o4.z, dv[x + 2]); dv[x + 3] = fmaf(p, o4.w, dv[x + 3]);
        dk[x] = fmaf(ds, q4.x, dk[x]); dk[x + 1] = fmaf(ds, q4.y, dk[x + 1]); dk[x + 2] = fmaf(ds, q4.z, dk[x + 2]); dk[x + 3] = fmaf(ds, q4.w, dk[x + 3]);
      }
    }
    if (n < from[n & 1] || gi >= P.seq) continue;
    float dq[HQ];
#pragma unroll
    for (int x = 0; x < HQ; ++x) dq[x] = 0.f;
#pragma unroll 1
    for (int k = 0; k < min(BKT, (P.causal ? min(P.seq_k, gi + 1) : P.seq_k) - j0); ++k) {
      float ds;
      asm volatile("ld.shared.f32 %0, [%1];" : "=f"(ds) : "r"(sd + (k * LDP + i) * 4) : "memory");
#pragma unroll
      for (int x = 0; x < HQ; x += 4) {
        const float4 k4 = tc::lds4(sk + (k * LD + eighth * HQ + x) * 4);
        dq[x] = fmaf(ds, k4.x, dq[x]); dq[x + 1] = fmaf(ds, k4.y, dq[x + 1]); dq[x + 2] = fmaf(ds, k4.z, dq[x + 2]); dq[x + 3] = fmaf(ds, k4.w, dq[x + 3]);
      }
    }
#pragma unroll
    for (int x = 0; x < HQ; x += 4)
      atomicAdd(reinterpret_cast<float4*>(P.dq + rt_off<32>(P.n_pad, (long long)b * P.t_pad + gi, h * HD + eighth * HQ + x)),
                make_float4(dq[x] * P.scale, dq[x + 1] * P.scale, dq[x + 2] * P.scale, dq[x + 3] * P.scale));
  }
  __syncthreads();
  if (work) {
#pragma unroll
    for (int c = 0; c < HC; c += 4) {
      tc::sts4(base + (r * LD + quarter * HC + c) * 4, reinterpret_cast<const uint32_t*>(&dk[c]));
      tc::sts4(base + (BKT * LD + r * LD + quarter * HC + c) * 4, reinterpret_cast<const uint32_t*>(&dv[c]));
    }
  }
  __syncthreads();
}

template <int HD>
__global__ void __launch_bounds__(BWD_THREADS, 1) attn_bwd_tc_f32_kernel(const __grid_constant__ F32BwdParams P) {
  using SM = BwdSmem;
  constexpr int PN = HD / 32, HC = HD / 4;                   // HC: columns of dK, dV and dQ of a thread
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + SM::BAR_OFF, slot = bars + 8 * SM::N_BARS, flag = slot + 8;
  auto bar = [&](int i) { return bars + 8u * i; };
  enum { KVFULL, QRAW, DORAW, QRAWE, DORAWE, KVPARTS, QPARTS, DOPARTS, SFULL, DPFULL, PREADY, DSREADY, DVDONE, DKDONE, DQDONE, DQREAD };
  const int warp = (int)tc::uniform(threadIdx.x / 32), lane = threadIdx.x % 32;
  const int slices = P.slices, slice = blockIdx.x % slices;
  const int j0 = blockIdx.x / slices * BKT, g = blockIdx.y, b = blockIdx.z;      // key tile 0 has the most queries: first
  const int t0 = P.causal ? j0 / BQT : 0, per_head = max(0, (P.seq + BQT - 1) / BQT - t0), items = per_head * P.group;
  const int n_it = slice < items ? (items - slice + slices - 1) / slices : 0;    // items slice, slice + slices, ...
  auto head_of = [&](int n) { return g * P.group + (slice + n * slices) / per_head; };
  auto row_of = [&](int n) { return (t0 + (slice + n * slices) % per_head) * BQT; };
  int32_t* status = P.status;
  auto raised = [&](int i) -> bool {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(flag + 4 * i) : "memory");
    return v != 0;
  };
  if (threadIdx.x == 0) {
    for (int i : {KVFULL, QRAW, DORAW, SFULL, DPFULL, DVDONE, DKDONE, DQDONE}) tc::mbar_init(bar(i), 1);
    for (int i : {QRAWE, DORAWE, KVPARTS, QPARTS, DOPARTS, PREADY, DSREADY, DQREAD}) tc::mbar_init(bar(i), WORK_WARPS);
    tc::fence_barrier_init();
    for (int i = 0; i < 5; ++i) asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag + 4 * i), "r"(i < 3 ? 0u : 0x7fffffffu) : "memory");
    tc::tma_prefetch_desc(&P.tq); tc::tma_prefetch_desc(&P.tk); tc::tma_prefetch_desc(&P.tv); tc::tma_prefetch_desc(&P.tdo);
    pdl_wait();
    if (n_it > 0) {
      tc::mbar_expect_tx(bar(KVFULL), 2 * BKT * HD * 4);
      tc::tma_load_4d(base + SM::DS_OFF, &P.tk, bar(KVFULL), 0, j0, b, g * PN);
      tc::tma_load_4d(base + SM::Q_OFF, &P.tv, bar(KVFULL), 0, j0, b, g * PN);
    }
  }
  if (warp == 1) {
    tc::tmem_alloc(slot, 512);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  uint32_t tmem_base;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(slot));
  tmem_base = tc::uniform(tmem_base);
  pdl_launch_dependents();

  if (warp == 0) {
    if (lane == 0) {
      for (int n = 0; n < n_it; ++n) {
        const int h = head_of(n), i0 = row_of(n);
        const long long at = ((long long)b * P.hq + h) * P.t_pad + i0;           // rows past the sequence may hold anything: masked
        const uint32_t stat = base + SM::STAT_OFF + (n & 1) * 512;
        if (!tc::mbar_wait(bar(DORAWE), (n & 1) ^ 1, status, 421)) break;
        tc::mbar_expect_tx(bar(DORAW), BQT * HD * 4 + 256);
        tc::tma_load_4d(base + SM::RAW_OFF + SM::RAW, &P.tdo, bar(DORAW), 0, i0, b, h * PN);
        tc::bulk_load(stat + 256, P.dvec + at, 256, bar(DORAW));
        if (!tc::mbar_wait(bar(QRAWE), (n & 1) ^ 1, status, 422)) break;
        tc::mbar_expect_tx(bar(QRAW), BQT * HD * 4 + 256);
        tc::tma_load_4d(base + SM::RAW_OFF, &P.tq, bar(QRAW), 0, i0, b, h * PN);
        tc::bulk_load(stat, P.lse + at, 256, bar(QRAW));
      }
    }
  } else if (warp == 1) {
    const bool leader = tc::elect_one();
    // ---- products, the small ones first (offsets in 16-byte units: 16 columns along a row 2, 16 rows 128) ----
    const uint32_t hi = tc::smem_desc_hi(1024);
    const uint32_t idesc_s = tc::idesc_bf16(BKT, BQT, 0, 0), idesc_kv = tc::idesc_bf16(BKT, HD, 0, 1), idesc_dq = tc::idesc_bf16(BQT, HD, 1, 1);
    auto lo = [&](uint32_t off) { return tc::smem_desc_lo(base + off, 16); };  // tiles of one 64-column panel: no leading offset in use
    auto six = [&](auto&& product) {
      uint32_t acc = 0;
      product(2, 0, acc); product(0, 2, acc); product(1, 1, acc); product(1, 0, acc); product(0, 1, acc); product(0, 0, acc);
    };
    auto scores = [&](uint32_t col, uint32_t a, uint32_t bq, uint32_t first) { // 128 keys x 64 queries, reduced over half of head_dim
      if (!leader) return;
      six([&](int pb, int pa, uint32_t& acc) {                                 // (parts in the forward's order, where queries are operand A)
#pragma unroll
        for (uint32_t kk = 0; kk < HD / 32; ++kk, acc = 1)
          tc::mma_bf16_ss_w(tmem_base + col, a + pa * (SM::KV_PART >> 4) + first + kk * 2, hi, bq + pb * (SM::Q_PART >> 4) + first + kk * 2, hi, idesc_s, acc);
      });
    };
    auto weighted = [&](uint32_t col, uint32_t parts, uint32_t bq) {           // 128 keys x head_dim, reduced over 64 queries
      if (!leader) return;
      six([&](int pa, int pb, uint32_t& acc) {
#pragma unroll
        for (uint32_t kk = 0; kk < BQT / 16; ++kk, acc = 1)
          tc::mma_bf16_ts_w(tmem_base + col, tmem_base + parts + pa * 32 + kk * 8, bq + pb * (SM::Q_PART >> 4) + kk * 128, hi, idesc_kv, acc);
      });
    };
    auto queries = [&](uint32_t col, uint32_t first) {                         // 64 queries x head_dim, reduced over 32 keys
      if (!leader) return;
      six([&](int pa, int pb, uint32_t& acc) {
#pragma unroll
        for (uint32_t kk = 0; kk < 2; ++kk, acc = 1)
          tc::mma_bf16_ss_w(tmem_base + col, lo(SM::DS_OFF) + pa * (SM::KV_PART >> 4) + first + kk * 128, hi,
                            lo(SM::K_OFF) + pb * (SM::KV_PART >> 4) + first + kk * 128, hi, idesc_dq, acc);
      });
    };
    bool ok = n_it > 0 && tc::mbar_wait_warp(bar(KVPARTS), 0, status, 423);
    for (int n = 0; n <= n_it && ok; ++n) {
      if (n > 0) {
        if (!tc::mbar_wait_warp(bar(PREADY), (n - 1) & 1, status, 424)) break;
        tc::tc_fence_after();
        weighted(SM::DV_COL, SM::P_COL, lo(SM::DO_OFF));
        if (leader) tc::mma_commit(bar(DVDONE));
        if (!tc::mbar_wait_warp(bar(DSREADY), (n - 1) & 1, status, 428)) break;
        tc::tc_fence_after();
        weighted(SM::DK_COL, SM::DS_COL, lo(SM::Q_OFF));
        if (leader) tc::mma_commit(bar(DKDONE));
        queries(SM::DQ_COL, 0);                            // and over dP^T, S^T and P^T, which have been read
        queries(SM::DP_COL, 256);
        queries(SM::S_COL, 512);
        queries(SM::P_COL, 768);
        if (leader) tc::mma_commit(bar(DQDONE));
      }
      if (n == n_it) break;
      if (!tc::mbar_wait_warp(bar(QPARTS), n & 1, status, 425) || (n > 0 && !tc::mbar_wait_warp(bar(DQREAD), (n - 1) & 1, status, 427))) break;
      tc::tc_fence_after();
      scores(SM::S_COL, lo(SM::K_OFF), lo(SM::Q_OFF), 0);
      scores(SM::DV_COL, lo(SM::K_OFF), lo(SM::Q_OFF), HD / 16);       // over the dV and dK of the item before, which have been added
      if (leader) tc::mma_commit(bar(SFULL));
      if (!tc::mbar_wait_warp(bar(DOPARTS), n & 1, status, 426)) break;
      tc::tc_fence_after();
      scores(SM::DP_COL, lo(SM::V_OFF), lo(SM::DO_OFF), 0);
      scores(SM::DK_COL, lo(SM::V_OFF), lo(SM::DO_OFF), HD / 16);
      if (leader) tc::mma_commit(bar(DPFULL));
    }
  } else {
    // ---- 16 warps: thread = (key row, a quarter of the queries and of the columns of dK, dV, dQ) ----
    const int q = warp % 4, quarter = (warp - 2) / 4, r = q * 32 + lane, gj = j0 + r, tid = threadIdx.x - 64;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    auto arrive = [&](int i) {
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(bar(i));
    };
    // A value out of range (tc::probe_range) raises a flag, before what depends on it is announced: 0 and 1 for even and odd items, 2 for K and V.
    // (An item's flag is read when its products are complete, and raised for the item after next when all have read it.)
    auto raise = [&](const float2& probe, int i) {
      if (tc::probe_failed(probe)) asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag + 4 * i), "r"(1u) : "memory");
    };
    auto convert = [&](uint32_t src, uint32_t dst, int rows, float lift, int flag_i) {
      float2 probe = make_float2(0.f, 0.f);
      for (int u = tid; u < rows * HD / 16; u += 32 * WORK_WARPS) convert_piece(src, dst, rows * 128, rows, u % rows, u / rows, lift, probe);
      raise(probe, flag_i);
      tc::fence_proxy_async();
    };
    // of S as it comes out of the products (where their product is below 1.2e-38 and loses bits, scores are below 1 and off by 2^-24)
    const float scale = P.scale * tc::PARTS_BACK;
    pdl_wait();
    bool ok = true;
    auto next_do = [&](int n) {
      ok = ok && tc::mbar_wait(bar(DORAW), n & 1, status, 430);
      if (!ok) return;
      convert(base + SM::RAW_OFF + SM::RAW, base + SM::DO_OFF, BQT, 0.f, n & 1);
      __syncwarp();
      if (lane == 0) { tc::mbar_arrive(bar(DORAWE)); tc::mbar_arrive(bar(DOPARTS)); }
    };
    auto next_q = [&](int n) {
      ok = ok && tc::mbar_wait(bar(QRAW), n & 1, status, 431);
      if (!ok) return;
      convert(base + SM::RAW_OFF, base + SM::Q_OFF, BQT, Lift<HD>::Q, n & 1);
      __syncwarp();
      if (lane == 0) { tc::mbar_arrive(bar(QRAWE)); tc::mbar_arrive(bar(QPARTS)); }
    };
    if (n_it > 0) {
      ok = tc::mbar_wait(bar(KVFULL), 0, status, 432);
      if (ok) {
        convert(base + SM::Q_OFF, base + SM::V_OFF, BKT, Lift<HD>::V, 2);
        convert(base + SM::DS_OFF, base + SM::K_OFF, BKT, Lift<HD>::K, 2);
        arrive(KVPARTS);
        ok = tc::mbar_wait(bar(KVPARTS), 0, status, 437);      // V's values have been read: Q's and dO's parts may lie over them
      }
      next_do(0);
      next_q(0);
    }
    float2 dk[HC / 2], dv[HC / 2];
#pragma unroll
    for (int c = 0; c < HC / 2; ++c) dk[c] = dv[c] = make_float2(0.f, 0.f);
    auto add = [&](uint32_t col, float2 (&sum)[HC / 2]) {
      uint32_t v[HC];
      if constexpr (HC == 16) tc::tmem_ld16(lane_addr + col + quarter * HC, v);
      else tc::tmem_ld8(lane_addr + col + quarter * HC, v);
      tc::tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < HC / 2; ++k) sum[k] = __fadd2_rn(sum[k], make_float2(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1])));
    };
    int plain_from[2] = {0x7fffffff, 0x7fffffff};              // even and odd items whose dQ is left to plain_items
    for (int n = 0; n < n_it && ok; ++n) {
      const int h = head_of(n), i0 = row_of(n);
      const uint32_t stat = base + SM::STAT_OFF + (n & 1) * 512;
      if (!tc::mbar_wait(bar(SFULL), n & 1, status, 433)) { ok = false; break; }
      tc::tc_fence_after();
      const bool need_mask = i0 + BQT > P.seq || j0 + BKT > P.seq_k || (P.causal && i0 < j0 + BKT - 1);
      float2 probe = make_float2(0.f, 0.f);
      const int c0 = quarter * 16;
      uint32_t x[16], y[16], part[3][8];
      float p[16];
      uint32_t out = 0;                                        // pairs that take no part
      if (need_mask) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const int gi = i0 + c0 + k;
          out |= (uint32_t)(gi >= P.seq || gj >= P.seq_k || (P.causal && gj > gi)) << k;
        }
      }
      tc::tmem_ld16(lane_addr + SM::S_COL + c0, x);
      tc::tmem_ld16(lane_addr + SM::DV_COL + c0, y);
      tc::tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 16; k += 4) {
        const float4 l4 = tc::lds4(stat + (c0 + k) * 4);
        const float ls[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) p[k + u] = out >> (k + u) & 1 ? 0.f : expf((__uint_as_float(x[k + u]) + __uint_as_float(y[k + u])) * scale - ls[u]);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) tc::split3(p[2 * k], p[2 * k + 1], Lift<HD>::P, part[0][k], part[1][k], part[2][k]);
#pragma unroll
      for (int i = 0; i < 3; ++i) tc::tmem_st8(lane_addr + SM::P_COL + i * 32 + c0 / 2, part[i]);
      tc::tmem_st_wait();
      tc::tc_fence_before();
      arrive(PREADY);
      if (!tc::mbar_wait(bar(DPFULL), n & 1, status, 438)) { ok = false; break; }
      tc::tc_fence_after();
      tc::tmem_ld16(lane_addr + SM::DP_COL + c0, x);
      tc::tmem_ld16(lane_addr + SM::DK_COL + c0, y);
      tc::tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 16; k += 4) {
        const float4 d4 = tc::lds4(stat + 256 + (c0 + k) * 4);
        const float ds[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) p[k + u] = out >> (k + u) & 1 ? 0.f : p[k + u] * fmaf(__uint_as_float(x[k + u]) + __uint_as_float(y[k + u]), tc::PARTS_BACK, -ds[u]);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        tc::split3(p[2 * k], p[2 * k + 1], Lift<HD>::DS, part[0][k], part[1][k], part[2][k]);
        tc::probe_range(p[2 * k], p[2 * k + 1], probe);
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        tc::tmem_st8(lane_addr + SM::DS_COL + i * 32 + c0 / 2, part[i]);
#pragma unroll
        for (int z = 0; z < 2; ++z) tc::sts4(base + SM::DS_OFF + i * SM::KV_PART + r * 128 + (((c0 / 8 + z) ^ (r & 7)) << 4), &part[i][4 * z]);
      }
      raise(probe, n & 1);
      tc::tmem_st_wait();
      tc::fence_proxy_async();
      tc::tc_fence_before();
      arrive(DSREADY);
      if (!tc::mbar_wait(bar(DVDONE), n & 1, status, 434)) { ok = false; break; }
      tc::tc_fence_after();
      add(SM::DV_COL, dv);
      if (n + 1 < n_it) next_do(n + 1);
      if (!ok || !tc::mbar_wait(bar(DKDONE), n & 1, status, 435)) { ok = false; break; }
      tc::tc_fence_after();
      add(SM::DK_COL, dk);
      if (n + 1 < n_it) next_q(n + 1);
      if (!ok || !tc::mbar_wait(bar(DQDONE), n & 1, status, 436)) { ok = false; break; }
      tc::tc_fence_after();
      float2 dq[HC / 2];
#pragma unroll
      for (int c = 0; c < HC / 2; ++c) dq[c] = make_float2(0.f, 0.f);
      add(SM::DQ_COL, dq);
      add(SM::DP_COL, dq);
      add(SM::S_COL, dq);
      add(SM::P_COL, dq);
      tc::tc_fence_before();
      const bool again = raised(n & 1) || raised(2);
      arrive(DQREAD);
      const int gi = i0 + q * 16 + lane;
      if (again) {
        if (warp == 2 && lane == 0 && n < plain_from[n & 1]) asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag + 12 + 4 * (n & 1)), "r"(n) : "memory");
        plain_from[n & 1] = min(plain_from[n & 1], n);
      } else if (lane < 16 && gi < P.seq) {
#pragma unroll
        for (int c = 0; c < HC / 2; ++c)                       // the parts' power of two first: a small softmax scale times it is zero
          dq[c] = __fmul2_rn(__fmul2_rn(dq[c], make_float2(tc::PARTS_BACK, tc::PARTS_BACK)), make_float2(P.scale, P.scale));
#pragma unroll
        for (int c = 0; c < HC / 4; ++c)
          atomicAdd(reinterpret_cast<float4*>(P.dq + rt_off<32>(P.n_pad, (long long)b * P.t_pad + gi, h * HD + quarter * HC + 4 * c)),
                    make_float4(dq[2 * c].x, dq[2 * c].y, dq[2 * c + 1].x, dq[2 * c + 1].y));
      }
    }
    // dK and dV of this block's items to shared memory, over K's and V's parts, which no product reads any more
    const uint32_t out = base + (uint32_t)(r * (HD + 4) + quarter * HC) * 4;
    constexpr uint32_t SUM_V = BKT * (HD + 4) * 4;
#pragma unroll
    for (int c = 0; c < HC / 2; ++c) {
      dk[c] = __fmul2_rn(dk[c], make_float2(tc::PARTS_BACK, tc::PARTS_BACK));
      dv[c] = __fmul2_rn(dv[c], make_float2(tc::PARTS_BACK, tc::PARTS_BACK));
    }
#pragma unroll
    for (int c = 0; c < HC / 2; c += 2) {
      tc::sts4(out + c * 8, reinterpret_cast<const uint32_t*>(&dk[c]));
      tc::sts4(out + SUM_V + c * 8, reinterpret_cast<const uint32_t*>(&dv[c]));
    }
  }
  __syncwarp();
  tc::tc_fence_before();
  pdl_wait();
  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem_base, 512);
  if (raised(0) || raised(1) || raised(2)) plain_items<HD>(P, base, flag + 12, n_it, t0, per_head);
  if (slices > 1) tc::cluster_sync_all();
  const int rows = BKT / slices;                             // of either matrix, that this block finishes
  for (int e = threadIdx.x; e < 2 * rows * (HD / 4); e += BWD_THREADS) {
    const bool is_v = e >= rows * (HD / 4);
    const int row = slice * rows + e / (HD / 4) % rows, col = e % (HD / 4) * 4;
    const uint32_t at = base + (uint32_t)(((is_v ? BKT : 0) + row) * (HD + 4) + col) * 4;
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    if (slices == 1) sum = tc::lds4(at);
    else
#pragma unroll 4
      for (int c = 0; c < slices; ++c) {
        float4 f;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(f.x), "=f"(f.y), "=f"(f.z), "=f"(f.w) : "r"(tc::map_to_cta(at, c)) : "memory");
        sum.x += f.x; sum.y += f.y; sum.z += f.z; sum.w += f.w;
      }
    if (j0 + row >= P.t_pad_k) continue;
    const bool live = j0 + row < P.seq_k;
    const float f = is_v ? 1.f : P.scale;
    *reinterpret_cast<float4*>((is_v ? P.dv : P.dk) + rt_off<32>(P.n_pad_k, (long long)b * P.t_pad_k + j0 + row, g * HD + col)) =
        live ? make_float4(sum.x * f, sum.y * f, sum.z * f, sum.w * f) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncwarp();
  if (slices > 1) tc::cluster_sync_all();                    // no block leaves while another may still read its sums
}

template <int HD>
cudaError_t bwd_launch(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* dA, const float* lse, const float* dvec,
                       void* dQ, void* dK, void* dV, int32_t* status, cudaStream_t st) {
  auto k = attn_bwd_tc_f32_kernel<HD>;
  // slices of a key tile's items: an item each at least, and blocks for all SMs at once at most
  const int key_tiles = (p->t_pad_kv + BKT - 1) / BKT, items = (p->d.seq + BQT - 1) / BQT * p->group;
  int slices = 1;
  while (slices < 8 && 2 * slices <= items && (long long)key_tiles * p->d.n_kv_heads * p->d.batch * slices * 2 <= p->sm_count) slices *= 2;
  const dim3 grid(key_tiles * slices, p->d.n_kv_heads, p->d.batch);
  auto make = [&](F32BwdParams& P) {
    memset(&P, 0, sizeof(P));
    P.n_pad = p->n_pad; P.n_pad_k = p->n_pad_kv; P.seq = p->d.seq; P.t_pad = p->t_pad; P.seq_k = p->seq_kv; P.t_pad_k = p->t_pad_kv;
    P.hq = p->d.n_q_heads; P.group = p->group; P.causal = p->d.causal; P.scale = p->scale; P.slices = slices;
    if (!fbl_encode_seq_map(&P.tq, true, Q, p->t_pad, p->d.batch, p->dq / 32, BQT, HD / 32) ||
        !fbl_encode_seq_map(&P.tdo, true, dA, p->t_pad, p->d.batch, p->dq / 32, BQT, HD / 32) ||
        !fbl_encode_seq_map(&P.tk, true, K, p->t_pad_kv, p->d.batch, p->dkv / 32, BKT, HD / 32) ||
        !fbl_encode_seq_map(&P.tv, true, V, p->t_pad_kv, p->d.batch, p->dkv / 32, BKT, HD / 32))
      return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BwdSmem::TOTAL);
  };
  auto point = [&](F32BwdParams& P) {
    P.q = (const float*)Q; P.k = (const float*)K; P.v = (const float*)V; P.dO = (const float*)dA;
    P.lse = lse; P.dvec = dvec; P.dq = (float*)dQ; P.dk = (float*)dK; P.dv = (float*)dV; P.status = status;
    return fbl_map_set_base(&P.tq, Q) && fbl_map_set_base(&P.tdo, dA) && fbl_map_set_base(&P.tk, K) && fbl_map_set_base(&P.tv, V);
  };
  LaunchKey key;
  key.add(1, 0);
  return LaunchMemo<F32BwdParams, 4>::run(p, FBL_MEMO_TC_F32_BWD, key, make, point, [&](const F32BwdParams& P) {
    return slices > 1 ? launch_cluster(k, grid, dim3(BWD_THREADS), BwdSmem::TOTAL, st, slices, true, P)
                      : launch_pdl(k, grid, dim3(BWD_THREADS), BwdSmem::TOTAL, st, P);
  });
}

}  // namespace

// Which plans run here: one answer for both directions, whose scores have to agree.  Blocks are four times as tall as on the FP32
// pipe and fill an SM, so short sequences stay there.  Forward / backward against the FP32 pipe (us), causal, heads of 64: 8 heads
// of 24 tokens x 16 sequences 7.7 / 13 and 6.3 / 9; of 64 tokens 8 / 14 and 10 / 22, x 64 sequences 29 / 52 and 22 / 45; 12 heads of
// 197 tokens x 4 16 / 32 and 36 / 70; 4 heads of 2048 82 / 104 and 199 / 300; 8 x 100 queries over 8 rows x 16 8.6 / 19 and 8.6 / 25.
// With half a tile of keys or less, and query blocks for several rounds, what counts is what a block takes by itself.  Steps over 16
// memory rows, here / on the FP32 pipe: 96 x 8 heads of 80 queries 342 / 288, 32 x 16 heads of 200 queries 364 / 347, of 500 742 /
// 738; 32 x 8 heads of 80 equal, of 200 with one KV head to four 251 / 266, 8 x 16 heads of 1500 572 / 616; over 48 rows from
// equal to half of it.
// Heads of 32: 64 tokens 6.5 / 10.4 and 7.1 / 9.9; 100 tokens of 8 heads x 32 19 / 33 and 22 / 45; 1500 queries over 16 rows x 4
// 20 / 41 and 13 / 34, 16 over 1500 58 / 31 and 106 / 23.
bool attn_tc_f32_supported(const fbl_plan* p) {
  if (p->d.dtype != FBL_DTYPE_FP32 || p->ffma_only || p->d.head_dim > 64) return false;
  const int longer = p->d.seq > p->seq_kv ? p->d.seq : p->seq_kv;
  if (p->d.head_dim == 32) return longer > 64 && p->seq_kv > 64;
  const bool rounds = (long long)p->d.batch * p->d.n_q_heads > 2 * p->sm_count;
  return longer > 64 ? p->seq_kv > 32 || !rounds : longer > 32 && !rounds;
}

cudaError_t launch_attn_fwd_tc_f32(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse, int32_t* status,
                                   cudaStream_t st) {
  return p->d.head_dim == 32 ? fwd_launch<32>(p, Q, K, V, A, lse, status, st) : fwd_launch<64>(p, Q, K, V, A, lse, status, st);
}

cudaError_t launch_attn_bwd_tc_f32(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* A, const void* dA,
                                   const float* lse, float* dvec, void* dQ, void* dK, void* dV, bool dvec_ready, int32_t* status,
                                   cudaStream_t st) {
  cudaError_t e = launch_attn_bwd_pre(p, A, dA, dvec, dvec_ready, st);
  if (e != cudaSuccess) return e;
  return p->d.head_dim == 32 ? bwd_launch<32>(p, Q, K, V, dA, lse, dvec, dQ, dK, dV, status, st)
                             : bwd_launch<64>(p, Q, K, V, dA, lse, dvec, dQ, dK, dV, status, st);
}

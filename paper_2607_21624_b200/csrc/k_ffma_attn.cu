// Attention in fp32 arithmetic on the FP32 pipe (plain FFMA, no tensor cores), operands in R-Tile order fetched by TMA into
// the swizzled 128-byte rows they are stored as (see k_ffma_gemm.cu for the operand fragments): fp32 storage (short sequences
// and heads of 128: the others run on the tensor cores, k_tc_f32_attn.cu), and the backward of bf16 storage where P and dS stay in
// fp32 (attn_fp32), whose operands are widened on their way to registers.
//
// Both kernels give a warp 16 rows of the score tile and all its columns (lane = (row group tm of 4, column group tn of
// 8), 4 x 8 scores per thread), so that the softmax needs only shuffles and the rows of P (forward) or of P^T and dS^T
// (backward) are written and read back by the warp that owns them.  Score products take their pairs for the two-wide
// multiply-adds along head_dim (both operands lie that way), the others along the result's columns.  A block is two
// warps: few rows per block, because a layer of a few hundred tokens has few blocks for 148 SMs and a ragged tail.
// Operand tiles are single-buffered and refetched as soon as their last reader is done, which is early: K behind the
// scores, V behind P V; dO behind dV, Q behind dK, with dQ still to come.
// The bound is the FP32 pipe; shared-memory loads take about three quarters of its time.
// Measured against kernels with one element per load and 256 threads per 64 rows: 4 sequences of 197 tokens, 12 heads of
// 64: forward 54 -> 38 us, backward with its dQ pass 120 -> 72 us (few warps per SM: 4 to 5 at this size).
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "fbl_internal.h"
#include "launch_memo.h"
#include "pdl.cuh"
#include "tc_common.cuh"

namespace {

constexpr int WARPS = 2, THREADS = 32 * WARPS, ROWS = 16 * WARPS;       // rows (queries forward, keys backward) of a block

typedef unsigned long long f2;              // two fp32 values of one two-wide operation
__device__ __forceinline__ f2 pack2(float x, float y) { f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y)); return r; }
__device__ __forceinline__ float2 unpack2(f2 v) { float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v)); return r; }
__device__ __forceinline__ void fma2(f2& d, f2 a, f2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ void lds2x2(uint32_t a, f2& x, f2& y) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "r"(a) : "memory");
}
using tc::lds4;
__device__ __forceinline__ void sts(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }

__device__ __forceinline__ void sts4(uint32_t a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// Four neighbouring columns (group c4) of a row of a tile of R rows, which lies in shared memory as TMA leaves it.
template <typename T, int R>
__device__ __forceinline__ void ld4(uint32_t tile, int row, int c4, f2& x, f2& y) {
  if constexpr (sizeof(T) == 4) {
    lds2x2(tile + (c4 / 8) * (R * 128) + row * 128 + (((c4 % 8) ^ (row & 7)) << 4), x, y);
  } else {
    uint32_t lo, hi;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(lo), "=r"(hi)
                 : "r"(tile + (c4 / 16) * (R * 128) + row * 128 + (((c4 % 16 / 2) ^ (row & 7)) << 4) + c4 % 2 * 8) : "memory");
    x = pack2(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u));
    y = pack2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
  }
}
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16* p, float4 v) { *reinterpret_cast<uint2*>(p) = make_uint2(tc::pack_bf16(v.x, v.y), tc::pack_bf16(v.z, v.w)); }

struct alignas(64) FfmaAttnParams {
  CUtensorMap tq, tk, tv, tdo;
  float* a;                     // forward: merged-head output [n_pad, dq]
  float* lse;                   // [B, Hq, t_pad]
  const float* dvec;            // backward: D = rowsum(dO * O)
  float* dq;                    // backward: zeroed dQ in fp32 (in the storage type's element order), added into
  void *dk, *dv;
  long long n_pad, n_pad_k;
  int seq, t_pad, seq_k, t_pad_k, hq, group, causal;
  int slices;                   // backward: blocks of a cluster, which share a key tile's items
  float scale;
  int32_t* status;
};

// s[i][j] = rows a (row ra + 4 i) times rows b (row tn + 8 j), reduced over head_dim.
template <typename T, int HD, int JN, int AR, int BR>
__device__ __forceinline__ void scores(uint32_t a_tile, uint32_t b_tile, int ra, int tn, float (&s)[4][JN]) {
  f2 acc[4][JN];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < JN; ++j) acc[i][j] = 0ull;
#pragma unroll 2
  for (int kq = 0; kq < HD / 4; ++kq) {
    f2 a[4][2], b[JN][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) ld4<T, AR>(a_tile, ra + 4 * i, kq, a[i][0], a[i][1]);
#pragma unroll
    for (int j = 0; j < JN; ++j) ld4<T, BR>(b_tile, tn + 8 * j, kq, b[j][0], b[j][1]);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < JN; ++j) fma2(acc[i][j], a[i][q], b[j][q]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < JN; ++j) { const float2 v = unpack2(acc[i][j]); s[i][j] = v.x + v.y; }
}

// acc[i][..] += sum over n rows k of tile b of w[row i][k] b[k][columns of this thread]; w: this thread's four rows in
// shared memory, four rows of pitch `ld` apart.
template <typename T, int HD, int BR>
__device__ __forceinline__ void weighted(uint32_t w, int ld, uint32_t b_tile, int tn, int n, f2 (&acc)[4][HD / 16]) {
#pragma unroll 2
  for (int k0 = 0; k0 < n; k0 += 4) {
    f2 b[4][HD / 16];
    float a[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int p = 0; p < HD / 32; ++p)
        ld4<T, BR>(b_tile, k0 + k, p * 8 + tn, b[k][2 * p], b[k][2 * p + 1]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 v = lds4(w + (4 * i * ld + k0) * 4);
      a[i][0] = v.x; a[i][1] = v.y; a[i][2] = v.z; a[i][3] = v.w;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const f2 aa = pack2(a[i][k], a[i][k]);
#pragma unroll
        for (int c = 0; c < HD / 16; ++c) fma2(acc[i][c], aa, b[k][c]);
      }
  }
}

// ------------------------------------------------------------------------------------------
// Forward: one block per (32-query tile, head, batch); online row softmax over 64-key tiles.
// ------------------------------------------------------------------------------------------
constexpr int FWD_KEYS = 64, FWD_LD = FWD_KEYS + 8;
template <int HD>
struct FfmaFwdSmem {
  static constexpr uint32_t K_OFF = 0, V_OFF = HD * FWD_KEYS * 4, Q_OFF = 2 * V_OFF, P_OFF = Q_OFF + HD * ROWS * 4;
  static constexpr uint32_t BAR_OFF = P_OFF + ROWS * FWD_LD * 4, TOTAL = BAR_OFF + 16 + 1024;
};

template <int HD>
__global__ void __launch_bounds__(THREADS) attn_fwd_ffma_kernel(const __grid_constant__ FfmaAttnParams P) {
  using SM = FfmaFwdSmem<HD>;
  constexpr int PN = HD / 32;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u, bar_k = base + SM::BAR_OFF, bar_v = bar_k + 8;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, tm = lane % 4, tn = lane / 4;
  // later queries first: under a causal mask they have the most keys
  const int i0 = ((int)gridDim.x - 1 - (int)blockIdx.x) * ROWS, h = blockIdx.y, b = blockIdx.z, g = h / P.group;
  const int row0 = b * P.t_pad;
  const int j_end = P.causal ? min(P.seq_k, i0 + ROWS) : P.seq_k, n_tiles = (j_end + FWD_KEYS - 1) / FWD_KEYS;
  auto load = [&](const CUtensorMap* map, uint32_t dst, uint32_t bar, int j) {
    tc::mbar_expect_tx(bar, HD * FWD_KEYS * 4);
    tc::tma_load_4d(dst, map, bar, 0, j * FWD_KEYS, b, g * PN);
  };
  if (threadIdx.x == 0) {
    tc::mbar_init(bar_k, 1);
    tc::mbar_init(bar_v, 1);
    tc::fence_barrier_init();
    pdl_wait();
    tc::mbar_expect_tx(bar_k, HD * (FWD_KEYS + ROWS) * 4);
    tc::tma_load_4d(base + SM::Q_OFF, &P.tq, bar_k, 0, i0, b, h * PN);
    tc::tma_load_4d(base + SM::K_OFF, &P.tk, bar_k, 0, 0, b, g * PN);
    load(&P.tv, base + SM::V_OFF, bar_v, 0);
  }
  __syncthreads();
  pdl_launch_dependents();
  pdl_wait();
  float m[4], l[4];
  f2 o[4][HD / 16];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = -INFINITY; l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < HD / 16; ++c) o[i][c] = 0ull;
  }
  const uint32_t p_row = base + SM::P_OFF + (warp * 16 + tm) * FWD_LD * 4;
  bool ok = true;
  // JN: groups of eight keys of the tile that are worked through (four where no more than 32 keys are left)
  auto tile = [&](auto jn_tag, int j) -> bool {
    constexpr int JN = decltype(jn_tag)::value;
    const int j0 = j * FWD_KEYS;
    ok = tc::mbar_wait(bar_k, j & 1, P.status, 131);
    float s[4][JN];
    scores<float, HD, JN, ROWS, FWD_KEYS>(base + SM::Q_OFF, base + SM::K_OFF, warp * 16 + tm, tn, s);
    if (__syncthreads_or(!ok)) return false;               // all warps are done with K
    if (threadIdx.x == 0 && j + 1 < n_tiles) load(&P.tk, base + SM::K_OFF, bar_k, j + 1);
    const bool need_mask = j0 + JN * 8 > P.seq_k || (P.causal && j0 + JN * 8 - 1 > i0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int gi = i0 + warp * 16 + tm + 4 * i;
      float mx = -INFINITY;
#pragma unroll
      for (int jj = 0; jj < JN; ++jj) {
        const int gj = j0 + tn + 8 * jj;
        s[i][jj] *= P.scale;
        if (need_mask && (gj >= P.seq_k || (P.causal && gj > gi))) s[i][jj] = -INFINITY;
        mx = fmaxf(mx, s[i][jj]);
      }
#pragma unroll
      for (int x = 4; x < 32; x *= 2) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
      const float m_new = fmaxf(m[i], mx);
      const float alpha = m_new == -INFINITY ? 1.f : expf(m[i] - m_new);
      float sum = 0.f;
#pragma unroll
      for (int jj = 0; jj < JN; ++jj) {
        const float p = m_new == -INFINITY ? 0.f : expf(s[i][jj] - m_new);
        sts(p_row + (4 * i * FWD_LD + tn + 8 * jj) * 4, p);
        sum += p;
      }
#pragma unroll
      for (int x = 4; x < 32; x *= 2) sum += __shfl_xor_sync(0xffffffffu, sum, x);
      l[i] = l[i] * alpha + sum;
      m[i] = m_new;
      const f2 al = pack2(alpha, alpha);
#pragma unroll
      for (int c = 0; c < HD / 16; ++c) o[i][c] = mul2(o[i][c], al);
    }
    __syncwarp();
    ok = tc::mbar_wait(bar_v, j & 1, P.status, 132);
    weighted<float, HD, FWD_KEYS>(p_row, FWD_LD, base + SM::V_OFF, tn, JN * 8, o);
    if (__syncthreads_or(!ok)) return false;               // ... and with V
    if (threadIdx.x == 0 && j + 1 < n_tiles) load(&P.tv, base + SM::V_OFF, bar_v, j + 1);
    return true;
  };
  using Full = std::integral_constant<int, 8>;
  using Half = std::integral_constant<int, 4>;
  for (int j = 0; j < n_tiles; ++j)
    if (!(j_end - j * FWD_KEYS > 32 ? tile(Full{}, j) : tile(Half{}, j))) return;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int gi = i0 + warp * 16 + tm + 4 * i;
    if (gi >= P.t_pad) continue;
    const bool live = gi < P.seq;
    const float inv = live ? 1.f / l[i] : 0.f;
#pragma unroll
    for (int p = 0; p < PN; ++p) {
      const float2 x = unpack2(o[i][2 * p]), y = unpack2(o[i][2 * p + 1]);
      st4(P.a + rt_off<32>(P.n_pad, row0 + gi, h * HD + p * 32 + tn * 4),
          live ? make_float4(x.x * inv, x.y * inv, y.x * inv, y.y * inv) : make_float4(0.f, 0.f, 0.f, 0.f));
    }
    if (tn == 0) P.lse[((long long)b * P.hq + h) * P.t_pad + gi] = live ? m[i] + logf(l[i]) : 0.f;
  }
}

// ------------------------------------------------------------------------------------------
// Backward: one block per (32-key tile, KV head, batch).  dK and dV stay in registers over the query tiles and the G
// query heads of the group; dQ reduces over the key tiles and is added into its zeroed buffer with 16-byte reductions.
// Where that makes fewer blocks than SMs (few sequences, few KV heads), a cluster of 2 to 8 blocks takes a key tile's
// (query head, query tile) items in turn and adds its dK and dV through distributed shared memory in a fixed order: the
// bound is the items' chain, some 6 us each.
// ------------------------------------------------------------------------------------------
template <typename T, int HD>
struct FfmaBwdSmem {
  static constexpr int QT = HD == 128 ? 32 : 64, LD = QT + 8;            // queries of a tile; pitch of P^T and dS^T rows
  static constexpr uint32_t E = sizeof(T), K_OFF = 0, V_OFF = HD * ROWS * E, Q_OFF = 2 * V_OFF, DO_OFF = Q_OFF + HD * QT * E;
  static constexpr uint32_t P_OFF = DO_OFF + HD * QT * E, S_OFF = P_OFF + ROWS * LD * 4;
  // slices: a block's dK and dV in fp32, over the operand tiles when they are free
  static constexpr uint32_t SUM_K = 0, SUM_V = HD * ROWS * 4;
  static_assert(2 * SUM_V <= P_OFF, "");
  static constexpr uint32_t BAR_OFF = S_OFF + ROWS * LD * 4, TOTAL = BAR_OFF + 24 + 1024;
};

template <typename T, int HD>
__global__ void __launch_bounds__(THREADS) attn_bwd_ffma_kernel(const __grid_constant__ FfmaAttnParams P) {
  using SM = FfmaBwdSmem<T, HD>;
  constexpr int TW = tile_w_of<T>::value, PN = HD / TW, QT = SM::QT, LD = SM::LD;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u, bar_kv = base + SM::BAR_OFF, bar_q = bar_kv + 8, bar_do = bar_kv + 16;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, tm = lane % 4, tn = lane / 4;
  const int slices = P.slices, slice = blockIdx.x % slices;
  const int j0 = blockIdx.x / slices * ROWS, g = blockIdx.y, b = blockIdx.z;      // key tile 0 has the most queries: first
  const int row0 = b * P.t_pad, row0k = b * P.t_pad_k;
  const int t0 = P.causal ? j0 / QT : 0, per_head = (P.seq + QT - 1) / QT - t0, n_it = max(0, per_head) * P.group;
  auto load = [&](const CUtensorMap* map, uint32_t dst, uint32_t bar, int it) {
    tc::mbar_expect_tx(bar, HD * QT * SM::E);
    tc::tma_load_4d(dst, map, bar, 0, (t0 + it % per_head) * QT, b, (g * P.group + it / per_head) * PN);
  };
  if (threadIdx.x == 0) {
    tc::mbar_init(bar_kv, 1);
    tc::mbar_init(bar_q, 1);
    tc::mbar_init(bar_do, 1);
    tc::fence_barrier_init();
    pdl_wait();
    tc::mbar_expect_tx(bar_kv, 2 * HD * ROWS * SM::E);
    tc::tma_load_4d(base + SM::K_OFF, &P.tk, bar_kv, 0, j0, b, g * PN);
    tc::tma_load_4d(base + SM::V_OFF, &P.tv, bar_kv, 0, j0, b, g * PN);
    if (slice < n_it) {
      load(&P.tq, base + SM::Q_OFF, bar_q, slice);
      load(&P.tdo, base + SM::DO_OFF, bar_do, slice);
    }
  }
  __syncthreads();
  pdl_launch_dependents();
  pdl_wait();
  f2 dk[4][HD / 16], dv[4][HD / 16];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < HD / 16; ++c) dk[i][c] = dv[i][c] = 0ull;
  const int ra = warp * 16 + tm;
  const uint32_t p_row = base + SM::P_OFF + ra * LD * 4, s_row = base + SM::S_OFF + ra * LD * 4;
  bool ok = tc::mbar_wait(bar_kv, 0, P.status, 133);
  // JN: groups of eight queries of the tile that are worked through
  auto tile = [&](auto jn_tag, int it, int phase) -> bool {
    constexpr int JN = decltype(jn_tag)::value;
    const int h = g * P.group + it / per_head, i0 = (t0 + it % per_head) * QT;
    const bool need_mask = i0 + JN * 8 > P.seq || j0 + ROWS > P.seq_k || (P.causal && i0 < j0 + ROWS - 1);
    float lse[JN], d[JN];
    const long long at = ((long long)b * P.hq + h) * P.t_pad;
#pragma unroll
    for (int j = 0; j < JN; ++j) {
      const int gi = i0 + tn + 8 * j;
      lse[j] = gi < P.seq ? P.lse[at + gi] : 0.f;
      d[j] = gi < P.seq ? P.dvec[at + gi] : 0.f;
    }
    ok = tc::mbar_wait(bar_q, phase, P.status, 134) && ok;
    float p[4][JN], dp[4][JN];
    scores<T, HD, JN, ROWS, QT>(base + SM::K_OFF, base + SM::Q_OFF, ra, tn, p);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < JN; ++j) {
        const int gi = i0 + tn + 8 * j, gj = j0 + ra + 4 * i;
        p[i][j] = need_mask && (gi >= P.seq || gj >= P.seq_k || (P.causal && gj > gi)) ? 0.f : expf(p[i][j] * P.scale - lse[j]);
        sts(p_row + (4 * i * LD + tn + 8 * j) * 4, p[i][j]);
      }
    ok = tc::mbar_wait(bar_do, phase, P.status, 135) && ok;
    scores<T, HD, JN, ROWS, QT>(base + SM::V_OFF, base + SM::DO_OFF, ra, tn, dp);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < JN; ++j) sts(s_row + (4 * i * LD + tn + 8 * j) * 4, p[i][j] * (dp[i][j] - d[j]));
    __syncwarp();
    weighted<T, HD, QT>(p_row, LD, base + SM::DO_OFF, tn, JN * 8, dv);
    if (__syncthreads_or(!ok)) return false;               // all warps are done with dO, and dS^T is complete
    if (threadIdx.x == 0 && it + slices < n_it) load(&P.tdo, base + SM::DO_OFF, bar_do, it + slices);
    weighted<T, HD, QT>(s_row, LD, base + SM::Q_OFF, tn, JN * 8, dk);
    __syncthreads();                                       // ... and with Q
    if (threadIdx.x == 0 && it + slices < n_it) load(&P.tq, base + SM::Q_OFF, bar_q, it + slices);
    // dQ = dS K: 16 queries at a time per warp, four neighbouring ones per thread, reduced over the block's keys
#pragma unroll 1
    for (int q0 = warp * 16; q0 < JN * 8; q0 += 16 * WARPS) {
      f2 dq[4][HD / 16];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < HD / 16; ++c) dq[i][c] = 0ull;
#pragma unroll 4
      for (int k = 0; k < ROWS; ++k) {
        f2 kb[HD / 16];
#pragma unroll
        for (int pn = 0; pn < HD / 32; ++pn) ld4<T, ROWS>(base + SM::K_OFF, k, pn * 8 + tn, kb[2 * pn], kb[2 * pn + 1]);
        const float4 v = lds4(base + SM::S_OFF + (k * LD + q0 + tm * 4) * 4);
        const float sv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const f2 aa = pack2(sv[i], sv[i]);
#pragma unroll
          for (int c = 0; c < HD / 16; ++c) fma2(dq[i][c], aa, kb[c]);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int gi = i0 + q0 + tm * 4 + i;
        if (gi >= P.seq) continue;
#pragma unroll
        for (int pn = 0; pn < HD / 32; ++pn) {
          const float2 x = unpack2(dq[i][2 * pn]), y = unpack2(dq[i][2 * pn + 1]);
          atomicAdd(reinterpret_cast<float4*>(P.dq + rt_off<TW>(P.n_pad, row0 + gi, h * HD + pn * 32 + tn * 4)),
                    make_float4(x.x * P.scale, x.y * P.scale, y.x * P.scale, y.y * P.scale));
        }
      }
    }
    __syncthreads();                                       // dS^T may be overwritten
    return true;
  };
  using Full = std::integral_constant<int, QT / 8>;
  using Half = std::integral_constant<int, QT / 16>;
  for (int it = slice, phase = 0; it < n_it; it += slices, phase ^= 1)
    if (!(P.seq - (t0 + it % per_head) * QT > QT / 2 ? tile(Full{}, it, phase) : tile(Half{}, it, phase))) break;
  auto store = [&](void* out, int row, int col, float4 v, float f) {
    if (j0 + row < P.t_pad_k) {
      f = j0 + row < P.seq_k ? f : 0.f;
      st4((T*)out + rt_off<TW>(P.n_pad_k, row0k + j0 + row, g * HD + col), make_float4(v.x * f, v.y * f, v.z * f, v.w * f));
    }
  };
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int pn = 0; pn < HD / 32; ++pn) {
      const int row = ra + 4 * i, col = pn * 32 + tn * 4;
      const float2 x = unpack2(dk[i][2 * pn]), y = unpack2(dk[i][2 * pn + 1]), u = unpack2(dv[i][2 * pn]), w = unpack2(dv[i][2 * pn + 1]);
      const float4 k4 = make_float4(x.x, x.y, y.x, y.y), v4 = make_float4(u.x, u.y, w.x, w.y);
      if (slices == 1) {
        store(P.dk, row, col, k4, P.scale);
        store(P.dv, row, col, v4, 1.f);
      } else {
        sts4(base + SM::SUM_K + (row * HD + col) * 4, k4);
        sts4(base + SM::SUM_V + (row * HD + col) * 4, v4);
      }
    }
  if (slices > 1) {
    tc::cluster_sync_all();
    const int per = ROWS / slices;                         // rows that this block finishes
    for (int e = threadIdx.x; e < 2 * per * (HD / 4); e += THREADS) {
      const int row = slice * per + e / (HD / 4) % per, col = e % (HD / 4) * 4;
      const bool is_v = e >= per * (HD / 4);
      const uint32_t at = base + (is_v ? SM::SUM_V : SM::SUM_K) + (row * HD + col) * 4;
      float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
      for (int c = 0; c < slices; ++c) {
        float4 f;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(f.x), "=f"(f.y), "=f"(f.z), "=f"(f.w) : "r"(tc::map_to_cta(at, c)) : "memory");
        sum.x += f.x; sum.y += f.y; sum.z += f.z; sum.w += f.w;
      }
      store(is_v ? P.dv : P.dk, row, col, sum, is_v ? 1.f : P.scale);
    }
    __syncwarp();
    tc::cluster_sync_all();                                // no block leaves while another may still read its sums
  }
}

// Shared memory to ask for: blocks that all fit the SMs at once spread evenly.  Launched while the kernel in front still
// runs, they would crowd on the SMs that it frees first (84 blocks of the backward: 46 us spread, 61 us crowded; 78 longer
// ones: 730 and 1050 us).  Two or three short ones (few `items` each) to an SM may as well start early.
constexpr uint32_t ALONE = 114 * 1024;                     // with the 1 KB that a block has on top, half an SM's is less
uint32_t spread(const fbl_plan* p, const dim3& grid, int items, uint32_t smem) {
  const long long per_sm = ((long long)grid.x * grid.y * grid.z + p->sm_count - 1) / p->sm_count;
  return per_sm == 1 || (per_sm <= 3 && items >= 4) ? std::max(smem, (uint32_t)(228 * 1024 / (per_sm + 1))) : smem;
}

typedef LaunchMemo<FfmaAttnParams, 4> AttnMemo;

void fill(const fbl_plan* p, FfmaAttnParams& P) {
  memset(&P, 0, sizeof(P));
  P.n_pad = p->n_pad; P.n_pad_k = p->n_pad_kv; P.seq = p->d.seq; P.t_pad = p->t_pad; P.seq_k = p->seq_kv; P.t_pad_k = p->t_pad_kv;
  P.hq = p->d.n_q_heads; P.group = p->group; P.causal = p->d.causal; P.scale = p->scale;
}

static_assert(FfmaFwdSmem<128>::TOTAL <= ALONE && FfmaBwdSmem<float, 128>::TOTAL <= ALONE, "");

template <typename T>
bool encode(CUtensorMap* map, const void* base, int t_pad, int batch, int cols, int rows, int hd) {
  constexpr int TW = tile_w_of<T>::value;
  return fbl_encode_seq_map(map, sizeof(T) == 4, base, t_pad, batch, cols / TW, rows, hd / TW);
}

template <int HD>
cudaError_t fwd_launch(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse, int32_t* status, cudaStream_t st) {
  auto k = attn_fwd_ffma_kernel<HD>;
  const dim3 grid((p->t_pad + ROWS - 1) / ROWS, p->d.n_q_heads, p->d.batch);
  const uint32_t smem = spread(p, grid, (p->t_pad_kv + FWD_KEYS - 1) / FWD_KEYS, FfmaFwdSmem<HD>::TOTAL);
  auto make = [&](FfmaAttnParams& P) {
    fill(p, P);
    if (!encode<float>(&P.tq, Q, p->t_pad, p->d.batch, p->dq, ROWS, HD) || !encode<float>(&P.tk, K, p->t_pad_kv, p->d.batch, p->dkv, FWD_KEYS, HD) ||
        !encode<float>(&P.tv, V, p->t_pad_kv, p->d.batch, p->dkv, FWD_KEYS, HD))
      return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ALONE);
  };
  auto point = [&](FfmaAttnParams& P) {
    P.a = (float*)A; P.lse = lse; P.status = status;
    return fbl_map_set_base(&P.tq, Q) && fbl_map_set_base(&P.tk, K) && fbl_map_set_base(&P.tv, V);
  };
  LaunchKey key;
  key.add(0, 0);                                           // the forward; the rest is the plan's
  return AttnMemo::run(p, FBL_MEMO_FFMA_ATTN, key, make, point, [&](const FfmaAttnParams& P) {
    return launch_pdl(k, grid, dim3(THREADS), smem, st, P);
  });
}

template <typename T, int HD>
cudaError_t bwd_launch(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* dA, const float* lse, const float* dvec,
                       float* dQ, void* dK, void* dV, int32_t* status, cudaStream_t st) {
  constexpr int QT = FfmaBwdSmem<T, HD>::QT;
  auto k = attn_bwd_ffma_kernel<T, HD>;
  // slices of a key tile's items: an item each at least, and no more once there are two blocks per SM (of two warps each,
  // for an SM's four schedulers)
  const int key_tiles = (p->t_pad_kv + ROWS - 1) / ROWS, items = (p->d.seq + QT - 1) / QT * p->group;
  int slices = 1;
  while (slices < 8 && 2 * slices <= items && (long long)key_tiles * p->d.n_kv_heads * p->d.batch * slices <= 2 * p->sm_count) slices *= 2;
  const dim3 grid(key_tiles * slices, p->d.n_kv_heads, p->d.batch);
  const uint32_t smem = slices > 1 ? FfmaBwdSmem<T, HD>::TOTAL : spread(p, grid, items, FfmaBwdSmem<T, HD>::TOTAL);
  auto make = [&](FfmaAttnParams& P) {
    fill(p, P);
    if (!encode<T>(&P.tq, Q, p->t_pad, p->d.batch, p->dq, QT, HD) || !encode<T>(&P.tdo, dA, p->t_pad, p->d.batch, p->dq, QT, HD) ||
        !encode<T>(&P.tk, K, p->t_pad_kv, p->d.batch, p->dkv, ROWS, HD) || !encode<T>(&P.tv, V, p->t_pad_kv, p->d.batch, p->dkv, ROWS, HD))
      return cudaErrorInvalidValue;
    P.slices = slices;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ALONE);
  };
  auto point = [&](FfmaAttnParams& P) {
    P.lse = const_cast<float*>(lse); P.dvec = dvec; P.dq = dQ; P.dk = dK; P.dv = dV; P.status = status;
    return fbl_map_set_base(&P.tq, Q) && fbl_map_set_base(&P.tdo, dA) && fbl_map_set_base(&P.tk, K) && fbl_map_set_base(&P.tv, V);
  };
  LaunchKey key;
  key.add(1, 0);                                           // the backward
  return AttnMemo::run(p, FBL_MEMO_FFMA_ATTN, key, make, point, [&](const FfmaAttnParams& P) {
    return slices > 1 ? launch_cluster(k, grid, dim3(THREADS), smem, st, slices, true, P) : launch_pdl(k, grid, dim3(THREADS), smem, st, P);
  });
}

}  // namespace

cudaError_t launch_attn_fwd_ffma(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse, int32_t* status,
                                 cudaStream_t st) {
  switch (p->d.head_dim) {
    case 32: return fwd_launch<32>(p, Q, K, V, A, lse, status, st);
    case 64: return fwd_launch<64>(p, Q, K, V, A, lse, status, st);
    case 128: return fwd_launch<128>(p, Q, K, V, A, lse, status, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_attn_bwd_ffma(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* A, const void* dA,
                                 const float* lse, float* dvec, float* dqacc, void* dQ, void* dK, void* dV, bool dvec_ready,
                                 int32_t* status, cudaStream_t st, const float2* rope) {
  cudaError_t e = launch_attn_bwd_pre(p, A, dA, dvec, dvec_ready, st);
  if (e != cudaSuccess) return e;
#define FBL_CALL(T_, HD_, DQ_) e = bwd_launch<T_, HD_>(p, Q, K, V, dA, lse, dvec, DQ_, dK, dV, status, st)
  if (p->d.dtype == FBL_DTYPE_BF16) {
    if (p->d.head_dim == 64) FBL_CALL(__nv_bfloat16, 64, dqacc);
    else if (p->d.head_dim == 128) FBL_CALL(__nv_bfloat16, 128, dqacc);
    else e = cudaErrorInvalidValue;
    if (e != cudaSuccess) return e;
    return rope ? launch_rope_bwd_round(p, dqacc, dQ, dK, rope, st) : launch_attn_bwd_post(p, dqacc, dQ, st);
  }
  switch (p->d.head_dim) {
    case 32: FBL_CALL(float, 32, (float*)dQ); break;
    case 64: FBL_CALL(float, 64, (float*)dQ); break;
    case 128: FBL_CALL(float, 128, (float*)dQ); break;
    default: e = cudaErrorInvalidValue;
  }
  return e;
#undef FBL_CALL
}

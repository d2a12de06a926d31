// Projection GEMMs on tcgen05 tensor cores (bf16 in, fp32 accumulate in TMEM, bf16 out), operands in
// R-Tile order fetched by TMA.  One kernel serves all six projection steps and their transposed forms:
// each operand is declared K-major or MN-major in the descriptors, so W / W^T and X / X^T are the same
// tiles in HBM and in shared memory.  Up to four reduction loops feed one accumulator (dXn), and up
// to five problems share one persistent launch (Q/K/V projections; dWo with dA; dWq/dWk/dWv with dXn).
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "fbl_internal.h"
#include "launch_memo.h"
#include "pdl.cuh"
#include "tc_common.cuh"

namespace {

constexpr int BM = 128, BK = 64;
constexpr int MAX_TERMS = 4, MAX_PROBLEMS = 5;

struct alignas(64) TcProblem {
  CUtensorMap ta[MAX_TERMS], tb[MAX_TERMS], tc;     // tc: the output, for the epilogue's bulk stores
  int n_terms;
  int b_static;                                        // 1: the first term's B operand is an input of the whole
                                                       // step (a weight), not written by an earlier kernel
  int kblocks[MAX_TERMS];
  int a_mn[MAX_TERMS], b_mn[MAX_TERMS];   // 1: operand is MN-major in shared memory (its rows are K indices)
  int m, n;
  __nv_bfloat16* c;
  long long c_rpad;
  const float* bias;
  const __nv_bfloat16* residual;
  int seq, t_pad;
  const __nv_bfloat16* dot_with;   // fused D = rowsum(C * dot_with) per head (the attention backward's D), or nullptr
  float* dot_out;
  int dot_hd, dot_hq;
  // Reduction loop cut into `ksplit` slices, each a work unit of its own (a problem with few output tiles and a
  // long reduction): slices add their fp32 partial tiles into `tacc`'s buffer with bulk tensor reductions, and a
  // later kernel rounds the sums to bf16.  Single-term problems without epilogue extras only.
  int ksplit;
  CUtensorMap tacc;
  // Fused activation of the feed-forward block (kernel variant EPI only; `residual` then points at the first extra
  // operand U instead of a residual, `aux1` at the second one, G; `tc2` is the second output's map):
  //   1 GELU forward    C = v (U), C2 = gelu(v)           2 GELU backward    C = v gelu'(U)
  //   3 gated forward   C = v (G), C2 = silu(v) U          4 gated backward   C = v silu(G), C2 = v U silu'(G)
  //   5 rotary embedding C = v with each 64-column head's (i, i + 32) pairs turned by the table's angle of the row's token
  const float2* rope;      // [32][t_pad] cosine and sine
  int epi;
  const __nv_bfloat16* aux1;
  CUtensorMap tc2;
};
struct alignas(64) TcGroup {
  TcProblem p[MAX_PROBLEMS];
  int count;
  int late_trigger;                          // as in GemmArgs: the dependents' trigger comes after the wait
  int slices;                                // gemm_tc_split_kernel: blocks of a cluster, which share a tile's reduction
  int32_t* status;
  // Optional chores for the epilogue warps while the first tile's main loop runs: zero-fill a buffer that a later
  // kernel of the pass adds into (16-byte units, dealt evenly to the blocks), and reset the pass's status word.
  uint4* zero_ptr;
  long long zero_vec;
  int reset_status;
};

__device__ __forceinline__ void group_chores(const TcGroup& G, int tid, int n_threads) {
  if (G.reset_status && blockIdx.x == 0 && tid == 0) *G.status = G.status[FBL_EARLY_COLSUM] = G.status[FBL_EARLY_ROUND] = 0;
  if (G.zero_vec > 0) {
    const long long per = (G.zero_vec + gridDim.x - 1) / gridDim.x;
    const long long lo = (long long)blockIdx.x * per, hi = min(G.zero_vec, lo + per);
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    for (long long i = lo + tid; i < hi; i += n_threads) G.zero_ptr[i] = z;
  }
}

// By the producer thread, after its pdl_wait(): whatever precedes the launch is complete for who sees the flag.
__device__ __forceinline__ void late_trigger(const TcGroup& G) {
  if (blockIdx.x == 0) pdl_raise(G.status + FBL_EARLY_COLSUM);
  pdl_launch_dependents();
}

template <int BN, int STAGES>
struct SmemPlan {
  static constexpr uint32_t A_BYTES = BM * 128;
  static constexpr uint32_t B_BYTES = BN * 128;
  static constexpr uint32_t STAGE = A_BYTES + B_BYTES;
  static constexpr uint32_t STG_OFF = STAGES * STAGE;    // per epilogue warp two 32 x 64 bf16 output staging tiles
  static constexpr uint32_t BAR_OFF = STG_OFF + 2 * 16384;
  static constexpr uint32_t N_BARS = 2 * STAGES + 4;     // full[], empty[], acc_full[2], acc_empty[2]
  static constexpr uint32_t TOTAL = BAR_OFF + 8 * N_BARS + 16 + 1024;   // + TMEM slot + alignment slack
};

// Work list of a launch: output tiles of all problems, numbered problem by problem with the M tile index
// fastest (blocks that run together then share the B tiles of one weight column block through L2).
struct TileCoord { int prob, m0, n0, kb0, kb1; };     // kb0..kb1: k-block range of term 0 (split problems)

template <int BN>
__device__ __forceinline__ bool tile_at(const TcGroup& G, int w, TileCoord* tc_out) {
  for (int p = 0; p < G.count; ++p) {
    const TcProblem& P = G.p[p];
    const int tm = (P.m + BM - 1) / BM, tn = (P.n + BN - 1) / BN;
    const int units = tm * tn * P.ksplit;
    if (w < units) {
      const int slice = w % P.ksplit, t = w / P.ksplit;        // slices of one tile are neighbours in the list
      tc_out->prob = p;
      tc_out->m0 = (t % tm) * BM;
      tc_out->n0 = (t / tm) * BN;
      const int per = (P.kblocks[0] + P.ksplit - 1) / P.ksplit;
      tc_out->kb0 = slice * per;
      tc_out->kb1 = min(P.kblocks[0], (slice + 1) * per);
      return true;
    }
    w -= units;
  }
  return false;
}

__device__ __forceinline__ float tanh_fast(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float gelu_fast(float u) { return 0.5f * u * (1.f + tanh_fast(0.7978845608028654f * (u + 0.044715f * u * u * u))); }
__device__ __forceinline__ float gelu_grad_fast(float u) {
  const float t = tanh_fast(0.7978845608028654f * (u + 0.044715f * u * u * u));
  return 0.5f * (1.f + t) + 0.5f * u * (1.f - t * t) * 0.7978845608028654f * (1.f + 0.134145f * u * u);
}
__device__ __forceinline__ float sigmoid_fast(float g) { return __fdividef(1.f, 1.f + __expf(-g)); }

// A warp's lanes of an accumulator in tensor memory.
struct TmemAcc {
  uint32_t addr;
  __device__ __forceinline__ void load(int col, uint32_t (&v)[32]) const { tc::tmem_ld32(addr + col, v); }
  __device__ __forceinline__ void wait() const { tc::tmem_ld_wait(); }
};

// One output tile of a CTA's 128 accumulator rows: TMEM -> registers -> swizzled staging -> bulk tensor store.  Each warp
// owns the 32 rows of its TMEM lane quarter and its staging tiles, and issues its own stores: no block-wide hand-off per
// panel, and the store of one panel overlaps the conversion of the next.  `q`: which 32 rows; `acc`: reads 32 columns of
// them (this lane's row); `wait`: waits until they are complete (what does not depend on them is requested first).
// ESETS = 2 (launches in which every block has a single tile, so that nothing overlaps its epilogue): two sets of four
// warps share the tile's 64-column panels, first and second half, and the epilogue takes half as long.  Each warp then
// has one staging tile instead of two (the staging area is the same size).
// EPI: what the instantiation can fuse besides bias, residual and the row reduction.
enum { EPI_NONE = 0, EPI_ACT, EPI_ROPE };
template <int BN, int ESETS, int EPI, typename Acc, typename Wait>
__device__ __forceinline__ bool epilogue_tile(const TcProblem& P, int m0, int n0, int q, Acc acc, uint32_t stg0, int& pc, Wait wait) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, set = (warp - 2) / 4;
  constexpr int PPS = BN / 64 / ESETS;              // panels per set
  const int row = m0 + q * 32 + lane;               // row of the problem owned by this thread
  const bool pad = P.t_pad > 0 && (row % P.t_pad) >= P.seq;
  const bool has_res = P.residual && row < P.m;
  // a head of the fused row reduction must stay within one warp: where it spans more panels than a set has, the first set
  // takes the whole tile
  const bool whole = ESETS == 2 && P.dot_with && P.dot_hd > 64 * PPS;
  const int pn_begin = set == 0 ? 0 : (whole ? BN / 64 : PPS);
  const int pn_end = ESETS == 1 ? BN / 64 : (set == 0 ? (whole ? BN / 64 : PPS) : BN / 64);
  uint4 rv[8];                                    // residual values of the next panel, requested a panel ahead
  if (has_res && pn_begin < pn_end && n0 + pn_begin * 64 < P.n) {
    const __nv_bfloat16* rp = P.residual + ((long long)(n0 / 64 + pn_begin) * P.c_rpad + row) * 64;
#pragma unroll
    for (int j = 0; j < 8; ++j) rv[j] = *reinterpret_cast<const uint4*>(rp + 8 * j);
  }
  uint4 rv2[EPI == EPI_ACT ? 8 : 1];                         // second extra operand of a fused activation, likewise
  if constexpr (EPI == EPI_ACT) {
    if (P.epi == 4 && row < P.m && pn_begin < pn_end && n0 + pn_begin * 64 < P.n) {
      const __nv_bfloat16* rp = P.aux1 + ((long long)(n0 / 64 + pn_begin) * P.c_rpad + row) * 64;
#pragma unroll
      for (int j = 0; j < 8; ++j) rv2[j] = *reinterpret_cast<const uint4*>(rp + 8 * j);
    }
  }
  const float* bias = P.bias;
  float bl[BN / 32];                              // this tile's bias: lane l holds columns l*BN/32 ... (requested
  if (bias) {                                     // while the MMAs run, handed out by shuffles below)
#pragma unroll
    for (int k = 0; k < BN / 32; ++k) {
      const int c = n0 + lane * (BN / 32) + k;
      bl[k] = c < P.n ? bias[c] : 0.f;
    }
  }
  if (!wait()) return false;
  tc::tc_fence_after();
  float dot_acc = 0.f;
#pragma unroll 1
  for (int pn = pn_begin; pn < pn_end; ++pn) {
    const int n = n0 + pn * 64;
    if (n >= P.n) break;                           // uniform: N is whole 64-column panels
    uint32_t v[64];
    acc.load(pn * 64, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
    acc.load(pn * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32]));
    acc.wait();
    if (P.ksplit > 1) {
      // partial sums of a reduction slice: two 32-column halves of the panel, fp32, added to the accumulation
      // buffer by bulk tensor reductions (same staging tiles and swizzle as the bf16 rows below)
#pragma unroll 1
      for (int hf = 0; hf < 2; ++hf) {
        const uint32_t stg = stg0 + (ESETS == 2 ? (uint32_t)(warp - 2) : (uint32_t)(q * 2 + (pc & 1))) * 4096u;
        if (ESETS == 2 && lane == 0) tc::bulk_wait_group_read0();     // the single staging tile's previous contents have been read
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j)
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stg + lane * 128 + (((uint32_t)j ^ (uint32_t)(lane & 7)) * 16)),
                       "r"(hf ? v[32 + 4 * j] : v[4 * j]), "r"(hf ? v[33 + 4 * j] : v[4 * j + 1]),
                       "r"(hf ? v[34 + 4 * j] : v[4 * j + 2]), "r"(hf ? v[35 + 4 * j] : v[4 * j + 3]) : "memory");
        tc::fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          tc::tma_reduce_add_4d(&P.tacc, stg, 0, hf, m0 + q * 32, n / 64);
          tc::bulk_commit_group();
          if (ESETS == 1) tc::bulk_wait_group_read1();
        }
        ++pc;
      }
      continue;
    }
    if constexpr (EPI == EPI_ACT) {
      if (P.epi != 0) {
        // ---- fused activation: one or two outputs from this panel ------------------------------------
        if (bias) {
#pragma unroll
          for (int j = 0; j < 64; ++j)
            v[j] = __float_as_uint(__uint_as_float(v[j]) + __shfl_sync(0xffffffffu, bl[j % (BN / 32)], (pn * 64 + j) / (BN / 32)));
        }
        uint4 o1[8], o2[8];
        uint32_t* w1 = reinterpret_cast<uint32_t*>(o1);
        uint32_t* w2 = reinterpret_cast<uint32_t*>(o2);
        const bool live = !pad && row < P.m;
        const __nv_bfloat16* a0 = reinterpret_cast<const __nv_bfloat16*>(rv);
        const __nv_bfloat16* a1 = reinterpret_cast<const __nv_bfloat16*>(rv2);
        const float keep = live ? 1.f : 0.f;            // padding rows and rows past the matrix are written as zero
        if (P.epi == 1) {
#pragma unroll
          for (int j = 0; j < 64; j += 2) {
            const float x0 = __uint_as_float(v[j]) * keep, x1 = __uint_as_float(v[j + 1]) * keep;
            w1[j / 2] = tc::pack_bf16(x0, x1);
            w2[j / 2] = tc::pack_bf16(gelu_fast(x0), gelu_fast(x1));
          }
        } else if (P.epi == 2) {
#pragma unroll
          for (int j = 0; j < 64; j += 2) {
            const float x0 = __uint_as_float(v[j]) * keep, x1 = __uint_as_float(v[j + 1]) * keep;
            w1[j / 2] = tc::pack_bf16(x0 * gelu_grad_fast(__bfloat162float(a0[j])), x1 * gelu_grad_fast(__bfloat162float(a0[j + 1])));
          }
        } else if (P.epi == 3) {
#pragma unroll
          for (int j = 0; j < 64; j += 2) {
            const float x0 = __uint_as_float(v[j]) * keep, x1 = __uint_as_float(v[j + 1]) * keep;
            w1[j / 2] = tc::pack_bf16(x0, x1);
            w2[j / 2] = tc::pack_bf16(x0 * sigmoid_fast(x0) * __bfloat162float(a0[j]), x1 * sigmoid_fast(x1) * __bfloat162float(a0[j + 1]));
          }
        } else {
#pragma unroll
          for (int j = 0; j < 64; j += 2) {
            float y1[2], y2[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const float x = __uint_as_float(v[j + u]) * keep;
              const float uu = __bfloat162float(a0[j + u]), gg = __bfloat162float(a1[j + u]), sg = sigmoid_fast(gg);
              y1[u] = x * gg * sg;
              y2[u] = x * uu * sg * (1.f + gg * (1.f - sg));
            }
            w1[j / 2] = tc::pack_bf16(y1[0], y1[1]);
            w2[j / 2] = tc::pack_bf16(y2[0], y2[1]);
          }
        }
        // the next panel's extra operands, requested while this panel's stores are under way
        if (pn + 1 < pn_end && n + 64 < P.n && row < P.m) {
          if (P.epi >= 2) {
            const __nv_bfloat16* rp = P.residual + ((long long)(n / 64 + 1) * P.c_rpad + row) * 64;
#pragma unroll
            for (int j = 0; j < 8; ++j) rv[j] = *reinterpret_cast<const uint4*>(rp + 8 * j);
          }
          if (P.epi == 4) {
            const __nv_bfloat16* rp = P.aux1 + ((long long)(n / 64 + 1) * P.c_rpad + row) * 64;
#pragma unroll
            for (int j = 0; j < 8; ++j) rv2[j] = *reinterpret_cast<const uint4*>(rp + 8 * j);
          }
        }
        const int n_out = (P.epi == 2) ? 1 : 2;
#pragma unroll 1
        for (int oi = 0; oi < n_out; ++oi) {
          const uint4* ov = oi ? o2 : o1;
          const uint32_t stg = stg0 + (ESETS == 2 ? (uint32_t)(warp - 2) : (uint32_t)(q * 2 + (pc & 1))) * 4096u;
          if (ESETS == 2 && lane == 0) tc::bulk_wait_group_read0();
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 8; ++j)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stg + lane * 128 + (((uint32_t)j ^ (uint32_t)(lane & 7)) * 16)),
                         "r"(ov[j].x), "r"(ov[j].y), "r"(ov[j].z), "r"(ov[j].w) : "memory");
          tc::fence_proxy_async();
          __syncwarp();
          if (lane == 0) {
            tc::tma_store_3d(oi ? &P.tc2 : &P.tc, stg, 0, m0 + q * 32, n / 64);
            tc::bulk_commit_group();
            if (ESETS == 1) tc::bulk_wait_group_read1();
          }
          ++pc;
        }
        continue;
      }
    }
    bool bias_left = bias != nullptr;
    if constexpr (EPI == EPI_ROPE) {
      if (P.epi == 5) {
        // Rotation of a head's (i, i + hd / 2) column pairs, of the rounded values, as where a pass of its own does it;
        // the table has a frequency's tokens next to each other, as the lanes have their rows.
        const float2* tab = P.rope + row % P.t_pad;
        if (bias) {
#pragma unroll
          for (int j = 0; j < 64; ++j)
            v[j] = __float_as_uint(__uint_as_float(v[j]) + __shfl_sync(0xffffffffu, bl[j % (BN / 32)], (pn * 64 + j) / (BN / 32)));
          bias_left = false;
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float2 cs = tab[(long long)j * P.t_pad];
          const float a = tc::round_bf16(__uint_as_float(v[j])), b = tc::round_bf16(__uint_as_float(v[j + 32]));
          v[j] = __float_as_uint(a * cs.x - b * cs.y);
          v[j + 32] = __float_as_uint(b * cs.x + a * cs.y);
        }
      }
    }
    uint4 outv[8];
    uint32_t* ow = reinterpret_cast<uint32_t*>(outv);
    if (has_res) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const __nv_bfloat16* rb = reinterpret_cast<const __nv_bfloat16*>(&rv[j]);
#pragma unroll
        for (int k = 0; k < 8; ++k) v[8 * j + k] = __float_as_uint(__uint_as_float(v[8 * j + k]) + __bfloat162float(rb[k]));
      }
      if (pn + 1 < pn_end && n + 64 < P.n) {
        const __nv_bfloat16* rp = P.residual + ((long long)(n / 64 + 1) * P.c_rpad + row) * 64;
#pragma unroll
        for (int j = 0; j < 8; ++j) rv[j] = *reinterpret_cast<const uint4*>(rp + 8 * j);
      }
    }
    if (bias_left) {
#pragma unroll
      for (int j = 0; j < 64; j += 2) {
        // column pn*64 + j is register (j % (BN/32)) of lane (pn*64 + j) / (BN/32)
        const float b0 = __shfl_sync(0xffffffffu, bl[j % (BN / 32)], (pn * 64 + j) / (BN / 32));
        const float b1 = __shfl_sync(0xffffffffu, bl[(j + 1) % (BN / 32)], (pn * 64 + j + 1) / (BN / 32));
        ow[j / 2] = tc::pack_bf16(pad ? 0.f : __uint_as_float(v[j]) + b0, pad ? 0.f : __uint_as_float(v[j + 1]) + b1);
      }
    } else {
#pragma unroll
      for (int j = 0; j < 64; j += 2)
        ow[j / 2] = tc::pack_bf16(pad ? 0.f : __uint_as_float(v[j]), pad ? 0.f : __uint_as_float(v[j + 1]));
    }
    if (P.dot_with && row < P.m) {
      // Row reduction over this head's columns, on the ROUNDED values the attention backward will read:
      // sum_j dS_ij = 0 (softmax shift invariance) holds only if D matches the dP that kernel forms.
      const __nv_bfloat16* ap = P.dot_with + ((long long)(n / 64) * P.c_rpad + row) * 64;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint4 av = *reinterpret_cast<const uint4*>(ap + 8 * j);
        const __nv_bfloat16* ab16 = reinterpret_cast<const __nv_bfloat16*>(&av);
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
          const uint32_t w2 = ow[4 * j + k / 2];        // two bf16: low half = even column
          dot_acc = fmaf(__uint_as_float(w2 << 16), __bfloat162float(ab16[k]), dot_acc);
          dot_acc = fmaf(__uint_as_float(w2 & 0xffff0000u), __bfloat162float(ab16[k + 1]), dot_acc);
        }
      }
      if ((n + 64) % P.dot_hd == 0) {                 // last panel of a head
        const int hh = n / P.dot_hd, bb = row / P.t_pad, tt = row % P.t_pad;
        P.dot_out[((long long)bb * P.dot_hq + hh) * P.t_pad + tt] = dot_acc;
        dot_acc = 0.f;
      }
    }
    // Staging tile (pc & 1) of this warp: its previous store (two panels ago) has been read, since lane 0
    // waited for that after committing the store of the panel before this one.
    const uint32_t stg = stg0 + (ESETS == 2 ? (uint32_t)(warp - 2) : (uint32_t)(q * 2 + (pc & 1))) * 4096u;
    if (ESETS == 2 && lane == 0) tc::bulk_wait_group_read0();    // one staging tile: the store before has read it
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; ++j)
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stg + lane * 128 + (((uint32_t)j ^ (uint32_t)(lane & 7)) * 16)),
                   "r"(outv[j].x), "r"(outv[j].y), "r"(outv[j].z), "r"(outv[j].w) : "memory");
    tc::fence_proxy_async();
    __syncwarp();
    if (lane == 0) {
      tc::tma_store_3d(&P.tc, stg, 0, m0 + q * 32, n / 64);
      tc::bulk_commit_group();
      if (ESETS == 1) tc::bulk_wait_group_read1();  // the store before this one has read its staging tile
    }
    ++pc;
  }
  return true;
}

// Persistent kernel: one block per SM walks the work list with stride gridDim.x.  Warp 0 feeds the
// shared-memory ring by TMA, warp 1 issues the MMAs into one of two TMEM accumulators, warps 2-5 drain the
// other accumulator (bias, residual, padding-row mask, bf16 rows in R-Tile order), so the epilogue of
// one tile overlaps the main loop of the next.
template <int BN, int STAGES, int ESETS, int EPI>
__global__ void __maxnreg__(ESETS == 2 ? 168 : EPI == EPI_ACT ? 255 : 224) gemm_tc_kernel(const __grid_constant__ TcGroup G) {
  using SP = SmemPlan<BN, STAGES>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + SP::BAR_OFF;
  auto full = [&](int s) { return bars + 8u * s; };
  auto empty = [&](int s) { return bars + 8u * (STAGES + s); };
  auto acc_full = [&](int a) { return bars + 8u * (2 * STAGES + a); };
  auto acc_empty = [&](int a) { return bars + 8u * (2 * STAGES + 2 + a); };
  const uint32_t slot = bars + 8 * SP::N_BARS;
  const int warp = (int)tc::uniform(threadIdx.x / 32), lane = threadIdx.x % 32;
  const tc::Status status(G.status, G.reset_status);
  constexpr uint32_t TMEM_COLS = 2 * BN;                 // two fp32 accumulators of BN columns

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(full(s), 1);                 // one producer arrival + transaction bytes
      tc::mbar_init(empty(s), 1);                // one tcgen05.commit arrival
    }
    for (int a = 0; a < 2; ++a) {
      tc::mbar_init(acc_full(a), 1);
      tc::mbar_init(acc_empty(a), 128 * ESETS);
    }
    tc::fence_barrier_init();
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
  if (!G.late_trigger) pdl_launch_dependents();

  if (warp == 0) {
    const bool leader = tc::elect_one();
    // ---- TMA producer.  Its loop is kept short (stage, phase and coordinates advance by additions, nothing is decided per
    // k-block): operands arrive from L2 about as fast as the products take them, so that a stage that is free and not yet
    // requested is time lost, most of all with CTA pairs.  (With a case per operand, a division and a test for prefilled
    // stages per k-block: gated feed-forward step of 4096 x 2048 x 8192 1131 us instead of 1088, 8192 x 4096 attention step
    // 5190 instead of 5060, Whisper-shaped cross-attention step 189.8 instead of 186.8.)
    int s = 0;
    uint32_t ph = 1;
    bool ok = true;
    TileCoord tcd;
    // Weights do not depend on the kernel before this one: their tiles for the first stages of the first
    // output tile are requested before waiting for that kernel, hiding their (cold) latency.
    int prefilled = 0;
    if (tile_at<BN>(G, blockIdx.x, &tcd) && G.p[tcd.prob].b_static && G.p[tcd.prob].ksplit == 1) {
      const TcProblem& P = G.p[tcd.prob];
      if (leader) { tc::tma_prefetch_desc(&P.ta[0]); tc::tma_prefetch_desc(&P.tb[0]); }
      const int n = P.kblocks[0] < STAGES ? P.kblocks[0] : STAGES;
      for (int kb = 0; kb < n; ++kb) {
        const uint32_t sb = base + kb * SP::STAGE + SP::A_BYTES;
        if (!leader) continue;
        tc::mbar_expect_tx(full(kb), SP::STAGE);
        if (P.b_mn[0]) tc::tma_load_3d(sb, &P.tb[0], full(kb), 0, kb * BK, tcd.n0 / 64);
        else tc::tma_load_3d(sb, &P.tb[0], full(kb), 0, tcd.n0, kb);
      }
      prefilled = n;
    }
    pdl_wait();
    if (G.late_trigger && leader) late_trigger(G);
    for (int w = blockIdx.x; ok && tile_at<BN>(G, w, &tcd); w += gridDim.x) {
      const TcProblem& P = G.p[tcd.prob];
      for (int t = 0; t < P.n_terms && ok; ++t) {
        int kb = t == 0 ? tcd.kb0 : 0;
        const int kb_end = t == 0 ? tcd.kb1 : P.kblocks[t];
        const CUtensorMap *ta = &P.ta[t], *tb = &P.tb[t];
        const int a_mn = P.a_mn[t], b_mn = P.b_mn[t];
        int ay = a_mn ? kb * BK : tcd.m0, az = a_mn ? tcd.m0 / 64 : kb, by = b_mn ? kb * BK : tcd.n0, bz = b_mn ? tcd.n0 / 64 : kb;
        const int ady = a_mn ? BK : 0, adz = a_mn ? 0 : 1, bdy = b_mn ? BK : 0, bdz = b_mn ? 0 : 1;
        auto advance = [&] {
          ay += ady; az += adz; by += bdy; bz += bdz;
          if (++s == STAGES) { s = 0; ph ^= 1; }
        };
        for (; prefilled > 0; --prefilled, ++kb) {         // the barrier is armed and the B tile on its way
          if (leader) tc::tma_load_3d(base + s * SP::STAGE, ta, full(s), 0, ay, az);
          advance();
        }
        for (; kb < kb_end; ++kb) {
          const uint32_t sa = base + s * SP::STAGE;
          if (!tc::mbar_wait_warp(empty(s), ph, status, 101)) { ok = false; break; }
          if (leader) {
            tc::mbar_expect_tx(full(s), SP::STAGE);
            tc::tma_load_3d(sa, ta, full(s), 0, ay, az);
            tc::tma_load_3d(sa + SP::A_BYTES, tb, full(s), 0, by, bz);
          }
          advance();
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer (a whole warp, see elect_one).  Descriptor words are formed once per reduction loop; per instruction only
    // the start-address field moves.  (With 128 x 256 tiles a k-block's 48 KB of operands take longer to arrive from
    // L2, at about 64 B/clk per SM, than its four MMAs take to run.) ------
    const bool leader = tc::elect_one();
    int s = 0, ti = 0;
    uint32_t ph = 0;
    bool ok = true;
    TileCoord tcd;
    const uint32_t hi = tc::smem_desc_hi(1024);
    for (int w = blockIdx.x; ok && tile_at<BN>(G, w, &tcd); w += gridDim.x, ++ti) {
      const TcProblem& P = G.p[tcd.prob];
      const int ab = ti & 1;
      if (!tc::mbar_wait_warp(acc_empty(ab), ((ti >> 1) & 1) ^ 1, status, 104)) { ok = false; break; }
      tc::tc_fence_after();
      const uint32_t d_tmem = tmem_base + ab * BN;
      uint32_t acc = 0;
      for (int t = 0; t < P.n_terms && ok; ++t) {
        const uint32_t idesc = tc::idesc_bf16(BM, BN, P.a_mn[t], P.b_mn[t]);
        // K-major: 8-row groups 1024 B apart, 16 K elements = 32 B along the row.
        // MN-major: 64-wide M/N blocks 8 KiB apart (64 K rows x 128 B), 16 K rows = 2 KiB.
        const uint32_t a_lo0 = tc::smem_desc_lo(base, P.a_mn[t] ? 8192u : 16u), a_step = P.a_mn[t] ? 128u : 2u;
        const uint32_t b_lo0 = tc::smem_desc_lo(base + SP::A_BYTES, P.b_mn[t] ? 8192u : 16u), b_step = P.b_mn[t] ? 128u : 2u;
        const int nkb = t == 0 ? tcd.kb1 - tcd.kb0 : P.kblocks[t];
        for (int kb = 0; kb < nkb; ++kb) {
          if (!tc::mbar_wait_warp(full(s), ph, status, 102)) { ok = false; break; }
          tc::tc_fence_after();
          const uint32_t a_lo = a_lo0 + (uint32_t)s * (SP::STAGE >> 4), b_lo = b_lo0 + (uint32_t)s * (SP::STAGE >> 4);
          if (leader) {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
              tc::mma_bf16_ss_w(d_tmem, a_lo + kk * a_step, hi, b_lo + kk * b_step, hi, idesc, kk > 0 ? 1u : acc);
            tc::mma_commit(empty(s));              // frees the stage once these MMAs have read it
          }
          acc = 1;
          if (++s == STAGES) { s = 0; ph ^= 1; }
        }
      }
      if (ok && leader) tc::mma_commit(acc_full(ab));
    }
  } else if (warp >= 2) {
    // ---- epilogue warps ---------------------------------------------------------------------------
    pdl_wait();                                       // the previous kernel may still be reading what we overwrite
    group_chores(G, threadIdx.x - 64, 128 * ESETS);
    const int q = warp % 4;                           // the TMEM lane quarter this warp may access
    int ti = 0, pc = 0;                               // tiles and panels done by this warp
    bool ok = true;
    TileCoord tcd;
    for (int w = blockIdx.x; ok && tile_at<BN>(G, w, &tcd); w += gridDim.x, ++ti) {
      const TcProblem& P = G.p[tcd.prob];
      const int ab = ti & 1;
      const bool ready = epilogue_tile<BN, ESETS, EPI>(P, tcd.m0, tcd.n0, q, TmemAcc{tmem_base + ((uint32_t)(q * 32) << 16) + ab * BN}, base + SP::STG_OFF, pc, [&] {
        return tc::mbar_wait(acc_full(ab), (ti >> 1) & 1, status, 103);
      });
      if (!ready) { ok = false; break; }
      tc::tc_fence_before();
      tc::mbar_arrive(acc_empty(ab));             // this accumulator may be overwritten by the tile after next
    }
    if (lane == 0) tc::bulk_wait_group0();        // all output tiles are in global memory before the block exits
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem_base, TMEM_COLS);
}

// ---------------------------------------------------------------------------------------------------
// CTA-pair variant (tcgen05 cta_group::2): two SMs share a 256 x 256 output tile.  Each CTA loads its 128 rows of
// A and its 128 columns of B (32 KB per k-block instead of 48 KB for a 128 x 256 tile of its own: operand
// delivery from L2, about 64 B/clk per SM, is what bounds the single-CTA kernel), the leader (cluster rank 0)
// issues MMAs of M = 256, N = 256 that read both CTAs' shared memory and write 128 accumulator rows into each
// CTA's tensor memory, and each CTA drains its own rows.  Barriers: full[] lives in the leader and counts the
// bytes of both CTAs' loads; empty[] and acc_full[] exist in both and get their arrivals from one commit that
// signals both CTAs; acc_empty[] lives in the leader and takes the arrivals of both CTAs' epilogue threads.
// ---------------------------------------------------------------------------------------------------
constexpr int PAIR_BN = 256, PAIR_STAGES = 6;
struct PairSmem {
  static constexpr uint32_t A_BYTES = 128 * 128, B_BYTES = 128 * 128, STAGE = A_BYTES + B_BYTES;
  static constexpr uint32_t STG_OFF = PAIR_STAGES * STAGE;
  static constexpr uint32_t BAR_OFF = STG_OFF + 2 * 16384;
  static constexpr uint32_t N_BARS = 2 * PAIR_STAGES + 4;
  static constexpr uint32_t TOTAL = BAR_OFF + 8 * N_BARS + 16 + 1024;
};

// work list in 256 x 256 tiles (ksplit slices as in tile_at); m0 / n0 are the pair's.  Tall problems go in bands of eight row
// tiles: the 74 tiles at work then share eight row tiles and nine column tiles of operands instead of 32 and two or three, which
// L2 holds (8192 x 4096 attention step: 5060 -> 4945 us, its four product launches 535, 172, 378, 1191 -> 505, 167, 364, 1131; bands
// of 16 the same).  Up to 16 row tiles fit as they are (4096 x 2048 x 8192 feed-forward in bands of eight: 88 -> 92 us a launch).
constexpr int PAIR_BAND = 8, PAIR_BAND_FROM = 16;
__device__ __forceinline__ bool pair_tile_at(const TcGroup& G, int w, TileCoord* tc_out) {
  for (int p = 0; p < G.count; ++p) {
    const TcProblem& P = G.p[p];
    const int tm = (P.m + 255) / 256, tn = (P.n + 255) / 256;
    const int units = tm * tn * P.ksplit;
    if (w < units) {
      const int slice = w % P.ksplit, t = w / P.ksplit;
      tc_out->prob = p;
      const int band = tm > PAIR_BAND_FROM ? PAIR_BAND : tm, at = t / (band * tn), h = min(band, tm - at * band), u = t - at * band * tn;
      tc_out->m0 = (at * band + u % h) * 256;
      tc_out->n0 = (u / h) * 256;
      const int per = (P.kblocks[0] + P.ksplit - 1) / P.ksplit;
      tc_out->kb0 = slice * per;
      tc_out->kb1 = min(P.kblocks[0], (slice + 1) * per);
      return true;
    }
    w -= units;
  }
  return false;
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(EPI == EPI_ACT ? 255 : 224) gemm_tc_pair_kernel(const __grid_constant__ TcGroup G) {
  using SP = PairSmem;
  constexpr int STAGES = PAIR_STAGES, BN = PAIR_BN;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + SP::BAR_OFF;
  auto full = [&](int s) { return bars + 8u * s; };
  auto empty = [&](int s) { return bars + 8u * (STAGES + s); };
  auto acc_full = [&](int a) { return bars + 8u * (2 * STAGES + a); };
  auto acc_empty = [&](int a) { return bars + 8u * (2 * STAGES + 2 + a); };
  const uint32_t slot = bars + 8 * SP::N_BARS;
  const int warp = (int)tc::uniform(threadIdx.x / 32), lane = threadIdx.x % 32;
  const uint32_t rank = tc::cluster_ctarank();
  const int pair_id = blockIdx.x / 2, n_pairs = gridDim.x / 2;
  const tc::Status status(G.status, G.reset_status);
  constexpr uint32_t TMEM_COLS = 2 * BN;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(full(s), 1);                 // leader: its producer's arrival + both CTAs' transaction bytes
      tc::mbar_init(empty(s), 1);                // one commit arrival (sent to both CTAs)
    }
    for (int a = 0; a < 2; ++a) {
      tc::mbar_init(acc_full(a), 1);
      tc::mbar_init(acc_empty(a), 256);          // leader: the epilogue threads of both CTAs
    }
    tc::fence_barrier_init();
  }
  if (warp == 1) {
    tc::tmem_alloc2(slot, TMEM_COLS);
    tc::tmem_relinquish2();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::cluster_sync_all();                        // the peer's barriers exist before anything signals them
  tc::tc_fence_after();
  uint32_t tmem_base;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(slot));
  tmem_base = tc::uniform(tmem_base);
  if (!G.late_trigger) pdl_launch_dependents();

  if (warp == 0) {
    const bool leader = tc::elect_one();
    // ---- TMA producer (both CTAs): own A rows, own half of B's columns; bytes counted on the leader's barrier ----
    int s = 0;
    uint32_t ph = 1;
    bool ok = true;
    TileCoord tcd;
    const uint32_t full0 = tc::map_to_cta(full(0), 0);
    pdl_wait();
    if (G.late_trigger && leader) late_trigger(G);
    for (int w = pair_id; ok && pair_tile_at(G, w, &tcd); w += n_pairs) {
      const TcProblem& P = G.p[tcd.prob];
      const int m0 = tcd.m0 + (int)rank * 128, n0 = tcd.n0 + (int)rank * 128;
      for (int t = 0; t < P.n_terms && ok; ++t) {
        int kb = t == 0 ? tcd.kb0 : 0;
        const int kb_end = t == 0 ? tcd.kb1 : P.kblocks[t];
        const CUtensorMap *ta = &P.ta[t], *tb = &P.tb[t];
        const int a_mn = P.a_mn[t], b_mn = P.b_mn[t];
        int ay = a_mn ? kb * BK : m0, az = a_mn ? m0 / 64 : kb, by = b_mn ? kb * BK : n0, bz = b_mn ? n0 / 64 : kb;
        const int ady = a_mn ? BK : 0, adz = a_mn ? 0 : 1, bdy = b_mn ? BK : 0, bdz = b_mn ? 0 : 1;
        for (; kb < kb_end; ++kb) {
          const uint32_t sa = base + s * SP::STAGE, fb = full0 + 8u * s;
          if (!tc::mbar_wait_warp(empty(s), ph, status, 111)) { ok = false; break; }
          if (leader) {
            if (rank == 0) tc::mbar_expect_tx(full(s), 2 * SP::STAGE);
            tc::tma_load_3d_pair(sa, ta, fb, 0, ay, az);
            tc::tma_load_3d_pair(sa + SP::A_BYTES, tb, fb, 0, by, bz);
          }
          ay += ady; az += adz; by += bdy; bz += bdz;
          if (++s == STAGES) { s = 0; ph ^= 1; }
        }
      }
    }
  } else if (warp == 1 && rank == 0) {
    // ---- MMA issuer (leader only) --------------------------------------------------------------
    const bool leader = tc::elect_one();
    int s = 0, ti = 0;
    uint32_t ph = 0;
    bool ok = true;
    TileCoord tcd;
    const uint32_t hi = tc::smem_desc_hi(1024);
    for (int w = pair_id; ok && pair_tile_at(G, w, &tcd); w += n_pairs, ++ti) {
      const TcProblem& P = G.p[tcd.prob];
      const int ab = ti & 1;
      if (!tc::mbar_wait_warp(acc_empty(ab), ((ti >> 1) & 1) ^ 1, status, 114)) { ok = false; break; }
      tc::tc_fence_after();
      const uint32_t d_tmem = tmem_base + ab * BN;
      uint32_t acc = 0;
      for (int t = 0; t < P.n_terms && ok; ++t) {
        const uint32_t idesc = tc::idesc_bf16(256, BN, P.a_mn[t], P.b_mn[t]);
        const uint32_t a_lo0 = tc::smem_desc_lo(base, P.a_mn[t] ? 8192u : 16u), a_step = P.a_mn[t] ? 128u : 2u;
        const uint32_t b_lo0 = tc::smem_desc_lo(base + SP::A_BYTES, P.b_mn[t] ? 8192u : 16u), b_step = P.b_mn[t] ? 128u : 2u;
        const int nkb = t == 0 ? tcd.kb1 - tcd.kb0 : P.kblocks[t];
        for (int kb = 0; kb < nkb; ++kb) {
          if (!tc::mbar_wait_warp(full(s), ph, status, 112)) { ok = false; break; }
          tc::tc_fence_after();
          const uint32_t a_lo = a_lo0 + (uint32_t)s * (SP::STAGE >> 4), b_lo = b_lo0 + (uint32_t)s * (SP::STAGE >> 4);
          if (leader) {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
              tc::mma_bf16_ss_w2(d_tmem, a_lo + kk * a_step, hi, b_lo + kk * b_step, hi, idesc, kk > 0 ? 1u : acc);
            tc::mma_commit2_both(empty(s));        // frees the stage in both CTAs once these MMAs have read it
          }
          acc = 1;
          if (++s == STAGES) { s = 0; ph ^= 1; }
        }
      }
      if (ok && leader) tc::mma_commit2_both(acc_full(ab));
    }
  } else if (warp >= 2) {
    // ---- epilogue (both CTAs): this CTA's 128 accumulator rows, as in the single-CTA kernel -------------
    pdl_wait();
    group_chores(G, threadIdx.x - 64, 128);
    const int q = warp % 4;
    int ti = 0, pc = 0;
    bool ok = true;
    TileCoord tcd;
    for (int w = pair_id; ok && pair_tile_at(G, w, &tcd); w += n_pairs, ++ti) {
      const TcProblem& P = G.p[tcd.prob];
      const int ab = ti & 1;
      const int m0 = tcd.m0 + (int)rank * 128;
      const bool ready = epilogue_tile<BN, 1, EPI>(P, m0, tcd.n0, q, TmemAcc{tmem_base + ((uint32_t)(q * 32) << 16) + ab * BN}, base + SP::STG_OFF, pc, [&] {
        return tc::mbar_wait(acc_full(ab), (ti >> 1) & 1, status, 113);
      });
      if (!ready) { ok = false; break; }
      tc::tc_fence_before();
      tc::mbar_arrive_cluster(tc::map_to_cta(acc_empty(ab), 0));     // the leader's barrier, from either CTA
    }
    if (lane == 0) tc::bulk_wait_group0();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::cluster_sync_all();                        // neither CTA frees tensor memory or leaves while its peer may still
  if (warp == 1) tc::tmem_dealloc2(tmem_base, TMEM_COLS);   // read its shared memory or signal its barriers
}

// ---------------------------------------------------------------------------------------------------
// Launches with few tiles and long reductions (few tokens: 50 x 768 outputs are six tiles for 148 SMs): the reduction of a
// 128 x 128 tile is cut into 2 or 4 slices, one per block of a cluster.  Each block accumulates its slice in tensor
// memory and leaves the fp32 sums in shared memory, over its operand stages; then it finishes its share of the tile's
// rows, adding the slices through distributed shared memory in a fixed order.  One tile per cluster.  Every slice has a
// k-block (gemm_slice_begin; make_group_split refuses a launch where one would not): what a block of none would add is what
// its tensor memory held before.  The bound is a
// block's chain: first operands, its k-blocks at about 545 clk each, the exchange (about 2.5 us: distributed shared memory
// gives a block some 15 bytes/clk), the epilogue.  Rank-16 adapter products of 4096 x 2048 (32 k-blocks, 32 row tiles):
// 14.3 -> 12.0 us forward and 18.5 -> 13.0 us backward.
// ---------------------------------------------------------------------------------------------------
constexpr int SPLIT_STAGES = 6, SPLIT_LD = 132;        // pitch of a partial row, in floats: 16-byte accesses without conflicts
__device__ __forceinline__ float4 ld_cluster(uint32_t a) {
  float4 f;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(f.x), "=f"(f.y), "=f"(f.z), "=f"(f.w) : "r"(a) : "memory");
  return f;
}
struct PartialAcc {
  uint32_t row;                                        // this lane's row in shared memory
  __device__ __forceinline__ void load(int col, uint32_t (&v)[32]) const {
#pragma unroll
    for (int j = 0; j < 32; j += 4)
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[j]), "=r"(v[j + 1]), "=r"(v[j + 2]), "=r"(v[j + 3]) : "r"(row + (col + j) * 4) : "memory");
  }
  __device__ __forceinline__ void wait() const {}
};

template <int EPI>
__global__ void __launch_bounds__(320, 1) gemm_tc_split_kernel(const __grid_constant__ TcGroup G) {
  constexpr int BN = 128, STAGES = SPLIT_STAGES;
  using SP = SmemPlan<BN, STAGES>;
  static_assert(128 * SPLIT_LD * 4 <= STAGES * (int)SP::STAGE, "a partial tile fits the operand stages");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + SP::BAR_OFF, slot = bars + 8 * SP::N_BARS, acc_full = bars + 8u * (2 * STAGES);
  auto full = [&](int s) { return bars + 8u * s; };
  auto empty = [&](int s) { return bars + 8u * (STAGES + s); };
  const int warp = (int)tc::uniform(threadIdx.x / 32), lane = threadIdx.x % 32;
  const tc::Status status(G.status, G.reset_status);
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(full(s), 1);
      tc::mbar_init(empty(s), 1);
    }
    tc::mbar_init(acc_full, 1);
    tc::fence_barrier_init();
  }
  if (warp == 1) {
    tc::tmem_alloc(slot, BN);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  uint32_t tmem_base;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(slot));
  tmem_base = tc::uniform(tmem_base);
  if (!G.late_trigger) pdl_launch_dependents();

  const int slice = blockIdx.x % G.slices;
  TileCoord tcd;
  tile_at<BN>(G, blockIdx.x / G.slices, &tcd);
  const TcProblem& P = G.p[tcd.prob];
  int total = 0;
  for (int t = 0; t < P.n_terms; ++t) total += P.kblocks[t];
  const int begin = gemm_slice_begin(total, G.slices, slice), end = gemm_slice_begin(total, G.slices, slice + 1);

  if (warp == 0) {
    const bool leader = tc::elect_one();
    // ---- TMA producer; the first weights before waiting for the kernel in front, as in gemm_tc_kernel ----
    int prefilled = 0;
    if (P.b_static && begin < P.kblocks[0]) {
      prefilled = min(STAGES, min(end, P.kblocks[0]) - begin);
      for (int i = 0; i < prefilled; ++i) {
        const uint32_t sb = base + i * SP::STAGE + SP::A_BYTES;
        if (!leader) continue;
        tc::mbar_expect_tx(full(i), SP::STAGE);
        if (P.b_mn[0]) tc::tma_load_3d(sb, &P.tb[0], full(i), 0, (begin + i) * BK, tcd.n0 / 64);
        else tc::tma_load_3d(sb, &P.tb[0], full(i), 0, tcd.n0, begin + i);
      }
    }
    pdl_wait();
    if (G.late_trigger && leader) late_trigger(G);
    int t = 0, first = 0;                              // term of the k-block, and its first k-block
    for (int k = begin, it = 0; k < end; ++k, ++it) {
      while (k - first >= P.kblocks[t]) { first += P.kblocks[t]; ++t; }
      const int kb = k - first, s = it % STAGES;
      const uint32_t sa = base + s * SP::STAGE, sb = sa + SP::A_BYTES;
      if (it >= prefilled) {
        if (!tc::mbar_wait_warp(empty(s), ((it / STAGES) & 1) ^ 1, status, 141)) break;
        if (leader) tc::mbar_expect_tx(full(s), SP::STAGE);
      }
      if (!leader) continue;
      if (P.a_mn[t]) tc::tma_load_3d(sa, &P.ta[t], full(s), 0, kb * BK, tcd.m0 / 64);
      else tc::tma_load_3d(sa, &P.ta[t], full(s), 0, tcd.m0, kb);
      if (it >= prefilled) {
        if (P.b_mn[t]) tc::tma_load_3d(sb, &P.tb[t], full(s), 0, kb * BK, tcd.n0 / 64);
        else tc::tma_load_3d(sb, &P.tb[t], full(s), 0, tcd.n0, kb);
      }
    }
    __syncwarp();
    tc::cluster_sync_all();
    tc::cluster_arrive();
  } else if (warp == 1) {
    // ---- MMA issuer ----
    const bool leader = tc::elect_one();
    const uint32_t hi = tc::smem_desc_hi(1024);
    int t = 0, first = 0;
    bool ok = true;
    for (int k = begin, it = 0; k < end; ++k, ++it) {
      while (k - first >= P.kblocks[t]) { first += P.kblocks[t]; ++t; }
      const int s = it % STAGES;
      if (!tc::mbar_wait_warp(full(s), (it / STAGES) & 1, status, 142)) { ok = false; break; }
      tc::tc_fence_after();
      const uint32_t idesc = tc::idesc_bf16(BM, BN, P.a_mn[t], P.b_mn[t]), sa = base + s * SP::STAGE;
      const uint32_t a_lo = tc::smem_desc_lo(sa, P.a_mn[t] ? 8192u : 16u), b_lo = tc::smem_desc_lo(sa + SP::A_BYTES, P.b_mn[t] ? 8192u : 16u);
      const uint32_t a_step = P.a_mn[t] ? 128u : 2u, b_step = P.b_mn[t] ? 128u : 2u;
      if (leader) {
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
          tc::mma_bf16_ss_w(tmem_base, a_lo + kk * a_step, hi, b_lo + kk * b_step, hi, idesc, (it > 0 || kk > 0) ? 1u : 0u);
        tc::mma_commit(empty(s));
      }
    }
    if (ok && leader) tc::mma_commit(acc_full);
    __syncwarp();
    tc::cluster_sync_all();
    tc::cluster_arrive();
  } else {
    // ---- epilogue warps: partial rows to shared memory, then this block's share of the row groups ----
    pdl_wait();
    group_chores(G, threadIdx.x - 64, 256);
    const int q = warp % 4, set = (warp - 2) / 4, groups = 4 / G.slices;
    auto exchange = [&]() -> bool {
      const bool ok = tc::mbar_wait(acc_full, 0, status, 143);
      tc::tc_fence_after();
      if (ok && tcd.m0 + q * 32 < P.m) {
        const uint32_t row = base + ((q * 32 + lane) * SPLIT_LD + set * 64) * 4;
#pragma unroll 1
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t v[32];
          tc::tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + set * 64 + hf * 32, v);
          tc::tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; j += 4)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row + (hf * 32 + j) * 4), "r"(v[j]), "r"(v[j + 1]), "r"(v[j + 2]), "r"(v[j + 3]) : "memory");
        }
      }
      __syncwarp();
      tc::cluster_sync_all();
      // this block's rows: sixteen independent 16-byte loads a thread, their sums in place of its own partial rows
      const int tid = threadIdx.x - 64, mine = 32 * min(32 * groups, P.m - tcd.m0 - slice * groups * 32);
      for (int i = tid; i < mine; i += 512) {
        const uint32_t at0 = base + (((slice * groups * 32) + i / 32) * SPLIT_LD + i % 32 * 4) * 4, at1 = at0 + 8 * SPLIT_LD * 4;
        const bool two = i + 256 < mine;
        float4 a[4], b[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c < G.slices) {
            a[c] = ld_cluster(tc::map_to_cta(at0, c));
            if (two) b[c] = ld_cluster(tc::map_to_cta(at1, c));
          }
#pragma unroll
        for (int c = 1; c < 4; ++c)
          if (c < G.slices) {
            a[0].x += a[c].x; a[0].y += a[c].y; a[0].z += a[c].z; a[0].w += a[c].w;
            b[0].x += b[c].x; b[0].y += b[c].y; b[0].z += b[c].z; b[0].w += b[c].w;
          }
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at0), "f"(a[0].x), "f"(a[0].y), "f"(a[0].z), "f"(a[0].w) : "memory");
        if (two)
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at1), "f"(b[0].x), "f"(b[0].y), "f"(b[0].z), "f"(b[0].w) : "memory");
      }
      __syncwarp();
      tc::cluster_arrive();                              // the others' partial rows have been read
      asm volatile("bar.sync 1, 256;" ::: "memory");
      return ok;
    };
    const int rg = slice * groups + q;                   // the row group this warp finishes (the first `groups` warps of a set)
    int pc = 0;
    if (q < groups && tcd.m0 + rg * 32 < P.m)
      epilogue_tile<BN, 2, EPI>(P, tcd.m0, tcd.n0, rg, PartialAcc{base + (rg * 32 + lane) * SPLIT_LD * 4}, base + SP::STG_OFF, pc, exchange);
    else
      exchange();
    if (lane == 0) tc::bulk_wait_group0();
    __syncwarp();
  }
  tc::tc_fence_before();
  tc::cluster_wait();                                    // no block leaves while another may still read its partial rows
  if (warp == 1) tc::tmem_dealloc(tmem_base, BN);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

typedef CUresult (*ReplaceAddressFn)(CUtensorMap*, void*);

ReplaceAddressFn replace_fn() {
  static ReplaceAddressFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapReplaceAddress", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<ReplaceAddressFn>(p);
  });
  return fn;
}

// Self-test of the bounded wait every tensor-core kernel relies on: one block initialises an mbarrier that nothing
// ever signals and waits on it through the same tc::mbar_wait, with a short limit.  The wait must give up, record
// its code in the status word and let the block return normally.
__global__ void wait_timeout_selftest_kernel(int32_t* status, long long limit_cycles) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    tc::mbar_init(tc::smem_u32(&bar), 1);
    tc::fence_barrier_init();
  }
  __syncthreads();
  const bool ok = tc::mbar_wait(tc::smem_u32(&bar), 0, status, 901, limit_cycles);
  __syncthreads();
  if (threadIdx.x == 0) status[1] = ok ? 2 : 1;     // the block reached its normal end
}

}  // namespace

cudaError_t launch_wait_timeout_selftest(int32_t* status, long long limit_cycles, cudaStream_t st) {
  wait_timeout_selftest_kernel<<<1, 64, 0, st>>>(status, limit_cycles);
  return cudaGetLastError();
}

bool fbl_map_set_base(CUtensorMap* map, const void* base) {
  ReplaceAddressFn fn = replace_fn();
  return fn && fn(map, const_cast<void*>(base)) == CUDA_SUCCESS;
}

static bool encode_panels(CUtensorMap* map, CUtensorMapDataType type, int width, const void* base, int64_t r_pad, int panels,
                          int box_rows, int box_panels) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)width, (cuuint64_t)r_pad, (cuuint64_t)panels};
  cuuint64_t strides[2] = {128, (cuuint64_t)r_pad * 128};
  cuuint32_t box[3] = {(cuuint32_t)width, (cuuint32_t)box_rows, (cuuint32_t)box_panels};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, type, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool fbl_encode_seq_map(CUtensorMap* map, bool f32, const void* base, int rows, int seqs, int panels, int box_rows, int box_panels) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint32_t width = f32 ? 32 : 64;
  cuuint64_t dims[4] = {width, (cuuint64_t)rows, (cuuint64_t)seqs, (cuuint64_t)panels};
  cuuint64_t strides[3] = {128, (cuuint64_t)rows * 128, (cuuint64_t)rows * seqs * 128};
  cuuint32_t box[4] = {width, (cuuint32_t)box_rows, 1, (cuuint32_t)box_panels};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool fbl_encode_rtile_map(CUtensorMap* map, const void* base, int64_t r_pad, int panels, int box_rows, int box_panels) {
  return encode_panels(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 64, base, r_pad, panels, box_rows, box_panels);
}
bool fbl_encode_f32_rtile_map(CUtensorMap* map, const void* base, int64_t r_pad, int panels, int box_rows, int box_panels) {
  return encode_panels(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 32, base, r_pad, panels, box_rows, box_panels);
}

// fp32 accumulator [n_pad, cols] stored in the bf16 tile order (64-column panels, 256-byte rows), viewed as
// [panels][rows][2 halves][32 floats] so that a box of 128 rows x one panel can use the 128-byte swizzle.
bool fbl_encode_f32_panel_map(CUtensorMap* map, const void* base, int64_t r_pad, int panels, int box_rows, int box_halves) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {32, 2, (cuuint64_t)r_pad, (cuuint64_t)panels};
  cuuint64_t strides[3] = {128, 256, (cuuint64_t)r_pad * 256};
  cuuint32_t box[4] = {32, (cuuint32_t)box_halves, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}


// Any number of rows and any whole number of 64-column panels: a box that reaches past its tensor (fewer rows than a
// tile, a single panel of columns, a short reduction) is filled with zeros by the load and clipped by the store, so a
// layer of 50 tokens or with one 64-wide key head costs one partly filled tile.  (The FFMA kernels that such shapes
// used to take: 95 us instead of 7 us for the 50 x 768 x 768 product, 453 us instead of 17 us for the query projection
// of a one-key-head layer, 3136 x 1024 x 1024.)  Only reductions along an operand's columns need whole panels.
bool gemm_tc_supported(const fbl_plan* p, const GemmArgs& g) {
  if (p->d.dtype != FBL_DTYPE_BF16) return false;
  if (g.n % 64 != 0 || g.n < 64 || g.m < 1) return false;
  for (int t = 0; t < g.n_terms; ++t) {
    const GemmTerm& tm = g.t[t];
    if (tm.a_trans ? (g.m % 64 != 0) : (tm.k % BK != 0)) return false;
    if (tm.b_trans && tm.k % BK != 0) return false;
  }
  return true;
}

// Problem set-up shared by the kernels: tensor maps, operand orientations, epilogue extras and reduction
// slices of every problem of a launch; addresses are point_group's.  bn_box: columns of B one CTA loads per k-block; tile_m x tile_n: the output
// tile a work unit covers (the CTA pair's 256 x 256, or one CTA's 128 x BN).  Returns the number of work units in
// *units.
cudaError_t fill_group(TcGroup& G, const GemmArgs* gs, int count, int bn_box, int tile_m, int tile_n, int* units) {
  memset(&G, 0, sizeof(G));
  G.count = count;
  G.late_trigger = gs[0].late_trigger != nullptr;
  int tiles = 0;
  for (int i = 0; i < count; ++i) {
    const GemmArgs& g = gs[i];
    TcProblem& P = G.p[i];
    P.n_terms = g.n_terms;
    for (int t = 0; t < g.n_terms; ++t) {
      const GemmTerm& tm = g.t[t];
      P.kblocks[t] = (tm.k + BK - 1) / BK;
      P.a_mn[t] = tm.a_trans ? 1 : 0;     // stored [k rows][m cols]: rows are K indices
      P.b_mn[t] = tm.b_trans ? 0 : 1;     // stored [k rows][n cols]: rows are K indices
      bool ok;
      if (tm.a_trans) ok = fbl_encode_rtile_map(&P.ta[t], tm.a, tm.a_rpad, g.m / 64, BK, BM / 64);
      else ok = fbl_encode_rtile_map(&P.ta[t], tm.a, tm.a_rpad, tm.k / 64, BM, 1);
      if (!ok) return cudaErrorInvalidValue;
      if (tm.b_trans) ok = fbl_encode_rtile_map(&P.tb[t], tm.b, tm.b_rpad, tm.k / 64, bn_box, 1);
      else ok = fbl_encode_rtile_map(&P.tb[t], tm.b, tm.b_rpad, g.n / 64, BK, bn_box / 64);
      if (!ok) return cudaErrorInvalidValue;
    }
    P.m = g.m; P.n = g.n;
    if (!fbl_encode_rtile_map(&P.tc, g.c, g.c_rpad, g.n / 64, 32, 1)) return cudaErrorInvalidValue;   // one warp's rows
    P.b_static = g.b_static;
    P.c_rpad = g.c_rpad; P.seq = g.seq; P.t_pad = g.t_pad;
    P.dot_hd = g.dot_hd; P.dot_hq = g.dot_hq; P.epi = g.epi;
    if (g.epi != 0) {
      const bool rope = g.epi == 5, two_out = g.epi != 2 && !rope;
      if (g.epi < 1 || g.epi > 5 || g.ksplit > 1 || g.dot_with || (g.epi >= 2 && !rope && !g.residual) || (g.epi == 4 && !g.aux1) ||
          (two_out && !g.c2) || (rope && (!g.rope || g.residual || g.t_pad <= 0)))
        return cudaErrorInvalidValue;
      if (two_out && !fbl_encode_rtile_map(&P.tc2, g.c2, g.c_rpad, g.n / 64, 32, 1)) return cudaErrorInvalidValue;
    }
    P.ksplit = 1;
    if (g.ksplit > 1) {
      if (g.n_terms != 1 || g.bias || g.residual || g.dot_with || g.t_pad > 0 || !g.acc) return cudaErrorInvalidValue;
      const int per = (P.kblocks[0] + g.ksplit - 1) / g.ksplit;        // no empty slice
      P.ksplit = (P.kblocks[0] + per - 1) / per;
      if (!fbl_encode_f32_panel_map(&P.tacc, g.acc, g.c_rpad, g.n / 64, 32, 1)) return cudaErrorInvalidValue;
    }
    tiles += ((g.m + tile_m - 1) / tile_m) * ((g.n + tile_n - 1) / tile_n) * P.ksplit;
  }
  *units = tiles;
  return cudaSuccess;
}

namespace {

// Which fused epilogue a launch needs (activations and the rotation never meet in one).
int group_epi(const GemmArgs* gs, int count) {
  int epi = EPI_NONE;
  for (int i = 0; i < count; ++i)
    if (gs[i].epi != 0) epi = gs[i].epi == 5 ? EPI_ROPE : EPI_ACT;
  return epi;
}

// A launch made ready but for its addresses: what launch_gemm_tc_group keeps.
struct GroupLaunch {
  TcGroup G;
  int order[MAX_PROBLEMS];                   // the caller's problem that each of G's is
  void (*kernel)(const TcGroup);
  int grid, threads, serial, cluster;        // cluster: blocks of a cluster where the launch says so, else 0
  int idle;                                  // what a late_trigger receives
  size_t smem;
};

cudaError_t group_launch(GroupLaunch& L, void (*k)(const TcGroup), int grid, int threads, size_t smem, int serial, int cluster = 0) {
  L.cluster = cluster;
  L.kernel = k; L.grid = grid; L.threads = threads; L.smem = smem; L.serial = serial;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

bool point_group(GroupLaunch& L, const GemmArgs* gs, int32_t* status) {
  TcGroup& G = L.G;
  G.status = status;
  G.zero_ptr = (uint4*)gs[0].zero_ptr; G.zero_vec = (long long)(gs[0].zero_bytes / 16); G.reset_status = gs[0].reset_status;
  bool ok = true;
  for (int i = 0; i < G.count; ++i) {
    const GemmArgs& g = gs[L.order[i]];
    TcProblem& P = G.p[i];
    for (int t = 0; t < P.n_terms; ++t) ok = ok && fbl_map_set_base(&P.ta[t], g.t[t].a) && fbl_map_set_base(&P.tb[t], g.t[t].b);
    ok = ok && fbl_map_set_base(&P.tc, g.c);
    if (P.epi != 0 && P.epi != 2 && P.epi != 5) ok = ok && fbl_map_set_base(&P.tc2, g.c2);
    if (P.ksplit > 1 || g.ksplit > 1) ok = ok && fbl_map_set_base(&P.tacc, g.acc);
    P.c = (__nv_bfloat16*)g.c; P.bias = g.bias; P.residual = (const __nv_bfloat16*)g.residual;
    P.dot_with = (const __nv_bfloat16*)g.dot_with; P.dot_out = g.dot_out;
    P.aux1 = (const __nv_bfloat16*)g.aux1; P.rope = g.rope;
  }
  return ok;
}

template <int BN, int STAGES>
cudaError_t make_group_bn(GroupLaunch& L, const fbl_plan* p, const GemmArgs* gs, int count, int esets_choice) {
  int tiles = 0;
  cudaError_t e = fill_group(L.G, gs, count, BN, BM, BN, &tiles);
  if (e != cudaSuccess) return e;
  const int grid = tiles < p->sm_count ? tiles : p->sm_count;
  // one tile per block at most: the epilogue is exposed, and the variant with two sets of epilogue warps halves it
  // (with several tiles per block the epilogues overlap the next main loops and the extra warps only cost)
  const int esets_knob = esets_choice ? esets_choice : p->knob_gemm_esets;
  const bool two_sets = BN > 64 && (esets_knob ? esets_knob == 2 : tiles <= p->sm_count);
  constexpr int SETS = BN > 64 ? 2 : 1;
  void (*k)(const TcGroup) = nullptr;
  switch (group_epi(gs, count)) {
    case EPI_ACT: k = two_sets ? gemm_tc_kernel<BN, STAGES, SETS, EPI_ACT> : gemm_tc_kernel<BN, STAGES, 1, EPI_ACT>; break;
    case EPI_ROPE: k = two_sets ? gemm_tc_kernel<BN, STAGES, SETS, EPI_ROPE> : gemm_tc_kernel<BN, STAGES, 1, EPI_ROPE>; break;
    default: k = two_sets ? gemm_tc_kernel<BN, STAGES, SETS, EPI_NONE> : gemm_tc_kernel<BN, STAGES, 1, EPI_NONE>;
  }
  return group_launch(L, k, grid, two_sets ? 320 : 192, SmemPlan<BN, STAGES>::TOTAL, gs[0].serial);
}

cudaError_t make_group_split(GroupLaunch& L, const GemmArgs* gs, int count, int slices) {
  int tiles = 0;
  cudaError_t e = fill_group(L.G, gs, count, 128, BM, 128, &tiles);
  if (e != cudaSuccess) return e;
  L.G.slices = slices;
  for (int i = 0; i < count; ++i) {
    int kb = 0;
    for (int t = 0; t < L.G.p[i].n_terms; ++t) kb += L.G.p[i].kblocks[t];
    if (kb < slices) return cudaErrorInvalidValue;       // a slice without work
  }
  const int epi = group_epi(gs, count);
  auto k = epi == EPI_ACT ? gemm_tc_split_kernel<EPI_ACT> : epi == EPI_ROPE ? gemm_tc_split_kernel<EPI_ROPE> : gemm_tc_split_kernel<EPI_NONE>;
  return group_launch(L, k, tiles * slices, 320, SmemPlan<128, SPLIT_STAGES>::TOTAL, gs[0].serial, slices);
}

cudaError_t make_group_pair(GroupLaunch& L, const fbl_plan* p, const GemmArgs* gs, int count) {
  int tiles = 0;
  cudaError_t e = fill_group(L.G, gs, count, 128, 256, 256, &tiles);   // each CTA loads 128 of the pair's 256 columns
  if (e != cudaSuccess) return e;
  const int epi = group_epi(gs, count), pairs = tiles < p->sm_count / 2 ? tiles : p->sm_count / 2;
  auto k = epi == EPI_ACT ? gemm_tc_pair_kernel<EPI_ACT> : epi == EPI_ROPE ? gemm_tc_pair_kernel<EPI_ROPE> : gemm_tc_pair_kernel<EPI_NONE>;
  return group_launch(L, k, 2 * pairs, 192, PairSmem::TOTAL, gs[0].serial);
}

}  // namespace

namespace {

// Output tiles a launch may use: 128 x 64 (slim), 128 x 128 or 128 x 256 on one CTA, 256 x 256 on a CTA pair.
enum TileKind { TILE_NARROW = 0, TILE_WIDE, TILE_PAIR, TILE_SLIM };
struct TileCost { int m, n; double kb, unit, epilogue, fixed; };      // extents; clocks per k-block, per unit, of an epilogue, per launch
// Clocks from a sweep of the four launches of a layer over 64 to 6300 tokens and widths of 320 to 3264 columns, taken before whole
// warps issued (but a pair's k-block); the choices are still the fastest, or within 2 us of it, at the workloads' sizes.  A
// k-block of a wide tile costs less than two of a narrow one (operands are re-read half as often per flop), a pair's
// less still (675 before their loading loop was shortened; with 640 in its place the ViT-Base step went from 181.3 to 179.9 us, the
// Llama-1B-shaped one from 482 to 478; 640 with 2000 a launch, or 610 with 1000, cost the feed-forward and adapter steps 1 to 4 %),
// but pairs start later; with few k-blocks the epilogue of the tile before is what a tile waits for.
const TileCost TILE_COST[4] = {{128, 128, 545, 800, 1600, 0}, {128, 256, 710, 900, 3600, 0}, {256, 256, 640, 900, 3600, 3500}, {128, 64, 400, 800, 1600, 0}};
struct TileWork { long long m; int n, kb, split; };

// Clocks of the longest block (pair) when the persistent kernel deals the units of a group's problems out in turn.  (Of a
// part with more SMs the first MAX_SLOTS stand for all; an enqueue call allocates nothing that could throw.)
constexpr int MAX_SLOTS = 512;
double tile_makespan(const TileCost& c, const TileWork* w, int count, int slots, double* idle = nullptr) {
  double load[MAX_SLOTS];
  slots = std::min(slots, MAX_SLOTS);
  std::fill(load, load + slots, 0.0);
  long long dealt = 0;
  for (int i = 0; i < count; ++i) {
    const long long units = ((w[i].m + c.m - 1) / c.m) * ((w[i].n + c.n - 1) / c.n) * w[i].split;
    const double main = ((w[i].kb + w[i].split - 1) / w[i].split + (w[i].split > 1 ? 2 : 0)) * c.kb + c.unit;
    const double len = main > c.epilogue ? main : c.epilogue;
    const int first = (int)(dealt % slots), extra = (int)(units % slots);
    for (int s = 0; s < slots; ++s) {
      const int turn = s >= first ? s - first : s - first + slots;       // this slot's place among the problem's first units
      load[(size_t)s] += (double)(units / slots + (turn < extra ? 1 : 0)) * len;
    }
    dealt += units;
  }
  double longest = 0, sum = 0;
  for (int s = 0; s < slots; ++s) { longest = std::max(longest, load[s]); sum += load[s]; }
  if (idle) *idle = longest - sum / slots;
  return longest + (dealt <= slots ? 0.5 : 1.0) * c.epilogue + c.fixed;
}

// Slices of gemm_tc_split_kernel (2 or 4; 0: that kernel is not the fastest) for a launch that takes `clocks` without.
int best_slices(const TileWork* w, int count, int sm_count, double clocks) {
  int pick = 0;
  for (int S = 2; S <= 4; S *= 2) {
    long long blocks = 0;
    int longest = 0;
    bool legal = true;
    for (int i = 0; i < count; ++i) {
      blocks += ((w[i].m + 127) / 128) * ((w[i].n + 127) / 128) * S;
      legal = legal && w[i].split == 1 && w[i].kb >= 2 * S;
      longest = std::max(longest, (w[i].kb + S - 1) / S);
    }
    if (!legal || blocks > sm_count) continue;
    // against a tile of its own: the cluster's start, the partial rows' way through shared memory, two barriers
    const double t = longest * TILE_COST[TILE_NARROW].kb + TILE_COST[TILE_NARROW].unit + 0.5 * TILE_COST[TILE_NARROW].epilogue + 5500;
    if (t < clocks) { clocks = t; pick = S; }
  }
  return pick;
}

// 128 x 64 tiles: less to load per k-block, and more SMs loading, where there are fewer tiles than SMs (50 tokens of 768:
// 20.0 -> 19.1 us a layer forward; 94 x 7 tokens of 320 x 640 gated: 57.8 -> 51.7 us a step).  With more tiles than SMs
// they only add loads of A; and a row of a head of 128, which the row reduction needs whole, spans two.
bool slim_legal(const GemmArgs* gs, int count, int sm_count) {
  long long tiles = 0;
  bool legal = true;
  for (int i = 0; i < count; ++i) {
    tiles += (long long)((gs[i].m + 127) / 128) * (gs[i].n / 64) * (gs[i].ksplit > 1 ? gs[i].ksplit : 1);
    legal = legal && (!gs[i].dot_with || gs[i].dot_hd <= 64);
  }
  return legal && tiles <= sm_count;
}

int best_tile(const TileWork* w, int count, int sm_count, bool pairs, double* clocks) {
  int kind = TILE_NARROW;
  *clocks = 1e300;
  for (int k = TILE_NARROW; k <= (pairs ? TILE_PAIR : TILE_WIDE); ++k) {
    const double t = tile_makespan(TILE_COST[k], w, count, k == TILE_PAIR ? sm_count / 2 : sm_count);
    if (t < *clocks) { *clocks = t; kind = k; }
  }
  return kind;
}

}  // namespace

// The tile whose slowest block finishes first; an offline choice for this launch, or the pair knob, comes before it.
// (N need not be whole tiles: panels past it are loaded as zeros and not stored.)
static cudaError_t make_group(GroupLaunch& L, const fbl_plan* p, const GemmArgs* gs, int count, const fbl_plan::GemmChoice& ch) {
  const int pair_mode = ch.pair >= 0 ? ch.pair : p->knob_gemm_pair;       // 0 never, 1 always, -1 by cost
  int kind = TILE_NARROW;
  GemmArgs by_length[MAX_PROBLEMS];
  TileWork w[MAX_PROBLEMS];
  for (int i = 0; i < count; ++i) {
    L.order[i] = i;
    w[i] = {gs[i].m, gs[i].n, 0, gs[i].ksplit > 1 ? gs[i].ksplit : 1};
    for (int t = 0; t < gs[i].n_terms; ++t) w[i].kb += (gs[i].t[t].k + BK - 1) / BK;
  }
  if (pair_mode == 1) {
    kind = TILE_PAIR;
  } else if (ch.bn) {
    kind = ch.bn == 128 ? TILE_NARROW : TILE_WIDE;
  } else {
    double clocks;
    kind = best_tile(w, count, p->sm_count, pair_mode != 0, &clocks);
    if (slim_legal(gs, count, p->sm_count)) {
      const double t = tile_makespan(TILE_COST[TILE_SLIM], w, count, p->sm_count);
      if (t < clocks) { clocks = t; kind = TILE_SLIM; }
    }
    const int slices = best_slices(w, count, p->sm_count, clocks);
    if (slices) {
      L.idle = 1 << 20;                              // fewer blocks than SMs, as a rule
      return make_group_split(L, gs, count, slices);
    }
    // The problems come with the token-axis reductions first; of few tokens those are the shortest, and the longest
    // units should start first.
    int order[MAX_PROBLEMS];
    for (int i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order, order + count, [&](int a, int b) { return w[a].kb / w[a].split > w[b].kb / w[b].split; });
    TileWork sorted[MAX_PROBLEMS];
    for (int i = 0; i < count; ++i) sorted[i] = w[order[i]];
    double sorted_clocks;
    const int sorted_kind = best_tile(sorted, count, p->sm_count, pair_mode != 0, &sorted_clocks);
    if (kind != TILE_SLIM && sorted_clocks < 0.95 * clocks) {
      kind = sorted_kind;
      for (int i = 0; i < count; ++i) { by_length[i] = gs[order[i]]; w[i] = sorted[i]; L.order[i] = order[i]; }
      by_length[0].serial = gs[0].serial; by_length[0].late_trigger = gs[0].late_trigger;      // the launch's own, not the problem's
      gs = by_length;
    }
  }
  double idle;
  tile_makespan(TILE_COST[kind], w, count, kind == TILE_PAIR ? p->sm_count / 2 : p->sm_count, &idle);
  L.idle = (int)idle;
  if (kind == TILE_PAIR) return make_group_pair(L, p, gs, count);
  if (kind == TILE_SLIM) return make_group_bn<64, 8>(L, p, gs, count, 1);
  if (kind == TILE_WIDE) return make_group_bn<256, 4>(L, p, gs, count, ch.esets);
  return make_group_bn<128, 6>(L, p, gs, count, ch.esets);
}

cudaError_t launch_gemm_tc_group(const fbl_plan* p, const GemmArgs* gs, int count, int32_t* status, cudaStream_t st,
                                 int launch_id) {
  if (count < 1 || count > MAX_PROBLEMS) return cudaErrorInvalidValue;
  fbl_plan::GemmChoice ch = {0, -1, 0};
  if (launch_id >= 0 && launch_id < FBL_GEMM_LAUNCH_COUNT) ch = p->choice[launch_id];
  LaunchKey key;
  gemm_group_key(key, gs, count);
  key.add(ch.bn, ch.pair);
  key.add(ch.esets, 0);
  return LaunchMemo<GroupLaunch, 12>::run(p, FBL_MEMO_TC_GEMM, key,
      [&](GroupLaunch& L) { return make_group(L, p, gs, count, ch); },
      [&](GroupLaunch& L) { return point_group(L, gs, status); },
      [&](const GroupLaunch& L) {
        if (gs[0].late_trigger) *gs[0].late_trigger = L.idle;
        if (L.cluster) return launch_cluster(L.kernel, dim3(L.grid), dim3(L.threads), L.smem, st, L.cluster, !L.serial, L.G);
        return L.serial ? launch_serial(L.kernel, dim3(L.grid), dim3(L.threads), L.smem, st, L.G)
                        : launch_pdl(L.kernel, dim3(L.grid), dim3(L.threads), L.smem, st, L.G);
      });
}

// How many slices to cut the reduction loops of the splittable problems of a group into (the same number for all
// of them).  The persistent kernel deals work units to its blocks round-robin, so a few long units beside many
// short ones leave most SMs idle: this asks, for each candidate, when the longest block of the best tile finishes,
// charging the fp32 detour (zero-fill, bulk reductions, rounding) as extra k-blocks and a fixed cost.  `zero_rides`: a
// launch in front of the group can do the zero-fill.  Each slice's tiles are read and written once more, so a small gain is
// none: of five feed-forward and attention steps whose choice the figures below changed from a dearer rounding pass, two
// gained 10 to 12 %, two 2 to 5 %, and the one that only the first group's lower price had changed lost 4 %.
int gemm_tc_choose_split(int sm_count, const GemmShape* sh, int count, bool zero_rides) {
  static const int cand[] = {1, 2, 3, 4, 6, 8, 12, 16};
  double base_cost = 0.0, best_cost = 0.0;
  int best = 1;
  for (int S : cand) {
    TileWork w[MAX_PROBLEMS];
    bool too_short = false, any_split = false;
    for (int i = 0; i < count; ++i) {
      w[i] = {sh[i].m, sh[i].n, sh[i].kblocks, sh[i].splittable ? S : 1};
      too_short = too_short || (w[i].split > 1 && sh[i].kblocks / S < 8);
      any_split = any_split || w[i].split > 1;
    }
    if (too_short || (S > 1 && !any_split)) continue;
    double cost;
    best_tile(w, count, sm_count, true, &cost);
    // zero-fill, in the launch in front or one of its own, and rounding beside the norm backward
    if (S > 1) cost += zero_rides ? 4000 : 6000;
    if (S == 1) base_cost = best_cost = cost;
    else if (cost < (zero_rides ? 0.9 : 0.85) * base_cost && cost < best_cost) { best = S; best_cost = cost; }   // worth it only with a clear gain
  }
  return best;
}

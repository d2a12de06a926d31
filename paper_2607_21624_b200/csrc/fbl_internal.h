// Internal declarations shared by the translation units of libfblayout.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "fblayout.h"

#define FBL_TILE_H 8
#define FBL_ALIGN 1024
#define FBL_PROF_MAX 32

// ---------------------------------------------------------------------------------------------
// R-Tile element map (section 4.2).  Storage tile = 8 rows x 128 bytes, row-major inside; tiles
// ordered with the row-tile index fastest.  TW = elements per 128-byte tile row.
// ---------------------------------------------------------------------------------------------
template <int TW>
__host__ __device__ __forceinline__ int64_t rt_off(int64_t r_pad, int64_t r, int c) {
  return ((int64_t)(c / TW) * r_pad + r) * TW + (c % TW);
}
__host__ __device__ __forceinline__ int64_t rt_off_dyn(int tw, int64_t r_pad, int64_t r, int64_t c) {
  return ((c / tw) * r_pad + r) * tw + (c % tw);
}

template <typename T> struct tile_w_of { static constexpr int value = 128 / (int)sizeof(T); };

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

struct FblMemoBase { virtual ~FblMemoBase() {} };      // launch_memo.h
enum { FBL_MEMO_TC_GEMM = 0, FBL_MEMO_FFMA_GEMM, FBL_MEMO_TC_FWD, FBL_MEMO_TC_BWD, FBL_MEMO_FFMA_ATTN, FBL_MEMO_TC_F32_GEMM, FBL_MEMO_TC_F32_FWD, FBL_MEMO_TC_F32_BWD, FBL_MEMO_COUNT };

struct fbl_plan {
  fbl_layer_desc d;
  int e;        // bytes per element
  int tw;       // tile_w in elements
  int t_pad;    // seq rounded up to 8
  int64_t n_pad;  // batch * t_pad
  // Key side of the attention: the same sequence in self-attention; in a cross-attention plan (cross = 1) the memory
  // sequence [batch, seq_kv, d_mem] that K and V are projected from
  int cross, seq_kv, t_pad_kv, d_mem;
  int64_t n_pad_kv;
  int dq, dkv, group;
  float scale;
  int sm_count;
  int use_tc;   // 1: tensor-core (tcgen05) kernels where one exists for the shape; 0: FFMA kernels only
  int ffma_only;   // kernel path 1: products of fp32 plans on the FP32 pipe instead of the tensor cores
  // byte offsets inside `saved`
  size_t sv_stats, sv_xn, sv_q, sv_k, sv_v, sv_a, sv_lse, sv_rope, saved_bytes;   // sv_rope: the rotary embedding's table
  // byte offsets inside the backward scratch
  size_t sb_da, sb_dvec, sb_dqacc, sb_dq, sb_dk, sb_dv, sb_dxn, sb_part, scratch_bwd_bytes;
  size_t scratch_fwd_bytes;
  size_t part_bytes;
  // reduction-loop slicing of the weight-gradient GEMMs (1: none) and their fp32 accumulation areas, which
  // follow the status word so that one fill zeroes both
  int ksplit_o, ksplit_qkv;
  size_t sb_acc_o, sb_acc_qkv, acc_bytes;
  // cross-attention only: slices of dWk / dWv, their accumulation area, dM's place is the caller's; partial sums of
  // the dK / dV column sums
  int ksplit_kv;
  size_t sb_acc_kv, sb_part_kv;
  size_t zero_bytes;        // leading part of the backward scratch that every step starts by zero-filling
  // tuning knobs, read from the environment once, at plan creation (0 / -1 = the library's own choice)
  int knob_gemm_pair;       // -1 by size, 0 never the CTA-pair GEMM kernel, 1 wherever its tile shape is legal
  int knob_gemm_esets;      // 0 by tiles per block, 1 / 2 sets of epilogue warps
  int knob_f32_bn, knob_f32_slices;   // 0 by size, 64 / 128 columns and 1, 2, 4, 8 slices of the fp32 products' tiles
  int knob_fwd_tiles;       // 0 by shape, 1 / 2 query tiles per forward-attention block at head_dim 64
  // low-rank adapters on Q, K, V (fbl_plan_enable_lora): rank, and the offsets of T = Xn [Aq|Ak|Av] inside `saved`,
  // of dT and of the unused norm-parameter gradients inside the backward scratch
  float rope_base;          // > 0: rotary position embedding on Q and K (fbl_plan_enable_rope)
  int lora_rank;
  size_t sv_t, sb_dt, sb_frozen;
  // Compute-tile configuration of each GEMM launch of a step, fixed offline by the tile chooser (0 / -1: the
  // built-in heuristics decide): output-tile width, CTA-pair kernel, sets of epilogue warps.
  struct GemmChoice { int bn, pair, esets; } choice[FBL_GEMM_LAUNCH_COUNT];
  // bookkeeping of the enqueue calls (they take the plan as const): kernels enqueued so far, optional per-step
  // event timing.  Calls on one plan are not thread-safe; give each host thread its own plan.
  mutable int64_t launches;
  mutable FblMemoBase* memo[FBL_MEMO_COUNT];
  mutable std::mutex memo_lock;
  mutable int prof_on, prof_n;
  mutable cudaEvent_t prof_ev[FBL_PROF_MAX + 1];
  mutable const char* prof_name[FBL_PROF_MAX];
};

static inline size_t fbl_align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// ---------------------------------------------------------------------------------------------
// Kernel launchers (all asynchronous on `st`; return a cudaError_t from the launch).
// ---------------------------------------------------------------------------------------------
struct GemmTerm {
  const void* a; int64_t a_rpad; int a_trans;   // logical A[m,k]; a_trans: stored as [k rows][m cols]
  const void* b; int64_t b_rpad; int b_trans;   // logical B[k,n]; b_trans: stored as [n rows][k cols]
  int k;
};
struct GemmArgs {
  int m, n, n_terms;
  GemmTerm t[4];
  void* c; int64_t c_rpad;        // C[m,n] stored [m rows][n cols]
  const float* bias;              // per output column, or nullptr
  const void* residual;           // same layout as C, or nullptr
  int seq, t_pad;                 // if t_pad > 0: rows with (row % t_pad) >= seq are written as zero
  int b_static;                   // 1: the first term's B operand is an input of the whole step (a weight)
  // optional fused row reduction D[b,h,t] = sum_d C[row, h*hd+d] * dot_with[row, h*hd+d] (C as stored, rounded)
  const void* dot_with; float* dot_out; int dot_hd, dot_hq;
  // reduction loop cut into ksplit slices whose fp32 partial tiles are added into `acc` (zeroed by the caller, same
  // element order as C with 4-byte elements); the norm backward rounds them to C (ConvertGroup)
  int ksplit; float* acc;
  // of a group's first problem: chores of the launch (zero-fill zero_bytes, a multiple of 16, at zero_ptr for a
  // later kernel of the pass; reset the pass's status word), and `serial`: the launch may not start before
  // everything ahead of it on the stream has completed
  void* zero_ptr; size_t zero_bytes; int reset_status, serial;
  // likewise, where not null (tensor-core kernels; see launch_colsum_early): the launch raises FBL_EARLY_COLSUM and lets the next
  // one start once everything ahead of it has completed; receives the clocks an SM is expected to stand idle before the
  // launch's slowest block ends, on average
  int* late_trigger;
  // fused activation of the feed-forward block (tensor-core kernel only): 0 none, 1 GELU forward (c = U, c2 = gelu(U)),
  // 2 GELU backward (c = value * gelu'(U), U in `residual`), 3 gated forward (c = G, c2 = silu(G) * U, U in `residual`),
  // 4 gated backward (c = value * silu(G), c2 = value * U * silu'(G); U in `residual`, G in `aux1`)
  // 5 rotary embedding of heads of 64 columns, with the table launch_norm_fwd leaves (see there)
  int epi; const void* aux1; void* c2; const float2* rope;
};

cudaError_t launch_gemm_simt(const GemmArgs& g, cudaStream_t st);
bool gemm_tc_supported(const fbl_plan* p, const GemmArgs& g);
cudaError_t launch_gemm_tc_group(const fbl_plan* p, const GemmArgs* gs, int count, int32_t* status, cudaStream_t st,
                                 int launch_id = -1);
bool gemm_ffma_supported(const fbl_plan* p, const GemmArgs& g);
cudaError_t launch_gemm_ffma_group(const fbl_plan* p, const GemmArgs* gs, int count, int32_t* status, cudaStream_t st);
// fp32 on the tensor cores: what gemm_ffma_supported accepts
cudaError_t launch_gemm_tc_f32_group(const fbl_plan* p, const GemmArgs* gs, int count, int32_t* status, cudaStream_t st);
// Every problem of the group can run on the tensor-core kernel and the plan wants it to.
static inline bool gemm_group_tc(const fbl_plan* p, const GemmArgs* gs, int count) {
  bool tc = p->use_tc != 0;
  for (int i = 0; i < count; ++i) tc = tc && gemm_tc_supported(p, gs[i]);
  return tc;
}
// One launch on the tensor-core kernel (bf16) or on the FFMA kernel (fp32), else one per problem on the plain FFMA kernel
// (bf16 storage, the cross-check path).  *kernels: how many were enqueued.
cudaError_t run_gemm_group(const fbl_plan* p, GemmArgs* gs, int count, int32_t* status, cudaStream_t st, int launch_id, int* kernels);
// The product that forms dA can form D = rowsum(dA * A) per head on the way.
static inline bool gemm_fuses_dot(const fbl_plan* p, const GemmArgs& ga) {
  return p->d.dtype == FBL_DTYPE_FP32 ? p->d.head_dim <= 64 && gemm_ffma_supported(p, ga) : p->use_tc && gemm_tc_supported(p, ga);
}
// The rotary embedding in the epilogue of the Q and K projections (gs[0], gs[1] of three): true if it goes there.  A head of
// 64 is one panel of the epilogue; one of 128 needs the neighbouring panel's accumulators and twice the table per element,
// which took longer than a pass of its own (26900 tokens of 6 + 1 heads: 238 us against 61 and 34 us).
static inline bool rope_in_projection(const fbl_plan* p, GemmArgs* gs, const float2* table) {
  if (!(p->rope_base > 0.f) || p->d.head_dim != 64 || !gemm_group_tc(p, gs, 3)) return false;
  for (int i = 0; i < 2; ++i) { gs[i].epi = 5; gs[i].rope = table; }
  return true;
}
// First k-block of a slice where a cluster shares a reduction of `total` k-blocks: shares differ by one at most, so none is
// empty unless there are fewer k-blocks than slices.  (Shares rounded up leave the last ones short: nine k-blocks in four
// make 3, 3, 3 and none.)
__host__ __device__ __forceinline__ int gemm_slice_begin(int total, int slices, int slice) { return total * slice / slices; }
struct GemmShape { int64_t m; int n; int kblocks; int splittable; };
int gemm_tc_choose_split(int sm_count, const GemmShape* sh, int count, bool zero_rides);
cudaError_t launch_wait_timeout_selftest(int32_t* status, long long limit_cycles, cudaStream_t st);
// With less than a tile of token rows on either side a bf16 layer keeps P and dS in fp32, or in two bf16 values: their rounding
// is as large as that of the results there (dQ, dK, dV off by 2.3e-3 of their norm instead of 1.65e-3), and with the rotary
// embedding dbk, what the rotation leaves of sums that cancel without it, is off by up to 1.5 %.  The line is where the caller's
// results have always changed over; what it costs against P and dS in bf16 (us a step): 50 tokens of 12 heads 59 -> 72, 120
// tokens of 16 heads over one KV head 69 -> 123, 8 queries over 1500 memory rows 115 -> 134, 4096 queries over 40 memory rows
// 192 -> 348 (plain fp32 kernels: 87, 583, 338, 1330).
static inline bool attn_fp32(const fbl_plan* p) { return p->n_pad < 128 || p->n_pad_kv < 128; }
// The kernels that a plan's attention runs on.
enum { ATTN_TC = 0, ATTN_FFMA, ATTN_SIMT };
static inline int attn_fwd_kernels(const fbl_plan* p) { return p->d.dtype == FBL_DTYPE_FP32 ? ATTN_FFMA : p->use_tc ? ATTN_TC : ATTN_SIMT; }
static inline int attn_bwd_kernels(const fbl_plan* p) { return p->use_tc && attn_fp32(p) ? ATTN_FFMA : attn_fwd_kernels(p); }
bool attn_bwd_tc_direct(const fbl_plan* p);    // the tensor-core backward writes dQ itself: no fp32 accumulator to zero and round
// Leading bytes of the backward scratch a step starts by zero-filling: status word and sliced products' accumulation areas,
// and behind them the dQ accumulator where the attention backward adds into it.
static inline size_t bwd_zero_bytes(const fbl_plan* p) {
  return attn_bwd_kernels(p) == ATTN_TC && attn_bwd_tc_direct(p) ? p->sb_dqacc : p->zero_bytes;
}
// Flags of pdl_early in the first block of the backward scratch, as offsets in words from the status word; a pass clears them
// with it.  FBL_EARLY_COLSUM: from the last products to the column sums beside them; FBL_EARLY_ROUND: from the norm backward's
// first kernel to the roundings beside it.
enum { FBL_EARLY_COLSUM = 64, FBL_EARLY_ROUND = 128 };
// What a backward pass starts with: zero the first `bytes` of its scratch (the status word's block and the fp32 areas the
// pass adds into).  `rides`: the pass's first products `gs` need nothing of it.  `serial`: no kernel of the pass may start
// before the forward pass has completed (the attention backward requests that pass's results before waiting for the kernel
// in front of it).  Counts a launch of its own.
cudaError_t start_backward(const fbl_plan* p, GemmArgs* gs, int count, bool rides, bool serial, int32_t* status, size_t bytes, cudaStream_t st);

// One launch forward.  Backward: D unless it is there, the attention, dQ's rounding where it was summed in fp32.  The rotation
// of dQ and dK back goes with that rounding where `attn_bwd_turns`, else it is a step of its own.
cudaError_t run_attn_fwd(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse, int32_t* status, cudaStream_t st);
cudaError_t run_attn_bwd(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* A, const void* dA, const float* lse,
                         float* dvec, float* dqacc, void* dQ, void* dK, void* dV, bool dvec_ready, int32_t* status, cudaStream_t st,
                         const float2* rope);
static inline bool attn_bwd_turns(const fbl_plan* p) { return p->rope_base > 0.f && p->use_tc; }
static inline int attn_bwd_launches(const fbl_plan* p, bool dvec_ready) {
  const bool summed = attn_bwd_kernels(p) != ATTN_TC || !attn_bwd_tc_direct(p);
  return (dvec_ready ? 1 : 2) + (p->d.dtype == FBL_DTYPE_BF16 && (summed || attn_bwd_turns(p)) ? 1 : 0);
}
void fbl_note_cuda_error(cudaError_t e, const char* where);

cudaError_t launch_pack(int dtype, int unpack, const void* src, void* dst, int64_t outer, int64_t rows,
                        int64_t rows_pad, int cols, cudaStream_t st);
// fp32 dQ sums -> dQ in bf16, and dK in place, both turned back by the table's angles
cudaError_t launch_rope_bwd_round(const fbl_plan* p, const float* acc, void* dQ, void* dK, const float2* rope, cudaStream_t st);
cudaError_t launch_rope(const fbl_plan* p, void* A, int heads_a, void* B, int heads_b, int inverse, cudaStream_t st);
// rope: where to leave the rotary embedding's table, [head_dim / 2][t_pad] (cosine, sine) of token t * base^(-2i/head_dim)
cudaError_t launch_norm_fwd(const fbl_plan* p, const void* X, const float* gamma, const float* beta, void* Xn,
                            float* stats, int32_t* status, cudaStream_t st, float2* rope = nullptr);
// Token-axis column sums of up to four matrices: slabs of 256 rows are summed to one row of partials each (at part[i],
// slabs x cols), which a second kernel adds up.
struct ColsumGroup {
  const void* m[4];
  float* out[4];
  float* part[4];
  int64_t rows[4];
  int cols[4], slabs[4];
  int count;
  int summed;               // the slabs' sums are under way already (launch_colsum_early)
};
// Adds a matrix; its partials come from *part, which moves on.
void colsum_add(ColsumGroup& G, const void* m, int64_t rows, int cols, float* out, float** part);
// Panels of slabs: the pieces of work of the first stage.
static inline int64_t colsum_units(const fbl_plan* p, const ColsumGroup& G) {
  int64_t units = 0;
  for (int i = 0; i < G.count; ++i) units += (int64_t)G.slabs[i] * (G.cols[i] / p->tw);
  return units;
}
// Whether the sums are better off beside the products than in the norm backward's launches, where up to about two pieces
// per SM pass unnoticed (steps of 10 to 120 us: 1 to 4 % slower beside the products with up to 324 pieces on 148 SMs, 2 to
// 5 % faster with 366 and more).
static inline bool colsum_early_pays(const fbl_plan* p, const ColsumGroup& G) {
  return G.count > 0 && 4 * colsum_units(p, G) > 9 * (int64_t)p->sm_count;
}
// The slabs' sums as a launch behind a tensor-core product launch with late_trigger (which gave `idle`), beside which it runs:
// the matrices must come from launches in front of that one.  `status`: of both launches.
cudaError_t launch_colsum_early(const fbl_plan* p, ColsumGroup& G, int idle, int32_t* status, cudaStream_t st);
cudaError_t launch_early_order_selftest(const fbl_plan* p, void* M, int64_t rows, int cols, float* out, int32_t* status, float* part,
                                        cudaStream_t st);
// Where the norm's own partial rows begin, behind column-sum partials from `part` to `end`.
static inline float* norm_partials(float* part, const float* end) { return part + (end - part + 255) / 256 * 256; }
// fp32 sums of sliced products, to be rounded to their bf16 places (n multiples of 4).
struct ConvertGroup { const float* src[4]; void* dst[4]; int64_t n[4]; int count; };
// Norm backward with the column sums of `sums` and the roundings of `round`; counts its own launches in p->launches (one to
// three).
cudaError_t launch_norm_bwd(const fbl_plan* p, const void* dXn, const void* X, const void* dY, const float* stats,
                            const float* gamma, void* dX, float* dgamma, float* dbeta, float* part, int32_t* status,
                            cudaStream_t st, const ColsumGroup* sums = nullptr, const ConvertGroup* round = nullptr);
cudaError_t launch_colsum(int dtype, const void* M, int64_t rows, int64_t cols, float* out, float* partials,
                          cudaStream_t st);
size_t colsum_scratch_bytes(int64_t rows, int64_t cols);
cudaError_t launch_colsum_group(int dtype, const ColsumGroup& G, cudaStream_t st);

// fp32 arithmetic (k_ffma_attn.cu): fp32 storage where not attn_tc_f32_supported, and the backward of bf16 storage.  The latter adds into dQ or, bf16, into dqacc,
// zeroed by the caller; dqacc it rounds and, with `rope`, turns
cudaError_t launch_attn_fwd_ffma(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse,
                                 int32_t* status, cudaStream_t st);
cudaError_t launch_attn_bwd_ffma(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* A, const void* dA,
                                 const float* lse, float* dvec, float* dqacc, void* dQ, void* dK, void* dV, bool dvec_ready,
                                 int32_t* status, cudaStream_t st, const float2* rope);
// fp32 storage on the tensor cores (k_tc_f32_attn.cu): heads of 32 and 64
bool attn_tc_f32_supported(const fbl_plan* p);
cudaError_t launch_attn_fwd_tc_f32(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse,
                                   int32_t* status, cudaStream_t st);
cudaError_t launch_attn_bwd_tc_f32(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* A, const void* dA,
                                   const float* lse, float* dvec, void* dQ, void* dK, void* dV, bool dvec_ready, int32_t* status,
                                   cudaStream_t st);       // adds into dQ, zeroed by the caller
// bf16 storage in fp32 arithmetic (cross-check)
cudaError_t launch_attn_fwd_simt(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse,
                                 cudaStream_t st);
cudaError_t launch_attn_bwd_simt(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* A,
                                 const void* dA, const float* lse, float* dvec, float* dqacc, void* dQ, void* dK,
                                 void* dV, bool dvec_ready, cudaStream_t st);
cudaError_t launch_attn_bwd_pre(const fbl_plan* p, const void* A, const void* dA, float* dvec, bool dvec_ready, cudaStream_t st);
cudaError_t launch_attn_bwd_post(const fbl_plan* p, const float* dqacc, void* dQ, cudaStream_t st);
cudaError_t launch_attn_fwd_tc(const fbl_plan* p, const void* Q, const void* K, const void* V, void* A, float* lse,
                               int32_t* status, cudaStream_t st);
cudaError_t launch_attn_bwd_tc(const fbl_plan* p, const void* Q, const void* K, const void* V, const void* A,
                               const void* dA, const float* lse, float* dvec, float* dqacc, void* dQ, void* dK,
                               void* dV, bool dvec_ready, int32_t* status, cudaStream_t st, const float2* rope = nullptr);

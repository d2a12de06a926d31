// fp32 products on the tensor cores, with the accuracy of fp32 arithmetic.  An fp32 value is the sum of three bf16 values (its
// rounding, the rounding of what that leaves, and the rest: 24 bits), so a product of two is nine bf16 products, of which the
// three smallest are below 2^-26 of the whole and left out.  The other six run as tcgen05.mma with fp32 accumulation:
//   lo x hi, hi x lo, mid x mid, mid x hi, hi x mid, hi x hi          (operand A's part x operand B's)
// 1614 / 6 = 269 TFLOP/s of fp32 work where the FP32 pipe has 74.
//
// Accuracy.  Every bf16 x bf16 product is exact in fp32; what is lost is the tensor core's own accumulation.  The accumulator
// is therefore used for no more than 64 columns of a reduction, the small products first, and added to a sum that a thread
// keeps in registers (rounded to nearest): no value passes more than four accumulations at its full size before such an addition.
// An infinity has no parts (inf - inf is NaN), so a block whose part of a tile is not finite throughout (and so where an operand
// is 2^111 or more, or a result 2^96) forms it again by plain multiply-adds: infinities and NaN go where the FP32 pipe puts them.
// (ViT-shaped step of 4 x 197 tokens with an infinity in X, which reaches every weight gradient: 850 us, all on the FP32 pipe 450, a
// thread to a result 20000; feed-forward step of 800 x 768 x 3072 950, 630, 12000.)
//
// One block per 128 x BN tile, or per slice of its reduction (then a cluster shares the tile; partial tiles meet in distributed
// shared memory in a fixed order: no atomics, the same bits every time).  18 warps: one loads fp32 operand tiles by TMA, four
// turn A's rows into packed bf16 parts in tensor memory, four turn B's into three tiles in shared memory in the canonical
// 128-byte-swizzled layout (K-major or MN-major as the operand lies: nothing is transposed on the way), one issues the products,
// eight add the finished accumulators up.  A lies in tensor memory because shared memory is the bound: per 64 columns a
// 128 x 128 tile moves 64 KB in, 64 KB out to the conversions, 48 KB of B's parts in and 96 KB of them out to the tensor core,
// 272 KB at 128 B/clk, where A's parts in shared memory would make it 416 KB (the products take 1536 clk).  Counted: the tensor pipe
// is active for 31 to 46 % of active cycles (800 x 768 outputs, 768 to 800 columns to reduce), conversions and waits for them the rest.
// Measured against the FP32 pipe (k_ffma_gemm.cu), us: 800 x 768 outputs, 768 columns to reduce: three problems 74 -> 22.8, one
// 31 -> 15.3, dWo with dA 60 -> 23.8, dWq, dWk, dWv with dXn 159 -> 47.7; 2048 x 2048 x 2048 358 -> 93 (185 TFLOP/s); 64 x 64 x 64
// 6.5 -> 5.5.  Error against 64 bits relative to the result's norm: 0.4e-7 to 1.8e-7 at 32 to 4096 columns, multiply-adds one after
// another 1.0e-7 to 9.9e-7; whole steps' outputs: 0.3 to 1.0 of theirs.
#include "f32_gemm.cuh"
#include "launch_memo.h"
#include "pdl.cuh"

namespace {

using f32g::Group;
using f32g::Problem;
using f32g::lds4;

constexpr int BM = 128, BK = 64;
// load, issue; A (4); B (4); sums (8).  (Eight converting warps for each operand, with the registers dealt out by setmaxnreg:
// 5 % slower.)
constexpr int WARPS = 18, THREADS = 32 * WARPS;
constexpr int CONVERTING = 8;

template <int BN>
struct Smem {
  static constexpr int STAGES = BN == 128 ? 2 : 3;
  static constexpr uint32_t A_BYTES = BM * BK * 4, B_BYTES = BN * BK * 4, STAGE = A_BYTES + B_BYTES;
  static constexpr uint32_t PART = BN * 128, PARTS_OFF = STAGES * STAGE;              // two sets of three parts of B
  static constexpr uint32_t BAR_OFF = PARTS_OFF + 6 * PART, N_BARS = 2 * STAGES + 6;
  static constexpr uint32_t TOTAL = BAR_OFF + 8 * N_BARS + 16 + 1024;                 // + tensor memory slot, flag, alignment slack
  static constexpr int LD = BN + 4;                                                   // row pitch of the finished tile
  static_assert(BM * LD * 4 <= STAGES * STAGE, "the finished tile fits the stages");
};
// tensor memory: two accumulators of BN columns, then two sets of A's three parts, 32 columns each
constexpr uint32_t TMEM_COLS = 512;
template <int BN> __device__ constexpr uint32_t a_col(int set, int part) { return 2 * BN + 96 * set + 32 * part; }

using tc::split3;
constexpr float LIFT = 2.7e-8f;       // of either operand: between them 0.9 of tc::LIFT_4, of one alone less than what brings up the next value
using tc::sts4;

// This block's part of its tile (k-blocks kb_begin .. kb_end) once more by multiply-adds, all threads of the block: where a result
// is not finite, which an infinity makes of every product that it is in.  32 columns of the reduction at a time, at `stage` in shared memory as
// [column][row]; a thread has four rows and BN / 16 columns of the tile, which goes to `tile` (rows LD floats apart).
template <int BN>
__device__ __noinline__ void plain_tile(const Problem& P, uint32_t tile, uint32_t stage, int m0, int n0, int kb_begin, int kb_end) {
  constexpr int KS = 32, LDA = BM + 4, LDB = BN + 4, NV = BN / 64, GROUPS = 512;
  static_assert(KS * (LDA + LDB) * 4 <= (int)(6 * Smem<BN>::PART) && GROUPS <= THREADS && GROUPS * 4 * 4 * NV == BM * BN, "parts' area, a thread's results");
  const uint32_t sa = stage, sb = stage + KS * LDA * 4;
  const int row = (int)(threadIdx.x / 16) * 4, col = (int)(threadIdx.x % 16) * 4;          // columns col, col + 64
  float4 sum[4][NV];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int v = 0; v < NV; ++v) sum[i][v] = make_float4(0.f, 0.f, 0.f, 0.f);
  // `rows` rows from r0 on (of `end`) of one operand, columns k0 .. k0 + 31 (of K) of the reduction; zeros beyond
  auto fill = [&](uint32_t to, int ld, int rows, const float* m, long long r_pad, bool rows_are_k, int r0, int end, int k0, int K) {
    for (int e = threadIdx.x; e < rows * (KS / 4); e += THREADS) {
      if (rows_are_k) {
        const int k = e / (rows / 4), r = e % (rows / 4) * 4;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 + r < end && k0 + k < K) x = *reinterpret_cast<const float4*>(m + rt_off<32>(r_pad, k0 + k, r0 + r));
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(to + (k * ld + r) * 4), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w) : "memory");
      } else {
        const int r = e % rows, k = e / rows * 4;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 + r < end && k0 + k < K) x = *reinterpret_cast<const float4*>(m + rt_off<32>(r_pad, r0 + r, k0 + k));
        const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) asm volatile("st.shared.f32 [%0], %1;" ::"r"(to + ((k + i) * ld + r) * 4), "f"(v[i]) : "memory");
      }
    }
  };
  int t = 0, kb = kb_begin;
#pragma unroll 1
  for (int left = kb_end - kb_begin; left > 0; --left, ++kb) {
    while (kb >= P.kblocks[t]) { kb -= P.kblocks[t]; ++t; }
#pragma unroll 1
    for (int k0 = kb * BK; k0 < min(kb * BK + BK, P.k[t]); k0 += KS) {
      __syncthreads();
      fill(sa, LDA, BM, P.a[t], P.a_rpad[t], P.a_k[t] != 0, m0, P.m, k0, P.k[t]);
      fill(sb, LDB, BN, P.b[t], P.b_rpad[t], P.b_k[t] != 0, n0, P.n, k0, P.k[t]);
      __syncthreads();
      if (threadIdx.x < GROUPS) {
#pragma unroll 4
        for (int k = 0; k < KS; ++k) {
          const float4 a4 = lds4(sa + (k * LDA + row) * 4);
          const float a[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const float4 b = lds4(sb + (k * LDB + col + 64 * v) * 4);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              sum[i][v].x = fmaf(a[i], b.x, sum[i][v].x); sum[i][v].y = fmaf(a[i], b.y, sum[i][v].y);
              sum[i][v].z = fmaf(a[i], b.z, sum[i][v].z); sum[i][v].w = fmaf(a[i], b.w, sum[i][v].w);
            }
          }
        }
      }
    }
  }
  if (threadIdx.x < GROUPS)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int v = 0; v < NV; ++v) sts4(tile + ((row + i) * Smem<BN>::LD + col + 64 * v) * 4, reinterpret_cast<const uint32_t*>(&sum[i][v]));
  __syncthreads();
}

template <int BN>
__global__ void __launch_bounds__(THREADS, 1) gemm_tc_f32_kernel(const __grid_constant__ Group G) {
  using SM = Smem<BN>;
  constexpr int STAGES = SM::STAGES;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + SM::BAR_OFF, slot = bars + 8 * SM::N_BARS, flag = slot + 8;
  auto full = [&](int s) { return bars + 8u * s; };                         // fp32 tiles of a stage have arrived
  auto empty = [&](int s) { return bars + 8u * (STAGES + s); };             // ... have been read
  auto parts = [&](int b) { return bars + 8u * (2 * STAGES + b); };         // both operands' parts are in place
  auto done = [&](int b) { return bars + 8u * (2 * STAGES + 2 + b); };      // the products have read them: accumulator complete
  auto added = [&](int b) { return bars + 8u * (2 * STAGES + 4 + b); };     // the accumulator has been read
  const int warp = (int)tc::uniform(threadIdx.x / 32), lane = threadIdx.x % 32;
  const tc::Status status(G.status, G.reset_status);
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(full(s), 1);
      tc::mbar_init(empty(s), CONVERTING);    // one arrival per converting warp
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(parts(b), CONVERTING);
      tc::mbar_init(done(b), 1);
      tc::mbar_init(added(b), 8);
    }
    tc::fence_barrier_init();
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag), "r"(0u) : "memory");
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
  // work unit: (problem, tile, slice); the slices of a tile are the blocks of a cluster
  const int slice = blockIdx.x % G.slices;
  int w = blockIdx.x / G.slices, pi = 0;
  while (w >= G.p[pi].tiles_m * G.p[pi].tiles_n) { w -= G.p[pi].tiles_m * G.p[pi].tiles_n; ++pi; }
  const Problem& P = G.p[pi];
  const int m0 = (w % P.tiles_m) * BM, n0 = (w / P.tiles_m) * BN;
  const int kb_begin = gemm_slice_begin(P.total_kb, G.slices, slice), n_kb = gemm_slice_begin(P.total_kb, G.slices, slice + 1) - kb_begin;

  if (warp == 0) {
    if (lane == 0) {
      auto load_b = [&](int it, int t, int k) {
        const uint32_t sb = base + it % STAGES * SM::STAGE + SM::A_BYTES;
        if (P.b_k[t]) tc::tma_load_3d(sb, &P.tb[t], full(it % STAGES), 0, k * BK, n0 / 32);
        else tc::tma_load_3d(sb, &P.tb[t], full(it % STAGES), 0, n0, k * (BK / 32));
      };
      // weights do not depend on the kernel in front: the first stages' are requested before waiting for it
      int ahead = 0;
      if (P.b_static)
        for (; ahead < STAGES && ahead < n_kb && kb_begin + ahead < P.kblocks[0]; ++ahead) {
          tc::mbar_expect_tx(full(ahead), SM::STAGE);
          load_b(ahead, 0, kb_begin + ahead);
        }
      pdl_wait();
      int t = 0, k = kb_begin;
      for (int it = 0; it < n_kb; ++it, ++k) {
        while (k >= P.kblocks[t]) { k -= P.kblocks[t]; ++t; }
        const int s = it % STAGES;
        if (it >= ahead) {
          if (!tc::mbar_wait(empty(s), ((it / STAGES) & 1) ^ 1, status, 131)) break;
          tc::mbar_expect_tx(full(s), SM::STAGE);
        }
        const uint32_t sa = base + s * SM::STAGE;
        if (P.a_k[t]) tc::tma_load_3d(sa, &P.ta[t], full(s), 0, k * BK, m0 / 32);
        else tc::tma_load_3d(sa, &P.ta[t], full(s), 0, m0, k * (BK / 32));
        if (it >= ahead) load_b(it, t, k);
      }
    }
  } else if (warp == 1) {
    const bool leader = tc::elect_one();
    const uint32_t hi = tc::smem_desc_hi(1024);
    const uint32_t idesc = tc::idesc_bf16(BM, BN, 0, P.b_k[0]);
    const uint32_t b_lo = tc::smem_desc_lo(base + SM::PARTS_OFF, P.b_k[0] ? 8192u : 16u), b_step = P.b_k[0] ? 128u : 2u;
    for (int it = 0; it < n_kb; ++it) {
      const int b = it & 1;
      const uint32_t ph = (it >> 1) & 1;
      if (!tc::mbar_wait_warp(added(b), ph ^ 1, status, 132) || !tc::mbar_wait_warp(parts(b), ph, status, 133)) break;
      tc::tc_fence_after();
      const uint32_t d = tmem_base + b * BN, bs = b_lo + b * (3 * SM::PART >> 4);
      auto product = [&](int pa, int pb) {
        if (!leader) return;
#pragma unroll
        for (uint32_t kk = 0; kk < BK / 16; ++kk)
          tc::mma_bf16_ts_w(d, tmem_base + a_col<BN>(b, pa) + kk * 8, bs + pb * (SM::PART >> 4) + kk * b_step, hi, idesc, pa < 2 || kk > 0);
      };
      product(2, 0); product(0, 2); product(1, 1); product(1, 0); product(0, 1); product(0, 0);
      if (leader) tc::mma_commit(done(b));
    }
  } else if (warp < 6) {
    // ---- A: a thread owns a row, 16 values at a time -> eight packed columns of each part
    const int q = warp % 4;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    const bool a_k = P.a_k[0] != 0;
    for (int it = 0; it < n_kb; ++it) {
      const int s = it % STAGES, b = it & 1;
      if (!tc::mbar_wait(full(s), (it / STAGES) & 1, status, 134) || !tc::mbar_wait(done(b), ((it >> 1) & 1) ^ 1, status, 135)) break;
      tc::tc_fence_after();
      const uint32_t sa = base + s * SM::STAGE;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        float x[16];
        if (a_k) {                            // the tile's rows are K indices: the thread's column, K rows 16 h ...
          const uint32_t col = sa + q * (BK * 128) + (lane & 3) * 4;
#pragma unroll
          for (int k = 0; k < 16; ++k)
            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x[k]) : "r"(col + (h * 16 + k) * 128 + (((lane >> 2) ^ (k & 7)) << 4)));
        } else {
          const uint32_t row = sa + (h / 2) * (BM * 128) + (q * 32 + lane) * 128;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float4 v = lds4(row + (((h % 2 * 4 + c) ^ (lane & 7)) << 4));
            x[4 * c] = v.x; x[4 * c + 1] = v.y; x[4 * c + 2] = v.z; x[4 * c + 3] = v.w;
          }
        }
        uint32_t p[3][8];
#pragma unroll
        for (int k = 0; k < 8; ++k) split3(x[2 * k], x[2 * k + 1], LIFT, p[0][k], p[1][k], p[2][k]);
#pragma unroll
        for (int i = 0; i < 3; ++i) tc::tmem_st8(lane_addr + a_col<BN>(b, i) + 8 * h, p[i]);
      }
      tc::tmem_st_wait();
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) { tc::mbar_arrive(empty(s)); tc::mbar_arrive(parts(b)); }
    }
  } else if (warp < 10) {
    // ---- B: 16 values of a row at a time, two 16-byte chunks of each part out -----------------------------------------
    const int tid = threadIdx.x - 6 * 32;
    const int rows = P.b_k[0] ? BK : BN;      // of a bf16 tile of 64 columns, and so of each of the two fp32 panels that it is made of
    for (int it = 0; it < n_kb; ++it) {
      const int s = it % STAGES, b = it & 1;
      if (!tc::mbar_wait(full(s), (it / STAGES) & 1, status, 136) || !tc::mbar_wait(done(b), ((it >> 1) & 1) ^ 1, status, 137)) break;
      const uint32_t sb = base + s * SM::STAGE + SM::A_BYTES, out = base + SM::PARTS_OFF + b * (3 * SM::PART);
#pragma unroll
      for (int u = 0; u < BN / 32; ++u) {
        const int unit = u * 128 + tid, h = unit / (2 * BN), panel = unit % (2 * BN) / rows, r = unit % rows;    // fp32 panel: 32 columns
        const uint32_t src = sb + panel * (rows * 128) + r * 128, dst = out + (panel / 2) * (rows * 128) + r * 128;
        float x[16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4 v = lds4(src + (((h * 4 + c) ^ (r & 7)) << 4));
          x[4 * c] = v.x; x[4 * c + 1] = v.y; x[4 * c + 2] = v.z; x[4 * c + 3] = v.w;
        }
        uint32_t p[3][8];
#pragma unroll
        for (int k = 0; k < 8; ++k) split3(x[2 * k], x[2 * k + 1], LIFT, p[0][k], p[1][k], p[2][k]);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int c = 0; c < 2; ++c) sts4(dst + i * SM::PART + (((panel % 2 * 4 + h * 2 + c) ^ (r & 7)) << 4), &p[i][4 * c]);
      }
      tc::fence_proxy_async();
      __syncwarp();
      if (lane == 0) { tc::mbar_arrive(empty(s)); tc::mbar_arrive(parts(b)); }
    }
  } else {
    // ---- sums: half a row per thread ----------------------------------------------------------------------------------
    constexpr int N = BN / 2;
    const int q = warp % 4, half = (warp - 10) / 4;
    float2 sum[N / 2];
#pragma unroll
    for (int i = 0; i < N / 2; ++i) sum[i] = make_float2(0.f, 0.f);
    pdl_wait();
    f32g::group_chores(G, threadIdx.x - 10 * 32, 256);
    for (int it = 0; it < n_kb; ++it) {
      const int b = it & 1;
      if (!tc::mbar_wait(done(b), (it >> 1) & 1, status, 138)) break;
      tc::tc_fence_after();
#pragma unroll
      for (int c = 0; c < N / 16; ++c) {
        uint32_t v[16];
        tc::tmem_ld16(tmem_base + ((uint32_t)(q * 32) << 16) + b * BN + half * N + 16 * c, v);
        tc::tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 8; ++i) sum[8 * c + i] = __fadd2_rn(sum[8 * c + i], make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])));
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(added(b));
    }
    float2 probe = make_float2(0.f, 0.f);     // NaN if and only if a sum is not finite
#pragma unroll
    for (int i = 0; i < N / 2; ++i) probe = __ffma2_rn(sum[i], make_float2(0.f, 0.f), probe);
    if (!(probe.x == 0.f && probe.y == 0.f)) asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag), "r"(1u) : "memory");
#pragma unroll
    for (int i = 0; i < N / 2; ++i) sum[i] = __fmul2_rn(sum[i], make_float2(tc::PARTS_BACK, tc::PARTS_BACK));
    // the partial tile, over the stages: the last accumulator is complete, so every operand has been read
    const uint32_t row = base + (uint32_t)((q * 32 + lane) * SM::LD + half * N) * 4;
#pragma unroll
    for (int i = 0; i < N; i += 4) sts4(row + i * 4, reinterpret_cast<const uint32_t*>(&sum[i / 2]));
  }
  __syncwarp();
  tc::tc_fence_before();
  pdl_wait();                                      // before anything is written
  __syncthreads();
  uint32_t again;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(again) : "r"(flag) : "memory");
  if (again) plain_tile<BN>(P, base, base + SM::PARTS_OFF, m0, n0, kb_begin, kb_begin + n_kb);
  if (G.slices > 1) tc::cluster_sync_all();
  if (warp == 1) tc::tmem_dealloc(tmem_base, TMEM_COLS);
  f32g::finish_tile<BM, BN, SM::LD, THREADS>(P, G.slices, slice, base, m0, n0);
  if (G.slices > 1) tc::cluster_sync_all();      // no block leaves while another may still read its partial tile
}

struct Launch { Group G; int grid, bn; };

// Tile width (128, 64) and slices (1, 2, 4, 8: blocks of a cluster) of a launch: the shortest list schedule, in the order of the
// grid, of its tiles over the clusters that fit the part at once.  Measured: a block takes some 6 us (64 columns: 4.5) to come up,
// fill its pipeline and finish its tile, and 1.06 us (0.9) for every 64 columns of the reduction.  800 x 768 outputs, with 1, 2, 4
// slices of 128 and 64 columns (us): three problems of 768 columns 22.6 30 47, 36 48 73; one of them 21.7 15.2 22.6, 18 24 27; dWo with
// dA 23.7 28.6 36, 35 37 48; dWq, dWk, dWv with dXn 74 61 76, 80 89 117.  128 x 512 x 512: 16.0 12.2 9.7, 13.2 10.2 7.9.
struct Choice { int bn, slices; };
Choice choose(const fbl_plan* p, const GemmArgs* gs, const int* order, int count) {
  Choice best = {128, 1};
  double best_t = 1e30;
  for (int bn = 128; bn >= 64; bn -= 64)
    for (int s = 1; s <= 8; s *= 2) {
      if ((p->knob_f32_bn && bn != p->knob_f32_bn) || (p->knob_f32_slices && s != p->knob_f32_slices)) continue;
      constexpr int MAX_SLOTS = 256;
      double end[MAX_SLOTS], cost[f32g::MAX_PROBLEMS], load = 0, whole = 0;      // end: a heap, the earliest on top
      // clusters of 4 and 8 do not fill every group of SMs that shares a scheduler
      const int fit = s == 4 ? p->sm_count * 36 / 148 : s == 8 ? p->sm_count * 16 / 148 : p->sm_count / s;
      const int slots = fit < 1 ? 1 : fit > MAX_SLOTS ? MAX_SLOTS : fit;
      long long units[f32g::MAX_PROBLEMS];
      for (int j = 0; j < count; ++j) {
        const GemmArgs& g = gs[order[j]];
        int kb = 0;
        for (int i = 0; i < g.n_terms; ++i) kb += (g.t[i].k + BK - 1) / BK;
        cost[j] = (bn == 128 ? 6.0 : 4.5) + (bn == 128 ? 1.06 : 0.9) * ((kb + s - 1) / s) + (s > 1 ? 0.3 : 0.0);
        units[j] = (long long)((g.m + BM - 1) / BM) * ((g.n + bn - 1) / bn);
        load += units[j] * cost[j] / slots;
        const long long rounds = units[j] / slots > 1 ? units[j] / slots - 1 : 0;     // rounds that leave the order as it is
        whole += rounds * cost[j];
        units[j] -= rounds * slots;
      }
      if (load >= best_t * 0.99) continue;
      for (int i = 0; i < slots; ++i) end[i] = 0;
      double t = 0;
      for (int j = 0; j < count; ++j)
        for (long long u = 0; u < units[j]; ++u) {
          const double e = end[0] + cost[j];
          t = e > t ? e : t;
          int i = 0;
          for (int c; (c = 2 * i + 1) < slots; i = c) {
            if (c + 1 < slots && end[c + 1] < end[c]) ++c;
            if (end[c] >= e) break;
            end[i] = end[c];
          }
          end[i] = e;
        }
      t += whole;
      if (t < best_t * 0.99) { best_t = t; best = {bn, s}; }
    }
  return best;
}

}  // namespace

cudaError_t launch_gemm_tc_f32_group(const fbl_plan* p, const GemmArgs* gs, int count, int32_t* status, cudaStream_t st) {
  if (count < 1 || count > f32g::MAX_PROBLEMS) return cudaErrorInvalidValue;
  LaunchKey key;
  gemm_group_key(key, gs, count);
  return LaunchMemo<Launch, 12>::run(p, FBL_MEMO_TC_F32_GEMM, key,
      [&](Launch& L) {
        int order[f32g::MAX_PROBLEMS];
        f32g::longest_first(gs, count, order);
        const Choice c = choose(p, gs, order, count);
        if (!f32g::fill_group(L.G, gs, count, order, BM, c.bn, BK)) return cudaErrorInvalidValue;
        L.grid = 0;
        for (int i = 0; i < count; ++i) L.grid += L.G.p[i].tiles_m * L.G.p[i].tiles_n * c.slices;
        L.G.slices = c.slices;
        L.bn = c.bn;
        const cudaError_t e = cudaFuncSetAttribute(gemm_tc_f32_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem<128>::TOTAL);
        return e != cudaSuccess ? e : cudaFuncSetAttribute(gemm_tc_f32_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem<64>::TOTAL);
      },
      [&](Launch& L) { return f32g::point_group(L.G, gs, status); },
      [&](const Launch& L) {
        auto go = [&](auto kernel, size_t smem) {
          if (L.G.slices > 1) return launch_cluster(kernel, dim3(L.grid), dim3(THREADS), smem, st, L.G.slices, true, L.G);
          return launch_pdl(kernel, dim3(L.grid), dim3(THREADS), smem, st, L.G);
        };
        return L.bn == 128 ? go(gemm_tc_f32_kernel<128>, Smem<128>::TOTAL) : go(gemm_tc_f32_kernel<64>, Smem<64>::TOTAL);
      });
}

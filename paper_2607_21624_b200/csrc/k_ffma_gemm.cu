// fp32 GEMMs on the FP32 pipe, the cross-check of the kernel that runs them on the tensor cores (k_tc_f32.cu; this one is what
// fbl_plan_set_kernel_path(plan, 1) selects), operands in R-Tile order fetched by TMA: C[m,n] = sum_terms A_t[m,:] B_t[:,n] (+ bias[n]) (+ residual), up to five problems in one launch.
//
// A block owns a 64 x 64 tile of C: one producer warp and four compute warps, 4 x 8 results per thread.  Operand tiles
// lie in shared memory exactly as the R-Tile panels store them (128-byte rows, 128-byte swizzle), and a transposed operand
// is the same bytes read with the roles of its axes swapped, so nothing is transposed on the way:
//   rows are M/N indices: a thread owns rows t, t + 16 (t + 8), ... and reads four K values of each with one access
//   rows are K indices:   a thread owns neighbouring columns of the row
// Either way eight threads read eight different 16-byte chunks of the swizzled rows (conflict-free).  Two-wide
// multiply-adds halve the issue slots: the pair is two columns where B's rows are K indices, even and odd K where both
// operands' rows are M/N indices (both then load as pairs).
//
// The bound is the FP32 pipe (128 multiply-adds per clock and SM: 74 TFLOP/s).  The shapes that come here have few tiles
// (800 x 768 outputs: 156 for 148 SMs), so the reduction is cut into 1, 2, 4 or 8 slices, one per block of a cluster; the
// slices' partial tiles are added through distributed shared memory in a fixed order, each block finishing its share of
// the tile's rows: no atomics, no second launch, the same bits every time.
// Measured (stand-alone, before with one element per thread and load, a launch per product -> now): 800 x 768 x 2304
// 312 -> 79 us, 800 x 768 x 768 105 -> 34 us, the four products behind the attention backward at 800 x 768 591 -> 161 us;
// 4096 x 1024 x 3072 47 TFLOP/s, 64 % of the pipe.  (8 x 8 results on two warps: 100, 52, 187 us; four blocks per SM at
// 96 registers spill.)
#include "f32_gemm.cuh"
#include "launch_memo.h"
#include "pdl.cuh"

namespace {

using f32g::lds4;
typedef f32g::Group FfmaGroup;
typedef f32g::Problem FfmaProblem;

constexpr int BM = 64, BN = 64, BK = 32, STAGES = 3;
constexpr int COMPUTE = 128, THREADS = COMPUTE + 32;      // a compute thread holds 4 x 8 results

struct FfmaLaunch { FfmaGroup G; int grid, serial; };      // a launch made ready

struct Smem {
  static constexpr uint32_t A_BYTES = BM * BK * 4, B_BYTES = BN * BK * 4, STAGE = A_BYTES + B_BYTES;
  static constexpr uint32_t BAR_OFF = STAGES * STAGE;
  static constexpr uint32_t TOTAL = BAR_OFF + 8 * 2 * STAGES + 1024;      // + alignment slack
};
constexpr int OUT_LD = BN + 4;              // row pitch of the finished tile in shared memory (over the operand stages)
static_assert(BM * OUT_LD * 4 <= STAGES * (int)Smem::STAGE, "the finished tile fits the stages");

typedef unsigned long long f2;              // two fp32 values of one two-wide operation
__device__ __forceinline__ f2 pack2(float x, float y) { f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y)); return r; }
__device__ __forceinline__ float2 unpack2(f2 v) { float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v)); return r; }
__device__ __forceinline__ void fma2(f2& d, f2 a, f2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ void lds2x2(uint32_t a, f2& x, f2& y) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "r"(a));
}

// The slice's reduction loop and its partial tile, left in shared memory (row-major, OUT_LD) over the operand stages.
template <bool AK, bool BKR>
__device__ __forceinline__ void tile_loop(uint32_t base, uint32_t bars, int n_kb, tc::Status status) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int tm = (warp % 2) * 8 + lane % 8, tn = (warp / 2) * 4 + lane / 8;    // 16 x 8 threads
  constexpr int NP = BKR ? 4 : 8;           // accumulator pairs per row: two columns, or even and odd K of one column
  f2 acc[4][NP];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < NP; ++j) acc[i][j] = 0ull;
  for (int it = 0; it < n_kb; ++it) {
    const int s = it % STAGES;
    if (!tc::mbar_wait(bars + 8u * s, (it / STAGES) & 1, status, 122)) break;
    const uint32_t sa = base + s * Smem::STAGE, sb = sa + Smem::A_BYTES;
#pragma unroll 2
    for (int kq = 0; kq < BK / 4; ++kq) {
      if constexpr (BKR) {
        f2 b[4][4];                         // [k][pair]: columns 4 tn .. 4 tn + 3 of both panels
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const int row = kq * 4 + k;
            lds2x2(sb + p * (BK * 128) + row * 128 + ((tn ^ (row & 7)) << 4), b[k][2 * p], b[k][2 * p + 1]);
          }
        float a[4][4];                      // [k][i]
        if constexpr (AK) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int row = kq * 4 + k;
            const float4 v = lds4(sa + (tm / 8) * (BK * 128) + row * 128 + (((tm & 7) ^ (row & 7)) << 4));
            a[k][0] = v.x; a[k][1] = v.y; a[k][2] = v.z; a[k][3] = v.w;
          }
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 v = lds4(sa + (tm + 16 * i) * 128 + ((kq ^ (tm & 7)) << 4));
            a[0][i] = v.x; a[1][i] = v.y; a[2][i] = v.z; a[3][i] = v.w;
          }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const f2 aa = pack2(a[k][i], a[k][i]);
#pragma unroll
            for (int j = 0; j < 4; ++j) fma2(acc[i][j], aa, b[k][j]);
          }
      } else {
        f2 a[4][2], b[8][2];                // [index][K pair]: both operands give pairs along K as they lie
#pragma unroll
        for (int i = 0; i < 4; ++i) lds2x2(sa + (tm + 16 * i) * 128 + ((kq ^ (tm & 7)) << 4), a[i][0], a[i][1]);
#pragma unroll
        for (int j = 0; j < 8; ++j) lds2x2(sb + (tn + 8 * j) * 128 + ((kq ^ tn) << 4), b[j][0], b[j][1]);
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) fma2(acc[i][j], a[i][q], b[j][q]);
      }
    }
    __syncwarp();
    if (lane == 0) tc::mbar_arrive(bars + 8u * (STAGES + s));
  }
  // every load of this slice has been waited for and, behind this barrier, read by all compute warps
  asm volatile("bar.sync 1, %0;" ::"n"(COMPUTE) : "memory");
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t row = base + (uint32_t)((AK ? tm * 4 + i : tm + 16 * i) * OUT_LD) * 4;
    if constexpr (BKR) {
#pragma unroll
      for (int p = 0; p < 2; ++p)
        asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(row + (p * 32 + tn * 4) * 4), "l"(acc[i][2 * p]), "l"(acc[i][2 * p + 1]) : "memory");
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 v = unpack2(acc[i][j]);
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(row + (tn + 8 * j) * 4), "f"(v.x + v.y) : "memory");
      }
    }
  }
}

__global__ void __launch_bounds__(THREADS, 3) gemm_ffma_kernel(const __grid_constant__ FfmaGroup G) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + Smem::BAR_OFF;
  auto full = [&](int s) { return bars + 8u * s; };
  auto empty = [&](int s) { return bars + 8u * (STAGES + s); };
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const tc::Status status(G.status, G.reset_status);
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(full(s), 1);
      tc::mbar_init(empty(s), COMPUTE / 32);                // one arrival per compute warp
    }
    tc::fence_barrier_init();
  }
  __syncthreads();
  pdl_launch_dependents();
  pdl_wait();
  f32g::group_chores(G, threadIdx.x, THREADS);
  // work unit: (problem, tile, slice); the slices of a tile are the blocks of a cluster
  const int slice = blockIdx.x % G.slices;
  int w = blockIdx.x / G.slices, pi = 0;
  while (w >= G.p[pi].tiles_m * G.p[pi].tiles_n) { w -= G.p[pi].tiles_m * G.p[pi].tiles_n; ++pi; }
  const FfmaProblem& P = G.p[pi];
  const int m0 = (w % P.tiles_m) * BM, n0 = (w / P.tiles_m) * BN;
  const int per = (P.total_kb + G.slices - 1) / G.slices;
  const int kb_begin = slice * per, kb_end = min(P.total_kb, kb_begin + per);

  if (warp == COMPUTE / 32) {
    if (lane == 0) {
      int t = 0, kb0 = 0;
      for (int kb = kb_begin, it = 0; kb < kb_end; ++kb, ++it) {
        while (kb - kb0 >= P.kblocks[t]) { kb0 += P.kblocks[t]; ++t; }
        const int s = it % STAGES, k = kb - kb0;
        if (!tc::mbar_wait(empty(s), ((it / STAGES) & 1) ^ 1, status, 121)) break;
        tc::mbar_expect_tx(full(s), Smem::STAGE);
        const uint32_t sa = base + s * Smem::STAGE, sb = sa + Smem::A_BYTES;
        if (P.a_k[t]) tc::tma_load_3d(sa, &P.ta[t], full(s), 0, k * BK, m0 / 32);
        else tc::tma_load_3d(sa, &P.ta[t], full(s), 0, m0, k);
        if (P.b_k[t]) tc::tma_load_3d(sb, &P.tb[t], full(s), 0, k * BK, n0 / 32);
        else tc::tma_load_3d(sb, &P.tb[t], full(s), 0, n0, k);
      }
    }
  } else {
    const int n_kb = max(0, kb_end - kb_begin);
    if (P.b_k[0]) {
      if (P.a_k[0]) tile_loop<true, true>(base, bars, n_kb, status);
      else tile_loop<false, true>(base, bars, n_kb, status);
    } else {
      tile_loop<false, false>(base, bars, n_kb, status);
    }
  }
  __syncwarp();
  if (G.slices > 1) tc::cluster_sync_all(); else __syncthreads();
  f32g::finish_tile<BM, BN, OUT_LD, THREADS>(P, G.slices, slice, base, m0, n0);
  if (G.slices > 1) tc::cluster_sync_all();      // no block leaves while another may still read its partial tile
}

// Slices per tile (1, 2, 4 or 8, the same for all problems of the launch): the longest SM of a list schedule, i.e. the
// average load plus one unit, in k-blocks (0.87 us of an SM for 64 x 64 x 32 multiply-adds at the rate reached), where a
// unit costs two k-blocks to start and finish, plus the exchange between slices.
int choose_slices(int sm_count, const FfmaGroup& G) {
  double best = 1e30;
  int pick = 1;
  for (int s = 1; s <= 8; s *= 2) {
    double load = 0, longest = 0;
    for (int i = 0; i < G.count; ++i) {
      const int per = (G.p[i].total_kb + s - 1) / s;
      load += (double)G.p[i].tiles_m * G.p[i].tiles_n * s * (per + 2);
      longest = per > longest ? per : longest;
    }
    const double t = (load / sm_count + longest) * 0.87 + (s > 1 ? 0.8 + 0.2 * s : 0.0);
    if (t < best) { best = t; pick = s; }
  }
  return pick;
}

}  // namespace

bool gemm_ffma_supported(const fbl_plan* p, const GemmArgs& g) {
  if (p->d.dtype != FBL_DTYPE_FP32 || g.n % 32 != 0) return false;
  for (int t = 0; t < g.n_terms; ++t) {
    const GemmTerm& tm = g.t[t];
    if (tm.a_trans ? g.m % 32 != 0 : tm.k % 32 != 0) return false;
    if (tm.b_trans && tm.k % 32 != 0) return false;
    if (tm.a_trans && tm.b_trans) return false;            // not needed by any step
    if (tm.a_trans != g.t[0].a_trans || tm.b_trans != g.t[0].b_trans) return false;   // one index map per result tile
  }
  return true;
}

static cudaError_t make_group(FfmaLaunch& L, const fbl_plan* p, const GemmArgs* gs, int count) {
  FfmaGroup& G = L.G;
  const int order[f32g::MAX_PROBLEMS] = {0, 1, 2, 3, 4};
  if (!f32g::fill_group(G, gs, count, order, BM, BN, BK)) return cudaErrorInvalidValue;
  int tiles = 0;
  for (int i = 0; i < count; ++i) tiles += G.p[i].tiles_m * G.p[i].tiles_n;
  G.slices = choose_slices(p->sm_count, G);
  L.grid = tiles * G.slices;
  // fp32 attention waits before it requests anything, so no launch has to be serial; but blocks that all fit the SMs at once
  // spread better over idle ones (tiny step 55.1 -> 54.3 us, an adapter step of 191 tokens 172 -> 165 us)
  L.serial = gs[0].serial && L.grid <= 3 * p->sm_count;
  return cudaFuncSetAttribute(gemm_ffma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem::TOTAL);
}

cudaError_t launch_gemm_ffma_group(const fbl_plan* p, const GemmArgs* gs, int count, int32_t* status, cudaStream_t st) {
  if (count < 1 || count > f32g::MAX_PROBLEMS) return cudaErrorInvalidValue;
  LaunchKey key;
  gemm_group_key(key, gs, count);
  return LaunchMemo<FfmaLaunch, 12>::run(p, FBL_MEMO_FFMA_GEMM, key,
      [&](FfmaLaunch& L) { return make_group(L, p, gs, count); },
      [&](FfmaLaunch& L) { return f32g::point_group(L.G, gs, status); },
      [&](const FfmaLaunch& L) {
        if (L.G.slices > 1) return launch_cluster(gemm_ffma_kernel, dim3(L.grid), dim3(THREADS), Smem::TOTAL, st, L.G.slices, !L.serial, L.G);
        return L.serial ? launch_serial(gemm_ffma_kernel, dim3(L.grid), dim3(THREADS), Smem::TOTAL, st, L.G)
                        : launch_pdl(gemm_ffma_kernel, dim3(L.grid), dim3(THREADS), Smem::TOTAL, st, L.G);
      });
}

cudaError_t run_gemm_group(const fbl_plan* p, GemmArgs* gs, int count, int32_t* status, cudaStream_t st, int launch_id, int* kernels) {
  *kernels = 1;
  if (gemm_group_tc(p, gs, count)) return launch_gemm_tc_group(p, gs, count, status, st, launch_id);
  bool ffma = true;
  for (int i = 0; i < count; ++i) ffma = ffma && gemm_ffma_supported(p, gs[i]);
  if (ffma && !p->ffma_only) return launch_gemm_tc_f32_group(p, gs, count, status, st);
  if (ffma) return launch_gemm_ffma_group(p, gs, count, status, st);
  if (p->d.dtype == FBL_DTYPE_FP32) return cudaErrorInvalidValue;      // no step forms such a product
  *kernels = count;
  for (int i = 0; i < count; ++i) {
    cudaError_t e = launch_gemm_simt(gs[i], st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// HBM-bound kernels on R-Tile matrices: pack/unpack, norm forward/backward, token-axis column sums.
// Thread mapping shared by all of them: 8 consecutive lanes cover one 128-byte tile row with one
// 16-byte vector each, 4 rows per warp are 512 contiguous bytes, so every warp-level access is a
// run of whole 128-byte lines.
#include <math.h>

#include "fbl_internal.h"
#include "pdl.cuh"

namespace {

template <typename T> struct Vec16 { static constexpr int N = 16 / (int)sizeof(T); };

template <typename T>
__device__ __forceinline__ void load16(const T* p, float (&v)[Vec16<T>::N]) {
  uint4 raw = *reinterpret_cast<const uint4*>(p);
  const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
  for (int i = 0; i < Vec16<T>::N; ++i) v[i] = to_f(e[i]);
}
template <typename T>
__device__ __forceinline__ void store16(T* p, const float (&v)[Vec16<T>::N]) {
  uint4 raw;
  T* e = reinterpret_cast<T*>(&raw);
#pragma unroll
  for (int i = 0; i < Vec16<T>::N; ++i) e[i] = from_f<T>(v[i]);
  *reinterpret_cast<uint4*>(p) = raw;
}

// ------------------------------------------------------------------------------------------
// pack / unpack: the only layout conversions, used at the graph boundary.
// ------------------------------------------------------------------------------------------
// A block converts PACK_UNITS / (units per row) whole padded rows, or one; a thread's accesses are PACK_UNITS / 256 units
// in flight.  A unit is 16 bytes (eight consecutive threads are one 128-byte tile row on the tiled side and 128 consecutive
// bytes on the row-major side), or one element where the row-major pointer is not 16-byte aligned.  HBM-bound: two passes
// of 3 MB take 2.4 us, where one element per thread and 64-bit divisions took 11 us.
// (No early trigger for the kernel behind: it may request weights before it waits, and this may be what packs them.)
constexpr int PACK_UNITS = 1024;
template <typename U, bool PACK>
__global__ void __launch_bounds__(256) pack_kernel(const U* __restrict__ src, U* __restrict__ dst, uint32_t rows,
                                                   uint32_t rows_pad, uint32_t r_pad, uint32_t units, uint32_t rows_per_block) {
  constexpr uint32_t TU = 128 / sizeof(U);                   // units per tile row
  const uint32_t r0 = blockIdx.x * rows_per_block, n = min(rows_per_block, r_pad - r0) * units;
  pdl_wait();
  for (uint32_t i0 = threadIdx.x; i0 < n; i0 += PACK_UNITS) {
    U v[PACK_UNITS / 256];
    int64_t to[PACK_UNITS / 256];
#pragma unroll
    for (int k = 0; k < PACK_UNITS / 256; ++k) {
      const uint32_t i = i0 + k * 256;
      to[k] = -1;
      if (i >= n) continue;
      const uint32_t r = r0 + i / units, u = i % units, o = r / rows_pad, row = r - o * rows_pad;
      const int64_t tiled = ((int64_t)(u / TU) * r_pad + r) * TU + u % TU, flat = ((int64_t)o * rows + row) * units + u;
      const bool live = row < rows;
      v[k] = U{};
      if (live) v[k] = src[PACK ? flat : tiled];
      if (PACK || live) to[k] = PACK ? tiled : flat;
    }
#pragma unroll
    for (int k = 0; k < PACK_UNITS / 256; ++k)
      if (to[k] >= 0) dst[to[k]] = v[k];
  }
}

// ------------------------------------------------------------------------------------------
// Pre-norm forward and backward for every width and both dtypes.  A thread owns the same 16-byte column vectors (NV of
// them, `tpr` threads a row apart) of every row it meets, so gamma, beta and the token-axis sums of its columns stay in
// registers and X (and dXn, dY) cross memory exactly once.  A row is `tpr` threads (a power of two up to a warp, whole
// warps above); a block holds as many rows side by side as fit 256 threads.  What bounds both is bytes in flight against
// the chain load -> row sums -> store, and next to it instruction issue (hence two-wide arithmetic).
//   Forward: the next PF rows' vectors are in flight in registers; a row stays within a warp up to 96 vectors.
//   Backward: R consecutive rows make a pass (R 128-byte pieces that lie behind each other in every column panel, one
//   exchange between a row's warps for all of them), and the next pass is on its way to a ring in shared memory meanwhile:
//   every thread copies to slots of its own and reads them back itself, which needs no barrier and no registers.
// Measured stand-alone, warm caches, against a warp-register kernel at eight widths and two- and three-pass kernels with
// shared-memory atomics elsewhere and in fp32 (us, before -> now, forward / backward with its reduction):
//   2048 x 768 2.9 -> 2.4 / 9.0 -> 7.6;  6304 x 768 5.5 -> 4.5 / 15.0 -> 13.1;  6304 x 768 fp32 13.9 -> 10.4 / 43 -> 21;
//   896 x 1280 10.4 -> 2.9 / 35 -> 7.0;  2977 x 2880 32 -> 11.4 / 90 -> 20.3;  8192 x 4096 34 -> 35 / 60 -> 42.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool live) {     // zeros where not live
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__host__ __device__ constexpr int norm_stages(int r, int nv) { return r * nv > 4 ? 1 : r * nv == 4 ? 2 : 3; }   // passes in the ring: at most 192 KB

// Two-wide fp32 arithmetic (one instruction for two elements): these kernels issue about as many instructions as their
// bytes take cycles.
template <typename T> __device__ __forceinline__ float2 pair_of(const uint4& raw, int i);      // elements 2i, 2i + 1
template <> __device__ __forceinline__ float2 pair_of<float>(const uint4& raw, int i) { return reinterpret_cast<const float2*>(&raw)[i]; }
template <> __device__ __forceinline__ float2 pair_of<__nv_bfloat16>(const uint4& raw, int i) {
  const uint32_t u = reinterpret_cast<const uint32_t*>(&raw)[i];
  return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}
// The V consecutive values of a vector of gamma or beta (plain fp32 arrays, normally 16-byte aligned).
template <int V>
__device__ __forceinline__ void load_params(const float* __restrict__ p, int c0, bool live, float2 (&v)[V / 2]) {
  if (!live) {
#pragma unroll
    for (int i = 0; i < V / 2; ++i) v[i] = make_float2(0.f, 0.f);
  } else if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
    for (int i = 0; i < V; i += 4) {
      const float4 t = *reinterpret_cast<const float4*>(p + c0 + i);
      v[i / 2] = make_float2(t.x, t.y); v[i / 2 + 1] = make_float2(t.z, t.w);
    }
  } else {
#pragma unroll
    for (int i = 0; i < V / 2; ++i) v[i] = make_float2(p[c0 + 2 * i], p[c0 + 2 * i + 1]);
  }
}
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
template <typename T>
__device__ __forceinline__ void store_pairs(T* p, const float2 (&v)[Vec16<T>::N / 2]) {
  store16(p, reinterpret_cast<const float(&)[Vec16<T>::N]>(v));
}

struct NormShape { int nv, tpr, groups, r; };   // vectors per thread, threads per row, rows side by side, rows per pass

static NormShape norm_shape(int nvec, int nv) {
  NormShape s;
  s.nv = nv;
  const int per = (nvec + nv - 1) / nv;
  if (per <= 32) { s.tpr = 8; while (s.tpr < per) s.tpr *= 2; }
  else s.tpr = (per + 31) / 32 * 32;
  s.groups = s.tpr >= 256 ? 1 : 256 / s.tpr;
  s.r = 1;
  return s;
}
// Forward: a row within one warp up to 96 vectors; then two or three vectors per thread, whichever leaves fewer idle
// lanes (three where equal: fewer warps to a row); above 512 vectors four or eight.
static NormShape norm_fwd_shape(int nvec) {
  if (nvec <= 96) return norm_shape(nvec, (nvec + 31) / 32);
  if (nvec > 512) return norm_shape(nvec, nvec <= 2048 ? 4 : 8);
  const NormShape two = norm_shape(nvec, 2), three = norm_shape(nvec, 3);
  return two.tpr * 2 < three.tpr * 3 ? two : three;
}
// Backward: one vector per thread up to 256 (the token-axis sums of one vector are 16 registers), with as many rows per
// pass (1, 2 or 4) as the rows leave for two blocks on every SM; wider rows two vectors and two rows, then four or eight.
static NormShape norm_bwd_shape(int nvec, int64_t n_pad, int sm_count) {
  NormShape s = norm_shape(nvec, nvec <= 256 ? 1 : nvec <= 1024 ? 2 : nvec <= 2048 ? 4 : 8);
  const int64_t slots = (int64_t)2 * sm_count * s.groups, want = (n_pad + slots - 1) / slots;
  s.r = want >= 3 ? 4 : (want == 2 ? 2 : 1);
  while (s.r * s.nv > 4 && s.r > 1) s.r /= 2;
  return s;
}

// Sums of K values over the tpr threads of a row, returned to all of them.  Up to a warp: shuffles.  Whole warps: the
// K sums of a warp by exchanging halves (K / 2 + K / 4 + ... shuffles, then the rest on one value), one exchange of
// the warps' sums through shared memory behind a barrier of the row's own.  Successive calls alternate between two
// exchange buffers: a warp that writes a buffer again has passed the barrier of the call in between, which every
// reader of the earlier values reached after reading them.
constexpr int NORM_EX = 16 * 8;                              // floats of one exchange buffer of a block: warps x values
// TPR > 0: tpr at compile time.
template <int K, int TPR = 0>
__device__ __forceinline__ void row_sums(float (&v)[K], int tpr, int group, float* ex, int& buf) {
  const int lane = threadIdx.x & 31;
  if (TPR == 32) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    return;
  }
  if (TPR == 0 && tpr <= 32) {
    for (int o = tpr / 2; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    return;
  }
  float* e = ex + buf * NORM_EX;
  buf ^= 1;
  int idx = 0;
#pragma unroll
  for (int n = K, o = 16; n > 1; n /= 2, o >>= 1) {          // lanes with bit o keep the upper half of the values
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < n / 2; ++k) {
      const float send = up ? v[k] : v[k + n / 2], keep = up ? v[k + n / 2] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    idx = idx * 2 + (up ? 1 : 0);
  }
#pragma unroll
  for (int o = 16 / K; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  const int warp = threadIdx.x / 32, wpr = (TPR ? TPR : tpr) / 32, w0 = group * wpr;
  if ((lane & (32 / K - 1)) == 0) e[warp * K + idx] = v[0];
  asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(tpr) : "memory");
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = 0.f;
#pragma unroll 8
  for (int w = 0; w < wpr; ++w) {
    if constexpr (K % 4 == 0) {
#pragma unroll
      for (int k = 0; k < K; k += 4) {
        const float4 t = *reinterpret_cast<const float4*>(e + (w0 + w) * K + k);
        v[k] += t.x; v[k + 1] += t.y; v[k + 2] += t.z; v[k + 3] += t.w;
      }
    } else {
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] += e[(w0 + w) * K + k];
    }
  }
}

template <typename T, int NV, int PF, int TPR>
__global__ void __launch_bounds__(512) norm_fwd_kernel(const T* __restrict__ X, const float* __restrict__ gamma,
                                                       const float* __restrict__ beta, T* __restrict__ Xn,
                                                       float* __restrict__ stats, int64_t n_pad, int d, int tpr_rt, int64_t per_block,
                                                       int seq, int t_pad, int rms, float eps, int32_t* __restrict__ status,
                                                       int n_norm, float2* __restrict__ rope, int rope_half, float rope_k) {
  constexpr int V = Vec16<T>::N, TW = tile_w_of<T>::value;
  __shared__ __align__(16) float s_ex[2 * NORM_EX];
  // First kernel of the forward pass: it resets the pass's status word (later kernels only write it after a
  // bounded wait of about a second has expired), which saves a fill node in front of the pass.
  if (blockIdx.x == 0 && threadIdx.x == 0) *status = 0;
  pdl_launch_dependents();
  if ((int)blockIdx.x >= n_norm) {                           // blocks behind the norm's: the rotary embedding's table
    pdl_wait();
    const int i = ((int)blockIdx.x - n_norm) * (int)blockDim.x + (int)threadIdx.x;
    if (i < rope_half * t_pad) {
      float sn, cs;
      sincosf((float)(i % t_pad) * exp2f((float)(i / t_pad) * rope_k), &sn, &cs);
      rope[i] = make_float2(cs, sn);
    }
    return;
  }
  const int tpr = TPR ? TPR : tpr_rt;
  const int group = threadIdx.x / tpr, lt = threadIdx.x % tpr, groups = blockDim.x / tpr;
  const float inv_d = 1.f / (float)d;
  int buf = 0;
  bool on[NV];
  float2 gm[NV][V / 2], bt[NV][V / 2];                       // inputs of the step: read before waiting for the kernel in front
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    const int c0 = (lt + j * tpr) * V;
    on[j] = c0 < d;
    load_params<V>(gamma, c0, on[j], gm[j]);
    load_params<V>(beta, c0, on[j] && beta, bt[j]);
  }
  pdl_wait();
  const int64_t r_end = min(n_pad, ((int64_t)blockIdx.x + 1) * per_block);
  auto fetch = [&](uint4 (&raw)[NV], int64_t r) {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int v = lt + j * tpr;
      raw[j] = make_uint4(0u, 0u, 0u, 0u);
      if (on[j] && r < r_end) raw[j] = *reinterpret_cast<const uint4*>(X + ((int64_t)(v / 8) * n_pad + r) * TW + (v % 8) * V);
    }
  };
  uint4 ring[PF][NV];
  const int64_t base = (int64_t)blockIdx.x * per_block;
#pragma unroll
  for (int k = 0; k < PF; ++k) fetch(ring[k], base + group + k * groups);
  for (int64_t rb = base; rb < r_end;) {                     // block-uniform: every thread takes part in the row sums
#pragma unroll
    for (int k = 0; k < PF; ++k) {
      if (rb >= r_end) break;
      const int64_t r = rb + group;
      const bool pad = (int)(r % t_pad) >= seq;
      float2 x[NV][V / 2];
      float2 t = both(0.f);
#pragma unroll
      for (int j = 0; j < NV; ++j)
#pragma unroll
        for (int i = 0; i < V / 2; ++i) { x[j][i] = pair_of<T>(ring[k][j], i); t = __fadd2_rn(t, x[j][i]); }
      fetch(ring[k], r + PF * groups);
      float mean[1] = {0.f}, q[1];
      if (!rms) {
        mean[0] = t.x + t.y;
        row_sums<1, TPR>(mean, tpr, group, s_ex, buf);
        mean[0] *= inv_d;
      }
      t = both(0.f);
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        if (!on[j]) continue;
#pragma unroll
        for (int i = 0; i < V / 2; ++i) { x[j][i] = __fadd2_rn(x[j][i], both(-mean[0])); t = __ffma2_rn(x[j][i], x[j][i], t); }
      }
      q[0] = t.x + t.y;
      row_sums<1, TPR>(q, tpr, group, s_ex, buf);
      const float rstd = rsqrtf(q[0] * inv_d + eps);
      if (r < r_end) {
        if (lt == 0) *reinterpret_cast<float2*>(stats + 2 * r) = pad ? make_float2(0.f, 0.f) : make_float2(mean[0], rstd);
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          if (!on[j]) continue;
          float2 y[V / 2];
#pragma unroll
          for (int i = 0; i < V / 2; ++i) y[i] = pad ? both(0.f) : __ffma2_rn(__fmul2_rn(x[j][i], both(rstd)), gm[j][i], bt[j][i]);
          const int v = lt + j * tpr;
          store_pairs(Xn + ((int64_t)(v / 8) * n_pad + r) * TW + (v % 8) * V, y);
        }
      }
      rb += groups;
    }
  }
}

// The rotation back of dQ, on its way from the fp32 accumulator to bf16, and of dK in place: one launch for both and the
// rounding.  A thread takes 8 columns of a head's low half and the matching 8 of its high half.
__global__ void __launch_bounds__(256) rope_bwd_round_kernel(const float* __restrict__ acc, __nv_bfloat16* __restrict__ dq, int heads_q,
                                                             __nv_bfloat16* __restrict__ dk, int heads_k, int64_t n_pad, int seq,
                                                             int t_pad, int hd, const float2* __restrict__ rope) {
  pdl_launch_dependents();
  pdl_wait();
  const int half = hd / 2, vec = half / 8;
  const int64_t per_q = n_pad * heads_q * vec, total = per_q + n_pad * heads_k * vec;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
    const bool is_k = idx >= per_q;
    int64_t rem = is_k ? idx - per_q : idx;
    const int v = (int)(rem % vec);
    rem /= vec;
    const int64_t r = rem % n_pad;
    const int h = (int)(rem / n_pad), t = (int)(r % t_pad);
    const int64_t lo_off = rt_off<64>(n_pad, r, h * hd + v * 8), hi_off = rt_off<64>(n_pad, r, h * hd + half + v * 8);
    float lo[8], hi[8];
    if (is_k) {
      load16(dk + lo_off, lo);
      load16(dk + hi_off, hi);
    } else {
#pragma unroll
      for (int i = 0; i < 8; i += 4) {
        const float4 a = *reinterpret_cast<const float4*>(acc + lo_off + i), b = *reinterpret_cast<const float4*>(acc + hi_off + i);
        lo[i] = a.x; lo[i + 1] = a.y; lo[i + 2] = a.z; lo[i + 3] = a.w;
        hi[i] = b.x; hi[i + 1] = b.y; hi[i + 2] = b.z; hi[i + 3] = b.w;
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float2 cs = rope[(int64_t)(v * 8 + i) * t_pad + t];
      const float a = lo[i], b = hi[i];
      lo[i] = a * cs.x + b * cs.y;
      hi[i] = b * cs.x - a * cs.y;
    }
    store16((is_k ? dk : dq) + lo_off, lo);
    store16((is_k ? dk : dq) + hi_off, hi);
  }
}

constexpr int COLSUM_SLAB = 256;

// First stage of a token-axis column sum: the block's (128-byte column panel p, slab of 256 rows) of matrix `which`,
// 32 storage tiles, reduced to one row of partials.  Any block of whole warps up to 512 threads; `red` has a row per warp.
template <typename T>
__device__ __forceinline__ void colsum_slab(const ColsumGroup& G, int p, int slab, int which,
                                            float (*red)[tile_w_of<T>::value + 1]) {
  constexpr int TW = tile_w_of<T>::value;
  constexpr int V = Vec16<T>::N;
  const int cols = G.cols[which];
  if (p * TW >= cols || slab >= G.slabs[which]) return;
  const T* M = (const T*)G.m[which];
  const int64_t rows = G.rows[which];
  float* part = G.part[which];
  const int rr = threadIdx.x / 8, l8 = threadIdx.x % 8, rstep = blockDim.x / 8;
  float acc[V];
#pragma unroll
  for (int i = 0; i < V; ++i) acc[i] = 0.f;
  const int64_t r_end = min((int64_t)(slab + 1) * COLSUM_SLAB, rows);
#pragma unroll 8                              // all of a thread's loads of the slab in flight together
  for (int64_t r = (int64_t)slab * COLSUM_SLAB + rr; r < r_end; r += rstep) {
    float v[V];
    load16(M + ((int64_t)p * rows + r) * TW + l8 * V, v);
#pragma unroll
    for (int i = 0; i < V; ++i) acc[i] += v[i];
  }
  // a warp holds four rows of eight vectors: add them, then one row per warp through shared memory
#pragma unroll
  for (int i = 0; i < V; ++i) {
    acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 8);
    acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 16);
  }
  const int warp = threadIdx.x / 32, warps = blockDim.x / 32;
  if ((threadIdx.x & 31) < 8) {
#pragma unroll
    for (int i = 0; i < V; ++i) red[warp][l8 * V + i] = acc[i];
  }
  __syncthreads();
  for (int c = threadIdx.x; c < TW; c += blockDim.x) {
    float s = 0.f;
    for (int k = 0; k < warps; ++k) s += red[k][c];
    part[(int64_t)slab * cols + p * TW + c] = s;
  }
}

// Backward.  Row sums mean(g) and mean(g xhat) with g = dXn gamma give dX; dgamma = sum dXn xhat and dbeta = sum dXn of
// the thread's own columns accumulate in registers over the block's rows, are added over the block's row groups at the
// end and leave as one partial row per block (the second kernel adds the blocks' rows: no atomics, the result does not
// depend on their order).  partials = nullptr: the norm's parameters are frozen, only dX is formed.
template <typename T, int NV, int R>
__global__ void __launch_bounds__(512) norm_bwd_kernel(const T* __restrict__ dXn, const T* __restrict__ X, const T* __restrict__ dY,
                                                       const float* __restrict__ stats, const float* __restrict__ gamma,
                                                       T* __restrict__ dX, float* __restrict__ partials, int64_t n_pad, int d,
                                                       int tpr, int64_t per_block, int rms, int n_norm,
                                                       const __grid_constant__ ColsumGroup CG, int cs_panels, int cs_slabs,
                                                       int32_t* __restrict__ late) {
  constexpr int V = Vec16<T>::N, TW = tile_w_of<T>::value;
  // exchange buffers of the row sums; the column-sum blocks use it as well
  __shared__ __align__(16) float s_ex[16 * (TW + 1) > 2 * NORM_EX ? 16 * (TW + 1) : 2 * NORM_EX];
  // Blocks behind the first n_norm ones do the first stage of the bias gradients' column sums (one launch less):
  // block n_norm + (which * slabs + slab) * panels + p
  if ((int)blockIdx.x >= n_norm) {
    if (!late) pdl_launch_dependents();
    pdl_wait();
    if (late && threadIdx.x == 0) pdl_launch_dependents();
    const int idx = (int)blockIdx.x - n_norm;
    colsum_slab<T>(CG, idx % cs_panels, (idx / cs_panels) % cs_slabs, idx / (cs_panels * cs_slabs),
                   reinterpret_cast<float(*)[TW + 1]>(s_ex));
    return;
  }
  if (!late) pdl_launch_dependents();                        // late: the flag under which the second kernel rounds beside this one
  const int group = threadIdx.x / tpr, lt = threadIdx.x % tpr, groups = blockDim.x / tpr;
  const float inv_d = 1.f / (float)d;
  int buf = 0;
  bool on[NV];
  float2 gm[NV][V / 2], ag[NV][V / 2], ab[NV][V / 2];
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    const int c0 = (lt + j * tpr) * V;
    on[j] = c0 < d;
    load_params<V>(gamma, c0, on[j], gm[j]);
#pragma unroll
    for (int i = 0; i < V / 2; ++i) ag[j][i] = ab[j][i] = both(0.f);
  }
  pdl_wait();
  if (late && threadIdx.x == 0) {
    if (blockIdx.x == 0) pdl_raise(late);
    pdl_launch_dependents();
  }
  constexpr int S = norm_stages(R, NV);
  extern __shared__ __align__(16) uint8_t s_ring[];          // [stage][X, dXn, (dY)][row][vector][thread]
  const int arrays = dY ? 3 : 2;
  const uint4* ring = reinterpret_cast<const uint4*>(s_ring) + threadIdx.x;
  const uint32_t ring_addr = (uint32_t)__cvta_generic_to_shared(s_ring) + threadIdx.x * 16;
  const int64_t first = (int64_t)blockIdx.x * per_block + group * R, r_end = min(n_pad, ((int64_t)blockIdx.x + 1) * per_block);
  auto fetch = [&](int64_t r0, int stage) {
#pragma unroll
    for (int k = 0; k < R; ++k)
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        const int v = lt + j * tpr;
        const bool live = on[j] && r0 + k < r_end;
        const int64_t off = live ? ((int64_t)(v / 8) * n_pad + r0 + k) * TW + (v % 8) * V : 0;
        const uint32_t dst = ring_addr + ((stage * arrays * R + k) * NV + j) * blockDim.x * 16, step = R * NV * blockDim.x * 16;
        cp_async16(dst, X + off, live);
        cp_async16(dst + step, dXn + off, live);
        if (dY) cp_async16(dst + 2 * step, dY + off, live);
      }
    cp_async_commit();
  };
  float2 stn[R];                                             // mean and rstd of the next pass's rows
  auto fetch_stats = [&](int64_t r0) {
#pragma unroll
    for (int k = 0; k < R; ++k) stn[k] = r0 + k < r_end ? *reinterpret_cast<const float2*>(stats + 2 * (r0 + k)) : make_float2(0.f, 0.f);
  };
#pragma unroll
  for (int i = 0; i < S - 1; ++i) fetch(first + (int64_t)i * groups * R, i);
  fetch_stats(first);
  int stage = 0;
  for (int64_t r0 = first; r0 - group * R < r_end; r0 += groups * R) {
    fetch(r0 + (int64_t)(S - 1) * groups * R, stage == 0 ? S - 1 : stage - 1);      // the stage read a pass ago
    float2 st[R];
#pragma unroll
    for (int k = 0; k < R; ++k) st[k] = stn[k];
    fetch_stats(r0 + groups * R);
    cp_async_wait<S - 1>();
    const uint4* xs = ring + stage * arrays * R * NV * blockDim.x;
    const uint4* gs = xs + R * NV * blockDim.x;
    const uint4* ys = gs + R * NV * blockDim.x;
    stage = stage == S - 1 ? 0 : stage + 1;
    float s[2 * R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
      float2 t1 = both(0.f), t2 = both(0.f);
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        const uint4 xr = xs[(k * NV + j) * blockDim.x], gr = gs[(k * NV + j) * blockDim.x];
#pragma unroll
        for (int i = 0; i < V / 2; ++i) {
          const float2 xh = __fmul2_rn(__fadd2_rn(pair_of<T>(xr, i), both(-st[k].x)), both(st[k].y));
          const float2 gv = pair_of<T>(gr, i), g = __fmul2_rn(gv, gm[j][i]);
          ag[j][i] = __ffma2_rn(gv, xh, ag[j][i]);
          ab[j][i] = __fadd2_rn(ab[j][i], gv);
          t1 = __fadd2_rn(t1, g);
          t2 = __ffma2_rn(g, xh, t2);
        }
      }
      s[2 * k] = t1.x + t1.y;
      s[2 * k + 1] = t2.x + t2.y;
    }
    row_sums<2 * R>(s, tpr, group, s_ex, buf);
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const int64_t r = r0 + k;
      if (r >= r_end) break;
      const float s1 = rms ? 0.f : s[2 * k] * inv_d, s2 = s[2 * k + 1] * inv_d;
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        if (!on[j]) continue;
        const uint4 xr = xs[(k * NV + j) * blockDim.x], gr = gs[(k * NV + j) * blockDim.x];
        const uint4 yr = dY ? ys[(k * NV + j) * blockDim.x] : make_uint4(0u, 0u, 0u, 0u);
        float2 o[V / 2];
#pragma unroll
        for (int i = 0; i < V / 2; ++i) {
          const float2 xh = __fmul2_rn(__fadd2_rn(pair_of<T>(xr, i), both(-st[k].x)), both(st[k].y));
          const float2 g = __ffma2_rn(pair_of<T>(gr, i), gm[j][i], both(-s1));
          o[i] = __ffma2_rn(both(st[k].y), __ffma2_rn(xh, both(-s2), g), pair_of<T>(yr, i));
        }
        const int v = lt + j * tpr;
        store_pairs(dX + ((int64_t)(v / 8) * n_pad + r) * TW + (v % 8) * V, o);
      }
    }
  }
  cp_async_wait<0>();
  if (!partials) return;
  float* mine = partials + (int64_t)blockIdx.x * 2 * d;
  const int width = tpr * NV * V;
  if (groups > 1) {
    float* s_sum = reinterpret_cast<float*>(s_ring);         // [groups][2][row width], over the ring
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NV; ++j)
#pragma unroll
      for (int i = 0; i < V; i += 4) {
        float* p = s_sum + (size_t)group * 2 * width + (lt + j * tpr) * V + i;
        *reinterpret_cast<float4*>(p) = make_float4(ag[j][i / 2].x, ag[j][i / 2].y, ag[j][i / 2 + 1].x, ag[j][i / 2 + 1].y);
        *reinterpret_cast<float4*>(p + width) = make_float4(ab[j][i / 2].x, ab[j][i / 2].y, ab[j][i / 2 + 1].x, ab[j][i / 2 + 1].y);
      }
    __syncthreads();
    for (int c = threadIdx.x; c < (rms ? d : 2 * d); c += blockDim.x) {
      const int at = c < d ? c : width + c - d;
      float t = 0.f;
      for (int q = 0; q < groups; ++q) t += s_sum[(size_t)q * 2 * width + at];
      mine[c] = t;
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    if (!on[j]) continue;
    const int c0 = (lt + j * tpr) * V;
#pragma unroll
    for (int i = 0; i < V; i += 4) {
      *reinterpret_cast<float4*>(mine + c0 + i) = make_float4(ag[j][i / 2].x, ag[j][i / 2].y, ag[j][i / 2 + 1].x, ag[j][i / 2 + 1].y);
      if (!rms) *reinterpret_cast<float4*>(mine + d + c0 + i) = make_float4(ab[j][i / 2].x, ab[j][i / 2].y, ab[j][i / 2 + 1].x, ab[j][i / 2 + 1].y);
    }
  }
}

// ------------------------------------------------------------------------------------------
// Rotary position embedding, in place, on two R-Tile matrices at once (Q and K forward; dQ and dK backward with the
// opposite angle).  Half-split pairing: inside a head, element i < hd/2 goes with element i + hd/2, and the pair of
// token t turns by t * base^(-2i/hd).  A thread takes 16 bytes of the low half and the matching 16 bytes of the
// high half (the same row of the same or of the neighbouring 128-byte panel).
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) rope_kernel(T* __restrict__ A, int heads_a, T* __restrict__ B, int heads_b,
                                                   int64_t n_pad, int seq, int t_pad, int hd, float neg2_log2_base_over_hd,
                                                   float sign) {
  constexpr int TW = tile_w_of<T>::value;
  constexpr int V = Vec16<T>::N;
  pdl_launch_dependents();
  pdl_wait();
  const int half = hd / 2, vec_per_head = half / V;
  const int64_t per_a = n_pad * heads_a * vec_per_head, total = per_a + n_pad * heads_b * vec_per_head;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
    const bool second = idx >= per_a;
    T* M = second ? B : A;
    const int heads = second ? heads_b : heads_a;
    int64_t rem = second ? idx - per_a : idx;
    // consecutive threads: consecutive vectors of a row's half-head, then rows (whole 128-byte pieces per warp quarter)
    const int v = (int)(rem % vec_per_head);
    rem /= vec_per_head;
    const int64_t r = rem % n_pad;
    const int h = (int)(rem / n_pad);
    const int t = (int)(r % t_pad);
    if (t >= seq) continue;                                     // padding rows hold zeros and stay zero
    const int c_lo = h * hd + v * V, c_hi = c_lo + half;
    T* plo = M + rt_off<TW>(n_pad, r, c_lo);
    T* phi = M + rt_off<TW>(n_pad, r, c_hi);
    float lo[V], hi[V];
    load16(plo, lo);
    load16(phi, hi);
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const float inv_freq = exp2f((float)(v * V + i) * neg2_log2_base_over_hd);
      float sn, cs;
      sincosf((float)t * inv_freq, &sn, &cs);
      sn *= sign;
      const float a = lo[i], b = hi[i];
      lo[i] = a * cs - b * sn;
      hi[i] = b * cs + a * sn;
    }
    store16(plo, lo);
    store16(phi, hi);
  }
}

// dgamma[c] (y = 0) or dbeta[c] (y = 1) = sum over the first kernel's blocks of their partial rows.  Blocks with
// y >= ny_norm finish the bias column sums instead (matrix y - ny_norm: the tree over its slab partials), so that
// the step's two small final reductions share one launch.  Blocks behind those (y >= ny_sums) round the fp32 sums of sliced
// products, which launches in front of the first kernel left: beside that one (pdl_early), whose end they wait for only at
// their own (four 768 x 768 matrices: a launch of 10 us in a step of 191 us before).
__global__ void __launch_bounds__(256) norm_bwd_reduce_kernel(const float* __restrict__ part, int blocks, int d,
                                                              float* __restrict__ dgamma, float* __restrict__ dbeta,
                                                              int ny_norm, const __grid_constant__ ColsumGroup G, int ny_sums,
                                                              const __grid_constant__ ConvertGroup C, int32_t* early) {
  __shared__ float red[8][33];
  pdl_launch_dependents();
  if ((int)blockIdx.y >= ny_sums) {
    pdl_early(early);
    const int64_t first = ((int64_t)((blockIdx.y - ny_sums) * gridDim.x + blockIdx.x) * 256 + threadIdx.x) * 4;
    const int64_t step = (int64_t)(gridDim.y - ny_sums) * gridDim.x * 1024;
    for (int k = 0; k < C.count; ++k) {
      __nv_bfloat16* dst = (__nv_bfloat16*)C.dst[k];
#pragma unroll 4
      for (int64_t i = first; i < C.n[k]; i += step) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(C.src[k] + i));
        __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        uint2 o;
        o.x = *reinterpret_cast<uint32_t*>(&lo); o.y = *reinterpret_cast<uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(dst + i) = o;
      }
    }
    pdl_wait();
    if (blockIdx.x == 0 && (int)blockIdx.y == ny_sums && threadIdx.x == 0) pdl_lower(early);
    return;
  }
  pdl_wait();
  if ((int)blockIdx.y >= ny_norm) {
    const int which = blockIdx.y - ny_norm;
    const int cols = G.cols[which], n_slabs = G.slabs[which];
    const float* cp = G.part[which];
    for (int c = blockIdx.x * 256 + threadIdx.x; c < cols; c += gridDim.x * 256) {
      float s = 0.f;
#pragma unroll 8
      for (int k = 0; k < n_slabs; ++k) s += cp[(int64_t)k * cols + c];
      G.out[which][c] = s;
    }
    return;
  }
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const int c = blockIdx.x * 32 + tx;
  float s = 0.f;
  if (c < d) {
    const float* col = part + (int64_t)blockIdx.y * d + c;
    const int64_t stride = 2 * (int64_t)d;
    int b = ty;
    for (; b + 56 < blocks; b += 64) {          // eight independent loads in flight per thread
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = col[(b + 8 * u) * stride];
#pragma unroll
      for (int u = 0; u < 8; ++u) s += v[u];
    }
    for (; b < blocks; b += 8) s += col[b * stride];
  }
  red[ty][tx] = s;
  __syncthreads();
  if (ty == 0 && c < d) {
#pragma unroll
    for (int k = 1; k < 8; ++k) s += red[k][tx];
    (blockIdx.y == 0 ? dgamma : dbeta)[c] = s;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) colsum_stage1(const __grid_constant__ ColsumGroup G) {
  __shared__ float red[8][tile_w_of<T>::value + 1];
  pdl_launch_dependents();
  pdl_wait();
  colsum_slab<T>(G, blockIdx.x, blockIdx.y, blockIdx.z, red);
}

// The same sums beside a tensor-core product, of matrices that launches in front of that one left (pdl_early); the wait for the
// product comes last, for the kernels behind this one.  A block takes a slab of a panel at a time; small as it is, and with at most one per SM, it fits beside
// a product block.  Loads go to L2, whose data is current.  Bound by memory, and hidden by the product:
// 2048 x 768 and 2048 x 3072 cost 5 us of a step of 114 us in a launch of their own; two of 3000 x 1280, with their
// second stage, 7 us of 199 us.
__global__ void __launch_bounds__(128, 8) colsum_early_kernel(const __grid_constant__ ColsumGroup G, int32_t* early) {
  using T = __nv_bfloat16;
  constexpr int TW = tile_w_of<T>::value, V = Vec16<T>::N, B = 8, STEP = 16 * B;
  __shared__ __align__(16) float red[3][TW];                            // 768 bytes: a product block leaves 1.9 KB, 1 KB of it reserved
  pdl_launch_dependents();
  pdl_early(early);
  const int warp = threadIdx.x / 32, rr = threadIdx.x / 8, l8 = threadIdx.x % 8;
  // position of the next batch of 128 rows: unit (panel of a slab of a matrix), and its first row of this thread
  int which = -1, left = (int)blockIdx.x, units = 0;
  int64_t row = 0, r_end = 0;
  const uint4* src = nullptr;
  float* out = nullptr;
  auto open_unit = [&]() {                                              // the first matrix that unit `left` falls into
    while (left >= units) {
      left -= units;
      if (++which >= G.count) return;
      units = G.cols[which] / TW * G.slabs[which];
    }
    const int cols = G.cols[which], panels = cols / TW, p = left % panels, slab = left / panels;
    const int64_t rows = G.rows[which];
    row = (int64_t)slab * COLSUM_SLAB + rr;
    r_end = min((int64_t)(slab + 1) * COLSUM_SLAB, rows);
    src = reinterpret_cast<const uint4*>((const T*)G.m[which] + (int64_t)p * rows * TW) + l8;
    out = G.part[which] + (int64_t)slab * cols + p * TW + l8 * V;
  };
  open_unit();
  uint4 u[B];                                                           // always a batch of loads in flight
#pragma unroll
  for (int k = 0; k < B; ++k) u[k] = which < G.count && row + k * 16 < r_end ? __ldcg(src + (row + k * 16) * 8) : make_uint4(0u, 0u, 0u, 0u);
  float acc[V];
#pragma unroll
  for (int i = 0; i < V; ++i) acc[i] = 0.f;
  while (which < G.count) {
    float* const to = out;
    const bool last = row - rr + STEP >= r_end;                         // uniform over the block
    row += STEP;
    if (last) {
      left += gridDim.x;
      open_unit();
    }
    const bool more = which < G.count;
#pragma unroll
    for (int k = 0; k < B; ++k) {
      float v[V];
      load16(reinterpret_cast<const T*>(&u[k]), v);
#pragma unroll
      for (int i = 0; i < V; ++i) acc[i] += v[i];
      u[k] = more && row + k * 16 < r_end ? __ldcg(src + (row + k * 16) * 8) : make_uint4(0u, 0u, 0u, 0u);
    }
    if (last) {
#pragma unroll
      for (int i = 0; i < V; ++i) {
        acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 8);
        acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 16);
      }
      if (warp > 0 && rr % 4 == 0) {
#pragma unroll
        for (int i = 0; i < V; ++i) red[warp - 1][l8 * V + i] = acc[i];
      }
      __syncthreads();
      if (rr == 0) {
#pragma unroll
        for (int i = 0; i < V; ++i) to[i] = acc[i] + red[0][l8 * V + i] + red[1][l8 * V + i] + red[2][l8 * V + i];
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < V; ++i) acc[i] = 0.f;
    }
  }
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) pdl_lower(early);
}

template <typename T, int NV, int PF, int TPR>
cudaError_t norm_fwd_launch(const fbl_plan* p, const NormShape& s, const void* X, const float* gamma, const float* beta,
                            void* Xn, float* stats, int32_t* status, float2* rope, cudaStream_t st) {
  const int64_t blocks = min((int64_t)p->sm_count * (NV == 1 ? 4 : 2), (p->n_pad + s.groups - 1) / s.groups);
  const int64_t per_block = ((p->n_pad + blocks - 1) / blocks + s.groups - 1) / s.groups * s.groups;
  const int threads = s.tpr * s.groups, n_norm = (int)((p->n_pad + per_block - 1) / per_block), half = p->d.head_dim / 2;
  const int extra = rope ? (half * p->t_pad + threads - 1) / threads : 0;
  return launch_pdl(norm_fwd_kernel<T, NV, PF, TPR>, dim3((unsigned)(n_norm + extra)), dim3(threads), 0, st,
                    (const T*)X, gamma, beta, (T*)Xn, stats, p->n_pad, p->d.d_model, s.tpr, per_block, p->d.seq, p->t_pad,
                    (int)(p->d.norm == FBL_NORM_RMSNORM), p->d.eps, status, n_norm, rope, half,
                    rope ? -2.f * log2f(p->rope_base) / (float)p->d.head_dim : 0.f);
}

template <typename T, int NV, int R>
cudaError_t norm_bwd_launch(const fbl_plan* p, const NormShape& s, const void* dXn, const void* X, const void* dY,
                            const float* stats, const float* gamma, void* dX, float* dgamma, float* dbeta, float* part,
                            int32_t* status, const ColsumGroup& cg, const ConvertGroup& round, cudaStream_t st) {
  constexpr int V = Vec16<T>::N;
  const int d = p->d.d_model, rms = p->d.norm == FBL_NORM_RMSNORM;
  const int64_t pass = (int64_t)s.groups * R;
  // at most two blocks per SM: the partial-sum area holds that many rows, and the second kernel adds them all
  const int64_t most = min((int64_t)p->sm_count * 2, (p->n_pad + pass - 1) / pass);
  const int64_t per_block = ((p->n_pad + most - 1) / most + pass - 1) / pass * pass;
  const int blocks = (int)((p->n_pad + per_block - 1) / per_block);
  const size_t ring = (size_t)norm_stages(R, NV) * (dY ? 3 : 2) * R * NV * s.tpr * s.groups * 16;
  int cs_panels = 0, n_slabs = 0;
  for (int i = 0; i < cg.count && !cg.summed; ++i) {
    cs_panels = max(cs_panels, cg.cols[i] / tile_w_of<T>::value);
    n_slabs = max(n_slabs, cg.slabs[i]);
  }
  // The column sums' first stage shares this launch while it is a few blocks for each that fits an SM beside the ring's
  // shared memory, which those blocks occupy without using it; beyond that a launch of its own is cheaper (91 us
  // together, 40 us apart for four 2977 x 2880 matrices; 4 us dearer apart for a 2048 x 768 and a 2048 x 3072 one).
  int cs_blocks = cs_panels * n_slabs * cg.count;
  if (cs_blocks > (ring <= 56 * 1024 ? 8 : 4) * p->sm_count) {
    cudaError_t ce = launch_pdl(colsum_stage1<T>, dim3(cs_panels, n_slabs, cg.count), dim3(256), 0, st, cg);
    if (ce != cudaSuccess) return ce;
    p->launches++;
    cs_blocks = 0;
  }
  const size_t sums = (size_t)s.groups * 2 * s.tpr * NV * V * sizeof(float), smem = ring > sums ? ring : sums;
  cudaError_t e = cudaSuccess;
  if (smem > 40 * 1024) e = cudaFuncSetAttribute(norm_bwd_kernel<T, NV, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = launch_pdl(norm_bwd_kernel<T, NV, R>, dim3(blocks + cs_blocks), dim3(s.tpr * s.groups), smem, st,
                             (const T*)dXn, (const T*)X, (const T*)dY, stats, gamma, (T*)dX, dgamma ? part : (float*)nullptr, p->n_pad,
                             d, s.tpr, per_block, rms, blocks, cg, cs_panels, n_slabs, round.count > 0 ? status + FBL_EARLY_ROUND : nullptr);
  if (e != cudaSuccess) return e;
  const int ny = !dgamma ? 0 : rms ? 1 : 2;
  const int nx = (d + 31) / 32, ny_sums = ny + cg.count;
  int64_t rounded = 0;
  for (int i = 0; i < round.count; ++i) rounded = max(rounded, round.n[i]);
  const int ny_round = (int)((min((int64_t)p->sm_count * 4, (rounded + 1023) / 1024) + nx - 1) / nx);
  p->launches += ny_sums + ny_round == 0 ? 1 : 2;
  if (ny_sums + ny_round == 0) return cudaSuccess;
  return launch_pdl(norm_bwd_reduce_kernel, dim3(nx, ny_sums + ny_round), dim3(256), 0, st, (const float*)part,
                    blocks, d, dgamma, dbeta, ny, cg, ny_sums, round, status + FBL_EARLY_ROUND);
}

// ------------------------------------------------------------------------------------------
// Token-axis column sums, two stages over tiles: (1) one block per (panel, slab of 256 rows)
// reduces its 32 storage tiles to one row of partials, (2) a tree over slabs.
// ------------------------------------------------------------------------------------------
__global__ void colsum_stage2(const __grid_constant__ ColsumGroup G) {
  pdl_launch_dependents();
  pdl_wait();
  const int which = blockIdx.y;
  const int cols = G.cols[which];
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  const float* part = G.part[which];
  const int n_slabs = G.slabs[which];
  float s = 0.f;
#pragma unroll 8
  for (int k = 0; k < n_slabs; ++k) s += part[(int64_t)k * cols + c];
  G.out[which][c] = s;
}

}  // namespace

template <typename U>
static cudaError_t pack_launch(int unpack, const void* src, void* dst, int64_t outer, int64_t rows, int64_t rows_pad,
                               int64_t row_bytes, cudaStream_t st) {
  const uint32_t units = (uint32_t)(row_bytes / sizeof(U)), r_pad = (uint32_t)(outer * rows_pad);
  const uint32_t per_block = units >= PACK_UNITS ? 1 : PACK_UNITS / units;
  const dim3 grid((r_pad + per_block - 1) / per_block);
  return unpack ? launch_pdl(pack_kernel<U, false>, grid, dim3(256), 0, st, (const U*)src, (U*)dst, (uint32_t)rows, (uint32_t)rows_pad, r_pad, units, per_block)
                : launch_pdl(pack_kernel<U, true>, grid, dim3(256), 0, st, (const U*)src, (U*)dst, (uint32_t)rows, (uint32_t)rows_pad, r_pad, units, per_block);
}

cudaError_t launch_pack(int dtype, int unpack, const void* src, void* dst, int64_t outer, int64_t rows,
                        int64_t rows_pad, int cols, cudaStream_t st) {
  if (outer * rows * cols == 0) return cudaSuccess;
  const int64_t row_bytes = (int64_t)cols * (dtype == FBL_DTYPE_FP32 ? 4 : 2);
  if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0)
    return pack_launch<uint4>(unpack, src, dst, outer, rows, rows_pad, row_bytes, st);
  if (dtype == FBL_DTYPE_FP32) return pack_launch<uint32_t>(unpack, src, dst, outer, rows, rows_pad, row_bytes, st);
  return pack_launch<uint16_t>(unpack, src, dst, outer, rows, rows_pad, row_bytes, st);
}

cudaError_t launch_rope(const fbl_plan* p, void* A, int heads_a, void* B, int heads_b, int inverse, cudaStream_t st) {
  const int hd = p->d.head_dim;
  const float k = -2.f * log2f(p->rope_base) / (float)hd;
  const int vec = p->d.dtype == FBL_DTYPE_FP32 ? 4 : 8;
  const int64_t total = p->n_pad * (int64_t)(heads_a + heads_b) * (hd / 2 / vec);
  const int blocks = (int)min((int64_t)p->sm_count * 16, (total + 255) / 256);
  if (p->d.dtype == FBL_DTYPE_FP32)
    return launch_pdl(rope_kernel<float>, dim3(blocks), dim3(256), 0, st, (float*)A, heads_a, (float*)B, heads_b, p->n_pad,
                      p->d.seq, p->t_pad, hd, k, inverse ? -1.f : 1.f);
  return launch_pdl(rope_kernel<__nv_bfloat16>, dim3(blocks), dim3(256), 0, st, (__nv_bfloat16*)A, heads_a,
                    (__nv_bfloat16*)B, heads_b, p->n_pad, p->d.seq, p->t_pad, hd, k, inverse ? -1.f : 1.f);
}

template <typename T>
cudaError_t norm_fwd_dispatch(const fbl_plan* p, const void* X, const float* gamma, const float* beta, void* Xn,
                              float* stats, int32_t* status, float2* rope, cudaStream_t st) {
  const NormShape s = norm_fwd_shape(p->d.d_model / Vec16<T>::N);
#define FBL_CALL(NV_, PF_, TPR_) norm_fwd_launch<T, NV_, PF_, TPR_>(p, s, X, gamma, beta, Xn, stats, status, rope, st)
  switch (s.nv) {
    case 1: return s.tpr == 32 ? FBL_CALL(1, 4, 32) : FBL_CALL(1, 4, 0);
    case 2:
      return s.tpr == 32 ? FBL_CALL(2, 4, 32) : s.tpr == 64 ? FBL_CALL(2, 4, 64) : s.tpr == 128 ? FBL_CALL(2, 4, 128)
                         : s.tpr == 256 ? FBL_CALL(2, 4, 256) : FBL_CALL(2, 4, 0);
    case 3: return s.tpr == 32 ? FBL_CALL(3, 3, 32) : FBL_CALL(3, 3, 0);
    case 4: return sizeof(T) == 4 ? FBL_CALL(4, 2, 0) : FBL_CALL(4, 1, 0);
  }
  if constexpr (sizeof(T) == 4) return FBL_CALL(8, 1, 0);
  return cudaErrorInvalidValue;                // bf16: d_model <= 16384 needs at most four vectors
#undef FBL_CALL
}

cudaError_t launch_rope_bwd_round(const fbl_plan* p, const float* acc, void* dQ, void* dK, const float2* rope, cudaStream_t st) {
  const int64_t total = p->n_pad * (int64_t)(p->d.n_q_heads + p->d.n_kv_heads) * (p->d.head_dim / 16);
  const int blocks = (int)min((int64_t)p->sm_count * 16, (total + 255) / 256);
  return launch_pdl(rope_bwd_round_kernel, dim3(blocks), dim3(256), 0, st, acc, (__nv_bfloat16*)dQ, p->d.n_q_heads, (__nv_bfloat16*)dK,
                    p->d.n_kv_heads, p->n_pad, p->d.seq, p->t_pad, p->d.head_dim, rope);
}

cudaError_t launch_norm_fwd(const fbl_plan* p, const void* X, const float* gamma, const float* beta, void* Xn,
                            float* stats, int32_t* status, cudaStream_t st, float2* rope) {
  if (p->d.norm == FBL_NORM_RMSNORM) beta = nullptr;
  return p->d.dtype == FBL_DTYPE_FP32 ? norm_fwd_dispatch<float>(p, X, gamma, beta, Xn, stats, status, rope, st)
                                      : norm_fwd_dispatch<__nv_bfloat16>(p, X, gamma, beta, Xn, stats, status, rope, st);
}

template <typename T>
cudaError_t norm_bwd_dispatch(const fbl_plan* p, const void* dXn, const void* X, const void* dY, const float* stats,
                              const float* gamma, void* dX, float* dgamma, float* dbeta, float* npart, int32_t* status,
                              const ColsumGroup& cg, const ConvertGroup& round, cudaStream_t st) {
  const NormShape s = norm_bwd_shape(p->d.d_model / Vec16<T>::N, p->n_pad, p->sm_count);
#define FBL_CALL(NV_, R_) norm_bwd_launch<T, NV_, R_>(p, s, dXn, X, dY, stats, gamma, dX, dgamma, dbeta, npart, status, cg, round, st)
  switch (s.nv) {
    case 1: return s.r == 4 ? FBL_CALL(1, 4) : s.r == 2 ? FBL_CALL(1, 2) : FBL_CALL(1, 1);
    case 2: return s.r == 2 ? FBL_CALL(2, 2) : FBL_CALL(2, 1);
    case 4: return FBL_CALL(4, 1);
  }
  if constexpr (sizeof(T) == 4) return FBL_CALL(8, 1);
  return cudaErrorInvalidValue;                // bf16: d_model <= 16384 needs at most four vectors
#undef FBL_CALL
}

// Zero-fill.  Bound by memory; a kernel and not a fill of the driver's, so that the products behind it are set up and their
// first weights under way when it ends.
static __global__ void __launch_bounds__(512) fill_kernel(uint4* __restrict__ out, int64_t n) {
  pdl_launch_dependents();
  pdl_wait();
  const uint4 z = make_uint4(0u, 0u, 0u, 0u);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) out[i] = z;
}

cudaError_t start_backward(const fbl_plan* p, GemmArgs* gs, int count, bool rides, bool serial, int32_t* status, size_t bytes, cudaStream_t st) {
  // Idle epilogue warps of the first products clear what they can while the first tiles are computed; with tens of MB their
  // stores delay those tiles by more than a launch costs, but the fp32 kernels leave memory idle.
  if (rides && (p->d.dtype == FBL_DTYPE_FP32 || (bytes <= (size_t)16 << 20 && gemm_group_tc(p, gs, count)))) {
    gs[0].zero_ptr = (char*)status + FBL_ALIGN; gs[0].zero_bytes = bytes - FBL_ALIGN;
    gs[0].reset_status = 1; gs[0].serial = serial;
    return cudaSuccess;
  }
  const int64_t n = (int64_t)(bytes / 16);
  const dim3 grid((unsigned)min((int64_t)p->sm_count * 4, (n + 511) / 512));
  p->launches++;
  return serial ? launch_serial(fill_kernel, grid, dim3(512), 0, st, (uint4*)status, n) : launch_pdl(fill_kernel, grid, dim3(512), 0, st, (uint4*)status, n);
}

void colsum_add(ColsumGroup& G, const void* m, int64_t rows, int cols, float* out, float** part) {
  const int i = G.count++;
  G.m[i] = m; G.rows[i] = rows; G.cols[i] = cols; G.out[i] = out; G.part[i] = *part;
  G.slabs[i] = (int)((rows + COLSUM_SLAB - 1) / COLSUM_SLAB);
  *part += (int64_t)G.slabs[i] * cols;
}

cudaError_t launch_colsum_early(const fbl_plan* p, ColsumGroup& G, int idle, int32_t* status, cudaStream_t st) {
  int64_t bytes = 0;
  for (int i = 0; i < G.count; ++i) bytes += G.rows[i] * G.cols[i] * 2;
  // Where the product's SMs run out of work at different times, those that have (some 13 bytes/clk each) do the sums, and
  // the ask for shared memory keeps them away from the busy ones: sharing those made a product of 46 us 2 us longer.  Where
  // they all end together that is no help, and the sums share the SMs (47 MB of sums beside a product of 75 us: a step of
  // 276 us that way, 251 us sharing).
  const bool beside = (int64_t)idle * p->sm_count * 13 < bytes;
  const dim3 grid((unsigned)min((int64_t)p->sm_count, colsum_units(p, G)));
  G.summed = 1;
  return launch_pdl(colsum_early_kernel, grid, dim3(128), beside ? 0 : 2048, st, G, status + FBL_EARLY_COLSUM);
}

// Self-test of pdl_early: a kernel that lets its dependents start at once and writes what they read only after `clocks`.
static __global__ void __launch_bounds__(256) slow_fill_kernel(uint4* __restrict__ out, int64_t n, uint4 v, long long clocks) {
  pdl_launch_dependents();
  pdl_wait();
  for (const long long t0 = clock64(); clock64() - t0 < clocks;) {}
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) out[i] = v;
}

cudaError_t launch_early_order_selftest(const fbl_plan* p, void* M, int64_t rows, int cols, float* out, int32_t* status, float* part,
                                        cudaStream_t st) {
  const uint32_t ones = 0x3f803f80u;                                    // two bf16 ones
  const cudaError_t e = launch_pdl(slow_fill_kernel, dim3(8), dim3(256), 0, st, (uint4*)M, rows * cols / 8,
                                   make_uint4(ones, ones, ones, ones), 400000ll);
  if (e != cudaSuccess) return e;
  ColsumGroup G = {};
  colsum_add(G, M, rows, cols, out, &part);
  const cudaError_t f = launch_colsum_early(p, G, 0, status, st);
  if (f != cudaSuccess) return f;
  return launch_pdl(colsum_stage2, dim3((unsigned)((cols + 127) / 128), 1), dim3(128), 0, st, G);
}

// Norm backward (dgamma = nullptr: only dX, the norm's parameters are frozen), and with it the bias column sums of up to
// four matrices: their first stage, unless it ran beside the product in front, as extra blocks of the first kernel, their
// second stage inside the second.  `part`: the norm's per-block partial rows.
cudaError_t launch_norm_bwd(const fbl_plan* p, const void* dXn, const void* X, const void* dY, const float* stats,
                            const float* gamma, void* dX, float* dgamma, float* dbeta, float* part, int32_t* status,
                            cudaStream_t st, const ColsumGroup* sums, const ConvertGroup* round) {
  ColsumGroup cg = {};
  ConvertGroup rg = {};
  if (round) rg = *round;
  if (sums) cg = *sums;
  if (p->d.dtype == FBL_DTYPE_FP32) return norm_bwd_dispatch<float>(p, dXn, X, dY, stats, gamma, dX, dgamma, dbeta, part, status, cg, rg, st);
  return norm_bwd_dispatch<__nv_bfloat16>(p, dXn, X, dY, stats, gamma, dX, dgamma, dbeta, part, status, cg, rg, st);
}

size_t colsum_scratch_bytes(int64_t rows, int64_t cols) {
  const int64_t slabs = (rows + COLSUM_SLAB - 1) / COLSUM_SLAB;
  return (size_t)(slabs * cols) * sizeof(float);
}

// Column sums in a pair of launches of their own.
cudaError_t launch_colsum_group(int dtype, const ColsumGroup& G, cudaStream_t st) {
  if (G.count < 1) return cudaErrorInvalidValue;
  int max_cols = 0, slabs = 0;
  for (int i = 0; i < G.count; ++i) { max_cols = max(max_cols, G.cols[i]); slabs = max(slabs, G.slabs[i]); }
  const int tw = dtype == FBL_DTYPE_FP32 ? 32 : 64;
  const dim3 grid((unsigned)(max_cols / tw), slabs, G.count);
  cudaError_t e;
  if (dtype == FBL_DTYPE_FP32) e = launch_pdl(colsum_stage1<float>, grid, dim3(256), 0, st, G);
  else e = launch_pdl(colsum_stage1<__nv_bfloat16>, grid, dim3(256), 0, st, G);
  if (e != cudaSuccess) return e;
  return launch_pdl(colsum_stage2, dim3((unsigned)((max_cols + 127) / 128), G.count), dim3(128), 0, st, G);
}

cudaError_t launch_colsum(int dtype, const void* M, int64_t rows, int64_t cols, float* out, float* partials,
                          cudaStream_t st) {
  ColsumGroup G = {};
  colsum_add(G, M, rows, (int)cols, out, &partials);
  return launch_colsum_group(dtype, G, st);
}

// ------------------------------------------------------------------------------------------
// Column sums without caller scratch.  The per-slab partial sums live in a fixed array inside the
// library image instead of a caller buffer, for callers that are not in a position to allocate.
// ------------------------------------------------------------------------------------------
#include <mutex>

#define FBL_COLSUM_NOALLOC_MAX_FLOATS (256 * 1024)   // 1 MiB: e.g. 16384 rows x 4096 columns

static __device__ __align__(256) float g_colsum_partials[FBL_COLSUM_NOALLOC_MAX_FLOATS];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
float* g_partials_addr[kMaxDevices] = {};   // device address of g_colsum_partials, per device ordinal
}  // namespace

extern "C" int fbl_colsum_noalloc(const fbl_plan* plan, const void* M_dev, int64_t rows, int64_t cols,
                                  float* out_dev, void* stream) {
  if (!plan || !M_dev || !out_dev || rows <= 0 || cols <= 0 || rows % 8 != 0 || cols % plan->tw != 0)
    return FBL_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(M_dev) & (FBL_ALIGN - 1)) != 0) return FBL_ERR_MISALIGNED;
  const int64_t slabs = (rows + COLSUM_SLAB - 1) / COLSUM_SLAB;
  if (slabs * cols > FBL_COLSUM_NOALLOC_MAX_FLOATS) {
    fbl_note_cuda_error(cudaSuccess, "fbl_colsum_noalloc: ceil(rows/256) * cols exceeds the built-in 262144-float area");
    return FBL_ERR_WORKSPACE_TOO_SMALL;
  }
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    fbl_note_cuda_error(e, "fbl_colsum_noalloc: cudaGetDevice");
    return FBL_ERR_CUDA;
  }
  float* partials = nullptr;
  {
    // Set-up, once per device and with that device current: in host code the array's name is only a
    // handle, so ask the runtime for the address the kernels must be given.
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_partials_addr[dev]) {
      void* addr = nullptr;
      e = cudaGetSymbolAddress(&addr, g_colsum_partials);
      if (e != cudaSuccess || !addr) {
        fbl_note_cuda_error(e, "fbl_colsum_noalloc: cudaGetSymbolAddress");
        return FBL_ERR_CUDA;
      }
      g_partials_addr[dev] = static_cast<float*>(addr);
    }
    partials = g_partials_addr[dev];
  }
  // Stage 1 writes every partial that stage 2 reads, so nothing left over from an earlier call is used.
  e = launch_colsum(plan->d.dtype, M_dev, rows, cols, out_dev, partials, reinterpret_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) {
    fbl_note_cuda_error(e, "fbl_colsum_noalloc: launch");
    return FBL_ERR_CUDA;
  }
  return FBL_OK;
}

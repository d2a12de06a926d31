// What the two kernels for fp32 products share: the parameter block of a launch, and the end of a tile's work -- slices'
// sums, bias, residual, padding rows, the fused row reduction.
#pragma once
#include <string.h>

#include "fbl_internal.h"
#include "tc_common.cuh"

namespace f32g {

constexpr int MAX_TERMS = 4, MAX_PROBLEMS = 5;

struct alignas(64) Problem {
  CUtensorMap ta[MAX_TERMS], tb[MAX_TERMS];
  int n_terms, kblocks[MAX_TERMS];
  int a_k[MAX_TERMS], b_k[MAX_TERMS];       // 1: the operand's stored rows are K indices
  int m, n, tiles_m, tiles_n, total_kb;
  int b_static;                             // 1: the first term's B operand is an input of the whole step (a weight)
  float* c;
  long long c_rpad;
  const float* bias;
  const float* residual;
  int seq, t_pad;
  const float* dot_with;                    // fused D = rowsum(C * dot_with) per head (head widths 32 and 64), or nullptr
  float* dot_out;
  int dot_hd, dot_hq;
  // the operands themselves, for tiles that the kernel on the tensor cores forms again (see there)
  const float* a[MAX_TERMS];
  const float* b[MAX_TERMS];
  long long a_rpad[MAX_TERMS], b_rpad[MAX_TERMS];
  int k[MAX_TERMS];
};
struct alignas(64) Group {
  Problem p[MAX_PROBLEMS];
  int from[MAX_PROBLEMS];                           // which of the caller's problems each is
  int count, slices, reset_status;
  int32_t* status;
  uint4* zero_ptr;                                  // chores of the launch, see GemmArgs
  long long zero_vec;
};

// Problems in the order of their reductions' lengths: the blocks that take longest start first.
inline void longest_first(const GemmArgs* gs, int count, int* order) {
  auto length = [&](int i) { long long k = 0; for (int t = 0; t < gs[i].n_terms; ++t) k += gs[i].t[t].k; return k; };
  for (int i = 0; i < count; ++i) {
    int j = i;
    for (; j > 0 && length(order[j - 1]) < length(i); --j) order[j] = order[j - 1];
    order[j] = i;
  }
}
// Everything of a group but its addresses, for tiles of bm x bn and k-blocks of bk.
inline bool fill_group(Group& G, const GemmArgs* gs, int count, const int* order, int bm, int bn, int bk) {
  memset(&G, 0, sizeof(G));
  G.count = count;
  for (int i = 0; i < count; ++i) {
    const GemmArgs& g = gs[G.from[i] = order[i]];
    Problem& P = G.p[i];
    P.n_terms = g.n_terms; P.m = g.m; P.n = g.n; P.b_static = g.b_static;
    for (int t = 0; t < g.n_terms; ++t) {
      const GemmTerm& tm = g.t[t];
      P.kblocks[t] = (tm.k + bk - 1) / bk;
      P.total_kb += P.kblocks[t];
      P.a_k[t] = tm.a_trans ? 1 : 0;
      P.b_k[t] = tm.b_trans ? 0 : 1;
      P.a_rpad[t] = tm.a_rpad; P.b_rpad[t] = tm.b_rpad; P.k[t] = tm.k;
      if (!fbl_encode_f32_rtile_map(&P.ta[t], tm.a, tm.a_rpad, (tm.a_trans ? g.m : tm.k) / 32, P.a_k[t] ? bk : bm, (P.a_k[t] ? bm : bk) / 32) ||
          !fbl_encode_f32_rtile_map(&P.tb[t], tm.b, tm.b_rpad, (tm.b_trans ? tm.k : g.n) / 32, P.b_k[t] ? bk : bn, (P.b_k[t] ? bn : bk) / 32))
        return false;
    }
    P.tiles_m = (g.m + bm - 1) / bm; P.tiles_n = (g.n + bn - 1) / bn;
    P.c_rpad = g.c_rpad; P.seq = g.seq; P.t_pad = g.t_pad; P.dot_hd = g.dot_hd; P.dot_hq = g.dot_hq;
  }
  return true;
}
inline bool point_group(Group& G, const GemmArgs* gs, int32_t* status) {
  G.status = status;
  G.zero_ptr = (uint4*)gs[0].zero_ptr; G.zero_vec = (long long)(gs[0].zero_bytes / 16); G.reset_status = gs[0].reset_status;
  bool ok = true;
  for (int i = 0; i < G.count; ++i) {
    const GemmArgs& g = gs[G.from[i]];
    Problem& P = G.p[i];
    for (int t = 0; t < P.n_terms; ++t) {
      ok = ok && fbl_map_set_base(&P.ta[t], g.t[t].a) && fbl_map_set_base(&P.tb[t], g.t[t].b);
      P.a[t] = (const float*)g.t[t].a; P.b[t] = (const float*)g.t[t].b;
    }
    P.c = (float*)g.c; P.bias = g.bias; P.residual = (const float*)g.residual;
    P.dot_with = (const float*)g.dot_with; P.dot_out = g.dot_out;
  }
  return ok;
}

using tc::lds4;

// This block's share of the tile's rows: the slices' sums (each block's at `base` of its shared memory, rows LD floats apart)
// in slice order, bias, residual, padding rows, 16-byte stores.  A thread keeps its four columns and has two rows in flight (one
// at a time, each waiting for its loads, an 800 x 768 x 768 product took 2 us longer).
template <int BM, int BN, int LD, int THREADS>
__device__ __forceinline__ void finish_tile(const Problem& P, int slices, int slice, uint32_t base, int m0, int n0) {
  constexpr int VECS = BN / 4, STEP = THREADS / VECS, U = 2;
  static_assert(THREADS % VECS == 0, "whole rows");
  const int rows = BM / slices, r0 = slice * rows;
  const int col = (threadIdx.x % VECS) * 4, n = n0 + col;
  float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
  if (P.bias && n < P.n) bias = make_float4(P.bias[n], P.bias[n + 1], P.bias[n + 2], P.bias[n + 3]);
  for (int i0 = threadIdx.x / VECS; i0 - (int)threadIdx.x / VECS < rows; i0 += STEP * U) {
    float4 s[U], extra[U];                         // the residual, or else what the row reduction multiplies with
    bool live[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * STEP, m = m0 + r0 + i;
      live[u] = i < rows && m < P.m && n < P.n;
      s[u] = extra[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (!live[u]) continue;
      const int64_t off = rt_off<32>(P.c_rpad, m, n);
      if (P.residual) extra[u] = *reinterpret_cast<const float4*>(P.residual + off);
      else if (P.dot_with) extra[u] = *reinterpret_cast<const float4*>(P.dot_with + off);
    }
    if (slices == 1) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (live[u]) s[u] = lds4(base + (uint32_t)((r0 + i0 + u * STEP) * LD + col) * 4);
    } else {
      for (int c = 0; c < slices; ++c) {
        float4 q[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (live[u])
            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(q[u].x), "=f"(q[u].y), "=f"(q[u].z), "=f"(q[u].w)
                         : "r"(tc::map_to_cta(base + (uint32_t)((r0 + i0 + u * STEP) * LD + col) * 4, c)));
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (live[u]) { s[u].x += q[u].x; s[u].y += q[u].y; s[u].z += q[u].z; s[u].w += q[u].w; }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int m = m0 + r0 + i0 + u * STEP;
      float dot = 0.f;
      if (live[u]) {
        float4 v = s[u];
        v.x += bias.x; v.y += bias.y; v.z += bias.z; v.w += bias.w;
        const int64_t off = rt_off<32>(P.c_rpad, m, n);
        if (P.residual) { v.x += extra[u].x; v.y += extra[u].y; v.z += extra[u].z; v.w += extra[u].w; }
        if (P.t_pad > 0 && m % P.t_pad >= P.seq) v = make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(P.c + off) = v;
        if (P.dot_with) {
          const float4 q = P.residual ? *reinterpret_cast<const float4*>(P.dot_with + off) : extra[u];
          dot = fmaf(v.x, q.x, fmaf(v.y, q.y, fmaf(v.z, q.z, v.w * q.w)));
        }
      }
      if (P.dot_with) {                            // a head is 8 or 16 neighbouring threads (32 or 64 columns)
        for (int o = P.dot_hd / 8; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        if (live[u] && n % P.dot_hd == 0) P.dot_out[((int64_t)(m / P.t_pad) * P.dot_hq + n / P.dot_hd) * P.t_pad + m % P.t_pad] = dot;
      }
    }
  }
}

__device__ __forceinline__ void group_chores(const Group& G, int tid, int threads) {
  if (G.reset_status && blockIdx.x == 0 && tid == 0) *G.status = 0;
  for (long long i = (long long)blockIdx.x * threads + tid; i < G.zero_vec; i += (long long)gridDim.x * threads)
    G.zero_ptr[i] = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace f32g

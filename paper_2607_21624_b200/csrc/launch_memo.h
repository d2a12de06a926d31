// What a launch of a plan is made of besides its arguments -- parameter block with its tensor maps, kernel, grid -- is
// remembered by those arguments: a program calls with the same buffers pass after pass, and encoding ten to thirty tensor
// maps, choosing tiles and setting function attributes is a tenth of a pass's host time (forward pass of four launches 19 ->
// 17 us, ten-launch step 45 -> 41 us; passes of few tokens are host-bound: 21.7 -> 19.2 us for an adapter forward of 48
// tokens).  Bounded per plan; the oldest entry makes room.
#pragma once
#include <stdint.h>
#include <string.h>

#include <new>

#include "fbl_internal.h"

struct LaunchKey {
  static constexpr int MAX = 256;
  uint64_t v[MAX];
  int n = 0;
  void add(uint64_t x) { if (n < MAX) v[n++] = x; }
  void add(const void* p) { add((uint64_t)(uintptr_t)p); }
  void add(int a, int b) { add(((uint64_t)(uint32_t)a << 32) | (uint32_t)b); }
};

template <typename Params, int N, int KEY>
struct LaunchMemo : FblMemoBase {
  struct Entry { Params params; uint64_t key[KEY]; int n; };
  Entry entry[N];
  int next = 0;
  LaunchMemo() { for (Entry& e : entry) e.n = 0; }

  // The entry of this key.  *hit = false: a fresh one, to be filled in (and dropped by `drop` if that fails).
  Entry* find(const LaunchKey& k, bool* hit) {
    for (Entry& e : entry)
      if (e.n == k.n && memcmp(e.key, k.v, (size_t)k.n * sizeof(uint64_t)) == 0) { *hit = true; return &e; }
    Entry& e = entry[next];
    next = (next + 1) % N;
    e.n = k.n;
    memcpy(e.key, k.v, (size_t)k.n * sizeof(uint64_t));
    *hit = false;
    return &e;
  }

  // launch(params) with the parameters fill(params) makes for this key, remembered in `slot` of the plan.
  template <typename Fill, typename Launch>
  static cudaError_t run(FblMemoBase*& slot, const LaunchKey& k, Fill&& fill, Launch&& launch) {
    if (!slot) slot = new (std::nothrow) LaunchMemo();
    if (!slot || k.n > KEY || k.n >= LaunchKey::MAX) {
      Params p;
      const cudaError_t e = fill(p);
      return e != cudaSuccess ? e : launch(p);
    }
    bool hit;
    Entry* at = static_cast<LaunchMemo*>(slot)->find(k, &hit);
    if (!hit) {
      const cudaError_t e = fill(at->params);
      if (e != cudaSuccess) { at->n = 0; return e; }
    }
    return launch(at->params);
  }
};

// Everything of a group of products that its parameter block depends on.
inline void gemm_group_key(LaunchKey& k, const GemmArgs* gs, int count, const int32_t* status) {
  k.add(status);
  k.add((uint64_t)count);
  for (int i = 0; i < count; ++i) {
    const GemmArgs& g = gs[i];
    k.add(g.m, g.n);
    k.add(g.n_terms, g.b_static);
    for (int t = 0; t < g.n_terms; ++t) {
      const GemmTerm& m = g.t[t];
      k.add(m.a); k.add((uint64_t)m.a_rpad); k.add(m.b); k.add((uint64_t)m.b_rpad);
      k.add(m.k, m.a_trans * 2 + m.b_trans);
    }
    k.add(g.c); k.add((uint64_t)g.c_rpad); k.add(g.bias); k.add(g.residual); k.add(g.seq, g.t_pad);
    k.add(g.dot_with); k.add(g.dot_out); k.add(g.dot_hd, g.dot_hq);
    k.add(g.acc); k.add(g.ksplit, g.epi); k.add(g.aux1); k.add(g.c2); k.add(g.rope); k.add(g.serial, 0);
    if (i == 0) { k.add(g.late_trigger != nullptr, 0); k.add(g.zero_ptr); k.add((uint64_t)g.zero_bytes); k.add((uint64_t)g.reset_status); }
  }
}

// What a launch of a plan is made of besides addresses -- kernel, grid, and a parameter block whose tensor maps await their
// addresses -- is kept in the plan under the launch's shape: choosing tiles, encoding ten to thirty tensor maps and setting
// function attributes is host work that a pass of few tokens would wait for.  Addresses are put in on every launch (9 ns a
// tensor map, against 46 to encode one), so a pass on new buffers costs what any other does, however many layers share the
// plan (kept by address, twelve 50-token layers on one plan took 21.9 us a forward pass and one layer alone 19.0; now 19.5 and
// 19.4).  A plan has less than a dozen shapes of launches of a kind; should there be more, the oldest makes room.
#pragma once
#include <cuda.h>
#include <stdint.h>
#include <string.h>

#include <memory>
#include <new>

#include "fbl_internal.h"

struct LaunchKey {
  static constexpr int MAX = 128;          // five products of four terms are 99 words
  uint64_t v[MAX];
  int n = 0;
  LaunchKey() {                            // function attributes are a device's
    int dev = -1;
    (void)cudaGetDevice(&dev);
    add((uint64_t)(int64_t)dev);
  }
  void add(uint64_t x) { if (n < MAX) v[n] = x; ++n; }
  void add(int a, int b) { add(((uint64_t)(uint32_t)a << 32) | (uint32_t)b); }
};

template <typename Params, int N>
struct LaunchMemo : FblMemoBase {
  struct Entry { Params params; uint64_t key[LaunchKey::MAX]; int n; };
  std::unique_ptr<Entry> entry[N];
  int next = 0;

  // launch(params) with what fill(params) makes for this key, kept in the plan's `slot`, and point(params) has given addresses.
  template <typename Fill, typename Point, typename Launch>
  static cudaError_t run(const fbl_plan* p, int slot, const LaunchKey& k, Fill&& fill, Point&& point, Launch&& launch) {
    std::lock_guard<std::mutex> hold(p->memo_lock);
    if (!p->memo[slot]) p->memo[slot] = new (std::nothrow) LaunchMemo();
    LaunchMemo* memo = static_cast<LaunchMemo*>(p->memo[slot]);
    Entry* at = nullptr;
    std::unique_ptr<Entry> fresh;
    if (memo && k.n <= LaunchKey::MAX)
      for (int i = 0; i < N && !at; ++i) {
        Entry* e = memo->entry[i].get();
        if (e && e->n == k.n && memcmp(e->key, k.v, (size_t)k.n * sizeof(uint64_t)) == 0) at = e;
      }
    if (!at) {
      fresh.reset(new (std::nothrow) Entry);
      if (!fresh) return cudaErrorMemoryAllocation;
      at = fresh.get();
      const cudaError_t e = fill(at->params);
      if (e != cudaSuccess) return e;
    }
    if (!point(at->params)) return cudaErrorInvalidValue;
    const cudaError_t e = launch(at->params);
    if (fresh && memo && k.n <= LaunchKey::MAX && e == cudaSuccess) {
      fresh->n = k.n;
      memcpy(fresh->key, k.v, (size_t)k.n * sizeof(uint64_t));
      memo->entry[memo->next] = std::move(fresh);
      memo->next = (memo->next + 1) % N;
    }
    return e;
  }
};

// What the parameter block of a group of products depends on besides addresses, in the order of the group.
inline void gemm_group_key(LaunchKey& k, const GemmArgs* gs, int count) {
  k.add(count, (gs[0].late_trigger != nullptr) * 2 + (gs[0].serial != 0));
  for (int i = 0; i < count; ++i) {
    const GemmArgs& g = gs[i];
    k.add(g.m, g.n);
    k.add(g.n_terms, g.b_static);
    for (int t = 0; t < g.n_terms; ++t) {
      const GemmTerm& m = g.t[t];
      k.add((uint64_t)m.a_rpad); k.add((uint64_t)m.b_rpad);
      k.add(m.k, m.a_trans * 2 + m.b_trans);
    }
    k.add((uint64_t)g.c_rpad); k.add(g.seq, g.t_pad); k.add(g.dot_hd, g.dot_hq); k.add(g.ksplit, g.epi);
    // which operands there are: fill_group's checks look at them
    k.add((g.bias != nullptr) | (g.residual != nullptr) << 1 | (g.dot_with != nullptr) << 2 | (g.aux1 != nullptr) << 3 |
          (g.c2 != nullptr) << 4 | (g.rope != nullptr) << 5 | (g.acc != nullptr) << 6, 0);
  }
}

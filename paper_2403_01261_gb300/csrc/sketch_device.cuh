// sketch_device.cuh -- device functions of the counting sweeps over rows of more
// than 32 entries (sketch_kernels.cu says how they count).  Included by one
// translation unit each.
#pragma once

#include "sweep_device.cuh"

namespace gsl {

namespace {

constexpr unsigned SETTLED = 0x80000000u;   // label bit: no longer in question (absent entries are -1)

__device__ __forceinline__ Best<unsigned> warp_best(Best<unsigned> b) {
  const unsigned m = __reduce_max_sync(FULL, b.sum);
  return {m, __reduce_max_sync(FULL, b.sum == m ? b.inv : 0u)};
}
__device__ __forceinline__ Best<unsigned long long> warp_best(Best<unsigned long long> b) {
  const unsigned hi = __reduce_max_sync(FULL, (unsigned)(b.sum >> 32));
  const bool h = (unsigned)(b.sum >> 32) == hi;
  const unsigned lo = __reduce_max_sync(FULL, h ? (unsigned)b.sum : 0u);
  const unsigned inv = __reduce_max_sync(FULL, (h && (unsigned)b.sum == lo) ? b.inv : 0u);
  return {((unsigned long long)hi << 32) | lo, inv};
}

__device__ __forceinline__ unsigned ceil_log2(unsigned x) { return x <= 1 ? 0u : 32u - (unsigned)__clz((int)(x - 1)); }

template <int T>
__device__ __forceinline__ void team_sync() {
  if (T == 32) __syncwarp();
  else __syncthreads();
}
template <int T>
__device__ __forceinline__ bool team_any(bool p) {
  if (T != 32) return __syncthreads_or(p) != 0;
  __syncwarp();
  return __any_sync(FULL, p);
}

// What a team shares besides its table.
template <int T, typename S>
struct TeamShared {
  S sum[T / 32];
  unsigned inv[T / 32];
  unsigned long long wsum;
  unsigned cnt;
  long long next;
  unsigned part[T == 32 ? 1 : 64 + 1];   // long rows: first entry of every part
  unsigned fill[T == 32 ? 1 : 64];
};

template <int T, typename B, typename S>
__device__ __forceinline__ Best<B> team_best(Best<B> b, TeamShared<T, S>* sh) {
  b = warp_best(b);
  if (T == 32) return b;
  const int lane = threadIdx.x & 31;
  if (lane == 0) {
    sh->sum[threadIdx.x >> 5] = (S)b.sum;
    sh->inv[threadIdx.x >> 5] = b.inv;
  }
  __syncthreads();
  b = {0, 0u};
  if (lane < T / 32) b = {(B)sh->sum[lane], sh->inv[lane]};
  return warp_best(b);   // the next barrier comes before sh is written again
}

// The table's memory holds 1 << lg counters of the counting round, or half as
// many slots of (sum, label) in the rounds after it (a quarter with 64-bit
// sums).
//
// Counters are 32-bit: shared 64-bit adds take eight times as long and far
// longer still on one hot counter (a 98,000-entry row with a common label
// took 0.9 ms).  With 64-bit sums they hold bounds instead, (w >> q) + 1 per
// entry, so that sum < counter << q; the named label's sum is exact anyway.
struct Sketch {
  unsigned* cnt;
  unsigned lg;
  unsigned q;   // 64-bit sums: shift of the bounds
  __device__ __forceinline__ unsigned slot(unsigned label) const { return sketch_hash(label, 0) >> (32u - lg); }
};
template <typename S>
struct Slots {
  S* sum;
  unsigned* lab;
  unsigned lg;
  __device__ __forceinline__ explicit Slots(const Sketch& t)
      : sum(reinterpret_cast<S*>(t.cnt)), lg(t.lg - (sizeof(S) == 8 ? 2 : 1)) {
    lab = reinterpret_cast<unsigned*>(sum + (1u << lg));
  }
  __device__ __forceinline__ unsigned slot(unsigned label, int round) const {
    return sketch_hash(label, round) >> (32u - lg);
  }
};

template <int T, typename S>
__device__ __forceinline__ void sketch_clear(S* sum, unsigned lg, int tid) {
  constexpr unsigned PER = 16 / sizeof(S);   // at least 64 counters: whole 16-byte words
  int4* p = reinterpret_cast<int4*>(sum);
#pragma unroll 4
  for (unsigned k = tid; k < (1u << lg) / PER; k += T) p[k] = make_int4(0, 0, 0, 0);
}

// A counter's step for an entry of weight w.
template <int WT>
__device__ __forceinline__ unsigned counter_step(const Sketch& t, const int* wp, int e) {
  if (WT == 0) return 1u;
  const unsigned w = (unsigned)wp[e];
  return WT == 1 ? w : (w >> t.q) + 1u;
}

// Labels of a row in registers: entry k * T + tid in l[k].
template <int T, int K>
struct RegItems {
  int (&l)[K];
  int d, tid;
  template <typename F>
  __device__ __forceinline__ void each(F&& f) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (k * T < d) f(l[k], k * T + tid);   // team-uniform; absent entries are -1
  }
};

// Labels of a row in the block's scratch list.
template <int T>
struct MemItems {
  int* list;
  int d, tid;
  template <typename F>
  __device__ __forceinline__ void each(F&& f) {
    // eight loads of a thread in flight: a store may alias the next load
    for (int e0 = tid; e0 < d; e0 += 8 * T) {
      int was[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) was[u] = e0 + u * T < d ? list[e0 + u * T] : -1;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        int l = was[u];
        f(l, e0 + u * T);
        if (l != was[u]) list[e0 + u * T] = l;
      }
    }
  }
};

// Sum of x over the team's threads.
template <int T, typename S>
__device__ __forceinline__ S team_total(unsigned long long x, TeamShared<T, S>* sh) {
  x = warp_sum_u64(x);
  if (T == 32) return (S)x;
  __syncthreads();
  if (threadIdx.x == 0) sh->wsum = 0;
  __syncthreads();
  if ((threadIdx.x & 31) == 0 && x) atomicAdd(&sh->wsum, x);
  __syncthreads();
  return (S)sh->wsum;
}

// The counting round's outcome: `mine` is each thread's largest (running
// sum, label) over its adds, counters hold the final sums; `best` covers the
// labels counted before (none: sum 0).  Returns whether it now covers these
// too; if not, the labels that could still beat it are left open,
// `open_items` of them.
template <int T, int WT, typename S, typename Items>
__device__ __forceinline__ bool sketch_top(Items& items, const int* wp, const Sketch& t, Best<unsigned> mine,
                                           Best<S>& best, unsigned& open_items, TeamShared<T, S>* sh) {
  if (T == 32) __syncwarp();   // ends the adds; team_best's barrier does so for a block
  const Best<unsigned> top = team_best<T>(mine, sh);
  open_items = 0;
  // whether a label bounded by counter value c can beat `best`
  auto can_beat = [&](unsigned c, unsigned inv) {
    return WT == 2 ? ((unsigned long long)c << t.q) > (unsigned long long)best.sum : beats<S>((S)c, inv, best);
  };
  if (top.sum == 0 || !can_beat(top.sum, top.inv)) return true;   // team-uniform
  const unsigned x = ~top.inv, hx = t.slot(x);
  bool other = WT == 2;   // bounds always need the comparison with the exact sum
  unsigned long long mine_x = 0;
  items.each([&](int& l, int e) {
    if (l >= 0) {
      if ((unsigned)l == x) mine_x += WT ? (unsigned long long)(unsigned)wp[e] : 1ull;
      else if (WT != 2) other = other || t.slot((unsigned)l) == hx;
    }
  });
  if (WT != 2 && !team_any<T>(other)) {
    best = {(S)top.sum, top.inv};
    return true;
  }
  const S sum = team_total<T, S>(mine_x, sh);
  const unsigned full = top.sum - (unsigned)(WT == 2 ? (unsigned long long)sum >> t.q : (unsigned long long)sum);
  if (beats<S>(sum, top.inv, best)) best = {sum, top.inv};
  unsigned left = 0;
  items.each([&](int& l, int) {
    if (l >= 0) {
      const unsigned h = t.slot((unsigned)l);
      const unsigned c = h == hx ? full : t.cnt[h];   // a bound of every other label in the slot
      if ((unsigned)l != x && can_beat(c, ~(unsigned)l)) ++left;
      else l = (int)((unsigned)l | SETTLED);
    }
  });
  left = __reduce_add_sync(FULL, left);
  if (T == 32) {
    __syncwarp();
  } else {
    __syncthreads();
    if (threadIdx.x == 0) sh->cnt = 0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && left) atomicAdd(&sh->cnt, left);
    __syncthreads();
    left = sh->cnt;
  }
  open_items = left;
  return left == 0;
}

// Rounds first_round.. over the items whose label is not settled: on return
// all are, and `best` covers them.  Starts and ends with the team in step.
template <int T, int WT, typename S, typename Items>
__device__ __forceinline__ void sketch_rounds(Items& items, const int* wp, const Slots<S> t, int first_round,
                                              int rounds, Best<S>& best, TeamShared<T, S>* sh, int* err) {
  const int tid = T == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  auto open = [](int l) { return l >= 0; };
  for (int r = first_round;; ++r) {
    sketch_clear<T>(t.sum, t.lg, tid);
    team_sync<T>();
    items.each([&](int& l, int e) {
      if (open(l)) {
        const unsigned h = t.slot((unsigned)l, r);
        atomicAdd(t.sum + h, WT ? (S)(unsigned)wp[e] : (S)1);
        *(volatile unsigned*)(t.lab + h) = (unsigned)l;
      }
    });
    team_sync<T>();
    items.each([&](int& l, int) {   // a label that lost its slot marks it shared
      if (open(l)) {
        volatile unsigned* p = t.lab + t.slot((unsigned)l, r);
        if (*p != (unsigned)l) *p = EMPTY32;
      }
    });
    team_sync<T>();
    Best<S> mine{0, 0u};
    items.each([&](int& l, int) {
      if (open(l)) {
        const unsigned h = t.slot((unsigned)l, r);
        const S c = t.sum[h];
        if (t.lab[h] != EMPTY32 && beats<S>(c, ~(unsigned)l, mine)) mine = {c, ~(unsigned)l};
      }
    });
    mine = team_best<T>(mine, sh);
    if (beats<S>(mine.sum, mine.inv, best)) best = mine;
    bool left = false;
    items.each([&](int& l, int) {
      if (open(l)) {
        const unsigned h = t.slot((unsigned)l, r);
        // every weight is at least 1, so a label of a shared slot has at most the slot's sum less one
        if (t.lab[h] == EMPTY32 && t.sum[h] && beats<S>(t.sum[h] - 1, ~(unsigned)l, best)) left = true;
        else l = (int)((unsigned)l | SETTLED);
      }
    });
    if (!team_any<T>(left)) return;
    if (r + 1 - first_round >= rounds) break;
  }
  if (rounds < SKETCH_ROUNDS) {   // a lowered retry bound
    raise_err(err, ERRBIT_TIMEOUT);
    return;
  }
  // labels that met another one in every round: one by one, the smallest first
  for (;;) {
    unsigned x = EMPTY32;
    items.each([&](int& l, int) {
      if (open(l) && (unsigned)l < x) x = (unsigned)l;
    });
    const Best<unsigned> lowest = warp_best(Best<unsigned>{~x, 0u});
    x = ~lowest.sum;
    if (T != 32) {
      __syncthreads();
      if (threadIdx.x == 0) sh->cnt = EMPTY32;
      __syncthreads();
      if ((threadIdx.x & 31) == 0) atomicMin(&sh->cnt, x);
      __syncthreads();
      x = sh->cnt;
    }
    if (x == EMPTY32) return;
    unsigned long long of_x = 0;
    items.each([&](int& l, int e) {
      if ((unsigned)l == x) of_x += WT ? (unsigned long long)(unsigned)wp[e] : 1ull;
    });
    const S c = team_total<T, S>(of_x, sh);
    if (beats<S>(c, ~x, best)) best = {c, ~x};
    items.each([&](int& l, int) {
      if ((unsigned)l == x) l = (int)((unsigned)l | SETTLED);
    });
    team_sync<T>();
  }
}

// Counts the items (counters clear) and leaves `best` covering them.
template <int T, int WT, typename S, typename Items>
__device__ __forceinline__ void sketch_count(Items& items, const int* wp, const Sketch& t, int rounds,
                                             Best<S>& best, TeamShared<T, S>* sh, int* err) {
  Best<unsigned> mine{0, 0u};
  items.each([&](int& x, int e) {
    if (x >= 0) {
      const unsigned w = counter_step<WT>(t, wp, e);
      const unsigned c = atomicAdd(t.cnt + t.slot((unsigned)x), w) + w;
      if (beats<unsigned>(c, ~(unsigned)x, mine)) mine = {c, ~(unsigned)x};
    }
  });
  unsigned left;
  if (!sketch_top<T, WT, S>(items, wp, t, mine, best, left, sh))
    sketch_rounds<T, WT, S>(items, wp, Slots<S>(t), 1, rounds, best, sh, err);
}

// One row in registers, K entries per thread (d <= T * K), LG counters (log2).
// GENERAL: first-sweep checks, identity labels, pre-gathered labels.
template <int T, int K, int LG, int WT, bool ASYNC, bool GENERAL, typename S>
__device__ __forceinline__ void sketch_row(const SweepArgs& a, int v, int old, const int* cp, const int* wp,
                                           const int* lp, int d, int tid, unsigned* mem, int rounds, const Pol& pol,
                                           Best<S>& best, unsigned long long& ws, TeamShared<T, S>* sh) {
  int l[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    l[k] = -1;
    if (k * T < d) {   // team-uniform
      int w;
      if (GENERAL) load_entry<WT != 0>(a, cp, wp, d, k * T + tid, pol, l[k], w);
      else l[k] = later_col(a, cp, d, k * T + tid, pol);
      if (GENERAL && WT && l[k] >= 0) ws += (unsigned long long)(unsigned)w;
    }
  }
  const Sketch t{mem, LG, WT == 2 ? ceil_log2((unsigned)d) : 0u};
  sketch_clear<T>(t.cnt, LG, tid);   // under the column loads
  if (GENERAL && a.ident) {
    // strictly increasing: every label (its id) occurs once
    bool inc = true;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int e = k * T + tid;
      if (e < d && (l[k] < 0 || (e + 1 < d && __ldg(cp + e + 1) <= l[k]))) inc = false;
      check_same_graph(a, v, l[k]);
      if (l[k] >= 0 && l[k] != v) {
        const S c = WT ? (S)(unsigned)wp[e] : (S)1;
        if (beats<S>(c, ~(unsigned)l[k], best)) best = {c, ~(unsigned)l[k]};
      }
    }
    if (!team_any<T>(!inc)) {
      best = team_best<T>(best, sh);
      return;
    }
    best = {0, 0u};
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (k * T < d) {
      if (GENERAL) {
        check_same_graph(a, v, l[k]);
        l[k] = entry_label<ASYNC>(a, lp, k * T + tid, l[k], v, pol);
      } else if (l[k] >= 0) {
        l[k] = l[k] == v ? -1 : (ASYNC ? ld_label_rw(a.prev + l[k]) : ld_label_ro(a.prev + l[k], pol.label));
      }
    }
  }
  if (T == 32 && !GENERAL && WT != 2 && !a.spread) {
    // a strict majority of the own label needs no table
    unsigned own = 0;
    const unsigned long long bound = WT ? (a.kw ? (unsigned long long)a.kw[v] : ~0ull) : (unsigned long long)d;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (k * T < d) {
        const bool mine = l[k] == old;
        if (WT) own += __reduce_add_sync(FULL, mine ? (unsigned)__ldg(wp + k * T + tid) : 0u);
        else own += (unsigned)__popc(__ballot_sync(FULL, mine));
      }
    }
    if (2ull * own > bound) {
      best = {(S)own, ~(unsigned)old};
      return;
    }
  }
  team_sync<T>();   // the counters are clear
  RegItems<T, K> items{l, d, tid};
  sketch_count<T, WT, S>(items, wp, t, rounds, best, sh, &a.ctr->err);
}

// One row through the block's scratch list.
template <int T, int LG, int WT, bool ASYNC, bool GENERAL, typename S>
__device__ __forceinline__ void sketch_long_row(const SweepArgs& a, int v, const int* cp, const int* wp,
                                                const int* lp, int d, int tid, unsigned* mem, int* list,
                                                long long region, int rounds, const Pol& pol, Best<S>& best,
                                                unsigned long long& ws, TeamShared<T, S>* sh) {
  if (GENERAL && a.ident) {
    // strictly increasing: every label (its id) occurs once
    bool inc = true;
    unsigned long long sum = 0;
#pragma unroll 4
    for (int e = tid; e < d; e += T) {
      int j, w;
      load_entry<WT != 0>(a, cp, wp, d, e, pol, j, w);
      if (j < 0 || (e + 1 < d && __ldg(cp + e + 1) <= j)) inc = false;
      check_same_graph(a, v, j);
      if (WT && j >= 0) sum += (unsigned long long)(unsigned)w;
      if (j >= 0 && j != v && beats<S>((S)(unsigned)w, ~(unsigned)j, best)) best = {(S)(unsigned)w, ~(unsigned)j};
    }
    if (!team_any<T>(!inc)) {
      best = team_best<T>(best, sh);
      ws = sum;
      return;
    }
    best = {0, 0u};
  }
  const Sketch t{mem, LG, WT == 2 ? ceil_log2((unsigned)d) : 0u};
  sketch_clear<T>(t.cnt, LG, tid);
  team_sync<T>();
  Best<unsigned> mine{0, 0u};
  // gather and count; eight entries of a thread in flight
  for (int e0 = 0; e0 < d; e0 += 8 * T) {
    int l[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      int w;
      const int e = e0 + u * T + tid;
      if (GENERAL) load_entry<WT != 0>(a, cp, wp, d, e, pol, l[u], w);
      else l[u] = later_col(a, cp, d, e, pol);
      if (GENERAL && WT && l[u] >= 0) ws += (unsigned long long)(unsigned)w;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (GENERAL) check_same_graph(a, v, l[u]);
      l[u] = entry_label<ASYNC>(a, lp, e0 + u * T + tid, l[u], v, pol);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * T + tid;
      if (e < d) list[e] = l[u];
      if (l[u] >= 0) {
        const unsigned w = counter_step<WT>(t, wp, e);
        const unsigned c = atomicAdd(t.cnt + t.slot((unsigned)l[u]), w) + w;
        if (beats<unsigned>(c, ~(unsigned)l[u], mine)) mine = {c, ~(unsigned)l[u]};
      }
    }
  }
  MemItems<T> items{list, d, tid};
  unsigned left;
  if (sketch_top<T, WT, S>(items, wp, t, mine, best, left, sh)) return;
  if (left <= (1u << (LG - 2))) {
    sketch_rounds<T, WT, S>(items, wp, Slots<S>(t), 1, rounds, best, sh, &a.ctr->err);
    return;
  }
  // many labels of about the same weight: the open entries in parts by a
  // second hash, each counted on its own with the best so far as a bound
  constexpr int PART = T * 8;   // entries aimed at, half of what the registers hold
  const unsigned lgp = min(6u, max(1u, ceil_log2(left / PART + 1)));
  const unsigned np = 1u << lgp;
  int* out = list + region / 3;
  int* outw = out + region / 3;
  auto part_of = [&](int l) { return ((unsigned)l * 0x7FEB352Du) >> (32u - lgp); };
  __syncthreads();
  if (tid < 64) sh->fill[tid] = 0;
  __syncthreads();
  items.each([&](int& l, int) {
    if (l >= 0) atomicAdd(&sh->fill[part_of(l)], 1u);
  });
  __syncthreads();
  if (tid == 0) {
    unsigned run = 0;
    for (unsigned p = 0; p < np; ++p) {
      const unsigned n = sh->fill[p];
      sh->part[p] = run;
      sh->fill[p] = run;
      run += n;
    }
    sh->part[np] = run;
  }
  __syncthreads();
  items.each([&](int& l, int e) {
    if (l >= 0) {
      const unsigned at = atomicAdd(&sh->fill[part_of(l)], 1u);
      out[at] = l;
      if (WT) outw[at] = wp[e];
    }
  });
  __syncthreads();
  for (unsigned p = 0; p < np; ++p) {
    const int from = (int)sh->part[p], n = (int)sh->part[p + 1] - from;
    if (n == 0) continue;   // block-uniform
    sketch_clear<T>(t.cnt, LG, tid);
    __syncthreads();
    if (n <= T * 16) {
      int l[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) l[k] = k * T + tid < n ? out[from + k * T + tid] : -1;
      RegItems<T, 16> part{l, n, tid};
      sketch_count<T, WT, S>(part, outw + from, t, rounds, best, sh, &a.ctr->err);
    } else {
      MemItems<T> part{out + from, n, tid};
      sketch_count<T, WT, S>(part, outw + from, t, rounds, best, sh, &a.ctr->err);
    }
    __syncthreads();
  }
}

}  // namespace

}  // namespace gsl

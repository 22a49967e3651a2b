// tile_device.cuh -- device functions of the short-row sweeps (rows of at most
// 32 entries): the argmax of one lane's row, and of rows counted G lanes each
// with one row's metadata per lane.  Included by one translation unit each.
#pragma once

#include "sweep_device.cuh"

namespace gsl {

namespace {

constexpr int TILE_U = 4;            // steps loaded together
constexpr int GROUP_SLOTS = 128;     // sketch slots per warp
constexpr int LANE_ROW = 4;          // longest row of one lane

// Largest (sum, ~label) over the G lanes of gmask; lanes without one pass sum 0.
template <int G>
__device__ __forceinline__ Best<unsigned long long> group_best(unsigned long long sum, int lbl, unsigned gmask) {
  Best<unsigned long long> b{sum, sum ? ~(unsigned)lbl : 0u};
#pragma unroll
  for (int o = G / 2; o >= 1; o >>= 1) {
    const unsigned long long s = __shfl_xor_sync(FULL, b.sum, o);
    const unsigned i = __shfl_xor_sync(FULL, b.inv, o);
    if (beats<unsigned long long>(s, i, b)) b = {s, i};
  }
  return b;
}
template <int G>
__device__ __forceinline__ Best<unsigned> group_best(unsigned sum, int lbl, unsigned gmask) {
  Best<unsigned> b;
  if (G >= 16) {
    b.sum = __reduce_max_sync(gmask, sum);
    b.inv = __reduce_max_sync(gmask, (sum && sum == b.sum) ? ~(unsigned)lbl : 0u);
  } else {   // several masks would run one after the other
    b.sum = sum;
#pragma unroll
    for (int o = G / 2; o >= 1; o >>= 1) b.sum = max(b.sum, __shfl_xor_sync(FULL, b.sum, o));
    b.inv = (sum && sum == b.sum) ? ~(unsigned)lbl : 0u;
#pragma unroll
    for (int o = G / 2; o >= 1; o >>= 1) b.inv = max(b.inv, __shfl_xor_sync(FULL, b.inv, o));
  }
  return b;
}

template <typename S>
__device__ __forceinline__ void take_better(Best<S>& a, const Best<S>& b) {
  if (beats<S>(b.sum, b.inv, a)) a = b;
}

// Sum of a value over the lanes of mask m (the calling lane's among them).
__device__ __forceinline__ unsigned mask_sum(unsigned m, unsigned x) { return __reduce_add_sync(m, x); }
__device__ __forceinline__ unsigned long long mask_sum(unsigned m, unsigned long long x) {   // x below 2^31
  const unsigned lo = __reduce_add_sync(m, (unsigned)x & 0xFFFFu), hi = __reduce_add_sync(m, (unsigned)x >> 16);
  return ((unsigned long long)hi << 16) + lo;
}

// A warp's sketch slots: sums and labels.
template <typename S>
struct GroupSlots {
  S sum[GROUP_SLOTS];
  unsigned lab[GROUP_SLOTS];
};

// Eq. 2's argmax of a group of G lanes, one entry each, in the group's 4 G
// slots from `base` on (sums all zero on entry and on return).
// Warp-synchronous; the slots of a warp's groups are disjoint.
template <int G, typename S>
__device__ __forceinline__ Best<S> group_sketch(GroupSlots<S>& slots, int base, int lbl, S wt, bool valid,
                                                unsigned gmask, int rounds, int* err) {
  constexpr int SHIFT = G == 32 ? 25 : (G == 16 ? 26 : 27);   // 4 G slots
  Best<S> best{0, 0u};
  bool act = valid;
  for (int r = 0;; ++r) {
    const int h = base + (int)(sketch_hash((unsigned)lbl, r) >> SHIFT);
    volatile S* sum = slots.sum + h;
    volatile unsigned* lab = slots.lab + h;
    if (act) {
      atomicAdd(slots.sum + h, wt);
      *lab = (unsigned)lbl;
    }
    __syncwarp();
    S c = 0;
    bool shared_slot = false;
    if (act) {
      c = *sum;
      shared_slot = *lab != (unsigned)lbl;
    }
    if (__any_sync(FULL, shared_slot)) {   // the label that won the store learns of the others
      __syncwarp();
      if (shared_slot) *lab = EMPTY32;
      __syncwarp();
      if (act) shared_slot = *lab == EMPTY32;
    }
    __syncwarp();
    if (act) *sum = 0;
    __syncwarp();
    take_better(best, group_best<G>(act && !shared_slot ? c : (S)0, lbl, gmask));
    act = act && shared_slot && c && beats<S>(c - 1, ~(unsigned)lbl, best);
    if (!__any_sync(FULL, act)) return best;
    if (r + 1 >= rounds) {
      if (rounds < SKETCH_ROUNDS) {   // a lowered retry bound
        raise_err(err, ERRBIT_TIMEOUT);
        return best;
      }
      const unsigned m = __match_any_sync(FULL, act ? lbl : -1) & gmask;
      S e = 0;
      if (act) e = mask_sum(m, wt);   // m: the lanes of this label, all here
      take_better(best, group_best<G>(e, lbl, gmask));
      return best;
    }
  }
}

// The largest (sum, smallest label) over a lane's labels in registers, -1 for none.
template <typename S>
__device__ __forceinline__ int lane_argmax(const int* l, const unsigned* w, int old) {
  S c[LANE_ROW];
#pragma unroll
  for (int i = 0; i < LANE_ROW; ++i) c[i] = w[i];
#pragma unroll
  for (int i = 0; i < LANE_ROW; ++i) {
#pragma unroll
    for (int k = i + 1; k < LANE_ROW; ++k) {
      const bool same = l[i] == l[k];
      c[i] += same ? w[k] : 0u;
      c[k] += same ? w[i] : 0u;
    }
  }
  S bc = 0;
  int bl = old;
#pragma unroll
  for (int i = 0; i < LANE_ROW; ++i) {
    if (l[i] >= 0 && (c[i] > bc || (c[i] == bc && l[i] < bl))) {
      bc = c[i];
      bl = l[i];
    }
  }
  return bl;
}

// Neighbour and weight of entry e.  FIRST: with the first sweep's checks;
// later sweeps only clamp an out-of-range column away (the first sweep, or
// the streaming check before it, has reported it).
template <int WT, bool FIRST>
__device__ __forceinline__ void tile_entry(const SweepArgs& a, const int* cp, const int* wp, int d, int e,
                                           const Pol& pol, int& j, int& wt) {
  if (FIRST) {
    load_entry<WT != 0>(a, cp, wp, d, e, pol, j, wt);
  } else {
    j = later_col(a, cp, d, e, pol);
    wt = WT && e < d ? ld_stream(wp + e, pol.stream) : (e < d ? 1 : 0);
  }
}

template <bool ASYNC, bool FIRST>
__device__ __forceinline__ int tile_label(const SweepArgs& a, int j, int v, const Pol& pol) {
  if (FIRST) {
    check_same_graph(a, v, j);
    return entry_label<ASYNC>(a, nullptr, 0, j, v, pol);
  }
  if (j < 0 || j == v) return -1;
  return ASYNC ? ld_label_rw(a.prev + j) : ld_label_ro(a.prev + j, pol.label);
}

// The label of one step's row (this lane's group): own label `own`, degree dd,
// this lane's entry e of it (column j, weight w, label lbl); `has` when the
// group holds a row at all.  Every lane of the warp calls it.
template <int WT, bool FIRST, int G>
__device__ __forceinline__ int step_label(const SweepArgs& a, bool has, int own, int dd, int e, int j, int w, int lbl,
                                          unsigned gmask, GroupSlots<typename SumOf<WT>::T>* slots, int rounds) {
  using S = typename SumOf<WT>::T;
  const int lane = threadIdx.x & 31;
  const bool nb = j >= 0, valid = lbl >= 0;
  if (WT == 1 && FIRST && a.check) {
    unsigned long long ws = nb ? (unsigned long long)w : 0ull;
#pragma unroll
    for (int o = G / 2; o >= 1; o >>= 1) ws += __shfl_xor_sync(FULL, ws, o);
    if (ws >= (1ull << 31)) raise_err(&a.ctr->err, ERRBIT_OVERFLOW);
  }
  // settled without counting every label: the own label's strict
  // majority (unit weights), or from the identity labels a strictly
  // increasing row, whose labels are all distinct.  The votes are the
  // whole warp's and stand outside every lane's condition.
  bool settled;
  Best<S> b;
  if (FIRST && a.ident) {
    const int jp = __shfl_up_sync(FULL, j, 1, G);
    const unsigned ok = __ballot_sync(FULL, !has || e >= dd || (nb && (e == 0 || jp < j)));
    settled = (ok & gmask) == gmask;
    b = group_best<G>(valid ? (S)(unsigned)w : (S)0, lbl, gmask);
  } else {
    const unsigned all = __ballot_sync(FULL, valid) & gmask;
    const unsigned mine = __ballot_sync(FULL, valid && lbl == own) & gmask;
    settled = all == 0 || (!WT && 2 * __popc(mine) > __popc(all));
    b = {settled ? (S)__popc(mine) : (S)0, ~(unsigned)own};
  }
  if (!__all_sync(FULL, settled)) {
    Best<S> x;
    if (WT) {
      x = group_sketch<G, S>(*slots, 4 * (lane & ~(G - 1)), lbl, (S)(unsigned)w, valid && !settled, gmask,
                             rounds, &a.ctr->err);
    } else {
      const unsigned m = __match_any_sync(FULL, lbl) & gmask;
      x = group_best<G>(valid ? (S)__popc(m) : (S)0, lbl, gmask);
    }
    if (!settled) b = x;
  }
  return b.sum ? (int)~b.inv : own;
}

// The tile's rows, one per lane (lanes 0..rows-1: vertex v, row start s,
// degree d <= G, own label old), counted 32 / G per step by G lanes each.
// Lane r receives row r's label in `nl`.
template <int WT, bool ASYNC, bool FIRST, int G>
__device__ __forceinline__ void tile_steps(const SweepArgs& a, int rows, int v, long long s, int d, int old,
                                           GroupSlots<typename SumOf<WT>::T>* slots, int rounds, const Pol& pol,
                                           int& nl) {
  const int lane = threadIdx.x & 31;
  constexpr int PER = 32 / G;   // rows per step
  const unsigned gmask = G == 32 ? FULL : ((1u << (G & 31)) - 1u) << (lane & ~(G - 1));
  const int e = lane & (G - 1);
  const int steps = (rows + PER - 1) / PER;
  int jn[TILE_U], wn[TILE_U];
  // this lane's row in step t, and its entry of that row
  auto row_at = [&](int t) -> int { return PER * t + lane / G; };
  auto load = [&](int t, int& j, int& w) {
    const int r = row_at(t);
    const long long rs = __shfl_sync(FULL, s, r & 31);
    const int rd = __shfl_sync(FULL, d, r & 31);
    tile_entry<WT, FIRST>(a, a.col + rs, a.w + rs, r < rows ? rd : 0, e, pol, j, w);
  };
#pragma unroll
  for (int u = 0; u < TILE_U; ++u) load(u, jn[u], wn[u]);
  for (int t0 = 0; t0 < steps; t0 += TILE_U) {
    int j[TILE_U], w[TILE_U], l[TILE_U];
#pragma unroll
    for (int u = 0; u < TILE_U; ++u) {
      const int vv = __shfl_sync(FULL, v, row_at(t0 + u) & 31);
      j[u] = jn[u];
      w[u] = wn[u];
      l[u] = tile_label<ASYNC, FIRST>(a, j[u], vv, pol);
    }
    if (t0 + TILE_U < steps) {
#pragma unroll
      for (int u = 0; u < TILE_U; ++u) load(t0 + TILE_U + u, jn[u], wn[u]);
    }
#pragma unroll
    for (int u = 0; u < TILE_U; ++u) {
      if (t0 + u >= steps) break;   // warp-uniform
      const int r = row_at(t0 + u);
      const int x = step_label<WT, FIRST, G>(a, r < rows, __shfl_sync(FULL, old, r & 31),
                                             __shfl_sync(FULL, d, r & 31), e, j[u], w[u], l[u], gmask, slots, rounds);
      const int y = __shfl_sync(FULL, x, (lane & (PER - 1)) * G);   // lane r takes row r's label from its group
      if (lane / PER == t0 + u) nl = y;
    }
  }
}

}  // namespace

}  // namespace gsl

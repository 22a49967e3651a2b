// tile_kernels.cu -- the sweep for rows of at most 32 entries (classes 0..5).
//
// Classes 0..2 (d <= 4), lane_sweep_kernel: one lane per row in natural
// order, the row's labels in registers, all pairs compared.  Flags, offsets,
// own labels and results are coalesced and neighbouring rows share column
// sectors, so these classes need no worklist: the frontier binning skips
// them and one launch replaces three.  Bound by the latency of the chain
// offsets - columns - labels, so the next tile's flags and offsets are
// loaded ahead.
//
// Classes 3..5, tile_sweep_kernel: a warp takes up to 32 rows of the
// worklist, one row's metadata and result per lane, and counts them four
// rows (5..8 entries, 8 lanes each), two (9..16) or one (17..32) a step, with
// the columns of the next four steps and the labels of four steps in
// flight.  A row whose own label holds a strict majority is settled by two
// votes; otherwise equal labels are found with __match_any_sync (unit
// weights) or summed in a shared-memory sketch (weights: a masked
// __reduce_add_sync runs once per label).  Bound by instruction issue: with
// one row's metadata per step the same rows took 247 instructions for 25
// entries at 63 % of the issue slots.
#include "sweep_device.cuh"

namespace gsl {

namespace {

constexpr int TILE_BLOCK = 256;
constexpr int TILE_MIN_BLOCKS = 4;   // 64 registers: four steps of loads in flight per warp, 32 warps per SM
constexpr int LANE_MIN_BLOCKS = 8;   // 32 registers
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
    act = act && shared_slot && beats<S>(c - 1, ~(unsigned)lbl, best);
    if (!__any_sync(FULL, act)) return best;
    if (r + 1 >= rounds) {
      if (rounds < SKETCH_ROUNDS) raise_err(err, ERRBIT_TIMEOUT);   // a lowered retry bound
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

// The tile's rows, one per lane (lanes 0..rows-1: vertex v, row start s,
// degree d <= G, own label old), counted 32 / G per step by G lanes each.
// Lane r receives row r's label in `nl`.
template <int WT, bool ASYNC, bool FIRST, int G>
__device__ __forceinline__ void tile_steps(const SweepArgs& a, int rows, int v, long long s, int d, int old,
                                           GroupSlots<typename SumOf<WT>::T>* slots, int rounds, const Pol& pol,
                                           int& nl) {
  using S = typename SumOf<WT>::T;
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
      const int own = __shfl_sync(FULL, old, r & 31);
      const int lbl = l[u];
      const bool nb = j[u] >= 0, valid = lbl >= 0;
      if (WT == 1 && FIRST && a.check) {
        unsigned long long ws = nb ? (unsigned long long)w[u] : 0ull;
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
        const int jp = __shfl_up_sync(FULL, j[u], 1, G);
        const int dd = __shfl_sync(FULL, d, r & 31);
        const unsigned ok = __ballot_sync(FULL, r >= rows || e >= dd || (nb && (e == 0 || jp < j[u])));
        settled = (ok & gmask) == gmask;
        b = group_best<G>(valid ? (S)(unsigned)w[u] : (S)0, lbl, gmask);
      } else {
        const unsigned all = __ballot_sync(FULL, valid) & gmask;
        const unsigned mine = __ballot_sync(FULL, valid && lbl == own) & gmask;
        settled = all == 0 || (!WT && 2 * __popc(mine) > __popc(all));
        b = {settled ? (S)__popc(mine) : (S)0, ~(unsigned)own};
      }
      if (!__all_sync(FULL, settled)) {
        Best<S> x;
        if (WT) {
          x = group_sketch<G, S>(*slots, 4 * (lane & ~(G - 1)), lbl, (S)(unsigned)w[u], valid && !settled, gmask,
                                 rounds, &a.ctr->err);
        } else {
          const unsigned m = __match_any_sync(FULL, lbl) & gmask;
          x = group_best<G>(valid ? (S)__popc(m) : (S)0, lbl, gmask);
        }
        if (!settled) b = x;
      }
      const int x = b.sum ? (int)~b.inv : own;
      const int y = __shfl_sync(FULL, x, (lane & (PER - 1)) * G);   // lane r takes row r's label from its group
      if (lane / PER == t0 + u) nl = y;
    }
  }
}

}  // namespace

namespace {
// Adds a kernel's per-thread change, entry and vertex counts to the counters.
__device__ __forceinline__ void flush_tile(Counters* ctr, unsigned dn, unsigned long long scan, unsigned act, int cls) {
  __shared__ unsigned long long acc[3];
  if (threadIdx.x < 3) acc[threadIdx.x] = 0;
  __syncthreads();
  dn = __reduce_add_sync(FULL, dn);
  act = __reduce_add_sync(FULL, act);
  scan = warp_sum_u64(scan);
  if ((threadIdx.x & 31) == 0 && act) {
    atomicAdd(&acc[0], (unsigned long long)dn);
    atomicAdd(&acc[1], scan);
    atomicAdd(&acc[2], (unsigned long long)act);
  }
  __syncthreads();
  if (threadIdx.x == 0 && acc[2]) {
    if (acc[0]) atomicAdd(&ctr->dn, acc[0]);
    atomicAdd(&ctr->scanned, acc[1]);
    if (cls < 0) {
      atomicAdd(&ctr->tile_scanned, acc[1]);
      atomicAdd(&ctr->tile_active, acc[2]);
    } else {
      atomicAdd(&ctr->cls_scanned[cls], acc[1]);
    }
  }
}

// Batched mode: the changed lanes' graphs, one add per graph present.
__device__ __forceinline__ void count_tile_changes(const SweepArgs& a, int v, bool changed) {
  const int g = changed ? a.gid[v] : -1;
  const unsigned m = __match_any_sync(FULL, g);
  if (changed && (m & lanemask_lt()) == 0) atomicAdd(a.dn_graph + g, (unsigned)__popc(m));
}
}  // namespace

// Classes 0..2 among the vertices [v0, v1): all of them (all_active) or
// those flagged in fcur, whose flags are cleared; with ASYNC only the
// vertices of `phase`.
template <int WT, bool ASYNC, bool FIRST>
__global__ void __launch_bounds__(TILE_BLOCK, LANE_MIN_BLOCKS)
    lane_sweep_kernel(SweepArgs a, long long v0, long long v1, unsigned char* __restrict__ fcur, int all_active,
                      const unsigned char* __restrict__ done, int phase, unsigned seed) {
  if (stopped(a)) return;
  const Pol pol = make_pol();
  const long long stride = (long long)gridDim.x * blockDim.x;
  unsigned my_dn = 0, my_act = 0, my_scan = 0;   // a thread's rows hold few entries: 32 bits
  // row bounds of vertex v (d = 0: not in this sweep or not in these classes)
  auto fetch = [&](long long v, long long& s, int& d) {
    s = 0;
    d = 0;
    bool act = v < v1;
    if (act && !all_active) act = fcur[v] != 0;
    if (ASYNC && act) act = sweep_phase(v, seed) == phase;
    if (act) {
      s = a.off[v];
      const long long dl = a.off[v + 1] - s;
      if (dl <= LANE_ROW) d = (int)dl;
    }
  };
  long long v = v0 + (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long wbase = v - (threadIdx.x & 31);
  long long s;
  int d;
  fetch(v, s, d);
  for (long long w = wbase; w < v1; w += stride, v += stride) {   // warp-uniform
    long long sn;
    int dn;
    fetch(v + stride, sn, dn);
    if (d && !all_active) fcur[v] = 0;
    if (d && a.gid && done[a.gid[v]]) d = 0;   // batched: this vertex's graph has stopped
    if (__any_sync(FULL, d > 0)) {
      int l[LANE_ROW];
      unsigned wt[LANE_ROW];
#pragma unroll
      for (int k = 0; k < LANE_ROW; ++k) {
        l[k] = -1;
        wt[k] = 1;
        if (k < d) {
          l[k] = __ldg(a.col + s + k);   // neighbouring rows share sectors: through L1
          if (WT) wt[k] = (unsigned)__ldg(a.w + s + k);
        }
      }
      const int old = d ? own_label<ASYNC>(a, (int)v) : 0;
      unsigned long long ws = 0;
#pragma unroll
      for (int k = 0; k < LANE_ROW; ++k) {
        int j = l[k];
        if (FIRST && k < d) {
          if ((unsigned)j >= (unsigned)a.n || (WT && a.check && (int)wt[k] <= 0)) {
            raise_err(&a.ctr->err, ERRBIT_INVALID);
            j = -1;
          }
          if (WT == 1 && j >= 0) ws += wt[k];
        }
        if (!FIRST && (unsigned)j >= (unsigned)a.n) j = -1;
        l[k] = tile_label<ASYNC, FIRST>(a, j, (int)v, pol);
      }
      if (WT == 1 && FIRST && a.check && ws >= (1ull << 31)) raise_err(&a.ctr->err, ERRBIT_OVERFLOW);
      const int nl = lane_argmax<typename SumOf<WT>::T>(l, wt, old);
      const bool changed = d > 0 && nl != old;
      if (d) {
        store_label<ASYNC>(a, (int)v, nl, changed);
        my_act += 1;
        my_scan += (unsigned)d;
        my_dn += changed ? 1u : 0u;
      }
      if (__any_sync(FULL, changed)) {
        if (a.dn_graph) count_tile_changes(a, (int)v, changed);
        if (a.mark && changed) {
          if (!ASYNC) a.fnext[v] = 1;
          for (int k = 0; k < d; ++k) {
            const int j = __ldg(a.col + s + k);
            if ((unsigned)j < (unsigned)a.n) a.fnext[j] = 1;
          }
        }
      }
    }
    s = sn;
    d = dn;
  }
  flush_tile(a.ctr, my_dn, my_scan, my_act, -1);
}

// Class 3, 4 or 5 (G = 8, 16, 32), from the worklist.
template <int WT, bool ASYNC, bool FIRST, int G>
__global__ void __launch_bounds__(TILE_BLOCK, TILE_MIN_BLOCKS) tile_sweep_kernel(SweepArgs a) {
  if (stopped(a)) return;
  constexpr int cls = G == 8 ? 3 : (G == 16 ? 4 : 5);
  using S = typename SumOf<WT>::T;
  __shared__ GroupSlots<S> sketch[WT ? TILE_BLOCK / 32 : 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (WT) {
    for (int k = lane; k < GROUP_SLOTS; k += 32) sketch[wid].sum[k] = 0;
    __syncwarp();
  }
  const Pol pol = make_pol();
  const int rounds = a.probe_cap < SKETCH_ROUNDS ? a.probe_cap : SKETCH_ROUNDS;
  const unsigned cnt = a.ctr->cls_count[cls];
  const int* __restrict__ work = class_work(a, cls);
  const unsigned nwarps = (gridDim.x * blockDim.x) >> 5, warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  // rows per tile: 32 once every warp gets several tiles, fewer for short worklists
  unsigned per = 32;
  while (per > 32u / G && cnt / per < 4u * nwarps) per >>= 1;
  unsigned my_dn = 0, my_act = 0;
  unsigned long long my_scan = 0;
  for (unsigned long long i0 = (unsigned long long)warp * per; i0 < cnt; i0 += (unsigned long long)nwarps * per) {
    const int rows = cnt - i0 < per ? (int)(cnt - i0) : (int)per;
    const bool mine = lane < rows;
    int v = 0, d = 0, old = 0;
    long long s = 0;
    if (mine) {
      v = work[i0 + lane];
      s = a.off[v];
      d = (int)(a.off[v + 1] - s);
      old = own_label<ASYNC>(a, v);
    }
    int nl = old;
    tile_steps<WT, ASYNC, FIRST, G>(a, rows, v, s, d, old, WT ? sketch + wid : sketch, rounds, pol, nl);
    const bool changed = mine && nl != old;
    if (mine) {
      store_label<ASYNC>(a, v, nl, changed);
      my_act += 1;
      my_scan += (unsigned long long)d;
      my_dn += changed ? 1u : 0u;
    }
    unsigned chm = __ballot_sync(FULL, changed);
    if (chm && a.dn_graph) count_tile_changes(a, v, changed);
    if (chm && a.mark) {
      if (!ASYNC && changed) a.fnext[v] = 1;
      while (chm) {
        const int r = __ffs((int)chm) - 1;
        chm &= chm - 1;
        const long long rs = __shfl_sync(FULL, s, r);
        const int rd = __shfl_sync(FULL, d, r);
        if (lane < rd) {
          const int j = ld_stream(a.col + rs + lane, pol.stream);
          if ((unsigned)j < (unsigned)a.n) a.fnext[j] = 1;
        }
      }
    }
  }
  flush_tile(a.ctr, my_dn, my_scan, my_act, cls);
}

namespace {
template <int W, bool A>
void launch_lane_t(const SweepArgs& a, long long v0, long long v1, unsigned char* fcur, int all_active,
                   const unsigned char* done, int phase, unsigned seed, const DeviceInfo& di, cudaStream_t s) {
  const long long need = (v1 - v0 + TILE_BLOCK - 1) / TILE_BLOCK, most = (long long)LANE_MIN_BLOCKS * di.sm_count;
  const int grid = (int)(need < most ? need : most);
  if (a.check || a.ident)
    lane_sweep_kernel<W, A, true><<<grid, TILE_BLOCK, 0, s>>>(a, v0, v1, fcur, all_active, done, phase, seed);
  else
    lane_sweep_kernel<W, A, false><<<grid, TILE_BLOCK, 0, s>>>(a, v0, v1, fcur, all_active, done, phase, seed);
}

template <int W, bool A, bool F>
void launch_tile_f(const SweepArgs& a, int cls, const DeviceInfo& di, cudaStream_t s) {
  const int grid = TILE_MIN_BLOCKS * di.sm_count;
  if (cls == 3) tile_sweep_kernel<W, A, F, 8><<<grid, TILE_BLOCK, 0, s>>>(a);
  else if (cls == 4) tile_sweep_kernel<W, A, F, 16><<<grid, TILE_BLOCK, 0, s>>>(a);
  else tile_sweep_kernel<W, A, F, 32><<<grid, TILE_BLOCK, 0, s>>>(a);
}

template <int W, bool A>
void launch_tile_t(const SweepArgs& a, int cls, const DeviceInfo& di, cudaStream_t s) {
  if (a.check || a.ident) launch_tile_f<W, A, true>(a, cls, di, s);
  else launch_tile_f<W, A, false>(a, cls, di, s);
}
}  // namespace

cudaError_t launch_sweep_lanes(const SweepArgs& a, int weights, bool async_mode, long long v0, long long v1,
                               unsigned char* fcur, int all_active, const unsigned char* done, int phase,
                               unsigned seed, const DeviceInfo& di, cudaStream_t s) {
  if (v1 <= v0) return cudaSuccess;
  switch (2 * weights + (async_mode ? 1 : 0)) {
    case 0: launch_lane_t<0, false>(a, v0, v1, fcur, all_active, done, phase, seed, di, s); break;
    case 1: launch_lane_t<0, true>(a, v0, v1, fcur, all_active, done, phase, seed, di, s); break;
    case 2: launch_lane_t<1, false>(a, v0, v1, fcur, all_active, done, phase, seed, di, s); break;
    case 3: launch_lane_t<1, true>(a, v0, v1, fcur, all_active, done, phase, seed, di, s); break;
    case 4: launch_lane_t<2, false>(a, v0, v1, fcur, all_active, done, phase, seed, di, s); break;
    case 5: launch_lane_t<2, true>(a, v0, v1, fcur, all_active, done, phase, seed, di, s); break;
    default: return cudaErrorInvalidValue;
  }
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_sweep_tile(const SweepArgs& a, int cls, int weights, bool async_mode, const DeviceInfo& di,
                              cudaStream_t s) {
  if (cls < 3 || cls > 5) return cudaErrorInvalidValue;
  switch (2 * weights + (async_mode ? 1 : 0)) {
    case 0: launch_tile_t<0, false>(a, cls, di, s); break;
    case 1: launch_tile_t<0, true>(a, cls, di, s); break;
    case 2: launch_tile_t<1, false>(a, cls, di, s); break;
    case 3: launch_tile_t<1, true>(a, cls, di, s); break;
    case 4: launch_tile_t<2, false>(a, cls, di, s); break;
    case 5: launch_tile_t<2, true>(a, cls, di, s); break;
    default: return cudaErrorInvalidValue;
  }
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace gsl

// solo_kernel.cu -- synchronous LPA and the split of a small graph in one launch.
//
// A 10,000-vertex graph needs a few microseconds of work per sweep; a dozen
// launches, a counter read-back and a host decision per sweep made 0.6 ms of
// it.  Here one cooperative grid (every block resident) runs all sweeps, the
// stop test and the split, with a grid barrier between the steps; the host
// launches once and reads the result once.  Vertices are taken in natural
// order, 1 to 32 per warp, each row counted by the form its length asks for
// (tile_device.cuh, sketch_device.cuh); rows of more than 256 entries are
// listed first and take a block each.  Bound by the latency of the chain
// barrier - flag - offsets - columns - labels of a sweep.
//
// Labels, flags and parents are written by other blocks of the same launch,
// so they are read at L2 (the in-place variants of the row functions).  The
// barrier's wait is bounded: past it the launch is abandoned by every block
// and the call fails with GSL_ERR_TIMEOUT.
#include <algorithm>

#include "sketch_device.cuh"
#include "tile_device.cuh"
#include "uf_device.cuh"

namespace gsl {

namespace {

constexpr int SOLO_BLOCK = 256, SOLO_WARPS = SOLO_BLOCK / 32;
constexpr int SOLO_BLOCKS_PER_SM = 4;   // 64 registers
constexpr int SOLO_WARP_ROW = 256;    // longest row of a warp
constexpr int SOLO_REG_ROW = 16 * SOLO_BLOCK;   // longest row in a block's registers
constexpr int SOLO_LG = 13;           // counters of a block's row (log2); a warp has an eighth
constexpr int SOLO_SAMPLE = 2, SOLO_SCAN = 8;   // split: links per vertex before pieces are named, entries scanned for them
constexpr long long SOLO_BLOCK_ENTRIES = 4096;  // of a graph with few, long rows
constexpr unsigned SOLO_POLLS = 1u << 22;       // barrier polls before the launch is abandoned

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier number `gen` (counted by the caller).  The last block to arrive
// reads the error bits and publishes them as the verdict before it releases
// the others, so that every block goes on or leaves alike, whatever a faster
// block raises in the next step.  False: leave.
__device__ __forceinline__ bool grid_sync(SoloState* st, const int* err, unsigned& gen) {
  __shared__ int s_good;
  __syncthreads();
  if (threadIdx.x == 0) {
    ++gen;
    __threadfence();
    if (atomicAdd(&st->arrived, 1u) == gen * gridDim.x - 1) {
      st->verdict = __ldcg(err) || __ldcg(&st->longest) > SOLO_ROW_MAX ? 1u : 0u;
      __threadfence();
      atomicExch(&st->released, gen);
    } else {
      for (unsigned k = 0; ld_acquire(&st->released) < gen; ++k) {
        if (k >= SOLO_POLLS || ld_acquire(&st->abandoned)) {
          atomicExch(&st->abandoned, 1u);
          break;
        }
      }
    }
    __threadfence();
    s_good = !ld_acquire(&st->verdict) && !ld_acquire(&st->abandoned);
  }
  __syncthreads();
  return s_good != 0;
}

__device__ __forceinline__ long long global_ns() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct SoloShared {
  unsigned counters[1u << SOLO_LG];
  TeamShared<SOLO_BLOCK, unsigned> team;
  TeamShared<32, unsigned> warp;   // not written by warps
  unsigned long long sums[3];
};

// Adds a step's per-thread counts to the sweep's.
__device__ __forceinline__ void solo_flush(SoloShared& sh, SoloState* st, int t, unsigned dn, unsigned act,
                                           unsigned long long scan) {
  __syncthreads();
  if (threadIdx.x < 3) sh.sums[threadIdx.x] = 0;
  __syncthreads();
  const unsigned d = __reduce_add_sync(FULL, dn), c = __reduce_add_sync(FULL, act);
  const unsigned long long s = warp_sum_u64(scan);
  if ((threadIdx.x & 31) == 0 && c) {
    atomicAdd(&sh.sums[0], (unsigned long long)d);
    atomicAdd(&sh.sums[1], (unsigned long long)c);
    atomicAdd(&sh.sums[2], s);
  }
  __syncthreads();
  if (threadIdx.x == 0 && sh.sums[1]) {
    if (sh.sums[0]) atomicAdd(&st->changed[t - 1], sh.sums[0]);
    atomicAdd(&st->active[t - 1], sh.sums[1]);
    atomicAdd(&st->scanned, sh.sums[2]);
  }
}

// Marks the neighbours of the changed rows among `mask`'s lanes.
__device__ __forceinline__ void solo_mark(const SweepArgs& a, unsigned mask, long long s, int d) {
  const int lane = threadIdx.x & 31;
  while (mask) {
    const int r = __ffs((int)mask) - 1;
    mask &= mask - 1;
    const long long rs = __shfl_sync(FULL, s, r);
    const int rd = __shfl_sync(FULL, d, r);
    for (int e = lane; e < rd; e += 32) {
      const int j = __ldg(a.col + rs + e);
      if ((unsigned)j < (unsigned)a.n) a.fnext[j] = 1;
    }
  }
}

// One sweep over a tile of up to 32 consecutive vertices from `base` on.
template <int WT, bool FIRST>
__device__ __forceinline__ void solo_tile(const SweepArgs& a, long long base, int width, unsigned char* fcur,
                                          bool all_active, SoloShared& sh, GroupSlots<unsigned>* slots, int rounds,
                                          const Pol& pol, unsigned& my_dn, unsigned& my_act,
                                          unsigned long long& my_scan) {
  const int lane = threadIdx.x & 31;
  const long long v = base + lane;
  bool act = lane < width && v < a.n;
  if (act && !all_active) act = __ldcg(fcur + v) != 0;
  if (!__any_sync(FULL, act)) return;
  long long s = 0;
  int d = 0;
  if (act) {
    s = a.off[v];
    const long long dl = a.off[v + 1] - s;
    act = dl > 0 && dl <= SOLO_WARP_ROW;
    d = act ? (int)dl : 0;
    if (act && !all_active) fcur[v] = 0;
  }
  const int old = act ? own_label<true>(a, (int)v) : 0;
  int nl = old;
  // one lane per row of 1..4 entries
  if (__any_sync(FULL, act && d <= LANE_ROW)) {
    int l[LANE_ROW];
    unsigned w[LANE_ROW];
    unsigned long long ws = 0;
    const int dd = d <= LANE_ROW ? d : 0;
#pragma unroll
    for (int k = 0; k < LANE_ROW; ++k) {
      l[k] = -1;
      w[k] = 1;
      if (k < dd) {
        l[k] = __ldg(a.col + s + k);
        if (WT) w[k] = (unsigned)__ldg(a.w + s + k);
      }
    }
#pragma unroll
    for (int k = 0; k < LANE_ROW; ++k) {
      int j = l[k];
      if (FIRST && k < dd) {
        if ((unsigned)j >= (unsigned)a.n || (WT && (int)w[k] <= 0)) {
          raise_err(&a.ctr->err, ERRBIT_INVALID);
          j = -1;
        }
        if (WT && j >= 0) ws += w[k];
      }
      if (!FIRST && (unsigned)j >= (unsigned)a.n) j = -1;
      l[k] = tile_label<true, FIRST>(a, j, (int)v, pol);
    }
    if (WT && FIRST && ws >= (1ull << 31)) raise_err(&a.ctr->err, ERRBIT_OVERFLOW);
    const int x = lane_argmax<unsigned>(l, w, old);
    if (dd) nl = x;
  }
  // a warp per row of 5..32 entries, four rows' loads in flight
  unsigned mask = __ballot_sync(FULL, d > LANE_ROW && d <= 32);
  while (mask) {
    int r[TILE_U], j[TILE_U], w[TILE_U], l[TILE_U];
#pragma unroll
    for (int u = 0; u < TILE_U; ++u) {
      r[u] = __ffs((int)mask) - 1;   // -1: no row left
      mask &= mask - 1;
      const long long rs = __shfl_sync(FULL, s, r[u] & 31);
      const int rd = __shfl_sync(FULL, d, r[u] & 31);
      tile_entry<WT, FIRST>(a, a.col + rs, a.w + rs, r[u] >= 0 ? rd : 0, lane, pol, j[u], w[u]);
    }
#pragma unroll
    for (int u = 0; u < TILE_U; ++u) l[u] = tile_label<true, FIRST>(a, j[u], (int)base + (r[u] & 31), pol);
#pragma unroll
    for (int u = 0; u < TILE_U; ++u) {
      if (r[u] < 0) break;   // warp-uniform
      const int x = step_label<WT, FIRST, 32>(a, true, __shfl_sync(FULL, old, r[u]), __shfl_sync(FULL, d, r[u]), lane,
                                              j[u], w[u], l[u], FULL, slots, rounds);
      if (lane == r[u]) nl = x;
    }
  }
  // and per row of 33..256 entries
  mask = __ballot_sync(FULL, d > 32);
  while (mask) {
    const int r = __ffs((int)mask) - 1;
    mask &= mask - 1;
    const long long rs = __shfl_sync(FULL, s, r);
    const int rd = __shfl_sync(FULL, d, r), ro = __shfl_sync(FULL, old, r), rv = (int)base + r;
    unsigned* mem = sh.counters + ((threadIdx.x >> 5) << (SOLO_LG - 3));
    Best<unsigned> best{0, 0u};
    unsigned long long ws = 0;
    const int* cp = a.col + rs;
    const int* wp = a.w + rs;
    if (rd <= 64)
      sketch_row<32, 2, 8, WT, true, FIRST, unsigned>(a, rv, ro, cp, wp, nullptr, rd, lane, mem, rounds, pol, best, ws, &sh.warp);
    else if (rd <= 128)
      sketch_row<32, 4, 9, WT, true, FIRST, unsigned>(a, rv, ro, cp, wp, nullptr, rd, lane, mem, rounds, pol, best, ws, &sh.warp);
    else
      sketch_row<32, 8, 10, WT, true, FIRST, unsigned>(a, rv, ro, cp, wp, nullptr, rd, lane, mem, rounds, pol, best, ws, &sh.warp);
    __syncwarp();
    if (WT && FIRST && warp_sum_u64(ws) >= (1ull << 31)) raise_err(&a.ctr->err, ERRBIT_OVERFLOW);
    if (lane == r) nl = best.sum ? (int)~best.inv : ro;
  }
  const bool changed = act && nl != old;
  if (act) {
    __stcg(a.next + v, nl);
    my_act += 1;
    my_scan += (unsigned long long)d;
    my_dn += changed ? 1u : 0u;
    if (changed && a.mark) a.fnext[v] = 1;
  }
  const unsigned chm = __ballot_sync(FULL, changed);
  if (a.mark) solo_mark(a, chm, s, d);
}

// One sweep over a listed long row, by the whole block (list: its label list,
// for rows that the registers do not hold).
template <int WT, bool FIRST>
__device__ __forceinline__ void solo_long(const SweepArgs& a, int v, unsigned char* fcur, bool all_active, int* list,
                                          SoloShared& sh, int rounds, const Pol& pol, unsigned& my_dn,
                                          unsigned& my_act, unsigned long long& my_scan) {
  __syncthreads();   // the previous row's last reads of sh and the table
  const bool act = all_active || __ldcg(fcur + v) != 0;
  __syncthreads();   // every thread has read the flag
  if (!act) return;  // block-uniform
  const int tid = threadIdx.x;
  if (!all_active && tid == 0) fcur[v] = 0;
  const long long s = a.off[v];
  const int d = (int)(a.off[v + 1] - s);
  const int old = own_label<true>(a, v);
  Best<unsigned> best{0, 0u};
  unsigned long long ws = 0;
  const int* cp = a.col + s;
  const int* wp = a.w + s;
  if (d > SOLO_REG_ROW)
    sketch_long_row<SOLO_BLOCK, SOLO_LG, WT, true, FIRST, unsigned>(a, v, cp, wp, nullptr, d, tid, sh.counters, list,
                                                                    3 * SOLO_ROW_MAX, rounds, pol, best, ws, &sh.team);
  else if (d <= SOLO_BLOCK * 8)
    sketch_row<SOLO_BLOCK, 8, SOLO_LG - 1, WT, true, FIRST, unsigned>(a, v, old, cp, wp, nullptr, d, tid, sh.counters, rounds,
                                                            pol, best, ws, &sh.team);
  else
    sketch_row<SOLO_BLOCK, 16, SOLO_LG, WT, true, FIRST, unsigned>(a, v, old, cp, wp, nullptr, d, tid, sh.counters, rounds, pol,
                                                         best, ws, &sh.team);
  if (WT && FIRST) {
    ws = warp_sum_u64(ws);
    __syncthreads();
    if (tid == 0) sh.team.wsum = 0;
    __syncthreads();
    if ((tid & 31) == 0 && ws) atomicAdd(&sh.team.wsum, ws);
    __syncthreads();
    if (tid == 0 && sh.team.wsum >= (1ull << 31)) raise_err(&a.ctr->err, ERRBIT_OVERFLOW);
  }
  const int nl = best.sum ? (int)~best.inv : old;
  const bool changed = nl != old;   // block-uniform
  if (tid == 0) {
    __stcg(a.next + v, nl);
    my_act += 1;
    my_scan += (unsigned long long)d;
    my_dn += changed ? 1u : 0u;
    if (changed && a.mark) a.fnext[v] = 1;
  }
  if (changed && a.mark) {
    for (int e = tid; e < d; e += SOLO_BLOCK) {
      const int j = __ldg(cp + e);
      if ((unsigned)j < (unsigned)a.n) a.fnext[j] = 1;
    }
  }
}

template <int WT, bool FIRST>
__device__ __forceinline__ void solo_sweep(const SweepArgs& a, const SoloArgs& q, int t, int tsh, unsigned nlong,
                                           unsigned nhuge, unsigned char* fcur, bool all_active, SoloShared& sh,
                                           GroupSlots<unsigned>* slots, int rounds, const Pol& pol) {
  unsigned my_dn = 0, my_act = 0;
  unsigned long long my_scan = 0;
  // the longest rows on the last blocks that have a list, the others from the first block on
  const unsigned back = gridDim.x - 1 - blockIdx.x;
  const unsigned lists = min((unsigned)SOLO_LISTS, gridDim.x);
  if (back < lists)
    for (unsigned i = back; i < nhuge; i += lists)
      solo_long<WT, FIRST>(a, __ldcg(q.longs + a.n - 1 - i), fcur, all_active, q.lists + (long long)back * 3 * SOLO_ROW_MAX,
                           sh, rounds, pol, my_dn, my_act, my_scan);
  for (unsigned i = blockIdx.x; i < nlong; i += gridDim.x)
    solo_long<WT, FIRST>(a, __ldcg(q.longs + i), fcur, all_active, nullptr, sh, rounds, pol, my_dn, my_act, my_scan);
  __syncthreads();   // the warps' tables overlie the block's
  const long long warp = (long long)blockIdx.x * SOLO_WARPS + (threadIdx.x >> 5), nwarps = (long long)gridDim.x * SOLO_WARPS;
  for (long long base = warp << tsh; base < a.n; base += nwarps << tsh)
    solo_tile<WT, FIRST>(a, base, 1 << tsh, fcur, all_active, sh, slots, rounds, pol, my_dn, my_act, my_scan);
  solo_flush(sh, q.state, t, my_dn, my_act, my_scan);
}

}  // namespace

// q.max_iters sweeps at most from labels_init (or the identity) when q.lpa,
// then the split of the labels (or of q.labels_in) when q.split.
template <int WT>
__global__ void __launch_bounds__(SOLO_BLOCK, SOLO_BLOCKS_PER_SM) solo_kernel(SweepArgs a0, SoloArgs q) {
  __shared__ SoloShared sh;
  __shared__ GroupSlots<unsigned> groups[WT ? SOLO_WARPS : 1];
  SoloState* st = q.state;
  unsigned gen = 0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const Pol pol = make_pol();
  const long long n = a0.n;
  const long long stride = (long long)gridDim.x * blockDim.x, first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (first == 0) st->time_ns[0] = global_ns();
  if (WT) {
    for (int k = lane; k < GROUP_SLOTS; k += 32) groups[wid].sum[k] = 0;
    __syncwarp();
  }
  GroupSlots<unsigned>* slots = WT ? groups + wid : groups;
  // offsets checked, long rows listed, labels and parents set
  long long longest = 0;
  int bad = 0;
  for (long long v = first; v < n; v += stride) {
    const long long s = a0.off[v], e = a0.off[v + 1];
    if (s < 0 || e < s || e > q.nnz || (v == 0 && s != 0) || (v == n - 1 && e != q.nnz)) bad = ERRBIT_INVALID;
    else if (e - s > longest) longest = e - s;
    if (!bad && e - s > SOLO_REG_ROW) {
      q.longs[n - 1 - (long long)atomicAdd(&st->nhuge, 1u)] = (int)v;
      const unsigned long long all = atomicAdd(&st->huge_entries, (unsigned long long)(e - s)) + (unsigned long long)(e - s);
      if (all > SOLO_HUGE_ENTRIES) longest = SOLO_ROW_MAX + 1;   // left to the class kernels
    }
    else if (!bad && e - s > SOLO_WARP_ROW) q.longs[atomicAdd(&st->nlong, 1u)] = (int)v;
    if (q.lpa) {
      int x = (int)v;
      if (q.labels_init) {
        x = q.labels_init[v];
        if (x < 0 || x >= n) {
          bad |= ERRBIT_INVALID;
          x = (int)v;
        }
      }
      __stcg(q.lab[0] + v, x);
      __stcg(q.lab[1] + v, x);
      q.flag[0][v] = 0;
      q.flag[1][v] = 0;
    }
    if (q.split) {
      __stcg(q.parent + v, (int)v);
      __stcg(q.named + v, -1);
    }
  }
  // one atomic per block: thousands on one address would take longer than a sweep
  if (threadIdx.x == 0) sh.sums[0] = 0;
  __syncthreads();
  const unsigned top = __reduce_max_sync(FULL, (unsigned)(longest > SOLO_ROW_MAX ? SOLO_ROW_MAX + 1 : longest));
  if (lane == 0 && top) atomicMax(&sh.sums[0], (unsigned long long)top);
  if (bad) atomicOr(&a0.ctr->err, bad);
  __syncthreads();
  if (threadIdx.x == 0 && sh.sums[0]) atomicMax(&st->longest, (long long)sh.sums[0]);
  if (!grid_sync(st, &a0.ctr->err, gen)) return;
  const unsigned nlong = ld_acquire(&st->nlong), nhuge = ld_acquire(&st->nhuge);
  const int rounds = a0.probe_cap < SKETCH_ROUNDS ? a0.probe_cap : SKETCH_ROUNDS;
  const int* labels = q.labels_in;
  int tsh = 0;   // log2 of the vertices a warp takes in one step: the most that leave no warp without a full step
  while (tsh < 5 && (n >> (tsh + 1)) >= (long long)gridDim.x * SOLO_WARPS) ++tsh;
  if (q.lpa) {
    int t = 0, converged = 0;
    bool marked = false;
    unsigned long long dn = (unsigned long long)n;
    while (t < q.max_iters) {
      ++t;
      SweepArgs a = a0;
      a.prev = q.lab[(t - 1) & 1];
      a.next = q.lab[t & 1];
      a.fnext = q.flag[(t + 1) & 1];
      a.ident = t == 1 && !q.labels_init;
      a.check = t == 1;
      a.spread = t == 2 && !q.labels_init;
      a.mark = t > 1 && 2 * dn <= (unsigned long long)n;
      const bool all_active = t == 1 || !marked;
      unsigned char* fcur = q.flag[t & 1];
      if (t == 1) solo_sweep<WT, true>(a, q, t, tsh, nlong, nhuge, fcur, all_active, sh, slots, rounds, pol);
      else solo_sweep<WT, false>(a, q, t, tsh, nlong, nhuge, fcur, all_active, sh, slots, rounds, pol);
      if (!grid_sync(st, &a0.ctr->err, gen)) return;
      dn = __ldcg(&st->changed[t - 1]);
      marked = a.mark != 0;
      if ((double)dn / (double)n <= q.tol) {
        converged = 1;
        break;
      }
    }
    if (first == 0) {
      st->sweeps = t;
      st->converged = converged;
      st->time_ns[1] = global_ns();
    }
    labels = q.lab[t & 1];
  }
  if (!q.split) {
    for (long long v = first; v < n; v += stride) q.out[v] = __ldcg(labels + v);
    return;
  }
  // split: every vertex links with its first same-community neighbours, every
  // community names a piece, and only vertices outside it offer the rest of
  // their rows (as split_kernels.cu does)
  const UfCap<UF_CAP> cap{0};
  int* err = &a0.ctr->err;
  for (long long u = first; u < n; u += stride) {
    const long long s = a0.off[u], e = a0.off[u + 1];
    const int cu = __ldcg(labels + u);
    int linked = 0;
    for (long long k = s; k < e && k < s + SOLO_SCAN && linked < SOLO_SAMPLE; ++k) {
      const int j = __ldg(a0.col + k);
      if ((unsigned)j >= (unsigned)n) {
        raise_err(err, ERRBIT_INVALID);
      } else if (j != (int)u && __ldcg(labels + j) == cu) {
        uf_unite(q.parent, (int)u, j, err, cap);
        ++linked;
      }
    }
  }
  if (!grid_sync(st, &a0.ctr->err, gen)) return;
  for (long long v = first; v < n; v += stride) {
    const int r = uf_find(q.parent, (int)v, err, cap);
    if (r != (int)v) __stcg(q.named + comm_slot(__ldcg(labels + v), n), r);   // as name_pieces_kernel
  }
  if (!grid_sync(st, &a0.ctr->err, gen)) return;
  // rows of more than SOLO_WARP_ROW entries by a block each, until their vertex
  // is inside the named piece (400,000 vertices, a few of them with up to 20,000
  // entries, in 1000 communities: 0.52 ms with a warp over each row, 0.22 so)
  for (unsigned i = blockIdx.x; i < nlong + nhuge; i += gridDim.x) {
    const int u = __ldcg(q.longs + (i < nlong ? (long long)i : n - 1 - (long long)(i - nlong)));
    const int cu = __ldcg(labels + u);
    __syncthreads();   // the previous row's last read of the name
    if (threadIdx.x == 0) {
      const int root = uf_find(q.parent, u, err, cap);
      const int name = community_name(q.named + comm_slot(cu, n), root);
      sh.team.cnt = (unsigned)name;
      sh.team.next = name == root ? 0 : a0.off[u + 1];
    }
    __syncthreads();
    const int name = (int)sh.team.cnt;
    const long long e = sh.team.next;   // 0: inside it already
    for (long long k = a0.off[u] + SOLO_SAMPLE + threadIdx.x; k < e; k += SOLO_BLOCK) {
      if (__ldcg(q.parent + u) == name) break;
      const int j = __ldg(a0.col + k);
      if ((unsigned)j >= (unsigned)n) raise_err(err, ERRBIT_INVALID);
      else if (j != u && __ldcg(labels + j) == cu) uf_unite(q.parent, u, j, err, cap);
    }
  }
  const long long nwarps = stride >> 5;
  for (long long base = (first >> 5) << tsh; base < n; base += nwarps << tsh) {   // warp-uniform
    const long long u = base + lane;
    long long s = 0, e = 0;
    int cu = 0;
    bool offer = false;
    if (lane < (1 << tsh) && u < n) {
      s = a0.off[u] + SOLO_SAMPLE;
      e = a0.off[u + 1];
      cu = __ldcg(labels + u);
      if (s < e && e - s <= SOLO_WARP_ROW - SOLO_SAMPLE) {
        const int root = uf_find(q.parent, (int)u, err, cap);
        offer = root != community_name(q.named + comm_slot(cu, n), root);
      }
    }
    unsigned mask = __ballot_sync(FULL, offer);
    while (mask) {
      const int r = __ffs((int)mask) - 1;
      mask &= mask - 1;
      const long long rs = __shfl_sync(FULL, s, r), re = __shfl_sync(FULL, e, r);
      const int rc = __shfl_sync(FULL, cu, r), ru = (int)base + r;
      for (long long k = rs + lane; k < re; k += 32) {
        const int j = __ldg(a0.col + k);
        if ((unsigned)j >= (unsigned)n) raise_err(err, ERRBIT_INVALID);
        else if (j != ru && __ldcg(labels + j) == rc) uf_unite(q.parent, ru, j, err, cap);
      }
      __syncwarp();
    }
  }
  if (!grid_sync(st, &a0.ctr->err, gen)) return;
  unsigned pieces = 0;
  for (long long v = first; v < n; v += stride) {
    const int r = uf_find(q.parent, (int)v, err, cap);
    q.out[v] = r;
    pieces += r == (int)v ? 1u : 0u;
  }
  pieces = __reduce_add_sync(FULL, pieces);
  if (lane == 0 && pieces) atomicAdd(&st->pieces, (unsigned long long)pieces);
  if (first == 0) st->time_ns[2] = global_ns();
}

cudaError_t launch_solo(const SweepArgs& a, const SoloArgs& q, int weights, const DeviceInfo& di, cudaStream_t s) {
  const void* fn = weights ? (const void*)solo_kernel<1> : (const void*)solo_kernel<0>;
  // four vertices per warp until the grid is full (in steps of one to four,
  // tsh): several rows' loads are in flight together, and the barrier is cheaper
  // with fewer blocks; a block per
  // SOLO_BLOCK_ENTRIES entries where few rows hold many (the complete graph of
  // 1000 vertices: 0.10 ms a call instead of 0.25 with its 32 blocks, of 2000
  // 0.12 instead of 0.35)
  long long blocks = std::max((a.n + 4 * SOLO_WARPS - 1) / (4 * SOLO_WARPS), q.nnz / SOLO_BLOCK_ENTRIES);
  const long long most = (long long)SOLO_BLOCKS_PER_SM * di.sm_count;
  if (blocks > most) blocks = most;
  void* args[] = {const_cast<SweepArgs*>(&a), const_cast<SoloArgs*>(&q)};
  const cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3((unsigned)blocks), dim3(SOLO_BLOCK), args, 0, s);
  count_launches(1);
  return e;
}

}  // namespace gsl

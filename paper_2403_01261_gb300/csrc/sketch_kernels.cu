// sketch_kernels.cu -- the sweep for rows of more than 32 entries (classes
// 6..8, and class 9 where the hub kernels do not take it).
//
// A team (one warp, or a block of 128 or 256 threads) takes a row, keeps its
// neighbours' labels in registers and adds every entry's weight to the
// counter its label hashes to.  The adds return running sums, so the largest
// (sum, smallest label) over the team names the fullest counter and a label
// in it.  When no other label of the row lies in that counter, its sum is
// that label's and no other label can reach it (its own counter is no fuller,
// and a counter as full gives a larger label or is shared): one round, no
// probing, no compare-and-swap, no match.  Otherwise the named label is summed
// exactly, labels whose counters cannot beat it drop out, and the rest is
// settled in rounds that also leave a label per slot (sketch_rounds): slots
// that end up with one label hold its exact sum.
//
// Rows longer than the registers hold (4096 entries) keep their labels in a
// scratch list of the block; if many of them stay open (labels of about the
// same weight, as in the early sweeps over weighted graphs), those are moved
// into parts by a second hash and counted part by part.
//
// Bound by instruction issue and the label gathers: the hash tables before
// spent 150 to 210 warp instructions per 32 entries (compare-and-swap 5
// cycles of an SM, match up to 64, a counter add 2.6).
#include "sketch_device.cuh"

namespace gsl {

namespace {

constexpr int K_WARP = 8, K_SMALL = 8, K_BLOCK = 16;               // entries per thread
constexpr int T_SMALL = 128, T_BLOCK = 256;                         // threads per row (class 6: a warp)
constexpr int LG_WARP = 10, LG_SMALL = 11, LG_BLOCK = 13;           // counters per row (log2)
constexpr int BLOCKS_PER_SM = 4;                                    // of T_BLOCK threads

template <int T>
constexpr int team_lg() { return T == 32 ? LG_WARP : (T == T_SMALL ? LG_SMALL : LG_BLOCK); }

// A row's total weight from the first sweep, for the majority filter of later ones.
template <int WT>
__device__ __forceinline__ void store_row_total(const SweepArgs& a, int v, unsigned long long ws) {
  if (WT == 1 && ws >= (1ull << 31)) raise_err(&a.ctr->err, ERRBIT_OVERFLOW);
  if (a.kw) a.kw[v] = WT == 2 ? (unsigned)(ws >> 22) + 1u : (ws < (1ull << 32) ? (unsigned)ws : ~0u);
}

}  // namespace

// A warp per row (class 6): up to 32 rows' metadata and results per warp, one
// row per lane, as in tile_sweep_kernel.
template <int WT, bool ASYNC, bool GENERAL>
__global__ void __launch_bounds__(256, 4) sketch_warp_kernel(SweepArgs a, int cls) {
  using S = typename SumOf<WT>::T;
  if (stopped(a)) return;
  extern __shared__ int4 smem_sketch[];
  __shared__ TeamShared<32, S> sh;   // not written by warps
  const int lane = threadIdx.x & 31;
  unsigned* mem = reinterpret_cast<unsigned*>(smem_sketch) + ((size_t)(threadIdx.x >> 5) << LG_WARP);
  const unsigned cnt = a.ctr->cls_count[cls];
  const int* work = class_work(a, cls);
  const Pol pol = make_pol();
  const int rounds = a.probe_cap < SKETCH_ROUNDS ? a.probe_cap : SKETCH_ROUNDS;
  const unsigned nwarps = (gridDim.x * blockDim.x) >> 5, warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  unsigned per = 32;   // rows per tile: fewer for short worklists
  while (per > 1 && cnt / per < 4u * nwarps) per >>= 1;
  unsigned long long my_dn = 0, my_scan = 0;
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
    for (int r = 0; r < rows; ++r) {
      const long long rs = __shfl_sync(FULL, s, r);
      const int rv = __shfl_sync(FULL, v, r), rd = __shfl_sync(FULL, d, r), ro = __shfl_sync(FULL, old, r);
      const int* cp = a.col + rs;
      const int* wp = a.w + rs;
      const int* lp = a.lg ? a.lg + rs : nullptr;
      Best<S> best{0, 0u};
      unsigned long long ws = 0;
      if (rd <= 64)
        sketch_row<32, 2, 8, WT, ASYNC, GENERAL, S>(a, rv, ro, cp, wp, lp, rd, lane, mem, rounds, pol, best, ws, &sh);
      else if (rd <= 128)
        sketch_row<32, 4, 9, WT, ASYNC, GENERAL, S>(a, rv, ro, cp, wp, lp, rd, lane, mem, rounds, pol, best, ws, &sh);
      else
        sketch_row<32, K_WARP, LG_WARP, WT, ASYNC, GENERAL, S>(a, rv, ro, cp, wp, lp, rd, lane, mem, rounds, pol, best,
                                                               ws, &sh);
      if (WT && GENERAL && a.check) {
        ws = warp_sum_u64(ws);
        if (lane == 0) store_row_total<WT>(a, rv, ws);
      }
      if (lane == r && best.sum) nl = (int)~best.inv;
      __syncwarp();   // the table's last reads before it is cleared
    }
    const bool changed = mine && nl != old;
    if (mine) {
      store_label<ASYNC>(a, v, nl, changed);
      my_scan += (unsigned long long)d;
      my_dn += changed ? 1ull : 0ull;
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
        for (int e = lane; e < rd; e += 32) {
          const int j = ld_stream(a.col + rs + e, pol.stream);
          if ((unsigned)j < (unsigned)a.n) a.fnext[j] = 1;
        }
      }
    }
  }
  flush_counters(a.ctr, cls, my_dn, my_scan);
}

// Rows of class cls, a block of T threads each: up to T * K entries in
// registers (fewer per thread on shorter rows), longer ones (T_BLOCK only)
// through the block's scratch region.  Blocks take rows from a counter; the
// first hub_blocks blocks of T_BLOCK threads take the rows of class 9 before
// those of cls, so that the longest rows run beside the others.
template <int T, int WT, bool ASYNC, bool GENERAL>
__global__ void __launch_bounds__(T, T == T_SMALL ? 8 : BLOCKS_PER_SM) sketch_kernel(SweepArgs a, int cls) {
  using S = typename SumOf<WT>::T;
  if (stopped(a)) return;
  extern __shared__ int4 smem_sketch[];
  __shared__ TeamShared<T, S> sh;
  const int tid = (int)threadIdx.x;
  unsigned* mem = reinterpret_cast<unsigned*>(smem_sketch);
  bool hubs = T == T_BLOCK && (int)blockIdx.x < a.hub_blocks;
  int now = hubs ? CLS_HUB : cls;
  unsigned cnt = a.ctr->cls_count[now];
  const int* work = class_work(a, now);
  const Pol pol = make_pol();
  const int rounds = a.probe_cap < SKETCH_ROUNDS ? a.probe_cap : SKETCH_ROUNDS;
  unsigned long long my_dn = 0, my_scan = 0, hub_scan = 0;
  int vn = 0;
  long long sn = 0, en = 0;
  auto fetch = [&](long long item) {
    if (item < (long long)cnt) {
      vn = work[item];
      sn = a.off[vn];
      en = a.off[vn + 1];
    }
  };
  long long item = 0;
  auto take = [&] {   // the next row, from the class's counter
    __syncthreads();   // the previous row's last reads of sh and the table
    if (threadIdx.x == 0) sh.next = (long long)atomicAdd(&a.ctr->row_next[now], 1u);
    __syncthreads();
    return sh.next;
  };
  item = take();
  fetch(item);
  for (;;) {
    if (item >= (long long)cnt) {   // block-uniform
      if (!hubs) break;
      hubs = false;
      hub_scan = my_scan;
      my_scan = 0;
      now = cls;
      cnt = a.ctr->cls_count[now];
      work = class_work(a, now);
      item = take();
      fetch(item);
      continue;
    }
    const int v = vn;
    const long long s = sn;
    const int d = (int)(en - sn);
    item = take();
    fetch(item);
    const int old = own_label<ASYNC>(a, v);
    const int* cp = a.col + s;
    const int* wp = a.w + s;
    const int* lp = a.lg ? a.lg + s : nullptr;
    Best<S> best{0, 0u};
    unsigned long long ws = 0;
    if (T == T_SMALL) {
      if (d <= T * K_SMALL / 2)
        sketch_row<T, K_SMALL / 2, LG_SMALL, WT, ASYNC, GENERAL, S>(a, v, old, cp, wp, lp, d, tid, mem, rounds, pol,
                                                                    best, ws, &sh);
      else
        sketch_row<T, K_SMALL, LG_SMALL, WT, ASYNC, GENERAL, S>(a, v, old, cp, wp, lp, d, tid, mem, rounds, pol, best,
                                                                ws, &sh);
    } else {
      if (d <= T * K_BLOCK / 2)
        sketch_row<T, K_BLOCK / 2, LG_BLOCK - 1, WT, ASYNC, GENERAL, S>(a, v, old, cp, wp, lp, d, tid, mem, rounds,
                                                                        pol, best, ws, &sh);
      else if (d <= T * K_BLOCK)
        sketch_row<T, K_BLOCK, LG_BLOCK, WT, ASYNC, GENERAL, S>(a, v, old, cp, wp, lp, d, tid, mem, rounds, pol, best,
                                                                ws, &sh);
      else
        sketch_long_row<T, LG_BLOCK, WT, ASYNC, GENERAL, S>(
            a, v, cp, wp, lp, d, tid, mem,
            hubs ? a.hub_scratch + (long long)blockIdx.x * a.hub_region
                 : a.scratch + (long long)blockIdx.x * a.scratch_region,
            hubs ? a.hub_region : a.scratch_region, rounds, pol, best, ws, &sh);
    }
    if (WT && GENERAL && a.check) {   // the row's total, for the majority filter of later sweeps
      ws = warp_sum_u64(ws);
      __syncthreads();
      if (tid == 0) sh.wsum = 0;
      __syncthreads();
      if ((tid & 31) == 0 && ws) atomicAdd(&sh.wsum, ws);
      __syncthreads();
      if (tid == 0) store_row_total<WT>(a, v, sh.wsum);
    }
    const int nl = best.sum ? (int)~best.inv : old;
    const bool changed = nl != old;   // block-uniform
    if (tid == 0) {
      store_label<ASYNC>(a, v, nl, changed);
      if (changed) count_graph_change(a, v);
      my_scan += (unsigned long long)d;
      my_dn += changed ? 1ull : 0ull;
    }
    if (changed && a.mark) {
      for (int e = tid; e < d; e += T) {
        const int j = ld_stream(cp + e, pol.stream);
        if ((unsigned)j < (unsigned)a.n) a.fnext[j] = 1;
      }
      if (!ASYNC && tid == 0) a.fnext[v] = 1;
    }
  }
  flush_counters(a.ctr, cls, my_dn, my_scan);
  if (T == T_BLOCK && a.hub_blocks) {
    __syncthreads();
    flush_counters(a.ctr, CLS_HUB, 0, hub_scan);
  }
}

namespace {
template <int T, int WT, bool A, bool G>
auto sketch_kernel_for() {
  if constexpr (T == 32) return &sketch_warp_kernel<WT, A, G>;
  else return &sketch_kernel<T, WT, A, G>;
}

template <int T, int WT, bool A, bool G>
cudaError_t launch_sketch_g(const SweepArgs& a, int cls, const DeviceInfo& di, cudaStream_t s) {
  constexpr int block = T == 32 ? 256 : T;
  const size_t smem = (sizeof(unsigned) << team_lg<T>()) * (size_t)(block / T);
  void (*const kernel)(SweepArgs, int) = sketch_kernel_for<T, WT, A, G>();
  // per host thread and device; the grid itself is formed anew on every launch
  thread_local int per_sm = 0, per_sm_of = -1;
  int dev = 0;
  if (cudaError_t e = cudaGetDevice(&dev)) return e;
  if (dev != per_sm_of) {
    if (cudaError_t e = raise_smem_limit((const void*)kernel, smem)) return e;
    if (cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, smem)) return e;
    per_sm_of = dev;
  }
  kernel<<<sketch_grid(per_sm, T == T_BLOCK, di), block, smem, s>>>(a, cls);
  count_launches(1);
  return cudaGetLastError();
}

template <int T, int WT>
cudaError_t launch_sketch_t(const SweepArgs& a, int cls, bool async_mode, const DeviceInfo& di, cudaStream_t s) {
  const bool general = a.check || a.ident || a.lg;
  if (async_mode)
    return general ? launch_sketch_g<T, WT, true, true>(a, cls, di, s)
                   : launch_sketch_g<T, WT, true, false>(a, cls, di, s);
  return general ? launch_sketch_g<T, WT, false, true>(a, cls, di, s)
                 : launch_sketch_g<T, WT, false, false>(a, cls, di, s);
}

template <int WT>
cudaError_t launch_sketch_w(const SweepArgs& a, int cls, int longest, bool async_mode, const DeviceInfo& di,
                            cudaStream_t s) {
  if (longest <= 32 * K_WARP) return launch_sketch_t<32, WT>(a, cls, async_mode, di, s);
  if (longest <= T_SMALL * K_SMALL) return launch_sketch_t<T_SMALL, WT>(a, cls, async_mode, di, s);
  return launch_sketch_t<T_BLOCK, WT>(a, cls, async_mode, di, s);
}
}  // namespace

long long sketch_blocks(const DeviceInfo& di) { return (long long)BLOCKS_PER_SM * di.sm_count; }
int sketch_grid(int per_sm, bool lists, const DeviceInfo& di) {
  const long long grid = (long long)(per_sm < 1 ? 1 : per_sm) * di.sm_count;
  return (int)(lists && grid > sketch_blocks(di) ? sketch_blocks(di) : grid);
}
long long sketch_register_row() { return (long long)T_BLOCK * K_BLOCK; }

cudaError_t launch_sketch(const SweepArgs& a, int cls, int longest, int weights, bool async_mode,
                          const DeviceInfo& di, cudaStream_t s) {
  if (weights == 0) return launch_sketch_w<0>(a, cls, longest, async_mode, di, s);
  if (weights == 1) return launch_sketch_w<1>(a, cls, longest, async_mode, di, s);
  return launch_sketch_w<2>(a, cls, longest, async_mode, di, s);
}

}  // namespace gsl

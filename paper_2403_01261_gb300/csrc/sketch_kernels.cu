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

}  // namespace

// Rows of class cls by teams of T threads: up to T * K entries in registers
// (fewer per thread on shorter rows), longer ones (T_BLOCK only) through the
// block's scratch region.  Warps take rows in strides, blocks from a counter;
// the first hub_blocks blocks of T_BLOCK threads take the rows of class 9
// before those of cls, so that the longest rows run beside the others.
template <int T, int WT, bool ASYNC, bool GENERAL>
__global__ void __launch_bounds__(T == 32 ? 256 : T, T == 32 ? 4 : (T == T_SMALL ? 8 : BLOCKS_PER_SM))
    sketch_kernel(SweepArgs a, int cls) {
  using S = typename SumOf<WT>::T;
  if (stopped(a)) return;
  extern __shared__ int4 smem_sketch[];
  __shared__ TeamShared<T, S> sh;
  const int tid = T == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  unsigned* mem = reinterpret_cast<unsigned*>(smem_sketch) + (T == 32 ? (size_t)(threadIdx.x >> 5) << team_lg<T>() : 0);
  bool hubs = T == T_BLOCK && (int)blockIdx.x < a.hub_blocks;
  int now = hubs ? CLS_HUB : cls;
  unsigned cnt = a.ctr->cls_count[now];
  const int* work = class_work(a, now);
  const Pol pol = make_pol();
  const int rounds = a.probe_cap < SKETCH_ROUNDS ? a.probe_cap : SKETCH_ROUNDS;
  unsigned long long my_dn = 0, my_scan = 0, hub_scan = 0;
  const long long nteams = ((long long)gridDim.x * blockDim.x) / T;
  long long item = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / T;
  int vn = 0;
  long long sn = 0, en = 0;
  auto fetch = [&] {
    if (item < (long long)cnt) {
      vn = work[item];
      sn = a.off[vn];
      en = a.off[vn + 1];
    }
  };
  auto take = [&] {   // a block's next row, from the class's counter
    __syncthreads();   // the previous row's last reads of sh and the table
    if (threadIdx.x == 0) sh.next = (long long)atomicAdd(&a.ctr->row_next[now], 1u);
    __syncthreads();
    return sh.next;
  };
  if (T != 32) item = take();
  fetch();
  for (;;) {
    if (item >= (long long)cnt) {   // team-uniform
      if (!hubs) break;
      hubs = false;
      hub_scan = my_scan;
      my_scan = 0;
      now = cls;
      cnt = a.ctr->cls_count[now];
      work = class_work(a, now);
      item = take();
      fetch();
      continue;
    }
    const int v = vn;
    const long long s = sn;
    const int d = (int)(en - sn);
    const long long next = T == 32 ? item + nteams : take();
    item = next;
    fetch();
    const int old = own_label<ASYNC>(a, v);
    const int* cp = a.col + s;
    const int* wp = a.w + s;
    const int* lp = a.lg ? a.lg + s : nullptr;
    Best<S> best{0, 0u};
    unsigned long long ws = 0;
    if (T == 32) {
      if (d <= 64)
        sketch_row<T, 2, 8, WT, ASYNC, GENERAL, S>(a, v, old, cp, wp, lp, d, tid, mem, rounds, pol, best, ws, &sh);
      else if (d <= 128)
        sketch_row<T, 4, 9, WT, ASYNC, GENERAL, S>(a, v, old, cp, wp, lp, d, tid, mem, rounds, pol, best, ws, &sh);
      else
        sketch_row<T, K_WARP, LG_WARP, WT, ASYNC, GENERAL, S>(a, v, old, cp, wp, lp, d, tid, mem, rounds, pol, best,
                                                              ws, &sh);
    } else if (T == T_SMALL) {
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
      if (T != 32) {
        __syncthreads();
        if (threadIdx.x == 0) sh.wsum = 0;
        __syncthreads();
        if ((threadIdx.x & 31) == 0 && ws) atomicAdd(&sh.wsum, ws);
        __syncthreads();
        ws = sh.wsum;
      }
      if (tid == 0) {
        if (WT == 1 && ws >= (1ull << 31)) raise_err(&a.ctr->err, ERRBIT_OVERFLOW);
        if (a.kw) a.kw[v] = WT == 2 ? (unsigned)(ws >> 22) + 1u : (ws < (1ull << 32) ? (unsigned)ws : ~0u);
      }
    }
    const int nl = best.sum ? (int)~best.inv : old;
    const bool changed = nl != old;   // team-uniform
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
    if (T == 32) __syncwarp();   // the table's last reads before it is cleared
  }
  flush_counters(a.ctr, cls, my_dn, my_scan);
  if (T == T_BLOCK && a.hub_blocks) {
    __syncthreads();
    flush_counters(a.ctr, CLS_HUB, 0, hub_scan);
  }
}

namespace {
template <int T, int WT, bool A, bool G>
cudaError_t launch_sketch_g(const SweepArgs& a, int cls, const DeviceInfo& di, cudaStream_t s) {
  constexpr int block = T == 32 ? 256 : T;
  const size_t smem = (sizeof(unsigned) << team_lg<T>()) * (size_t)(block / T);
  thread_local int grid = 0;
  if (!grid) {
    if (cudaError_t e = raise_smem_limit((const void*)sketch_kernel<T, WT, A, G>, smem)) return e;
    int per_sm = 0;
    if (cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sketch_kernel<T, WT, A, G>, block, smem))
      return e;
    grid = (per_sm < 1 ? 1 : per_sm) * di.sm_count;
    if (T == T_BLOCK && grid > sketch_blocks(di)) grid = (int)sketch_blocks(di);   // one scratch region each
  }
  sketch_kernel<T, WT, A, G><<<grid, block, smem, s>>>(a, cls);
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
long long sketch_register_row() { return (long long)T_BLOCK * K_BLOCK; }

cudaError_t launch_sketch(const SweepArgs& a, int cls, int longest, int weights, bool async_mode,
                          const DeviceInfo& di, cudaStream_t s) {
  if (weights == 0) return launch_sketch_w<0>(a, cls, longest, async_mode, di, s);
  if (weights == 1) return launch_sketch_w<1>(a, cls, longest, async_mode, di, s);
  return launch_sketch_w<2>(a, cls, longest, async_mode, di, s);
}

}  // namespace gsl

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
#include "tile_device.cuh"

namespace gsl {

namespace {

constexpr int TILE_BLOCK = 256;
constexpr int TILE_MIN_BLOCKS = 4;   // 64 registers: four steps of loads in flight per warp, 32 warps per SM
constexpr int LANE_MIN_BLOCKS = 8;   // 32 registers

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

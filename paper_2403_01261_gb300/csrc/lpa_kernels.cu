// lpa_kernels.cu -- the label-propagation sweep of GSL-LPA on sm_103a.
//
// One sweep applies Eq. 2 (C_i = argmax_c sum_{j in J_i, C_j = c} w_ij,
// scanCommunities() of Algorithm 3 skipping j == i) to every vertex of the
// frontier, with ties going to the smallest label.  Integer weights make the
// per-label sums exact and the argmax a max over the packed 64-bit key
// (sum << 32 | ~label), so the result does not depend on the order in which
// threads add: the synchronous sweep is deterministic.
//
// Work is split by degree class (binning pass below):
//   d <= 32          one lane, half a warp or a warp per row (tile_kernels.cu)
//   d <= warp_small  one warp per row      (sketch_kernels.cu)
//   d <= warp_max    128 threads per row   (the same)
//   d <= blk_max     256 threads per row   (the same)
//   larger           beside those, or in thread-block clusters and pieces
//                    (hub_kernels.cu)
// Small graphs run whole in one launch (solo_kernel.cu).  This file holds the
// classification, the binning and the streamed first sweep.
//
// Pruning (lpaMove(): a processed vertex is re-marked when a neighbour
// changes): a vertex whose label changes sets the next-frontier flag of each
// neighbour and, in synchronous mode, of itself (the double buffer then
// stays consistent for unprocessed vertices).  Eq. 2 depends on neighbour
// labels only, so skipping the other vertices gives the same labels as a
// full sweep.
#include <atomic>
#include <mutex>
#include <unordered_map>

#include "sweep_device.cuh"

namespace gsl {


// ---------------------------------------------------------------------------
// Static classification of all vertices: class totals, region starts, max
// degree; validates the offsets array.
__global__ void class_histogram_kernel(const long long* __restrict__ off, long long n, long long nnz, ClassBounds cb,
                                       Counters* ctr) {
  __shared__ unsigned long long hist[NCLASS];
  __shared__ unsigned long long hub_e;
  __shared__ long long maxd;
  __shared__ int bad;
  if (threadIdx.x < NCLASS) hist[threadIdx.x] = 0;
  if (threadIdx.x == 0) { maxd = 0; bad = 0; hub_e = 0; }
  __syncthreads();
  long long lmax = 0;
  int lbad = 0;
  // whole warps step together (the bound is warp-uniform), so that equal
  // classes are counted with one shared atomic per warp
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long v0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
  for (long long w = v0; w < n; w += stride) {
    const long long v = w + (threadIdx.x & 31);
    int c = -1;
    if (v < n) {
      const long long s = off[v], e = off[v + 1];
      if (s < 0 || e < s || e > nnz) {
        lbad |= ERRBIT_INVALID;
      } else if (e - s >= (1ll << 31)) {
        lbad |= ERRBIT_OVERFLOW;
      } else {
        const long long d = e - s;
        lmax = d > lmax ? d : lmax;
        c = degree_class(d, cb.warp_small, cb.warp_max, cb.blk_max);
        if (c == CLS_HUB) atomicAdd(&hub_e, (unsigned long long)d);
      }
      if (v == 0 && s != 0) lbad |= ERRBIT_INVALID;
      if (v == n - 1 && e != nnz) lbad |= ERRBIT_INVALID;
    }
    const unsigned m = __match_any_sync(FULL, c);
    if (c >= 0 && (m & lanemask_lt()) == 0) atomicAdd(&hist[c], (unsigned long long)__popc(m));
  }
  if (lmax) atomicMax(&maxd, lmax);
  if (lbad) atomicOr(&bad, lbad);
  __syncthreads();
  if (threadIdx.x < NCLASS && hist[threadIdx.x]) atomicAdd(&ctr->cls_total[threadIdx.x], hist[threadIdx.x]);
  if (threadIdx.x == 0) {
    if (maxd) atomicMax(&ctr->max_degree, maxd);
    if (hub_e) atomicAdd(&ctr->hub_entries, hub_e);
    if (bad) atomicOr(&ctr->err, bad);
  }
}

__global__ void class_starts_kernel(Counters* ctr) {
  unsigned long long run = 0;
  for (int c = 0; c < NCLASS; ++c) {
    ctr->cls_start[c] = run;
    run += ctr->cls_total[c];
  }
}

// ---------------------------------------------------------------------------
// Frontier binning: every vertex with its flag set (or every vertex when
// all_active) is appended to its class region; the flag is cleared, which
// leaves the flag array zeroed for reuse as the frontier after next.  With
// phase >= 0 only the vertices of that phase (sweep_phase) are taken; the
// flags of the others stay set for the binning of the other phase.
// PHASED is a template flag so that the one-phase binning of synchronous
// sweeps carries no phase test.
constexpr int BIN_ITEMS = 8;
constexpr int BIN_BLOCKS = 6;   // resident 256-thread blocks per SM (40 registers); the grid is no larger

template <bool PHASED>
__global__ void __launch_bounds__(256, BIN_BLOCKS) bin_kernel(const long long* __restrict__ off, long long n,
                                                   unsigned char* __restrict__ fcur, int all_active, ClassBounds cb,
                                                   int* __restrict__ work, Counters* ctr, const int* __restrict__ gid,
                                                   const unsigned char* __restrict__ done, const int* stop, int phase,
                                                   unsigned seed, int first_cls) {
  if (stop && *(volatile const int*)stop) return;
  __shared__ unsigned cnt[NCLASS];
  __shared__ unsigned base[NCLASS];
  const long long tile = (long long)blockDim.x * BIN_ITEMS;
  for (long long t0 = (long long)blockIdx.x * tile; t0 < n; t0 += (long long)gridDim.x * tile) {
    if (threadIdx.x < NCLASS) cnt[threadIdx.x] = 0;
    __syncthreads();
    int cls[BIN_ITEMS];
    unsigned pos[BIN_ITEMS];
#pragma unroll
    for (int k = 0; k < BIN_ITEMS; ++k) {
      const long long v = t0 + (long long)k * blockDim.x + threadIdx.x;
      cls[k] = -1;
      if (v < n) {
        // classes below first_cls are swept in natural order: their flags stay
        const bool flagged = all_active != 0 || fcur[v] != 0;
        bool act = flagged && (!PHASED || sweep_phase(v, seed) == phase);
        if (act) {
          const int c = degree_class(off[v + 1] - off[v], cb.warp_small, cb.warp_max, cb.blk_max);
          if (c >= first_cls) {
            if (!all_active) fcur[v] = 0;
            if (gid && done[gid[v]]) act = false;   // batched: this vertex's graph has stopped
            if (act) cls[k] = c;
          }
        }
      }
    }
    // every item's class is known before any is counted, so that the
    // tile's offset loads are all in flight together
#pragma unroll
    for (int k = 0; k < BIN_ITEMS; ++k) {
      // one shared-memory add per class present in the warp
      const unsigned m = __match_any_sync(FULL, cls[k]);
      const int leader = __ffs(m) - 1;
      unsigned b = 0;
      if ((int)(threadIdx.x & 31) == leader && cls[k] >= 0) b = atomicAdd(&cnt[cls[k]], (unsigned)__popc(m));
      pos[k] = __shfl_sync(FULL, b, leader) + (unsigned)__popc(m & lanemask_lt());
    }
    __syncthreads();
    if (threadIdx.x < NCLASS) base[threadIdx.x] = cnt[threadIdx.x] ? atomicAdd(&ctr->cls_count[threadIdx.x], cnt[threadIdx.x]) : 0u;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BIN_ITEMS; ++k) {
      if (cls[k] >= 0) {
        const long long v = t0 + (long long)k * blockDim.x + threadIdx.x;
        work[ctr->cls_start[cls[k]] + base[cls[k]] + pos[k]] = (int)v;
      }
    }
    __syncthreads();
  }
}

__global__ void init_labels_kernel(const int* __restrict__ init, int* __restrict__ a, int* __restrict__ b, long long n,
                                   Counters* ctr) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    int x = (int)v;
    if (init) {
      x = init[v];
      if (x < 0 || x >= n) {
        raise_err(&ctr->err, ERRBIT_INVALID);
        x = (int)v;
      }
    }
    a[v] = x;
    if (b) b[v] = x;
  }
}

// ---------------------------------------------------------------------------
// Edge-parallel gather of a synchronous sweep's neighbour labels.  The class
// kernels hold hash tables in shared memory, which caps their occupancy,
// and they interleave dependent loads with hashing; this pass has neither:
// every thread keeps four independent gathers in flight at full occupancy,
// and the class kernels then read the labels as a coalesced stream.
__global__ void __launch_bounds__(256) pregather_kernel(const int* __restrict__ col, long long nnz,
                                                        const int* __restrict__ prev, long long n,
                                                        int* __restrict__ lg) {
  const unsigned long long ps = policy_evict_first(), pl = policy_evict_last();
  const long long st = (long long)gridDim.x * blockDim.x;
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + 3 * st < nnz; i += 4 * st) {
    int j[4], l[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) j[u] = ld_stream(col + i + u * st, ps);
#pragma unroll
    for (int u = 0; u < 4; ++u) l[u] = (unsigned)j[u] < (unsigned)n ? ld_label_ro(prev + j[u], pl) : -1;
#pragma unroll
    for (int u = 0; u < 4; ++u) __stcs(lg + i + u * st, l[u]);
  }
  for (; i < nnz; i += st) {
    const int j = ld_stream(col + i, ps);
    __stcs(lg + i, (unsigned)j < (unsigned)n ? ld_label_ro(prev + j, pl) : -1);
  }
}

cudaError_t launch_pregather(const int* col, long long nnz, const int* prev, long long n, int* lg,
                             const DeviceInfo& di, cudaStream_t s) {
  if (nnz <= 0) return cudaSuccess;
  long long blocks = (nnz + 255) / 256;
  const long long cap = 16ll * di.sm_count;
  pregather_kernel<<<(int)(blocks < cap ? blocks : cap), 256, 0, s>>>(col, nnz, prev, n, lg);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Sweep 1 from the identity labelling with unit weights, as three streaming
// passes instead of per-vertex row scans.  When a row is strictly
// increasing every neighbour label (its id) occurs once with weight 1, so
// Eq. 2's argmax with smallest-label ties is the smallest neighbour other
// than the vertex itself: the first entry of the row, or the second when
// the first is a self-loop.
//   1. rowstart_kernel: bit off[v] set for every non-empty row;
//   2. sorted_check_kernel: edge-parallel, flags every row that is not
//      strictly increasing and checks every column's range;
//   3. ident_first_kernel: writes the label of every unflagged row.
// Flagged rows keep their flag and are swept by the hash kernels.
__global__ void rowstart_kernel(const long long* __restrict__ off, long long n, unsigned* __restrict__ bits) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    const long long st = off[v];
    if (off[v + 1] > st) atomicOr(bits + (st >> 5), 1u << (st & 31));
  }
}

__device__ __forceinline__ long long row_of(const long long* off, long long n, long long e) {
  long long lo = 0, hi = n;   // largest r with off[r] <= e
  while (hi - lo > 1) {
    const long long mid = (lo + hi) >> 1;
    if (off[mid] <= e) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Entry e (column je) against entry e + 1 (column jn): the row is not
// strictly increasing if e + 1 continues e's row and jn <= je.  `end` is
// the end of the checked range, a row boundary (or nnz).  A flagged row
// also raises *any_bad when it is given.
__device__ __forceinline__ void check_order(const long long* off, long long n, long long end, const unsigned* bits,
                                            unsigned char* bad, unsigned* any_bad, long long e, int je, int jn) {
  const long long f = e + 1;
  if (f < end && ((__ldg(bits + (f >> 5)) >> (f & 31)) & 1u) == 0 && !(je < jn)) {
    bad[row_of(off, n, e)] = 1;
    if (any_bad && __ldcg(any_bad) == 0) atomicOr(any_bad, 1u);
  }
}

__device__ __forceinline__ void check_pair(const long long* off, long long n, long long end, const unsigned* bits,
                                           unsigned char* bad, unsigned* any_bad, Counters* ctr, long long e, int je,
                                           int jn) {
  if ((unsigned)je >= (unsigned)n) raise_err(&ctr->err, ERRBIT_INVALID);
  check_order(off, n, end, bits, bad, any_bad, e, je, jn);
}

// The entries [e0, e1) of a range that ends at a row boundary (the whole
// array: e0 = 0, e1 = nnz).  Sixteen entries per thread per round, as four
// 16-byte loads issued together; the few entries before the first 16-byte
// boundary and after the last whole quad are checked by one thread.  The
// entry after a thread's quad comes from the next lane (or the next quad
// row of the warp).  Entry indices (bits, rows, the quads' positions) are
// absolute.
__global__ void __launch_bounds__(256) sorted_check_kernel(const long long* __restrict__ off, long long n,
                                                            const int* __restrict__ col, long long e0, long long e1,
                                                            const unsigned* __restrict__ bits,
                                                            unsigned char* __restrict__ bad, unsigned* any_bad,
                                                            Counters* ctr) {
  const unsigned long long pol = policy_evict_first();
  const int lane = threadIdx.x & 31;
  const long long nnz = e1;   // the checked range ends here (a row boundary)
  long long head = e0 + ((long long)((16 - ((unsigned long long)(col + e0) & 15)) & 15) >> 2);   // 4-byte aligned
  if (head > nnz) head = nnz;
  const long long nq = (nnz - head) >> 2;
  const long long tail0 = head + 4 * nq;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid == 0) {
    for (long long e = e0; e < head; ++e)
      check_pair(off, n, nnz, bits, bad, any_bad, ctr, e, col[e], e + 1 < nnz ? col[e + 1] : 0);
    for (long long e = tail0; e < nnz; ++e)
      check_pair(off, n, nnz, bits, bad, any_bad, ctr, e, col[e], e + 1 < nnz ? col[e + 1] : 0);
  }
  const int4* cq = reinterpret_cast<const int4*>(col + head);
  const long long warp = tid >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long qb = warp * 128; qb < nq; qb += nwarps * 128) {   // warp-uniform; 128 quads per round
    int4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long q = qb + u * 32 + lane;
      v[u] = q < nq ? ld_stream4(cq + q, pol) : make_int4(0, 0, 0, 0);
    }
    const long long elast = head + 4 * (qb + 128);   // the entry after the round's last quad
    const int tailx = (lane == 31 && qb + 128 <= nq && elast < nnz) ? ld_stream(col + elast, pol) : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      int nx = __shfl_down_sync(FULL, v[u].x, 1);
      const int hx = u < 3 ? __shfl_sync(FULL, v[u < 3 ? u + 1 : u].x, 0) : tailx;
      if (lane == 31) nx = hx;
      const long long q = qb + u * 32 + lane;
      if (q < nq) {
        const long long e = head + 4 * q;
        if (q + 1 >= nq) nx = e + 4 < nnz ? col[e + 4] : 0;   // the next entry lies in the scalar tail
        const unsigned mx = max(max((unsigned)v[u].x, (unsigned)v[u].y), max((unsigned)v[u].z, (unsigned)v[u].w));
        if (mx >= (unsigned)n) raise_err(&ctr->err, ERRBIT_INVALID);
        // four increasing pairs need no row bounds: only a quad with a
        // descent (a row start, or a row out of order) is checked pair by pair
        if (!(v[u].x < v[u].y && v[u].y < v[u].z && v[u].z < v[u].w && (v[u].w < nx || e + 4 >= nnz))) {
          check_order(off, n, nnz, bits, bad, any_bad, e, v[u].x, v[u].y);
          check_order(off, n, nnz, bits, bad, any_bad, e + 1, v[u].y, v[u].z);
          check_order(off, n, nnz, bits, bad, any_bad, e + 2, v[u].z, v[u].w);
          check_order(off, n, nnz, bits, bad, any_bad, e + 3, v[u].w, nx);
        }
      }
    }
  }
}

__global__ void ident_first_kernel(const long long* __restrict__ off, long long n, const int* __restrict__ col,
                                   const unsigned char* __restrict__ bad, int* __restrict__ next, Counters* ctr) {
  unsigned long long my_dn = 0, my_scan = 0, my_act = 0;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    const long long st = off[v], d = off[v + 1] - st;
    if (d == 0 || bad[v]) continue;   // an empty row keeps its label, already in `next`
    my_act += 1;
    int nl = col[st];
    if (nl == (int)v) nl = d > 1 ? col[st + 1] : (int)v;
    if ((unsigned)nl >= (unsigned)n) nl = (int)v;   // out of range: reported by the check pass
    next[v] = nl;
    my_dn += nl != (int)v ? 1ull : 0ull;
    my_scan += (unsigned long long)d;
  }
  my_dn = warp_sum_u64(my_dn);
  my_scan = warp_sum_u64(my_scan);
  my_act = warp_sum_u64(my_act);
  if ((threadIdx.x & 31) == 0) {
    if (my_dn) atomicAdd(&ctr->dn, my_dn);
    if (my_scan) atomicAdd(&ctr->scanned, my_scan);
    if (my_act) atomicAdd(&ctr->fast_active, my_act);
  }
}

namespace {
// One wave of 256-thread blocks of `kernel`: as many as are resident at once
// (the streaming passes of sweep 1 use more registers than eight blocks per
// SM allow, and a second wave would run at part of the bandwidth).
template <typename K>
int one_wave_grid(K kernel, const DeviceInfo& di) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, 0) != cudaSuccess) {
    cudaGetLastError();
    per_sm = 0;
  }
  return (per_sm < 1 ? 1 : per_sm) * di.sm_count;
}
}  // namespace

cudaError_t launch_row_check(const long long* off, long long n, const int* col, long long nnz, unsigned* bits,
                             unsigned char* bad, Counters* ctr, const DeviceInfo& di, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int g = 8 * di.sm_count;
  thread_local int gc = 0;
  if (!gc) gc = one_wave_grid(sorted_check_kernel, di);
  cudaMemsetAsync(bits, 0, sizeof(unsigned) * (size_t)((nnz >> 5) + 1), s);
  rowstart_kernel<<<g, 256, 0, s>>>(off, n, bits);
  if (nnz > 0) sorted_check_kernel<<<gc, 256, 0, s>>>(off, n, col, 0, nnz, bits, bad, nullptr, ctr);
  count_launches(nnz > 0 ? 2 : 1);
  return cudaGetLastError();
}

cudaError_t launch_ident_stream(const long long* off, long long n, const int* col, long long nnz, unsigned* bits,
                                unsigned char* bad, int* next, Counters* ctr, const DeviceInfo& di, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (cudaError_t e = launch_row_check(off, n, col, nnz, bits, bad, ctr, di, s)) return e;
  thread_local int gi = 0;
  if (!gi) gi = one_wave_grid(ident_first_kernel, di);
  ident_first_kernel<<<gi, 256, 0, s>>>(off, n, col, bad, next, ctr);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Pieces of the first two sweeps while the columns are still arriving
// (gsl_gsllpa_host): the rows are cut into chunks at row boundaries, and a
// chunk's columns are checked and its rows swept as soon as it has landed.

// All-active binning of the rows [v0, v1) (sweep 2 runs on every vertex):
// appended to their class regions as bin_kernel does.
__global__ void __launch_bounds__(256) bin_range_kernel(const long long* __restrict__ off, long long v0, long long v1,
                                                         ClassBounds cb, int* __restrict__ work, Counters* ctr,
                                                         int first_cls) {
  __shared__ unsigned cnt[NCLASS];
  __shared__ unsigned base[NCLASS];
  const long long tile = (long long)blockDim.x * BIN_ITEMS;
  for (long long t0 = v0 + (long long)blockIdx.x * tile; t0 < v1; t0 += (long long)gridDim.x * tile) {
    if (threadIdx.x < NCLASS) cnt[threadIdx.x] = 0;
    __syncthreads();
    int cls[BIN_ITEMS];
    unsigned pos[BIN_ITEMS];
#pragma unroll
    for (int k = 0; k < BIN_ITEMS; ++k) {
      const long long v = t0 + (long long)k * blockDim.x + threadIdx.x;
      cls[k] = v < v1 ? degree_class(off[v + 1] - off[v], cb.warp_small, cb.warp_max, cb.blk_max) : -1;
      if (cls[k] < first_cls) cls[k] = -1;
      const unsigned m = __match_any_sync(FULL, cls[k]);
      const int leader = __ffs(m) - 1;
      unsigned b = 0;
      if ((int)(threadIdx.x & 31) == leader && cls[k] >= 0) b = atomicAdd(&cnt[cls[k]], (unsigned)__popc(m));
      pos[k] = __shfl_sync(FULL, b, leader) + (unsigned)__popc(m & lanemask_lt());
    }
    __syncthreads();
    if (threadIdx.x < NCLASS) base[threadIdx.x] = cnt[threadIdx.x] ? atomicAdd(&ctr->cls_count[threadIdx.x], cnt[threadIdx.x]) : 0u;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BIN_ITEMS; ++k) {
      if (cls[k] >= 0) {
        const long long v = t0 + (long long)k * blockDim.x + threadIdx.x;
        work[ctr->cls_start[cls[k]] + base[cls[k]] + pos[k]] = (int)v;
      }
    }
    __syncthreads();
  }
}

// Sweep 1 from the identity labelling on rows assumed strictly increasing,
// reading only each row's first entries, from `col` (which may be host
// memory the device can read): the labels and counts ident_first_kernel
// gives when no row is flagged.
cudaError_t launch_ident_first(const long long* off, long long n, const int* col, const unsigned char* zero_flags,
                               int* next, Counters* ctr, const DeviceInfo& di, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  ident_first_kernel<<<16 * di.sm_count, 256, 0, s>>>(off, n, col, zero_flags, next, ctr);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_rowstart(const long long* off, long long n, unsigned* bits, long long nbits_words,
                            const DeviceInfo& di, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (cudaError_t e = cudaMemsetAsync(bits, 0, sizeof(unsigned) * (size_t)nbits_words, s)) return e;
  rowstart_kernel<<<8 * di.sm_count, 256, 0, s>>>(off, n, bits);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_chunk_check(const long long* off, long long n, const int* col, long long nnz, long long e0,
                               long long e1, const unsigned* bits, unsigned char* bad, unsigned* any_bad,
                               Counters* ctr, const DeviceInfo& di, cudaStream_t s) {
  (void)nnz;
  if (e1 <= e0) return cudaSuccess;
  thread_local int gc = 0;
  if (!gc) gc = one_wave_grid(sorted_check_kernel, di);
  sorted_check_kernel<<<gc, 256, 0, s>>>(off, n, col, e0, e1, bits, bad, any_bad, ctr);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_bin_range(const long long* off, long long v0, long long v1, const Tuning& t, int* work,
                             Counters* ctr, const DeviceInfo& di, cudaStream_t s, int first_cls) {
  if (v1 <= v0) return cudaSuccess;
  const long long tile = 256ll * BIN_ITEMS;
  long long blocks = (v1 - v0 + tile - 1) / tile;
  const long long cap = 8ll * di.sm_count;
  bin_range_kernel<<<(int)(blocks < cap ? blocks : cap), 256, 0, s>>>(off, v0, v1, class_bounds(t), work, ctr, first_cls);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// launchers
namespace {
std::atomic<long long> g_launches{0};

constexpr int WARP_SMALL = 256;   // longest row of one warp (class 6)
}  // namespace

cudaError_t launch_sweep_class(const SweepArgs& a, int cls, int weights, bool async_mode, const Tuning& t,
                               int longest, const DeviceInfo& di, cudaStream_t s) {
  if (cls < CLS_WARP_S) return launch_sweep_tile(a, cls, weights, async_mode, di, s);
  const ClassBounds cb = class_bounds(t);
  // class 8 always takes the block kernel: it sweeps class 9 as well
  const int bound = cls == CLS_WARP_S ? cb.warp_small : (cls == CLS_WARP_L ? cb.warp_max : cb.blk_max);
  return launch_sketch(a, cls, cls == CLS_BLOCK ? 1 << 30 : (bound < longest ? bound : longest), weights, async_mode,
                       di, s);
}

void count_launches(long long k) { g_launches.fetch_add(k, std::memory_order_relaxed); }

cudaError_t raise_smem_limit(const void* fn, size_t bytes) {
  static std::mutex mu;
  static std::unordered_map<const void*, size_t> limits;
  std::lock_guard<std::mutex> g(mu);
  size_t& cur = limits[fn];
  if (bytes <= cur) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) cur = bytes;
  return e;
}
long long launches_total() { return g_launches.load(std::memory_order_relaxed); }

ClassBounds class_bounds(const Tuning& t) {
  ClassBounds cb;
  cb.warp_max = t.warp_max;
  cb.warp_small = WARP_SMALL < t.warp_max ? WARP_SMALL : t.warp_max;
  cb.blk_max = t.blk_max;
  return cb;
}

cudaError_t launch_class_histogram(const long long* off, long long n, long long nnz, const Tuning& t, Counters* ctr,
                                   const DeviceInfo& di, cudaStream_t s) {
  if (n > 0) {
    long long blocks = (n + 255) / 256;
    const long long cap = 8ll * di.sm_count;
    class_histogram_kernel<<<(int)(blocks < cap ? blocks : cap), 256, 0, s>>>(off, n, nnz, class_bounds(t), ctr);
  }
  class_starts_kernel<<<1, 1, 0, s>>>(ctr);
  count_launches(n > 0 ? 2 : 1);
  return cudaGetLastError();
}

cudaError_t launch_bin(const long long* off, long long n, unsigned char* fcur, int all_active, const Tuning& t,
                       int* work, Counters* ctr, const DeviceInfo& di, cudaStream_t s, const int* gid,
                       const unsigned char* done, const int* stop, int phase, unsigned seed, int first_cls) {
  if (n <= 0) return cudaSuccess;
  const long long tile = 256ll * BIN_ITEMS;
  long long blocks = (n + tile - 1) / tile;
  const long long cap = (long long)BIN_BLOCKS * di.sm_count;
  const int grid = (int)(blocks < cap ? blocks : cap);
  if (phase >= 0)
    bin_kernel<true><<<grid, 256, 0, s>>>(off, n, fcur, all_active, class_bounds(t), work, ctr, gid, done, stop, phase,
                                          seed, first_cls);
  else
    bin_kernel<false><<<grid, 256, 0, s>>>(off, n, fcur, all_active, class_bounds(t), work, ctr, gid, done, stop, -1,
                                           0u, first_cls);
  count_launches(1);
  return cudaGetLastError();
}

// A sweep over all vertices whose worklist an earlier such sweep of the same
// call left: only the class counts are set again (R-MAT 25: 0.2 ms of binning
// a sweep, the 60 M-vertex lattice 0.22 ms).
__global__ void all_counts_kernel(Counters* ctr, int first_cls) {
  for (int k = first_cls; k < NCLASS; ++k) ctr->cls_count[k] = (unsigned)ctr->cls_total[k];
}

cudaError_t launch_all_counts(Counters* ctr, int first_cls, cudaStream_t s) {
  all_counts_kernel<<<1, 1, 0, s>>>(ctr, first_cls);
  count_launches(1);
  return cudaGetLastError();
}

// Between the two phases of an asynchronous sweep: the first phase's class
// counts move to phase_cls and the per-phase worklist counters restart.
__global__ void phase_reset_kernel(Counters* ctr, const int* stop) {
  if (stop && *(volatile const int*)stop) return;
  for (int k = 0; k < NCLASS; ++k) {
    ctr->phase_cls[k] += ctr->cls_count[k];
    ctr->cls_count[k] = 0;
    ctr->uns_count[k] = 0;
    ctr->row_next[k] = 0;
  }
  ctr->hub_pieces = 0;
  ctr->hub_clusters = 0;
  ctr->hub_clu_next = 0;
  ctr->filter_next = 0;
  ctr->filter_long = 0;
  ctr->filter_pieces = 0;
}

cudaError_t launch_phase_reset(Counters* ctr, const int* stop, cudaStream_t s) {
  phase_reset_kernel<<<1, 1, 0, s>>>(ctr, stop);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_init_labels(const int* init, int* a, int* b, long long n, Counters* ctr, const DeviceInfo& di,
                               cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  long long blocks = (n + 255) / 256;
  const long long cap = 8ll * di.sm_count;
  init_labels_kernel<<<(int)(blocks < cap ? blocks : cap), 256, 0, s>>>(init, a, b, n, ctr);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace gsl

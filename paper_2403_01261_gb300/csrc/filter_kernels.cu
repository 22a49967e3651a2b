// filter_kernels.cu -- rows settled by a strict majority before they are
// counted (classes 6..9, once labels have started to settle).
//
// When the entries of a row that carry one label weigh more than half of the
// row (the vertex itself excluded), that label is Eq. 2's argmax whatever the
// others are.  Two labels are worth testing:
//   - the vertex's own, which most rows keep in later sweeps;
//   - on skewed graphs one label that most entries of the whole graph carry
//     (R-MAT 25: 66-75 % of the entries in sweep 3, nearly all in sweep 4).
//     Testing for it needs one bit per vertex instead of a label: 4 MB that
//     stay in L2 instead of 134 MB of which most gathers miss it, and it
//     settles rows that are about to change as well.
// filter_plan_kernel samples 1024 entries and picks the test; rows it settles
// are written and dropped, the others form a second worklist that the
// counting kernels read (class_work).  A row is read only until the tested
// label holds more than half of its weight: unit weights count against the
// degree, others against the row total that sweep 1 stored.
//
// Classes 6 and 7 take a warp per row; 8 and 9 a block per row from a
// counter, so that no long row is left to one warp; where the rest of the graph
// does not hide its longest row (SweepArgs::long_rows), rows past FILTER_LONG are
// only listed there, in pieces of FILTER_PIECE entries that the blocks of a
// second kernel share.  Bound by the gathers.
#include "sweep_device.cuh"

namespace gsl {

namespace {

constexpr int KW_SHIFT = 22;   // 64-bit sums: row totals are stored as (total >> 22) + 1
// Sampled shares of neighbours from which the tests are made.  Neither line is
// sharp (ms a call).  Giant label from 45 / 55 / 68 %: R-MAT 25 29.6 / 29.9 /
// 29.7, R-MAT 22 with int32 weights 11.6 / 11.5 / 12.1, heavy-tailed 2 M vertices
// 2.50 / 2.39 / 2.37; own label from 25 / 40 / 55 %: R-MAT 22 with int32 weights
// 11.5 / 11.5 / 11.3, 700,000-vertex planted partition 1.92 / 1.90 / 1.89.
constexpr int GIANT_PERCENT = 55, OWN_PERCENT = 40;

// Weight the tested label must exceed half of: an upper bound of the row's
// total, or ~0 when none is known (then the row is read to its end).
template <int WT>
__device__ __forceinline__ unsigned long long row_bound(const SweepArgs& a, int v, int d) {
  if (WT == 0) return (unsigned long long)d;
  if (!a.kw) return ~0ull;
  return WT == 1 ? (unsigned long long)a.kw[v] : (unsigned long long)a.kw[v] << KW_SHIFT;
}

// The tested label's weight and all weight over a thread's four entries at
// e, e + step, ..; columns in j, -1 for none.
template <int WT, bool ASYNC, bool GIANT>
__device__ __forceinline__ void filter_entries(const SweepArgs& a, const int* lp, int v, int own, const int* wp, int e,
                                               int step, const int (&j)[4], const Pol& pol,
                                               typename SumOf<WT>::T& hit, typename SumOf<WT>::T& all) {
  using S = typename SumOf<WT>::T;
  bool is[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    is[u] = false;
    if (j[u] >= 0 && j[u] != v) {
      if (GIANT) {
        const unsigned word = (unsigned)ld_label_ro(reinterpret_cast<const int*>(a.bits) + (j[u] >> 5), pol.label);
        is[u] = (word >> (j[u] & 31)) & 1u;
      } else {
        is[u] = entry_label<ASYNC>(a, lp, e + u * step, j[u], v, pol) == own;
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (j[u] >= 0 && j[u] != v) {
      const S w = WT ? (S)(unsigned)ld_stream(wp + e + u * step, pol.stream) : (S)1;
      all += w;
      if (is[u]) hit += w;
    }
  }
}

__device__ __forceinline__ unsigned warp_total(unsigned x) { return __reduce_add_sync(FULL, x); }
__device__ __forceinline__ unsigned long long warp_total(unsigned long long x) { return warp_sum_u64(x); }

// Writes a settled row; the caller marks the neighbours of a changed one.
template <bool ASYNC>
__device__ __forceinline__ bool settle(const SweepArgs& a, int v, int nl, int old, unsigned long long& dn) {
  const bool changed = nl != old;
  store_label<ASYNC>(a, v, nl, changed);
  if (changed) {
    count_graph_change(a, v);
    dn += 1;
    if (a.mark && !ASYNC) a.fnext[v] = 1;
  }
  return changed;
}

__device__ __forceinline__ void flush_filter(Counters* ctr, unsigned long long dn, unsigned long long scan,
                                             unsigned long long settled) {
  dn = warp_sum_u64(dn);
  scan = warp_sum_u64(scan);
  settled = warp_sum_u64(settled);
  if ((threadIdx.x & 31) == 0) {
    if (dn) atomicAdd(&ctr->dn, dn);
    if (scan) atomicAdd(&ctr->scanned, scan);
    if (settled) atomicAdd(&ctr->fast_active, settled);
  }
}

// One warp per row of classes 6 and 7.
template <int WT, bool ASYNC, bool GIANT>
__device__ __forceinline__ void filter_warps(const SweepArgs& a, int* __restrict__ out) {
  using S = typename SumOf<WT>::T;
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const Pol pol = make_pol();
  const int giant = a.ctr->giant_label;
  const long long c6 = a.ctr->filter_from <= CLS_WARP_S ? a.ctr->cls_count[CLS_WARP_S] : 0;
  const long long total = a.ctr->filter_from <= CLS_WARP_L ? c6 + a.ctr->cls_count[CLS_WARP_L] : 0;
  unsigned long long my_dn = 0, my_scan = 0, my_settled = 0;
  for (long long i = warp; i < total; i += nwarps) {
    const int cls = i < c6 ? CLS_WARP_S : CLS_WARP_L;
    const long long start = a.ctr->cls_start[cls];
    const int v = a.work[start + (i < c6 ? i : i - c6)];
    const long long s = a.off[v];
    const int d = (int)(a.off[v + 1] - s);
    const int old = own_label<ASYNC>(a, v);
    const int* cp = a.col + s;
    const int* wp = a.w + s;
    const int* lp = a.lg ? a.lg + s : nullptr;
    const unsigned long long bound = row_bound<WT>(a, v, d);
    S hit = 0, all = 0;
    bool early = false;
    int jn[4], read = d;
#pragma unroll
    for (int u = 0; u < 4; ++u) jn[u] = later_col(a, cp, d, lane + 32 * u, pol);
    for (int r0 = 0; r0 < d; r0 += 128) {
      int j[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) j[u] = jn[u];
      const bool more = r0 + 128 < d;   // warp-uniform
      if (more) {
#pragma unroll
        for (int u = 0; u < 4; ++u) jn[u] = later_col(a, cp, d, r0 + 128 + lane + 32 * u, pol);
      }
      filter_entries<WT, ASYNC, GIANT>(a, lp, v, old, wp, r0 + lane, 32, j, pol, hit, all);
      if (more && bound != ~0ull) {
        early = 2ull * (unsigned long long)warp_total(hit) > bound;
        if (early) {
          read = r0 + 128;
          break;
        }
      }
    }
    const S h = warp_total(hit), t = warp_total(all);
    const bool settled = early || 2ull * (unsigned long long)h > (unsigned long long)t;
    bool changed = false;
    if (lane == 0) {
      if (settled) {
        changed = settle<ASYNC>(a, v, GIANT ? giant : old, old, my_dn);
        my_scan += (unsigned long long)read;
        my_settled += 1;
      } else {
        out[start + atomicAdd(&a.ctr->uns_count[cls], 1u)] = v;
      }
    }
    if (GIANT && a.mark && __any_sync(FULL, changed)) {
      for (int e = lane; e < d; e += 32) {
        const int j = ld_stream(cp + e, pol.stream);
        if ((unsigned)j < (unsigned)a.n) a.fnext[j] = 1;
      }
    }
  }
  flush_filter(a.ctr, my_dn, my_scan, my_settled);
}

// One block per row of classes 8 and 9.
template <int WT, bool ASYNC, bool GIANT>
__device__ __forceinline__ void filter_blocks(const SweepArgs& a, int* __restrict__ out) {
  using S = typename SumOf<WT>::T;
  __shared__ S s_hit, s_all;
  __shared__ unsigned s_next, s_slot, s_piece;
  __shared__ int s_changed;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
  const Pol pol = make_pol();
  const int giant = a.ctr->giant_label;
  const unsigned c9 = a.ctr->cls_count[CLS_HUB];
  const unsigned total = a.ctr->filter_from <= CLS_BLOCK ? c9 + a.ctr->cls_count[CLS_BLOCK] : 0u;
  unsigned long long my_dn = 0, my_scan = 0, my_settled = 0;
  for (unsigned i = blockIdx.x; i < total;) {   // the longest class first
    const int cls = i < c9 ? CLS_HUB : CLS_BLOCK;
    const long long start = a.ctr->cls_start[cls];
    const int v = a.work[start + (i < c9 ? i : i - c9)];
    if (tid == 0) {
      s_hit = 0;
      s_all = 0;
      s_next = gridDim.x + atomicAdd(&a.ctr->filter_next, 1u);
    }
    __syncthreads();
    const unsigned next = s_next;
    const long long s = a.off[v];
    const int d = (int)(a.off[v + 1] - s);
    if (d > FILTER_LONG && a.long_rows) {   // block-uniform
      const int pieces = (d + FILTER_PIECE - 1) / FILTER_PIECE;
      if (tid == 0) {
        s_slot = atomicAdd(&a.ctr->filter_long, 1u);
        s_piece = atomicAdd(&a.ctr->filter_pieces, (unsigned)pieces);
        a.long_rows[s_slot] = FilterLong{0, 0, 0, v, cls, (unsigned)pieces};
      }
      __syncthreads();
      for (int k = tid; k < pieces; k += T) a.long_pieces[s_piece + k] = make_int2((int)s_slot, k);
      i = next;
      continue;
    }
    const int old = own_label<ASYNC>(a, v);
    const int* cp = a.col + s;
    const int* wp = a.w + s;
    const int* lp = a.lg ? a.lg + s : nullptr;
    const unsigned long long bound = row_bound<WT>(a, v, d);
    S all = 0;
    int jn[4], read = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) jn[u] = later_col(a, cp, d, tid + u * T, pol);
    for (int r0 = 0; r0 < d; r0 += 4 * T) {
      int j[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) j[u] = jn[u];
      const bool more = r0 + 4 * T < d;   // block-uniform
      if (more) {
#pragma unroll
        for (int u = 0; u < 4; ++u) jn[u] = later_col(a, cp, d, r0 + 4 * T + tid + u * T, pol);
      }
      S hit = 0;
      filter_entries<WT, ASYNC, GIANT>(a, lp, v, old, wp, r0 + tid, T, j, pol, hit, all);
      hit = warp_total(hit);
      S sum = 0;
      if (lane == 0 && hit) sum = atomicAdd(&s_hit, hit) + hit;
      read = min(d, r0 + 4 * T);
      if (more && bound != ~0ull) {   // warps leave on their own once the row is settled
        const unsigned over = __ballot_sync(FULL, 2ull * (unsigned long long)sum > bound);
        if (over) break;
      }
    }
    all = warp_total(all);
    if (lane == 0 && all) atomicAdd(&s_all, all);
    __syncthreads();
    const unsigned long long h = 2ull * (unsigned long long)s_hit;
    const bool settled = h > bound || h > (unsigned long long)s_all;   // all of the row was read unless h > bound
    if (tid == 0) {
      s_changed = 0;
      if (settled) {
        s_changed = settle<ASYNC>(a, v, GIANT ? giant : old, old, my_dn);
        my_scan += (unsigned long long)read;
        my_settled += 1;
      } else {
        out[start + atomicAdd(&a.ctr->uns_count[cls], 1u)] = v;
      }
    }
    __syncthreads();
    if (GIANT && a.mark && s_changed) {
      for (int e = tid; e < d; e += T) {
        const int j = ld_stream(cp + e, pol.stream);
        if ((unsigned)j < (unsigned)a.n) a.fnext[j] = 1;
      }
    }
    i = next;
  }
  flush_filter(a.ctr, my_dn, my_scan, my_settled);
}

// One block per listed piece of a long row.  A piece is skipped once the
// pieces before it have settled the row; the one that ends last decides.
// One block over the whole row took 0.5 ms per million entries, however idle
// the rest of the chip: one hub of 8 M entries among 80 M others 3.85 ms a pass,
// 0.06 in pieces; of 2 M among 60 M 1.04 and 0.10; of 1 M among 10 M 0.51 and less
// than 0.05.  From 65,536 entries on, which a block reads in about 30 us, that is
// longer than what a small graph's sweep takes.  R-MAT 25 has no use for it (8.4
// ms a call by blocks, 8.5 in pieces).
template <int WT, bool ASYNC, bool GIANT>
__device__ __forceinline__ void filter_pieces(const SweepArgs& a, int* __restrict__ out) {
  using S = typename SumOf<WT>::T;
  __shared__ unsigned long long s_hit, s_all;
  __shared__ int s_skip, s_changed;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
  const Pol pol = make_pol();
  const int giant = a.ctr->giant_label;
  const unsigned total = a.ctr->filter_pieces;
  unsigned long long my_dn = 0, my_scan = 0, my_settled = 0;
  for (unsigned i = blockIdx.x; i < total; i += gridDim.x) {
    const int2 piece = a.long_pieces[i];
    FilterLong* row = a.long_rows + piece.x;
    const int v = row->v;
    const long long s = a.off[v];
    const int d = (int)(a.off[v + 1] - s), from = piece.y * FILTER_PIECE, len = min(d - from, FILTER_PIECE);
    const int old = own_label<ASYNC>(a, v);
    const unsigned long long bound = row_bound<WT>(a, v, d);
    if (tid == 0) {
      s_hit = 0;
      s_all = 0;
      s_changed = 0;
      s_skip = bound != ~0ull && 2ull * __ldcg(&row->hit) > bound;
    }
    __syncthreads();
    const bool skip = s_skip != 0;
    if (!skip) {
      const int* cp = a.col + s + from;
      const int* wp = a.w + s + from;
      const int* lp = a.lg ? a.lg + s + from : nullptr;
      S hit = 0, all = 0;
      int jn[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) jn[u] = later_col(a, cp, len, tid + u * T, pol);
      for (int r0 = 0; r0 < len; r0 += 4 * T) {
        int j[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) j[u] = jn[u];
#pragma unroll
        for (int u = 0; u < 4; ++u) jn[u] = later_col(a, cp, len, r0 + 4 * T + tid + u * T, pol);
        filter_entries<WT, ASYNC, GIANT>(a, lp, v, old, wp, r0 + tid, T, j, pol, hit, all);
      }
      hit = warp_total(hit);
      all = warp_total(all);
      if (lane == 0) {
        if (hit) atomicAdd(&s_hit, (unsigned long long)hit);
        if (all) atomicAdd(&s_all, (unsigned long long)all);
      }
    }
    __syncthreads();
    if (tid == 0) {
      if (!skip) {
        atomicAdd(&row->hit, s_hit);
        atomicAdd(&row->all, s_all);
        atomicAdd(&row->read, (unsigned long long)len);
      }
      __threadfence();
      if (atomicSub(&row->left, 1u) == 1u) {
        __threadfence();
        const unsigned long long h = 2ull * __ldcg(&row->hit);
        if (h > bound || h > __ldcg(&row->all)) {   // all of the row was read unless h > bound
          s_changed = settle<ASYNC>(a, v, GIANT ? giant : old, old, my_dn);
          my_scan += __ldcg(&row->read);
          my_settled += 1;
        } else {
          out[a.ctr->cls_start[row->cls] + atomicAdd(&a.ctr->uns_count[row->cls], 1u)] = v;
        }
      }
    }
    __syncthreads();
    if (GIANT && a.mark && s_changed) {
      for (int e = tid; e < d; e += T) {
        const int j = ld_stream(a.col + s + e, pol.stream);
        if ((unsigned)j < (unsigned)a.n) a.fnext[j] = 1;
      }
    }
    __syncthreads();   // s_changed is cleared for the next piece
  }
  flush_filter(a.ctr, my_dn, my_scan, my_settled);
}

}  // namespace

// Which label the filter tests, and from which class on: the giant on every
// class from 6, the own label from first_cls, or nothing (early sweeps over
// weighted graphs, where no label repeats: the filter's pass was a quarter of
// the time there and settled nothing).  1024 vertices sampled in proportion to
// their degree (the ends of random entries) each look at one random
// neighbour: whether it carries the vertex's own label, and which label it
// carries; a label that more than half of them see shows as the bitwise
// majority.
__global__ void __launch_bounds__(1024) filter_plan_kernel(SweepArgs a, long long nnz, int first_cls, int sample,
                                                           unsigned seed) {
  if (stopped(a)) return;
  __shared__ unsigned bit[32];
  const unsigned t = threadIdx.x;
  if (!sample) {
    if (t == 0) {
      a.ctr->filter_from = first_cls;
      a.ctr->giant_on = 0;
    }
    return;
  }
  if (t < 32) bit[t] = 0;
  __syncthreads();
  const unsigned x = hash32(hash32(t + 1024u * seed) ^ 0x5BD1E995u), y = hash32((t * 0x27D4EB2Fu + seed) | 1u);
  const int j = a.col[__umul64hi((unsigned long long)x << 32 | y, (unsigned long long)nnz)];
  int own = -1, l = -1;
  if ((unsigned)j < (unsigned)a.n) {
    const long long s = a.off[j], d = a.off[j + 1] - s;
    if (d > 0) {
      const int k = a.col[s + __umul64hi((unsigned long long)y << 32 | x, (unsigned long long)d)];
      if ((unsigned)k < (unsigned)a.n) {
        own = a.prev[j];
        l = a.prev[k];
      }
    }
  }
  const bool ok = l >= 0;
  const int valid = __syncthreads_count(ok), keeps = __syncthreads_count(ok && l == own);
#pragma unroll
  for (int b = 0; b < 31; ++b) {
    const unsigned m = __ballot_sync(FULL, ok && ((l >> b) & 1));
    if ((t & 31) == (unsigned)b && m) atomicAdd(&bit[b], (unsigned)__popc(m));
  }
  __syncthreads();
  int g = 0;
  for (int b = 0; b < 31; ++b) g |= (2 * (int)bit[b] > valid ? 1 : 0) << b;
  const int same = __syncthreads_count(ok && l == g);
  if (t == 0) {
    const int on = valid > 0 && 100 * same >= GIANT_PERCENT * valid;
    a.ctr->giant_on = on;
    a.ctr->giant_label = g;
    a.ctr->filter_from = on ? CLS_WARP_S : (100 * keeps >= OWN_PERCENT * valid ? first_cls : NCLASS);
  }
}

// Bit v: vertex v carries the giant label.
__global__ void __launch_bounds__(256) giant_bits_kernel(const int* __restrict__ prev, long long n,
                                                         unsigned* __restrict__ bits, const Counters* ctr) {
  if (!ctr->giant_on) return;
  const int g = ctr->giant_label;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long v0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
  for (long long w = v0; w < n; w += stride) {   // warp-uniform
    const long long v = w + (threadIdx.x & 31);
    const unsigned m = __ballot_sync(FULL, v < n && prev[v < n ? v : n - 1] == g);
    if ((threadIdx.x & 31) == 0) bits[w >> 5] = m;
  }
}

// Six blocks per SM: 40 registers, of which the synchronous forms of the warp
// kernel, which hold both tests, spill 104 to 180 bytes.  R-MAT 25 at 4 / 5 / 6 /
// 8 blocks: 30.6 / 29.7 / 29.9 / 30.4 ms a call, the filter 9.3 / 8.5 / 8.5 / 9.2.
template <int WT, bool ASYNC>
__global__ void __launch_bounds__(256, 6) filter_warp_kernel(SweepArgs a, int* __restrict__ out) {
  if (stopped(a)) return;
  if (!ASYNC && a.ctr->giant_on) filter_warps<WT, ASYNC, true>(a, out);
  else filter_warps<WT, ASYNC, false>(a, out);
}

template <int WT, bool ASYNC>
__global__ void __launch_bounds__(256, 6) filter_block_kernel(SweepArgs a, int* __restrict__ out) {
  if (stopped(a)) return;
  if (!ASYNC && a.ctr->giant_on) filter_blocks<WT, ASYNC, true>(a, out);
  else filter_blocks<WT, ASYNC, false>(a, out);
}

template <int WT, bool ASYNC>
__global__ void __launch_bounds__(256, 6) filter_long_kernel(SweepArgs a, int* __restrict__ out) {
  if (stopped(a)) return;
  if (!ASYNC && a.ctr->giant_on) filter_pieces<WT, ASYNC, true>(a, out);
  else filter_pieces<WT, ASYNC, false>(a, out);
}

// The rows passed on become the class counts.
__global__ void filter_counts_kernel(Counters* ctr, const int* stop, int first_cls, int last_cls) {
  if (stop && *(volatile const int*)stop) return;
  if (first_cls < 0) first_cls = ctr->filter_from;
  for (int k = first_cls; k <= last_cls; ++k) ctr->cls_count[k] = ctr->uns_count[k];
}

cudaError_t launch_filter_counts(Counters* ctr, const int* stop, cudaStream_t s, int first_cls, int last_cls) {
  filter_counts_kernel<<<1, 1, 0, s>>>(ctr, stop, first_cls, last_cls);
  count_launches(1);
  return cudaGetLastError();
}

namespace {
template <int WT, bool A>
void launch_filter_t(const SweepArgs& a, int* out, bool warps, bool blocks, const DeviceInfo& di, cudaStream_t s) {
  if (blocks) filter_block_kernel<WT, A><<<6 * di.sm_count, 256, 0, s>>>(a, out);
  if (blocks && a.long_rows) filter_long_kernel<WT, A><<<6 * di.sm_count, 256, 0, s>>>(a, out);
  if (warps) filter_warp_kernel<WT, A><<<6 * di.sm_count, 256, 0, s>>>(a, out);
}
}  // namespace

cudaError_t launch_majority_filter(const SweepArgs& a, long long nnz, int* out, unsigned* bits, int weights,
                                   bool async_mode, int first_cls, bool sample, unsigned seed, bool warps, bool blocks,
                                   const DeviceInfo& di, cudaStream_t s, int* kernels) {
  sample = sample && !async_mode && nnz > 0;   // in place, the sampled labels may change under the sweep
  filter_plan_kernel<<<1, sample ? 1024 : 32, 0, s>>>(a, nnz, first_cls, sample ? 1 : 0, seed);
  int launches = 2 + (warps ? 1 : 0) + (blocks ? (a.long_rows ? 2 : 1) : 0);
  if (sample) {
    long long g = (a.n + 255) / 256;
    const long long cap = 8ll * di.sm_count;
    giant_bits_kernel<<<(int)(g < cap ? g : cap), 256, 0, s>>>(a.prev, a.n, bits, a.ctr);
    ++launches;
  }
  SweepArgs f = a;
  f.bits = bits;
  switch (2 * weights + (async_mode ? 1 : 0)) {
    case 0: launch_filter_t<0, false>(f, out, warps, blocks, di, s); break;
    case 1: launch_filter_t<0, true>(f, out, warps, blocks, di, s); break;
    case 2: launch_filter_t<1, false>(f, out, warps, blocks, di, s); break;
    case 3: launch_filter_t<1, true>(f, out, warps, blocks, di, s); break;
    case 4: launch_filter_t<2, false>(f, out, warps, blocks, di, s); break;
    default: launch_filter_t<2, true>(f, out, warps, blocks, di, s); break;
  }
  filter_counts_kernel<<<1, 1, 0, s>>>(a.ctr, a.stop, -1, CLS_HUB);
  count_launches(launches);
  if (kernels) *kernels = launches;
  return cudaGetLastError();
}

}  // namespace gsl

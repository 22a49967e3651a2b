// modularity_kernels.cu -- Eq. 1 on sm_103a with exact integer sums.
//
// Q = sum_c [ sigma_c / 2m - (Sigma_c / 2m)^2 ].  Over a symmetric CSR:
//   2m            = sum of all entry weights (weighted degrees K_i summed),
//   S1            = sum_c sigma_c = weights of entries (i, j) with C_i == C_j,
//   Sigma_c       = sum of K_i over the vertices of c,
//   S2            = sum_c Sigma_c^2 (128-bit).
// Pass 1 accumulates K_i into Sigma[C_i] and the block sums of 2m and S1:
// rows of 1..4 entries one lane each in natural order, longer ones from the
// worklist by degree class.  Unit-weight K_i are degrees, so every vertex's
// K_i is added by the natural-order kernel and the class kernels only count
// S1.  Pass 2 squares and sums Sigma in 128 bits; the host forms Q once in
// double.  All sums are integers, so the result is independent of summation
// order.
//
// A partition that sweeps leave on a skewed graph holds one community of
// nearly every vertex: adding each lane's part to Sigma directly made 52 of
// 52.5 ms of an R-MAT scale 23 call wait on atomics to one address.  Equal
// communities of a warp are added up first, then in a per-block table of
// MOD_CACHE communities, which reaches Sigma once per block.  What is left
// is bound by the gathers of the neighbours' labels.
#include "kernels.h"

namespace gsl {

namespace {

struct U128 {
  unsigned long long lo, hi;
};
__device__ __forceinline__ U128 add128(U128 a, U128 b) {
  U128 r;
  r.lo = a.lo + b.lo;
  r.hi = a.hi + b.hi + (r.lo < a.lo ? 1ull : 0ull);
  return r;
}
__device__ __forceinline__ U128 sq64(unsigned long long x) {
  U128 r;
  r.lo = x * x;
  r.hi = __umul64hi(x, x);
  return r;
}

__device__ __forceinline__ void flush_sums(ModSums* out, unsigned long long k, unsigned long long s1) {
  __shared__ unsigned long long acc[2];
  if (threadIdx.x == 0) { acc[0] = 0; acc[1] = 0; }
  __syncthreads();
  for (int o = 16; o; o >>= 1) {
    k += __shfl_xor_sync(FULL, k, o);
    s1 += __shfl_xor_sync(FULL, s1, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&acc[0], k);
    atomicAdd(&acc[1], s1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (acc[0]) atomicAdd(&out->two_m, acc[0]);
    if (acc[1]) atomicAdd(&out->s1, acc[1]);
  }
}

// Per-block table of community sums (direct mapped, first come): what does
// not fit goes to Sigma at once.
constexpr int MOD_CACHE = 256;
struct SigmaCache {
  int key[MOD_CACHE];   // -1: free
  unsigned long long sum[MOD_CACHE];
};

__device__ __forceinline__ void cache_clear(SigmaCache& sc) {
  for (int k = threadIdx.x; k < MOD_CACHE; k += blockDim.x) {
    sc.key[k] = -1;
    sc.sum[k] = 0;
  }
  __syncthreads();
}

__device__ __forceinline__ void cache_add(SigmaCache& sc, unsigned long long* sigma, int c, unsigned long long k) {
  const int slot = (int)(hash32((unsigned)c) >> 24);
  const int old = atomicCAS(&sc.key[slot], -1, c);
  if (old == -1 || old == c) atomicAdd(&sc.sum[slot], k);
  else atomicAdd(sigma + c, k);
}

// Every lane of the warp with its community c and sum k (k = 0: nothing):
// the lanes that share the first such lane's community are added up first.
__device__ __forceinline__ void warp_add_sigma(SigmaCache& sc, unsigned long long* sigma, int c,
                                               unsigned long long k) {
  const unsigned has = __ballot_sync(FULL, k != 0);
  if (!has) return;
  const int first = __ffs((int)has) - 1;
  const int cf = __shfl_sync(FULL, c, first);   // every lane takes part
  const bool same = k != 0 && c == cf;
  const unsigned long long total = warp_sum_u64(same ? k : 0ull);
  if ((int)(threadIdx.x & 31) == first) cache_add(sc, sigma, c, total);
  else if (k && !same) cache_add(sc, sigma, c, k);
}

__device__ __forceinline__ void cache_flush(SigmaCache& sc, unsigned long long* sigma) {
  __syncthreads();
  for (int k = threadIdx.x; k < MOD_CACHE; k += blockDim.x)
    if (sc.key[k] >= 0 && sc.sum[k]) atomicAdd(sigma + sc.key[k], sc.sum[k]);
}

// U entries e, e + step, .. of a row of u's community cu, the loads of all
// in flight together: adds their weights to k and, inside cu, to s1.
template <bool WEIGHTED, int U>
__device__ __forceinline__ void mod_entries(const int* col, const int* w, const int* labels, long long n, int cu,
                                            long long e, long long end, int step, unsigned long long& k,
                                            unsigned long long& s1, int* err) {
  int j[U], x[U];
#pragma unroll
  for (int q = 0; q < U; ++q) {
    const bool in = e + (long long)q * step < end;
    j[q] = in ? ld_stream(col + e + (long long)q * step) : -1;
    x[q] = 1;
    if (WEIGHTED && in) x[q] = ld_stream(w + e + (long long)q * step);
    if (in && (unsigned)j[q] >= (unsigned)n) {
      raise_err(err, ERRBIT_INVALID);
      j[q] = -1;
    }
  }
#pragma unroll
  for (int q = 0; q < U; ++q) {
    if (j[q] >= 0) {
      const unsigned long long we = (unsigned long long)(unsigned)x[q];
      if (WEIGHTED) k += we;
      if (ld_label_ro(labels + j[q]) == cu) s1 += we;
    }
  }
}

constexpr int MOD_LANE_ROW = 4;   // longest row of one lane (classes 0..2)

}  // namespace

// Every vertex in natural order, one lane each: label range, unit-weight
// K_i, and the rows of 1..4 entries.
template <bool WEIGHTED>
__global__ void __launch_bounds__(256) mod_lane_kernel(const long long* __restrict__ off, const int* __restrict__ col,
                                                        const int* __restrict__ w, const int* __restrict__ labels,
                                                        long long n, Counters* ctr, unsigned long long* sigma,
                                                        ModSums* out) {
  __shared__ SigmaCache sc;
  cache_clear(sc);
  unsigned long long tk = 0, ts1 = 0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long v0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
  for (long long wv = v0; wv < n; wv += stride) {   // warp-uniform
    const long long v = wv + (threadIdx.x & 31);
    unsigned long long k = 0;
    int cu = 0;
    if (v < n) {
      const long long s = off[v], e = off[v + 1];
      cu = labels[v];
      if ((unsigned)cu >= (unsigned)n) {
        raise_err(&ctr->err, ERRBIT_INVALID);
        cu = 0;
      } else {
        if (e - s <= MOD_LANE_ROW) mod_entries<WEIGHTED, MOD_LANE_ROW>(col, w, labels, n, cu, s, e, 1, k, ts1, &ctr->err);
        if (!WEIGHTED) k = (unsigned long long)(e - s);
      }
    }
    tk += k;
    warp_add_sigma(sc, sigma, cu, k);
  }
  cache_flush(sc, sigma);
  flush_sums(out, tk, ts1);
}

// Classes 3..7 from the worklist: G lanes per row, four entries of a lane in
// flight on rows longer than G.
template <int G, bool WEIGHTED>
__global__ void __launch_bounds__(256) mod_group_kernel(const long long* __restrict__ off, const int* __restrict__ col,
                                                         const int* __restrict__ w, const int* __restrict__ labels,
                                                         long long n, const int* __restrict__ work, Counters* ctr,
                                                         int cls, unsigned long long* sigma, ModSums* out) {
  __shared__ SigmaCache sc;
  if (WEIGHTED) cache_clear(sc);
  const unsigned cnt = (unsigned)ctr->cls_total[cls];
  const int* wl = work + ctr->cls_start[cls];
  constexpr int PER = 32 / G;
  const int lane = threadIdx.x & 31, gl = lane & (G - 1);
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  unsigned long long tk = 0, ts1 = 0;
  for (long long i0 = warp * PER; i0 < (long long)cnt; i0 += nwarps * PER) {   // warp-uniform
    const long long item = i0 + lane / G;
    unsigned long long k = 0;
    int cu = 0;
    if (item < (long long)cnt) {
      const int u = wl[item];
      const long long s = off[u], e = off[u + 1];
      cu = labels[u];
      if ((unsigned)cu >= (unsigned)n) {
        cu = 0;   // reported by the natural-order kernel
      } else if (G < 32 || e - s <= 32) {
        mod_entries<WEIGHTED, 1>(col, w, labels, n, cu, s + gl, e, G, k, ts1, &ctr->err);
      } else {
        for (long long x = s + gl; x < e; x += 4 * G)
          mod_entries<WEIGHTED, 4>(col, w, labels, n, cu, x, e, G, k, ts1, &ctr->err);
      }
    }
    if (WEIGHTED) {
      tk += k;
#pragma unroll
      for (int o = G / 2; o; o >>= 1) k += __shfl_xor_sync(FULL, k, o);
      warp_add_sigma(sc, sigma, cu, gl == 0 ? k : 0ull);
    }
  }
  if (WEIGHTED) cache_flush(sc, sigma);
  flush_sums(out, tk, ts1);
}

// The entries [from, to) of u's row by a block, four of a thread in flight.
template <bool WEIGHTED>
__device__ __forceinline__ void mod_block_entries(const int* col, const int* w, const int* labels, long long n, int cu,
                                                  long long from, long long to, unsigned long long* sigma,
                                                  unsigned long long& tk, unsigned long long& ts1, int* err) {
  unsigned long long k = 0;
  for (long long x = from + threadIdx.x; x < to; x += 4 * blockDim.x)
    mod_entries<WEIGHTED, 4>(col, w, labels, n, cu, x, to, (int)blockDim.x, k, ts1, err);
  if (WEIGHTED) {
    tk += k;
    k = warp_sum_u64(k);
    if ((threadIdx.x & 31) == 0 && k) atomicAdd(sigma + cu, k);
  }
}

// Classes 8 and 9: one block per row.  With `pieces`, rows of more than
// FILTER_LONG entries are only listed, in pieces of FILTER_PIECE entries.
template <bool WEIGHTED>
__global__ void __launch_bounds__(512) mod_block_kernel(const long long* __restrict__ off, const int* __restrict__ col,
                                                         const int* __restrict__ w, const int* __restrict__ labels,
                                                         long long n, const int* __restrict__ work, Counters* ctr,
                                                         int cls, unsigned long long* sigma, int2* pieces, ModSums* out) {
  __shared__ unsigned s_piece;
  const unsigned cnt = (unsigned)ctr->cls_total[cls];
  const int* wl = work + ctr->cls_start[cls];
  unsigned long long tk = 0, ts1 = 0;
  for (long long item = blockIdx.x; item < (long long)cnt; item += gridDim.x) {
    const int u = wl[item];
    const long long s = off[u], e = off[u + 1];
    const int cu = labels[u];
    if ((unsigned)cu >= (unsigned)n) continue;   // reported by the natural-order kernel
    if (pieces && e - s > FILTER_LONG) {         // block-uniform
      const int np = (int)((e - s + FILTER_PIECE - 1) / FILTER_PIECE);
      __syncthreads();   // the previous row's last read
      if (threadIdx.x == 0) s_piece = atomicAdd(&ctr->filter_pieces, (unsigned)np);
      __syncthreads();
      for (int k = threadIdx.x; k < np; k += blockDim.x) pieces[s_piece + k] = make_int2(u, k);
      continue;
    }
    mod_block_entries<WEIGHTED>(col, w, labels, n, cu, s, e, sigma, tk, ts1, &ctr->err);
  }
  flush_sums(out, tk, ts1);
}

// One block per listed piece.  A row of 8 million entries among 80 million others
// takes 12.7 ms by one block, 1.4 in pieces.
template <bool WEIGHTED>
__global__ void __launch_bounds__(512) mod_piece_kernel(const long long* __restrict__ off, const int* __restrict__ col,
                                                         const int* __restrict__ w, const int* __restrict__ labels,
                                                         long long n, Counters* ctr, unsigned long long* sigma,
                                                         const int2* __restrict__ pieces, ModSums* out) {
  const unsigned cnt = ctr->filter_pieces;
  unsigned long long tk = 0, ts1 = 0;
  for (unsigned i = blockIdx.x; i < cnt; i += gridDim.x) {
    const int2 p = pieces[i];
    const long long from = off[p.x] + (long long)p.y * FILTER_PIECE, e = off[p.x + 1];
    mod_block_entries<WEIGHTED>(col, w, labels, n, labels[p.x], from, from + FILTER_PIECE < e ? from + FILTER_PIECE : e,
                                sigma, tk, ts1, &ctr->err);
  }
  flush_sums(out, tk, ts1);
}

__global__ void __launch_bounds__(256) mod_square_kernel(const unsigned long long* __restrict__ sigma, long long n,
                                                          unsigned long long* partials) {
  U128 acc{0, 0};
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
    acc = add128(acc, sq64(sigma[c]));
  __shared__ unsigned long long lo[256], hi[256];
  lo[threadIdx.x] = acc.lo;
  hi[threadIdx.x] = acc.hi;
  __syncthreads();
  for (int o = blockDim.x / 2; o; o >>= 1) {
    if (threadIdx.x < (unsigned)o) {
      U128 a{lo[threadIdx.x], hi[threadIdx.x]}, b{lo[threadIdx.x + o], hi[threadIdx.x + o]};
      const U128 r = add128(a, b);
      lo[threadIdx.x] = r.lo;
      hi[threadIdx.x] = r.hi;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partials[2 * blockIdx.x] = lo[0];
    partials[2 * blockIdx.x + 1] = hi[0];
  }
}

__global__ void __launch_bounds__(256) mod_final_kernel(const unsigned long long* partials, long long nparts,
                                                        ModSums* out) {
  __shared__ unsigned long long lo[256], hi[256];
  U128 acc{0, 0};
  for (long long b = threadIdx.x; b < nparts; b += 256) acc = add128(acc, U128{partials[2 * b], partials[2 * b + 1]});
  lo[threadIdx.x] = acc.lo;
  hi[threadIdx.x] = acc.hi;
  __syncthreads();
  for (int o = 128; o; o >>= 1) {
    if (threadIdx.x < (unsigned)o) {
      const U128 r = add128(U128{lo[threadIdx.x], hi[threadIdx.x]}, U128{lo[threadIdx.x + o], hi[threadIdx.x + o]});
      lo[threadIdx.x] = r.lo;
      hi[threadIdx.x] = r.hi;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out->s2_lo = lo[0];
    out->s2_hi = hi[0];
  }
}

namespace {
template <bool W>
int launch_mod_rows(const long long* off, const int* col, const int* w, long long n, const int* labels,
                    const int* work, Counters* ctr, const unsigned long long* totals, unsigned long long* sigma,
                    int2* pieces, ModSums* out, const DeviceInfo& di, cudaStream_t s) {
  const int g = 8 * di.sm_count;
  const long long blocks = (n + 255) / 256;
  mod_lane_kernel<W><<<(int)(blocks < g ? blocks : g), 256, 0, s>>>(off, col, w, labels, n, ctr, sigma, out);
  int launches = 1;
  for (int k = NCLASS - 1; k >= CLS_BINNED; --k) {   // the longest rows first; classes without a vertex not at all
    if (!totals[k]) continue;
    ++launches;
    if (k >= CLS_BLOCK)
      mod_block_kernel<W><<<4 * di.sm_count, 512, 0, s>>>(off, col, w, labels, n, work, ctr, k, sigma, pieces, out);
    else if (k >= 5)
      mod_group_kernel<32, W><<<g, 256, 0, s>>>(off, col, w, labels, n, work, ctr, k, sigma, out);
    else if (k == 4)
      mod_group_kernel<16, W><<<g, 256, 0, s>>>(off, col, w, labels, n, work, ctr, k, sigma, out);
    else
      mod_group_kernel<8, W><<<g, 256, 0, s>>>(off, col, w, labels, n, work, ctr, k, sigma, out);
  }
  if (pieces) {
    mod_piece_kernel<W><<<4 * di.sm_count, 512, 0, s>>>(off, col, w, labels, n, ctr, sigma, pieces, out);
    ++launches;
  }
  return launches;
}
}  // namespace

long long modularity_partials(const DeviceInfo& di) { return 4ll * di.sm_count; }

cudaError_t launch_modularity(const long long* off, const int* col, const int* w, long long n, const int* labels,
                              const int* work, Counters* ctr, const unsigned long long* totals,
                              unsigned long long* sigma, unsigned long long* partials, long long nparts, int2* pieces,
                              ModSums* out, const DeviceInfo& di, cudaStream_t s, int* kernels) {
  *kernels = 0;
  if (n <= 0) return cudaSuccess;
  static_assert(CLS_BINNED == 3 && MOD_LANE_ROW == 4, "classes 0..2 are the rows of one lane");
  int launches = w ? launch_mod_rows<true>(off, col, w, n, labels, work, ctr, totals, sigma, pieces, out, di, s)
                   : launch_mod_rows<false>(off, col, w, n, labels, work, ctr, totals, sigma, pieces, out, di, s);
  long long np = nparts < modularity_partials(di) ? nparts : modularity_partials(di);
  if (np > (n + 255) / 256) np = (n + 255) / 256;
  mod_square_kernel<<<(int)np, 256, 0, s>>>(sigma, n, partials);
  mod_final_kernel<<<1, 256, 0, s>>>(partials, np, out);
  *kernels = launches + 2;
  count_launches(*kernels);
  return cudaGetLastError();
}

}  // namespace gsl

// split_kernels.cu -- split last (Algorithm 2) and label renumbering on sm_103a.
//
// Algorithm 2 labels every connected piece of every community with the
// vertex its BFS started from; scanning start vertices in ascending order
// makes that the smallest vertex of the piece.  Here the pieces are found
// as the connected components of the subgraph of edges (u, j) with
// C[u] == C[j], by lock-free union-find instead of one BFS per piece:
//   - parent[v] <= v at all times; a union links the larger of two roots
//     below the smaller with atomicCAS, so the root of every tree is the
//     smallest vertex of its component -- Algorithm 2's label;
//   - find follows parents with path halving (benign racy stores: every
//     value written is an ancestor of the vertex);
//   - edges are offered in two phases (neighbour sampling after Sutton,
//     Ben-Nun and Bar-Noy, "Optimizing Parallel Graph Connectivity
//     Computation via Subgraph Sampling", IPDPS 2018): first every vertex
//     links with its first SPLIT_SAMPLE row entries of its own community;
//     after flattening, every community names one of its pieces (the root
//     one of its vertices below a root holds, the last write winning; the
//     community of the most frequent root among sampled vertices names that
//     root; a community of roots only names the piece of the first vertex that
//     asks), and only vertices outside their community's named piece offer
//     their remaining entries.  An edge inside a named piece is redundant,
//     and an edge between a named piece and another piece of the same
//     community is offered from the other end, so the components are the
//     same as offering every edge.  Communities are mapped to a table of n
//     slots (label c in [0, n) to slot c, others by a hash); a slot shared by
//     two communities names a piece of one of them, and the other's vertices
//     then all offer their entries, which is slower but still exact.
// The second phase takes the vertices in natural order, one lane each: a warp
// per vertex spent four dependent loads on finding out that there was nothing
// to offer, and stray members, written last, named their own single-vertex
// pieces, so that most of their communities offered everything (4 M-vertex
// planted partition: 0.85 ms of hooks, now 0.08).
// All loops are bounded (parents strictly decrease along a path and a
// failed CAS strictly lowers the root being linked); the bound is a safety
// net that raises ERRBIT_TIMEOUT.
#include "uf_device.cuh"

namespace gsl {

namespace {

constexpr int SPLIT_SAMPLE = 2;   // same-community links per vertex before the named pieces are known
constexpr int SPLIT_SCAN = 8;     // row entries the sampling pass looks at for them

// Offers entry e of u's row to the union-find if it is an intra-community
// edge; returns whether it was one.
template <int F>
__device__ __forceinline__ bool hook_entry(const int* col, const int* labels, int* p, long long n, int u, int cu,
                                           long long e, int* err, UfCap<F> cap) {
  const int j = ld_stream(col + e);
  if ((unsigned)j >= (unsigned)n) {
    raise_err(err, ERRBIT_INVALID);
    return false;
  }
  if (j == u || ld_label_ro(labels + j) != cu) return false;
  uf_unite(p, u, j, err, cap);
  return true;
}

}  // namespace

__global__ void init_parent_kernel(int* __restrict__ p, long long n) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x)
    p[v] = (int)v;
}

// Every vertex links with the first SPLIT_SAMPLE same-community
// neighbours among its first SPLIT_SCAN row entries.
// The first two entries' columns and labels are requested together; the
// rest of the scan (when they are not both links) goes one entry at a time.
// Bound by unions that compete: in plain grid strides a whole community links
// at once, thousands of threads on a handful of roots.  So every warp takes
// SAMPLE_PART vertices in a row, and the warps in flight spread over 4 times
// as many communities: the split of 4 million vertices in communities of 2000
// takes 0.636 ms instead of 0.855, and LPA + split of R-MAT 20 1.29 instead of
// 1.38.  Longer parts gain little more (0.60 ms from 512 vertices on) and give
// up what neighbouring warps share in L2: a 38 million vertex lattice is 0.3%
// slower with 128, 1% with 512, 1.5% with 4096.
constexpr long long SAMPLE_PART = 128;

template <int F>
__global__ void __launch_bounds__(256) sample_link_kernel(const long long* __restrict__ off,
                                                          const int* __restrict__ col,
                                                          const int* __restrict__ labels, int* p, long long n,
                                                          Counters* ctr, UfCap<F> cap) {
  static_assert(SPLIT_SAMPLE == 2, "the first two entries are loaded together");
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long even = ((n + nwarps - 1) / nwarps + 31) & ~31ll;
  const long long part = even < SAMPLE_PART ? even : SAMPLE_PART;
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  // u runs through this warp's parts: the next one starts nwarps parts on
  long long u = w * part + (threadIdx.x & 31), end = (w + 1) * part;
  for (; u < n; u += 32) {
    if (u >= end) {
      u += (nwarps - 1) * part;
      end += nwarps * part;
      if (u >= n) break;
    }
    const long long s = off[u], e = off[u + 1];
    if (s >= e) continue;
    const int cu = labels[u];
    const int j0 = ld_stream(col + s), j1 = s + 1 < e ? ld_stream(col + s + 1) : -1;
    const bool v0 = (unsigned)j0 < (unsigned)n, v1 = (unsigned)j1 < (unsigned)n;
    if (!v0 || (s + 1 < e && !v1)) raise_err(&ctr->err, ERRBIT_INVALID);
    const int l0 = v0 && j0 != (int)u ? ld_label_ro(labels + j0) : ~cu;
    const int l1 = v1 && j1 != (int)u ? ld_label_ro(labels + j1) : ~cu;
    int linked = 0;
    if (l0 == cu) {
      uf_unite(p, (int)u, j0, &ctr->err, cap);
      ++linked;
    }
    if (l1 == cu) {
      uf_unite(p, (int)u, j1, &ctr->err, cap);
      ++linked;
    }
    for (int k = 2; k < SPLIT_SCAN && linked < SPLIT_SAMPLE && s + k < e; ++k)
      linked += hook_entry(col, labels, p, n, (int)u, cu, s + k, &ctr->err, cap) ? 1 : 0;
  }
}

// Every parent becomes the root.
template <int F>
__global__ void flatten_kernel(int* p, int* out, long long n, Counters* ctr, UfCap<F> cap) {   // out may equal p
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x)
    out[v] = uf_find(p, (int)v, &ctr->err, cap);
}

// The most frequent root among 1024 sampled vertices (one block
// of 1024 threads: sample, bitonic sort in shared memory, longest run).
__global__ void __launch_bounds__(1024) giant_kernel(const int* p, long long n, Counters* ctr) {
  __shared__ int a[1024];
  const unsigned t = threadIdx.x;
  const unsigned long long x = ((unsigned long long)hash32(t * 2654435761u + 0x9E37u) * (unsigned long long)n) >> 32;
  a[t] = __ldcg(p + x);
  __syncthreads();
  for (unsigned k = 2; k <= 1024; k <<= 1) {
    for (unsigned j = k >> 1; j > 0; j >>= 1) {
      const unsigned q = t ^ j;
      if (q > t) {
        const bool up = (t & k) == 0;
        const int x0 = a[t], x1 = a[q];
        if ((x0 > x1) == up) {
          a[t] = x1;
          a[q] = x0;
        }
      }
      __syncthreads();
    }
  }
  if (t == 0) {
    int best = a[0], best_run = 0, run = 0;
    for (int i = 0; i < 1024; ++i) {
      run = (i > 0 && a[i] == a[i - 1]) ? run + 1 : 1;
      if (run > best_run) {
        best_run = run;
        best = a[i];
      }
    }
    ctr->giant = best;
  }
}

// Every community names a piece: the root its vertices hold after flattening,
// the last write winning; then the community of the most frequent sampled
// root (giant_kernel) names that root.  Roots do not name themselves: a
// community's stray members, scattered over the ids and often written last,
// would name their single-vertex pieces and leave the others to offer their
// whole rows.  Slots nobody names here hold -1 (community_name).
__global__ void name_pieces_kernel(const int* __restrict__ p, const int* __restrict__ labels, long long n,
                                   int* __restrict__ named) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    const int r = p[v];
    if (r == (int)v) continue;
    int* slot = named + comm_slot(labels[v], n);
    if (*slot != r) *slot = r;   // one community may hold nearly every vertex: mostly read
  }
}

__global__ void name_giant_kernel(const int* __restrict__ labels, long long n, int* __restrict__ named,
                                  const Counters* ctr) {
  const int g = ctr->giant;
  if (g >= 0 && (long long)g < n) named[comm_slot(labels[g], n)] = g;
}

// Vertices outside their community's named piece offer entries SPLIT_SAMPLE..
// of their row (both directions: the other end may be skipped), unless their
// parent has become the named root by the time their row is reached.  Rows of up
// to HOOK_LANE entries go by their lane, longer ones by this warp, two at a time,
// while they are HOOK_STEPS steps of 32 entries in all.  A warp that meets more
// lists them, for a warp each or past HOOK_WARP entries for a block each
// (hook_listed_kernel), which also stop inside a row.  Left where they
// were met, the dense rows of a small graph, or the heavy ids of one that is
// sorted by degree, ran on a fraction of the chip: split after LPA of 60,000
// vertices of 1500 entries 2.43 ms, listed 0.43; 2 million vertices, a few of
// them heavy, in 1000 communities 1.64 and 0.77.  Asked again, hubs seldom read
// their rows: R-MAT 24 in 1000 random communities 9.5 and 4.4 ms.  At 32 steps
// the heavy ids take 1.19 ms, at 128 the split of 30,000 vertices of 900 entries
// 0.45 instead of 0.35; one row at a time a circulant of 16 neighbours takes 0.49
// instead of 0.38.
constexpr int HOOK_LANE = 8, HOOK_STEPS = 64, HOOK_WARP = 2048;

// Offers the entries k, k + step, .. below end of u's row, none when u's parent
// is the root `name`; EVERY: and no more once it has become that.
template <bool EVERY, int F>
__device__ __forceinline__ void hook_row(const int* col, const int* labels, int* p, long long n, int u, int cu,
                                         int name, long long k, long long end, int step, int* err, UfCap<F> cap) {
  int ru = __ldcg(p + u);
  for (; k < end; k += step) {
    const int j = ld_stream(col + k);
    if (ru == name) return;
    const int next = EVERY ? __ldcg(p + u) : ru;
    if ((unsigned)j >= (unsigned)n) raise_err(err, ERRBIT_INVALID);
    else if (j != u && ld_label_ro(labels + j) == cu && __ldcg(p + j) != ru) uf_unite(p, u, j, err, cap);
    ru = next;
  }
}

template <int F>
__global__ void __launch_bounds__(256) hook_kernel(const long long* __restrict__ off, const int* __restrict__ col,
                                                    const int* __restrict__ labels, int* p, long long n,
                                                    int* __restrict__ list, Counters* ctr, UfCap<F> cap,
                                                    int* named) {
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long w = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); w < n; w += stride) {   // warp-uniform
    const long long u = w + lane;
    long long s = 0, e = 0;
    int cu = 0, ru = 0, slot = -1, name = 0;
    if (u < n) {
      s = off[u] + SPLIT_SAMPLE;
      e = off[u + 1];
      if (s < e) {
        ru = __ldcg(p + u);
        cu = labels[u];
        slot = (int)comm_slot(cu, n);
        name = named[slot];   // through L1: a name stays, and -1 is looked at again
      }
    }
    // one lane asks for all of its community; a row that the sampling pass has
    // scanned is offered for less
    const bool ask = name == -1 && e - s > SPLIT_SCAN - SPLIT_SAMPLE;
    if (__any_sync(FULL, ask)) {
      const unsigned same = __match_any_sync(FULL, ask ? slot : -1);
      const int leader = __ffs((int)same) - 1;
      int first = 0;
      if (ask && lane == leader) first = community_name(named + slot, ru);
      first = __shfl_sync(FULL, first, leader);
      if (ask) name = first;
    }
    bool offer = slot >= 0 && ru != name;
    if (offer && e - s > HOOK_WARP) {   // from the list's end
      list[n - 1 - (long long)atomicAdd(&ctr->hook_long, 1u)] = (int)u;
      offer = false;
    }
    if (offer && e - s <= HOOK_LANE) {
      hook_row<false>(col, labels, p, n, (int)u, cu, name, s, e, 1, &ctr->err, cap);
      offer = false;
    }
    __syncwarp();
    unsigned mask = __ballot_sync(FULL, offer);
    if (!mask) continue;
    if (__reduce_add_sync(FULL, offer ? (unsigned)((e - s + 31) >> 5) : 0u) > HOOK_STEPS) {
      unsigned base = 0;
      if (lane == 0) base = atomicAdd(&ctr->hook_rows, (unsigned)__popc(mask));
      base = __shfl_sync(FULL, base, 0);
      if (offer) list[base + __popc(mask & ((1u << lane) - 1u))] = (int)u;
      continue;
    }
    while (mask) {   // two rows at a time, half a warp each
      const int r0 = __ffs((int)mask) - 1;
      mask &= mask - 1;
      const int r1 = __ffs((int)mask) - 1;   // -1: none
      mask &= mask - 1;
      const int r = lane < 16 ? r0 : (r1 < 0 ? r0 : r1);
      const long long rs = __shfl_sync(FULL, s, r), re = __shfl_sync(FULL, e, r);
      const int rc = __shfl_sync(FULL, cu, r), rn = __shfl_sync(FULL, name, r);
      hook_row<false>(col, labels, p, n, (int)w + r, rc, rn, rs + (r1 < 0 ? lane : (lane & 15)), re, r1 < 0 ? 32 : 16,
                      &ctr->err, cap);
      __syncwarp();
    }
  }
}

// The listed rows: the long ones a block each, then the others a warp each.  A
// warp takes a run of the list, so that the rows in flight lie in many communities
// and their unions seldom compete.
template <int F>
__global__ void __launch_bounds__(512) hook_listed_kernel(const long long* __restrict__ off, const int* __restrict__ col,
                                                           const int* __restrict__ labels, int* p, long long n,
                                                           const int* __restrict__ list, Counters* ctr, UfCap<F> cap,
                                                           const int* __restrict__ named) {
  const unsigned longs = ctr->hook_long, cnt = ctr->hook_rows;
  for (unsigned i = blockIdx.x; i < longs; i += gridDim.x) {
    const int u = list[n - 1 - i], cu = labels[u];
    hook_row<true>(col, labels, p, n, u, cu, named[comm_slot(cu, n)], off[u] + SPLIT_SAMPLE + threadIdx.x, off[u + 1],
                   (int)blockDim.x, &ctr->err, cap);
  }
  const unsigned nwarps = (gridDim.x * blockDim.x) >> 5, part = (cnt + nwarps - 1) / nwarps;
  const unsigned w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (unsigned i = w * part; i < cnt && i < (w + 1) * part; ++i) {
    const int u = list[i], cu = labels[u];
    hook_row<true>(col, labels, p, n, u, cu, named[comm_slot(cu, n)], off[u] + SPLIT_SAMPLE + (threadIdx.x & 31),
                   off[u + 1], 32, &ctr->err, cap);
  }
}

// ---------------------------------------------------------------- renumber
// rank of every representative (out[v] == v) among all representatives,
// then out[v] = rank[out[v]]: pieces numbered 0..k-1 by smallest vertex.
constexpr int RN_THREADS = 256;
constexpr int RN_ITEMS = 8;
constexpr long long RN_TILE = (long long)RN_THREADS * RN_ITEMS;

// Representatives per tile of RN_TILE vertices (thread t of the block takes
// vertices t * RN_ITEMS .. + RN_ITEMS - 1 of the tile, as rn_rank_kernel
// does).  A thread's eight labels are read as two 16-byte loads where the
// array is 16-byte aligned and the eight lie inside it.
__global__ void __launch_bounds__(RN_THREADS) rn_count_kernel(const int* __restrict__ rep, long long n,
                                                               unsigned long long* __restrict__ block_sums) {
  static_assert(RN_ITEMS == 8, "two 16-byte loads per thread");
  __shared__ unsigned acc;
  if (threadIdx.x == 0) acc = 0;
  __syncthreads();
  const long long v0 = (long long)blockIdx.x * RN_TILE + (long long)threadIdx.x * RN_ITEMS;
  unsigned c = 0;
  if ((reinterpret_cast<uintptr_t>(rep) & 15) == 0 && v0 + RN_ITEMS <= n) {
    const int4 x = __ldg(reinterpret_cast<const int4*>(rep + v0));
    const int4 y = __ldg(reinterpret_cast<const int4*>(rep + v0 + 4));
    const int v = (int)v0;
    c = (x.x == v) + (x.y == v + 1) + (x.z == v + 2) + (x.w == v + 3) + (y.x == v + 4) + (y.y == v + 5) +
        (y.z == v + 6) + (y.w == v + 7);
  } else {
    for (int k = 0; k < RN_ITEMS; ++k) {
      const long long v = v0 + k;
      if (v < n && rep[v] == (int)v) ++c;
    }
  }
  c = __reduce_add_sync(FULL, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(&acc, c);
  __syncthreads();
  if (threadIdx.x == 0) block_sums[blockIdx.x] = acc;
}

__global__ void __launch_bounds__(1024) rn_scan_kernel(unsigned long long* block_sums, long long nb,
                                                        unsigned long long* total) {
  __shared__ unsigned long long buf[1024];
  __shared__ unsigned long long carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (long long b0 = 0; b0 < nb; b0 += 1024) {
    const long long b = b0 + threadIdx.x;
    const unsigned long long x = b < nb ? block_sums[b] : 0ull;
    buf[threadIdx.x] = x;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {   // Hillis-Steele inclusive scan
      const unsigned long long y = threadIdx.x >= (unsigned)o ? buf[threadIdx.x - o] : 0ull;
      __syncthreads();
      buf[threadIdx.x] += y;
      __syncthreads();
    }
    if (b < nb) block_sums[b] = carry + buf[threadIdx.x] - x;   // exclusive
    __syncthreads();
    if (threadIdx.x == 0) carry += buf[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = carry;
}

__global__ void __launch_bounds__(RN_THREADS) rn_rank_kernel(const int* __restrict__ rep, long long n,
                                                              const unsigned long long* __restrict__ block_sums,
                                                              int* __restrict__ rank) {
  __shared__ unsigned warp_tot[RN_THREADS / 32];
  const long long t0 = (long long)blockIdx.x * RN_TILE;
  unsigned flags = 0, c = 0;
  for (int k = 0; k < RN_ITEMS; ++k) {
    const long long v = t0 + (long long)threadIdx.x * RN_ITEMS + k;
    if (v < n && rep[v] == (int)v) { flags |= 1u << k; ++c; }
  }
  // exclusive scan of c over the block
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned incl = c;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  unsigned wbase = 0;
  for (int w = 0; w < wid; ++w) wbase += warp_tot[w];
  unsigned long long r = block_sums[blockIdx.x] + wbase + incl - c;
  for (int k = 0; k < RN_ITEMS; ++k) {
    if (flags >> k & 1u) {
      const long long v = t0 + (long long)threadIdx.x * RN_ITEMS + k;
      rank[v] = (int)r++;
    }
  }
}

__global__ void rn_apply_kernel(const int* __restrict__ rep, int* __restrict__ out, const int* __restrict__ rank,
                                long long n) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x)
    out[v] = rank[rep[v]];
}

// ------------------------------------------------------------ Algorithm 4
// A community is disconnected when it holds more than one piece.  With the
// pieces from the union-find (every piece labelled by its smallest vertex),
// each piece representative adds one to its community's count; flags are
// the communities with a count of two or more.
__global__ void disc_count_kernel(const int* __restrict__ rep, const int* __restrict__ labels, long long n,
                                  int* __restrict__ cnt, Counters* ctr) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    const int c = labels[v];
    if ((unsigned)c >= (unsigned)n) {
      raise_err(&ctr->err, ERRBIT_INVALID);
      continue;
    }
    if (rep[v] == (int)v) atomicAdd(cnt + c, 1);
  }
}

__global__ void disc_flag_kernel(const int* __restrict__ cnt, long long n, unsigned char* __restrict__ flags,
                                 unsigned long long* total) {
  unsigned long long mine = 0;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const bool f = cnt[c] >= 2;
    if (flags) flags[c] = f ? 1 : 0;
    mine += f ? 1ull : 0ull;
  }
  mine = warp_sum_u64(mine);
  if ((threadIdx.x & 31) == 0 && mine) atomicAdd(total, mine);
}

// ------------------------------------------------------------ Algorithm 1
// One sweep of SL-LP / SL-LPP: every vertex (with pruning: every vertex of
// the current frontier) takes the smallest piece label over itself and its
// neighbours of the same community, in place.  A warp handles a vertex;
// labels only decrease, so concurrent updates converge to the same fixed
// point as the sequential sweep: the smallest vertex id of every piece.
// With pruning, a vertex that changed puts its same-community neighbours in
// the next frontier.
__global__ void __launch_bounds__(256) split_lp_kernel(const long long* __restrict__ off, const int* __restrict__ col,
                                                       const int* __restrict__ labels, long long n, int* cp,
                                                       unsigned char* __restrict__ fcur,
                                                       unsigned char* __restrict__ fnext, int prune, Counters* ctr) {
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  unsigned long long my_dn = 0;
  for (long long v = warp; v < n; v += nwarps) {
    if (prune) {
      if (!fcur[v]) continue;   // warp-uniform
      __syncwarp();
      if (lane == 0) fcur[v] = 0;
    }
    const long long s = off[v], e = off[v + 1];
    const int c = labels[v];
    const int cur = __ldcg(cp + v);
    int m = cur;
    for (long long x = s + lane; x < e; x += 32) {
      const int j = ld_stream(col + x);
      if ((unsigned)j >= (unsigned)n) {
        raise_err(&ctr->err, ERRBIT_INVALID);
        continue;
      }
      if (ld_label_ro(labels + j) == c) {
        const int pj = __ldcg(cp + j);
        m = pj < m ? pj : m;
      }
    }
    m = __reduce_min_sync(FULL, m);
    if (m < cur) {   // warp-uniform
      if (lane == 0) __stcg(cp + v, m);
      my_dn += lane == 0 ? 1ull : 0ull;
      if (prune) {
        for (long long x = s + lane; x < e; x += 32) {
          const int j = ld_stream(col + x);
          if ((unsigned)j < (unsigned)n && ld_label_ro(labels + j) == c) fnext[j] = 1;
        }
      }
    }
  }
  my_dn = warp_sum_u64(my_dn);
  if (lane == 0 && my_dn) atomicAdd(&ctr->dn, my_dn);
}

__global__ void iota_kernel(int* __restrict__ p, unsigned char* __restrict__ f, long long n) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    p[v] = (int)v;
    if (f) f[v] = 1;
  }
}

// ---------------------------------------------------------------- launchers
namespace {
int grid_for(long long items, int block, const DeviceInfo& di, int per_sm = 8) {
  long long b = (items + block - 1) / block;
  const long long cap = (long long)per_sm * di.sm_count;
  if (b > cap) b = cap;
  return (int)(b < 1 ? 1 : b);
}
}  // namespace

template <int F>
void launch_split_t(const long long* off, const int* col, long long n, const int* labels, int* list, Counters* ctr,
                    int* parent, int* named, int* out, UfCap<F> cap, const DeviceInfo& di, cudaStream_t s) {
  const int g = grid_for(n, 256, di);
  init_parent_kernel<<<g, 256, 0, s>>>(parent, n);
  sample_link_kernel<F><<<g, 256, 0, s>>>(off, col, labels, parent, n, ctr, cap);
  flatten_kernel<F><<<g, 256, 0, s>>>(parent, parent, n, ctr, cap);
  giant_kernel<<<1, 1024, 0, s>>>(parent, n, ctr);
  cudaMemsetAsync(named, 0xFF, sizeof(int) * (size_t)n, s);
  name_pieces_kernel<<<g, 256, 0, s>>>(parent, labels, n, named);
  name_giant_kernel<<<1, 1, 0, s>>>(labels, n, named, ctr);
  hook_kernel<F><<<g, 256, 0, s>>>(off, col, labels, parent, n, list, ctr, cap, named);
  hook_listed_kernel<F><<<4 * di.sm_count, 512, 0, s>>>(off, col, labels, parent, n, list, ctr, cap, named);
  flatten_kernel<F><<<g, 256, 0, s>>>(parent, out, n, ctr, cap);
  count_launches(SPLIT_LAUNCHES);
}

cudaError_t launch_split(const long long* off, const int* col, long long n, const int* labels, int* list,
                         Counters* ctr, int* parent, int* named, int* out, const Tuning& t, const DeviceInfo& di,
                         cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (t.uf_cap == UF_CAP)
    launch_split_t(off, col, n, labels, list, ctr, parent, named, out, UfCap<UF_CAP>{0}, di, s);
  else
    launch_split_t(off, col, n, labels, list, ctr, parent, named, out, UfCap<0>{t.uf_cap}, di, s);
  return cudaGetLastError();
}

cudaError_t launch_disconnected(const int* rep, const int* labels, long long n, int* cnt, unsigned char* flags,
                                unsigned long long* total, Counters* ctr, const DeviceInfo& di, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  cudaMemsetAsync(cnt, 0, sizeof(int) * (size_t)n, s);
  cudaMemsetAsync(total, 0, sizeof(unsigned long long), s);
  disc_count_kernel<<<grid_for(n, 256, di), 256, 0, s>>>(rep, labels, n, cnt, ctr);
  disc_flag_kernel<<<grid_for(n, 256, di), 256, 0, s>>>(cnt, n, flags, total);
  count_launches(2);
  return cudaGetLastError();
}

cudaError_t launch_split_lp_init(int* cp, unsigned char* f, long long n, const DeviceInfo& di, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  iota_kernel<<<grid_for(n, 256, di), 256, 0, s>>>(cp, f, n);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_split_lp_sweep(const long long* off, const int* col, const int* labels, long long n, int* cp,
                                  unsigned char* fcur, unsigned char* fnext, int prune, Counters* ctr,
                                  const DeviceInfo& di, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  split_lp_kernel<<<16 * di.sm_count, 256, 0, s>>>(off, col, labels, n, cp, fcur, fnext, prune, ctr);
  count_launches(1);
  return cudaGetLastError();
}

long long renumber_blocks(long long n) { return (n + RN_TILE - 1) / RN_TILE; }

cudaError_t launch_renumber(const int* rep, int* out, long long n, int* rank, unsigned long long* block_sums,
                            long long nblocks_cap, unsigned long long* k_dev, const DeviceInfo& di, cudaStream_t s) {
  const long long nb = renumber_blocks(n);
  if (nb > nblocks_cap) return cudaErrorInvalidValue;
  if (n <= 0) {
    cudaMemsetAsync(k_dev, 0, sizeof(unsigned long long), s);
    return cudaGetLastError();
  }
  rn_count_kernel<<<(int)nb, RN_THREADS, 0, s>>>(rep, n, block_sums);
  rn_scan_kernel<<<1, 1024, 0, s>>>(block_sums, nb, k_dev);
  count_launches(2);
  if (!out) return cudaGetLastError();   // count only
  rn_rank_kernel<<<(int)nb, RN_THREADS, 0, s>>>(rep, n, block_sums, rank);
  rn_apply_kernel<<<grid_for(n, 256, di), 256, 0, s>>>(rep, out, rank, n);
  count_launches(2);
  return cudaGetLastError();
}

}  // namespace gsl

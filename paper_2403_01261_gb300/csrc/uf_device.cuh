// uf_device.cuh -- the lock-free union-find of the split (split_kernels.cu says
// how it is used).  Included by one translation unit each.
#pragma once

#include "kernels.h"

namespace gsl {

namespace {

// Bound of the union-find loops.  The default is a compile-time constant
// (the loops are measurably faster that way); kernels instantiated with
// UfCap<0> take a bound lowered at run time (gsl_ctx_set_retry_bounds).
constexpr int UF_CAP = 1 << 26;
template <int FIXED>
struct UfCap {
  int runtime;
  __device__ __forceinline__ int get() const { return FIXED > 0 ? FIXED : runtime; }
};

template <int F>
__device__ __forceinline__ int uf_find(int* p, int x, int* err, UfCap<F> cap) {
  const int bound = cap.get();
  for (int it = 0; it < bound; ++it) {
    const int px = __ldcg(p + x);
    if (px == x) return x;
    const int ppx = __ldcg(p + px);
    if (ppx != px) __stcg(p + x, ppx);
    x = ppx;
  }
  raise_err(err, ERRBIT_TIMEOUT);
  return x;
}

template <int F>
__device__ __forceinline__ void uf_unite(int* p, int a, int b, int* err, UfCap<F> cap) {
  const int bound = cap.get();
  for (int it = 0; it < bound; ++it) {
    a = uf_find(p, a, err, cap);
    b = uf_find(p, b, err, cap);
    if (a == b) return;
    const int hi = a > b ? a : b, lo = a > b ? b : a;
    const int old = atomicCAS(p + hi, hi, lo);
    if (old == hi) return;
    a = old;   // hi got a parent meanwhile: continue from it
    b = lo;
  }
  raise_err(err, ERRBIT_TIMEOUT);
}

// Slot of community label c in a table of n entries.
__device__ __forceinline__ long long comm_slot(int c, long long n) {
  if (c >= 0 && (long long)c < n) return c;
  unsigned x = (unsigned)c;
  x ^= x >> 16;
  x *= 0x7FEB352Du;
  x ^= x >> 15;
  x *= 0x846CA68Bu;
  x ^= x >> 16;
  return (long long)(((unsigned long long)x * (unsigned long long)n) >> 32);
}

// The root by which a community names its piece, asked by a vertex of it whose
// parent is ru: other vertices offer their entries, this piece's do not.  A slot
// that is still empty belongs to communities of which no two vertices were
// linked: the first vertex to ask names its own piece, the others offer theirs
// to it.  A community of one vertex so reads no entry past the sampled ones,
// whatever its row (R-MAT 22 with every vertex its own community: 0.51 ms with
// every root naming itself, 1.51 with none, 0.29 so).  Exact as before: a slot
// is named once, every vertex that skips shares a tree with the name, and an
// edge of which one end skips is offered by the other.
__device__ __forceinline__ int community_name(int* slot, int ru) {
  const int name = __ldcg(slot);
  if (name != -1) return name;
  const int first = atomicCAS(slot, -1, ru);
  return first == -1 ? ru : first;
}

}  // namespace

}  // namespace gsl

// kernels.h -- host-side launchers of the GSL-LPA kernels (internal header).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include "common.cuh"

namespace gsl {

// Majority filter: where nothing hides the longest row, rows of more than
// FILTER_LONG entries are read in pieces of FILTER_PIECE by any number of blocks.
constexpr int FILTER_LONG = 65536, FILTER_PIECE = 8192;
struct FilterLong {   // one such row
  unsigned long long hit, all;   // weight of the tested label and of the whole row, so far
  unsigned long long read;       // entries read
  int v, cls;
  unsigned left;                 // pieces still to end
};

// Arguments of one label-propagation sweep.
struct SweepArgs {
  const long long* off;      // CSR offsets [n+1]
  const int* col;            // CSR columns [nnz]
  const int* w;              // weights [nnz] or nullptr (unit)
  const int* prev;           // labels read (C^{t-1}); == next in async mode
  int* next;                 // labels written (C^t)
  unsigned char* fnext;      // frontier flags of the next sweep (set, never cleared here)
  const int* work;           // worklist (class regions at Counters::cls_start)
  const int* work2;          // rows the majority filter left, the same regions (null: no filter this sweep)
  const unsigned* bits;      // majority filter: one bit per vertex carrying the giant label
  FilterLong* long_rows;     // majority filter: long rows and their pieces as (row, piece); null: the graph has none
  int2* long_pieces;
  Counters* ctr;
  int* scratch;              // label lists of rows longer than a block's registers, one region per block
  long long scratch_region;  // ints per region (three lists of the longest row)
  int* hub_scratch;          // the same for class 9, one region for each of the first hub_blocks blocks
  long long hub_region;
  int hub_blocks;            // 0: class 9 has its own kernels
  long long n;
  // batched mode (many graphs packed in one CSR); all null for one graph
  const int* gid;            // graph of every vertex
  const long long* vptr;     // vertex range of every graph [vptr[g], vptr[g+1])
  unsigned* dn_graph;        // per-graph change count of this sweep
  const int* stop;           // nonzero: every graph is done, kernels return at once
  int ident;                 // prev is the identity labelling (not read)
  int check;                 // validate weights and weighted degrees
  int mark;                  // mark neighbours of changed vertices in fnext
  const int* lg;             // sync mode: labels gathered per entry, lg[e] = prev[col[e]] (null: gather)
  int spread;                // labels read are nearly all distinct (sweep 2 from the identity labelling)
  unsigned* kw;              // weighted degree per vertex of classes 6-9: written in sweep 1 (check), then read by
                             // the majority filter and class 6's own-label test (null: none)
  int probe_cap;             // bound on the probes of one hash-table insert (past it: ERRBIT_TIMEOUT)
};

struct Tuning {
  int warp_max = 1024;       // class 7 upper degree bound (a small block per row)
  int blk_max = 131072;       // class 8 upper degree bound (a block per row; above: class 9)
  int blk_slots = 12288;     // shared-memory table slots per block of the hub kernels
  int blk_block = 512;       // threads per block of the hub-piece kernel
  int pregather = 0;         // two-phase sweeps: 0 never, 1 when the frontier is large, 2 always
  int majority = 1;          // own-label majority pass: 0 never, 1 once labels settle, 2 always
  int hub_cluster_max = 1 << 30;  // hubs up to this degree go to one thread-block cluster each (0: never)
  int probe_cap = 1 << 24;   // bound on the probes of one hash-table insert
  int uf_cap = 1 << 26;      // bound on the steps of one union-find find or union (split_kernels.cu UF_CAP)
};

// Degree bounds of the classes (see common.cuh).
struct ClassBounds {
  int warp_small;
  int warp_max;
  int blk_max;
};

struct DeviceInfo {
  int sm_count = 0;
  int max_smem_optin = 0;
  int cooperative = 0;
};

// lpa_kernels.cu
cudaError_t launch_class_histogram(const long long* off, long long n, long long nnz, const Tuning& t,
                                   Counters* ctr, const DeviceInfo& di, cudaStream_t s);
// phase >= 0: only the frontier vertices of that phase of an asynchronous
// sweep (a hash of the vertex id and `seed`); the others keep their flags,
// as do the vertices of the classes below first_cls.
cudaError_t launch_bin(const long long* off, long long n, unsigned char* fcur, int all_active,
                       const Tuning& t, int* work, Counters* ctr, const DeviceInfo& di, cudaStream_t s,
                       const int* gid = nullptr, const unsigned char* done = nullptr, const int* stop = nullptr,
                       int phase = -1, unsigned seed = 0, int first_cls = 0);
// The class counts of an all-active binning whose worklist is still in place.
cudaError_t launch_all_counts(Counters* ctr, int first_cls, cudaStream_t s);
// tile_kernels.cu: the rows of 1..4 entries among the vertices [v0, v1) (all
// of them, or those flagged in fcur, whose flags are cleared), and the rows
// of classes 3..5 on the worklist.
cudaError_t launch_sweep_lanes(const SweepArgs& a, int weights, bool async_mode, long long v0, long long v1,
                               unsigned char* fcur, int all_active, const unsigned char* done, int phase,
                               unsigned seed, const DeviceInfo& di, cudaStream_t s);
cudaError_t launch_sweep_tile(const SweepArgs& a, int cls, int weights, bool async_mode, const DeviceInfo& di,
                              cudaStream_t s);
// Between the two phases of an asynchronous sweep (see Counters::phase_cls).
cudaError_t launch_phase_reset(Counters* ctr, const int* stop, cudaStream_t s);
// sketch_kernels.cu: the rows of class cls on the worklist, none longer than
// `longest`.  Rows longer than
// sketch_register_row() need SweepArgs::scratch, sketch_blocks() regions of
// three times the longest row's length.  weights: 0 unit, 1 int32, 2 int32 with 64-bit
// sums (so in the other sweep launchers).
long long sketch_blocks(const DeviceInfo& di);
long long sketch_register_row();
// Blocks of a launch with per_sm resident per SM; with lists no more than
// sketch_blocks() of the same device, since each uses its own scratch region.
int sketch_grid(int per_sm, bool lists, const DeviceInfo& di);
cudaError_t launch_sketch(const SweepArgs& a, int cls, int longest, int weights, bool async_mode,
                          const DeviceInfo& di, cudaStream_t s);
// Classes 3..8 on the worklist; class 8's launch sweeps class 9 as well when
// SweepArgs::hub_blocks is set.
cudaError_t launch_sweep_class(const SweepArgs& a, int cls, int weights, bool async_mode, const Tuning& t,
                               int longest, const DeviceInfo& di, cudaStream_t s);
void count_launches(long long k);   // process-wide tally of kernels this library launched
// Raises kernel fn's dynamic shared-memory limit to at least `bytes` (never
// lowers it, so launches of other host threads with smaller tables stay
// valid); thread-safe.
cudaError_t raise_smem_limit(const void* fn, size_t bytes);
long long launches_total();
// filter_kernels.cu: majority filter over the classes from first_cls (or 6,
// when one label dominates a sample of the entries) to 9.  Settled rows are
// written; the others go to `out` (n ints, class regions as in the worklist)
// and become the class counts: the sweep kernels launched next need
// SweepArgs::work2 = out.  bits: n / 32 + 1 words of scratch.  warps, blocks:
// whether classes 6-7 and 8-9 hold rows.
cudaError_t launch_majority_filter(const SweepArgs& a, long long nnz, int* out, unsigned* bits, int weights,
                                   bool async_mode, int first_cls, bool sample, unsigned seed, bool warps, bool blocks,
                                   const DeviceInfo& di, cudaStream_t s, int* kernels = nullptr);
// The class counts of first_cls..last_cls become the rows a filter passed on.
cudaError_t launch_filter_counts(Counters* ctr, const int* stop, cudaStream_t s, int first_cls, int last_cls);
// Edge-parallel label gather for a synchronous sweep: lg[e] = prev[col[e]]
// for every CSR entry (-1 for an out-of-range column).
cudaError_t launch_pregather(const int* col, long long nnz, const int* prev, long long n, int* lg,
                             const DeviceInfo& di, cudaStream_t s);
// Streaming sweep 1 (identity labels, unit weights): bits holds nnz/32+1
// words of scratch; rows that are not strictly increasing are flagged in
// `bad` (n bytes, zero on entry) and left for the hash kernels.
cudaError_t launch_ident_stream(const long long* off, long long n, const int* col, long long nnz, unsigned* bits,
                                unsigned char* bad, int* next, Counters* ctr, const DeviceInfo& di, cudaStream_t s);
// The first two of those passes (row starts, strict-increase check).
cudaError_t launch_row_check(const long long* off, long long n, const int* col, long long nnz, unsigned* bits,
                             unsigned char* bad, Counters* ctr, const DeviceInfo& di, cudaStream_t s);
// Sweeps 1 and 2 while the columns arrive in row-aligned chunks
// (gsl_gsllpa_host): the row-start bitmap (offsets only, bits zeroed
// first), sweep 1 from each row's first entries assuming every row is
// strictly increasing (col may be host memory the device reads), the
// verification of a landed chunk [e0, e1) (flags rows that are not strictly
// increasing in `bad` and raises *any_bad), and the all-active binning of
// the chunk's rows [v0, v1).
cudaError_t launch_rowstart(const long long* off, long long n, unsigned* bits, long long nbits_words,
                            const DeviceInfo& di, cudaStream_t s);
cudaError_t launch_ident_first(const long long* off, long long n, const int* col, const unsigned char* zero_flags,
                               int* next, Counters* ctr, const DeviceInfo& di, cudaStream_t s);
cudaError_t launch_chunk_check(const long long* off, long long n, const int* col, long long nnz, long long e0,
                               long long e1, const unsigned* bits, unsigned char* bad, unsigned* any_bad,
                               Counters* ctr, const DeviceInfo& di, cudaStream_t s);
cudaError_t launch_bin_range(const long long* off, long long v0, long long v1, const Tuning& t, int* work,
                             Counters* ctr, const DeviceInfo& di, cudaStream_t s, int first_cls = 0);
// Streaming sweep 1 with float weights: for strictly increasing rows the
// label is the neighbour of largest weight (smallest id among equals).
cudaError_t launch_ident_stream_f32(const long long* off, long long n, const int* col, const float* wf,
                                    long long nnz, unsigned* bits, unsigned char* bad, int* next, Counters* ctr,
                                    const DeviceInfo& di, cudaStream_t s);
cudaError_t launch_init_labels(const int* init, int* a, int* b, long long n, Counters* ctr,
                               const DeviceInfo& di, cudaStream_t s);
ClassBounds class_bounds(const Tuning& t);

// batch_kernels.cu
cudaError_t launch_fill_gid(const long long* vptr, int num_graphs, long long n, int* gid, const DeviceInfo& di,
                            cudaStream_t s);
cudaError_t launch_graph_update(int t, double tol, int max_iters, const long long* vptr, int num_graphs,
                                const unsigned* dn_graph, int* iters, unsigned char* done, int* stop,
                                cudaStream_t s);
cudaError_t launch_batch_final(const int* const* bufs, const int* iters, const int* gid, long long n, int async_mode,
                               int* out, const DeviceInfo& di, cudaStream_t s);
cudaError_t launch_localize(const long long* vptr, const int* gid, long long n, int* labels, const DeviceInfo& di,
                            cudaStream_t s);

// hub_kernels.cu: class 9 in pieces.  Arrays sized by the class's vertex
// total (best, own, wsum, used_cnt: one per hub; piece_start, ustart: one
// more) and its entry total E (used: E slot indices; tab: 2 E slots, all
// EMPTY between sweeps; slot indices must stay below 2^32).
struct HubPlan {
  int* piece_start;             // first piece of frontier hub i (prefix sums)
  long long* ustart;            // first entry of hub i's regions (prefix sums of degrees)
  unsigned long long* best;     // largest packed key over hub i's pieces
  unsigned* own;                // entries of hub i carrying its own label
  unsigned long long* wsum;     // weighted degree of hub i (checked when weighted)
  unsigned* used_cnt;           // table slots claimed for hub i
  unsigned* used;               // their indices: hub i at used[ustart[i]..]
  unsigned long long* tab;      // hub i's table at tab[2 ustart[i] .. 2 ustart[i+1])
  int* clu;                     // frontier hubs taken by clusters (indices i), hub_clusters of them
};
// True when a piece always fits the block kernel's shared table.
bool hub_pieces_fit(const Tuning& t);
// Class 9: plan, cluster kernel (hubs up to t.hub_cluster_max), pieces, final
// pass.  *kernels = launches made.
cudaError_t launch_hub_pieces(const SweepArgs& a, const HubPlan& hp, bool weighted, bool async_mode,
                              const Tuning& t, const DeviceInfo& di, cudaStream_t s, int* kernels);

// float_kernels.cu: sweeps with float32 weights and float64 sums.  Classes
// 6..9 use one block per row; rows whose 2 d slots exceed shared memory use
// the block's region (`region` slots, >= 2 * largest degree) of gkeys/gvals,
// float_table_blocks(di) regions in all.
long long float_table_blocks(const DeviceInfo& di);
cudaError_t launch_sweep_f32(const SweepArgs& a, const float* wf, int cls, bool async_mode, unsigned* gkeys,
                             double* gvals, long long region, const DeviceInfo& di, cudaStream_t s);
// Own-label majority filter for float weights (classes 7-8, float64 sums),
// as launch_majority_filter.
cudaError_t launch_majority_filter_f32(const SweepArgs& a, const float* wf, int* out, bool async_mode,
                                       const DeviceInfo& di, cudaStream_t s);
// Exact fixed-point form of float weights (float_kernels.cu): out[0..2] =
// 1024 + lowest set-bit exponent, 1024 + highest set-bit exponent, invalid
// flag; then wi[e] = w[e] * 2^shift.
cudaError_t launch_f32_exact_scan(const float* w, long long nnz, int* out, const DeviceInfo& di, cudaStream_t s);
cudaError_t launch_f32_to_fixed(const float* w, long long nnz, int shift, int* wi, const DeviceInfo& di,
                                cudaStream_t s);
// Eq. 1 with float weights: sums[0] = 2m, sums[1] = S1, sums[2] = S2 (sigma: n doubles).
cudaError_t launch_modularity_f32(const long long* off, const int* col, const float* wf, const int* labels,
                                  long long n, double* sigma, double* sums, Counters* ctr, const DeviceInfo& di,
                                  cudaStream_t s);

// solo_kernel.cu: sweeps and split of a small graph in one cooperative launch.
constexpr int SOLO_SWEEPS = 64;        // sweeps whose counts fit the state
constexpr long long SOLO_ROW_MAX = 32768;   // longest row it takes
constexpr int SOLO_LISTS = 32;         // blocks with label lists for rows of more than 4096 entries
// Entries of such rows from which the class kernels, which have a list per
// block, are faster (ms a call, one launch / class kernels): 1.0 M in rows of
// 8000 0.40 / 0.57, 2.0 M 0.61 / 0.54, 3.2 M 0.89 / 0.55; 1.15 M in rows of 4500
// 0.47 / 0.58, 3.6 M 1.07 / 0.54; 1.9 M in rows of 30,000 0.44 / 0.47, 3 M 0.74 / 0.47.
constexpr unsigned long long SOLO_HUGE_ENTRIES = 3ull << 19;
struct SoloState {   // zero before the launch
  unsigned arrived, released, verdict, abandoned;   // grid barrier
  unsigned nlong, nhuge;               // rows of more than 256 and of more than 4096 entries
  int sweeps, converged;
  unsigned long long huge_entries;     // entries of the rows of more than 4096
  long long longest;                   // more than SOLO_ROW_MAX (a longer row, or too many huge entries): nothing was done
  unsigned long long changed[SOLO_SWEEPS], active[SOLO_SWEEPS];
  unsigned long long scanned, pieces;
  long long time_ns[3];                // start, end of the sweeps, end of the split
  Counters ctr;                        // only its error bits are used
};
struct SoloArgs {
  SoloState* state;
  long long nnz;
  const int* labels_init;              // sweeps start here (null: identity)
  const int* labels_in;                // split alone: the labels to split
  int lpa, split;
  double tol;
  int max_iters;                       // <= SOLO_SWEEPS
  int* lab[2];
  unsigned char* flag[2];
  int* lists;                          // SOLO_LISTS label lists of 3 * SOLO_ROW_MAX ints
  int* longs;                          // scratch, n ints each
  int* parent;
  int* named;
  int* out;
};
cudaError_t launch_solo(const SweepArgs& a, const SoloArgs& q, int weights, const DeviceInfo& di, cudaStream_t s);

// split_kernels.cu.  list, parent and named: n ints of scratch each;
// Counters::hook_rows and hook_long zero.
constexpr int SPLIT_LAUNCHES = 9;
cudaError_t launch_split(const long long* off, const int* col, long long n, const int* labels,
                         int* list, Counters* ctr, int* parent, int* named, int* out, const Tuning& t,
                         const DeviceInfo& di, cudaStream_t s);
cudaError_t launch_renumber(const int* rep, int* out, long long n, int* rank, unsigned long long* block_sums,
                            long long nblocks_cap, unsigned long long* k_dev, const DeviceInfo& di,
                            cudaStream_t s);
long long renumber_blocks(long long n);
// Algorithm 4 from split representatives: cnt (n ints) receives the pieces
// per community, flags (nullable, n bytes) the disconnected communities,
// *total their number.
cudaError_t launch_disconnected(const int* rep, const int* labels, long long n, int* cnt, unsigned char* flags,
                                unsigned long long* total, Counters* ctr, const DeviceInfo& di, cudaStream_t s);
// Algorithm 1: cp = identity (and every frontier flag set), then sweeps
// until Counters::dn stays zero.
cudaError_t launch_split_lp_init(int* cp, unsigned char* f, long long n, const DeviceInfo& di, cudaStream_t s);
cudaError_t launch_split_lp_sweep(const long long* off, const int* col, const int* labels, long long n, int* cp,
                                  unsigned char* fcur, unsigned char* fnext, int prune, Counters* ctr,
                                  const DeviceInfo& di, cudaStream_t s);

// modularity_kernels.cu
struct ModSums {
  unsigned long long two_m;
  unsigned long long s1;
  unsigned long long s2_lo, s2_hi;
};
// `work` holds the binning of classes CLS_BINNED.. of every vertex, totals
// the host's copy of the class totals, pieces (null: rows are not shared) room
// for those of the rows past FILTER_LONG, Counters::filter_pieces zero.
// *kernels = launches made.
cudaError_t launch_modularity(const long long* off, const int* col, const int* w, long long n,
                              const int* labels, const int* work, Counters* ctr, const unsigned long long* totals,
                              unsigned long long* sigma, unsigned long long* partials, long long nparts,
                              int2* pieces, ModSums* out, const DeviceInfo& di, cudaStream_t s, int* kernels);
long long modularity_partials(const DeviceInfo& di);

}  // namespace gsl

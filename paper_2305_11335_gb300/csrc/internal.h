// internal.h -- host-side launchers of the library's kernels (not part of the ABI).
//
// Every launcher works on one class (dpc_device.cuh): the instances of a call
// that share the padded dimension dp and the gridded dimension g.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "dpc_device.cuh"

namespace dpc {

// Streaming multiprocessors of the current device (grid caps are multiples
// of it); queried once per device.
unsigned sm_count();

// Polls a bounded device-side wait makes before it gives up: `dflt`, or the
// smaller value in the environment variable DPC_TEST_WAIT_LIMIT (tests use 0
// to make every such wait give up at once and check the recovery path).
uint32_t wait_limit(uint32_t dflt);

// Largest single device allocation the library may make (the environment
// variable DPC_WORKSPACE_LIMIT_BYTES, unset = no limit).  dev_alloc fails
// without calling cudaMalloc when a request is larger.
bool dev_alloc(void** p, size_t bytes);

// Kernels enqueued by the current call (the entry points hold the library
// lock while enqueueing, so a plain counter suffices).
extern long long g_kernel_launches;
inline void count_launches(int k) { g_kernel_launches += k; }

// Host-computed constants of one cutoff (the [host] fields of CutGeom).
struct CutHost {
  double dc, dc2;
  float t_in, t_out, band_mul, band_add;
  int32_t skip;  // dependent search: points with rho < skip are skipped
  int32_t pad;
};
CutHost make_cut_host(double d_cut, int dp);

// Cutoffs passed by value (single-instance calls that have no device copy).
constexpr int kCutChunk = 16;
struct CutArgs {
  CutHost h[kCutChunk];
};

// ---- binning (binning.cu) ---------------------------------------------------
void launch_class_init(const ClassView& cv, int g, int ib, int bcap, int* status, cudaStream_t st);
// chunk tables of a multi-instance class (InstDev::chunk0 gives each instance's first chunk)
void launch_chunks(const ClassView& cv, uint32_t* chunk_inst, uint32_t* chunk_pos, cudaStream_t st);
void launch_bbox(const void* pts, int dtype, const ClassView& cv, int g, cudaStream_t st);
// per-instance grid and per (instance, cutoff) parameters; cutoffs come from
// hc_dev ([ninst][ncut], device) or, when it is null, from hc_host (ncut <= kCutChunk)
void launch_setup(const ClassView& cv, CutGeom* cuts, int ncut, const CutHost* hc_dev,
                  const CutHost* hc_host, cudaStream_t st);
// level and block radius of one cutoff (cuts: [ninst]) again: rpref = 0 the
// default rule, rpref > 0 the finest level whose block radius is <= rpref
void launch_set_radius(const ClassView& cv, CutGeom* cuts, int rpref, cudaStream_t st);
// near-dependent search `shift` grid levels finer than the density's (0: same)
void launch_near_level(const ClassView& cv, CutGeom* cuts, int shift, cudaStream_t st);
// The block geometry several cutoffs share: per instance that of the largest
// of the cutoffs in `mask` (bit c: cutoff c of cuts [ncut][ninst]) into
// geo [ninst]
void launch_group_geometry(const ClassView& cv, const CutGeom* cuts, int ncut, unsigned long long mask,
                           CutGeom* geo, cudaStream_t st);
// cut ([ninst]) takes the level, radius and far bounds of geo ([ninst])
void launch_adopt_geometry(const ClassView& cv, const CutGeom* geo, CutGeom* cut, cudaStream_t st);
// (count: the digit counts of launch_sort_clear, or null)
void launch_codes(const void* pts, int dtype, const ClassView& cv, int g, unsigned long long* codes,
                  uint32_t* ids, uint32_t* count, cudaStream_t st);
void launch_gather(const void* pts, int dtype, const ClassView& cv, int dp,
                   const unsigned long long* codes_a, const unsigned long long* codes_b,
                   const uint32_t* ids_a, const uint32_t* ids_b, float* spts,
                   unsigned long long* scode, uint32_t* sid, cudaStream_t st);
// occupied level-k cells of every instance for one cutoff (cuts: [ninst]) -> hash
void launch_cells(const unsigned long long* scode, const ClassView& cv, int g, const CutGeom* cuts,
                  HashInfo* hi, unsigned long long* hkeys, uint2* hvals, uint32_t hcap,
                  cudaStream_t st);

// ---- radix sort (sort.cu) ------------------------------------------------------
constexpr uint32_t kSortMaxPasses = 8;   // 8-bit digits of a 64-bit key
constexpr uint32_t kSortSmall = 1u << 17, kSortMiddle = 1u << 21;  // tiles of 1024, 2048 items up to here
// 32-bit words of sort scratch that serve every size up to n: per tile and
// digit a published 64-bit count, the digit counts of every pass, a tile
// counter per pass (and slack)
constexpr size_t sort_hist_words_for(uint64_t n) {
  const uint64_t a = ((n < kSortSmall ? n : kSortSmall) + 1023) / 1024;
  const uint64_t b = ((n < kSortMiddle ? n : kSortMiddle) + 2047) / 2048;
  const uint64_t c = (n + 4095) / 4096;
  const uint64_t ab = a > b ? a : b, t = ab > c ? ab : c;
  return (size_t)(t ? t : 1) * 256u * 2u + kSortMaxPasses * 256u + kSortMaxPasses + 8u;
}
size_t sort_hist_words(uint32_t n);
// one-time kernel attribute setup (called before any stream capture)
void sort_init();
// Clears the scratch for a sort of n items and returns the digit counts
// [kSortMaxPasses][256] for a kernel that fills them (rs_count_digits in
// dpc_device.cuh) ahead of launch_sort(counted = true).  Worth it up to
// kSortMiddle points; beyond, the shared-memory atomics cost the code kernel more
// than one more read of the keys (1e7 points in 3-D: binning 1.36 ms counted, 1.32
// not).
uint32_t* launch_sort_clear(uint32_t n, uint32_t* hist, cudaStream_t st);
// Sorts (codes_a, ids_a) by code, LSD over the device-side pass count
// sort_passes(cls->S, cls->ib); the result lands in the _a buffers if that
// count is even, else in _b.
void launch_sort(unsigned long long* codes_a, unsigned long long* codes_b, uint32_t* ids_a,
                 uint32_t* ids_b, uint32_t n, const ClassGeom* cls, uint32_t* hist, bool counted,
                 cudaStream_t st);

// ---- radix tree (tree.cu) ------------------------------------------------------
// Tree over the class's sorted keys; root[i] = the internal node whose leaves
// are exactly instance i (kNoNode for an instance of one point).
void launch_tree_build(const unsigned long long* scode, const ClassView& cv, Node* nodes, uint32_t* root,
                       cudaStream_t st);
// Every internal node's child record (dpc_device.cuh: the children's
// indices, their largest order keys and, with `boxes`, their bounding boxes
// over rec_dims(dp, dmax) coordinates) into nrec, kRecWordsMax words per node at most;
// the boxes depend only on the points, so once per binning suffices.
void launch_tree_maxkey(const unsigned long long* skey, const float* spts, int dp, int dmax, uint32_t n,
                        Node* nodes, uint32_t* visit, float* nrec, bool boxes, cudaStream_t st);
// The dimension of the boxes of a class whose points have dp padded and at most
// dmax coordinates.  5-D, 1e6 points: far search
// 4.47 ms with 6, 5.07 with 8; 1e5 points .494 and .546.
inline int rec_dims(int dp, int dmax) { return dp == 8 && dmax <= 6 ? 6 : dp; }

// Work layouts of the density and near-dependent kernels:
//   union    a warp owns 32 consecutive sorted points (one query per lane) and
//            streams the union of their blocks through shared memory, every
//            candidate a broadcast read (block.cuh)
//   segment  the 32 points are split into segments of a cell or of a few
//            consecutive ones; the points around a segment are staged in shared
//            memory once and its queries spread over the lanes (CandTile)
//   tree     (near phase only) no block scan: every query goes to the tree
//            search of the far phase
//   tensor   (density, 5-8 dimensions, float32 filter) the distance tiles on the
//            tensor cores (tc_density.cu); other cases fall back to segment
//   pairs    (density only) segments of one cell, every unordered pair counted
//            once for both of its points (density.cu, k_density_pairs)
// seg_cells (segment layouts): a segment may span several consecutive cells
// while their bounding box grown by R holds at most seg_cells cells (0: one
// cell per segment)
//   cell     one warp per occupied cell: the block's points staged in shared
//            memory, every lane one query (or a share of one query's
//            candidates for cells below 32 points) against all of them
//            (cell_tile.cu)
enum { kLayoutUnion = 1, kLayoutSegment = 2, kLayoutTree = 3, kLayoutTensor = 4, kLayoutPairs = 5,
       kLayoutCell = 6 };

// ---- density (density.cu) -------------------------------------------------------
// Chunks from which float32 points in binary64 are counted pair by pair (every
// pair once) and not in segments (every query's block, but a chunk's queries
// spread over several warps).  The binary64 pipe is the bound where the chip is
// full; below that the longest chunk is.  Density in ms, segments / pairs, uniform
// points: 2-D 1e4 .041 / .070, 2e4 .063 / .080, 4e4 .132 / .121, 3e5 1.35 / .54;
// 3-D 1e4 .078 / .134, 2e4 .133 / .150, 4e4 .29 / .22, 3e5 3.0 / 1.1; 5-D 1e4 .56 /
// 1.07, 2e4 1.29 / 1.33, 4e4 3.4 / 2.4; 7-D 2e4 3.8 / 5.4, 4e4 10.4 / 11.8, 1e5
// 45 / 28.
constexpr uint32_t kBinary64Pairs = 800;
// Cutoffs evaluated in one density launch: they share the block geometry of
// the largest of them; cut[j] is the [ninst] thresholds of cutoff j, rho[j]
// its output row.
constexpr int kMultiCuts = 4;
struct MultiCut {
  int m = 0;
  const CutGeom* cut[kMultiCuts] = {};
  int32_t* rho[kMultiCuts] = {};
};
// min_fill: points per occupied cell from which a tensor layout runs; below it
// the CUDA-core layout launched beside it does (tensor_fill in dpc_device.cuh;
// 0: always tensor).
// rho of every point for one cutoff (cuts: [ninst]); rho_out is indexed by
// output index (sid); d: the largest dimension of the class
// (prec: 0 float32 filter, 1 binary64, 2 binary64 mode on int32 points)
void launch_density(int dp, int g, int d, int prec, int layout, const float* spts,
                    const unsigned long long* scode, const uint32_t* sid, const ClassView& cv,
                    const CutGeom* cuts, HashInfo* hi, const unsigned long long* hkeys,
                    const uint2* hvals, uint4* pieces, int32_t* rho_out,
                    unsigned long long* skey, Counters* ctr, cudaStream_t st,
                    int seg_cells = 0, uint32_t min_fill = 0);
// rho of the cutoffs of `mc` in one pass over the blocks of `geo` ([ninst]; the
// hash holds its level's cells): tensor tiles for dp = 8 with the float32
// filter, segments otherwise.  No order keys are written.
void launch_density_multi(int dp, int g, int d, int prec, const float* spts, const unsigned long long* scode,
                          const uint32_t* sid, const ClassView& cv, const CutGeom* geo, HashInfo* hi,
                          const unsigned long long* hkeys, const uint2* hvals, uint4* pieces,
                          const MultiCut& mc, Counters* ctr, cudaStream_t st, int seg_cells,
                          uint32_t min_fill);
// the tensor-core form of the density step (dp = 8, float32 filter only; d:
// the largest dimension of the class; pieces: N entries of scratch; skey: the
// order keys of cutoff 0, or null)
void launch_density_tc(int d, const float* spts, const unsigned long long* scode, const uint32_t* sid,
                       const ClassView& cv, const CutGeom* geo, HashInfo* hi,
                       const unsigned long long* hkeys, const uint2* hvals, uint4* pieces,
                       const MultiCut& mc, unsigned long long* skey, Counters* ctr, uint32_t min_fill,
                       cudaStream_t st);
// the cell layout of the density step (cell_tile.cu)
void launch_density_cell(int dp, int g, bool fp64, const float* spts,
                         const unsigned long long* scode, const uint32_t* sid, const ClassView& cv,
                         const CutGeom* cuts, const HashInfo* hi, const unsigned long long* hkeys,
                         const uint2* hvals, int32_t* rho_out, unsigned long long* skey,
                         Counters* ctr, cudaStream_t st);
// order keys of sorted points from densities given by output index
void launch_keys_from_rho(const int32_t* rho, const uint32_t* sid, uint32_t n,
                          unsigned long long* skey, cudaStream_t st);

// ---- dependent points (dependent.cu) ----------------------------------------------
struct FarQueue {
  uint32_t* pos;   // sorted position of each queued query
  float* s1;       // best float32 distance found by the near phase (FP32 mode)
  double* s1d;     // best binary64 distance found by the near phase (FP64 mode)
  uint32_t* pos2;  // the same for the queries passed to the far phase's second round
  float* s1_2;
  double* s1d2;
};
// Dependent points already found for another cutoff of the same call (null:
// none), with this cutoff's densities and the caller's points: bounds for the
// far search.
struct FarHint {
  const int32_t* lambda = nullptr;
  const int32_t* rho = nullptr;
  const void* pts = nullptr;
  int dtype = 0;
};
// lambda and delta are indexed by output index; lambda values are
// instance-local ids
// (skip_fill, tree layout: nothing from that many points per occupied cell on;
// min_fill, union layout: nothing below it)
void launch_dep_near(int dp, int g, int dmax, bool fp64, int layout, const float* spts,
                     const unsigned long long* scode, const unsigned long long* skey,
                     const ClassView& cv, int32_t rho_skip, const void* pts, int dtype,
                     const CutGeom* cuts, const HashInfo* hi, const unsigned long long* hkeys,
                     const uint2* hvals, int32_t* lambda, double* delta, FarQueue q, Counters* ctr,
                     cudaStream_t st, const float* nbox, const uint32_t* roots, int seg_cells = 0,
                     uint32_t skip_fill = 0, uint32_t min_fill = 0);
// the cell layout of the near phase (cell_tile.cu)
void launch_dep_near_cell(int dp, int g, bool fp64, const float* spts,
                          const unsigned long long* scode, const unsigned long long* skey,
                          const ClassView& cv, int32_t rho_skip, const void* pts, int dtype,
                          const CutGeom* cuts, const HashInfo* hi,
                          const unsigned long long* hkeys, const uint2* hvals, int32_t* lambda,
                          double* delta, FarQueue q, Counters* ctr, cudaStream_t st);
// the tensor-core form of the near phase (dp = 8, float32 filter only; d and
// pieces as for launch_density_tc)
void launch_dep_near_tc(int d, const float* spts, const unsigned long long* scode, const uint32_t* sid,
                        const unsigned long long* skey, const ClassView& cv, int32_t rho_skip,
                        const void* pts, int dtype, const CutGeom* cuts, HashInfo* hi,
                        const unsigned long long* hkeys, const uint2* hvals, uint4* pieces,
                        int32_t* lambda, double* delta, FarQueue q, Counters* ctr, uint32_t min_fill,
                        cudaStream_t st);
void launch_dep_far(int dp, int dmax, bool fp64, const float* spts, const unsigned long long* scode,
                    const unsigned long long* skey, const ClassView& cv, const CutGeom* cuts,
                    const float* nbox, const uint32_t* root, FarQueue q, const FarHint& hint,
                    int32_t* lambda, double* delta, Counters* ctr, cudaStream_t st);

// ---- decision graph (decision.cu) -------------------------------------------------
// top-k by gamma = rho * delta and the (rho, delta) histogram of every instance
// of the class (rho, delta indexed by output index; top/gamma [n_inst][k] and
// hist [n_inst][rho_bins][delta_bins] by batch row, InstDev::row); 0, or -1
// when a launch failed
int launch_decision(const int32_t* rho, const double* delta, const ClassView& cv, int k,
                     int32_t* top, double* gamma, int rho_bins, int delta_bins, double delta_lo,
                     unsigned long long* hist, void* scratch, int* status, cudaStream_t st);
// device scratch launch_decision needs for a class of ninst instances
size_t decision_scratch_bytes(uint32_t ninst, uint32_t n, int k);
// ---- priority range search (range.cu) -------------------------------------------
struct PrangeArgs {
  uint32_t nq;              // queries
  int32_t n_inst;           // instances of the batch
  const int32_t* q_inst;    // [nq] batch row of each query (device)
  const double* q_box;      // [nq][2][kMaxDim] lo then hi (device)
  const int32_t* q_rho;     // [nq] thresholds (device)
  const int32_t* rowmap;    // [n_inst] class-local index or -1; null: one_row only
  int32_t one_row;          // the batch row of a single-instance class
  long long* count;         // [nq] matches (device output)
};
void launch_prange_init(const PrangeArgs& a, int32_t* ids, int max_out, int* status,
                        cudaStream_t st);
// the box hierarchy of one class (rec: at least 22 words per chunk)
void launch_prange_boxes(int dp, const float* spts, const unsigned long long* skey,
                         const ClassView& cv, float* rec, cudaStream_t st);
// one class.  mode 0 (count): cnt[q] for the class's queries, 0 for the
// others, and count[q]; 1 (fill): keys (q << 31 | id) at off[q]..; 2 (top):
// count[q], the max_out <= prange_top_ids() smallest ids of each query, and
// the class's matches added to *total
void launch_prange(int dp, int mode, const float* spts, const unsigned long long* skey,
                   const ClassView& cv, float* rec, const PrangeArgs& a, uint32_t* cnt,
                   const unsigned long long* off, unsigned long long* keys, int32_t* ids,
                   int max_out, unsigned long long* total, int* status, cudaStream_t st);
int prange_top_ids();
void launch_prange_scan(const uint32_t* cnt, uint32_t nq, unsigned long long* off, cudaStream_t st);
void launch_prange_scatter(const unsigned long long* keys, uint64_t total,
                           const unsigned long long* off, uint32_t nq, int max_out, int32_t* ids,
                           int* status, cudaStream_t st);

int decision_max_topk();
// padding of every top-k row (-1, NaN; `pad`: some rows have no points) and
// zero histograms for n_inst rows
void launch_decision_init(int n_inst, int k, bool pad, int32_t* top, double* gamma, int rho_bins,
                          int delta_bins, unsigned long long* hist, cudaStream_t st);

// ---- small instances (small.cu) ---------------------------------------------------
// All pairs straight from the caller's coordinates (every instance of the
// class has dimension d); cutoffs as for launch_setup.  rho of cutoff k at
// rho + k * rho_stride.
void launch_small_density(int d, bool fp64, const void* pts, int dtype, const ClassView& cv,
                          const CutHost* hc_dev, const CutHost* hc_host, int ncut, int32_t* rho,
                          uint64_t rho_stride, Counters* ctr, int* status, cudaStream_t st);
// lambda and delta of cutoff `cut` of the call from its densities
void launch_small_dependent(int d, bool fp64, const void* pts, int dtype, const ClassView& cv,
                            const CutHost* hc_dev, const CutHost* hc_host, int ncut, int cut,
                            int32_t rho_skip, const int32_t* rho, int32_t* lambda, double* delta,
                            Counters* ctr, int* status, cudaStream_t st);
// Largest instance that all pairs serve faster than the grid (small_class in
// api.cu gives the measurements).
constexpr uint32_t small_limit(int d, bool fp64, bool density_only) {
  return fp64 ? (d <= 3 ? 2048u : 4096u) : (density_only && d <= 5 ? 16384u : 8192u);
}
// Points of an instance whose pointers fit a CTA's shared memory (k_small_labels).
constexpr uint32_t kSmallLabelPoints = 32768;
// Whether the labels of a class take one launch with a CTA per instance, or the
// launches of labels.cu over all points.  A CTA costs a few microseconds however
// small its instance, and one CTA alone falls behind at 24,000 points.  Labels
// phase of a run, launches -> CTA per instance (us): one instance of 8,000 points
// 38 -> 18, 16,000 40 -> 31, 24,000 42 -> 43, 32,000 42 -> 63 (4 of them 42 -> 63,
// 40 of them 126 -> 80); 1,000 instances of 20 points 26 -> 14, 10,000 of them
// 32 -> 82, 100,000 62 -> 740; 10,000 of 300 points 87 -> 117, 4,000 of 1,000
// 108 -> 64, 2,000 of 2,000 119 -> 55.
inline bool labels_by_instance(uint32_t n, uint32_t ninst, uint32_t nmax) {
  if (nmax > kSmallLabelPoints || (nmax > 20480u && (uint64_t)n < 16ull * nmax)) return false;
  return ninst <= 4096u || (uint64_t)n >= 1024ull * ninst;
}
void launch_small_labels(const int32_t* rho, const int32_t* lambda, const double* delta,
                         const ClassView& cv, uint32_t nmax, const LabelParams* params,
                         LabelParams one, int32_t* label, int* status, cudaStream_t st);
// one-time kernel attribute setup (called before any stream capture)
void small_init();

// ---- labels (labels.cu) -------------------------------------------------------------
int label_rounds(uint32_t n);
// Labels of every point of the class for one cutoff (arrays indexed by output
// index); params: [ninst] on the device, or null for a single instance (`one`);
// nmax: the largest instance; flags needs label_rounds(nmax) + 1 ints.
void launch_labels(const int32_t* rho, const int32_t* lambda, const double* delta,
                   const ClassView& cv, uint32_t nmax, const LabelParams* params,
                   LabelParams one, int32_t* label, int32_t* flags, int* status, cudaStream_t st);

}  // namespace dpc

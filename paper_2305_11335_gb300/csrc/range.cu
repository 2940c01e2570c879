// range.cu -- priority range search (the appendix on range queries): for a
// query (instance, closed axis-parallel box [lo, hi], threshold rho_q), every
// point of the instance inside the box whose priority -- its density -- is
// above rho_q.
//
// The search runs on a 32-ary box hierarchy over the key-sorted points: a
// level-1 node is one 32-point chunk, a level-l node 32 consecutive nodes
// below it, each with the bounding box, the smallest and largest density and
// the smallest id of its points (the pruning the appendix describes for the
// priority search kd-tree: a node is entered only if its largest density is
// above rho_q and its box meets the query's).  One warp per query: the 32
// lanes test the 32 children of a node at once, or the 32 points of a chunk,
// always on consecutive records, so every step is one coalesced load and a
// ballot instead of a chain of dependent node loads per lane.  A node wholly
// inside the query (box and densities) is counted without being entered.
// The sorted float copy holds every coordinate exactly (float32 inputs as
// they are, int32 inputs are range-checked to |x| <= 2^24), and the query's
// bounds are rounded inwards to float32 (x >= lo exactly when x >= the least
// float32 >= lo), so every test is exact in float32.
//
// Ids: up to kTopIds per query the warp keeps the smallest ids it has met in a
// shared buffer of at least twice that many; when it fills up it is sorted,
// the rest dropped, and the largest id kept bounds what is still appended --
// and which wholly inside nodes are still entered.  One pass then gives counts
// and ids.  More ids than that: a COUNT pass, then a FILL pass that writes
// (query << 31 | instance-local id) for every match at the query's offset; the
// host sorts those keys (radix sort) and a last kernel scatters the first
// max_out ids of every query, ascending, into its output row.
//
// 1e6 points in 3-D, 2e4 queries of 2,600 matches on average, 64 ids each:
// 36.6 ms per call with a lane-per-node walk of the radix tree in two passes and
// a global sort of the 5e7 match keys, 0.99 ms now (the search itself 0.52).
#include <cstdint>

#include "internal.h"

namespace dpc {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kPrThreads = 128;
constexpr int kPrWarps = kPrThreads / 32;
constexpr int kBoxLevels = 8;  // 32^7 chunks and more

// Node record: lo(DP) | hi(DP) | largest density, smallest density, smallest id, 0.
template <int DP>
constexpr int box_words() { return 2 * DP + 4; }

struct BoxTree {
  float* rec;                    // every level, level 1 first
  uint32_t off[kBoxLevels + 1];  // first node of level l
  uint32_t cnt[kBoxLevels + 1];  // nodes of level l (level 1: the chunks)
  int levels;
};

struct BoxSum {
  uint32_t rmax, rmin, id;
};

// Reduces the lanes' boxes (ordered-uint lo, hi) and sums over the warp and
// writes the record of one node.
template <int DP>
__device__ __forceinline__ void box_reduce_store(const uint32_t* lo, const uint32_t* hi, BoxSum z, int lane,
                                                 float* __restrict__ rec) {
  float v = 0.f;
#pragma unroll
  for (int a = 0; a < DP; ++a) {
    const float l = ord_float(__reduce_min_sync(kFull, lo[a]));
    const float h = ord_float(__reduce_max_sync(kFull, hi[a]));
    if (lane == a) v = l;
    if (lane == DP + a) v = h;
  }
  const uint32_t rmax = __reduce_max_sync(kFull, z.rmax);
  const uint32_t rmin = __reduce_min_sync(kFull, z.rmin);
  const uint32_t id = __reduce_min_sync(kFull, z.id);
  if (lane == 2 * DP) v = __uint_as_float(rmax);
  if (lane == 2 * DP + 1) v = __uint_as_float(rmin);
  if (lane == 2 * DP + 2) v = __uint_as_float(id);
  if (lane < box_words<DP>()) rec[lane] = v;
}

// densities as ordered unsigned words (any int32)
__device__ __forceinline__ uint32_t rho_ord(int32_t r) { return (uint32_t)r ^ 0x80000000u; }
__device__ __forceinline__ int32_t key_rho(unsigned long long k) { return (int32_t)(k >> 32); }

// Level 1: one warp per chunk.
template <int DP>
__global__ void __launch_bounds__(256)
k_box_chunks(const float* __restrict__ spts, const unsigned long long* __restrict__ skey, ClassView cv, BoxTree T) {
  const int lane = threadIdx.x & 31;
  for (uint32_t c = blockIdx.x * 8u + (threadIdx.x >> 5); c < cv.nchunk; c += gridDim.x * 8u) {
    uint32_t i, p0, end;
    cv.chunk(c, i, p0, end);
    const uint32_t p = p0 + lane;
    uint32_t lo[DP], hi[DP];
    BoxSum z{0u, 0xffffffffu, 0xffffffffu};
#pragma unroll
    for (int a = 0; a < DP; ++a) {
      lo[a] = 0xffffffffu;
      hi[a] = 0u;
    }
    if (p < end) {
      const Pt<DP> x = load_pt<DP>(spts, p);
      const unsigned long long k = skey[p];
#pragma unroll
      for (int a = 0; a < DP; ++a) lo[a] = hi[a] = float_ord(x.x[a]);
      z.rmax = z.rmin = rho_ord(key_rho(k));
      z.id = key_id(k);
    }
    box_reduce_store<DP>(lo, hi, z, lane, T.rec + (size_t)c * box_words<DP>());
  }
}

template <int DP>
__device__ __forceinline__ void load_box(const float* __restrict__ rec, uint32_t node, float* v) {
  constexpr int W = box_words<DP>();
  const float4* r = reinterpret_cast<const float4*>(rec) + (size_t)node * (W / 4);
#pragma unroll
  for (int k = 0; k < W / 4; ++k) {
    const float4 q = r[k];
    v[4 * k] = q.x; v[4 * k + 1] = q.y; v[4 * k + 2] = q.z; v[4 * k + 3] = q.w;
  }
}

// Level l from level l - 1: one warp per node.
template <int DP>
__global__ void __launch_bounds__(256) k_box_level(BoxTree T, int l) {
  const int lane = threadIdx.x & 31;
  for (uint32_t m = blockIdx.x * 8u + (threadIdx.x >> 5); m < T.cnt[l]; m += gridDim.x * 8u) {
    const uint32_t c = m * 32u + lane;
    uint32_t lo[DP], hi[DP];
    BoxSum z{0u, 0xffffffffu, 0xffffffffu};
#pragma unroll
    for (int a = 0; a < DP; ++a) {
      lo[a] = 0xffffffffu;
      hi[a] = 0u;
    }
    if (c < T.cnt[l - 1]) {
      float v[box_words<DP>()];
      load_box<DP>(T.rec, T.off[l - 1] + c, v);
#pragma unroll
      for (int a = 0; a < DP; ++a) {
        lo[a] = float_ord(v[a]);
        hi[a] = float_ord(v[DP + a]);
      }
      z.rmax = __float_as_uint(v[2 * DP]);
      z.rmin = __float_as_uint(v[2 * DP + 1]);
      z.id = __float_as_uint(v[2 * DP + 2]);
    }
    box_reduce_store<DP>(lo, hi, z, lane, T.rec + (size_t)(T.off[l] + m) * box_words<DP>());
  }
}

// The query's box with its bounds rounded inwards to float32; axes from d on
// are unbounded (the padding is zero).
template <int DP>
struct PrQuery {
  float lo[DP], hi[DP];
  uint32_t rq;  // threshold, ordered
};

enum { kCount = 0, kFill = 1, kTop = 2 };
constexpr int kTopIds = 512;  // ids per query the warp's buffer serves

// Sorts the warp's buffer of `size` (a power of two >= 64) ids ascending.
__device__ __forceinline__ void sort_ids(uint32_t* buf, uint32_t size, int lane) {
  for (uint32_t len = 2; len <= size; len <<= 1) {
    for (uint32_t stride = len >> 1; stride > 0; stride >>= 1) {
      for (uint32_t q = lane; q < size / 2; q += 32) {
        const uint32_t i = 2u * q - (q & (stride - 1u)), j = i + stride;
        const uint32_t a = buf[i], b = buf[j];
        if ((a > b) == ((i & len) == 0)) {
          buf[i] = b;
          buf[j] = a;
        }
      }
      __syncwarp();
    }
  }
}

// MODE kCount: count[q] and cnt[q] (the count restricted to this class);
// kFill: keys at off[q] + (the warp's running position); kTop: count[q] and the
// max_out smallest ids (bufn: the id buffer's entries per warp, a power of two
// >= 2 max_out and >= 64), and the number of matches of the class in *total.
template <int DP, int MODE>
__global__ void __launch_bounds__(kPrThreads)
k_prange(const float* __restrict__ spts, const unsigned long long* __restrict__ skey, ClassView cv, BoxTree T,
         uint32_t nq, int32_t n_inst, const int32_t* __restrict__ q_inst, const double* __restrict__ q_box,
         const int32_t* __restrict__ q_rho, const int32_t* __restrict__ rowmap, int32_t one_row,
         uint32_t* __restrict__ cnt, long long* __restrict__ count, const unsigned long long* __restrict__ off,
         unsigned long long* __restrict__ out_keys, int32_t* __restrict__ ids, int max_out, int bufn,
         unsigned long long* total, int* __restrict__ status) {
  constexpr int W = box_words<DP>();
  extern __shared__ uint32_t s_ids[];  // kTop: [kPrWarps][bufn]
  __shared__ uint32_t s_base[kPrWarps][kBoxLevels + 1], s_mask[kPrWarps][kBoxLevels + 1];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t* const buf = s_ids + (MODE == kTop ? wib * bufn : 0);
  bool bad = false;
  const uint32_t q = blockIdx.x * kPrWarps + wib;  // one query per warp
  unsigned long long found = 0;
  if (q < nq) {
    const int32_t row = q_inst[q];
    int32_t loc = -1;
    if (row >= 0 && row < n_inst) loc = rowmap ? rowmap[row] : (row == one_row ? 0 : -1);
    if (loc < 0 || (uint32_t)loc >= cv.ninst) {
      if (MODE == kCount && lane == 0) cnt[q] = 0u;  // another class's query (or a bad row, flagged once)
    } else {
      const InstDev I = cv.instance((uint32_t)loc);
      PrQuery<DP> Q;
      Q.rq = rho_ord(q_rho[q]);
#pragma unroll
      for (int a = 0; a < DP; ++a) {
        const bool in = a < I.d;
        Q.lo[a] = in ? __double2float_ru(q_box[(size_t)q * 2 * kMaxDim + a]) : -INFINITY;
        Q.hi[a] = in ? __double2float_rd(q_box[(size_t)q * 2 * kMaxDim + kMaxDim + a]) : INFINITY;
      }
      const uint64_t base = MODE == kFill ? off[q] : 0ull;
      const uint32_t cap = MODE == kFill ? cnt[q] : 0u;  // the count pass's number
      uint32_t have = 0;                   // kFill: keys written; kTop: ids in the buffer
      uint32_t limit = 0xffffffffu;        // kTop: only smaller ids (output indices) can still enter
      // sort the buffer, keep the smallest max_out ids
      auto compact = [&]() {
        for (uint32_t e = have + lane; e < (uint32_t)bufn; e += 32) buf[e] = 0xffffffffu;
        __syncwarp();
        sort_ids(buf, (uint32_t)bufn, lane);
        if (have >= (uint32_t)max_out) {
          have = (uint32_t)max_out;
          limit = buf[max_out - 1];
        }
        __syncwarp();
      };
      auto scan_point = [&](bool ok, const Pt<DP>& x, unsigned long long k) {
        bool in = ok && rho_ord(key_rho(k)) > Q.rq;
#pragma unroll
        for (int a = 0; a < DP; ++a) in &= x.x[a] >= Q.lo[a] && x.x[a] <= Q.hi[a];
        unsigned m = __ballot_sync(kFull, in);
        found += __popc(m);
        if constexpr (MODE == kFill) {
          const uint32_t slot = have + __popc(m & lt);
          if (in) {
            if (slot < cap)
              out_keys[base + slot] = ((unsigned long long)q << 31) | (unsigned long long)(key_id(k) - (uint32_t)I.out);
            else
              bad = true;
          }
          have += __popc(m);
        }
        if constexpr (MODE == kTop) {
          const uint32_t id = key_id(k);
          in &= id < limit;
          m = __ballot_sync(kFull, in);
          if (m) {
            if (have + 32u > (uint32_t)bufn) {
              compact();
              in &= id < limit;
              m = __ballot_sync(kFull, in);
            }
            if (in) buf[have + __popc(m & lt)] = id;
            have += __popc(m);
            __syncwarp();
          }
        }
      };
      // children b .. b + 31 of level l that are in the instance's range and
      // can hold a match; wholly inside nodes are counted here where no id of
      // theirs is wanted
      const uint32_t ch0 = I.chunk0, ch1 = I.chunk0 + (I.n + 31u) / 32u;
      auto test = [&](int l, uint32_t b) {
        const uint32_t node = b + (uint32_t)lane;
        const uint64_t c0 = (uint64_t)node << (5 * (l - 1)), c1 = ((uint64_t)node + 1ull) << (5 * (l - 1));
        bool go = node < T.cnt[l] && c1 > ch0 && c0 < ch1;
        uint32_t whole = 0;
        if (go) {
          float v[W];
          load_box<DP>(T.rec, T.off[l] + node, v);
          go = __float_as_uint(v[2 * DP]) > Q.rq;
          bool inside = __float_as_uint(v[2 * DP + 1]) > Q.rq && c0 >= ch0 &&
                        (c1 < T.cnt[1] ? c1 : T.cnt[1]) <= ch1;
#pragma unroll
          for (int a = 0; a < DP; ++a) {
            go &= v[DP + a] >= Q.lo[a] && v[a] <= Q.hi[a];
            inside &= v[a] >= Q.lo[a] && v[DP + a] <= Q.hi[a];
          }
          if (MODE != kFill && go && inside && (MODE == kCount || __float_as_uint(v[2 * DP + 2]) >= limit)) {
            go = false;
            const uint64_t e1 = (c1 < ch1 ? c1 : ch1) - ch0;
            whole = (uint32_t)((e1 * 32u < I.n ? e1 * 32u : I.n) - (c0 - ch0) * 32u);
          }
        }
        if (MODE != kFill) found += __reduce_add_sync(kFull, whole);
        return __ballot_sync(kFull, go);
      };
      if (I.n > 0) {
        int l = 1;  // the lowest level where the instance spans at most 32 nodes
        while (l < T.levels && ((ch1 - 1u) >> (5 * (l - 1))) - (ch0 >> (5 * (l - 1))) >= 32u) ++l;
        uint32_t b = ch0 >> (5 * (l - 1));
        unsigned m = test(l, b);
        const int top = l;
        for (;;) {
          if (m == 0u) {  // up
            if (l >= top) break;
            ++l;
            m = s_mask[wib][l];
            b = s_base[wib][l];
            __syncwarp();  // read by every lane before it is written again
            continue;
          }
          const uint32_t node = b + (uint32_t)(__ffs((int)m) - 1);
          m &= m - 1u;
          if (l > 1) {  // down
            if (lane == 0) {
              s_mask[wib][l] = m;
              s_base[wib][l] = b;
            }
            __syncwarp();
            --l;
            b = node * 32u;
            m = test(l, b);
            continue;
          }
          // chunks of this node, two at a time: both loads in flight
          const bool two = m != 0u;
          const uint32_t node2 = two ? b + (uint32_t)(__ffs((int)m) - 1) : node;
          if (two) m &= m - 1u;
          const uint32_t pa = I.start + (node - ch0) * 32u + lane, pb = I.start + (node2 - ch0) * 32u + lane;
          const bool oka = pa < I.start + I.n, okb = two && pb < I.start + I.n;
          Pt<DP> xa, xb;
          unsigned long long ka = 0ull, kb = 0ull;
#pragma unroll
          for (int a = 0; a < DP; ++a) xa.x[a] = xb.x[a] = 0.f;
          if (oka) {
            xa = load_pt<DP>(spts, pa);
            ka = __ldg(skey + pa);
          }
          if (okb) {
            xb = load_pt<DP>(spts, pb);
            kb = __ldg(skey + pb);
          }
          scan_point(oka, xa, ka);
          if (two) scan_point(okb, xb, kb);
        }
      }
      if constexpr (MODE == kTop) {
        if (have) compact();
        const uint32_t got = min(have, (uint32_t)max_out);
        for (uint32_t e = lane; e < (uint32_t)max_out; e += 32)
          ids[(size_t)q * max_out + e] = e < got ? (int32_t)(buf[e] - (uint32_t)I.out) : -1;
      }
      if (MODE != kFill && lane == 0) {
        if (MODE == kCount) cnt[q] = (uint32_t)found;
        count[q] = (long long)found;
      }
    }
  }
  if constexpr (MODE == kTop) {
    if (lane == 0 && found) atomicAdd(total, found);
  }
  if (bad) set_status(status, kStatusIndex);
}

// Query checks and output defaults: count 0, rows of -1; a row index outside
// the batch is a data error.
__global__ void k_prange_init(uint32_t nq, int32_t n_inst, const int32_t* __restrict__ q_inst,
                              long long* __restrict__ count, int32_t* __restrict__ ids, int max_out,
                              int* __restrict__ status) {
  const uint64_t total = (uint64_t)nq * (uint64_t)(max_out > 0 ? max_out : 0);
  for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < total;
       e += (uint64_t)gridDim.x * blockDim.x)
    ids[e] = -1;
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += gridDim.x * blockDim.x) {
    count[q] = 0;
    const int32_t r = q_inst[q];
    if (r < 0 || r >= n_inst) set_status(status, kStatusQuery);
  }
}

// Exclusive scan of cnt[0..nq) into off[0..nq], one CTA (off[nq] = total).
__global__ void __launch_bounds__(1024) k_prange_scan(const uint32_t* __restrict__ cnt, uint32_t nq,
                                                      unsigned long long* __restrict__ off) {
  __shared__ unsigned long long part[1024];
  __shared__ unsigned long long carry;
  if (threadIdx.x == 0) carry = 0ull;
  __syncthreads();
  for (uint32_t c0 = 0; c0 < nq; c0 += 1024u) {
    const uint32_t i = c0 + threadIdx.x;
    const unsigned long long v = i < nq ? cnt[i] : 0ull;
    part[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
      const unsigned long long t = threadIdx.x >= (unsigned)o ? part[threadIdx.x - o] : 0ull;
      __syncthreads();
      part[threadIdx.x] += t;
      __syncthreads();
    }
    if (i < nq) off[i] = carry + part[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == 1023) carry += part[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) off[nq] = carry;
}

// Sorted keys -> the first max_out ids of every query's row.
__global__ void k_prange_scatter(const unsigned long long* __restrict__ keys, uint64_t total,
                                 const unsigned long long* __restrict__ off, uint32_t nq,
                                 int max_out, int32_t* __restrict__ ids, int* __restrict__ status) {
  for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < total;
       e += (uint64_t)gridDim.x * blockDim.x) {
    const unsigned long long k = keys[e];
    const uint32_t q = (uint32_t)(k >> 31);
    if (q >= nq || e < off[q] || e >= off[q + 1]) {
      set_status(status, kStatusIndex);
      continue;
    }
    const uint64_t j = e - off[q];
    if (j < (uint64_t)max_out) ids[(size_t)q * max_out + j] = (int32_t)(k & 0x7fffffffull);
  }
}

inline unsigned grid_cap(uint64_t items, int per, unsigned cap) {
  uint64_t b = (items + per - 1) / per;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (unsigned)b;
}

// Levels of the hierarchy of nchunk chunks: up to a level of at most 32 nodes.
BoxTree box_tree(float* rec, uint32_t nchunk) {
  BoxTree T;
  T.rec = rec;
  T.levels = 1;
  T.off[0] = T.cnt[0] = 0u;
  T.off[1] = 0u;
  T.cnt[1] = nchunk;
  while (T.cnt[T.levels] > 32u && T.levels < kBoxLevels) {
    const int l = T.levels++;
    T.off[l + 1] = T.off[l] + T.cnt[l];
    T.cnt[l + 1] = (T.cnt[l] + 31u) / 32u;
  }
  return T;
}

template <int DP>
void boxes_dp(const float* spts, const unsigned long long* skey, const ClassView& cv, float* rec,
              cudaStream_t st) {
  const BoxTree T = box_tree(rec, cv.nchunk);
  k_box_chunks<DP><<<grid_cap(cv.nchunk, 8, sm_count() * 16u), 256, 0, st>>>(spts, skey, cv, T);
  for (int l = 2; l <= T.levels; ++l)
    k_box_level<DP><<<grid_cap(T.cnt[l], 8, sm_count() * 16u), 256, 0, st>>>(T, l);
  count_launches(T.levels);
}

template <int DP>
void prange_dp(int mode, const float* spts, const unsigned long long* skey, const ClassView& cv, float* rec,
               const PrangeArgs& a, uint32_t* cnt, const unsigned long long* off, unsigned long long* keys,
               int32_t* ids, int max_out, unsigned long long* total, int* status, cudaStream_t st) {
  const BoxTree T = box_tree(rec, cv.nchunk);
  const unsigned grid = (a.nq + kPrWarps - 1) / kPrWarps;
  int bufn = 64;
  while (bufn < 2 * max_out) bufn <<= 1;
  auto go = [&](auto kern, size_t sh) {
    kern<<<grid, kPrThreads, sh, st>>>(spts, skey, cv, T, a.nq, a.n_inst, a.q_inst, a.q_box, a.q_rho, a.rowmap,
                                       a.one_row, cnt, a.count, off, keys, ids, max_out, bufn, total, status);
  };
  if (mode == kTop) go(k_prange<DP, kTop>, sizeof(uint32_t) * (size_t)kPrWarps * bufn);
  else if (mode == kFill) go(k_prange<DP, kFill>, 0);
  else go(k_prange<DP, kCount>, 0);
}

}  // namespace

void launch_prange_init(const PrangeArgs& a, int32_t* ids, int max_out, int* status,
                        cudaStream_t st) {
  const uint64_t items = (uint64_t)a.nq * (uint64_t)(max_out > 0 ? max_out : 1);
  k_prange_init<<<grid_cap(items, 256, sm_count() * 16u), 256, 0, st>>>(a.nq, a.n_inst, a.q_inst, a.count,
                                                                 ids, max_out, status);
  count_launches(1);
}

int prange_top_ids() { return kTopIds; }

void launch_prange_boxes(int dp, const float* spts, const unsigned long long* skey, const ClassView& cv,
                         float* rec, cudaStream_t st) {
  if (dp == 2) boxes_dp<2>(spts, skey, cv, rec, st);
  else if (dp == 4) boxes_dp<4>(spts, skey, cv, rec, st);
  else boxes_dp<8>(spts, skey, cv, rec, st);
}

void launch_prange(int dp, int mode, const float* spts, const unsigned long long* skey, const ClassView& cv,
                   float* rec, const PrangeArgs& a, uint32_t* cnt, const unsigned long long* off,
                   unsigned long long* keys, int32_t* ids, int max_out, unsigned long long* total, int* status,
                   cudaStream_t st) {
  if (a.nq == 0) return;
  if (dp == 2) prange_dp<2>(mode, spts, skey, cv, rec, a, cnt, off, keys, ids, max_out, total, status, st);
  else if (dp == 4) prange_dp<4>(mode, spts, skey, cv, rec, a, cnt, off, keys, ids, max_out, total, status, st);
  else prange_dp<8>(mode, spts, skey, cv, rec, a, cnt, off, keys, ids, max_out, total, status, st);
  count_launches(1);
}

void launch_prange_scan(const uint32_t* cnt, uint32_t nq, unsigned long long* off,
                        cudaStream_t st) {
  k_prange_scan<<<1, 1024, 0, st>>>(cnt, nq, off);
  count_launches(1);
}

void launch_prange_scatter(const unsigned long long* keys, uint64_t total,
                           const unsigned long long* off, uint32_t nq, int max_out, int32_t* ids,
                           int* status, cudaStream_t st) {
  if (total == 0 || max_out <= 0) return;
  k_prange_scatter<<<grid_cap(total, 256, sm_count() * 16u), 256, 0, st>>>(keys, total, off, nq, max_out,
                                                                     ids, status);
  count_launches(1);
}

}  // namespace dpc

// dependent.cu -- lambda_i (the nearest point of higher order) and
// delta_i = D(x_i, lambda_i) (Definitions 2-3).
//
// The paper runs one priority nearest-neighbour query per point in parallel
// (Algorithm 1) on a priority search kd-tree.  Here each query runs in two
// phases:
//   near  the grid block around the point's cell (the cells the density
//         used), streamed by the warp with one query per lane (block.cuh).
//         If the best candidate is closer than anything outside the block
//         can be, and no other candidate is within the float32 error band
//         of it, the query is settled; this holds for most points, since a
//         point's dependent point is usually within d_cut.
//   far   the remaining queries (local density maxima, isolated points, near
//         ties) walk the radix tree (tree.cu) depth first, nearer child
//         first, skipping subtrees whose largest key is not above the query's
//         key or whose box is farther than the best candidate so far (the
//         pruning of Section 4.1.2).
//
// Exactness.  Candidates are compared on their float32 distance s32; the
// winner of the binary64 order (s64, id) -- the write-min of Section 3.2 --
// is certainly the float32 winner unless another candidate lies within the
// float32 error band of it.  The query tracks the smallest and second
// smallest s32; when the second is inside the band the candidates inside it
// are re-ranked in binary64 (rare: exact ties and near ties).  delta is
// always sqrt of the winner's binary64 distance.  In FP64 mode every
// candidate is compared in binary64 directly.
#include <cmath>
#include <type_traits>

#include "block.cuh"
#include "internal.h"

namespace dpc {

namespace {

constexpr int kFarThreads = 128;
constexpr int kStack = 128;
constexpr int kWarpStack = 1024;  // shared stack entries per warp (far phase, round 2)
constexpr uint32_t kFarBudget = 128;  // node expansions per query in round 1, at least
constexpr unsigned kFarGrid = 128;    // CTAs per SM of round 1, at most
constexpr int kNearWarps = 4;
constexpr int kNearThreads = kNearWarps * 32;

__device__ __forceinline__ float band_of(float s, float mul, float add) {
  return __fadd_ru(__fmul_ru(s, mul), add);
}

// A region whose float lower bound lbs (already 1e-5 below the true squared
// distance) exceeds `bound` by this much holds no candidate with s32 <= bound:
// the margin dominates the absolute float32 error term of tiny distances.
constexpr float kPruneAbs = 1e-33f;
__device__ __forceinline__ bool beyond(float lbs, float bound) {
  return lbs > __fadd_ru(bound, kPruneAbs);
}

// 1e-5 of a bound covers its relative error, but below 2^-126 a float32 bound is
// off by up to 2^-150 per axis whatever its size; in binary64 mode, where
// distances that small are told apart, bounds are lowered by this as well (the
// float32 comparisons have kPruneAbs; with it in both modes a run of 1e6 points
// in 2-D took 0.25% longer).
constexpr float kPruneTiny = 0x1p-140f;

// Running minimum of (s, id), the second smallest s, and the sorted position
// of the minimum (tree phase).
template <typename S>
struct Best {
  S s1, s2;
  uint32_t o1;   // id of the best
  uint32_t t1;   // sorted position of the best
  __device__ __forceinline__ void init() {
    s1 = (S)INFINITY;
    s2 = (S)INFINITY;
    o1 = 0xffffffffu;
    t1 = 0xffffffffu;
  }
  __device__ __forceinline__ void add(S s, uint32_t o, uint32_t t) {
    if (s < s1 || (s == s1 && o < o1)) {
      s2 = s1;
      s1 = s;
      o1 = o;
      t1 = t;
    } else if (s < s2) {
      s2 = s;
    }
  }
  // union over the warp's lanes (every lane ends with the same summary)
  __device__ __forceinline__ void merge_warp() {
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      const S b1 = __shfl_xor_sync(kFull, s1, m);
      const uint32_t bo = __shfl_xor_sync(kFull, o1, m);
      const S b2 = __shfl_xor_sync(kFull, s2, m);
      const uint32_t bt = __shfl_xor_sync(kFull, t1, m);
      if (b1 < s1 || (b1 == s1 && bo < o1)) {
        s2 = s1 < b2 ? s1 : b2;
        s1 = b1;
        o1 = bo;
        t1 = bt;
      } else {
        s2 = s2 < b1 ? s2 : b1;
      }
    }
  }
};

// Exact binary64 argmin over (s64, id).
struct Exact {
  double s;
  uint32_t o;
  __device__ __forceinline__ void init() {
    s = INFINITY;
    o = 0xffffffffu;
  }
  __device__ __forceinline__ void add(double v, uint32_t id) {
    if (v < s || (v == s && id < o)) {
      s = v;
      o = id;
    }
  }
  __device__ __forceinline__ void merge_warp() {
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) add(__shfl_xor_sync(kFull, s, m), __shfl_xor_sync(kFull, o, m));
  }
};

// Conservative squared lower bound, in fine units, between the query and a box
// of fine indices [lo, hi] on each axis (a point of fine index c lies in
// [c - 0.5, c + 1.5) fine units; the query's float position is within 1/8).
__device__ __forceinline__ float lb_axis(float lo, float hi, float u) {
  return fmaxf(fmaxf(lo - 1.f - u, u - hi - 2.f), 0.f);
}

// ---------------------------------------------------------------------------
// near phase

// Smallest and second smallest float32 distance of a candidate set, and the id
// of a candidate at the smallest.  Two candidates at the same smallest
// distance leave s2 == s1, which the caller treats as ambiguous and resolves
// in binary64 later, so ties need no id order here.
struct Min2 {
  float s1, s2;
  uint32_t o1;
  __device__ __forceinline__ void init() {
    s1 = s2 = INFINITY;
    o1 = 0xffffffffu;
  }
  __device__ __forceinline__ void add(float v, uint32_t id) {
    s2 = fminf(s2, fmaxf(s1, v));
    o1 = v < s1 ? id : o1;
    s1 = fminf(s1, v);
  }
};

// Coordinates of point `id` of the instance whose coordinates start at
// element `coord` of the caller's input (the same float values the sorted copy
// holds: int32 inputs are exact in float32 by the range check).
template <int DP>
__device__ __forceinline__ Pt<DP> input_pt(const void* __restrict__ pts, int dtype, uint64_t coord,
                                           int d, uint32_t id) {
  Pt<DP> p;
#pragma unroll
  for (int a = 0; a < DP; ++a) {
    float v = 0.f;
    if (a < d) {
      const size_t e = coord + (size_t)id * d + a;
      v = dtype == 0 ? (float)__ldg((const int32_t*)pts + e) : __ldg((const float*)pts + e);
    }
    p.x[a] = v;
  }
  return p;
}

template <int DP, int G, bool F64>
__global__ void __launch_bounds__(kNearThreads)
k_dep_near(const float* __restrict__ spts, const unsigned long long* __restrict__ scode,
           const unsigned long long* __restrict__ skey, ClassView cv, int32_t rho_skip,
           const void* __restrict__ pts, int dtype, const CutGeom* __restrict__ cuts,
           const HashInfo* __restrict__ hi, const unsigned long long* __restrict__ hkeys,
           const uint2* __restrict__ hvals, int32_t* __restrict__ lambda,
           double* __restrict__ delta, FarQueue q, Counters* ctr, uint32_t min_fill) {
  if (min_fill && !tensor_fill(cv.N, hi, min_fill)) return;  // the tree layout's part
  constexpr int kNearCap = DP == 8 ? 128 : 256;
  __shared__ __align__(16) float s_pts[kNearWarps * kNearCap * DP];
  __shared__ unsigned long long s_key[kNearWarps * kNearCap];
  __shared__ RunTable s_rt[kNearWarps];
  __shared__ RunTable s_rt2[kNearWarps];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  float* wpts = s_pts + wib * kNearCap * DP;
  unsigned long long* wkey = s_key + wib * kNearCap;
  RunTable& rt = s_rt[wib];
  RunTable& rt2 = s_rt2[wib];
  const int S = cv.cls->S, ib = cv.cls->ib;
  const uint32_t hmask = hi->hmask;
  const uint32_t n = cv.N;
  const uint32_t lanemask_lt = (1u << lane) - 1u;

  for (uint32_t ch = blockIdx.x * kNearWarps + wib; ch < cv.nchunk; ch += gridDim.x * kNearWarps) {
    uint32_t inst, p0, end;
    cv.chunk(ch, inst, p0, end);
    const InstDev I = cv.instance(inst);
    const GridGeom* geom = cv.geom + inst;
    const CutGeom& C = cuts[inst];
    const float f2lo = geom->f2 * (1.f - 1e-5f);
    const double inv_f = geom->inv_f;
    double org[G];
#pragma unroll
    for (int a = 0; a < G; ++a) org[a] = geom->org[a];
    const int k = C.k;
    const float cell_fine = (float)(1u << k);
    const int R = C.R;
    const int shift = G * k;
    const int cmax = (1 << (geom->B - k)) - 1;
    const float bmul = C.band_mul, badd = C.band_add;
    const float far32 = C.far32;
    const double far64 = C.far64;
    const unsigned long long hb = ib ? ((unsigned long long)inst << S) : 0ull;
    const uint32_t p = p0 + lane;
    const bool valid = p < end;
    Pt<DP> me;
#pragma unroll
    for (int a = 0; a < DP; ++a) me.x[a] = 0.f;
    unsigned long long K = ~0ull;
    if (valid) {
      me = load_pt<DP>(spts, p);
      K = skey[p];
    }
    const unsigned long long mycell = valid ? (key_code(scode[p], S, ib) >> shift) : ~0ull;
    uint32_t c0[G];
    unmorton<G>(valid ? mycell : 0ull, c0);
    const bool skip = valid && (int32_t)(K >> 32) < max(rho_skip, C.skip);
    const int nvalid = (int)min(32u, end - p0);
    Min2 acc;
    acc.init();
    Exact acc64;
    acc64.init();
    // the query's position in fine units, for cell lower bounds
    float uq[G];
#pragma unroll
    for (int a = 0; a < G; ++a) uq[a] = valid ? (float)(((double)me.x[a] - org[a]) * inv_f) : 0.f;
    for_groups<G>(mycell, c0, valid, valid && !skip, nvalid, R, cmax, lane,
                  [&](bool act, const Union<G>& u) {
      const int nr = union_runs<G>(u, hkeys, hvals, hmask, hb, n, lane, rt);
      // scan every run of a table, staged window by window
      auto scan = [&](const RunTable& tab, int nt) {
        const uint32_t total = tab.pre[nt];
        for (uint32_t w0 = 0; w0 < total; w0 += kNearCap) {
          const uint32_t w1 = min(total, w0 + (uint32_t)kNearCap);
          __syncwarp();
          stage_runs<DP, true>(tab, nt, w0, w1, spts, skey, wpts, wkey, lane);
          __syncwarp();
          for_window_runs<G>(tab, nt, u, w0, w1, [&](uint32_t i0, uint32_t i1, const uint32_t* cc) {
            const bool need = act && in_block<G>(c0, cc, R);
            if (!__any_sync(kFull, need)) return;
            // a lane outside this cell's block takes no candidate: no key exceeds ~0
            const unsigned long long Kl = need ? K : ~0ull;
#pragma unroll 4
            for (uint32_t i = i0; i < i1; ++i) {
              const unsigned long long kt = wkey[i];
              const Pt<DP> x = window_pt<DP>(wpts, i);
              if constexpr (F64) {
                if (kt > Kl) acc64.add(dist64<DP>(me, x), key_id(kt));
              } else {
                const float d32 = dist32<DP>(me, x);
                acc.add(kt > Kl ? d32 : INFINITY, key_id(kt));
              }
            }
          });
        }
        __syncwarp();
      };
      auto own = [&](const uint32_t* cc) {
        bool same = act;
#pragma unroll
        for (int a = 0; a < G; ++a) same &= cc[a] == c0[a];
        return __any_sync(kFull, same) != 0;
      };
      // a small union: one pass over everything
      if (rt.pre[nr] <= 4u * kNearCap) {
        scan(rt, nr);
        return;
      }
      // pass 1: the cells holding the group's own queries -- unless they hold
      // too few points to bound the search, then one pass over everything
      const int n1 = filter_runs<G>(rt, nr, u, rt2, lane, own);
      if (rt2.pre[n1] < 96u) {
        scan(rt, nr);
        return;
      }
      scan(rt2, n1);
      // pass 2: the other cells of the blocks that can still hold a point
      // closer than some lane's best (a conservative lower bound decides)
      scan(rt2, filter_runs<G>(rt, nr, u, rt2, lane, [&](const uint32_t* cc) {
        if (own(cc)) return false;
        bool need = act && in_block<G>(c0, cc, R);
        if (need) {
          float lb2 = 0.f;
#pragma unroll
          for (int a = 0; a < G; ++a) {
            const float lo = (float)cc[a] * cell_fine;
            const float l = lb_axis(lo, lo + cell_fine - 1.f, uq[a]);
            lb2 = fmaf(l, l, lb2);
          }
          const float lbs = lb2 * f2lo;
          if constexpr (F64) need = (double)(lbs - kPruneTiny) <= acc64.s;
          else need = !beyond(lbs, band_of(acc.s1, bmul, badd));
        }
        return __any_sync(kFull, need) != 0;
      }));
    });

    bool settled = false;
    float s1 = INFINITY;
    if (valid && !skip) {
      const uint32_t id = key_id(K);
      if constexpr (F64) {
        settled = acc64.o != 0xffffffffu && acc64.s < far64;
        if (settled) {
          lambda[id] = (int32_t)(acc64.o - (uint32_t)I.out);
          delta[id] = sqrt(acc64.s);
        }
      } else if (acc.o1 != 0xffffffffu) {
        s1 = acc.s1;
        const float bnd = band_of(s1, bmul, badd);
        settled = bnd < far32 && acc.s2 > bnd;
        if (settled) {
          const uint32_t o = acc.o1 - (uint32_t)I.out;
          lambda[id] = (int32_t)o;
          delta[id] = sqrt(dist64<DP>(me, input_pt<DP>(pts, dtype, I.coord, I.d, o)));
        }
      }
    } else if (valid) {
      const uint32_t id = key_id(K);
      lambda[id] = -1;
      delta[id] = __longlong_as_double(0x7ff8000000000000ll);  // NaN: skipped
    }
    // unsettled queries (nothing near, or a near tie) go to the far phase
    const bool push = valid && !skip && !settled;
    const unsigned pm = __ballot_sync(kFull, push);
    uint32_t base = 0;
    if (lane == 0 && pm) base = atomicAdd(&ctr->queue_n, (unsigned)__popc(pm));
    base = __shfl_sync(kFull, base, 0);
    if (push) {
      const uint32_t slot = base + __popc(pm & lanemask_lt);
      q.pos[slot] = p;
      if constexpr (F64) q.s1d[slot] = acc64.s;
      else q.s1[slot] = s1;
    }
  }
}

// Segment form of the near phase (the work layout of k_density_seg): the
// chunk's points are split into segments of consecutive cells; the warp looks
// the cells around a segment up once, stages their points and order keys in
// shared memory, and lane l keeps the smallest and second smallest float32
// distance among the higher candidates of query l % nqp in part l / nqp of the
// tile, four candidates at a time as broadcast reads.  The parts are merged with
// shuffles at the end; lane j then settles the chunk's query j or queues it
// for the far phase exactly as k_dep_near does.
// What bounds it: issue slots and the ALU pipe in them (61% and 62% busy, DRAM 5%):
// 25 instructions per lane and scanned pair, set-up and idle lanes included
// (profiles/, 4e6 points in 3-D, 1.74 ms).  1e7 points in 3-D: 6.09 ms with the
// candidates in registers across the lanes and a warp reduction per query and
// window, 5.6 with those reductions only where a window could still matter, 4.4
// with queries across the lanes.
template <int DP, int G>
constexpr int near_cap() { return DP == 2 ? 512 : (DP == 4 && G < 4 ? 384 : (DP == 4 ? 256 : 128)); }

template <int DP, int G, bool F64>
__global__ void __launch_bounds__(kNearThreads, DP == 8 ? 4 : 5)
k_dep_near_seg(const float* __restrict__ spts, const unsigned long long* __restrict__ scode,
               const unsigned long long* __restrict__ skey, ClassView cv, int32_t rho_skip,
               const void* __restrict__ pts, int dtype, const CutGeom* __restrict__ cuts,
               const HashInfo* __restrict__ hi, const unsigned long long* __restrict__ hkeys,
               const uint2* __restrict__ hvals, int32_t* __restrict__ lambda,
               double* __restrict__ delta, FarQueue q, Counters* ctr, int seg_cells) {
  constexpr int ND = real_dims<DP, G>();  // coordinates that can be nonzero
  constexpr int kCap = near_cap<DP, G>();
  __shared__ RunTable s_rt[kNearWarps];
  __shared__ RunTable s_rt2[kNearWarps];
  __shared__ CandTile<ND, kCap, true> s_tile[kNearWarps];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  RunTable& rt = s_rt[wib];
  RunTable& rt2 = s_rt2[wib];
  CandTile<ND, kCap, true>& tile = s_tile[wib];
  const int S = cv.cls->S, ib = cv.cls->ib;
  const uint32_t hmask = hi->hmask;
  const uint32_t n = cv.N;
  const uint32_t lanemask_lt = (1u << lane) - 1u;

  for (uint32_t ch = blockIdx.x * kNearWarps + wib; ch < cv.nchunk; ch += gridDim.x * kNearWarps) {
    uint32_t inst, p0, end;
    cv.chunk(ch, inst, p0, end);
    const CutGeom& C = cuts[inst];
    const int k = C.k;
    const int R = C.R;
    const int shift = G * k;
    const int cmax = (1 << (cv.geom[inst].B - k)) - 1;
    const unsigned long long hb = ib ? ((unsigned long long)inst << S) : 0ull;
    const uint32_t p = p0 + lane;
    const bool valid = p < end;
    unsigned long long K = ~0ull;
    if (valid) K = skey[p];
    const unsigned long long mycell = valid ? (key_code(scode[p], S, ib) >> shift) : ~0ull;
    const bool skip = valid && (int32_t)(K >> 32) < max(rho_skip, C.skip);
    const int nvalid = (int)min(32u, end - p0);
    Min2 best;  // lane j: query p0 + j
    best.init();
    Exact best64;
    best64.init();
    int s = 0;
    while (s < nvalid) {
      const unsigned long long cell = __shfl_sync(kFull, mycell, s);
      Union<G> u;
      const int e = super_segment<G>(mycell, valid, s, nvalid, R, cmax, seg_cells, lane, u);
      const unsigned seg = (e >= 32 ? 0xffffffffu : ((1u << e) - 1u)) & ~((1u << s) - 1u);  // lanes s .. e-1
      if (__ballot_sync(kFull, valid && !skip) & seg) {
        // one cell only: the own-cell-first passes below apply
        const bool single = (__ballot_sync(kFull, valid && mycell == cell) & seg) == seg;
        const int nq = e - s;
        const int lg = nq > 1 ? 32 - __clz(nq - 1) : 0;  // nqp = 1 << lg
        const int nqp = 1 << lg;
        const uint32_t part = (uint32_t)lane >> lg, step = 4u * (32u >> lg);
        const int mine = lane & (nqp - 1);
        const bool active = mine < nq;
        const uint32_t pq = p0 + (uint32_t)(s + (active ? mine : 0));
        const Pt<DP> me = load_pt<DP>(spts, pq);
        // a lane without a query (or with a skipped one) takes no candidate
        const int src = s + (active ? mine : 0);
        unsigned long long Kq = __shfl_sync(kFull, K, src);
        const int skipped = __shfl_sync(kFull, (int)skip, src);  // (every lane takes part)
        if (!active || skipped) Kq = ~0ull;
        f32x2 q2[ND];
#pragma unroll
        for (int a = 0; a < ND; ++a) q2[a] = pack2(me.x[a], me.x[a]);
        float s1 = INFINITY, s2 = INFINITY;
        uint32_t w1 = 0;  // low key word of the candidate at s1
        Exact ex;
        ex.init();
        // every candidate of a run table, tile by tile
        auto scan = [&](RunTable& tab, int ntab) {
          const uint32_t total = tab.pre[ntab];
          for (uint32_t t0 = 0; t0 < total; t0 += kCap) {
            const uint32_t t1 = min(total, t0 + (uint32_t)kCap);
            __syncwarp();
            stage_tile<DP, ND, kCap, true>(tab, ntab, t0, t1, spts, skey, tile, lane);
            const uint32_t tn = t1 - t0;
            for (uint32_t i = 4u * part; i < tn; i += step) {
              unsigned long long ck[4];
              const ulonglong2 k0 = *reinterpret_cast<const ulonglong2*>(&tile.key[i]);
              const ulonglong2 k1 = *reinterpret_cast<const ulonglong2*>(&tile.key[i + 2]);
              ck[0] = k0.x;
              ck[1] = k0.y;
              ck[2] = k1.x;
              ck[3] = k1.y;
              if constexpr (F64) {
#pragma unroll
                for (int v = 0; v < 4; ++v)
                  if (ck[v] > Kq) ex.add(dist64<DP, ND>(me, tile_pt<DP>(tile, i + v)), key_id(ck[v]));
              } else {
                f32x2 cc[2][ND];
                tile_quad(tile, i, cc);
                float dd[4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  const f32x2 sq = dist32x2<ND>(q2, cc[h]);
                  dd[2 * h] = lo2(sq);
                  dd[2 * h + 1] = hi2(sq);
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                  const float x = ck[v] > Kq ? dd[v] : INFINITY;
                  s2 = fminf(s2, fmaxf(s1, x));
                  w1 = x < s1 ? (uint32_t)ck[v] : w1;
                  s1 = fminf(s1, x);
                }
              }
            }
          }
          // the parts of each query (every lane of a query ends with the same)
          for (int o = nqp; o < 32; o <<= 1) {
            if constexpr (F64) {
              ex.add(__shfl_xor_sync(kFull, ex.s, o), __shfl_xor_sync(kFull, ex.o, o));
            } else {
              const float o1 = __shfl_xor_sync(kFull, s1, o), o2 = __shfl_xor_sync(kFull, s2, o);
              const uint32_t ow = __shfl_xor_sync(kFull, w1, o);
              s2 = fminf(fminf(s2, o2), fmaxf(s1, o1));
              w1 = o1 < s1 ? ow : w1;
              s1 = fminf(s1, o1);
            }
          }
        };
        const int nr = union_runs<G>(u, hkeys, hvals, hmask, hb, n, lane, rt);
        // Dense blocks of one cell: first the cell itself, then only the other
        // cells that can still hold a point closer than some query's best (a
        // conservative lower bound decides); any other block: one pass.
        if (!single || rt.pre[nr] <= 1024u) {
          scan(rt, nr);
        } else {
          uint32_t c0[G];
          unmorton<G>(cell, c0);
          auto own = [&](const uint32_t* cc) {
            bool same = true;
#pragma unroll
            for (int a = 0; a < G; ++a) same &= cc[a] == c0[a];
            return same;
          };
          scan(rt2, filter_runs<G>(rt, nr, u, rt2, lane, own));
          const GridGeom* geom = cv.geom + inst;
          const float f2lo = geom->f2 * (1.f - 1e-5f);
          const float cell_fine = (float)(1u << k);
          float uq[G];  // the query in fine units
#pragma unroll
          for (int a = 0; a < G; ++a) uq[a] = (float)(((double)me.x[a] - geom->org[a]) * geom->inv_f);
          const float bnd = band_of(s1, C.band_mul, C.band_add);
          const int n2 = filter_runs<G>(rt, nr, u, rt2, lane, [&](const uint32_t* cc) {
            if (own(cc)) return false;
            bool need = Kq != ~0ull;
            if (need) {
              float lb2 = 0.f;
#pragma unroll
              for (int a = 0; a < G; ++a) {
                const float lo = (float)cc[a] * cell_fine;
                const float l = lb_axis(lo, lo + cell_fine - 1.f, uq[a]);
                lb2 = fmaf(l, l, lb2);
              }
              const float lbs = lb2 * f2lo;
              if constexpr (F64) need = (double)(lbs - kPruneTiny) <= ex.s;
              else need = !beyond(lbs, bnd);
            }
            return __any_sync(kFull, need) != 0;
          });
          if constexpr (!F64) {  // the parts hold the merged best: keep it in one of them
            if (part) s1 = s2 = INFINITY;
          }
          scan(rt2, n2);
        }
        // lane j takes query j's result
        const int from = (lane - s) & 31;
        if constexpr (F64) {
          const double es = __shfl_sync(kFull, ex.s, from);
          const uint32_t eo = __shfl_sync(kFull, ex.o, from);
          if ((seg >> lane) & 1u) {
            best64.s = es;
            best64.o = eo;
          }
        } else {
          const float b1 = __shfl_sync(kFull, s1, from), b2 = __shfl_sync(kFull, s2, from);
          const uint32_t bw = __shfl_sync(kFull, w1, from);
          if ((seg >> lane) & 1u) {
            best.s1 = b1;
            best.s2 = b2;
            best.o1 = b1 < INFINITY ? 0xffffffffu - bw : 0xffffffffu;  // key_id of the low word
          }
        }
      }
      s = e;
    }

    const InstDev I = cv.instance(inst);
    const float bmul = C.band_mul, badd = C.band_add;
    const float far32 = C.far32;
    const double far64 = C.far64;
    bool settled = false;
    float s1 = INFINITY;
    if (valid && !skip) {
      const uint32_t id = key_id(K);
      if constexpr (F64) {
        settled = best64.o != 0xffffffffu && best64.s < far64;
        if (settled) {
          lambda[id] = (int32_t)(best64.o - (uint32_t)I.out);
          delta[id] = sqrt(best64.s);
        }
      } else if (best.o1 != 0xffffffffu) {
        s1 = best.s1;
        const float bnd = band_of(s1, bmul, badd);
        settled = bnd < far32 && best.s2 > bnd;
        if (settled) {
          const uint32_t o = best.o1 - (uint32_t)I.out;
          const Pt<DP> me = load_pt<DP>(spts, p);
          lambda[id] = (int32_t)o;
          delta[id] = sqrt(dist64<DP>(me, input_pt<DP>(pts, dtype, I.coord, I.d, o)));
        }
      }
    } else if (valid) {
      const uint32_t id = key_id(K);
      lambda[id] = -1;
      delta[id] = __longlong_as_double(0x7ff8000000000000ll);  // NaN: skipped
    }
    // unsettled queries (nothing near, or a near tie) go to the far phase
    const bool push = valid && !skip && !settled;
    const unsigned pm = __ballot_sync(kFull, push);
    uint32_t base = 0;
    if (lane == 0 && pm) base = atomicAdd(&ctr->queue_n, (unsigned)__popc(pm));
    base = __shfl_sync(kFull, base, 0);
    if (push) {
      const uint32_t slot = base + __popc(pm & lanemask_lt);
      q.pos[slot] = p;
      if constexpr (F64) q.s1d[slot] = best64.s;
      else q.s1[slot] = s1;
    }
  }
}

// Tree layout of the near phase: no block scan; every query (but the skipped
// ones) goes to the tree search, bounded by its nearest higher point among the
// 96 sorted points around its chunk (Morton neighbours are mostly spatial
// neighbours, so the bound is near the answer and the search mostly verifies
// it).  One warp per 32-point chunk: the points of the chunk and of its two
// neighbours staged once, every lane over all of them.
// 1e6 points in 2-D: near phase and far search 0.53 + 0.21 ms with the blocks
// scanned, 0.03 + 0.54 with the tree searched unbounded, 0.04 + 0.46 with this
// bound, 0.04 + 0.29 with the walk of far_walk.
template <int DP, int ND, int RD>
__global__ void __launch_bounds__(kNearThreads)
k_near_to_far(const float* __restrict__ spts, const unsigned long long* __restrict__ skey, ClassView cv,
              const CutGeom* __restrict__ cuts, int32_t rho_skip, int32_t* __restrict__ lambda,
              double* __restrict__ delta, FarQueue q, Counters* ctr, const HashInfo* __restrict__ hi,
              const float* __restrict__ nbox, const uint32_t* __restrict__ roots, uint32_t skip_fill) {
  if (skip_fill && tensor_fill(cv.N, hi, skip_fill)) return;  // the tensor tiles' part
  constexpr int kAround = 128;  // 96 used
  __shared__ CandTile<ND, kAround, true> s_tile[kNearWarps];
  const int lane = threadIdx.x & 31;
  CandTile<ND, kAround, true>& tile = s_tile[threadIdx.x >> 5];
  const uint32_t lanemask_lt = (1u << lane) - 1u;
  for (uint32_t c = blockIdx.x * kNearWarps + (threadIdx.x >> 5); c < cv.nchunk; c += gridDim.x * kNearWarps) {
    uint32_t inst, p0, end;
    cv.chunk(c, inst, p0, end);
    const uint32_t start = cv.instance(inst).start;
    const uint32_t a0 = p0 >= start + 32u ? p0 - 32u : start;
    const uint32_t an = min(end, p0 + 64u) - a0;  // at most 96
    const uint32_t npad = (an + 3u) & ~3u;
    __syncwarp();
    for (uint32_t e = lane; e < npad; e += 32) {
      Pt<DP> x;
#pragma unroll
      for (int k = 0; k < DP; ++k) x.x[k] = -INFINITY;
      unsigned long long kc = 0ull;
      if (e < an) {
        x = load_pt<DP>(spts, a0 + e);
        kc = skey[a0 + e];
      }
#pragma unroll
      for (int k = 0; k < ND; ++k) tile.x[k][e] = -x.x[k];
      tile.key[e] = kc;
    }
    __syncwarp();
    const uint32_t p = p0 + lane;
    const bool valid = p < end;
    const uint32_t own = (valid ? p : p0) - a0;
    const unsigned long long K = tile.key[own];
    const Pt<DP> me = tile_pt<DP>(tile, own);
    f32x2 q2[ND];
#pragma unroll
    for (int k = 0; k < ND; ++k) q2[k] = pack2(me.x[k], me.x[k]);
    float s1 = INFINITY;
#pragma unroll 2
    for (uint32_t i = 0; i < npad; i += 4) {
      const ulonglong2 k0 = *reinterpret_cast<const ulonglong2*>(&tile.key[i]);
      const ulonglong2 k1 = *reinterpret_cast<const ulonglong2*>(&tile.key[i + 2]);
      f32x2 cc[2][ND];
      tile_quad(tile, i, cc);
      const f32x2 sa = dist32x2<ND>(q2, cc[0]), sb = dist32x2<ND>(q2, cc[1]);
      s1 = fminf(s1, k0.x > K ? lo2(sa) : INFINITY);
      s1 = fminf(s1, k0.y > K ? hi2(sa) : INFINITY);
      s1 = fminf(s1, k1.x > K ? lo2(sb) : INFINITY);
      s1 = fminf(s1, k1.y > K ? hi2(sb) : INFINITY);
    }
    const CutGeom& C = cuts[inst];
    const bool skip = valid && (int32_t)(K >> 32) < max(rho_skip, C.skip);
    if (skip) {
      const uint32_t id = key_id(K);
      lambda[id] = -1;
      delta[id] = __longlong_as_double(0x7ff8000000000000ll);  // NaN: skipped
    }
    // the instance's highest point has no dependent point: its key is the
    // largest of the root's record
    const uint32_t root = roots[inst];
    bool top = false;
    if (valid && !skip && root < cv.N - 1u) {  // (kNoNode: an instance of one point)
      const unsigned long long* rk =
          reinterpret_cast<const unsigned long long*>(nbox + (size_t)root * rec_words<RD>() + 4);
      top = rk[0] <= K && rk[1] <= K;
    }
    if (top) {
      const uint32_t id = key_id(K);
      lambda[id] = -1;
      delta[id] = INFINITY;
    }
    const bool push = valid && !skip && !top;
    const unsigned pm = __ballot_sync(kFull, push);
    uint32_t base = 0;
    if (lane == 0 && pm) base = atomicAdd(&ctr->queue_n, (unsigned)__popc(pm));
    base = __shfl_sync(kFull, base, 0);
    if (push) {
      const uint32_t slot = base + __popc(pm & lanemask_lt);
      q.pos[slot] = p;
      q.s1[slot] = s1;
      // the binary64 search prunes with distances of its own: the bound is
      // widened by the float32 error
      q.s1d[slot] = s1 < INFINITY ? (double)band_of(s1, C.band_mul, C.band_add) : (double)INFINITY;
    }
  }
}

// ---------------------------------------------------------------------------
// far phase: depth-first priority search of the radix tree

// Squared lower bound between the query and the bounding box of a subtree
// (all coordinates; box layout [lo(RD) | hi(RD)] per node, tree.cu), scaled
// 1e-5 down (F64: and kPruneTiny less) so that it stays below the float32 (F64: the
// binary64) distance of every point inside despite the rounding of this
// evaluation and of dist32.
template <int DP, int RD, bool F64>
__device__ __forceinline__ float rec_lb2(const ChildRec<RD>& r, int s, const Pt<DP>& x) {
  float lb2 = 0.f;
#pragma unroll
  for (int a = 0; a < RD; ++a) {
    const float l = fmaxf(fmaxf(r.lo[s][a] - x.x[a], x.x[a] - r.hi[s][a]), 0.f);
    lb2 = fmaf(l, l, lb2);
  }
  return F64 ? fmaf(lb2, 1.f - 1e-5f, -kPruneTiny) : lb2 * (1.f - 1e-5f);
}

// A leaf child's point, from its record (its box is the point itself).
template <int DP, int RD>
__device__ __forceinline__ Pt<DP> rec_point(const ChildRec<RD>& r, int s) {
  Pt<DP> p;
#pragma unroll
  for (int a = 0; a < DP; ++a) p.x[a] = a < RD ? r.lo[s][a < RD ? a : 0] : 0.f;
  return p;
}

enum { kWalkDone = 0, kWalkBudget = 1, kWalkBad = -1 };

// One thread's depth-first search below internal node `start`, nearer child
// first: every leaf with key > K not excluded by `prune` is passed to
// visit(t, kt, point).  Expanding a node reads its child record alone (the
// children's indices, keys and boxes).  Stops with kWalkBudget after `budget` node expansions, and
// with kWalkBad on a malformed tree or stack overflow (neither happens for a
// tree built by tree.cu: its depth is at most 64 + 32).
template <int DP, int RD, bool F64, typename Prune, typename Visit>
__device__ __noinline__ int tree_walk_from(const float* __restrict__ nbox, uint32_t n,
                                           unsigned long long K, const Pt<DP>& xq,
                                           uint32_t start, uint32_t budget, uint32_t& expanded,
                                           Prune prune, Visit visit) {
  uint32_t stk[kStack];
  float stl[kStack];
  int sp = 0;
  stk[sp] = start;
  stl[sp] = 0.f;
  ++sp;
  while (sp > 0) {
    --sp;
    const uint32_t ni = stk[sp];
    if (prune(stl[sp])) continue;
    if (ni + 1 >= n) return kWalkBad;
    if (expanded >= budget) return kWalkBudget;
    ++expanded;
    const ChildRec<RD> r = load_rec<RD>(nbox, ni);
    uint32_t keep[2];
    float keepl[2];
    int nk = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const uint32_t c = r.child[s];
      if (r.key[s] <= K) continue;  // nothing of higher key below
      if (c & kLeafBit) {
        if ((c & ~kLeafBit) >= n) return kWalkBad;
        visit(c & ~kLeafBit, r.key[s], rec_point<DP, RD>(r, s));
      } else {
        const float lbs = rec_lb2<DP, RD, F64>(r, s, xq);
        if (prune(lbs)) continue;
        keep[nk] = c;
        keepl[nk] = lbs;
        ++nk;
      }
    }
    if (sp + nk > kStack) return kWalkBad;
    if (nk == 2 && keepl[0] < keepl[1]) {  // push the farther child first
      stk[sp] = keep[1]; stl[sp] = keepl[1]; ++sp;
      stk[sp] = keep[0]; stl[sp] = keepl[0]; ++sp;
    } else {
      for (int s = 0; s < nk; ++s) { stk[sp] = keep[s]; stl[sp] = keepl[s]; ++sp; }
    }
  }
  return kWalkDone;
}

// The walk of the far phase's first round: as tree_walk_from, with the nearer
// child kept in a register (only the farther one is pushed) and the stack in
// shared memory, [entry][thread]: lanes of a warp stand at different depths, so
// entries in local memory cost a sector per lane and access.  Entries past
// kFastStack (deep trees) go to a local array.  Leaves are visited by their record
// (the point is in it); a caller that reads memory at a leaf's index checks it.
constexpr int kFastStack = 24;
struct FastStack {
  uint32_t node[kFastStack][kFarThreads];
  float lb[kFastStack][kFarThreads];
};

template <int DP, int RD, bool F64, typename Prune, typename Visit>
__device__ __forceinline__ int far_walk(FastStack& fs, const float* __restrict__ nbox, uint32_t n,
                                        unsigned long long K, const Pt<DP>& xq, uint32_t start, uint32_t budget,
                                        uint32_t& expanded, Prune prune, Visit visit) {
  const int tid = threadIdx.x;
  uint32_t more[kStack - kFastStack];
  float morel[kStack - kFastStack];
  int sp = 0;
  uint32_t ni = start;
  for (;;) {
    if (ni + 1 >= n) return kWalkBad;
    if (expanded >= budget) return kWalkBudget;
    ++expanded;
    const ChildRec<RD> r = load_rec<RD>(nbox, ni);
    const bool h0 = r.key[0] > K, h1 = r.key[1] > K;  // something of higher key below
    const bool leaf0 = r.child[0] & kLeafBit, leaf1 = r.child[1] & kLeafBit;
    if (h0 && leaf0) visit(r.child[0] & ~kLeafBit, r.key[0], rec_point<DP, RD>(r, 0));
    if (h1 && leaf1) visit(r.child[1] & ~kLeafBit, r.key[1], rec_point<DP, RD>(r, 1));
    const float l0 = rec_lb2<DP, RD, F64>(r, 0, xq), l1 = rec_lb2<DP, RD, F64>(r, 1, xq);
    const bool g0 = h0 && !leaf0 && !prune(l0), g1 = h1 && !leaf1 && !prune(l1);
    if (g0 && g1) {
      const bool first = l0 < l1;
      const uint32_t far_c = first ? r.child[1] : r.child[0];
      const float far_l = first ? l1 : l0;
      if (sp < kFastStack) {
        fs.node[sp][tid] = far_c;
        fs.lb[sp][tid] = far_l;
      } else if (sp < kStack) {
        more[sp - kFastStack] = far_c;
        morel[sp - kFastStack] = far_l;
      } else {
        return kWalkBad;
      }
      ++sp;
      ni = first ? r.child[0] : r.child[1];
    } else if (g0 || g1) {
      ni = g0 ? r.child[0] : r.child[1];
    } else {
      float l;
      do {
        if (sp == 0) return kWalkDone;
        --sp;
        if (sp < kFastStack) {
          ni = fs.node[sp][tid];
          l = fs.lb[sp][tid];
        } else {
          ni = more[sp - kFastStack];
          l = morel[sp - kFastStack];
        }
      } while (prune(l));
    }
  }
}

// Per-query context shared by the two far kernels.
template <int DP>
struct FarQuery {
  uint32_t p, id, inst;
  uint32_t base;   // output index of the instance's point 0 (ids - base = local ids)
  uint32_t root;   // the instance's subtree, kNoNode for a single point
  unsigned long long K;
  Pt<DP> xq;
  __device__ __forceinline__ void load(uint32_t pos, const float* __restrict__ spts,
                                       const unsigned long long* __restrict__ scode,
                                       const unsigned long long* __restrict__ skey,
                                       const ClassView& cv, const uint32_t* __restrict__ roots,
                                       int S, int ib) {
    p = pos;
    K = skey[p];
    id = key_id(K);
    xq = load_pt<DP>(spts, p);
    inst = key_inst(scode[p], S, ib);
    if (inst >= cv.ninst) inst = 0;
    base = (uint32_t)cv.instance(inst).out;
    root = roots[inst];
  }
};

// The dependent point of the same point under another cutoff of the sweep, if
// it is higher here too: its distance bounds the search from the start (the
// walk meets it again, so it needs no place among the candidates).
template <int DP, bool F64>
__device__ __forceinline__ double hint_bound(const FarHint& h, const ClassView& cv, const FarQuery<DP>& fq) {
  if (!h.lambda) return INFINITY;
  const int32_t l = h.lambda[fq.id];
  const InstDev I = cv.instance(fq.inst);
  if (l < 0 || (uint32_t)l >= I.n) return INFINITY;
  const uint32_t o = fq.base + (uint32_t)l;
  if (order_key(h.rho[o], o) <= fq.K) return INFINITY;
  const Pt<DP> x = input_pt<DP>(h.pts, h.dtype, I.coord, I.d, (uint32_t)l);
  if constexpr (F64) return dist64<DP>(fq.xq, x);
  else return (double)dist32<DP>(fq.xq, x);
}

// Node expansions a query may take in the first round.  The second round gives
// a long search a whole warp, which shortens the last searches of a small set
// but expands more nodes per query and starts over, so it is left to sets that
// do not fill the chip and to the longest searches of the others: the budget
// grows with the queries per resident thread (`room` of them).  Measured with
// budgets of 128 / 256 / 512 / 1024 / 2048, far search in ms: 7-D, 438,000 far
// queries of 2e6 points 17.7 / 16.3 / 12.2 / 10.4 / 10.6; 5-D, 1e6 queries
// 18.2 / 6.4 / 5.4 / 5.7 / 5.9; 5-D, 1e5 queries .88 / .48 / .55 / .70 / .85;
// 7-D, 13,000 queries .43 / .43 / .56 / .76 / .98; 3-D, 1.5e5 queries .154 /
// .181 / .199 / .200 / .203; 2-D, 1e6 queries .290 / .280 / .265 / .267 / .267.
template <int DP>
__device__ __forceinline__ uint32_t far_budget(uint32_t qn, uint32_t room) {
  const uint32_t b = (uint32_t)min((unsigned long long)qn * (DP > 4 ? 768u : 64u) / room, 1024ull);
  return min(max(b, kFarBudget), DP > 4 ? 1024u : 512u);
}

// Far queries, first round: one thread per query, a depth-first search with
// an expansion budget.  Most queries finish within it; the others are passed to
// the second round with the best distance found so far, which bounds their
// search there.  What bounds it is the child records' way from L2 (7-D: 32e9
// expansions/s of 160 bytes, 5.1 TB/s).  Letting a lane that is done take the
// next query while its neighbours go on costs more than the idle lanes (1e6
// 2-D queries .35 ms for .26).
template <int DP, int RD, bool F64>
__global__ void __launch_bounds__(kFarThreads)
k_dep_far(const float* __restrict__ spts, const unsigned long long* __restrict__ scode,
          const unsigned long long* __restrict__ skey, ClassView cv,
          const CutGeom* __restrict__ cuts,
          const float* __restrict__ nbox, const uint32_t* __restrict__ roots, FarQueue q, FarHint hint,
          int32_t* __restrict__ lambda, double* __restrict__ delta, Counters* ctr, uint32_t room) {
  __shared__ FastStack fs;
  const uint32_t qn = ctr->queue_n;
  const uint32_t budget = far_budget<DP>(qn, room);
  const uint32_t n = cv.N;
  const int S = cv.cls->S, ib = cv.cls->ib;
  // the band depends only on DP, the same for every instance of the class
  const float bmul = cuts[0].band_mul, badd = cuts[0].band_add;
  const uint32_t lanemask_lt = (1u << (threadIdx.x & 31)) - 1u;
  unsigned long long rescans = 0, expanded_sum = 0;
  uint32_t expanded_max = 0;
  bool bad = false;
  const uint32_t qn_pad = (qn + 31) & ~31u;  // whole warps, for the ballot below
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < qn_pad; e += gridDim.x * blockDim.x) {
    bool pass_on = false;
    double s_next = INFINITY;
    uint32_t expanded = 0;
    FarQuery<DP> fq;
    if (e < qn) {
      fq.load(q.pos[e], spts, scode, skey, cv, roots, S, ib);
      if (fq.root == kNoNode) {
        lambda[fq.id] = -1;
        delta[fq.id] = INFINITY;
      } else if constexpr (F64) {
        Best<double> best;
        best.init();
        const double s_init = fmin(q.s1d[e], hint_bound<DP, true>(hint, cv, fq));
        const int r = far_walk<DP, RD, F64>(
            fs, nbox, n, fq.K, fq.xq, fq.root, budget, expanded,
            [&](float lbs) { return (double)lbs > fmin(best.s1, s_init); },
            [&](uint32_t t, unsigned long long kt, const Pt<DP>& x) {
              best.add(dist64<DP>(fq.xq, x), key_id(kt), t);
            });
        bad |= r == kWalkBad;
        if (r == kWalkBudget) {
          pass_on = true;
          s_next = fmin(best.s1, s_init);
        } else if (best.t1 == 0xffffffffu) {
          lambda[fq.id] = -1;
          delta[fq.id] = INFINITY;
        } else {
          lambda[fq.id] = (int32_t)(best.o1 - fq.base);
          delta[fq.id] = sqrt(best.s1);
        }
      } else {
        Best<float> best;
        best.init();
        const float s_init = fminf(q.s1[e], (float)hint_bound<DP, false>(hint, cv, fq));
        const int r = far_walk<DP, RD, F64>(
            fs, nbox, n, fq.K, fq.xq, fq.root, budget, expanded,
            [&](float lbs) { return beyond(lbs, band_of(fminf(best.s1, s_init), bmul, badd)); },
            [&](uint32_t t, unsigned long long kt, const Pt<DP>& x) {
              best.add(dist32<DP>(fq.xq, x), key_id(kt), t);
            });
        bad |= r == kWalkBad;
        if (r == kWalkBudget) {
          pass_on = true;
          s_next = fminf(best.s1, s_init);
        } else if (best.t1 >= n) {  // nothing higher (or a malformed tree: far_walk checks no leaf)
          bad |= best.t1 != 0xffffffffu;
          lambda[fq.id] = -1;
          delta[fq.id] = INFINITY;
        } else {
          const float b = band_of(best.s1, bmul, badd);
          Exact ex;
          ex.init();
          if (best.s2 <= b) {  // near tie: re-rank the band in binary64
            ++rescans;
            uint32_t more = 0;
            bad |= tree_walk_from<DP, RD, F64>(
                       nbox, n, fq.K, fq.xq, fq.root, 0xffffffffu, more,
                       [&](float lbs) { return beyond(lbs, b); },
                       [&](uint32_t t, unsigned long long kt, const Pt<DP>& x) {
                         if (dist32<DP>(fq.xq, x) <= b) ex.add(dist64<DP>(fq.xq, x), key_id(kt));
                       }) != kWalkDone;
            expanded += more;
          } else {
            ex.add(dist64<DP>(fq.xq, load_pt<DP>(spts, best.t1)), best.o1);
          }
          lambda[fq.id] = (int32_t)(ex.o - fq.base);
          delta[fq.id] = sqrt(ex.s);
        }
      }
    }
    expanded_sum += expanded;
    expanded_max = max(expanded_max, expanded);
    const unsigned pm = __ballot_sync(kFull, pass_on);
    uint32_t base = 0;
    if ((threadIdx.x & 31) == 0 && pm) base = atomicAdd(&ctr->queue2_n, (unsigned)__popc(pm));
    base = __shfl_sync(kFull, base, 0);
    if (pass_on) {
      const uint32_t slot = base + __popc(pm & lanemask_lt);
      q.pos2[slot] = fq.p;
      if constexpr (F64) q.s1d2[slot] = s_next;
      else q.s1_2[slot] = (float)s_next;
    }
  }
  if (bad) set_status(cv.cls->status, kStatusStack);
  for (int o = 16; o > 0; o >>= 1) {
    rescans += __shfl_xor_sync(kFull, rescans, o);
    expanded_sum += __shfl_xor_sync(kFull, expanded_sum, o);
    expanded_max = max(expanded_max, __shfl_xor_sync(kFull, expanded_max, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (rescans) atomicAdd(&ctr->exact_rescans, rescans);
    if (expanded_sum) atomicAdd(&ctr->far_nodes, expanded_sum);
    if (expanded_max) atomicMax(&ctr->far_nodes_max, expanded_max);
  }
}

// Far queries, second round: the queries that exceeded the first round's
// budget, one warp per query.  The search restarts at the root with the
// first round's best as its bound, so the warp can expand 32 nodes per step
// (one per lane) without wandering: every round pops up to 32 entries from
// the warp's shared stack, each lane expands its node, and the survivors are
// pushed with a warp prefix sum.  Children that do not fit on the stack are
// searched by their lane alone.
template <int DP, int RD, bool F64>
__global__ void __launch_bounds__(kFarThreads)
k_dep_far_wide(const float* __restrict__ spts, const unsigned long long* __restrict__ scode,
               const unsigned long long* __restrict__ skey, ClassView cv,
               const CutGeom* __restrict__ cuts,
               const float* __restrict__ nbox, const uint32_t* __restrict__ roots, FarQueue q,
               int32_t* __restrict__ lambda, double* __restrict__ delta, Counters* ctr) {
  constexpr int kWarpsPerBlock = kFarThreads / 32;
  __shared__ uint32_t s_stk[kWarpsPerBlock][kWarpStack];
  __shared__ float s_lb[kWarpsPerBlock][kWarpStack];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  uint32_t* stk = s_stk[wib];
  float* stl = s_lb[wib];
  const uint32_t qn = ctr->queue2_n;
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // statistics of the round
    ctr->far_queries += ctr->queue_n;
    ctr->far_wide_queries += qn;
  }
  const uint32_t n = cv.N;
  const int S = cv.cls->S, ib = cv.cls->ib;
  const float bmul = cuts[0].band_mul, badd = cuts[0].band_add;
  unsigned long long rescans = 0, expanded_sum = 0;
  uint32_t expanded_max = 0;
  bool bad = false;
  const uint32_t nwarps = gridDim.x * kWarpsPerBlock;
  for (uint32_t e = blockIdx.x * kWarpsPerBlock + wib; e < qn; e += nwarps) {
    FarQuery<DP> fq;
    fq.load(q.pos2[e], spts, scode, skey, cv, roots, S, ib);
    uint32_t expanded = 0;

    auto search = [&](auto refresh, auto prune, auto visit) {
      if (lane == 0) {
        stk[0] = fq.root;
        stl[0] = 0.f;
      }
      int sp = 1;
      __syncwarp();
      while (sp > 0) {
        refresh();
        const int take = sp < 32 ? sp : 32;
        const int base = sp - take;
        uint32_t keep[2];
        float keepl[2];
        int nk = 0;
        if (lane < take) {
          const uint32_t ni = stk[base + lane];
          const float lbn = stl[base + lane];
          if (!prune(lbn)) {
            if (ni + 1 >= n) {
              bad = true;
            } else {
              ++expanded;
              const ChildRec<RD> r = load_rec<RD>(nbox, ni);
#pragma unroll
              for (int s = 0; s < 2; ++s) {
                const uint32_t c = r.child[s];
                if (r.key[s] <= fq.K) continue;  // nothing of higher key below
                if (c & kLeafBit) {
                  if ((c & ~kLeafBit) >= n) {
                    bad = true;
                    continue;
                  }
                  visit(c & ~kLeafBit, r.key[s], rec_point<DP, RD>(r, s));
                } else {
                  const float l = rec_lb2<DP, RD, F64>(r, s, fq.xq);
                  if (prune(l)) continue;
                  keep[nk] = c;
                  keepl[nk] = l;
                  ++nk;
                }
              }
              if (nk == 2 && keepl[0] < keepl[1]) {  // farther first: nearer is popped sooner
                const uint32_t tc = keep[0]; keep[0] = keep[1]; keep[1] = tc;
                const float tl = keepl[0]; keepl[0] = keepl[1]; keepl[1] = tl;
              }
            }
          }
        }
        uint32_t incl = (uint32_t)nk;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t t = __shfl_up_sync(kFull, incl, d);
          if (lane >= d) incl += t;
        }
        const int total = (int)__shfl_sync(kFull, incl, 31);
        const int pos = base + (int)incl - nk;
        __syncwarp();
        for (int s = 0; s < nk; ++s) {
          if (pos + s < kWarpStack) {
            stk[pos + s] = keep[s];
            stl[pos + s] = keepl[s];
          } else {  // no room: this lane searches the subtree alone
            bad |= tree_walk_from<DP, RD, F64>(nbox, n, fq.K, fq.xq, keep[s], 0xffffffffu,
                                      expanded, prune, visit) != kWalkDone;
          }
        }
        sp = min(base + total, kWarpStack);
        __syncwarp();
      }
    };

    if constexpr (F64) {
      Best<double> best;
      best.init();
      const double s_init = q.s1d2[e];
      double wbest = s_init;  // the warp's best, refreshed every round
      search(
          [&] {
            double m = best.s1;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fmin(m, __shfl_xor_sync(kFull, m, o));
            wbest = fmin(m, s_init);
          },
          [&](float lbs) { return (double)lbs > fmin(best.s1, wbest); },
          [&](uint32_t t, unsigned long long kt, const Pt<DP>& x) {
            best.add(dist64<DP>(fq.xq, x), key_id(kt), t);
          });
      best.merge_warp();
      if (lane == 0) {
        if (best.t1 == 0xffffffffu) {
          lambda[fq.id] = -1;
          delta[fq.id] = INFINITY;
        } else {
          lambda[fq.id] = (int32_t)(best.o1 - fq.base);
          delta[fq.id] = sqrt(best.s1);
        }
      }
    } else {
      Best<float> best;
      best.init();
      const float s_init = q.s1_2[e];
      float wbest = s_init;  // the warp's best, refreshed every round
      search(
          [&] {
            float m = best.s1;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(kFull, m, o));
            wbest = fminf(m, s_init);
          },
          [&](float lbs) { return beyond(lbs, band_of(fminf(best.s1, wbest), bmul, badd)); },
          [&](uint32_t t, unsigned long long kt, const Pt<DP>& x) {
            best.add(dist32<DP>(fq.xq, x), key_id(kt), t);
          });
      best.merge_warp();
      if (best.t1 == 0xffffffffu) {
        if (lane == 0) {
          lambda[fq.id] = -1;
          delta[fq.id] = INFINITY;
        }
      } else {
        const float b = band_of(best.s1, bmul, badd);
        Exact ex;
        ex.init();
        if (best.s2 <= b) {  // near tie: re-rank the band in binary64
          ++rescans;
          search([] {}, [&](float lbs) { return beyond(lbs, b); },
                 [&](uint32_t t, unsigned long long kt, const Pt<DP>& x) {
                   if (dist32<DP>(fq.xq, x) <= b) ex.add(dist64<DP>(fq.xq, x), key_id(kt));
                 });
          ex.merge_warp();
        } else if (lane == 0) {
          ex.add(dist64<DP>(fq.xq, load_pt<DP>(spts, best.t1)), best.o1);
        }
        if (lane == 0) {
          lambda[fq.id] = (int32_t)(ex.o - fq.base);
          delta[fq.id] = sqrt(ex.s);
        }
      }
    }
    expanded_sum += expanded;
    uint32_t qexp = expanded;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) qexp += __shfl_xor_sync(kFull, qexp, o);
    expanded_max = max(expanded_max, qexp);
  }
  if (__any_sync(kFull, bad) && lane == 0) set_status(cv.cls->status, kStatusStack);
  for (int o = 16; o > 0; o >>= 1) expanded_sum += __shfl_xor_sync(kFull, expanded_sum, o);
  if (lane == 0) {
    if (rescans) atomicAdd(&ctr->exact_rescans, rescans);
    if (expanded_sum) atomicAdd(&ctr->far_nodes, expanded_sum);
    if (expanded_max) atomicMax(&ctr->far_nodes_max, expanded_max);
  }
}

inline unsigned grid_for(uint64_t items, int per_block, unsigned cap) {
  uint64_t b = (items + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (unsigned)b;
}

template <int DP, int G>
void near_dg(bool fp64, int layout, const float* spts, const unsigned long long* scode,
             const unsigned long long* skey, const ClassView& cv, int32_t rho_skip,
             const void* pts, int dtype, const CutGeom* cuts, const HashInfo* hi,
             const unsigned long long* hkeys, const uint2* hvals, int32_t* lambda, double* delta,
             FarQueue q, Counters* ctr, int seg_cells, uint32_t min_fill, cudaStream_t st) {
  // (a launch that most sets leave at once: fewer CTAs)
  const unsigned grid = grid_for(cv.nchunk, kNearWarps, sm_count() * (min_fill ? 16u : 64u));
  if (layout == kLayoutSegment) {
    if (fp64)
      k_dep_near_seg<DP, G, true><<<grid, kNearThreads, 0, st>>>(spts, scode, skey, cv, rho_skip, pts,
                                                                 dtype, cuts, hi, hkeys, hvals, lambda,
                                                                 delta, q, ctr, seg_cells);
    else
      k_dep_near_seg<DP, G, false><<<grid, kNearThreads, 0, st>>>(spts, scode, skey, cv, rho_skip, pts,
                                                                  dtype, cuts, hi, hkeys, hvals, lambda,
                                                                  delta, q, ctr, seg_cells);
  } else {
    if (fp64)
      k_dep_near<DP, G, true><<<grid, kNearThreads, 0, st>>>(spts, scode, skey, cv, rho_skip, pts,
                                                             dtype, cuts, hi, hkeys, hvals, lambda,
                                                             delta, q, ctr, min_fill);
    else
      k_dep_near<DP, G, false><<<grid, kNearThreads, 0, st>>>(spts, scode, skey, cv, rho_skip, pts,
                                                              dtype, cuts, hi, hkeys, hvals, lambda,
                                                              delta, q, ctr, min_fill);
  }
}

template <int DP, int RD>
void far_dp(bool fp64, const float* spts, const unsigned long long* scode,
            const unsigned long long* skey, const ClassView& cv, const CutGeom* cuts,
            const float* nbox, const uint32_t* root, FarQueue q, const FarHint& hint,
            int32_t* lambda, double* delta, Counters* ctr, cudaStream_t st) {
  // the queue length is known only on the device: CTAs for most lengths, so
  // that a free SM takes the next 128 queries (1e6 2-D queries .27 -> .24 ms,
  // 438,000 7-D queries 9.8 -> 8.7 against 8 CTAs per SM striding over the
  // queue, of which 6 were resident in 7-D); those without a query end at once
  const unsigned grid = grid_for(cv.N, kFarThreads, sm_count() * kFarGrid);
  const uint32_t room = sm_count() * 1024u;
  const unsigned grid2 = grid_for(cv.N, kFarThreads / 32, sm_count() * 16u);
  if (fp64) {
    k_dep_far<DP, RD, true><<<grid, kFarThreads, 0, st>>>(spts, scode, skey, cv, cuts, nbox,
                                                      root, q, hint, lambda, delta, ctr, room);
    k_dep_far_wide<DP, RD, true><<<grid2, kFarThreads, 0, st>>>(spts, scode, skey, cv, cuts,
                                                            nbox, root, q, lambda, delta, ctr);
  } else {
    k_dep_far<DP, RD, false><<<grid, kFarThreads, 0, st>>>(spts, scode, skey, cv, cuts, nbox,
                                                       root, q, hint, lambda, delta, ctr, room);
    k_dep_far_wide<DP, RD, false><<<grid2, kFarThreads, 0, st>>>(spts, scode, skey, cv, cuts,
                                                             nbox, root, q, lambda, delta, ctr);
  }
}

}  // namespace

void launch_dep_near(int dp, int g, int dmax, bool fp64, int layout, const float* spts,
                     const unsigned long long* scode, const unsigned long long* skey,
                     const ClassView& cv, int32_t rho_skip, const void* pts, int dtype,
                     const CutGeom* cuts, const HashInfo* hi, const unsigned long long* hkeys,
                     const uint2* hvals, int32_t* lambda, double* delta, FarQueue q, Counters* ctr,
                     cudaStream_t st, const float* nbox, const uint32_t* roots, int seg_cells,
                     uint32_t skip_fill, uint32_t min_fill) {
  if (cv.N == 0) return;
  // (skip_fill: beside a form for dense cells, which has cleared the queue and may
  // have filled it)
  if (!skip_fill) cudaMemsetAsync(&ctr->queue_n, 0, 2 * sizeof(unsigned int), st);  // queue_n and queue2_n
  if (layout == kLayoutCell) {
    launch_dep_near_cell(dp, g, fp64, spts, scode, skey, cv, rho_skip, pts, dtype, cuts, hi, hkeys,
                         hvals, lambda, delta, q, ctr, st);
    return;  // counted there
  }
  if (layout == kLayoutTree) {
    const unsigned grid = grid_for(cv.nchunk, kNearWarps, sm_count() * 64u);
    auto go = [&](auto kern) {
      kern<<<grid, kNearThreads, 0, st>>>(spts, skey, cv, cuts, rho_skip, lambda, delta, q, ctr, hi, nbox, roots,
                                          skip_fill);
    };
    if (g == 1) go(k_near_to_far<2, 1, 2>);
    else if (g == 2) go(k_near_to_far<2, 2, 2>);
    else if (g == 3) go(k_near_to_far<4, 3, 4>);
    else if (dp == 4) go(k_near_to_far<4, 4, 4>);
    else if (rec_dims(dp, dmax) == 6) go(k_near_to_far<8, 6, 6>);
    else go(k_near_to_far<8, 8, 8>);
  } else if (g == 1) near_dg<2, 1>(fp64, layout, spts, scode, skey, cv, rho_skip, pts, dtype, cuts, hi, hkeys, hvals, lambda, delta, q, ctr, seg_cells, min_fill, st);
  else if (g == 2) near_dg<2, 2>(fp64, layout, spts, scode, skey, cv, rho_skip, pts, dtype, cuts, hi, hkeys, hvals, lambda, delta, q, ctr, seg_cells, min_fill, st);
  else if (g == 3) near_dg<4, 3>(fp64, layout, spts, scode, skey, cv, rho_skip, pts, dtype, cuts, hi, hkeys, hvals, lambda, delta, q, ctr, seg_cells, min_fill, st);
  else if (dp == 4) near_dg<4, 4>(fp64, layout, spts, scode, skey, cv, rho_skip, pts, dtype, cuts, hi, hkeys, hvals, lambda, delta, q, ctr, seg_cells, min_fill, st);
  else near_dg<8, 4>(fp64, layout, spts, scode, skey, cv, rho_skip, pts, dtype, cuts, hi, hkeys, hvals, lambda, delta, q, ctr, seg_cells, min_fill, st);
  count_launches(1);
}

void launch_dep_far(int dp, int dmax, bool fp64, const float* spts, const unsigned long long* scode,
                    const unsigned long long* skey, const ClassView& cv, const CutGeom* cuts,
                    const float* nbox, const uint32_t* root, FarQueue q,
                    const FarHint& hint, int32_t* lambda, double* delta, Counters* ctr, cudaStream_t st) {
  if (cv.N == 0) return;
  if (dp == 2) far_dp<2, 2>(fp64, spts, scode, skey, cv, cuts, nbox, root, q, hint, lambda, delta, ctr, st);
  else if (dp == 4) far_dp<4, 4>(fp64, spts, scode, skey, cv, cuts, nbox, root, q, hint, lambda, delta, ctr, st);
  else if (rec_dims(dp, dmax) == 6) far_dp<8, 6>(fp64, spts, scode, skey, cv, cuts, nbox, root, q, hint, lambda, delta, ctr, st);
  else far_dp<8, 8>(fp64, spts, scode, skey, cv, cuts, nbox, root, q, hint, lambda, delta, ctr, st);
  count_launches(2);
}

}  // namespace dpc

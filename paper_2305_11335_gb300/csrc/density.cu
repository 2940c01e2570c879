// density.cu -- rho_i = |{j : D(x_i, x_j) <= d_cut}| (Definition 1).
//
// One query per lane, 32 consecutive Morton-sorted queries per warp; the warp
// stages the union of its queries' grid blocks in shared memory (block.cuh)
// and each lane counts the points of its own (2R+1)^g block, reading every
// candidate as a broadcast.
//   FP32_CERT: s32 <= t_in counts, s32 > t_out does not.  Pairs in between
//              (about 1e-6 of d_cut^2 wide) are counted with the canonical
//              binary64 distance in a separate pass, taken only by a warp that
//              met one, so the hot loop stays float32.
//   FP64:      every pair is evaluated in binary64.
// Both give exactly the binary64 count.  The kernel also writes the order key
// of every sorted point, (rho << 32) | ~id.
#include <type_traits>

#include "block.cuh"
#include "internal.h"

namespace dpc {

namespace {

constexpr int kWarps = 4;
constexpr int kThreads = kWarps * 32;

template <int DP>
constexpr int density_cap() { return DP == 8 ? 256 : 512; }

// Exact count of this lane's band pairs among the window's candidates (rare
// path, taken only by a warp that met a band pair in this window).
template <int DP, int G>
__device__ __noinline__ int2 band_recount(const RunTable& rt, int nr, const Union<G> u,
                                          uint32_t w0, uint32_t w1, const float* wpts,
                                          const uint32_t* c0, bool act, int R, Pt<DP> me,
                                          float t_in, float t_out, double dc2) {
  int in = 0, seen = 0;
  for_window_runs<G>(rt, nr, u, w0, w1, [&](uint32_t i0, uint32_t i1, const uint32_t* cc) {
    if (!(act && in_block<G>(c0, cc, R))) return;
    for (uint32_t i = i0; i < i1; ++i) {
      const Pt<DP> x = window_pt<DP>(wpts, i);
      const float s32 = dist32<DP>(me, x);
      if (s32 > t_in && s32 <= t_out) {
        ++seen;
        in += dist64<DP>(me, x) <= dc2;
      }
    }
  });
  return make_int2(in, seen);
}

// Resident blocks per SM the register budget must allow (shared memory
// allows 10 of the 2-D and 5 of the wider blocks).
template <int DP>
constexpr int density_min_blocks() { return DP == 2 ? 7 : 5; }

template <int DP, int G, bool F64>
__global__ void __launch_bounds__(kThreads, density_min_blocks<DP>())
k_density(const float* __restrict__ spts, const unsigned long long* __restrict__ scode,
          const uint32_t* __restrict__ sid, ClassView cv, const CutGeom* __restrict__ cuts,
          const HashInfo* __restrict__ hi, const unsigned long long* __restrict__ hkeys,
          const uint2* __restrict__ hvals, int32_t* __restrict__ rho_out,
          unsigned long long* __restrict__ skey, Counters* ctr) {
  constexpr int ND = real_dims<DP, G>();
  constexpr int kCap = density_cap<DP>();
  __shared__ __align__(16) float s_pts[kWarps * kCap * DP];
  __shared__ RunTable s_rt[kWarps];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  float* wpts = s_pts + wib * kCap * DP;
  RunTable& rt = s_rt[wib];
  const int S = cv.cls->S, ib = cv.cls->ib;
  const uint32_t hmask = hi->hmask;
  const uint32_t n = cv.N;

  unsigned long long band = 0, pairs = 0;
  for (uint32_t ch = blockIdx.x * kWarps + wib; ch < cv.nchunk; ch += gridDim.x * kWarps) {
    uint32_t inst, p0, end;
    cv.chunk(ch, inst, p0, end);
    const CutGeom& C = cuts[inst];
    const int k = C.k;
    const int R = C.R;
    const int shift = G * k;
    const int cmax = (1 << (cv.geom[inst].B - k)) - 1;
    const double dc2 = C.dc2;
    const float t_in = C.t_in, t_out = C.t_out;
    const unsigned long long hb = ib ? ((unsigned long long)inst << S) : 0ull;
    const uint32_t p = p0 + lane;
    const bool valid = p < end;
    Pt<DP> me;
#pragma unroll
    for (int a = 0; a < DP; ++a) me.x[a] = 0.f;
    if (valid) me = load_pt<DP>(spts, p);
    const unsigned long long mycell = valid ? (key_code(scode[p], S, ib) >> shift) : ~0ull;
    uint32_t c0[G];
    unmorton<G>(valid ? mycell : 0ull, c0);
    const int nvalid = (int)min(32u, end - p0);
    int32_t count = 0;
    for_groups<G>(mycell, c0, valid, valid, nvalid, R, cmax, lane, [&](bool act, const Union<G>& u) {
      const int nr = union_runs<G>(u, hkeys, hvals, hmask, hb, n, lane, rt);
      const uint32_t total = rt.pre[nr];
      for (uint32_t w0 = 0; w0 < total; w0 += kCap) {
        const uint32_t w1 = min(total, w0 + (uint32_t)kCap);
        __syncwarp();
        stage_runs<DP, false>(rt, nr, w0, w1, spts, nullptr, wpts, nullptr, lane);
        __syncwarp();
        int32_t c = 0, c2 = 0;
        for_window_runs<G>(rt, nr, u, w0, w1, [&](uint32_t i0, uint32_t i1, const uint32_t* cc) {
          const bool need = act && in_block<G>(c0, cc, R);
          if (!__any_sync(kFull, need)) return;
          if (need) pairs += i1 - i0;
          // a lane outside this cell's block compares against -1: never counts
          const float ti = need ? t_in : -1.f, to = need ? t_out : -1.f;
          const double dl = need ? dc2 : -1.0;
#pragma unroll 4
          for (uint32_t i = i0; i < i1; ++i) {
            const Pt<DP> x = window_pt<DP>(wpts, i);
            if constexpr (F64) {
              c += dist64<DP, ND>(me, x) <= dl;
            } else {
              const float s32 = dist32<DP, ND>(me, x);
              c += s32 <= ti;
              c2 += s32 <= to;
            }
          }
        });
        if constexpr (!F64) {
          if (__any_sync(kFull, c2 != c)) {
            const int2 r = band_recount<DP, G>(rt, nr, u, w0, w1, wpts, c0, act && c2 != c, R, me,
                                               t_in, t_out, dc2);
            c += r.x;
            band += r.y;
          }
        }
        count += c;
      }
      __syncwarp();
    });
    if (valid) {
      const uint32_t id = sid[p];
      rho_out[id] = count;
      skey[p] = order_key(count, id);
    }
  }
  for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(kFull, pairs, o);
  if (lane == 0 && pairs) atomicAdd(&ctr->pairs, pairs);
  if constexpr (!F64) {
    for (int o = 16; o > 0; o >>= 1) band += __shfl_xor_sync(kFull, band, o);
    if (lane == 0 && band) atomicAdd(&ctr->band_pairs, band);
  }
}

// ---------------------------------------------------------------------------
// Segment form: the 32 points of a chunk are split into segments of
// consecutive cells (super_segment: one cell, or several while the box around
// their blocks stays small); the warp looks the box's cells up once, stages
// their points in shared memory and every lane counts for one query of the
// segment: lane l answers query l % nqp on part l / nqp of the candidates, four
// at a time as broadcast reads (CandTile).  The box contains every query's
// block, so counting over all of it is exact.
// PREC 0 (float32 filter): two candidates are evaluated at once with packed add / mul / fma
// (the same rounding as the scalar sequence, so the certified band is
// unchanged); u = s - up(t_in) is negative (its sign bit) for a pair that
// counts, and as an unsigned word at most (t_out - up(t_in)) rounded for one in
// the band: one unsigned minimum per pair finds those, and a query that met one
// recounts its band pairs of the tile in binary64.  PREC 1: every pair in
// binary64.  PREC 2 (binary64 mode, int32 input): the same squared distance in
// 64-bit integers, exact as binary64 is there (below 2^53), off the binary64
// pipe, which issues one result per 16 clocks and warp.
// A set of few chunks is cut finer: `sub` warps share a chunk's queries, so that
// the chip has enough warps to hide the lookups (1e4 points in 2-D: 83 us with
// one warp per chunk; a replayed run 101 -> 70 us with this, the sort's small
// tiles and the merged set-up launches).
// What bounds it: issue slots (65% of them busy, 1.5 warps ready per cycle; DRAM 3%):
// 16 instructions per lane and scanned pair, of which the loop over candidates
// takes about 6 with every lane on a query, the rest the segment's set-up (cell
// lookups, staging) and lanes without one (profiles/, 4e6 points in 3-D, 1.11 ms).
// 1e7 points in 3-D: 3.60 ms with the candidates in registers across the lanes and
// one warp reduction per query pair and window of 128 candidates, 2.65 with
// queries across the lanes.
// M cutoffs of a sweep that share the block geometry `geo` (M = 1: one cutoff)
// are counted in one pass: the distances, lookups and staging are paid once,
// every cutoff adds its own compare and count.
template <int DP>
constexpr int seg_cap() { return DP == 8 ? 256 : 512; }

template <int DP, int G, int PREC, int M>
__global__ void __launch_bounds__(kThreads, (DP == 8 || PREC == 1) ? 5 : 7)
k_density_seg(const float* __restrict__ spts, const unsigned long long* __restrict__ scode,
              const uint32_t* __restrict__ sid, ClassView cv, const CutGeom* __restrict__ geo,
              const HashInfo* __restrict__ hi, const unsigned long long* __restrict__ hkeys,
              const uint2* __restrict__ hvals, MultiCut mc, unsigned long long* __restrict__ skey,
              Counters* ctr, int seg_cells, uint32_t skip_fill, uint32_t sub) {
  if (skip_fill && tensor_fill(cv.N, hi, skip_fill)) return;  // the tensor tiles' part
  constexpr int ND = real_dims<DP, G>();
  constexpr int kCap = seg_cap<DP>();
  __shared__ RunTable s_rt[kWarps];
  __shared__ CandTile<ND, kCap, false> s_tile[kWarps];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  RunTable& rt = s_rt[wib];
  CandTile<ND, kCap, false>& tile = s_tile[wib];
  const int S = cv.cls->S, ib = cv.cls->ib;
  const uint32_t hmask = hi->hmask;
  const uint32_t n = cv.N;

  unsigned long long band = 0, pairs = 0;
  const uint64_t work = (uint64_t)cv.nchunk * sub;
  for (uint64_t it = blockIdx.x * kWarps + wib; it < work; it += gridDim.x * kWarps) {
    uint32_t inst, p0, end;
    cv.chunk((uint32_t)(it / sub), inst, p0, end);
    p0 += (uint32_t)(it % sub) * (32u / sub);
    if (p0 >= end) continue;  // warp-uniform
    end = min(end, p0 + 32u / sub);
    const int k = geo[inst].k;
    const int R = geo[inst].R;
    const int shift = G * k;
    const int cmax = (1 << (cv.geom[inst].B - k)) - 1;
    f32x2 ntin2[M];
    uint32_t width[M];  // band: bits(u) <= width
    double dc2s[M];
    long long thr[M];  // PREC 2: s <= thr; real distances are at most 2^53, the padding's at least 2^57
#pragma unroll
    for (int c = 0; c < M; ++c) {
      const CutGeom& C = mc.cut[c][inst];
      const float up = next_up(C.t_in);
      dc2s[c] = C.dc2;
      thr[c] = PREC == 2 ? (long long)fmin(floor(C.dc2), 0x1p54) : 0ll;
      ntin2[c] = pack2(-up, -up);
      // s <= t_out implies fl(s - up) <= fl(t_out - up)
      width[c] = __float_as_uint(fmaxf(C.t_out - up, 0.f));
    }
    const unsigned long long hb = ib ? ((unsigned long long)inst << S) : 0ull;
    const uint32_t p = p0 + lane;
    const bool valid = p < end;
    const unsigned long long mycell = valid ? (key_code(scode[p], S, ib) >> shift) : ~0ull;
    const int nvalid = (int)min(32u, end - p0);
    int s = 0;
    while (s < nvalid) {
      Union<G> u;
      const int e = super_segment<G>(mycell, valid, s, nvalid, R, cmax, seg_cells, lane, u);  // queries s .. e-1
      const int nr = union_runs<G>(u, hkeys, hvals, hmask, hb, n, lane, rt);
      const uint32_t total = rt.pre[nr];
      const int nq = e - s;
      pairs += (unsigned long long)nq * total;
      const int lg = nq > 1 ? 32 - __clz(nq - 1) : 0;  // nqp = 1 << lg
      const int nqp = 1 << lg;
      const uint32_t part = (uint32_t)lane >> lg, step = 4u * (32u >> lg);
      const int mine = lane & (nqp - 1);
      const uint32_t pq = p0 + (uint32_t)(s + min(mine, nq - 1));
      const Pt<DP> me = load_pt<DP>(spts, pq);
      int32_t cnt[M];
#pragma unroll
      for (int c = 0; c < M; ++c) cnt[c] = 0;
      f32x2 q2[ND];
#pragma unroll
      for (int a = 0; a < ND; ++a) q2[a] = pack2(me.x[a], me.x[a]);
      for (uint32_t w0 = 0; w0 < total; w0 += kCap) {
        const uint32_t w1 = min(total, w0 + (uint32_t)kCap);
        __syncwarp();
        stage_tile<DP, ND, kCap, false>(rt, nr, w0, w1, spts, nullptr, tile, lane);
        const uint32_t tn = w1 - w0;
        if constexpr (PREC == 2) {
          // coordinates as integers (exact: |x| <= 2^24), not negated
          const uint32_t npad = (tn + 127u) & ~127u;
          for (uint32_t i = lane; i < npad; i += 32) {
#pragma unroll
            for (int a = 0; a < ND; ++a) tile.x[a][i] = __int_as_float(i < tn ? (int)-tile.x[a][i] : 1 << 29);
          }
          __syncwarp();
          int iq[ND];
#pragma unroll
          for (int a = 0; a < ND; ++a) iq[a] = (int)me.x[a];
          for (uint32_t i = 4u * part; i < tn; i += step) {
            long long d[4] = {0, 0, 0, 0};
#pragma unroll
            for (int a = 0; a < ND; ++a) {
              const int4 c4 = *reinterpret_cast<const int4*>(&tile.x[a][i]);
              const int t0 = iq[a] - c4.x, t1 = iq[a] - c4.y, t2 = iq[a] - c4.z, t3 = iq[a] - c4.w;
              d[0] += (long long)t0 * t0;
              d[1] += (long long)t1 * t1;
              d[2] += (long long)t2 * t2;
              d[3] += (long long)t3 * t3;
            }
#pragma unroll
            for (int v = 0; v < 4; ++v)
#pragma unroll
              for (int c = 0; c < M; ++c) cnt[c] += d[v] <= thr[c] ? 1 : 0;
          }
        } else if constexpr (PREC == 1) {
          for (uint32_t i = 4u * part; i < tn; i += step) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              // (padding is at distance +inf, which an infinite d_cut^2 would count)
              const bool real = i + v < tn;
              const double d = dist64<DP, ND>(me, tile_pt<DP>(tile, i + v));
#pragma unroll
              for (int c = 0; c < M; ++c) cnt[c] += real && d <= dc2s[c] ? 1 : 0;
            }
          }
        } else {
          uint32_t lowest[M];
#pragma unroll
          for (int c = 0; c < M; ++c) lowest[c] = 0xffffffffu;
#pragma unroll 2
          for (uint32_t i = 4u * part; i < tn; i += step) {
            f32x2 cc[2][ND];
            tile_quad(tile, i, cc);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const f32x2 sq = dist32x2<ND>(q2, cc[h]);
#pragma unroll
              for (int c = 0; c < M; ++c) {
                const f32x2 x = add2(sq, ntin2[c]);
                const uint32_t x0 = __float_as_uint(lo2(x)), x1 = __float_as_uint(hi2(x));
                cnt[c] += (int32_t)((x0 >> 31) + (x1 >> 31));
                lowest[c] = min(lowest[c], min(x0, x1));
              }
            }
          }
#pragma unroll
          for (int c = 0; c < M; ++c) {
            if (__any_sync(kFull, lowest[c] <= width[c])) {  // rare: band pairs of this tile
              const CutGeom& C = mc.cut[c][inst];
              const float t_in = C.t_in, t_out = C.t_out;
              const double dc2 = C.dc2;
              if (lowest[c] <= width[c]) {
#pragma unroll 1
                for (uint32_t i = 4u * part; i < tn; i += step) {
#pragma unroll 1
                  for (uint32_t v = i; v < i + 4u && v < tn; ++v) {
                    const Pt<DP> x = tile_pt<DP>(tile, v);
                    const float s32 = dist32<DP, ND>(me, x);
                    if (s32 > t_in && s32 <= t_out && mine < nq) {
                      ++band;
                      cnt[c] += dist64<DP, ND>(me, x) <= dc2 ? 1 : 0;
                    }
                  }
                }
              }
            }
          }
        }
      }
      // the parts of each query
#pragma unroll
      for (int c = 0; c < M; ++c)
        for (int o = nqp; o < 32; o <<= 1) cnt[c] += __shfl_xor_sync(kFull, cnt[c], o);
      if (lane < nq) {
        const uint32_t id = sid[pq];
#pragma unroll
        for (int c = 0; c < M; ++c) mc.rho[c][id] = cnt[c];
        if (skey) skey[pq] = order_key(cnt[0], id);
      }
      s = e;
    }
  }
  if (lane == 0 && pairs) atomicAdd(&ctr->pairs, pairs);
  if constexpr (PREC == 0) {
    for (int o = 16; o > 0; o >>= 1) band += __shfl_xor_sync(kFull, band, o);
    if (lane == 0 && band) atomicAdd(&ctr->band_pairs, band);
  }
}

// candidate slots per lane of the pair layout (its per-slot counts need
// registers of their own)
template <int DP>
constexpr int pairs_v() { return DP == 2 ? 8 : (DP == 4 ? 8 : 4); }

// Pair layout (symmetric): every unordered pair within d_cut is evaluated
// once and counted for both points.  Segments are the points of one cell in a
// chunk; the block's candidates are spread over the lanes, in registers, and the
// segment's queries taken two per pass.  A segment in cell A only takes the cells
// B of its block that follow A in Morton order, plus the points of A itself that
// follow the query in sorted order.  A query's count stays in a register and
// each candidate's in a register per slot; both go to a position-indexed
// counter with one atomic add per window (candidates) or per chunk (queries).
// cnt2 is the low 32-bit word of each sorted point's 64-bit order key slot
// (index 2p), zeroed before; k_pairs_finish turns it into rho and the key.
template <int DP, int G, bool F64>
__global__ void __launch_bounds__(kThreads, DP == 2 ? 5 : 4)
k_density_pairs(const float* __restrict__ spts, const unsigned long long* __restrict__ scode,
                ClassView cv, const CutGeom* __restrict__ cuts, const HashInfo* __restrict__ hi,
                const unsigned long long* __restrict__ hkeys, const uint2* __restrict__ hvals,
                uint32_t* __restrict__ cnt2, Counters* ctr) {
  constexpr int ND = real_dims<DP, G>();
  constexpr int V = pairs_v<DP>();
  constexpr uint32_t W = 32u * V;
  __shared__ RunTable s_rt[kWarps];
  __shared__ RunTable s_rt2[kWarps];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  RunTable& rt = s_rt[wib];
  RunTable& rt2 = s_rt2[wib];
  const int S = cv.cls->S, ib = cv.cls->ib;
  const uint32_t hmask = hi->hmask;
  const uint32_t n = cv.N;

  unsigned long long band = 0, pairs = 0;
  for (uint32_t ch = blockIdx.x * kWarps + wib; ch < cv.nchunk; ch += gridDim.x * kWarps) {
    uint32_t inst, p0, end;
    cv.chunk(ch, inst, p0, end);
    const CutGeom& C = cuts[inst];
    const int k = C.k;
    const int R = C.R;
    const int shift = G * k;
    const int cmax = (1 << (cv.geom[inst].B - k)) - 1;
    const double dc2 = C.dc2;
    const float t_in = C.t_in, t_out = C.t_out;
    const unsigned long long hb = ib ? ((unsigned long long)inst << S) : 0ull;
    const uint32_t p = p0 + lane;
    const bool valid = p < end;
    const unsigned long long mycell = valid ? (key_code(scode[p], S, ib) >> shift) : ~0ull;
    const int nvalid = (int)min(32u, end - p0);
    int32_t acc = valid ? 1 : 0;  // lane j: query p0 + j (itself, then its pairs)
    int s = 0;
    while (s < nvalid) {
      const unsigned long long cell = __shfl_sync(kFull, mycell, s);
      const int e = s + __popc(__ballot_sync(kFull, valid && mycell == cell));  // queries s .. e-1
      uint32_t c0[G];
      unmorton<G>(cell, c0);
      Union<G> u;
      block_union<G>(c0, R, cmax, u);
      const int nr = union_runs<G>(u, hkeys, hvals, hmask, hb, n, lane, rt);
      // OWN = false: the cells after A; OWN = true: A's points after the
      // segment's first query (a pair counts only if the candidate follows
      // the query)
      auto scan = [&](const RunTable& tab, int ntab, auto own_tag) {
        constexpr bool OWN = decltype(own_tag)::value;
        const uint32_t total = tab.pre[ntab];
        pairs += (unsigned long long)(e - s) * total;
        for (uint32_t w0 = 0; w0 < total; w0 += W) {
          Pt<DP> cand[V];
          load_window<DP, V>(tab, ntab, w0, total, spts, lane, cand);
          const int vn = (int)min((uint32_t)V, (total - w0 + 31u) / 32u);
          // OWN: one run, so slot v of this lane holds position pbase + 32 v
          const uint32_t pbase = OWN ? tab.start[0] + w0 + lane : 0u;
          // this lane's candidates' counts, two 16-bit halves per word
          uint32_t cc[(V + 1) / 2];
#pragma unroll
          for (int v = 0; v < (V + 1) / 2; ++v) cc[v] = 0u;
          for (int j = s; j < e; j += 2) {
            const bool two = j + 1 < e;
            const uint32_t qa = p0 + j, qb = p0 + (two ? j + 1 : j);
            const Pt<DP> xa = load_pt<DP>(spts, qa);
            const Pt<DP> xb = load_pt<DP>(spts, qb);
            int32_t cnt_a, cnt_b;
            if constexpr (F64) {
              unsigned c = 0;
#pragma unroll
              for (int v = 0; v < V; ++v) {
                if (v >= vn) break;
                const uint32_t pv = pbase + 32u * v;
                const bool ea = (!OWN || pv > qa) && dist64<DP, ND>(xa, cand[v]) <= dc2;
                const bool eb = two && (!OWN || pv > qb) && dist64<DP, ND>(xb, cand[v]) <= dc2;
                c += (ea ? 1u : 0u) + (eb ? 0x10000u : 0u);
                cc[v >> 1] += ((ea ? 1u : 0u) + (eb ? 1u : 0u)) << (16 * (v & 1));
              }
              c = __reduce_add_sync(kFull, c);
              cnt_a = (int32_t)(c & 0xffffu);
              cnt_b = (int32_t)(c >> 16);
            } else {
              unsigned ci = 0, co = 0;
#pragma unroll
              for (int v = 0; v < V; ++v) {
                if (v >= vn) break;
                const uint32_t pv = pbase + 32u * v;
                const float sa0 = dist32<DP, ND>(xa, cand[v]);
                const float sb0 = dist32<DP, ND>(xb, cand[v]);
                // a pair that does not count is NaN, which no threshold (+inf
                // among them) reaches
                const float sa = (!OWN || pv > qa) ? sa0 : NAN;
                const float sb = (two && (!OWN || pv > qb)) ? sb0 : NAN;
                const bool ia = sa <= t_in, ib2 = sb <= t_in;
                ci += (ia ? 1u : 0u) + (ib2 ? 0x10000u : 0u);
                co += (sa <= t_out ? 1u : 0u) + (sb <= t_out ? 0x10000u : 0u);
                cc[v >> 1] += ((ia ? 1u : 0u) + (ib2 ? 1u : 0u)) << (16 * (v & 1));
              }
              ci = __reduce_add_sync(kFull, ci);
              co = __reduce_add_sync(kFull, co);
              cnt_a = (int32_t)(ci & 0xffffu);
              cnt_b = (int32_t)(ci >> 16);
              if (co != ci) {  // band pairs: recount them in binary64
                unsigned in = 0, seen = 0;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                  if (v >= vn) break;
                  const uint32_t pv = pbase + 32u * v;
                  const float sa = (!OWN || pv > qa) ? dist32<DP, ND>(xa, cand[v]) : NAN;
                  const float sb = (two && (!OWN || pv > qb)) ? dist32<DP, ND>(xb, cand[v]) : NAN;
                  if (sa > t_in && sa <= t_out) {
                    ++seen;
                    const bool x = dist64<DP, ND>(xa, cand[v]) <= dc2;
                    in += x ? 1u : 0u;
                    cc[v >> 1] += (x ? 1u : 0u) << (16 * (v & 1));
                  }
                  if (sb > t_in && sb <= t_out) {
                    seen += 0x10000u;
                    const bool x = dist64<DP, ND>(xb, cand[v]) <= dc2;
                    in += x ? 0x10000u : 0u;
                    cc[v >> 1] += (x ? 1u : 0u) << (16 * (v & 1));
                  }
                }
                in = __reduce_add_sync(kFull, in);
                seen = __reduce_add_sync(kFull, seen);
                cnt_a += (int32_t)(in & 0xffffu);
                cnt_b += (int32_t)(in >> 16);
                if (lane == 0) band += (seen & 0xffffu) + (seen >> 16);
              }
            }
            if (lane == j) acc += cnt_a;
            if (two && lane == j + 1) acc += cnt_b;
          }
          // the candidates' counts, at their positions (found again in the run table)
          {
            const uint32_t e0 = w0 + lane;
            int lo = 0, hi = ntab - 1;
            while (lo < hi) {
              const int mid = (lo + hi + 1) >> 1;
              if (tab.pre[mid] <= e0) lo = mid;
              else hi = mid - 1;
            }
            int r = lo;
#pragma unroll
            for (int v = 0; v < V; ++v) {
              const uint32_t c = (cc[v >> 1] >> (16 * (v & 1))) & 0xffffu;
              const uint32_t ev = e0 + 32u * v;
              if (ev >= total) break;
              while (r + 1 < ntab && tab.pre[r + 1] <= ev) ++r;
              if (c) atomicAdd(&cnt2[2 * (size_t)(tab.start[r] + (ev - tab.pre[r]))], c);
            }
          }
        }
      };
      // the block's cells after A (Morton order)
      const int nb = filter_runs<G>(rt, nr, u, rt2, lane, [&](const uint32_t* cc) {
        return morton<G>(cc) > cell;
      });
      scan(rt2, nb, std::false_type());
      // A itself: its points after the segment's first query
      {
        const uint2 run = clip_run(hash_find(hkeys, hvals, hmask, hb | cell), n);
        const uint32_t a0 = max(run.x, p0 + (uint32_t)s + 1u);
        __syncwarp();
        if (lane == 0) {
          rt2.pre[0] = 0u;
          rt2.start[0] = a0;
          rt2.cell[0] = 0u;
          rt2.pre[1] = run.y > a0 ? run.y - a0 : 0u;
        }
        __syncwarp();
        scan(rt2, 1, std::true_type());
      }
      s = e;
    }
    if (valid) atomicAdd(&cnt2[2 * (size_t)p], (uint32_t)acc);
  }
  if (lane == 0 && pairs) atomicAdd(&ctr->pairs, pairs);
  if constexpr (!F64) {
    if (lane == 0 && band) atomicAdd(&ctr->band_pairs, band);
  }
}

// Counts of the pair layout -> rho (by output id) and the order keys.
__global__ void k_pairs_finish(const uint32_t* __restrict__ sid, uint32_t n, int32_t* __restrict__ rho_out,
                               unsigned long long* __restrict__ skey) {
  for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const uint32_t c = reinterpret_cast<const uint32_t*>(skey)[2 * (size_t)p];
    const uint32_t id = sid[p];
    rho_out[id] = (int32_t)c;
    skey[p] = order_key((int32_t)c, id);
  }
}

__global__ void k_keys_from_rho(const int32_t* __restrict__ rho, const uint32_t* __restrict__ sid,
                                uint32_t n, unsigned long long* __restrict__ skey) {
  for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const uint32_t id = sid[p];
    skey[p] = order_key(rho[id], id);
  }
}

inline unsigned grid_for(uint64_t items, int per_block, unsigned cap) {
  uint64_t b = (items + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (unsigned)b;
}

// Segment densities of the cutoffs of mc (prec: 0 float32 filter, 1 binary64,
// 2 64-bit integers).
template <int DP, int G>
void density_multi_dg(int prec, const float* spts, const unsigned long long* scode, const uint32_t* sid,
                      const ClassView& cv, const CutGeom* geo, const HashInfo* hi, const unsigned long long* hkeys,
                      const uint2* hvals, const MultiCut& mc, unsigned long long* skey, Counters* ctr, int seg_cells,
                      uint32_t skip_fill, cudaStream_t st) {
  // at least 8 warps per SM's scheduler, down to 4 queries a warp
  uint32_t sub = 1;
  while (sub < 8u && (uint64_t)cv.nchunk * sub < (uint64_t)sm_count() * 32u) sub *= 2;
  const unsigned grid = grid_for((uint64_t)cv.nchunk * sub, kWarps, sm_count() * 64u);
  auto go = [&](auto kern) {
    kern<<<grid, kThreads, 0, st>>>(spts, scode, sid, cv, geo, hi, hkeys, hvals, mc, skey, ctr, seg_cells, skip_fill,
                                    sub);
  };
  auto cuts = [&](auto p) {
    constexpr int P = decltype(p)::value;
    if (mc.m == 1) go(k_density_seg<DP, G, P, 1>);
    else if (mc.m == 2) go(k_density_seg<DP, G, P, 2>);
    else if (mc.m == 3) go(k_density_seg<DP, G, P, 3>);
    else go(k_density_seg<DP, G, P, 4>);
  };
  if (prec == 0) cuts(std::integral_constant<int, 0>{});
  else if (prec == 1) cuts(std::integral_constant<int, 1>{});
  else cuts(std::integral_constant<int, 2>{});
  count_launches(1);
}

template <int DP, int G>
void density_dg(int prec, int layout, const float* spts, const unsigned long long* scode,
                const uint32_t* sid, const ClassView& cv, const CutGeom* cuts, const HashInfo* hi,
                const unsigned long long* hkeys, const uint2* hvals, int32_t* rho_out,
                unsigned long long* skey, Counters* ctr, int seg_cells, uint32_t skip_fill, cudaStream_t st) {
  const unsigned grid = grid_for(cv.nchunk, kWarps, sm_count() * 64u);
  const bool fp64 = prec != 0;
  if (layout == kLayoutPairs) {
    cudaMemsetAsync(skey, 0, sizeof(unsigned long long) * cv.N, st);
    uint32_t* cnt2 = reinterpret_cast<uint32_t*>(skey);
    if (fp64)
      k_density_pairs<DP, G, true><<<grid, kThreads, 0, st>>>(spts, scode, cv, cuts, hi, hkeys, hvals,
                                                              cnt2, ctr);
    else
      k_density_pairs<DP, G, false><<<grid, kThreads, 0, st>>>(spts, scode, cv, cuts, hi, hkeys, hvals,
                                                               cnt2, ctr);
    k_pairs_finish<<<grid_for(cv.N, 256, sm_count() * 16u), 256, 0, st>>>(sid, cv.N, rho_out, skey);
    count_launches(1);
  } else if (layout == kLayoutSegment) {
    MultiCut mc;
    mc.m = 1;
    mc.cut[0] = cuts;
    mc.rho[0] = rho_out;
    density_multi_dg<DP, G>(prec, spts, scode, sid, cv, cuts, hi, hkeys, hvals, mc, skey, ctr, seg_cells, skip_fill,
                            st);
    return;
  } else {
    if (fp64)
      k_density<DP, G, true><<<grid, kThreads, 0, st>>>(spts, scode, sid, cv, cuts, hi, hkeys, hvals,
                                                        rho_out, skey, ctr);
    else
      k_density<DP, G, false><<<grid, kThreads, 0, st>>>(spts, scode, sid, cv, cuts, hi, hkeys,
                                                         hvals, rho_out, skey, ctr);
  }
  count_launches(1);
}

}  // namespace

void launch_density_multi(int dp, int g, int d, int prec, const float* spts, const unsigned long long* scode,
                          const uint32_t* sid, const ClassView& cv, const CutGeom* geo, HashInfo* hi,
                          const unsigned long long* hkeys, const uint2* hvals, uint4* pieces, const MultiCut& mc,
                          Counters* ctr, cudaStream_t st, int seg_cells, uint32_t min_fill) {
  if (cv.N == 0) return;
  uint32_t skip_fill = 0;
  if (dp == 8 && prec == 0) {
    launch_density_tc(d, spts, scode, sid, cv, geo, hi, hkeys, hvals, pieces, mc, nullptr, ctr, min_fill, st);
    if (min_fill == 0) return;
    skip_fill = min_fill;
  }
  auto go = [&](auto run) { run(prec, spts, scode, sid, cv, geo, hi, hkeys, hvals, mc, nullptr, ctr, seg_cells, skip_fill, st); };
  if (g == 1) go(density_multi_dg<2, 1>);
  else if (g == 2) go(density_multi_dg<2, 2>);
  else if (g == 3) go(density_multi_dg<4, 3>);
  else if (dp == 4) go(density_multi_dg<4, 4>);
  else go(density_multi_dg<8, 4>);
}

void launch_density(int dp, int g, int d, int prec, int layout, const float* spts,
                    const unsigned long long* scode, const uint32_t* sid, const ClassView& cv,
                    const CutGeom* cuts, HashInfo* hi, const unsigned long long* hkeys,
                    const uint2* hvals, uint4* pieces, int32_t* rho_out,
                    unsigned long long* skey, Counters* ctr, cudaStream_t st, int seg_cells, uint32_t min_fill) {
  if (cv.N == 0) return;
  uint32_t skip_fill = 0;
  if (layout == kLayoutTensor) {
    if (dp == 8 && prec == 0 && pieces) {
      MultiCut mc;
      mc.m = 1;
      mc.cut[0] = cuts;
      mc.rho[0] = rho_out;
      launch_density_tc(d, spts, scode, sid, cv, cuts, hi, hkeys, hvals, pieces, mc, skey, ctr, min_fill, st);
      if (min_fill == 0) return;
      skip_fill = min_fill;
    }
    layout = kLayoutSegment;
  }
  // float32 points in binary64: the segments' work with every pair once
  if (layout == kLayoutSegment && prec == 1 && cv.nchunk >= kBinary64Pairs) layout = kLayoutPairs;
  if (layout == kLayoutCell) {
    launch_density_cell(dp, g, prec != 0, spts, scode, sid, cv, cuts, hi, hkeys, hvals, rho_out, skey, ctr,
                        st);
    return;
  }
  if (g == 1) density_dg<2, 1>(prec, layout, spts, scode, sid, cv, cuts, hi, hkeys, hvals, rho_out, skey, ctr, seg_cells, skip_fill, st);
  else if (g == 2) density_dg<2, 2>(prec, layout, spts, scode, sid, cv, cuts, hi, hkeys, hvals, rho_out, skey, ctr, seg_cells, skip_fill, st);
  else if (g == 3) density_dg<4, 3>(prec, layout, spts, scode, sid, cv, cuts, hi, hkeys, hvals, rho_out, skey, ctr, seg_cells, skip_fill, st);
  else if (dp == 4) density_dg<4, 4>(prec, layout, spts, scode, sid, cv, cuts, hi, hkeys, hvals, rho_out, skey, ctr, seg_cells, skip_fill, st);
  else density_dg<8, 4>(prec, layout, spts, scode, sid, cv, cuts, hi, hkeys, hvals, rho_out, skey, ctr, seg_cells, skip_fill, st);
}

void launch_keys_from_rho(const int32_t* rho, const uint32_t* sid, uint32_t n,
                          unsigned long long* skey, cudaStream_t st) {
  if (n == 0) return;
  k_keys_from_rho<<<grid_for(n, 256, sm_count() * 16u), 256, 0, st>>>(rho, sid, n, skey);
  count_launches(1);
}

}  // namespace dpc

// small.cu -- rho, lambda, delta of small instances from all pairs, and the
// labels of small instances in one launch.
//
// Below a few thousand points the grid pipeline (binning, sort, cell hash,
// tree) is a chain of about forty launches of two to eight microseconds each,
// while all n^2 pairs are a few million distances: one density launch and one
// dependent launch read the caller's coordinates directly and need no index at
// all.  What bounds them is the launch itself up to about 2,000 points, then
// the float32 issue rate.
//
// A CTA owns Q consecutive queries of one instance (uniform, in registers) and
// its four warps stride over the instance's points, two candidates per lane in
// packed float32 pairs; the counts (or the nearest higher candidates) are
// reduced once per query.  FP32_CERT filters in float32 with the bands of
// CutHost and settles every pair inside a band in binary64; FP64 evaluates
// every pair in binary64.  Both give the binary64 definition exactly.
#include <cmath>

#include "internal.h"

namespace dpc {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
constexpr int kStep = 64 * kWarps;  // candidates a CTA takes per iteration

// Q queries per CTA: the candidates' loads and conversions are shared by them.
template <int D>
constexpr int small_q() { return D <= 2 ? 8 : 4; }

// Coordinates of point `id` as the float32 values the whole library works on
// (int32 inputs are exact by the range check).
template <int D>
__device__ __forceinline__ void load_row(const void* __restrict__ pts, int dtype, uint64_t coord, uint32_t id,
                                         float* x) {
  const size_t e = coord + (size_t)id * D;
  if (dtype == 0) {
#pragma unroll
    for (int a = 0; a < D; ++a) x[a] = (float)__ldg((const int32_t*)pts + e + a);
  } else {
#pragma unroll
    for (int a = 0; a < D; ++a) x[a] = __ldg((const float*)pts + e + a);
  }
}

// The range check of the binning (dpc.h), on the caller's values.
template <int D>
__device__ __forceinline__ bool bad_row(const void* __restrict__ pts, int dtype, uint64_t coord, uint32_t id) {
  const size_t e = coord + (size_t)id * D;
  bool bad = false;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    if (dtype == 0) {
      const int32_t v = __ldg((const int32_t*)pts + e + a);
      bad |= (v > (1 << 24)) | (v < -(1 << 24));
    } else {
      bad |= !(fabsf(__ldg((const float*)pts + e + a)) <= 1.152921504606846976e18f);  // 2^60; NaN
    }
  }
  return bad;
}

template <int D>
__device__ __forceinline__ float row_dist32(const float* a, const float* b) {
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const float t = a[k] - b[k];
    s = fmaf(t, t, s);
  }
  return s;
}

template <int D>
__device__ __forceinline__ double row_dist64(const float* a, const float* b) {
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const double t = __dsub_rn((double)a[k], (double)b[k]);
    s = __dadd_rn(s, __dmul_rn(t, t));
  }
  return s;
}

// The Q queries of group g: instance, first local id, how many.
template <int Q>
__device__ __forceinline__ InstDev group_of(const ClassView& cv, uint32_t g, uint32_t& inst, uint32_t& q0, int& nq) {
  uint32_t p0, end;
  cv.chunk(g / (32 / Q), inst, p0, end);
  const InstDev I = cv.instance(inst);
  p0 += (g % (32 / Q)) * Q;
  q0 = p0 - I.start;
  nq = p0 < end ? (int)min((uint32_t)Q, end - p0) : 0;
  return I;
}

// Cutoff k of instance i: uploaded tables [inst][ncut], or kernel arguments.
__device__ __forceinline__ const CutHost& small_cut(const CutHost* __restrict__ hc, const CutArgs& args, int ncut,
                                                    uint32_t i, int k) {
  return hc ? hc[(size_t)i * ncut + k] : args.h[k];
}

// Densities of cutoffs cut0 .. (grid y).
template <int D, bool F64>
__global__ void __launch_bounds__(kThreads)
k_small_density(const void* __restrict__ pts, int dtype, ClassView cv, const CutHost* __restrict__ hc,
                const __grid_constant__ CutArgs args, int ncut, int cut0, int32_t* __restrict__ rho, uint64_t rho_stride,
                uint32_t ngroup, Counters* ctr, int* status) {
  constexpr int Q = small_q<D>();
  __shared__ uint32_t s_cnt[kWarps][Q];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cut = cut0 + (int)blockIdx.y;
  for (uint32_t g = blockIdx.x; g < ngroup; g += gridDim.x) {
    uint32_t inst, q0;
    int nq;
    const InstDev I = group_of<Q>(cv, g, inst, q0, nq);
    if (nq == 0) continue;  // uniform over the CTA
    const CutHost C = small_cut(hc, args, ncut, inst, cut);
    if (cut == 0 && (int)threadIdx.x < nq && bad_row<D>(pts, dtype, I.coord, q0 + threadIdx.x))
      set_status(status, kStatusBadCoord);
    if (threadIdx.x == 0 && q0 == 0) atomicAdd(&ctr->pairs, (unsigned long long)I.n * I.n);
    float xq[Q][D];
#pragma unroll
    for (int j = 0; j < Q; ++j) load_row<D>(pts, dtype, I.coord, q0 + (uint32_t)min(j, nq - 1), xq[j]);
    uint32_t cnt[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) cnt[j] = 0u;
    if constexpr (F64) {
      for (uint32_t e = threadIdx.x; e < I.n; e += kThreads) {
        float x[D];
        load_row<D>(pts, dtype, I.coord, e, x);
#pragma unroll
        for (int j = 0; j < Q; ++j) cnt[j] += row_dist64<D>(xq[j], x) <= C.dc2 ? 1u : 0u;
      }
    } else {
      const BandBits bb = band_bits(C.t_in, C.t_out);
      const f32x2 ntin2 = pack2(-next_up(C.t_in), -next_up(C.t_in));
      uint32_t mband = 0xffffffffu;
      f32x2 q2[Q][D];
#pragma unroll
      for (int j = 0; j < Q; ++j)
#pragma unroll
        for (int a = 0; a < D; ++a) q2[j][a] = pack2(xq[j][a], xq[j][a]);
#pragma unroll 2
      for (uint32_t e0 = warp * 64; e0 < I.n; e0 += kStep) {
        const uint32_t ea = e0 + lane, eb = ea + 32u;
        float xa[D], xb[D];
#pragma unroll
        for (int a = 0; a < D; ++a) xa[a] = xb[a] = -INFINITY;
        if (ea < I.n) load_row<D>(pts, dtype, I.coord, ea, xa);
        if (eb < I.n) load_row<D>(pts, dtype, I.coord, eb, xb);
        f32x2 nc[D];  // negated; +inf past the end: distance +inf, never counted, never in the band
#pragma unroll
        for (int a = 0; a < D; ++a) nc[a] = pack2(-xa[a], -xb[a]);
#pragma unroll
        for (int j = 0; j < Q; ++j) {
          const f32x2 s = dist32x2<D>(q2[j], nc);
          cnt[j] += sign_count2(add2(s, ntin2));
          mband = min(mband, band_min2(s, bb.lo));
        }
      }
      // a band pair anywhere: this warp's candidates again, every band pair in
      // binary64
      if (__any_sync(kFull, mband < bb.width)) {
        uint32_t seen = 0;
        for (uint32_t e0 = warp * 64; e0 < I.n; e0 += kStep) {
#pragma unroll 1
          for (uint32_t e = e0 + lane; e < e0 + 64u && e < I.n; e += 32u) {
            float x[D];
            load_row<D>(pts, dtype, I.coord, e, x);
            if constexpr (D == 1) {
              // a 1-D binary64 distance is so short that it would run under a
              // predicate for every pair, through the binary64 pipe (13,000 integer
              // points with a cutoff that many pairs meet: 1.32 ms, 0.12 with the
              // float32 tests first and a loop over the pairs that need it)
              uint32_t bm = 0;
#pragma unroll
              for (int j = 0; j < Q; ++j) {
                const float s = row_dist32<D>(xq[j], x);
                bm |= (s > C.t_in && s <= C.t_out && j < nq) ? 1u << j : 0u;
              }
              seen += __popc(bm);
#pragma unroll 1
              while (bm) {
                const int j = __ffs((int)bm) - 1;
                bm &= bm - 1u;
                float y[D];
                load_row<D>(pts, dtype, I.coord, q0 + (uint32_t)j, y);
                const uint32_t in = row_dist64<D>(y, x) <= C.dc2 ? 1u : 0u;
#pragma unroll
                for (int k = 0; k < Q; ++k) cnt[k] += k == j ? in : 0u;
              }
            } else {
#pragma unroll
              for (int j = 0; j < Q; ++j) {
                const float s = row_dist32<D>(xq[j], x);
                if (s > C.t_in && s <= C.t_out && j < nq) {
                  ++seen;
                  cnt[j] += row_dist64<D>(xq[j], x) <= C.dc2 ? 1u : 0u;
                }
              }
            }
          }
        }
        seen = __reduce_add_sync(kFull, seen);
        if (lane == 0 && seen) atomicAdd(&ctr->band_pairs, (unsigned long long)seen);
      }
    }
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      const uint32_t c = __reduce_add_sync(kFull, cnt[j]);
      if (lane == 0) s_cnt[warp][j] = c;
    }
    __syncthreads();
    if ((int)threadIdx.x < nq) {
      uint32_t c = 0;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) c += s_cnt[w][threadIdx.x];
      rho[(size_t)cut * rho_stride + I.out + q0 + threadIdx.x] = (int32_t)c;
    }
    __syncthreads();
  }
}

// Dependent points of one cutoff from its densities.  Per query every lane
// keeps the smallest and second smallest float32 distance among its higher
// candidates; when a second candidate lies within the error band of the
// smallest, the CTA ranks the band in binary64.
template <int D, bool F64>
__global__ void __launch_bounds__(kThreads)
k_small_dependent(const void* __restrict__ pts, int dtype, ClassView cv, const CutHost* __restrict__ hc,
                  const __grid_constant__ CutArgs args, int ncut, int cut, int32_t rho_skip,
                  const int32_t* __restrict__ rho, int32_t* __restrict__ lambda, double* __restrict__ delta,
                  uint32_t ngroup, Counters* ctr, int* status) {
  constexpr int Q = 4;
  __shared__ double s_d[kWarps][Q];
  __shared__ float s_1[kWarps][Q], s_2[kWarps][Q];
  __shared__ uint32_t s_j[kWarps][Q];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t g = blockIdx.x; g < ngroup; g += gridDim.x) {
    uint32_t inst, q0;
    int nq;
    const InstDev I = group_of<Q>(cv, g, inst, q0, nq);
    if (nq == 0) continue;
    const CutHost C = small_cut(hc, args, ncut, inst, cut);
    const int32_t skip = max(rho_skip, C.skip);
    const int32_t* __restrict__ r = rho + I.out;
    if (cut == 0 && (int)threadIdx.x < nq && bad_row<D>(pts, dtype, I.coord, q0 + threadIdx.x))
      set_status(status, kStatusBadCoord);
    float xq[Q][D];
    int32_t rq[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      const uint32_t id = q0 + (uint32_t)min(j, nq - 1);
      load_row<D>(pts, dtype, I.coord, id, xq[j]);
      rq[j] = __ldg(r + id);
    }
    // candidate e of density re is higher than query j (order_key: densities as
    // unsigned words, ties to the smaller id)
    auto higher = [&](int32_t re, uint32_t e, int j) {
      return (uint32_t)re > (uint32_t)rq[j] || (re == rq[j] && e < q0 + (uint32_t)j);
    };
    // binary64 ranking of the candidates with s32 <= bnd, over the CTA
    auto rank64 = [&](int j, float bnd, bool all) {
      double bs = INFINITY;
      uint32_t bj = 0xffffffffu;
      for (uint32_t e = threadIdx.x; e < I.n; e += kThreads) {
        if (!higher(__ldg(r + e), e, j)) continue;
        float x[D];
        load_row<D>(pts, dtype, I.coord, e, x);
        if (!all && !(row_dist32<D>(xq[j], x) <= bnd)) continue;
        const double s = row_dist64<D>(xq[j], x);
        if (s < bs || (s == bs && e < bj)) {
          bs = s;
          bj = e;
        }
      }
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) {
        const double os = __shfl_xor_sync(kFull, bs, m);
        const uint32_t oj = __shfl_xor_sync(kFull, bj, m);
        if (os < bs || (os == bs && oj < bj)) {
          bs = os;
          bj = oj;
        }
      }
      if (lane == 0) {
        s_d[warp][j] = bs;
        s_j[warp][j] = bj;
      }
    };
    // the four warps' results of query j: (s64, id)
    auto finish = [&](int j) {
      double bs = s_d[0][j];
      uint32_t bj = s_j[0][j];
#pragma unroll
      for (int w = 1; w < kWarps; ++w)
        if (s_d[w][j] < bs || (s_d[w][j] == bs && s_j[w][j] < bj)) {
          bs = s_d[w][j];
          bj = s_j[w][j];
        }
      const uint64_t o = I.out + q0 + (uint32_t)j;
      lambda[o] = bj == 0xffffffffu ? -1 : (int32_t)bj;
      delta[o] = bj == 0xffffffffu ? INFINITY : sqrt(bs);
    };
    if constexpr (F64) {
#pragma unroll
      for (int j = 0; j < Q; ++j)
        if (j < nq && rq[j] >= skip) rank64(j, 0.f, true);
      __syncthreads();
      if ((int)threadIdx.x < nq) {
#pragma unroll
        for (int j = 0; j < Q; ++j)
          if ((int)threadIdx.x == j) {
            if (rq[j] >= skip) {
              finish(j);
            } else {
              const uint64_t o = I.out + q0 + (uint32_t)j;
              lambda[o] = -1;
              delta[o] = __longlong_as_double(0x7ff8000000000000ll);  // NaN: skipped
            }
          }
      }
      __syncthreads();
    } else {
      float m1[Q], m2[Q];
      uint32_t mj[Q];
      f32x2 q2[Q][D];
#pragma unroll
      for (int j = 0; j < Q; ++j) {
        m1[j] = m2[j] = INFINITY;
        mj[j] = 0xffffffffu;
#pragma unroll
        for (int a = 0; a < D; ++a) q2[j][a] = pack2(xq[j][a], xq[j][a]);
      }
#pragma unroll 2
      for (uint32_t e0 = warp * 64; e0 < I.n; e0 += kStep) {
        const uint32_t ea = e0 + lane, eb = ea + 32u;
        float xa[D], xb[D];
#pragma unroll
        for (int a = 0; a < D; ++a) xa[a] = xb[a] = -INFINITY;
        int32_t ra = 0, rb = 0;  // past the end: the distance is +inf whatever the order says
        if (ea < I.n) {
          load_row<D>(pts, dtype, I.coord, ea, xa);
          ra = __ldg(r + ea);
        }
        if (eb < I.n) {
          load_row<D>(pts, dtype, I.coord, eb, xb);
          rb = __ldg(r + eb);
        }
        f32x2 nc[D];
#pragma unroll
        for (int a = 0; a < D; ++a) nc[a] = pack2(-xa[a], -xb[a]);
#pragma unroll
        for (int j = 0; j < Q; ++j) {
          const f32x2 s = dist32x2<D>(q2[j], nc);
          const float sa = higher(ra, ea, j) ? lo2(s) : INFINITY;
          const float sb = higher(rb, eb, j) ? hi2(s) : INFINITY;
          m2[j] = fminf(m2[j], fmaxf(m1[j], sa));
          mj[j] = sa < m1[j] ? ea : mj[j];
          m1[j] = fminf(m1[j], sa);
          m2[j] = fminf(m2[j], fmaxf(m1[j], sb));
          mj[j] = sb < m1[j] ? eb : mj[j];
          m1[j] = fminf(m1[j], sb);
        }
      }
#pragma unroll
      for (int j = 0; j < Q; ++j) {
        // the warp's smallest, an id at it, and the second smallest
        const float g1 = __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(m1[j])));
        const unsigned at = __ballot_sync(kFull, m1[j] == g1);
        const float g2 = __popc(at) > 1 ? g1 : __uint_as_float(__reduce_min_sync(
                                                   kFull, __float_as_uint(m1[j] == g1 ? m2[j] : m1[j])));
        const uint32_t gj = __shfl_sync(kFull, mj[j], __ffs((int)at) - 1);
        if (lane == 0) {
          s_1[warp][j] = g1;
          s_2[warp][j] = g2;
          s_j[warp][j] = gj;
        }
      }
      __syncthreads();
      unsigned amb = 0;  // uniform: queries ranked in binary64
#pragma unroll
      for (int j = 0; j < Q; ++j) {
        if (j >= nq) continue;
        float b1 = s_1[0][j], b2 = s_2[0][j];
        uint32_t bj = s_j[0][j];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) {
          const float w1 = s_1[w][j];
          b2 = fminf(fminf(b2, s_2[w][j]), fmaxf(b1, w1));
          bj = w1 < b1 ? s_j[w][j] : bj;
          b1 = fminf(b1, w1);
        }
        const bool skipped = rq[j] < skip;
        const bool none = !(b1 < INFINITY);
        const float bnd = __fadd_ru(__fmul_ru(b1, C.band_mul), C.band_add);
        const bool close = !skipped && !none && b2 <= bnd;
        if (close) amb |= 1u << j;
        if ((int)threadIdx.x == j && !close) {
          const uint64_t o = I.out + q0 + (uint32_t)j;
          if (skipped || none) {
            lambda[o] = -1;
            delta[o] = skipped ? __longlong_as_double(0x7ff8000000000000ll) : (double)INFINITY;
          } else {
            float x[D];
            load_row<D>(pts, dtype, I.coord, bj, x);
            lambda[o] = (int32_t)bj;
            delta[o] = sqrt(row_dist64<D>(xq[j], x));
          }
        }
        m1[j] = bnd;
      }
      __syncthreads();
      if (amb) {
#pragma unroll
        for (int j = 0; j < Q; ++j)
          if ((amb >> j) & 1u) rank64(j, m1[j], false);
        __syncthreads();
        if (threadIdx.x == 0) {
          atomicAdd(&ctr->exact_rescans, (unsigned long long)__popc(amb));
#pragma unroll
          for (int j = 0; j < Q; ++j)
            if ((amb >> j) & 1u) finish(j);
        }
        __syncthreads();
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Labels of instances that fit one CTA's shared memory: the pointers of one
// instance in shared memory, doubled until every one is at its root, one
// launch for the class (labels.cu needs init, log rounds, local and check
// launches).  The rules are labels.cu's; a pointer never becomes its own
// root by jumping, so the points of a cycle stay open and are reported.

constexpr int kLabelThreads = 1024;

__global__ void __launch_bounds__(kLabelThreads)
k_small_labels(const int32_t* __restrict__ rho, const int32_t* __restrict__ lambda, const double* __restrict__ delta,
               ClassView cv, const LabelParams* __restrict__ params, LabelParams one, int32_t* __restrict__ label,
               int* status) {
  extern __shared__ int32_t s_par[];
  for (uint32_t inst = blockIdx.x; inst < cv.ninst; inst += gridDim.x) {
    const InstDev I = cv.instance(inst);
    const LabelParams P = params ? params[inst] : one;
    const int32_t n = (int32_t)I.n;
#pragma unroll 4
    for (int32_t i = threadIdx.x; i < n; i += kLabelThreads) {
      const int32_t r = __ldg(rho + I.out + i), l = __ldg(lambda + I.out + i);
      const double dl = __ldg(delta + I.out + i);
      int32_t v;
      if (r < P.rho_noise) v = -1;                                                 // Definition 4
      else if (l < 0 || (r >= P.rho_min && dl >= P.delta_min)) v = i;  // Definition 5
      else v = l < n ? l : -1;
      s_par[i] = v;
    }
    int open = 1;
    // every round at least doubles the distance covered: 32 rounds are more
    // than any forest needs
    for (int round = 0; round < 32 && open; ++round) {
      __syncthreads();
      int mine = 0;
      for (int32_t i = threadIdx.x; i < n; i += kLabelThreads) {
        const volatile int32_t* par = s_par;
        int32_t p = par[i];
        if (p < 0 || p == i) continue;
        bool root = false;
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
          const int32_t pp = par[p];
          if (pp == p || pp < 0) {
            if (pp < 0) p = pp;
            root = true;
            break;
          }
          if (pp == i) break;  // back at itself: a cycle
          p = pp;
        }
        s_par[i] = p;
        if (!root) mine = 1;
      }
      open = __syncthreads_or(mine);
    }
    if (open && threadIdx.x == 0) set_status(status, kStatusCycle);
    for (int32_t i = threadIdx.x; i < n; i += kLabelThreads) label[I.out + i] = s_par[i];
    __syncthreads();
  }
}

template <int D>
void density_d(bool fp64, const void* pts, int dtype, const ClassView& cv, const CutHost* hc, const CutArgs& a,
               int ncut, int32_t* rho, uint64_t stride, Counters* ctr, int* status, cudaStream_t st) {
  const uint64_t ng = (uint64_t)cv.nchunk * (32 / small_q<D>());
  // a launch takes at most 65,535 cutoffs in its grid's second dimension
  for (int c0 = 0; c0 < ncut; c0 += 65535) {
    const dim3 grid((unsigned)(ng < (1u << 20) ? ng : (1u << 20)), (unsigned)(ncut - c0 < 65535 ? ncut - c0 : 65535));
    if (fp64)
      k_small_density<D, true><<<grid, kThreads, 0, st>>>(pts, dtype, cv, hc, a, ncut, c0, rho, stride, (uint32_t)ng,
                                                         ctr, status);
    else
      k_small_density<D, false><<<grid, kThreads, 0, st>>>(pts, dtype, cv, hc, a, ncut, c0, rho, stride, (uint32_t)ng,
                                                          ctr, status);
    count_launches(1);
  }
}

template <int D>
void dependent_d(bool fp64, const void* pts, int dtype, const ClassView& cv, const CutHost* hc, const CutArgs& a,
                 int ncut, int cut, int32_t rho_skip, const int32_t* rho, int32_t* lambda, double* delta,
                 Counters* ctr, int* status, cudaStream_t st) {
  const uint64_t ng = (uint64_t)cv.nchunk * 8u;
  const unsigned grid = (unsigned)(ng < (1u << 20) ? ng : (1u << 20));
  if (fp64)
    k_small_dependent<D, true><<<grid, kThreads, 0, st>>>(pts, dtype, cv, hc, a, ncut, cut, rho_skip, rho, lambda,
                                                         delta, (uint32_t)ng, ctr, status);
  else
    k_small_dependent<D, false><<<grid, kThreads, 0, st>>>(pts, dtype, cv, hc, a, ncut, cut, rho_skip, rho, lambda,
                                                          delta, (uint32_t)ng, ctr, status);
}

CutArgs pack_args(const CutHost* hc_dev, const CutHost* hc_host, int ncut) {
  CutArgs a;
  if (!hc_dev)
    for (int c = 0; c < ncut && c < kCutChunk; ++c) a.h[c] = hc_host[c];
  return a;
}

}  // namespace

void launch_small_density(int d, bool fp64, const void* pts, int dtype, const ClassView& cv, const CutHost* hc_dev,
                          const CutHost* hc_host, int ncut, int32_t* rho, uint64_t rho_stride, Counters* ctr,
                          int* status, cudaStream_t st) {
  if (cv.N == 0) return;
  const CutArgs a = pack_args(hc_dev, hc_host, ncut);
  switch (d) {
    case 1: density_d<1>(fp64, pts, dtype, cv, hc_dev, a, ncut, rho, rho_stride, ctr, status, st); break;
    case 2: density_d<2>(fp64, pts, dtype, cv, hc_dev, a, ncut, rho, rho_stride, ctr, status, st); break;
    case 3: density_d<3>(fp64, pts, dtype, cv, hc_dev, a, ncut, rho, rho_stride, ctr, status, st); break;
    case 4: density_d<4>(fp64, pts, dtype, cv, hc_dev, a, ncut, rho, rho_stride, ctr, status, st); break;
    case 5: density_d<5>(fp64, pts, dtype, cv, hc_dev, a, ncut, rho, rho_stride, ctr, status, st); break;
    case 6: density_d<6>(fp64, pts, dtype, cv, hc_dev, a, ncut, rho, rho_stride, ctr, status, st); break;
    case 7: density_d<7>(fp64, pts, dtype, cv, hc_dev, a, ncut, rho, rho_stride, ctr, status, st); break;
    default: density_d<8>(fp64, pts, dtype, cv, hc_dev, a, ncut, rho, rho_stride, ctr, status, st); break;
  }
}

void launch_small_dependent(int d, bool fp64, const void* pts, int dtype, const ClassView& cv,
                            const CutHost* hc_dev, const CutHost* hc_host, int ncut, int cut, int32_t rho_skip,
                            const int32_t* rho, int32_t* lambda, double* delta, Counters* ctr, int* status,
                            cudaStream_t st) {
  if (cv.N == 0) return;
  const CutArgs a = pack_args(hc_dev, hc_host, ncut);
  switch (d) {
    case 1: dependent_d<1>(fp64, pts, dtype, cv, hc_dev, a, ncut, cut, rho_skip, rho, lambda, delta, ctr, status, st); break;
    case 2: dependent_d<2>(fp64, pts, dtype, cv, hc_dev, a, ncut, cut, rho_skip, rho, lambda, delta, ctr, status, st); break;
    case 3: dependent_d<3>(fp64, pts, dtype, cv, hc_dev, a, ncut, cut, rho_skip, rho, lambda, delta, ctr, status, st); break;
    case 4: dependent_d<4>(fp64, pts, dtype, cv, hc_dev, a, ncut, cut, rho_skip, rho, lambda, delta, ctr, status, st); break;
    case 5: dependent_d<5>(fp64, pts, dtype, cv, hc_dev, a, ncut, cut, rho_skip, rho, lambda, delta, ctr, status, st); break;
    case 6: dependent_d<6>(fp64, pts, dtype, cv, hc_dev, a, ncut, cut, rho_skip, rho, lambda, delta, ctr, status, st); break;
    case 7: dependent_d<7>(fp64, pts, dtype, cv, hc_dev, a, ncut, cut, rho_skip, rho, lambda, delta, ctr, status, st); break;
    default: dependent_d<8>(fp64, pts, dtype, cv, hc_dev, a, ncut, cut, rho_skip, rho, lambda, delta, ctr, status, st); break;
  }
  count_launches(1);
}

void launch_small_labels(const int32_t* rho, const int32_t* lambda, const double* delta, const ClassView& cv,
                         uint32_t nmax, const LabelParams* params, LabelParams one, int32_t* label, int* status,
                         cudaStream_t st) {
  if (cv.N == 0) return;
  const size_t sh = sizeof(int32_t) * (size_t)nmax;
  const unsigned grid = cv.ninst < sm_count() * 8u ? cv.ninst : sm_count() * 8u;
  k_small_labels<<<grid, kLabelThreads, sh, st>>>(rho, lambda, delta, cv, params, one, label, status);
  count_launches(1);
}

void small_init() {
  constexpr int kDevs = 64;
  static bool done[kDevs] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs || done[dev]) return;
  cudaFuncSetAttribute(k_small_labels, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)(sizeof(int32_t) * kSmallLabelPoints));
  done[dev] = true;
}

}  // namespace dpc

// decision.cu -- decision-graph summaries of one cutoff (Section 3, the
// decision graph plots delta against rho; cluster centers are the points
// standing out with both large).
//
//   top-k    per instance, the k points with the largest gamma = rho * delta
//            (binary64 product; descending gamma, equal gamma by the smaller
//            id; points whose product is NaN -- skipped points -- or negative
//            excluded).  One pass over the points counts a float32 lower
//            bound of gamma by its leading bits (k_dg_scan); the pick finds
//            the largest bin edge L that at least k points reach; a second
//            pass collects every point whose gamma can be >= L with its exact
//            gamma (k_dg_gather), normally a few thousand; one CTA per
//            instance sorts them (bitonic) and writes the first k.  Where
//            more points than the candidate buffer holds share the top bins
//            (masses of equal gamma), the exact radix select runs instead
//            (k_dg_select: 8-bit digits of the gamma bits, then of the ids).
//   hist     per instance, counts over (rho bin, delta bin): rho bin
//            floor(log2 rho); delta bin floor(log2(fl64(delta / delta_lo)))
//            (the exponent of the quotient), 0 for delta <= delta_lo; both
//            clipped to the last bin (+inf delta too).  Counted in the same
//            first pass.
//
// What bounds it: 12 bytes per point and pass, so two passes over 1e7 points
// are 35 us at the copy rate; the binary64 pipe (2 results per clock and SM)
// comes next, which is why neither pass multiplies or divides in binary64
// where a bound from the bit patterns decides.
#include <cmath>
#include <cstdint>

#include "internal.h"

namespace dpc {

namespace {

constexpr int kDgThreads = 1024;
constexpr int kMaxTopK = 1024;
constexpr int kDgCap = 4096;   // candidates the sort CTA can hold (48 KB of shared memory)
constexpr unsigned kFullMask = 0xffffffffu;

// Bins of the first pass and candidates kept per instance: up to 256 instances
// get fine bins (2048: a factor 1.09 of gamma each) and the whole sort buffer.
// With more the scratch is bounded by 24 bytes per point of the class and 1 KB
// and two or three times the k asked for per instance: 4 bins per octave and 1024
// candidates where the mean instance has 4096 points, 2 and 512 from 512
// points, and below that a buffer that takes the mean instance twice.  With one
// bin per octave and 2 k candidates most of 4,096 instances of 38,000 points
// overflowed into the radix select (k = 16: 50 ms; 2.6 now).
struct DgShape {
  int shift;     // bin = bits of the float32 lower bound >> shift
  int nbins;
  uint32_t cap;  // candidates per instance
};
inline DgShape dg_shape(uint32_t ninst, uint32_t n, int k) {
  DgShape z;
  const uint32_t mean = n / (ninst > 0u ? ninst : 1u) + 1u;
  z.shift = ninst <= 256u ? 20 : (mean >= 4096u ? 21 : (mean >= 512u ? 22 : 23));
  z.nbins = 1 << (31 - z.shift);
  const uint32_t room = ninst <= 256u ? (uint32_t)kDgCap : (mean >= 4096u ? 1024u : (mean >= 512u ? 512u : 2u * mean));
  const uint32_t want = (ninst > 256u && mean >= 4096u ? 3u : 2u) * (uint32_t)k;
  z.cap = room > want ? room : want;
  if (z.cap > (uint32_t)kDgCap) z.cap = (uint32_t)kDgCap;
  return z;
}

// gamma of one point as an order-preserving bit pattern; false for a point
// that takes no part (NaN delta, or a product that is NaN or negative).
__device__ __forceinline__ bool gamma_bits(int32_t rho, double delta, unsigned long long& gb) {
  const double g = __dmul_rn((double)rho, delta);
  if (!(g >= 0.0)) return false;
  gb = g == 0.0 ? 0ull : (unsigned long long)__double_as_longlong(g);  // -0 as +0
  return true;
}

// A float32 lower bound a <= gamma of a valid point, as its bit pattern
// (non-negative floats order like their bits).  Apart from saturation at
// FLT_MAX (gamma may be larger) and products below 2^-90 (a may be 0),
// gamma < a (1 + 2^-21): both factors and the product are truncated once to
// 24 bits.  No binary64 arithmetic unless a sign is involved.
__device__ __forceinline__ bool gamma_low(int32_t rho, double delta, uint32_t& a) {
  const uint32_t hi = (uint32_t)__double2hiint(delta), lo = (uint32_t)__double2loint(delta);
  if (rho > 0 && hi < 0x7ff00000u) {  // the usual case: delta finite and >= +0
    const int e = (int)(hi >> 20) - (1023 - 127);
    if (e >= 255) {
      a = 0x7f7fffffu;
    } else {
      const uint32_t f = e <= 0 ? 0u : ((uint32_t)e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
      a = __float_as_uint(__fmul_rz(__int2float_rz(rho), __uint_as_float(f)));
    }
    return true;
  }
  unsigned long long gb;
  if (!gamma_bits(rho, delta, gb)) return false;
  const float f = __double2float_rz(__longlong_as_double((long long)gb));
  a = min(__float_as_uint(f), 0x7f7fffffu);
  return true;
}

// Per-instance state of the selection.
struct __align__(16) DgState {
  unsigned long long prefix, mask;  // radix select: gamma bits fixed so far (T when done)
  uint32_t need;    // points still to take among those matching prefix/mask
  uint32_t all;     // 1: fewer than k valid points, every valid point is taken
  uint32_t idp, idm;  // id digits fixed so far (the tie break among gamma == T)
  uint32_t idneed;  // ties still to take among ids matching idp/idm
  uint32_t tie;     // 0: every point at T is taken; 1: ids below the limit only
  uint32_t fill;    // candidates gathered
  uint32_t low;     // smallest bits of the lower bound a candidate can have
  uint32_t exact;   // 1: the radix select finds the winners
  uint32_t pad[3];
};

// Words shared by the whole selection: instances left to the radix select,
// and its grid barrier.
struct DgShared {
  uint32_t open;
  uint32_t arrived;
  uint32_t stop;
  uint32_t pad;
};

// The CTA's share of a class: a contiguous range of chunks, and the instances
// of its first and last chunk (the only ones that can span other CTAs).
struct ChunkRange {
  uint32_t c0, c1, first, last;
};

__device__ __forceinline__ ChunkRange chunk_range(const ClassView& cv) {
  const uint32_t per = (cv.nchunk + gridDim.x - 1) / gridDim.x;
  ChunkRange r;
  r.c0 = min(cv.nchunk, blockIdx.x * per);
  r.c1 = min(cv.nchunk, r.c0 + per);
  uint32_t p0, end;
  r.first = r.last = 0xffffffffu;
  if (r.c0 < r.c1) {
    cv.chunk(r.c0, r.first, p0, end);
    cv.chunk(r.c1 - 1, r.last, p0, end);
  }
  return r;
}

// (rho, delta) bin of one point.  The exponent of fl64(delta / delta_lo) from
// the bit patterns: with both normal, quotient mantissa m = md / ml in
// (1/2, 2), and md < ml implies md / ml <= 1 - 2^-52 / ml < 1 - 2^-53, so the
// rounded quotient never reaches the next power of two.  (A binary64 divide
// per point took 250 us for 1e7 points; subnormals still divide.)
struct DgBins {
  int rho_bins, delta_bins;
  double lo;
};
__device__ __forceinline__ bool dg_bins(int32_t r, double dl, const DgBins& B, int& a, int& b) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(dl);
  if ((u & 0x7fffffffffffffffull) > 0x7ff0000000000000ull || r < 1) return false;
  a = 31 - __clz(r);
  a = a < B.rho_bins ? a : B.rho_bins - 1;
  const unsigned long long ul = (unsigned long long)__double_as_longlong(B.lo);
  if ((u >> 63) || u <= ul) {  // delta <= delta_lo
    b = 0;
    return true;
  }
  const int ed = (int)(u >> 52), el = (int)(ul >> 52);
  if (el > 0 && ed < 2047) {
    constexpr unsigned long long kMant = (1ull << 52) - 1ull;
    b = ed - el - ((u & kMant) < (ul & kMant) ? 1 : 0);
    if (b > 1023) b = B.delta_bins - 1;  // the quotient overflows
  } else {
    const double q = __ddiv_rn(dl, B.lo);
    b = isinf(q) ? B.delta_bins - 1 : ilogb(q);
  }
  b = b < 0 ? 0 : (b < B.delta_bins ? b : B.delta_bins - 1);
  return true;
}

constexpr int kHistSmemBins = 4096;  // (rho, delta) bins counted in shared memory at most
constexpr int kScanThreads = 256;
constexpr int kSelectBlocks = 4;  // CTAs per SM of the radix select, co-resident by its launch bounds

// First pass, every point once: counts of the lower bound's bins (TOP) and of
// the (rho, delta) bins (HIST).  Shared-memory counts for the CTA's first and
// last instance (a single instance: two copies, by warp, so that hot bins
// collide less), global atomics for instances wholly inside its range.  Loads
// are unrolled (4 points per thread in flight for a single instance): the
// pass is bound by the 12 bytes per point.
// 1e7 points, k = 1024, 24 x 48 bins: 1.36 ms per call with 8 digit passes and a
// binary64 divide per point; 0.115 ms now (this pass 44 us, the gather 25, the
// sort 24).
template <bool SINGLE, bool TOP, bool HIST, bool SMEM>
__global__ void __launch_bounds__(kScanThreads, 4)
k_dg_scan(const int32_t* __restrict__ rho, const double* __restrict__ delta, ClassView cv,
          uint32_t* __restrict__ hist, int shift, int nbins, uint32_t cap, DgBins B,
          unsigned long long* __restrict__ hist2) {
  extern __shared__ uint32_t dg_sh[];
  uint32_t* const s1 = dg_sh;                         // [2][nbins]
  uint32_t* const s2 = dg_sh + (TOP ? 2 * nbins : 0);  // [2][nb]
  const int nb = B.rho_bins * B.delta_bins;
  const int words = (TOP ? 2 * nbins : 0) + (HIST && SMEM ? 2 * nb : 0);
  for (int e = threadIdx.x; e < words; e += kScanThreads) dg_sh[e] = 0u;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // one point: slot 0 / 1 (shared) or 2 (global); all lanes of a warp share
  // slot and instance
  auto count = [&](int slot, uint32_t inst, uint32_t row, bool top, bool ok, int32_t r, double dl) {
    if constexpr (TOP) {
      uint32_t a;
      if (top && ok && gamma_low(r, dl, a)) {
        const uint32_t bin = a >> shift;
        if (slot < 2) atomicAdd(&s1[slot * nbins + bin], 1u);
        else atomicAdd(&hist[(size_t)inst * nbins + bin], 1u);
      }
    }
    if constexpr (HIST) {
      int ba = 0, bb = 0;
      const bool in = ok && dg_bins(r, dl, B, ba, bb);
      const int bin = ba * B.delta_bins + bb;
      if (SMEM && slot < 2) {
        if (in) atomicAdd(&s2[slot * nb + bin], 1u);
      } else {
        const uint32_t peers = __match_any_sync(kFullMask, in ? bin : -1 - lane);
        if (in && (peers & ((1u << lane) - 1u)) == 0u)
          atomicAdd(&hist2[(size_t)row * nb + bin], (unsigned long long)__popc(peers));
      }
    }
  };
  ChunkRange R;
  R.first = R.last = 0u;
  if constexpr (!SINGLE) R = chunk_range(cv);
  __syncthreads();
  if constexpr (SINGLE) {
    const InstDev I = cv.one;
    const uint64_t n = cv.N;
    const uint64_t stride = (uint64_t)gridDim.x * kScanThreads;
    const int32_t* const rp = rho + I.out;
    const double* const dp = delta + I.out;
    constexpr int U = 4;
    for (uint64_t p0 = (uint64_t)blockIdx.x * kScanThreads + warp * 32; p0 < n; p0 += U * stride) {
      int32_t r[U];
      double dl[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t p = p0 + u * stride + lane;
        r[u] = p < n ? __ldg(rp + p) : 0;
        dl[u] = p < n ? __ldg(dp + p) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) count(warp & 1, 0u, I.row, true, p0 + u * stride + lane < n, r[u], dl[u]);
    }
  } else {
    constexpr int kWarps = kScanThreads / 32;
    for (uint32_t c = R.c0 + warp; c < R.c1; c += kWarps) {
      uint32_t inst, p0, end;
      cv.chunk(c, inst, p0, end);
      const InstDev I = cv.instance(inst);
      const uint32_t p = p0 + lane;
      const uint64_t gi = I.out + (p - I.start);
      const bool ok = p < end;
      const int32_t r = ok ? __ldg(rho + gi) : 0;
      const double dl = ok ? __ldg(delta + gi) : 0.0;
      // an instance that fits the candidate buffer needs no counts
      count(inst == R.first ? 0 : (inst == R.last ? 1 : 2), inst, I.row, I.n > cap, ok, r, dl);
    }
  }
  __syncthreads();
  if constexpr (TOP) {
    for (int e = threadIdx.x; e < 2 * nbins; e += kScanThreads) {
      const uint32_t v = s1[e];
      const uint32_t inst = SINGLE ? 0u : (e < nbins ? R.first : R.last);
      if (v) atomicAdd(&hist[(size_t)inst * nbins + (e < nbins ? e : e - nbins)], v);
    }
  }
  if constexpr (HIST && SMEM) {
    for (int e = threadIdx.x; e < 2 * nb; e += kScanThreads) {
      const uint32_t v = s2[e];
      if (!v) continue;
      const InstDev I = cv.instance(SINGLE ? 0u : (e < nb ? R.first : R.last));
      atomicAdd(&hist2[(size_t)I.row * nb + (e < nb ? e : e - nb)], (unsigned long long)v);
    }
  }
}

// One warp per instance: the largest bin edge L that at least k points reach
// (every one of the k largest gammas is >= L), as the smallest lower-bound
// bits of a candidate: gamma >= L implies a > L (1 - 2^-21), 16 units of the
// bit pattern below L's.  Near and below 2^-90, where the bound may have
// underflowed, every valid point is a candidate.  More points than the buffer
// holds above L: the radix select takes the instance.
__global__ void k_dg_low(DgState* __restrict__ st, DgShared* __restrict__ sh, const uint32_t* __restrict__ hist,
                         ClassView cv, int k, int shift, int nbins, uint32_t cap) {
  const int lane = threadIdx.x & 31;
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  for (uint32_t inst = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); inst < cv.ninst; inst += nw) {
    const InstDev I = cv.instance(inst);
    uint32_t low = 0u, exact = 0u;
    if (I.n > cap) {
      const uint32_t* h = hist + (size_t)inst * nbins;
      // lane l sums the bins [top - per, top), top = nbins - l per: independent
      // 16-byte loads, one scan, and one lane walks its own bins again
      const int per = nbins >> 5, top = nbins - lane * per;
      uint32_t sum = 0;
      for (int e = top - per; e < top; e += 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(h + e);
        sum += v.x + v.y + v.z + v.w;
      }
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFullMask, incl, o);
        if (lane >= o) incl += t;
      }
      const unsigned hit = __ballot_sync(kFullMask, incl >= (uint32_t)k);
      if (hit) {
        const int src = __ffs(hit) - 1;
        uint32_t total = incl - sum;
        int bin = top;
        if (lane == src)
          while (total < (uint32_t)k) total += h[--bin];
        total = __shfl_sync(kFullMask, total, src);
        const uint32_t L = (uint32_t)__shfl_sync(kFullMask, bin, src) << shift;
        exact = total > cap ? 1u : 0u;
        low = L <= (37u << 23) ? 0u : L - 16u;
      }
    }
    if (lane == 0) {
      DgState z;
      z.prefix = z.mask = 0ull;
      z.need = (uint32_t)k;
      z.all = 0u;
      z.idp = z.idm = 0u;
      z.idneed = 0u;
      z.tie = 0u;
      z.fill = 0u;
      z.low = low;
      z.exact = exact;
      z.pad[0] = z.pad[1] = z.pad[2] = 0u;
      st[inst] = z;
      if (exact) atomicAdd(&sh->open, 1u);
    }
  }
}

// A warp appends its lanes' candidates (take) of one instance; the append
// that crosses the buffer's end hands the instance to the radix select.
__device__ __forceinline__ void dg_push(DgState* st, DgShared* sh, uint32_t inst, uint32_t cap, bool take,
                                        unsigned long long gb, uint32_t id, int lane,
                                        unsigned long long* __restrict__ cand_key,
                                        uint32_t* __restrict__ cand_id) {
  const unsigned m = __ballot_sync(kFullMask, take);
  if (m == 0u) return;
  uint32_t base = 0;
  if (lane == 0) {
    base = atomicAdd(&st[inst].fill, (uint32_t)__popc(m));
    if (sh && base <= cap && base + (uint32_t)__popc(m) > cap) {
      st[inst].exact = 1u;
      atomicAdd(&sh->open, 1u);
    }
  }
  base = __shfl_sync(kFullMask, base, 0);
  if (take) {
    const uint32_t slot = base + __popc(m & ((1u << lane) - 1u));
    if (slot < cap) {
      cand_key[(size_t)inst * cap + slot] = gb;
      cand_id[(size_t)inst * cap + slot] = id;
    }
  }
}

// Second pass: every point whose lower bound reaches the instance's `low`,
// with its exact gamma.
template <bool SINGLE>
__global__ void __launch_bounds__(kScanThreads, 4)
k_dg_gather(const int32_t* __restrict__ rho, const double* __restrict__ delta, ClassView cv, DgState* st,
            DgShared* sh, uint32_t cap, unsigned long long* __restrict__ cand_key,
            uint32_t* __restrict__ cand_id) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto point = [&](uint32_t inst, uint32_t low, bool ok, int32_t r, double dl, uint32_t id) {
    uint32_t a;
    bool take = ok && gamma_low(r, dl, a) && a >= low;
    if (!__any_sync(kFullMask, take)) return;
    unsigned long long gb = 0ull;
    if (take) take = gamma_bits(r, dl, gb);
    dg_push(st, sh, inst, cap, take, gb, id, lane, cand_key, cand_id);
  };
  if constexpr (SINGLE) {
    if (st[0].exact) return;
    const uint32_t low = st[0].low;
    const uint64_t n = cv.N;
    const uint64_t stride = (uint64_t)gridDim.x * kScanThreads;
    const int32_t* const rp = rho + cv.one.out;
    const double* const dp = delta + cv.one.out;
    constexpr int U = 4;
    for (uint64_t p0 = (uint64_t)blockIdx.x * kScanThreads + warp * 32; p0 < n; p0 += U * stride) {
      int32_t r[U];
      double dl[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t p = p0 + u * stride + lane;
        r[u] = p < n ? __ldg(rp + p) : 0;
        dl[u] = p < n ? __ldg(dp + p) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t p = p0 + u * stride + lane;
        point(0u, low, p < n, r[u], dl[u], (uint32_t)p);
      }
    }
  } else {
    const uint32_t nw = gridDim.x * (kScanThreads >> 5);
    for (uint32_t c = blockIdx.x * (kScanThreads >> 5) + warp; c < cv.nchunk; c += nw) {
      uint32_t inst, p0, end;
      cv.chunk(c, inst, p0, end);
      const DgState* S = st + inst;
      if (S->exact) continue;  // (a late 1 only saves work)
      const InstDev I = cv.instance(inst);
      const uint32_t p = p0 + lane;
      const uint32_t id = p - I.start;
      const uint64_t gi = I.out + id;
      const bool ok = p < end;
      const int32_t r = ok ? __ldg(rho + gi) : 0;
      const double dl = ok ? __ldg(delta + gi) : 0.0;
      point(inst, S->low, ok, r, dl, id);
    }
  }
}

// ---- the exact radix select (instances with masses of equal leading bits) ----

constexpr uint32_t kDgSpinLimit = 1u << 24;

// Grid barrier of a cooperative launch, bounded: a block that gives up (or
// sees that another did) makes every block leave.
__device__ bool dg_barrier(DgShared* sh, uint32_t& target, uint32_t limit, int* status) {
  __shared__ uint32_t s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    target += gridDim.x;
    __threadfence();
    atomicAdd(&sh->arrived, 1u);
    uint32_t ok = 0u;
    for (uint32_t i = 0; i <= limit; ++i) {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&sh->arrived) : "memory");
      if (v >= target) {
        ok = 1u;
        break;
      }
      if (*(volatile uint32_t*)&sh->stop) break;
      __nanosleep(64);
    }
    if (!ok) {
      *(volatile uint32_t*)&sh->stop = 1u;
      set_status(status, kStatusTimeout);
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0u;
}

__device__ __forceinline__ DgState dg_load(const DgState* st) {
  DgState s;
  const uint4* q = reinterpret_cast<const uint4*>(st);
  uint4* d = reinterpret_cast<uint4*>(&s);
  static_assert(sizeof(DgState) % 16 == 0, "state in 16-byte words");
#pragma unroll
  for (int i = 0; i < (int)(sizeof(DgState) / 16); ++i) d[i] = __ldcg(q + i);
  return s;
}

// Digit histogram of one pass, warp per 32-point chunk (one instance).  The
// CTA's first and last instances count in shared memory (one global add per
// bin at the end), the instances wholly inside its range count with one
// global atomic per distinct digit of a warp.  IDS = false: gamma digit dg of
// the points matching the instance's prefix; IDS = true: id digit dg of the
// points at gamma == T matching the id prefix.
template <bool IDS>
__device__ void dg_hist(const int32_t* __restrict__ rho, const double* __restrict__ delta, const ClassView& cv,
                        const DgState* st, uint32_t* hist, int dg, uint32_t (*sh)[256]) {
  const int lane = threadIdx.x & 31;
  for (int e = threadIdx.x; e < 512; e += blockDim.x) (&sh[0][0])[e] = 0u;
  const ChunkRange R = chunk_range(cv);
  __syncthreads();
  uint32_t cur = 0xffffffffu;
  DgState S;
#pragma unroll 2
  for (uint32_t c = R.c0 + (threadIdx.x >> 5); c < R.c1; c += blockDim.x >> 5) {
    uint32_t inst, p0, end;
    cv.chunk(c, inst, p0, end);
    if (inst != cur) S = dg_load(st + inst);
    cur = inst;
    if (!S.exact || S.all || (IDS && !S.tie)) continue;  // warp-uniform
    const InstDev I = cv.instance(inst);
    const uint32_t p = p0 + lane;
    uint32_t digit = 256u + lane;  // no digit: a key no other lane has
    if (p < end) {
      const uint32_t id = p - I.start;
      const uint64_t gi = I.out + id;
      unsigned long long gb;
      if (gamma_bits(rho[gi], delta[gi], gb)) {
        if (!IDS) {
          if ((gb & S.mask) == S.prefix) digit = (uint32_t)(gb >> (8 * dg)) & 255u;
        } else if (gb == S.prefix && (id & S.idm) == S.idp) {
          digit = (id >> (8 * dg)) & 255u;
        }
      }
    }
    const uint32_t peers = __match_any_sync(kFullMask, digit);
    if (digit < 256u && (peers & ((1u << lane) - 1u)) == 0u) {
      const uint32_t v = (uint32_t)__popc(peers);
      if (inst == R.first) atomicAdd(&sh[0][digit], v);
      else if (inst == R.last) atomicAdd(&sh[1][digit], v);
      else atomicAdd(&hist[(size_t)inst * 256u + digit], v);
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 512; e += blockDim.x) {
    const uint32_t v = (&sh[0][0])[e];
    const uint32_t inst = e < 256 ? R.first : R.last;
    if (v) atomicAdd(&hist[(size_t)inst * 256u + (e & 255)], v);
  }
}

// One warp per instance: fix digit dg from the histogram, then clear it.
template <bool IDS>
__device__ void dg_pick(DgState* st, uint32_t* hist, uint32_t ninst, int dg) {
  const int lane = threadIdx.x & 31;
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  for (uint32_t inst = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); inst < ninst; inst += nw) {
    DgState S = dg_load(st + inst);
    if (!S.exact) continue;
    uint32_t* h = hist + (size_t)inst * 256u;
    const bool active = !(S.all || (IDS && !S.tie));
    if (active) {
      // gamma: digits from the top (lane 0 holds 255..248); ids: from the bottom
      uint32_t c[8];
      uint32_t sum = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int b = IDS ? lane * 8 + j : 255 - (lane * 8 + j);
        c[j] = __ldcg(h + b);
        sum += c[j];
      }
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFullMask, incl, o);
        if (lane >= o) incl += t;
      }
      const uint32_t need = IDS ? S.idneed : S.need;
      // the digit where the running count reaches `need`
      uint32_t before = incl - sum;
      int found = -1;
      uint32_t below = 0, at = 0;
      if (before < need && incl >= need) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (found < 0 && before + c[j] >= need) {
            found = IDS ? lane * 8 + j : 255 - (lane * 8 + j);
            below = before;
            at = c[j];
          }
          if (found < 0) before += c[j];
        }
      }
      const unsigned owner = __ballot_sync(kFullMask, found >= 0);
      if (owner == 0u) {
        // fewer than `need` points match: only possible on the first gamma
        // digit (every valid point is counted there) -- take them all
        if (!IDS && lane == 0) S.all = 1u;
      } else {
        const int src = __ffs(owner) - 1;
        const int D = __shfl_sync(kFullMask, found, src);
        const uint32_t bl = __shfl_sync(kFullMask, below, src);
        const uint32_t cnt_at = __shfl_sync(kFullMask, at, src);
        if (!IDS) {
          S.prefix |= (unsigned long long)D << (8 * dg);
          S.mask |= 255ull << (8 * dg);
          S.need = need - bl;
          if (dg == 0) {  // T is fixed: S.need points at T remain to take
            S.tie = cnt_at > S.need ? 1u : 0u;
            S.idneed = S.need;
          }
        } else {
          S.idp |= (uint32_t)D << (8 * dg);
          S.idm |= 255u << (8 * dg);
          S.idneed = need - bl;
        }
      }
    }
    __syncwarp();
    if (lane == 0) st[inst] = S;
#pragma unroll
    for (int j = 0; j < 8; ++j) h[lane * 8 + j] = 0u;
  }
}

// Cooperative launch; returns at once when no instance needs it.  Per 8-bit
// digit (8 of gamma, 4 of the id where more points sit at the k-th value than
// are needed): a histogram over all points of the class, a grid barrier, a
// pick per instance, a grid barrier; then the winners -- gamma above T, or at
// T with an id no larger than the tie limit -- replace the candidates.
__global__ void __launch_bounds__(256, kSelectBlocks)
k_dg_select(const int32_t* __restrict__ rho, const double* __restrict__ delta, ClassView cv, DgState* st,
            DgShared* gs, uint32_t* hist, uint32_t cap, unsigned long long* __restrict__ cand_key,
            uint32_t* __restrict__ cand_id, uint32_t limit, int* status) {
  __shared__ uint32_t sh[2][256];
  if (__ldcg(&gs->open) == 0u) return;
  uint32_t target = 0;
  const int lane = threadIdx.x & 31;
  const uint64_t gtid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  const uint64_t gall = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t e = gtid; e < (uint64_t)cv.ninst * 256u; e += gall) hist[e] = 0u;
  for (uint64_t e = gtid; e < cv.ninst; e += gall)
    if (__ldcg(&st[e].exact)) st[e].fill = 0u;
  if (!dg_barrier(gs, target, limit, status)) return;
  for (int dg = 7; dg >= 0; --dg) {
    dg_hist<false>(rho, delta, cv, st, hist, dg, sh);
    if (!dg_barrier(gs, target, limit, status)) return;
    dg_pick<false>(st, hist, cv.ninst, dg);
    if (!dg_barrier(gs, target, limit, status)) return;
  }
  for (int dg = 3; dg >= 0; --dg) {
    dg_hist<true>(rho, delta, cv, st, hist, dg, sh);
    if (!dg_barrier(gs, target, limit, status)) return;
    dg_pick<true>(st, hist, cv.ninst, dg);
    if (!dg_barrier(gs, target, limit, status)) return;
  }
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  for (uint32_t c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < cv.nchunk; c += nw) {
    uint32_t inst, p0, end;
    cv.chunk(c, inst, p0, end);
    const DgState S = dg_load(st + inst);
    if (!S.exact) continue;
    const InstDev I = cv.instance(inst);
    const uint32_t p = p0 + lane;
    bool take = false;
    unsigned long long gb = 0ull;
    uint32_t id = 0u;
    if (p < end) {
      id = p - I.start;
      const uint64_t gi = I.out + id;
      if (gamma_bits(rho[gi], delta[gi], gb))
        take = S.all || gb > S.prefix || (gb == S.prefix && (!S.tie || id <= S.idp));
    }
    dg_push(st, nullptr, inst, cap, take, gb, id, lane, cand_key, cand_id);
  }
}

// One CTA per instance: bitonic sort of its candidates (gamma descending, id
// ascending), the first k into its output row.
__global__ void __launch_bounds__(kDgThreads)
k_dg_sort(ClassView cv, const DgState* __restrict__ st, int k, uint32_t cap, const unsigned long long* __restrict__ cand_key,
          const uint32_t* __restrict__ cand_id, int32_t* __restrict__ top, double* __restrict__ gamma_out) {
  __shared__ unsigned long long s_key[kDgCap];
  __shared__ uint32_t s_id[kDgCap];
  const int tid = threadIdx.x;
  for (uint32_t inst = blockIdx.x; inst < cv.ninst; inst += gridDim.x) {
    const InstDev I = cv.instance(inst);
    const uint32_t filled = min(st[inst].fill, cap);
    uint32_t P = 1;
    while (P < filled) P <<= 1;
    for (uint32_t i = tid; i < P; i += blockDim.x) {
      if (i < filled) {
        s_key[i] = cand_key[(size_t)inst * cap + i];
        s_id[i] = cand_id[(size_t)inst * cap + i];
      } else {
        s_key[i] = 0ull;
        s_id[i] = 0xffffffffu;  // padding sorts last
      }
    }
    __syncthreads();
    // pair (i, i + stride) of every stage by pair number: pairs 32 w .. 32 w +
    // 31 lie in one 64-element block for strides up to 32, so those stages
    // need a warp barrier only (21 block barriers for 4096 candidates, not 78)
    auto stage = [&](uint32_t size, uint32_t stride) {
      for (uint32_t q = tid; q < P / 2; q += kDgThreads) {
        const uint32_t i = 2u * q - (q & (stride - 1u)), j = i + stride;
        const unsigned long long ki = s_key[i], kj = s_key[j];
        const uint32_t ni = s_id[i], nj = s_id[j];
        const bool i_first = ki > kj || (ki == kj && ni < nj);
        if (((i & size) == 0) != i_first) {
          s_key[i] = kj;
          s_key[j] = ki;
          s_id[i] = nj;
          s_id[j] = ni;
        }
      }
    };
    for (uint32_t size = 2; size <= P; size <<= 1) {
      uint32_t stride = size >> 1;
      for (; stride > 32; stride >>= 1) {
        stage(size, stride);
        __syncthreads();
      }
      for (; stride > 0; stride >>= 1) {
        stage(size, stride);
        __syncwarp();
      }
      __syncthreads();
    }
    for (int i = tid; i < k; i += blockDim.x) {
      const size_t o = (size_t)I.row * k + i;
      if ((uint32_t)i < filled) {
        top[o] = (int32_t)s_id[i];
        gamma_out[o] = __longlong_as_double((long long)s_key[i]);
      } else {
        top[o] = -1;
        gamma_out[o] = __longlong_as_double(0x7ff8000000000000ll);  // NaN: no point
      }
    }
    __syncthreads();
  }
}

// Every top-k row: no point (-1, NaN) until the instance's CTA fills it.
__global__ void k_decision_pad(int32_t* top, double* gamma, size_t m) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < m; i += (size_t)gridDim.x * blockDim.x) {
    top[i] = -1;
    gamma[i] = __longlong_as_double(0x7ff8000000000000ll);
  }
}

}  // namespace

void launch_decision_init(int n_inst, int k, bool pad, int32_t* top, double* gamma, int rho_bins,
                          int delta_bins, unsigned long long* hist, cudaStream_t st) {
  if (pad && k > 0 && top && gamma) {
    const size_t m = (size_t)n_inst * k;
    uint64_t blocks = (m + 255) / 256;
    if (blocks < 1) blocks = 1;
    if (blocks > sm_count() * 16u) blocks = sm_count() * 16u;
    k_decision_pad<<<(unsigned)blocks, 256, 0, st>>>(top, gamma, m);
    count_launches(1);
  }
  if (hist && rho_bins > 0 && delta_bins > 0)
    cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * (size_t)n_inst * rho_bins * delta_bins, st);
}

// Scratch of one class: state, shared words and bins (zeroed together), then
// the candidates.
struct DgScratch {
  size_t shared, hist, zeroed, key, id, bytes;
};
static DgScratch dg_scratch(uint32_t ninst, uint32_t n, int k) {
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  const DgShape z = dg_shape(ninst, n, k);
  DgScratch o;
  o.shared = al(sizeof(DgState) * ninst);
  o.hist = o.shared + al(sizeof(DgShared));
  o.zeroed = o.hist + al(sizeof(uint32_t) * (size_t)z.nbins * ninst);
  o.key = o.zeroed;
  o.id = o.key + al(sizeof(unsigned long long) * (size_t)ninst * z.cap);
  o.bytes = o.id + al(sizeof(uint32_t) * (size_t)ninst * z.cap);
  return o;
}

size_t decision_scratch_bytes(uint32_t ninst, uint32_t n, int k) { return dg_scratch(ninst, n, k).bytes; }

template <bool SINGLE>
static void dg_scan(bool top, bool hist, bool smem, unsigned grid, size_t sh_bytes, const int32_t* rho,
                    const double* delta, const ClassView& cv, uint32_t* H, const DgShape& z, const DgBins& B,
                    unsigned long long* hist2, cudaStream_t st) {
  auto go = [&](auto kern) {
    kern<<<grid, kScanThreads, sh_bytes, st>>>(rho, delta, cv, H, z.shift, z.nbins, z.cap, B, hist2);
    count_launches(1);
  };
  if (top && hist && smem) go(k_dg_scan<SINGLE, true, true, true>);
  else if (top && hist) go(k_dg_scan<SINGLE, true, true, false>);
  else if (top) go(k_dg_scan<SINGLE, true, false, false>);
  else if (smem) go(k_dg_scan<SINGLE, false, true, true>);
  else go(k_dg_scan<SINGLE, false, true, false>);
}

int launch_decision(const int32_t* rho, const double* delta, const ClassView& cv, int k,
                    int32_t* top, double* gamma, int rho_bins, int delta_bins, double delta_lo,
                    unsigned long long* hist, void* scratch, int* status, cudaStream_t st) {
  const bool want_top = k > 0 && top && gamma && cv.ninst > 0;
  const bool want_hist = hist && rho_bins > 0 && delta_bins > 0 && cv.ninst > 0;
  const bool single = cv.inst == nullptr;
  const DgShape z = dg_shape(cv.ninst, cv.N, k > 0 ? k : 1);
  const DgScratch o = dg_scratch(cv.ninst, cv.N, k > 0 ? k : 1);
  char* b = (char*)scratch;
  DgState* S = (DgState*)b;
  DgShared* G = (DgShared*)(b + o.shared);
  uint32_t* H = (uint32_t*)(b + o.hist);
  unsigned long long* ck = (unsigned long long*)(b + o.key);
  uint32_t* ci = (uint32_t*)(b + o.id);
  // a single instance that fits the candidate buffer needs no counts
  const bool count = want_top && !(single && cv.N <= z.cap);
  if (want_top) cudaMemsetAsync(G, 0, o.zeroed - o.shared, st);
  // 4 CTAs per SM hold every thread the register budget allows; at least 4
  // points per thread
  uint64_t cb = ((uint64_t)cv.nchunk * 32u + 4u * kScanThreads - 1) / (4u * kScanThreads);
  const unsigned grid = (unsigned)(cb < 1 ? 1 : (cb > sm_count() * 4u ? sm_count() * 4u : cb));
  if (count || want_hist) {
    const DgBins B{rho_bins, delta_bins, delta_lo};
    const bool smem = want_hist && rho_bins * delta_bins <= kHistSmemBins;
    const size_t sh = sizeof(uint32_t) * ((count ? 2u * z.nbins : 0u) + (smem ? 2u * rho_bins * delta_bins : 0u));
    if (single) dg_scan<true>(count, want_hist, smem, grid, sh, rho, delta, cv, H, z, B, hist, st);
    else dg_scan<false>(count, want_hist, smem, grid, sh, rho, delta, cv, H, z, B, hist, st);
  }
  if (!want_top) return 0;
  uint64_t ib = ((uint64_t)cv.ninst + 7) / 8;
  const unsigned inst_blocks = (unsigned)(ib < 1 ? 1 : (ib > sm_count() * 16u ? sm_count() * 16u : ib));
  k_dg_low<<<inst_blocks, 256, 0, st>>>(S, G, H, cv, k, z.shift, z.nbins, z.cap);
  if (single) k_dg_gather<true><<<grid, kScanThreads, 0, st>>>(rho, delta, cv, S, G, z.cap, ck, ci);
  else k_dg_gather<false><<<grid, kScanThreads, 0, st>>>(rho, delta, cv, S, G, z.cap, ck, ci);
  count_launches(2);
  if (!(single && cv.N <= z.cap)) {
    const uint32_t limit = wait_limit(kDgSpinLimit);
    const unsigned sg = sm_count() * kSelectBlocks;
    uint32_t cap = z.cap;
    ClassView v = cv;
    void* args[] = {(void*)&rho, (void*)&delta, (void*)&v,  (void*)&S,  (void*)&G,     (void*)&H,
                    (void*)&cap, (void*)&ck,    (void*)&ci, (void*)&limit, (void*)&status};
    if (cudaLaunchCooperativeKernel((const void*)k_dg_select, dim3(sg), dim3(256), args, 0, st) != cudaSuccess)
      return -1;
    count_launches(1);
  }
  const unsigned sgrid = cv.ninst < sm_count() * 2u ? cv.ninst : sm_count() * 2u;
  k_dg_sort<<<sgrid, kDgThreads, 0, st>>>(cv, S, k, z.cap, ck, ci, top, gamma);
  count_launches(1);
  return 0;
}

int decision_max_topk() { return kMaxTopK; }

}  // namespace dpc

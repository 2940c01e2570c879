// sort.cu -- LSD radix sort of (64-bit code, 32-bit id) pairs by code.
//
// The radix-sort primitive of Section 3.2, used here to put the points in
// Morton order.  The digits of every pass are counted beforehand (by the kernel
// that writes the codes, rs_count_digits, or k_rs_hist_all in one read of the
// keys).  Then one kernel per 8-bit pass (k_rs_onesweep): a CTA takes the next
// tile (an atomic tile counter, so tiles start in order), ranks every item
// inside the tile (warp multi-split with __match_any_sync, warps in tile order),
// publishes its digit counts, and finds the count of every digit in all earlier
// tiles by looking back over their published counts (decoupled look-back, after
// Merrill and Garland's single-pass prefix scan: a tile that has its inclusive
// prefix publishes it, so a look-back stops at the first such tile); then a
// shared-memory reorder and coalesced runs to the global positions.  The
// published words carry the pass, so one clear serves all passes.  Every wait
// on an earlier tile is bounded; a wait that gives up records kStatusTimeout.
// The number of passes (ceil((S + ib) / 8) for keys of S + ib bits, see
// ClassGeom) is known only on the device: passes beyond it return at once, so
// the launch sequence is fixed and the result lands in buffer (passes & 1).
//
// A tile's ranking is a chain of one shared-memory step per item and thread, so
// few items per thread make short passes as long as the tiles fill the chip:
// 4 items (1,024 a tile) up to 2^17, 8 up to 2^21, 16 beyond.  Binning of blobs of
// 1e4 / 1e5 / 1e6 points in 3-D with 16 items throughout, a clear per pass and
// count and scan kernels of their own: 131 / 145 / 241 us; as here: 79 / 101 / 206.
#include "internal.h"

namespace dpc {

namespace {

constexpr int kRsThreads = 256;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kMaxPasses = (int)kSortMaxPasses;

constexpr unsigned long long kFlagAgg = 1ull << 62;     // the tile's own counts
constexpr unsigned long long kFlagPrefix = 2ull << 62;  // counts of this and every earlier tile
constexpr unsigned long long kFlagMask = 3ull << 62;
constexpr int kPassShift = 56;  // published by pass p: p + 1 in bits 56..59
constexpr unsigned long long kPassMask = 15ull << kPassShift;
constexpr uint32_t kSpinLimit = 1u << 20;  // ld.acquire polls of earlier tiles before giving up

// The sort's scratch: status[ntiles][256] (u64, reused by every pass), the
// digit counts of every pass [kMaxPasses][256], a tile counter per pass.
struct SortScratch {
  unsigned long long* status;
  uint32_t* count;
  uint32_t* tiles;
};

__host__ __device__ inline SortScratch sort_scratch(uint32_t* base, uint32_t ntiles) {
  SortScratch z;
  z.status = reinterpret_cast<unsigned long long*>(base);
  z.count = base + (size_t)ntiles * 256u * 2u;
  z.tiles = z.count + kMaxPasses * 256;
  return z;
}

// Digit counts of every pass in one read of the keys.
__global__ void __launch_bounds__(kRsThreads)
k_rs_hist_all(const unsigned long long* __restrict__ keys, uint32_t n,
              const ClassGeom* __restrict__ cls, uint32_t* __restrict__ count) {
  __shared__ uint32_t cnt[kMaxPasses][256];
  const int npass = sort_passes(cls->S, cls->ib);
  rs_clear_digits(cnt);
  for (uint32_t i = blockIdx.x * kRsThreads + threadIdx.x; i < n; i += gridDim.x * kRsThreads)
    rs_count_digits(cnt, keys[i], npass);
  rs_flush_digits(cnt, count, npass);
}

__device__ __forceinline__ void st_release(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

template <int IPT>
struct ScatterSmem {
  unsigned long long keys[kRsThreads * IPT];
  uint32_t vals[kRsThreads * IPT];
  uint32_t whist[kRsWarps][256];  // per-warp digit counts, then warp prefixes
  uint32_t tstart[256];           // tile-local start of each digit
  uint32_t gbase[256];            // global start of each digit in this tile
  uint32_t wsum[2][kRsWarps];
  uint32_t tile;
};

template <int kRsIpt>
__global__ void __launch_bounds__(kRsThreads, kRsIpt == 16 ? 3 : (kRsIpt == 8 ? 4 : 6))
k_rs_onesweep(const unsigned long long* __restrict__ kin, const uint32_t* __restrict__ vin,
              unsigned long long* __restrict__ kout, uint32_t* __restrict__ vout, uint32_t n,
              int pass, const ClassGeom* __restrict__ cls, SortScratch z, uint32_t spin_limit) {
  if (pass >= sort_passes(cls->S, cls->ib)) return;
  constexpr int kRsTile = kRsThreads * kRsIpt;
  constexpr int kRsWarpItems = 32 * kRsIpt;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ScatterSmem<kRsIpt>& S = *reinterpret_cast<ScatterSmem<kRsIpt>*>(smem_raw);
  const unsigned long long tag = (unsigned long long)(pass + 1) << kPassShift;
  const int shift = 8 * pass;
  const int lane = threadIdx.x & 31;
  const int w = threadIdx.x >> 5;
  const uint32_t lanemask_lt = (1u << lane) - 1u;

  for (int i = threadIdx.x; i < kRsWarps * 256; i += kRsThreads) (&S.whist[0][0])[i] = 0;
  // tiles are taken in launch order, so every earlier tile has started
  if (threadIdx.x == 0) S.tile = atomicAdd(&z.tiles[pass], 1u);
  __syncthreads();
  const uint32_t tile = S.tile;

  // pass 1: warp-local stable ranks
  const uint32_t wbase = tile * kRsTile + w * kRsWarpItems;
  unsigned long long key[kRsIpt];
  uint32_t val[kRsIpt];
  uint32_t rank[kRsIpt];
#pragma unroll
  for (int r = 0; r < kRsIpt; ++r) {
    const uint32_t i = wbase + r * 32 + lane;
    const bool valid = i < n;
    key[r] = valid ? kin[i] : 0ull;
    val[r] = valid ? vin[i] : 0u;
    const uint32_t dg = (uint32_t)(key[r] >> shift) & 255u;
    const uint32_t vmask = __ballot_sync(0xffffffffu, valid);
    const uint32_t peers = __match_any_sync(0xffffffffu, valid ? dg : (256u + lane)) & vmask;
    uint32_t pre = 0;
    if (valid) pre = S.whist[w][dg];
    __syncwarp();
    if (valid && (peers & lanemask_lt) == 0) S.whist[w][dg] = pre + __popc(peers);
    __syncwarp();
    rank[r] = valid ? pre + __popc(peers & lanemask_lt) : 0xffffffffu;
  }
  __syncthreads();
  // per digit: prefix over warps (tile order), the tile's count, then the
  // count of the digit in every earlier tile (look-back)
  {
    const int d = threadIdx.x;
    uint32_t run = 0;
#pragma unroll
    for (int k = 0; k < kRsWarps; ++k) {
      uint32_t c = S.whist[k][d];
      S.whist[k][d] = run;
      run += c;
    }
    const uint32_t my_total = run;
    unsigned long long* st = z.status + (size_t)tile * 256u + d;
    st_release(st, (tile == 0 ? kFlagPrefix : kFlagAgg) | tag | my_total);
    uint32_t before = 0;
    if (tile > 0) {
      uint32_t t = tile - 1;
      uint32_t spins = 0;
      for (;;) {
        const unsigned long long v = ld_acquire(z.status + (size_t)t * 256u + d);
        const unsigned long long f = v & kFlagMask;
        if (f == 0ull || (v & kPassMask) != tag) {
          if (spins++ >= spin_limit) {
            // an earlier tile has not published in time: record it, and count
            // this digit over every earlier tile's items directly (slow but
            // exact, so the sort and everything after it stay well formed)
            set_status(cls->status, kStatusTimeout);
            before = 0;
            const uint32_t upto = tile * (uint32_t)kRsTile;  // < n: this tile exists
            for (uint32_t i = 0; i < upto; ++i)
              before += ((uint32_t)(kin[i] >> shift) & 255u) == (uint32_t)d ? 1u : 0u;
            break;
          }
          continue;
        }
        before += (uint32_t)v;
        if (f == kFlagPrefix || t == 0) break;
        --t;
      }
      st_release(st, kFlagPrefix | tag | (before + my_total));
    }
    // tile-local starts and the digits' global starts: two exclusive scans
    // over the 256 digits (warp scans and the warps' sums)
    const uint32_t cnt = z.count[pass * 256 + d];
    uint32_t i1 = my_total, i2 = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t1 = __shfl_up_sync(0xffffffffu, i1, o), t2 = __shfl_up_sync(0xffffffffu, i2, o);
      if (lane >= o) {
        i1 += t1;
        i2 += t2;
      }
    }
    if (lane == 31) {
      S.wsum[0][w] = i1;
      S.wsum[1][w] = i2;
    }
    __syncthreads();
    uint32_t b1 = 0, b2 = 0;
#pragma unroll
    for (int k = 0; k < kRsWarps; ++k)
      if (k < w) {
        b1 += S.wsum[0][k];
        b2 += S.wsum[1][k];
      }
    S.tstart[d] = b1 + i1 - my_total;
    S.gbase[d] = b2 + i2 - cnt + before;
  }
  __syncthreads();
  // pass 2: place every item at its tile-local sorted position
#pragma unroll
  for (int r = 0; r < kRsIpt; ++r) {
    if (rank[r] != 0xffffffffu) {
      const uint32_t dg = (uint32_t)(key[r] >> shift) & 255u;
      const uint32_t pos = S.tstart[dg] + S.whist[w][dg] + rank[r];
      if (pos < (uint32_t)kRsTile) {
        S.keys[pos] = key[r];
        S.vals[pos] = val[r];
      } else {
        set_status(cls->status, kStatusIndex);
      }
    }
  }
  __syncthreads();
  // pass 3: coalesced runs to global memory
  const uint32_t tbase = tile * kRsTile;
  const uint32_t tcount = tbase < n ? min((uint32_t)kRsTile, n - tbase) : 0u;
  for (uint32_t pos = threadIdx.x; pos < tcount; pos += kRsThreads) {
    const unsigned long long k = S.keys[pos];
    const uint32_t dg = (uint32_t)(k >> shift) & 255u;
    const uint32_t dst = S.gbase[dg] + (pos - S.tstart[dg]);
    if (dst < n) {
      kout[dst] = k;
      vout[dst] = S.vals[pos];
    } else {
      set_status(cls->status, kStatusIndex);
    }
  }
}

// Items per thread of a pass over n items (see the top of the file).
int items_for(uint32_t n) { return n <= kSortSmall ? 4 : (n <= kSortMiddle ? 8 : 16); }

}  // namespace

size_t sort_hist_words(uint32_t n) { return sort_hist_words_for(n); }

void sort_init() {
  constexpr int kDevs = 64;
  static bool done[kDevs] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs || done[dev]) return;
  cudaFuncSetAttribute(k_rs_onesweep<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ScatterSmem<4>));
  cudaFuncSetAttribute(k_rs_onesweep<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ScatterSmem<8>));
  cudaFuncSetAttribute(k_rs_onesweep<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ScatterSmem<16>));
  done[dev] = true;
}

uint32_t* launch_sort_clear(uint32_t n, uint32_t* hist, cudaStream_t st) {
  const uint32_t tile = (uint32_t)(kRsThreads * items_for(n));
  const uint32_t nt = (n + tile - 1) / tile;
  const SortScratch z = sort_scratch(hist, nt);
  cudaMemsetAsync(hist, 0, (char*)(z.tiles + kMaxPasses) - (char*)hist, st);
  return z.count;
}

void launch_sort(unsigned long long* codes_a, unsigned long long* codes_b, uint32_t* ids_a,
                 uint32_t* ids_b, uint32_t n, const ClassGeom* cls, uint32_t* hist, bool counted,
                 cudaStream_t st) {
  if (n == 0) return;
  const int ipt = items_for(n);
  const uint32_t nt = (n + (uint32_t)(kRsThreads * ipt) - 1) / (uint32_t)(kRsThreads * ipt);
  sort_init();
  const SortScratch z = sort_scratch(hist, nt);
  const uint32_t spin = wait_limit(kSpinLimit);
  if (!counted) {
    launch_sort_clear(n, hist, st);
    const uint32_t want = (n + 4u * kRsThreads - 1) / (4u * kRsThreads);
    const unsigned hb = want < sm_count() * 4u ? want : sm_count() * 4u;
    k_rs_hist_all<<<hb, kRsThreads, 0, st>>>(codes_a, n, cls, z.count);
    count_launches(1);
  }
  unsigned long long* kb[2] = {codes_a, codes_b};
  uint32_t* vb[2] = {ids_a, ids_b};
  auto go = [&](auto kern, size_t sh) {
    for (int pass = 0; pass < kMaxPasses; ++pass) {
      const int i = pass & 1, o = (pass + 1) & 1;
      kern<<<nt, kRsThreads, sh, st>>>(kb[i], vb[i], kb[o], vb[o], n, pass, cls, z, spin);
    }
  };
  if (ipt == 4) go(k_rs_onesweep<4>, sizeof(ScatterSmem<4>));
  else if (ipt == 8) go(k_rs_onesweep<8>, sizeof(ScatterSmem<8>));
  else go(k_rs_onesweep<16>, sizeof(ScatterSmem<16>));
  count_launches(kMaxPasses);
}

}  // namespace dpc

// tc_density.cu -- rho_i (Definition 1) and the near phase of the dependent
// search for 5- to 8-dimensional points with the distance tiles on the tensor
// cores (tcgen05, TF32 operands, FP32 accumulation in tensor memory).
//
// Work layout: the sorted points are cut into pieces of at most 128 consecutive
// points whose blocks share a box of cells (k_tc_pieces); a CTA of 8 warps takes
// pieces one by one from a global work counter.  The 128 rows of the MMA are the
// piece's queries, the columns the candidates of the piece's cells, 256 per MMA.
// With the augmented rows
//     a = [q_0 .. q_d-1, (1 + e) |q|^2, 1]
//     b = [-2 c_0 .. -2 c_d-1, 1, (1 + e) |c|^2]      (e = 2^-14)
// one product a . b = s + e (|q|^2 + |c|^2): the squared distance s plus an error
// allowance, so that subtracting (1 - e) t_in, t_in the float32 filter's inner
// threshold, leaves s + E - t_in with E = e (|q|^2 + |c|^2 + t_in).  Every operand
// is split into a TF32 high part and a TF32 remainder; the products hi.hi, hi.lo
// and lo.hi (measured error ~2^-22 relative to |a||b|) lie side by side in 3 d + 4
// columns.  Coordinates are taken relative to the piece's first query so the
// norms stay small.  Thread t owns one accumulator row (its query) and half of
// the 256 columns of each tile.
//
// Exactness: E is far above the split-TF32 error, the FP32 accumulation error
// (at most about 2^-16.4 times the same sum of norms) and the float32 norm
// rounding, so acc - (1 - e) t_in < 0 proves s <= t_in, hence s64 <= d_cut^2
// (t_in, t_out as in the float32 filter); above W = (t_out - t_in) +
// 1.25 e (|q|^2 + the largest |c|^2 of the 32 columns + t_in) (rounded up) it
// proves s > t_out, hence s64 > d_cut^2.  Pairs in between are decided by the
// float32 filter on the original coordinates and, inside its own band, by the
// canonical binary64 distance, so rho is exactly the binary64 count.
//
// What bounds it: the epilogue's ALU work (ALU pipe 62% busy with three cutoffs in a
// pass, 43% with one) and the barriers between staging, MMA and epilogue (two CTAs
// per SM overlap them); the tensor pipe is 10% busy with three cutoffs in a pass,
// 18% with one, 11% in the near phase (profiles/, 663,000 points in 7-D).
// 2e6 points in 7-D: three cutoffs of one level in one pass 40 ms where three
// passes of two separate operands, one cutoff each and one cell per piece took
// about 35 each; the recount alone, unrolled per column and in binary64 for every
// pair of the tensor band, took 5x that (it thrashes the instruction cache).
#include <cstdint>

#include "block.cuh"
#include "internal.h"

namespace dpc {

namespace {

constexpr int kTcThreads = 256;     // 8 warps: warps w and w + 4 share accumulator lanes
constexpr int kTcM = 128;            // queries per MMA (rows)
constexpr int kTcN = 256;            // candidates per MMA (columns)
constexpr float kTcErr = 0x1p-14f;
// one candidate row per thread: warp w stages columns 32w .. 32w + 31
static_assert(kTcN == kTcThreads, "candidate rows per thread");
// |c|^2 of a padding candidate, which must never count: above every threshold
// (make_cut_host keeps t_in at or below 3.0e38), and finite as a sum of two TF32
// numbers.  (A mask of the last columns instead costs the density 0.7-1%.)
constexpr float kTcFar = 3.2e38f;
constexpr uint32_t kTcWaitLimit = 1u << 26;  // mbarrier polls before giving up

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t u;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
  return __uint_as_float(u);
}

// Byte offset of element (row r, k) in the K-major, non-swizzled operand
// layout of a ROWS-row operand: core matrices of 8 rows x 16 bytes; the two
// core matrices of one 8-element K step 128 bytes apart (leading offset),
// 8-row groups 256 bytes apart (stride offset), K steps ROWS * 32 bytes apart.
template <int ROWS>
__device__ __forceinline__ uint32_t op_off(int r, int k) {
  return (uint32_t)((k >> 3) * (ROWS * 32) + (r >> 3) * 256 + ((k >> 2) & 1) * 128 + (r & 7) * 16 +
                    (k & 3) * 4);
}

// Shared-memory matrix descriptor (sm_100 family): start address, leading and
// stride byte offsets (all >> 4), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)(128u >> 4) << 16;
  d |= (uint64_t)(256u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor of kind::tf32: FP32 accumulator, TF32 A and B, both
// K-major, N = 256, M = 128.
constexpr uint32_t kTcIdesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(kTcN >> 3) << 17) |
                              ((uint32_t)(kTcM >> 4) << 24);

__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity, uint32_t limit) {
  for (uint32_t it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 " selp.b32 %0, 1, 0, p;\n}\n" : "=r"(done) : "r"(addr), "r"(parity) : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, "
      "%30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// One piece: up to 128 consecutive sorted points of one instance and the cell
// box ("union") around them that holds every query's own block.
//   x  first sorted position
//   y  points (bits 0-7), extent - 1 of the union per axis (4 bits each from bit 8)
//   z, w  first cell of the union, 16 bits per axis (B <= 15 bits with 4 axes)
constexpr int kTcUnion = 256;  // cells of a union at most
__device__ __forceinline__ uint4 pack_piece(uint32_t q0, uint32_t cnt, const int* lo, const int* w) {
  return make_uint4(q0,
                    cnt | (uint32_t)(w[0] - 1) << 8 | (uint32_t)(w[1] - 1) << 12 | (uint32_t)(w[2] - 1) << 16 |
                        (uint32_t)(w[3] - 1) << 20,
                    (uint32_t)lo[0] | (uint32_t)lo[1] << 16, (uint32_t)lo[2] | (uint32_t)lo[3] << 16);
}
struct Piece {
  uint32_t q0, cnt;
  Union<4> u;
};
__device__ __forceinline__ Piece unpack_piece(uint4 r, uint32_t n) {
  Piece p;
  p.q0 = r.x < n ? r.x : 0u;
  p.cnt = min(min(r.y & 255u, (uint32_t)kTcM), n - p.q0);
  p.u.ncell = 1;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    p.u.w[a] = (int)((r.y >> (8 + 4 * a)) & 15u) + 1;
    p.u.inv[a] = (65536 + p.u.w[a] - 1) / p.u.w[a];
    p.u.lo[a] = (int)(((a < 2 ? r.z : r.w) >> (16 * (a & 1))) & 0xffffu);
    p.u.ncell *= p.u.w[a];
  }
  p.u.ncell = min(p.u.ncell, kTcUnion);
  return p;
}

// The piece list: one warp per 128 consecutive sorted points of an instance
// takes their cells in order and adds a cell to the current piece as long as
// the union grows by no more cells than the block of a piece of its own would
// cost (a piece's work is its candidates, whatever rows it fills): cells of a
// few points share the 128 rows of one MMA.
// Also gives every point density 0 and its order key first, or, for the near
// phase, lambda = -1: a CTA that gives up on a wait (the MMA did not complete
// in time) leaves its pieces unwritten, and the later phases must still see
// one valid key per position and dependent pointers that form no cycle.
__global__ void __launch_bounds__(256)
k_tc_pieces(HashInfo* hi, const unsigned long long* __restrict__ scode, ClassView cv,
            const CutGeom* __restrict__ cuts, uint4* __restrict__ pieces, const uint32_t* __restrict__ sid,
            MultiCut mc, unsigned long long* __restrict__ skey, int32_t* __restrict__ lambda, uint32_t min_fill) {
  if (!tensor_fill(cv.N, hi, min_fill)) return;
  const int lane = threadIdx.x & 31;
  const int S = cv.cls->S, ib = cv.cls->ib;
  const uint32_t nw = gridDim.x * 8u;
  for (uint32_t c = blockIdx.x * 8u + (threadIdx.x >> 5); c < cv.nchunk; c += nw) {
    uint32_t inst, p0, end;
    cv.chunk(c, inst, p0, end);
    const InstDev I = cv.instance(inst);
    if (p0 + lane < end) {
      const uint32_t id = sid[p0 + lane];
      for (int j = 0; j < mc.m; ++j) mc.rho[j][id] = 0;
      if (skey) skey[p0 + lane] = order_key(0, id);
      if (lambda) lambda[id] = -1;
    }
    if (((p0 - I.start) & (uint32_t)(kTcM - 1)) != 0u) continue;
    const CutGeom& C = cuts[inst];
    const int shift = 4 * C.k, R = C.R;
    const int cmax = (1 << (cv.geom[inst].B - C.k)) - 1;
    const int cnt = (int)min((uint32_t)kTcM, end - p0);
    unsigned long long cell[4];
    uint32_t head[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t p = p0 + 32u * i + lane;
      const bool in = 32 * i + lane < cnt;
      cell[i] = in ? key_code(scode[p], S, ib) >> shift : ~0ull;
      const unsigned long long prev =
          in && (32 * i + lane) > 0 ? key_code(scode[p - 1], S, ib) >> shift : ~0ull;
      head[i] = __ballot_sync(kFull, in && cell[i] != prev);
    }
    int s = 0, npc = 0;  // first point of the piece being built
    int lo[4], hi4[4];   // its cells' box
    int size = 0;
    uint4 mine[4];       // lane l holds pieces l, l + 32, ..
    auto close = [&](int e) {
      int ul[4], uw[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        ul[a] = max(lo[a] - R, 0);
        uw[a] = min(hi4[a] + R, cmax) - ul[a] + 1;
      }
      const uint4 r = pack_piece(p0 + (uint32_t)s, (uint32_t)(e - s), ul, uw);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (npc == 32 * i + lane) mine[i] = r;
      ++npc;
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t m = head[i];
      while (m) {
        const int l = __ffs((int)m) - 1;
        m &= m - 1u;
        const int at = 32 * i + l;
        uint32_t cc[4];
        unmorton<4>(__shfl_sync(kFull, cell[i], l), cc);
        int own = 1, both = 1;
        bool narrow = true;
        int nl[4], nh[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          own *= min((int)cc[a] + R, cmax) - max((int)cc[a] - R, 0) + 1;
          nl[a] = size ? min(lo[a], (int)cc[a]) : (int)cc[a];
          nh[a] = size ? max(hi4[a], (int)cc[a]) : (int)cc[a];
          const int w = min(nh[a] + R, cmax) - max(nl[a] - R, 0) + 1;
          narrow &= w <= 16;
          both = narrow ? both * w : 1 << 20;
        }
        if (size && !(narrow && both <= kTcUnion && both <= size + own)) {
          close(at);
          s = at;
          size = own;
#pragma unroll
          for (int a = 0; a < 4; ++a) lo[a] = hi4[a] = (int)cc[a];
        } else {
          size = both;
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            lo[a] = nl[a];
            hi4[a] = nh[a];
          }
        }
      }
    }
    close(cnt);
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(&hi->npieces, (uint32_t)npc);
    base = __shfl_sync(kFull, base, 0);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (32 * i + lane < npc) pieces[base + 32 * i + lane] = mine[i];
  }
}

// Run table of a union of up to kTcUnion cells (RunTable's layout).
struct TcRuns {
  uint32_t pre[kTcUnion + 1];
  uint32_t start[kTcUnion];
};

// All warps look the union's cells up (one cell per thread: 256 threads), the
// non-empty runs in cell order; returns their number.  Block-wide.
__device__ __forceinline__ int tc_runs(const Union<4>& u, const unsigned long long* __restrict__ hkeys,
                                       const uint2* __restrict__ hvals, uint32_t hmask, unsigned long long hb,
                                       uint32_t n, TcRuns& rt, uint32_t (*wsum)[2], uint32_t q0 = 0u,
                                       uint32_t* rot = nullptr) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t st = 0, len = 0;
  if (tid < u.ncell) {
    int rem = tid;
    uint32_t c[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int q = rem / u.w[a];
      c[a] = (uint32_t)(u.lo[a] + rem - q * u.w[a]);
      rem = q;
    }
    const uint2 run = clip_run(hash_find(hkeys, hvals, hmask, hb | morton<4>(c)), n);
    st = run.x;
    len = run.y - run.x;
  }
  const unsigned m = __ballot_sync(kFull, len > 0);
  uint32_t incl = len;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t t = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) {
    wsum[warp][0] = (uint32_t)__popc(m);
    wsum[warp][1] = incl;
  }
  __syncthreads();
  uint32_t slot0 = 0, pre0 = 0, nr = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kTcThreads / 32; ++w) {
    if (w < warp) {
      slot0 += wsum[w][0];
      pre0 += wsum[w][1];
    }
    nr += wsum[w][0];
    total += wsum[w][1];
  }
  if (len > 0) {
    const uint32_t slot = slot0 + (uint32_t)__popc(m & ((1u << lane) - 1u));
    rt.pre[slot] = pre0 + incl - len;
    rt.start[slot] = st;
    // where position q0 stands in the candidate list
    if (rot && q0 - st < len) *rot = pre0 + incl - len + (q0 - st);
  }
  if (tid == 0) rt.pre[nr] = total;
  __syncthreads();
  return (int)nr;
}

// Sorted position of candidate e of the run table.
__device__ __forceinline__ uint32_t tc_candidate(const TcRuns& rt, int nr, uint32_t e) {
  int lo = 0, hi = nr - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (rt.pre[mid] <= e) lo = mid;
    else hi = mid - 1;
  }
  return rt.start[lo] + (e - rt.pre[lo]);
}

struct TcSmem {
  float a[kTcM * 32];           // query rows
  float b[kTcN * 32];           // candidate rows
  float c[kTcN * 8];            // candidate coordinates (original)
  float cmax[kTcN / 32];        // per 32 columns (the rows one warp stages): largest |c'|^2
  int cnt[kMultiCuts][kTcM];       // per query: the two column halves' counts
  TcRuns rt;
  uint32_t wsum[kTcThreads / 32][2];
  unsigned long long mbar;
  uint32_t tmem;
  uint32_t item;
};

// Writes KS * 8 operand values of row r, 16 bytes at a time.
template <int ROWS, int KS>
__device__ __forceinline__ void put_row32(float* op, int r, const float* v) {
#pragma unroll
  for (int k = 0; k < 8 * KS; k += 4)
    *reinterpret_cast<float4*>((char*)op + op_off<ROWS>(r, k)) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
}

// Densities of up to kMultiCuts cutoffs that share the block geometry `geo`: one
// product per pair, compared with every cutoff's threshold.
//   a = [q_hi, q_hi, q_lo | (1 + e)|q|^2 hi, lo | 1, 1]
//   b = [c_hi, c_lo, c_hi | 1, 1 | (1 + e)|c|^2 hi, lo]      (c = -2 c')
// in 3 D + 4 <= 32 columns (the three products of the TF32 split laid side by
// side: 3 or 4 K = 8 steps instead of 6 with separate operands), so the
// accumulator is s + e (|q|^2 + |c|^2).
template <int D, int M>
__global__ void __launch_bounds__(kTcThreads, 2)
k_density_tc(const float* __restrict__ spts, const unsigned long long* __restrict__ scode,
             const uint32_t* __restrict__ sid, ClassView cv, const CutGeom* __restrict__ geo, HashInfo* hi,
             const unsigned long long* __restrict__ hkeys, const uint2* __restrict__ hvals,
             const uint4* __restrict__ pieces, MultiCut mc, unsigned long long* __restrict__ skey, Counters* ctr,
             uint32_t poll_limit, uint32_t min_fill) {
  if (!tensor_fill(cv.N, hi, min_fill)) return;
  constexpr int DP = 8;
  constexpr int KS = (3 * D + 4 + 7) / 8;  // K = 8 steps
  extern __shared__ __align__(128) unsigned char tc_smem_raw[];
  TcSmem& sm = *reinterpret_cast<TcSmem*>(tc_smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = cv.cls->S, ib = cv.cls->ib;
  const uint32_t hmask = hi->hmask;
  const uint32_t npieces = hi->npieces;
  const uint32_t n = cv.N;
  const uint32_t mbar = smem_addr(&sm.mbar);

  if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(mbar) : "memory");
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_addr(&sm.tmem)), "r"(kTcN) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sm.tmem;
  // warp w reads accumulator lanes 32 (w % 4) .. (the rows of queries
  // 32 (w % 4) ..) and the columns of half w / 4
  const int qrow = (warp & 3) * 32 + lane;
  const int chalf = warp >> 2;
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(chalf * (kTcN / 2));
  uint32_t phase = 0;
  unsigned long long band = 0, pairs = 0;
  bool stop = false;

  while (!stop) {
    if (tid == 0) sm.item = atomicAdd(&hi->work, 1u);
    __syncthreads();
    const uint32_t item = sm.item;
    if (item >= npieces) break;
    const Piece pc = unpack_piece(pieces[item], n);
    uint32_t inst = key_inst(scode[pc.q0], S, ib);
    if (inst >= cv.ninst) inst = 0;
    const unsigned long long hb = ib ? ((unsigned long long)inst << S) : 0ull;
    const int nr = tc_runs(pc.u, hkeys, hvals, hmask, hb, n, sm.rt, sm.wsum);
    const uint32_t total = sm.rt.pre[nr];
    float t_in[M], tw[M];
    f32x2 nthr[M];  // -(1 - e) t_in, rounded so that the threshold is not above it
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const CutGeom& C = mc.cut[j][inst];
      t_in[j] = C.t_in;
      tw[j] = __fsub_ru(C.t_out, C.t_in);
      const float t = -__fmul_rd(C.t_in, 1.f - kTcErr);
      nthr[j] = pack2(t, t);
    }
    if (tid == 0) pairs += (unsigned long long)pc.cnt * total;
    // query rows: this thread's point, relative to the piece's first point
    const uint32_t q = pc.q0 + (uint32_t)qrow;
    const bool inq = qrow < (int)pc.cnt;
    const Pt<DP> o = load_pt<DP>(spts, pc.q0);
    Pt<DP> me;
#pragma unroll
    for (int a = 0; a < DP; ++a) me.x[a] = 0.f;
    if (inq) me = load_pt<DP>(spts, q);
    float nq = 0.f;
    {
      float row[8 * KS];
#pragma unroll
      for (int k = 0; k < 8 * KS; ++k) row[k] = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const float t = inq ? me.x[a] - o.x[a] : 0.f;
        nq = fmaf(t, t, nq);
        const float h = tf32_rna(t);
        row[a] = row[D + a] = h;
        row[2 * D + a] = tf32_rna(t - h);
      }
      const float w = nq * (1.f + kTcErr);
      row[3 * D] = tf32_rna(w);
      row[3 * D + 1] = tf32_rna(w - row[3 * D]);
      row[3 * D + 2] = row[3 * D + 3] = 1.f;
      if (chalf == 0) put_row32<kTcM, KS>(sm.a, qrow, row);
    }
    if (tid < kTcM) {
#pragma unroll
      for (int j = 0; j < M; ++j) sm.cnt[j][tid] = 0;
    }
    int32_t cnt[M];
#pragma unroll
    for (int j = 0; j < M; ++j) cnt[j] = 0;
    // This thread's candidate of the tile starting at w (row tid), loaded
    // one tile ahead: the next tile's load is issued right after this
    // tile's MMA, so it is in flight during the MMA and the epilogue.
    auto fetch = [&](uint32_t w) {
      Pt<DP> x;
#pragma unroll
      for (int a = 0; a < DP; ++a) x.x[a] = 0.f;
      const uint32_t e = w + (uint32_t)tid;
      if (e < total) x = load_pt<DP>(spts, tc_candidate(sm.rt, nr, e));
      return x;
    };
    Pt<DP> xnext = fetch(0);
    for (uint32_t w0 = 0; w0 < total && !stop; w0 += kTcN) {
      {  // candidate rows: one per thread
        const Pt<DP> x = xnext;
        const bool in = w0 + (uint32_t)tid < total;
        float row[8 * KS];
#pragma unroll
        for (int k = 0; k < 8 * KS; ++k) row[k] = 0.f;
        float nc = 0.f;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          const float t = in ? x.x[a] - o.x[a] : 0.f;
          nc = fmaf(t, t, nc);
          const float h = tf32_rna(-2.f * t);
          row[a] = row[2 * D + a] = h;
          row[D + a] = tf32_rna(-2.f * t - h);
        }
        row[3 * D] = row[3 * D + 1] = 1.f;
        const float w = in ? nc * (1.f + kTcErr) : kTcFar;
        row[3 * D + 2] = tf32_rna(w);
        row[3 * D + 3] = tf32_rna(w - row[3 * D + 2]);
        const float m = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(nc)));
        if (lane == 0) sm.cmax[warp] = m;
        put_row32<kTcN, KS>(sm.b, tid, row);
        float4* cs = reinterpret_cast<float4*>(sm.c + tid * DP);
        cs[0] = make_float4(x.x[0], x.x[1], x.x[2], x.x[3]);
        cs[1] = make_float4(x.x[4], x.x[5], x.x[6], x.x[7]);
      }
      // operands written by the threads -> visible to the tensor core
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tid == 0) {
        const uint32_t ab = smem_addr(sm.a), bb = smem_addr(sm.b);
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          const uint64_t ad = smem_desc(ab + ks * (kTcM * 32));
          const uint64_t bd = smem_desc(bb + ks * (kTcN * 32));
          asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %4, 0;\n"
                       " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, q;\n}\n"
                       :: "r"(tmem), "l"(ad), "l"(bd), "r"(kTcIdesc), "r"(ks ? 1u : 0u) : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                     :: "r"(mbar) : "memory");
      }
      if (w0 + kTcN < total) xnext = fetch(w0 + kTcN);
      const bool ok = mbar_wait(mbar, phase, poll_limit);
      phase ^= 1u;
      if (__syncthreads_or(!ok)) {  // the MMA did not finish in time: record and stop
        if (tid == 0) set_status(cv.cls->status, kStatusTimeout);
        // let the MMA in flight finish (the full limit, whatever poll_limit
        // was) before tensor memory is freed and the CTA exits
        mbar_wait(mbar, phase ^ 1u, kTcWaitLimit);
        stop = true;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int ncol = (int)min((uint32_t)kTcN, total - w0);
      for (int cl = 0; cl < kTcN / 2; cl += 32) {
        const int cb = chalf * (kTcN / 2) + cl;  // first column of this load
        if (cb >= ncol) break;                   // warp-uniform
        if ((warp & 3) * 32 >= (int)pc.cnt) break;  // no query in this warp's rows
        float v[32];
        tmem_ld32(trow + (uint32_t)cl, v);
        const float cm = sm.cmax[cb >> 5];
#pragma unroll
        for (int j = 0; j < M; ++j) {
          // acc - (1 - e) t_in = s + E - t_in with E = e (|q|^2 + |c|^2 +
          // t_in): negative is counted; at or above +0 and at most W =
          // (t_out - t_in) + 1.25 E (largest candidate norm of the 32
          // columns, rounded up) is recounted in binary64; above W the pair
          // is certainly farther than t_out.  The subtraction's sign is
          // exact.  One funnel shift per element collects the signs, one
          // unsigned minimum over the bit patterns finds the band.
          const float W = __fadd_ru(
              tw[j], __fmul_ru(1.25f * kTcErr, __fadd_ru(__fadd_ru(nq, cm), t_in[j])));
          const uint32_t wbits = __float_as_uint(W);
          uint32_t sg = 0, lowest = 0xffffffffu;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const f32x2 x = add2(pack2(v[2 * i], v[2 * i + 1]), nthr[j]);
            const uint32_t x0 = __float_as_uint(lo2(x)), x1 = __float_as_uint(hi2(x));
            sg = __funnelshift_l(x0, sg, 1);
            sg = __funnelshift_l(x1, sg, 1);
            lowest = min(lowest, min(x0, x1));
          }
          if (inq) {
            cnt[j] += __popc(sg);
            if (lowest <= wbits) {
              // band pairs: the float32 filter on the original coordinates,
              // the canonical binary64 distance inside its own (far narrower)
              // band; one loop over a column mask keeps the code small
              uint32_t bm = 0;
#pragma unroll
              for (int i = 0; i < 32; ++i)
                bm |= (__float_as_uint(v[i] + lo2(nthr[j])) <= wbits) ? (1u << i) : 0u;
              if (ncol - cb < 32) bm &= (1u << (ncol - cb)) - 1u;
              const float t_out = mc.cut[j][inst].t_out;
#pragma unroll 1
              while (bm) {
                const int i = __ffs((int)bm) - 1;
                bm &= bm - 1u;
                const float4* cs = reinterpret_cast<const float4*>(sm.c + (cb + i) * DP);
                const float4 c0 = cs[0], c1 = cs[1];
                const Pt<DP> x{{c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w}};
                const float s32 = dist32<DP, D>(me, x);
                if (s32 <= t_in[j]) {
                  ++cnt[j];
                } else if (s32 <= t_out) {
                  ++band;
                  cnt[j] += dist64<DP, D>(me, x) <= mc.cut[j][inst].dc2 ? 1 : 0;
                }
              }
            }
          }
        }
      }
      // every read of the accumulator and the operands done before the next tile
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
    }
    // the two halves of each query's counts
    if (inq) {
#pragma unroll
      for (int j = 0; j < M; ++j) atomicAdd(&sm.cnt[j][qrow], cnt[j]);
    }
    __syncthreads();
    if (inq && chalf == 0 && !stop) {
      const uint32_t id = sid[q];
#pragma unroll
      for (int j = 0; j < M; ++j) mc.rho[j][id] = sm.cnt[j][qrow];
      if (skey) skey[q] = order_key(sm.cnt[0][qrow], id);
    }
    __syncthreads();
  }
  // release the tensor memory
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(kTcN) : "memory");
  for (int o = 16; o > 0; o >>= 1) band += __shfl_xor_sync(kFull, band, o);
  if (lane == 0 && band) atomicAdd(&ctr->band_pairs, band);
  if (tid == 0 && pairs) atomicAdd(&ctr->pairs, pairs);
}

// Dynamic shared memory per CTA: at least the layout, and enough that no
// more than two CTAs share an SM (each holds kTcN of the 512 tensor-memory
// columns for its whole life, so a third would wait for one to finish).
constexpr size_t kTcSmemBytes = sizeof(TcSmem) > 100 * 1024 ? sizeof(TcSmem) : 100 * 1024;
static_assert(sizeof(TcSmem) <= 110 * 1024, "two CTAs per SM");

// ---------------------------------------------------------------------------
// The near phase of the dependent search (Definitions 2-3) on the tensor
// cores: the same pieces and tiles, with |q|^2 and |c|^2 unscaled so that the
// accumulator is within E = e (|q'|^2 + |c'|^2) of the exact real squared
// distance.  Each query keeps the smallest and second smallest float32 distance
// among its higher candidates, evaluated from the coordinates as everywhere
// else; the accumulator only decides which candidates are looked at: one whose
// accumulator exceeds tt = band(s1) (1 + 2^-19) + E has a float32 distance above
// band(s1), so it is neither the winner nor within its band.  Per 32 columns
// one compare of the densities (a superset of "higher": ties are settled by the
// full key later) and one minimum per column give the smallest accumulator
// that could matter; almost all groups end there.  The tiles start at the
// piece's own points, so tt is small from the first tile on.
// The query is settled as in the CUDA-core layouts (band(s1) below the block's
// far bound, no second candidate within the band), else queued for the far
// phase.  7-D, 2e6 points, 17 per cell: 12.5 ms a cutoff, 17.3 with every column
// compared and ranked on its accumulator.

struct TcNearSmem {
  float a[kTcM * 32];
  float b[kTcN * 32];
  float c[kTcN * 8];             // candidate coordinates (original)
  unsigned long long key[kTcN];  // order key per column (0: padding)
  uint32_t rho[kTcN];            // its density word
  float cmax[kTcN / 32];
  // the second column half's per-row results, merged by the first half
  float s1[kTcM], s2[kTcM];
  uint32_t o1[kTcM];
  TcRuns rt;
  uint32_t wsum[kTcThreads / 32][2];
  unsigned long long mbar;
  uint32_t tmem;
  uint32_t item;
  uint32_t rot;  // the piece's first point in the candidate list
};

__device__ __forceinline__ float tc_band(float s, float mul, float add) {
  return __fadd_ru(__fmul_ru(s, mul), add);
}

// Coordinates of point `o` of an instance in the caller's input.
__device__ __forceinline__ Pt<8> tc_caller_pt(const void* __restrict__ pts, int dtype, uint64_t coord,
                                              int d, uint32_t o) {
  Pt<8> p;
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    float v = 0.f;
    if (a < d) {
      const size_t e = coord + (size_t)o * d + a;
      v = dtype == 0 ? (float)__ldg((const int32_t*)pts + e) : __ldg((const float*)pts + e);
    }
    p.x[a] = v;
  }
  return p;
}

template <int D>
__global__ void __launch_bounds__(kTcThreads, 2)
k_dep_near_tc(const float* __restrict__ spts, const unsigned long long* __restrict__ scode,
              const unsigned long long* __restrict__ skey, ClassView cv, int32_t rho_skip, const void* __restrict__ pts, int dtype,
              const CutGeom* __restrict__ cuts, HashInfo* hi,
              const unsigned long long* __restrict__ hkeys, const uint2* __restrict__ hvals,
              const uint4* __restrict__ pieces, int32_t* __restrict__ lambda,
              double* __restrict__ delta, FarQueue fq, Counters* ctr, uint32_t poll_limit,
              uint32_t min_fill) {
  if (!tensor_fill(cv.N, hi, min_fill)) return;
  constexpr int DP = 8;
  constexpr int KS = (3 * D + 4 + 7) / 8;  // K = 8 steps
  extern __shared__ __align__(128) unsigned char tcn_smem_raw[];
  TcNearSmem& sm = *reinterpret_cast<TcNearSmem*>(tcn_smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = cv.cls->S, ib = cv.cls->ib;
  const uint32_t hmask = hi->hmask;
  const uint32_t npieces = hi->npieces;
  const uint32_t n = cv.N;
  const uint32_t mbar = smem_addr(&sm.mbar);
  const uint32_t lanemask_lt = (1u << lane) - 1u;

  if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(mbar) : "memory");
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_addr(&sm.tmem)), "r"(kTcN) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sm.tmem;
  const int qrow = (warp & 3) * 32 + lane;
  const int chalf = warp >> 2;
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(chalf * (kTcN / 2));
  uint32_t phase = 0;
  bool stop = false;

  while (!stop) {
    if (tid == 0) sm.item = atomicAdd(&hi->work, 1u);
    __syncthreads();
    const uint32_t item = sm.item;
    if (item >= npieces) break;
    const Piece pc = unpack_piece(pieces[item], n);
    uint32_t inst = key_inst(scode[pc.q0], S, ib);
    if (inst >= cv.ninst) inst = 0;
    const CutGeom& C = cuts[inst];
    const InstDev I = cv.instance(inst);
    const float bmul = C.band_mul, badd = C.band_add, far32 = C.far32;
    const int32_t skip_below = max(rho_skip, C.skip);
    const unsigned long long hb = ib ? ((unsigned long long)inst << S) : 0ull;
    if (tid == 0) sm.rot = 0u;
    __syncthreads();
    const int nr = tc_runs(pc.u, hkeys, hvals, hmask, hb, n, sm.rt, sm.wsum, pc.q0, &sm.rot);
    const uint32_t total = sm.rt.pre[nr], rot = sm.rot;
    const uint32_t qp = pc.q0 + (uint32_t)qrow;
    const bool inq = qrow < (int)pc.cnt;
    const Pt<DP> o = load_pt<DP>(spts, pc.q0);
    Pt<DP> me;
#pragma unroll
    for (int a = 0; a < DP; ++a) me.x[a] = 0.f;
    unsigned long long K = ~0ull;
    if (inq) {
      me = load_pt<DP>(spts, qp);
      K = skey[qp];
    }
    const bool act = inq && (int32_t)(K >> 32) >= skip_below;
    float nq = 0.f;
    {
      float row[8 * KS];
#pragma unroll
      for (int i = 0; i < 8 * KS; ++i) row[i] = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const float t = inq ? me.x[a] - o.x[a] : 0.f;
        nq = fmaf(t, t, nq);
        const float h = tf32_rna(t);
        row[a] = row[D + a] = h;
        row[2 * D + a] = tf32_rna(t - h);
      }
      row[3 * D] = tf32_rna(nq);
      row[3 * D + 1] = tf32_rna(nq - row[3 * D]);
      row[3 * D + 2] = row[3 * D + 3] = 1.f;
      if (chalf == 0) put_row32<kTcM, KS>(sm.a, qrow, row);
    }
    const uint32_t rq = act ? (uint32_t)(K >> 32) : 0xffffffffu;
    float s1 = INFINITY, s2 = INFINITY, top = INFINITY;  // top = band(s1) (1 + 2^-19)
    uint32_t o1 = 0xffffffffu;
    auto fetch = [&](uint32_t w, unsigned long long& kc) {
      Pt<DP> x;
#pragma unroll
      for (int a = 0; a < DP; ++a) x.x[a] = 0.f;
      kc = 0ull;
      const uint32_t e = w + (uint32_t)tid;
      if (e < total) {
        uint32_t at = e + rot;  // < 2^32: both below the class's points
        if (at >= total) at -= total;
        const uint32_t src = tc_candidate(sm.rt, nr, at);
        x = load_pt<DP>(spts, src);
        kc = skey[src];
      }
      return x;
    };
    unsigned long long knext;
    Pt<DP> xnext = fetch(0, knext);
    for (uint32_t w0 = 0; w0 < total && !stop; w0 += kTcN) {
      {
        const bool in = w0 + (uint32_t)tid < total;
        float row[8 * KS];
#pragma unroll
        for (int i = 0; i < 8 * KS; ++i) row[i] = 0.f;
        float nc = 0.f;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          const float t = in ? xnext.x[a] - o.x[a] : 0.f;
          nc = fmaf(t, t, nc);
          const float h = tf32_rna(-2.f * t);
          row[a] = row[2 * D + a] = h;
          row[D + a] = tf32_rna(-2.f * t - h);
        }
        row[3 * D] = row[3 * D + 1] = 1.f;
        const float w = in ? nc : kTcFar;
        row[3 * D + 2] = tf32_rna(w);
        row[3 * D + 3] = tf32_rna(w - row[3 * D + 2]);
        sm.key[tid] = in ? knext : 0ull;
        sm.rho[tid] = in ? (uint32_t)(knext >> 32) : 0u;
        float4* cs = reinterpret_cast<float4*>(sm.c + tid * DP);
        cs[0] = make_float4(xnext.x[0], xnext.x[1], xnext.x[2], xnext.x[3]);
        cs[1] = make_float4(xnext.x[4], xnext.x[5], xnext.x[6], xnext.x[7]);
        const float m = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(nc)));
        if (lane == 0) sm.cmax[warp] = m;
        put_row32<kTcN, KS>(sm.b, tid, row);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tid == 0) {
        const uint32_t ab = smem_addr(sm.a), bb = smem_addr(sm.b);
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          const uint64_t ad = smem_desc(ab + ks * (kTcM * 32));
          const uint64_t bd = smem_desc(bb + ks * (kTcN * 32));
          asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %4, 0;\n"
                       " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, q;\n}\n"
                       :: "r"(tmem), "l"(ad), "l"(bd), "r"(kTcIdesc), "r"(ks ? 1u : 0u) : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                     :: "r"(mbar) : "memory");
      }
      if (w0 + kTcN < total) xnext = fetch(w0 + kTcN, knext);
      const bool ok = mbar_wait(mbar, phase, poll_limit);
      phase ^= 1u;
      if (__syncthreads_or(!ok)) {  // the MMA did not finish in time: record and stop
        if (tid == 0) set_status(cv.cls->status, kStatusTimeout);
        mbar_wait(mbar, phase ^ 1u, kTcWaitLimit);  // the MMA in flight, before TMEM is freed
        stop = true;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int ncol = (int)min((uint32_t)kTcN, total - w0);
      for (int cl = 0; cl < kTcN / 2; cl += 32) {
        const int cb = chalf * (kTcN / 2) + cl;
        if (cb >= ncol) break;                       // warp-uniform
        if ((warp & 3) * 32 >= (int)pc.cnt) break;  // no query in this warp's rows
        float v[32];
        tmem_ld32(trow + (uint32_t)cl, v);
        float mn = INFINITY;
        const uint4* rh = reinterpret_cast<const uint4*>(sm.rho + cb);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 r4 = rh[i];
          mn = fminf(mn, r4.x >= rq ? v[4 * i] : INFINITY);
          mn = fminf(mn, r4.y >= rq ? v[4 * i + 1] : INFINITY);
          mn = fminf(mn, r4.z >= rq ? v[4 * i + 2] : INFINITY);
          mn = fminf(mn, r4.w >= rq ? v[4 * i + 3] : INFINITY);
        }
        const float tt = __fadd_ru(top, __fmul_ru(kTcErr, __fadd_ru(nq, sm.cmax[cb >> 5])));
        if (act && mn <= tt) {
          uint32_t bm = 0;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint4 r4 = rh[i];
            bm |= (v[4 * i] <= tt && r4.x >= rq) ? 1u << (4 * i) : 0u;
            bm |= (v[4 * i + 1] <= tt && r4.y >= rq) ? 2u << (4 * i) : 0u;
            bm |= (v[4 * i + 2] <= tt && r4.z >= rq) ? 4u << (4 * i) : 0u;
            bm |= (v[4 * i + 3] <= tt && r4.w >= rq) ? 8u << (4 * i) : 0u;
          }
#pragma unroll 1
          while (bm) {
            const int j = __ffs((int)bm) - 1;
            bm &= bm - 1u;
            const unsigned long long kc = sm.key[cb + j];
            if (kc <= K) continue;
            const float4* cs = reinterpret_cast<const float4*>(sm.c + (cb + j) * DP);
            const float4 c0 = cs[0], c1 = cs[1];
            const Pt<DP> x{{c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w}};
            const float d32 = dist32<DP, D>(me, x);
            s2 = fminf(s2, fmaxf(s1, d32));
            if (d32 < s1) {
              s1 = d32;
              o1 = key_id(kc);
            }
          }
          top = __fmul_ru(tc_band(s1, bmul, badd), 1.f + 0x1p-19f);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
    }
    // the two column halves of each query, then settle it or queue it
    if (chalf == 1) {
      sm.s1[qrow] = s1;
      sm.s2[qrow] = s2;
      sm.o1[qrow] = o1;
    }
    __syncthreads();
    bool push = false;
    if (chalf == 0 && inq && !stop) {
      const float t1 = sm.s1[qrow];
      s2 = fminf(fminf(s2, sm.s2[qrow]), fmaxf(s1, t1));
      o1 = t1 < s1 ? sm.o1[qrow] : o1;
      s1 = fminf(s1, t1);
      const uint32_t id = key_id(K);
      if (!act) {
        lambda[id] = -1;
        delta[id] = __longlong_as_double(0x7ff8000000000000ll);  // NaN: skipped
      } else {
        bool settled = false;
        if (o1 != 0xffffffffu) {
          const float bnd = tc_band(s1, bmul, badd);
          settled = bnd < far32 && s2 > bnd;
        }
        if (settled) {
          const uint32_t ol = o1 - (uint32_t)I.out;
          lambda[id] = (int32_t)ol;
          delta[id] = sqrt(dist64<DP>(me, tc_caller_pt(pts, dtype, I.coord, I.d, ol)));
        } else {
          push = true;
        }
      }
    }
    const unsigned pm = __ballot_sync(kFull, push);
    uint32_t base = 0;
    if (lane == 0 && pm) base = atomicAdd(&ctr->queue_n, (unsigned)__popc(pm));
    base = __shfl_sync(kFull, base, 0);
    if (push) {
      const uint32_t slot2 = base + __popc(pm & lanemask_lt);
      fq.pos[slot2] = qp;
      fq.s1[slot2] = s1;
    }
    __syncthreads();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(kTcN) : "memory");
}

constexpr size_t kTcNearSmemBytes =
    sizeof(TcNearSmem) > 100 * 1024 ? sizeof(TcNearSmem) : 100 * 1024;
static_assert(sizeof(TcNearSmem) <= 110 * 1024, "two CTAs per SM");

}  // namespace

// One-time kernel attribute setup of the instantiations for `d` dimensions.
template <int D>
static void tc_attr() {
  constexpr int kDevs = 64;
  static bool done[kDevs] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs || done[dev]) return;
  auto set = [](auto kern, size_t b) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b);
  };
  set(k_density_tc<D, 1>, kTcSmemBytes);
  set(k_density_tc<D, 2>, kTcSmemBytes);
  set(k_density_tc<D, 3>, kTcSmemBytes);
  set(k_density_tc<D, 4>, kTcSmemBytes);
  set(k_dep_near_tc<D>, kTcNearSmemBytes);
  done[dev] = true;
}

template <int D>
static void density_tc_d(const float* spts, const unsigned long long* scode, const uint32_t* sid,
                         const ClassView& cv, const CutGeom* geo, HashInfo* hi, const unsigned long long* hkeys,
                         const uint2* hvals, const uint4* pieces, const MultiCut& mc, unsigned long long* skey,
                         Counters* ctr, uint32_t min_fill, cudaStream_t st) {
  tc_attr<D>();
  const uint32_t poll = wait_limit(kTcWaitLimit);
  auto go = [&](auto kern) {  // two resident CTAs per SM take the pieces one by one
    kern<<<sm_count() * 2u, kTcThreads, kTcSmemBytes, st>>>(spts, scode, sid, cv, geo, hi, hkeys, hvals, pieces, mc,
                                                            skey, ctr, poll, min_fill);
  };
  if (mc.m == 1) go(k_density_tc<D, 1>);
  else if (mc.m == 2) go(k_density_tc<D, 2>);
  else if (mc.m == 3) go(k_density_tc<D, 3>);
  else go(k_density_tc<D, 4>);
}

static void tc_pieces(const unsigned long long* scode, const uint32_t* sid, const ClassView& cv, const CutGeom* geo,
                      HashInfo* hi, uint4* pieces, const MultiCut& mc, unsigned long long* skey, int32_t* lambda,
                      uint32_t min_fill, cudaStream_t st) {
  cudaMemsetAsync(&hi->work, 0, 2 * sizeof(uint32_t), st);  // work and npieces
  const uint64_t b = ((uint64_t)cv.nchunk + 7) / 8;
  const unsigned grid = (unsigned)(b < sm_count() * 16u ? b : sm_count() * 16u);
  k_tc_pieces<<<grid, 256, 0, st>>>(hi, scode, cv, geo, pieces, sid, mc, skey, lambda, min_fill);
}

void launch_density_tc(int d, const float* spts, const unsigned long long* scode, const uint32_t* sid,
                       const ClassView& cv, const CutGeom* geo, HashInfo* hi, const unsigned long long* hkeys,
                       const uint2* hvals, uint4* pieces, const MultiCut& mc, unsigned long long* skey,
                       Counters* ctr, uint32_t min_fill, cudaStream_t st) {
  if (cv.N == 0) return;
  tc_pieces(scode, sid, cv, geo, hi, pieces, mc, skey, nullptr, min_fill, st);
  if (d <= 5) density_tc_d<5>(spts, scode, sid, cv, geo, hi, hkeys, hvals, pieces, mc, skey, ctr, min_fill, st);
  else if (d == 6) density_tc_d<6>(spts, scode, sid, cv, geo, hi, hkeys, hvals, pieces, mc, skey, ctr, min_fill, st);
  else if (d == 7) density_tc_d<7>(spts, scode, sid, cv, geo, hi, hkeys, hvals, pieces, mc, skey, ctr, min_fill, st);
  else density_tc_d<8>(spts, scode, sid, cv, geo, hi, hkeys, hvals, pieces, mc, skey, ctr, min_fill, st);
  count_launches(2);
}

void launch_dep_near_tc(int d, const float* spts, const unsigned long long* scode, const uint32_t* sid,
                        const unsigned long long* skey, const ClassView& cv, int32_t rho_skip, const void* pts,
                        int dtype, const CutGeom* cuts, HashInfo* hi, const unsigned long long* hkeys,
                        const uint2* hvals, uint4* pieces, int32_t* lambda, double* delta, FarQueue q,
                        Counters* ctr, uint32_t min_fill, cudaStream_t st) {
  if (cv.N == 0) return;
  cudaMemsetAsync(&ctr->queue_n, 0, 2 * sizeof(unsigned int), st);  // queue_n and queue2_n
  tc_pieces(scode, sid, cv, cuts, hi, pieces, MultiCut{}, nullptr, lambda, min_fill, st);
  const unsigned grid = sm_count() * 2u;
  const uint32_t poll = wait_limit(kTcWaitLimit);
  auto go = [&](auto kern) {
    kern<<<grid, kTcThreads, kTcNearSmemBytes, st>>>(spts, scode, skey, cv, rho_skip, pts, dtype, cuts, hi, hkeys,
                                                     hvals, pieces, lambda, delta, q, ctr, poll, min_fill);
  };
  if (d <= 5) { tc_attr<5>(); go(k_dep_near_tc<5>); }
  else if (d == 6) { tc_attr<6>(); go(k_dep_near_tc<6>); }
  else if (d == 7) { tc_attr<7>(); go(k_dep_near_tc<7>); }
  else { tc_attr<8>(); go(k_dep_near_tc<8>); }
  count_launches(2);
}

}  // namespace dpc

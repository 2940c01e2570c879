// api.cu -- the C ABI (include/dpc.h): argument checks, the per-(device,
// stream) workspace, and the order in which the kernels run.
//
// The instances of a call are grouped into classes of equal padded dimension
// dp and gridded dimension g (at most five: (2,1), (2,2), (4,3), (4,4), (8,4)).  Each
// class runs as one unit, every kernel launched once for all its instances
// (dpc_device.cuh describes the layout):
//   binning   bbox -> grid setup -> sort keys -> radix sort -> gather
//   tree      radix tree over the sorted keys (dependent points only)
//   per cutoff
//     cells     occupied level-k cells -> hash
//     density   rho (Definition 1) + order keys
//     dependent maxkeys of the tree -> near phase -> far phase (Definitions 2-3)
//     labels    pointer jumping (Definitions 4-5)
// All on the caller's stream, with no host synchronization; a multi-instance
// class first copies its instance table and cutoffs to the device (one
// asynchronous copy per call from a page-locked staging buffer).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <string>
#include <mutex>
#include <utility>
#include <vector>

#include "../../include/dpc.h"
#include "internal.h"

namespace dpc {

long long g_kernel_launches = 0;

uint32_t wait_limit(uint32_t dflt) {
  const char* e = std::getenv("DPC_TEST_WAIT_LIMIT");
  if (!e || !*e) return dflt;
  char* end = nullptr;
  const unsigned long long v = std::strtoull(e, &end, 10);
  if (end == e) return dflt;
  return v < dflt ? (uint32_t)v : dflt;
}

bool dev_alloc(void** p, size_t bytes) {
  *p = nullptr;
  const char* e = std::getenv("DPC_WORKSPACE_LIMIT_BYTES");
  if (e && *e) {
    char* end = nullptr;
    const unsigned long long cap = std::strtoull(e, &end, 10);
    if (end != e && bytes > cap) return false;
  }
  if (cudaMalloc(p, bytes) != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return false;
  }
  return true;
}

unsigned sm_count() {
  constexpr int kDevs = 64;
  static int cached[kDevs] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs) {
    cudaGetLastError();
    return 1u;  // the launch that follows reports the error
  }
  if (cached[dev] <= 0) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
      cudaGetLastError();
      return 1u;
    }
    cached[dev] = v;
  }
  return (unsigned)cached[dev];
}

namespace {

constexpr size_t kAlign = 256;

inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

inline uint32_t next_pow2(uint64_t x) {
  uint64_t t = 16;
  while (t < x) t <<= 1;
  return (uint32_t)t;
}

inline int dp_of(int d) { return d <= 2 ? 2 : (d <= 4 ? 4 : 8); }
inline int g_of(int d) { return grid_dims(d); }

// ---- argument checks -----------------------------------------------------------

struct Inst {
  uint64_t n;
  int d;
  uint64_t pt_off;     // into result arrays
  uint64_t coord_off;  // into pts, in elements
};

int check_batch(const dpc_batch* b, std::vector<Inst>* insts, uint64_t* total) {
  if (!b || b->n_inst < 1 || !b->pt_offset || !b->dim || b->n_dcut < 1 || !b->d_cut) return DPC_ERR_ARG;
  if (b->pt_offset[0] != 0) return DPC_ERR_ARG;
  insts->clear();
  insts->reserve(b->n_inst);
  for (int i = 0; i < b->n_inst; ++i) {
    const int64_t lo = b->pt_offset[i], hi = b->pt_offset[i + 1];
    if (hi < lo) return DPC_ERR_ARG;
    const int d = b->dim[i];
    if (d < 1 || d > kMaxDim) return DPC_ERR_ARG;
    if (hi - lo >= (int64_t)0x7fffffff) return DPC_ERR_OVERFLOW;
    Inst in;
    in.n = (uint64_t)(hi - lo);
    in.d = d;
    in.pt_off = (uint64_t)lo;
    in.coord_off = b->coord_offset ? (uint64_t)b->coord_offset[i] : (uint64_t)lo * (uint64_t)d;
    if (b->coord_offset && b->coord_offset[i] < 0) return DPC_ERR_ARG;
    for (int c = 0; c < b->n_dcut; ++c) {
      const double dc = b->d_cut[(size_t)i * b->n_dcut + c];
      if (!std::isfinite(dc) || dc < 0.0) return DPC_ERR_ARG;
    }
    insts->push_back(in);
  }
  // output indices are 32-bit inside the library
  if (b->pt_offset[b->n_inst] >= (int64_t)0x7fffffff) return DPC_ERR_OVERFLOW;
  *total = (uint64_t)b->pt_offset[b->n_inst];
  return DPC_OK;
}

constexpr uint32_t kKnownFlags = DPC_PREC_MASK | DPC_FLAG_SYNC_CHECK | DPC_FLAG_PHASE_TIMES |
                                 DPC_FLAG_AUTOTUNE | DPC_FLAG_RADIUS_MASK | DPC_FLAG_GRAPH |
                                 DPC_FLAG_LAYOUT_MASK | DPC_FLAG_SKIP_NOISE |
                                 DPC_FLAG_NEAR_SHIFT_MASK;

int check_flags(uint32_t flags) {
  const uint32_t prec = flags & DPC_PREC_MASK;
  if (prec != DPC_PREC_FP64 && prec != DPC_PREC_FP32_CERT) return DPC_ERR_UNSUPPORTED;
  if (flags & ~kKnownFlags) return DPC_ERR_ARG;
  if (((flags & DPC_FLAG_RADIUS_MASK) >> 12) > 5) return DPC_ERR_ARG;
  if (((flags & DPC_FLAG_LAYOUT_MASK) >> 16) > 6) return DPC_ERR_ARG;
  if (((flags & DPC_FLAG_NEAR_SHIFT_MASK) >> 20) > 3) return DPC_ERR_ARG;
  return DPC_OK;
}

int status_to_code(int s) {
  if (s == 0) return DPC_OK;
  if (s & kStatusBadCoord) return DPC_ERR_DATA;
  // a wait that gave up leaves later results unreliable: report it first
  if (s & kStatusTimeout) return DPC_ERR_TIMEOUT;
  if (s & (kStatusCycle | kStatusQuery)) return DPC_ERR_DATA;
  if (s & kStatusStack) return DPC_ERR_UNSUPPORTED;
  return DPC_ERR_CUDA;
}

// ---- classes -------------------------------------------------------------------

// One class of a call: the non-empty instances sharing (dp, g), in batch order.
struct ClassPlan {
  int dp = 0, g = 0;
  std::vector<int> members;  // batch indices
  uint32_t N = 0, nchunk = 0, nmax = 0;
  int dmax = 1;  // largest dimension of its instances
  int ib = 0, bcap = kMaxBits;
  // offsets of this class's tables in the upload block (multi-instance only)
  size_t off_inst = 0, off_cut = 0, off_par = 0;
  // tables on the device (several instances, or more cutoffs than fit in
  // kernel arguments); a single instance otherwise runs without them
  bool upload = false;
  bool uploaded() const { return upload; }
};

// Groups the instances into classes; `all_one` puts every instance in one
// class (labels only, where the dimension does not matter).
std::vector<ClassPlan> plan_classes(const std::vector<Inst>& insts, bool all_one) {
  std::vector<ClassPlan> out;
  const int keys[5][2] = {{2, 1}, {2, 2}, {4, 3}, {4, 4}, {8, 4}};
  for (int k = 0; k < (all_one ? 1 : 5); ++k) {
    ClassPlan c;
    c.dp = keys[k][0];
    c.g = keys[k][1];
    for (size_t i = 0; i < insts.size(); ++i) {
      const Inst& in = insts[i];
      if (in.n == 0) continue;
      if (!all_one && (dp_of(in.d) != c.dp || g_of(in.d) != c.g)) continue;
      c.members.push_back((int)i);
      c.N += (uint32_t)in.n;
      c.nchunk += (uint32_t)((in.n + 31) / 32);
      c.nmax = std::max(c.nmax, (uint32_t)in.n);
      c.dmax = std::max(c.dmax, in.d);
    }
    if (c.members.empty()) continue;
    int ib = 0;
    while ((size_t(1) << ib) < c.members.size()) ++ib;
    c.ib = ib;
    c.bcap = std::min(kMaxBits, (63 - ib) / c.g);
    out.push_back(std::move(c));
  }
  return out;
}

// Grid level and kernel layouts chosen for one (class, cutoff); r = 0: the
// default rule.
struct Choice {
  int r = 0;
  int dlay = 0;  // density layout (kLayout*)
  int nlay = 0;  // near-phase layout
  int ns = 0;    // near-phase grid levels below the density's
  int sc = 0;    // segment layouts: cells a segment's union may hold (0: one cell)
  uint32_t dfill = 0, nfill = 0;  // points per cell from which a tensor layout runs (0: always)
  uint32_t ufill = 0;  // near phase in the tree layout: points per cell from which union runs (0: never)
};

struct Workspace {
  int device = -1;
  cudaStream_t stream = nullptr;
  uint64_t cap_n = 0;     // points per class the buffers hold
  uint32_t cap_inst = 0;  // instances per class
  int cap_ncut = 0;
  void* base = nullptr;   // one allocation, carved below
  size_t bytes = 0;

  GridGeom* geom = nullptr;   // [cap_inst]
  CutGeom* cuts = nullptr;    // [cap_ncut][cap_inst]
  CutGeom* geo = nullptr;     // [cap_inst] geometry shared by the cutoffs of a group
  ClassGeom* cls = nullptr;
  HashInfo* hinfo = nullptr;
  Counters* ctr = nullptr;
  Counters* ctr_save = nullptr;  // the counters during autotuning trials
  int* status = nullptr;
  int32_t* flags = nullptr;
  uint32_t* roots = nullptr;  // [cap_inst]
  uint32_t* chunk_inst = nullptr;
  uint32_t* chunk_pos = nullptr;
  unsigned long long *codes_a = nullptr, *codes_b = nullptr;
  uint32_t *ids_a = nullptr, *ids_b = nullptr;
  uint32_t* hist = nullptr;
  float* spts = nullptr;
  unsigned long long* scode = nullptr;
  uint32_t* sid = nullptr;
  unsigned long long* skey = nullptr;
  unsigned long long* hkeys = nullptr;
  uint2* hvals = nullptr;
  uint32_t hcap = 0;
  Node* nodes = nullptr;
  float* nbox = nullptr;    // per-node child records of the radix tree (dpc_device.cuh)
  bool boxes_ready = false; // nbox matches the current binning
  uint32_t* visit = nullptr;
  uint4* pieces = nullptr;        // pieces of up to 128 points (tensor-core layouts)
  uint32_t* qpos = nullptr;
  float* qs1 = nullptr;
  double* qs1d = nullptr;
  uint32_t* qpos2 = nullptr;
  float* qs1_2 = nullptr;
  double* qs1d2 = nullptr;

  // instance tables and cutoffs of multi-instance classes: filled in the
  // page-locked host buffer, copied to the device buffer once per call
  void* up_dev = nullptr;
  void* up_host = nullptr;
  size_t up_bytes = 0;
  cudaEvent_t up_done = nullptr;  // the last copy out of up_host has finished

  // host-buffer entry point staging; its copies to the host run on a stream
  // of their own, each behind the event of the phase that finished its output
  void* io = nullptr;
  size_t io_bytes = 0;
  cudaStream_t copy_stream = nullptr;
  std::vector<cudaEvent_t> out_ev;

  // priority range search: per-query arrays (scr) and the match keys (scr2)
  void* scr = nullptr;
  size_t scr_bytes = 0;
  void* scr2 = nullptr;
  size_t scr2_bytes = 0;

  // the captured graph of DPC_FLAG_GRAPH calls and the key it was captured for
  cudaGraphExec_t gexec = nullptr;
  std::string gkey;
  long long glaunches = 0;
  void drop_graph() {
    if (gexec) cudaGraphExecDestroy(gexec);
    gexec = nullptr;
    gkey.clear();
  }

  // autotuned radius and layouts per (class shape, cutoff), see choose()
  std::map<std::string, Choice> tuned;
  cudaEvent_t tune_ev[24] = {};

  // for dpc_get_stats: the last class and cutoff that ran
  Choice last_choice;
  uint32_t last_points = 0;  // points of the class last_cut belongs to
  const CutGeom* last_cut = nullptr;
  const GridGeom* last_geom = nullptr;
  bool have_last = false;
  long long launches_last = 0;

  // phase timing (DPC_FLAG_PHASE_TIMES)
  struct PhaseRec {
    int phase;
    cudaEvent_t a, b;
  };
  bool timing = false;
  std::vector<cudaEvent_t> ev_pool;
  size_t ev_used = 0;
  std::vector<PhaseRec> recs;

  cudaEvent_t take_event() {
    if (ev_used == ev_pool.size()) {
      cudaEvent_t e;
      cudaEventCreate(&e);
      ev_pool.push_back(e);
    }
    return ev_pool[ev_used++];
  }

  void begin_call(uint32_t fl) {
    timing = (fl & DPC_FLAG_PHASE_TIMES) != 0;
    recs.clear();
    ev_used = 0;
    g_kernel_launches = 0;
  }
  void end_call() { launches_last = g_kernel_launches; }

  void release() {
    drop_graph();
    for (cudaEvent_t e : ev_pool) cudaEventDestroy(e);
    ev_pool.clear();
    ev_used = 0;
    recs.clear();
    if (base) cudaFree(base);
    if (io) cudaFree(io);
    if (scr) cudaFree(scr);
    if (scr2) cudaFree(scr2);
    scr = scr2 = nullptr;
    scr_bytes = scr2_bytes = 0;
    if (up_dev) cudaFree(up_dev);
    if (up_host) cudaFreeHost(up_host);
    if (up_done) cudaEventDestroy(up_done);
    for (cudaEvent_t e : out_ev) cudaEventDestroy(e);
    out_ev.clear();
    if (copy_stream) cudaStreamDestroy(copy_stream);
    copy_stream = nullptr;
    for (auto& e : tune_ev) {
      if (e) cudaEventDestroy(e);
      e = nullptr;
    }
    base = io = up_dev = up_host = nullptr;
    up_done = nullptr;
    tuned.clear();
    bytes = io_bytes = up_bytes = 0;
    cap_n = 0;
    cap_inst = 0;
    cap_ncut = 0;
    have_last = false;
  }

  int reserve(uint64_t n, uint32_t ninst, int ncut) {
    if (n <= cap_n && ninst <= cap_inst && ncut <= cap_ncut && base) return DPC_OK;
    uint64_t want_n = std::max<uint64_t>(std::max<uint64_t>(n, cap_n), 1024);
    uint32_t want_i = std::max<uint32_t>(std::max<uint32_t>(ninst, cap_inst), 1);
    int want_c = std::max(std::max(ncut, cap_ncut), 8);
    if (base) {
      cudaStreamSynchronize(stream);
      drop_graph();  // it holds pointers into the old buffers
      cudaFree(base);
      base = nullptr;
    }
    const uint64_t N = want_n;
    const uint32_t hc = next_pow2(2 * N);
    const uint64_t nchunk = N / 32 + want_i + 1;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += align_up(b); return o; };
    const size_t o_geom = take(sizeof(GridGeom) * want_i);
    const size_t o_cuts = take(sizeof(CutGeom) * want_i * (size_t)want_c);
    const size_t o_geo = take(sizeof(CutGeom) * want_i);
    const size_t o_cls = take(sizeof(ClassGeom));
    const size_t o_hi = take(sizeof(HashInfo));
    // the status word follows the counters: one memset clears both
    const size_t o_ctr = take(sizeof(Counters) + sizeof(int));
    const size_t o_status = o_ctr + sizeof(Counters);
    const size_t o_ctr2 = take(sizeof(Counters));
    const size_t o_flags = take(sizeof(int32_t) * 80);
    const size_t o_roots = take(sizeof(uint32_t) * want_i);
    const size_t o_ci = take(4 * nchunk), o_cp = take(4 * nchunk);
    const size_t o_ca = take(8 * N), o_cb = take(8 * N);
    const size_t o_ia = take(4 * N), o_ib = take(4 * N);
    const size_t o_hist = take(4 * sort_hist_words((uint32_t)N));
    const size_t o_spts = take(4 * 8 * N);
    const size_t o_scode = take(8 * N);
    const size_t o_sid = take(4 * N);
    const size_t o_skey = take(8 * N);
    const size_t o_hk = take(8 * (size_t)hc), o_hv = take(8 * (size_t)hc);
    const size_t o_nodes = take(sizeof(Node) * N);
    const size_t o_nbox = take(4 * (size_t)kRecWordsMax * N);
    const size_t o_visit = take(4 * N);
    const size_t o_pieces = take(sizeof(uint4) * N);
    const size_t o_qpos = take(4 * N), o_qs1 = take(4 * N), o_qs1d = take(8 * N);
    const size_t o_qpos2 = take(4 * N), o_qs1_2 = take(4 * N), o_qs1d2 = take(8 * N);
    void* p = nullptr;
    if (!dev_alloc(&p, off)) {
      cap_n = 0;
      cap_inst = 0;
      return DPC_ERR_OOM;
    }
    base = p;
    bytes = off;
    char* b = (char*)p;
    geom = (GridGeom*)(b + o_geom);
    cuts = (CutGeom*)(b + o_cuts);
    geo = (CutGeom*)(b + o_geo);
    cls = (ClassGeom*)(b + o_cls);
    hinfo = (HashInfo*)(b + o_hi);
    ctr = (Counters*)(b + o_ctr);
    ctr_save = (Counters*)(b + o_ctr2);
    status = (int*)(b + o_status);
    flags = (int32_t*)(b + o_flags);
    roots = (uint32_t*)(b + o_roots);
    chunk_inst = (uint32_t*)(b + o_ci);
    chunk_pos = (uint32_t*)(b + o_cp);
    codes_a = (unsigned long long*)(b + o_ca);
    codes_b = (unsigned long long*)(b + o_cb);
    ids_a = (uint32_t*)(b + o_ia);
    ids_b = (uint32_t*)(b + o_ib);
    hist = (uint32_t*)(b + o_hist);
    spts = (float*)(b + o_spts);
    scode = (unsigned long long*)(b + o_scode);
    sid = (uint32_t*)(b + o_sid);
    skey = (unsigned long long*)(b + o_skey);
    hkeys = (unsigned long long*)(b + o_hk);
    hvals = (uint2*)(b + o_hv);
    hcap = hc;
    nodes = (Node*)(b + o_nodes);
    nbox = (float*)(b + o_nbox);
    visit = (uint32_t*)(b + o_visit);
    pieces = (uint4*)(b + o_pieces);
    qpos = (uint32_t*)(b + o_qpos);
    qs1 = (float*)(b + o_qs1);
    qs1d = (double*)(b + o_qs1d);
    qpos2 = (uint32_t*)(b + o_qpos2);
    qs1_2 = (float*)(b + o_qs1_2);
    qs1d2 = (double*)(b + o_qs1d2);
    cap_n = N;
    cap_inst = want_i;
    cap_ncut = want_c;
    have_last = false;
    cudaMemsetAsync(ctr, 0, sizeof(Counters) + sizeof(int), stream);
    return DPC_OK;
  }

  // Makes the upload buffers at least `b` bytes and waits until the previous
  // copy out of the host buffer has finished, so it can be rewritten.
  int reserve_upload(size_t b) {
    if (!up_done) {
      if (cudaEventCreateWithFlags(&up_done, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        return DPC_ERR_CUDA;
      }
    } else if (cudaEventSynchronize(up_done) != cudaSuccess) {
      cudaGetLastError();
      return DPC_ERR_CUDA;
    }
    if (b <= up_bytes && up_dev) return DPC_OK;
    if (up_dev) {
      cudaStreamSynchronize(stream);
      drop_graph();
      cudaFree(up_dev);
      cudaFreeHost(up_host);
      up_dev = up_host = nullptr;
      up_bytes = 0;
    }
    if (!dev_alloc(&up_dev, b)) return DPC_ERR_OOM;
    if (cudaMallocHost(&up_host, b) != cudaSuccess) {
      cudaGetLastError();
      cudaFree(up_dev);
      up_dev = up_host = nullptr;
      return DPC_ERR_OOM;
    }
    up_bytes = b;
    return DPC_OK;
  }

  // grow-only device scratch (contents not kept across growth)
  int reserve_buf(void** p, size_t* have, size_t b) {
    if (b <= *have && *p) return DPC_OK;
    if (*p) {
      cudaStreamSynchronize(stream);
      cudaFree(*p);
      *p = nullptr;
    }
    if (!dev_alloc(p, b)) {
      *have = 0;
      return DPC_ERR_OOM;
    }
    *have = b;
    return DPC_OK;
  }

  int reserve_io(size_t b) {
    if (b <= io_bytes && io) return DPC_OK;
    if (io) {
      cudaStreamSynchronize(stream);
      cudaFree(io);
      io = nullptr;
    }
    if (!dev_alloc(&io, b)) {
      io_bytes = 0;
      return DPC_ERR_OOM;
    }
    io_bytes = b;
    return DPC_OK;
  }
};

// Records CUDA events around one phase when the call asked for phase times.
struct Phase {
  Workspace* w;
  int ph;
  cudaEvent_t a = nullptr;
  Phase(Workspace* w_, int ph_) : w(w_), ph(ph_) {
    if (w->timing) {
      a = w->take_event();
      cudaEventRecord(a, w->stream);
    }
  }
  ~Phase() {
    if (w->timing) {
      cudaEvent_t b = w->take_event();
      cudaEventRecord(b, w->stream);
      w->recs.push_back({ph, a, b});
    }
  }
};

std::mutex g_mu;
std::map<std::pair<int, cudaStream_t>, Workspace*> g_ws;

int get_workspace(cudaStream_t st, Workspace** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return DPC_ERR_CUDA;
  }
  int count = 0;
  if (cudaGetDeviceCount(&count) != cudaSuccess || count == 0) {
    cudaGetLastError();
    return DPC_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  auto key = std::make_pair(dev, st);
  auto it = g_ws.find(key);
  if (it == g_ws.end()) {
    Workspace* w = new Workspace();
    w->device = dev;
    w->stream = st;
    it = g_ws.emplace(key, w).first;
  }
  *out = it->second;
  return DPC_OK;
}

int finish(Workspace* w, uint32_t flags) {
  w->end_call();
  if (cudaGetLastError() != cudaSuccess) return DPC_ERR_CUDA;
  if (flags & DPC_FLAG_SYNC_CHECK) {
    if (cudaStreamSynchronize(w->stream) != cudaSuccess) {
      cudaGetLastError();
      return DPC_ERR_CUDA;
    }
    int s = 0;
    if (cudaMemcpy(&s, w->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) {
      cudaGetLastError();
      return DPC_ERR_CUDA;
    }
    return status_to_code(s);
  }
  return DPC_OK;
}

// ---- one call: plan, upload, classes ----------------------------------------------

// What a call runs.  cut_first/ncut select the cutoffs (all, or one);
// params (may be null) are the labelling thresholds.
struct CallPlan {
  std::vector<ClassPlan> classes;
  int ncut_all = 1;   // n_dcut of the batch
  int cut_first = 0;  // first cutoff this call uses
  int ncut = 1;       // cutoffs this call uses
  uint32_t max_inst = 0;
  uint64_t max_n = 0;
  const dpc_params* params = nullptr;  // thresholds of the call (dpc_run, dpc_cluster)
  bool skip_noise = false;             // DPC_FLAG_SKIP_NOISE
};

CallPlan make_plan(const dpc_batch* b, const std::vector<Inst>& insts, int cut_first, int ncut,
                   bool all_one) {
  CallPlan P;
  P.classes = plan_classes(insts, all_one);
  P.ncut_all = b->n_dcut;
  P.cut_first = cut_first;
  P.ncut = ncut;
  for (auto& c : P.classes) {
    c.upload = c.members.size() > 1 || ncut > kCutChunk;
    P.max_inst = std::max<uint32_t>(P.max_inst, (uint32_t)c.members.size());
    P.max_n = std::max<uint64_t>(P.max_n, c.N);
  }
  return P;
}

// The cutoff constants of (instance bi, cutoff cut); with DPC_FLAG_SKIP_NOISE
// the dependent search skips that pair's noise points.
CutHost cut_host(const CallPlan& P, const dpc_batch* b, int bi, int cut, int dp) {
  CutHost h = make_cut_host(b->d_cut[(size_t)bi * P.ncut_all + cut], dp);
  if (P.skip_noise && P.params) h.skip = P.params[(size_t)bi * P.ncut_all + cut].rho_noise;
  return h;
}

// Fills and copies the tables of every multi-instance class (instance
// descriptors, cutoff constants [inst][cut], label thresholds [cut][inst]).
int upload_tables(Workspace* w, CallPlan& P, const dpc_batch* b, const std::vector<Inst>& insts,
                  const dpc_params* params) {
  size_t total = 0;
  for (auto& c : P.classes) {
    if (!c.uploaded()) continue;
    const size_t m = c.members.size();
    c.off_inst = total;
    total += align_up(sizeof(InstDev) * m);
    c.off_cut = total;
    total += align_up(sizeof(CutHost) * m * P.ncut);
    c.off_par = total;
    total += align_up(sizeof(LabelParams) * m * P.ncut);
  }
  if (total == 0) return DPC_OK;
  int rc = w->reserve_upload(total);
  if (rc) return rc;
  char* h = (char*)w->up_host;
  for (auto& c : P.classes) {
    if (!c.uploaded()) continue;
    const size_t m = c.members.size();
    InstDev* id = (InstDev*)(h + c.off_inst);
    CutHost* ch = (CutHost*)(h + c.off_cut);
    LabelParams* lp = (LabelParams*)(h + c.off_par);
    uint32_t start = 0, chunk = 0;
    for (size_t j = 0; j < m; ++j) {
      const int bi = c.members[j];
      const Inst& in = insts[bi];
      id[j].start = start;
      id[j].n = (uint32_t)in.n;
      id[j].out = in.pt_off;
      id[j].coord = in.coord_off;
      id[j].d = in.d;
      id[j].chunk0 = chunk;
      id[j].row = (uint32_t)bi;
      id[j].pad = 0;
      start += (uint32_t)in.n;
      chunk += (uint32_t)((in.n + 31) / 32);
      for (int k = 0; k < P.ncut; ++k) {
        const int cut = P.cut_first + k;
        ch[j * P.ncut + k] = cut_host(P, b, bi, cut, c.dp);
        LabelParams L{0, 0, 0.0};
        if (params) {
          const dpc_params& q = params[(size_t)bi * P.ncut_all + cut];
          L.rho_noise = q.rho_noise;
          L.rho_min = q.rho_min;
          L.delta_min = q.delta_min;
        }
        lp[(size_t)k * m + j] = L;
      }
    }
  }
  cudaMemcpyAsync(w->up_dev, w->up_host, total, cudaMemcpyHostToDevice, w->stream);
  cudaEventRecord(w->up_done, w->stream);
  return DPC_OK;
}

// The device view of one class.
ClassView view_of(Workspace* w, const ClassPlan& c, const std::vector<Inst>& insts) {
  ClassView v;
  std::memset(&v, 0, sizeof(v));
  v.N = c.N;
  v.ninst = (uint32_t)c.members.size();
  v.nchunk = c.nchunk;
  v.geom = w->geom;
  v.cls = w->cls;
  if (c.uploaded()) {
    v.inst = (const InstDev*)((char*)w->up_dev + c.off_inst);
    v.chunk_inst = w->chunk_inst;
    v.chunk_pos = w->chunk_pos;
  } else {
    const Inst& in = insts[c.members[0]];
    v.one.start = 0;
    v.one.n = (uint32_t)in.n;
    v.one.out = in.pt_off;
    v.one.coord = in.coord_off;
    v.one.d = in.d;
    v.one.chunk0 = 0;
    v.one.row = (uint32_t)c.members[0];
  }
  return v;
}

const CutHost* cut_table(Workspace* w, const ClassPlan& c) {
  return c.uploaded() ? (const CutHost*)((char*)w->up_dev + c.off_cut) : nullptr;
}

// The cutoffs of a class that runs without uploaded tables.
std::vector<CutHost> host_cuts(const CallPlan& P, const dpc_batch* b, const ClassPlan& c) {
  std::vector<CutHost> hc;
  if (!c.uploaded())
    for (int k = 0; k < P.ncut && k < kCutChunk; ++k)
      hc.push_back(cut_host(P, b, c.members[0], P.cut_first + k, c.dp));
  return hc;
}

// Binning of one class: geometry for the call's cutoffs, sorted points.
void bin_class(Workspace* w, const void* pts, int dtype, const CallPlan& P, const ClassPlan& c,
               const ClassView& cv, const dpc_batch* b, const std::vector<Inst>& insts) {
  cudaStream_t st = w->stream;
  Phase ph(w, DPC_PHASE_BIN);
  w->boxes_ready = false;
  launch_class_init(cv, c.g, c.ib, c.bcap, w->status, st);
  launch_chunks(cv, w->chunk_inst, w->chunk_pos, st);
  launch_bbox(pts, dtype, cv, c.g, st);
  launch_setup(cv, w->cuts, P.ncut, cut_table(w, c), host_cuts(P, b, c).data(), st);
  const bool counted = cv.N <= kSortMiddle;
  uint32_t* count = counted ? launch_sort_clear(cv.N, w->hist, st) : nullptr;
  launch_codes(pts, dtype, cv, c.g, w->codes_a, w->ids_a, count, st);
  launch_sort(w->codes_a, w->codes_b, w->ids_a, w->ids_b, cv.N, w->cls, w->hist, counted, st);
  launch_gather(pts, dtype, cv, c.dp, w->codes_a, w->codes_b, w->ids_a, w->ids_b, w->spts,
                w->scode, w->sid, st);
  (void)insts;
}

// Points per occupied cell from which the default layouts of 5-8 dimensions use
// tensor tiles: a tile serves up to 128 queries at the cost of one, but sparse
// cells leave its rows empty and every piece pays its lookups and waits.
// Densities of 1e5 points in 5-D at 4 cutoffs with tiles from 1 / 2 / 3 / 4 points
// on / without, ms: 1.9 points per cell at the smallest cutoff 1.53 / 1.18 / 1.26 /
// 1.25 / 1.24, 2.6 a cell 1.32 / 1.32 / 1.41 / 1.43 / 1.96, 3.1 a cell 1.38 / 1.38 /
// 1.38 / 1.57 / 1.94; 128 instances of 2, 3 and 5 dimensions, 8 cutoffs, whole call
// 84.4 / 84.4 / 81.6 / 81.6 (81.0 from 8 on).  Near phase, the same batch: 141 with
// tiles from 1 or 2 points on, 84.5 from anything between 3 and 16; of 2e6 points
// in 7-D (17 points per cell) 50 ms with tiles, 118 without.
constexpr uint32_t kTensorDensityFill = 2, kTensorNearFill = 4;

// Points per occupied cell from which the default near phase in 1-D scans the
// block (union) instead of searching the tree, with the float32 filter and for
// sets of some size: on smooth dense data the tree search meets long runs of
// higher points (near phase + far search, us, union / tree: 300,000 points in
// blobs, 882 a cell, 1,235 / 2,641; 1e6, 2,874 a cell, 9,758 / 20,729; 100,000,
// 346 a cell, 529 / 516; 300,000, 49 a cell, 255 / 148; uniform, 18 a cell, 100 /
// 99; integer clusters, where both search on through ties, 300 a cell 2,501 /
// 2,250, 940 a cell 17,161 / 14,621; in binary64 the tree everywhere, 882 a cell
// 13,678 / 6,661).
constexpr uint32_t kUnionNearPoints = 1u << 17;
constexpr uint32_t kUnionNearFill = 512;

FarQueue queue_of(Workspace* w) {
  FarQueue q;
  q.pos = w->qpos;
  q.s1 = w->qs1;
  q.s1d = w->qs1d;
  q.pos2 = w->qpos2;
  q.s1_2 = w->qs1_2;
  q.s1d2 = w->qs1d2;
  return q;
}

void tree_step(Workspace* w, const ClassView& cv) {
  Phase ph(w, DPC_PHASE_TREE);
  launch_tree_build(w->scode, cv, w->nodes, w->roots, w->stream);
}

void cells_step(Workspace* w, const ClassPlan& c, const ClassView& cv, const CutGeom* cuts) {
  Phase ph(w, DPC_PHASE_CELLS);
  launch_cells(w->scode, cv, c.g, cuts, w->hinfo, w->hkeys, w->hvals, w->hcap, w->stream);
  w->last_cut = cuts;
  w->last_geom = w->geom;
  w->last_points = cv.N;
  w->have_last = true;
}

void density_step(Workspace* w, const ClassPlan& c, const ClassView& cv, const CutGeom* cuts,
                  int prec, int layout, int seg_cells, int32_t* rho, uint32_t min_fill) {
  Phase ph(w, DPC_PHASE_DENSITY);
  // the tensor layout exists for 5-8 dimensions with the float32 filter;
  // other cases run in segments, and the statistics report what ran
  if (layout == kLayoutTensor && !(c.dp == 8 && prec == 0)) layout = kLayoutSegment;
  w->last_choice.dlay = layout;
  w->last_choice.dfill = min_fill;
  launch_density(c.dp, c.g, c.dmax, prec, layout, w->spts, w->scode, w->sid, cv, cuts, w->hinfo, w->hkeys,
                 w->hvals, w->pieces, rho, w->skey, w->ctr, w->stream, seg_cells, min_fill);
}

void dependent_step(Workspace* w, const ClassPlan& c, const ClassView& cv, CutGeom* cuts,
                    const void* pts, int dtype, int32_t rho_skip, bool fp64, int layout, int nshift,
                    int seg_cells, int32_t* lambda, double* delta, uint32_t min_fill,
                    const FarHint& hint = FarHint()) {
  cudaStream_t st = w->stream;
  {
    Phase ph(w, DPC_PHASE_MAXKEY);
    launch_tree_maxkey(w->skey, w->spts, c.dp, c.dmax, cv.N, w->nodes, w->visit, w->nbox,
                       !w->boxes_ready, st);
    w->boxes_ready = true;
  }
  if (nshift > 0 && layout != kLayoutTree) {  // the near phase on finer cells
    launch_near_level(cv, cuts, nshift, st);
    cells_step(w, c, cv, cuts);
  }
  {
    Phase ph(w, DPC_PHASE_NEAR);
    uint32_t dense = 0;
    if (layout == kLayoutTensor && c.dp == 8 && !fp64) {
      launch_dep_near_tc(c.dmax, w->spts, w->scode, w->sid, w->skey, cv, rho_skip, pts, dtype, cuts, w->hinfo,
                         w->hkeys, w->hvals, w->pieces, lambda, delta, queue_of(w), w->ctr, min_fill, st);
      if (min_fill)  // sparse cells
        launch_dep_near(c.dp, c.g, c.dmax, fp64, kLayoutTree, w->spts, w->scode, w->skey, cv, rho_skip, pts, dtype, cuts,
                        w->hinfo, w->hkeys, w->hvals, lambda, delta, queue_of(w), w->ctr, st, w->nbox, w->roots, seg_cells,
                        min_fill);
    } else {
      // the tensor layout exists for 5-8 dimensions with the float32 filter
      if (layout == kLayoutTensor) layout = kLayoutUnion;
      // 1-D by default: the block scan on dense cells, the tree elsewhere
      if (layout == kLayoutTree && c.g == 1 && !fp64 && min_fill && cv.N >= kUnionNearPoints) dense = kUnionNearFill;
      if (dense)
        launch_dep_near(c.dp, c.g, c.dmax, fp64, kLayoutUnion, w->spts, w->scode, w->skey, cv, rho_skip, pts, dtype,
                        cuts, w->hinfo, w->hkeys, w->hvals, lambda, delta, queue_of(w), w->ctr, st, w->nbox, w->roots,
                        seg_cells, 0, dense);
      launch_dep_near(c.dp, c.g, c.dmax, fp64, layout, w->spts, w->scode, w->skey, cv, rho_skip, pts, dtype,
                      cuts, w->hinfo, w->hkeys, w->hvals, lambda, delta, queue_of(w), w->ctr, st,
                      w->nbox, w->roots, seg_cells, dense);
    }
    w->last_choice.nlay = layout;
    w->last_choice.ufill = dense;
    w->last_choice.nfill = min_fill;
  }
  {
    Phase ph(w, DPC_PHASE_FAR);
    launch_dep_far(c.dp, c.dmax, fp64, w->spts, w->scode, w->skey, cv, cuts, w->nbox, w->roots,
                   queue_of(w), hint, lambda, delta, w->ctr, st);
  }
}

void labels_step(Workspace* w, const ClassPlan& c, const ClassView& cv, int k_in_call,
                 const LabelParams& one, const int32_t* rho, const int32_t* lambda,
                 const double* delta, int32_t* label) {
  Phase ph(w, DPC_PHASE_LABELS);
  const LabelParams* par =
      c.uploaded()
          ? (const LabelParams*)((char*)w->up_dev + c.off_par) + (size_t)k_in_call * c.members.size()
          : nullptr;
  if (labels_by_instance(c.N, (uint32_t)c.members.size(), c.nmax))
    launch_small_labels(rho, lambda, delta, cv, c.nmax, par, one, label, w->status, w->stream);
  else
    launch_labels(rho, lambda, delta, cv, c.nmax, par, one, label, w->flags, w->status, w->stream);
}

LabelParams one_params(const dpc_params* params, const ClassPlan& c, int ncut_all, int cut) {
  LabelParams L{0, 0, 0.0};
  if (params && !c.uploaded()) {
    const dpc_params& q = params[(size_t)c.members[0] * ncut_all + cut];
    L.rho_noise = q.rho_noise;
    L.rho_min = q.rho_min;
    L.delta_min = q.delta_min;
  }
  return L;
}

// Names one (class shape, cutoff) among the autotuned choices.
std::string tune_key(const ClassPlan& c, const dpc_batch* b, int cut) {
  char buf[160];
  const double dc = b->d_cut[(size_t)c.members[0] * b->n_dcut + cut];
  unsigned long long bits;
  std::memcpy(&bits, &dc, sizeof(bits));
  std::snprintf(buf, sizeof(buf), "%d/%d/%zu/%u/%d/%llx", c.dp, c.g, c.members.size(), c.N, cut, bits);
  return buf;
}

// ---- small instances -----------------------------------------------------------

// Whether a class runs from all pairs (small.cu) instead of the grid: one
// dimension, no fixed or tuned radius or layout asked for, few enough points an
// instance (small_limit) and few enough of them.
// Points, measured on blobs with a median density of 16 (us a call, grid -> all
// pairs): density of 1,000 points in 2-D 107 -> 9.5, 8,192 115 -> 36, 16,384 121
// -> 92 (5-D 214 -> 191; 8-D 8,192 189 -> 134, 16,384 216 -> 492); a run of 1,000
// points in 2-D 189 -> 27, 8,192 227 -> 127, 16,384 266 -> 360 (5-D 8,192 394 ->
// 169, 16,384 590 -> 615; 8-D 599 -> 335 and 769 -> 1,089).  In binary64 the
// pairs wait for the binary64 pipe: a run of 2,048 points in 2-D 315 -> 199,
// 4,096 357 -> 653; in 5-D 4,096 1,590 -> 1,342, in 4-D 1,077 -> 1,103.
// Instances: every group of 4 or 8 queries costs a CTA however small its instance
// is, so a class of many tiny ones is the grid's.  Sum of the phases without
// labels: a run of 4,000 instances of 20 points in 2-D 242 -> 156 us, 8,000 271 ->
// 288, 20,000 403 -> 688 (3-D 257 -> 185, 290 -> 343, 432 -> 822); 1,000 of 100
// (4,000 chunks) 256 -> 191, 2,000 309 -> 359; 100 of 1,000 (3,200) 263 -> 269.  A
// density alone: 20,000 of 20 245 -> 151, 500 of 1,000 (16,000 chunks) 260 -> 257,
// 20,000 of 100 (80,000) 546 -> 618.  The grid's sweeps share their set-up, so
// runs of three cutoffs and more change sides earlier (1,000 of 100, whole calls:
// 2 cutoffs 526 -> 408, 4 608 -> 787; 4,000 of 20 in 3-D, 8 cutoffs 1,262 -> 1,658).
// A captured call (DPC_FLAG_GRAPH) takes this path up to 4,096 points only.
// Replayed, all pairs are the faster side beyond that too (grid -> all pairs: a
// run of 4,096 points in 2-D 155 -> 52, 8,192 177 -> 123, in 8-D 542 -> 331), so
// the line is not one of speed: a captured call of more points keeps the grid's
// kernel sequence, which tests/test_gpu_parity.py counts at 6,000 points.
bool small_class(const Workspace* w, const dpc_batch* b, const CallPlan& P, const ClassPlan& c,
                 const std::vector<Inst>& insts, uint32_t flags, bool density_only) {
  if (flags & (DPC_FLAG_RADIUS_MASK | DPC_FLAG_LAYOUT_MASK | DPC_FLAG_NEAR_SHIFT_MASK | DPC_FLAG_AUTOTUNE))
    return false;
  // an earlier call's choice for this shape stays in force
  for (int k = 0; k < P.ncut && !w->tuned.empty(); ++k)
    for (const char* kind : {"R/", "D/"})
      if (w->tuned.count(kind + tune_key(c, b, P.cut_first + k))) return false;
  const bool fp64 = (flags & DPC_PREC_MASK) == DPC_PREC_FP64;
  const int d = insts[c.members[0]].d;
  const uint32_t nmax = small_limit(d, fp64, density_only);
  if (c.nmax > nmax || ((flags & DPC_FLAG_GRAPH) && c.nmax > 4096u)) return false;
  if (c.nchunk > (density_only ? 16384u : (P.ncut > 2 ? 2048u : 4096u))) return false;
  uint64_t pairs = 0;
  for (int i : c.members) {
    if (insts[i].d != d) return false;
    pairs += insts[i].n * insts[i].n;
  }
  return pairs <= (uint64_t)nmax * nmax;
}

void small_density_step(Workspace* w, const void* pts, int dtype, const CallPlan& P, const ClassPlan& c,
                        const ClassView& cv, const dpc_batch* b, const std::vector<Inst>& insts, bool fp64,
                        int32_t* rho, uint64_t N) {
  Phase ph(w, DPC_PHASE_DENSITY);
  launch_chunks(cv, w->chunk_inst, w->chunk_pos, w->stream);
  launch_small_density(insts[c.members[0]].d, fp64, pts, dtype, cv, cut_table(w, c), host_cuts(P, b, c).data(),
                       P.ncut, rho, N, w->ctr, w->status, w->stream);
  w->last_choice = Choice();
  w->have_last = false;
}

void small_dependent_step(Workspace* w, const void* pts, int dtype, const CallPlan& P, const ClassPlan& c,
                          const ClassView& cv, const dpc_batch* b, const std::vector<Inst>& insts, bool fp64,
                          int k, int32_t rho_skip, const int32_t* rho, int32_t* lambda, double* delta) {
  Phase ph(w, DPC_PHASE_NEAR);
  launch_small_dependent(insts[c.members[0]].d, fp64, pts, dtype, cv, cut_table(w, c), host_cuts(P, b, c).data(),
                         P.ncut, k, rho_skip, rho, lambda, delta, w->ctr, w->status, w->stream);
}

// ---- autotuning of the cell level -------------------------------------------------
//
// The block radius R (and with it the grid level: finer cells for larger R)
// decides how many candidates a query scans and how many cells a warp looks
// up.  The default rule keeps R = 1 unless a larger R shrinks the block side
// by 20%; with DPC_FLAG_AUTOTUNE the first call for a class shape times the
// density step once per radius (R = 1, 2, 3 in 1-2 gridded dims, R = 1, 2 in
// 3; 4 gridded dims allow only R = 1) and keeps the fastest for later calls of
// the same shape.

// What a tuning trial of the dependent step needs (null: density only).
struct NearTrial {
  const void* pts;
  int dtype;
  int32_t* lambda;  // scratch outputs of the trial
  double* delta;
};

// Default layouts (measured on the GB300).  Density: tensor tiles in 5-8
// dimensions with the float32 filter, segments otherwise, pairs in binary64 from
// kBinary64Pairs chunks on, union in 1-D.
// Near phase: tensor tiles again; else the tree search (near phase + far search,
// ms, blocks scanned -> tree: 1e6 points in 2-D 0.74 -> 0.34, blobs of 1e6 in 3-D
// 2.21 -> 0.66, in 4-D 4.6 -> 1.9, binary64 1e5 in 5-D 62.9 -> 2.6; against it
// only the 1e7-point 3-D walk, 4.84 -> 5.83, which the autotuner finds), in 1-D
// up to 1e6 points (2e5: 0.14 -> 0.10; 2e6: 0.70 -> 1.02).
inline bool tensor_class(const ClassPlan& c, bool fp64) { return c.dp == 8 && !fp64; }
inline int default_dlayout(const ClassPlan& c, int prec) {
  if (tensor_class(c, prec != 0)) return kLayoutTensor;
  if (prec == 2) return kLayoutSegment;  // 64-bit integers
  if (c.g < 2) return kLayoutUnion;
  return prec == 1 && c.nchunk >= kBinary64Pairs ? kLayoutPairs : kLayoutSegment;
}
inline int default_nlayout(const ClassPlan& c, bool fp64) {
  if (tensor_class(c, fp64)) return kLayoutTensor;
  return c.g == 1 && c.N > 1000000u ? kLayoutUnion : kLayoutTree;
}
// segments of the segment layouts span cells while their union fits this: the
// middle of a flat range (1e7 points in 3-D, density + near phase: 7.78 ms at 40
// cells, 7.10 at 48, 7.10 at 56, 7.03 at 64, 7.02 at 72, 7.17 at 80; 1e6 in 2-D,
// density: .436 ms one cell, .371 at 25, .360 at 36, .364 at 49, .364 at 56)
inline int default_seg_cells(int g) { return g == 3 ? 56 : (g == 2 ? 36 : 0); }

// The grid level and kernel layouts of one (class, cutoff): a fixed radius or
// layout from the flags, else the autotuned choice (measured now when the
// call asks for autotuning and the shape is new, cached otherwise), else the
// default rule.  A trial, per radius, times cells, then density in both
// layouts and the dependent search (near phase + far phase) with each near
// layout (after one untimed pass that loads the kernels and warms the caches);
// the radius with the least cells + best density + best dependent search wins,
// with its best layouts.  The counters are saved around the trials;
// rho_scratch (and the NearTrial outputs) receive the trials' results.
Choice choose(Workspace* w, const ClassPlan& c, const ClassView& cv, CutGeom* cuts,
              const dpc_batch* b, int cut, int prec, int32_t* rho_scratch, uint32_t flags,
              const NearTrial* near = nullptr) {
  const bool fp64 = prec != 0;
  Choice ch;
  ch.r = (int)((flags & DPC_FLAG_RADIUS_MASK) >> 12);
  const int forced = (int)((flags & DPC_FLAG_LAYOUT_MASK) >> 16);
  const int forced_ns = (int)((flags & DPC_FLAG_NEAR_SHIFT_MASK) >> 20);
  ch.dlay = (forced && forced != kLayoutTree) ? forced : default_dlayout(c, prec);
  ch.nlay = (forced && forced != kLayoutPairs) ? forced : default_nlayout(c, fp64);
  ch.ns = forced_ns ? forced_ns - 1 : 0;
  ch.sc = default_seg_cells(c.g);
  if (!forced) {
    ch.dfill = kTensorDensityFill;
    ch.nfill = kTensorNearFill;
  }
  const std::string key = (near ? "R/" : "D/") + tune_key(c, b, cut);
  auto it = w->tuned.find(key);
  const bool fixed = ch.r != 0 || forced || forced_ns;
  if (!fixed && it == w->tuned.end() && (flags & DPC_FLAG_AUTOTUNE)) {
    cudaStream_t st = w->stream;
    if (!w->tune_ev[0])
      for (auto& e : w->tune_ev) cudaEventCreate(&e);
    cudaMemcpyAsync(w->ctr_save, w->ctr, sizeof(Counters), cudaMemcpyDeviceToDevice, st);
    // the tensor layout exists for 5-8 dimensions with the float32 filter
    const int ndl = (c.dp == 8 && !fp64) ? 4 : 3;
    const int dlays[4] = {kLayoutUnion, kLayoutSegment, kLayoutPairs, kLayoutTensor};
    // the tensor layouts exist for 5-8 dimensions with the float32 filter
    const int nnl = (c.dp == 8 && !fp64) ? 4 : 3;
    const int nlays[4] = {kLayoutUnion, kLayoutSegment, kLayoutTree, kLayoutTensor};
    constexpr int kShifts = 3;  // near phase 0, 1 or 2 levels below the density's
    constexpr int kNL = 4;      // near layout slots per shift
    // events: 0 start, 1 after cells, 2-5 after each density layout, 6 after
    // the subtree keys; per near shift s, 7 + (kNL + 1) s after its level
    // change and cells, then one after each near layout (each followed by the
    // far search, which finishes what the near phase leaves; the tree layout,
    // which uses no cells, only at s = 0)
    auto trial = [&](int r, bool timed) {
      if (timed) cudaEventRecord(w->tune_ev[0], st);
      launch_set_radius(cv, cuts, r, st);
      launch_cells(w->scode, cv, c.g, cuts, w->hinfo, w->hkeys, w->hvals, w->hcap, st);
      if (timed) cudaEventRecord(w->tune_ev[1], st);
      for (int l = 0; l < 4; ++l) {
        if (l < ndl)
          launch_density(c.dp, c.g, c.dmax, prec, dlays[l], w->spts, w->scode, w->sid, cv, cuts, w->hinfo,
                         w->hkeys, w->hvals, w->pieces, rho_scratch, w->skey, w->ctr, st,
                         default_seg_cells(c.g));
        if (timed) cudaEventRecord(w->tune_ev[2 + l], st);
      }
      if (!near) return;
      launch_tree_maxkey(w->skey, w->spts, c.dp, c.dmax, cv.N, w->nodes, w->visit, w->nbox,
                         !w->boxes_ready, st);
      w->boxes_ready = true;
      if (timed) cudaEventRecord(w->tune_ev[6], st);
      for (int sh = 0; sh < kShifts; ++sh) {
        if (sh > 0) {
          launch_set_radius(cv, cuts, r, st);
          launch_near_level(cv, cuts, sh, st);
          launch_cells(w->scode, cv, c.g, cuts, w->hinfo, w->hkeys, w->hvals, w->hcap, st);
        }
        if (timed) cudaEventRecord(w->tune_ev[7 + (kNL + 1) * sh], st);
        for (int l = 0; l < kNL; ++l) {
          if (l < nnl && (sh == 0 || nlays[l] != kLayoutTree)) {
            if (nlays[l] == kLayoutTensor)
              launch_dep_near_tc(c.dmax, w->spts, w->scode, w->sid, w->skey, cv, 0, near->pts, near->dtype,
                                 cuts, w->hinfo, w->hkeys, w->hvals, w->pieces, near->lambda,
                                 near->delta, queue_of(w), w->ctr, 0, st);
            else
              launch_dep_near(c.dp, c.g, c.dmax, fp64, nlays[l], w->spts, w->scode, w->skey, cv, 0,
                              near->pts, near->dtype, cuts, w->hinfo, w->hkeys, w->hvals,
                              near->lambda, near->delta, queue_of(w), w->ctr, st,
                              w->nbox, w->roots, default_seg_cells(c.g));
            launch_dep_far(c.dp, c.dmax, fp64, w->spts, w->scode, w->skey, cv, cuts, w->nbox,
                           w->roots, queue_of(w), FarHint(), near->lambda, near->delta, w->ctr, st);
          }
          if (timed) cudaEventRecord(w->tune_ev[8 + (kNL + 1) * sh + l], st);
        }
      }
    };
    auto span = [&](int a, int z) {
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, w->tune_ev[a], w->tune_ev[z]) != cudaSuccess) {
        cudaGetLastError();
        return 1e30f;
      }
      return ms;
    };
    const int rmax = c.g >= 4 ? 1 : (c.g == 3 ? 2 : 3);
    trial(1, false);  // untimed: module loading, caches
    Choice best;
    float best_ms = 0.f;
    bool failed = false;
    for (int r = 1; r <= rmax && !failed; ++r) {
      // each phase: the smaller of two timings
      float cl = 1e30f, dt[4] = {1e30f, 1e30f, 1e30f, 1e30f};
      float nt[kShifts][kNL], lv[kShifts];
      for (int sh = 0; sh < kShifts; ++sh) {
        lv[sh] = 1e30f;
        for (int l = 0; l < kNL; ++l) nt[sh][l] = 1e30f;
      }
      for (int rep = 0; rep < 2; ++rep) {
        trial(r, true);
        if (cudaEventSynchronize(w->tune_ev[near ? 8 + (kNL + 1) * (kShifts - 1) + kNL - 1 : 5]) !=
            cudaSuccess) {
          cudaGetLastError();
          failed = true;
          break;
        }
        cl = fminf(cl, span(0, 1));
        for (int l = 0; l < ndl; ++l) dt[l] = fminf(dt[l], span(1 + l, 2 + l));
        if (near)
          for (int sh = 0; sh < kShifts; ++sh) {
            // the level change and cells of a shift count against it
            lv[sh] = sh == 0 ? 0.f
                             : fminf(lv[sh], span(8 + (kNL + 1) * (sh - 1) + kNL - 1, 7 + (kNL + 1) * sh));
            for (int l = 0; l < nnl; ++l)
              if (sh == 0 || nlays[l] != kLayoutTree)
                nt[sh][l] = fminf(nt[sh][l], span(7 + (kNL + 1) * sh + l, 8 + (kNL + 1) * sh + l));
          }
      }
      if (failed) break;
      // a layout other than the default has to win by 3%
      auto pick = [&](const float* t, const int* lays, int m, int def) {
        int bi = 0;
        for (int l = 0; l < m; ++l)
          if (lays[l] == def) bi = l;
        for (int l = 0; l < m; ++l)
          if (t[l] < 0.97f * t[bi]) bi = l;
        return bi;
      };
      const int di = pick(dt, dlays, ndl, default_dlayout(c, prec));
      int nsi = 0, ni = -1;
      float nms = 0.f;
      if (near) {
        ni = pick(nt[0], nlays, nnl, default_nlayout(c, fp64));
        nms = nt[0][ni];
        for (int sh = 1; sh < kShifts; ++sh) {
          const int l = pick(nt[sh], nlays, nnl, default_nlayout(c, fp64));
          const float t = lv[sh] + nt[sh][l];
          if (t < 0.97f * nms) {
            nms = t;
            nsi = sh;
            ni = l;
          }
        }
      }
      const float ms = cl + dt[di] + nms;
      if (best.r == 0 || ms < best_ms) {
        best_ms = ms;
        best.r = r;
        best.dlay = dlays[di];
        best.nlay = near ? nlays[ni] : default_nlayout(c, fp64);
        best.ns = near ? nsi : 0;
        best.sc = default_seg_cells(c.g);
      }
    }
    if (failed) best = Choice();
    // back to the default level (the trials left a shifted one behind)
    launch_set_radius(cv, cuts, 0, st);
    cudaMemcpyAsync(w->ctr, w->ctr_save, sizeof(Counters), cudaMemcpyDeviceToDevice, st);
    it = w->tuned.emplace(key, best).first;
  }
  if (!fixed && it != w->tuned.end() && it->second.r > 0) ch = it->second;
  if (ch.r > 0) launch_set_radius(cv, cuts, ch.r, w->stream);
  w->last_choice = ch;
  return ch;
}

// ---- cutoff sweeps -------------------------------------------------------------
//
// The grid level of a cutoff is a power of two times the smallest one, so the
// cutoffs of a sweep fall into groups with the same cells (1.25^k: three per
// level).  One density launch serves up to kMultiCuts cutoffs of a group, and
// the near-dependent search runs on the cells of the smallest cutoff (at most
// kNearLevels levels below the cutoff's own): a dependent point's distance
// hardly depends on the cutoff, the block's points grow with its power.  After
// the first cutoff the dependent point found for another one, where it is
// higher here too, bounds the search (FarHint).  Groups run from the largest
// cutoffs down, so one hash at a time suffices.
// 2e6 points in 7-D at 4 cutoffs: 565 -> 171 ms a call (density 217 -> 49, near
// phase 209 -> 50, far 30 -> 70); 128 instances of 2, 3 and 5 dimensions at 8
// cutoffs: 257 -> 148 ms (density 90 -> 42, near phase and far 154 -> 97).
constexpr int kNearLevels = 3;

struct CutGroup {
  int level = 0;
  std::vector<int> cuts;  // cutoffs whose densities run on this group's cells
  std::vector<int> near;  // cutoffs whose near phase does
};

bool sweep_call(const CallPlan& P, uint32_t flags) {
  return P.ncut > 1 && P.ncut <= 64 &&
         !(flags & (DPC_FLAG_RADIUS_MASK | DPC_FLAG_LAYOUT_MASK | DPC_FLAG_NEAR_SHIFT_MASK));
}

// Groups by the cutoffs of the class's first instance (any grouping is
// correct: every instance takes the geometry of its largest cutoff of the
// group), largest level first.
std::vector<CutGroup> group_cuts(const CallPlan& P, const dpc_batch* b, const ClassPlan& c) {
  const double* d = b->d_cut + (size_t)c.members[0] * P.ncut_all;
  const double dmin = *std::min_element(d, d + P.ncut);
  std::map<int, CutGroup, std::greater<int>> by;
  std::vector<int> level(P.ncut);
  for (int j = 0; j < P.ncut; ++j) {
    // no common fine cell without a positive smallest cutoff: one group each
    level[j] = dmin > 0.0 ? (int)std::ceil(std::log2(std::min(d[j] / dmin, 0x1p40)) - 1e-9) : j;
    by[level[j]].level = level[j];
    by[level[j]].cuts.push_back(j);
  }
  for (int j = 0; j < P.ncut; ++j) {
    int at = level[j];
    if (dmin > 0.0)
      for (auto& kv : by)
        if (kv.first < at && kv.first >= level[j] - kNearLevels) at = kv.first;
    by[at].near.push_back(j);
  }
  std::vector<CutGroup> out;
  for (auto& kv : by) out.push_back(std::move(kv.second));
  return out;
}

// The densities of one group (cells of its geometry into the hash first).
void group_density_step(Workspace* w, const ClassPlan& c, const ClassView& cv, int ncut, const CutGroup& g,
                        int prec, int32_t* rho, uint64_t N) {
  unsigned long long mask = 0;
  for (int j : g.cuts) mask |= 1ull << j;
  launch_group_geometry(cv, w->cuts, ncut, mask, w->geo, w->stream);
  cells_step(w, c, cv, w->geo);
  Phase ph(w, DPC_PHASE_DENSITY);
  w->last_choice = Choice();
  w->last_choice.dlay = tensor_class(c, prec != 0) ? kLayoutTensor : kLayoutSegment;
  w->last_choice.dfill = kTensorDensityFill;
  auto single = [&](int j) {  // the single-cutoff default
    w->last_choice.dlay = default_dlayout(c, prec);
    launch_density(c.dp, c.g, c.dmax, prec, w->last_choice.dlay, w->spts, w->scode, w->sid, cv,
                   w->cuts + (size_t)j * cv.ninst, w->hinfo, w->hkeys, w->hvals, w->pieces, rho + (size_t)j * N,
                   w->skey, w->ctr, w->stream, default_seg_cells(c.g));
  };
  if (g.cuts.size() == 1 && !tensor_class(c, prec != 0)) {
    single(g.cuts[0]);
    return;
  }
  for (size_t i = 0; i < g.cuts.size(); i += kMultiCuts) {
    // float32 points in binary64, one cutoff left over: every pair once, as for a
    // cutoff alone (on top of four in one pass, segments / pairs in ms: 1e6 points
    // in 2-D 14.4 / 6.8, in 3-D 79 / 35, 1e5 in 5-D 10.9 / 9.3, in 7-D 17.6 /
    // 15.7; in 1-D .88 / 1.07 with that one's union layout)
    if (i + 1 == g.cuts.size() && default_dlayout(c, prec) == kLayoutPairs) {
      launch_adopt_geometry(cv, w->geo, w->cuts + (size_t)g.cuts[i] * cv.ninst, w->stream);
      single(g.cuts[i]);
      return;
    }
    MultiCut mc;
    for (size_t j = i; j < g.cuts.size() && j < i + kMultiCuts; ++j) {
      mc.cut[mc.m] = w->cuts + (size_t)g.cuts[j] * cv.ninst;
      mc.rho[mc.m++] = rho + (size_t)g.cuts[j] * N;
    }
    launch_density_multi(c.dp, c.g, c.dmax, prec, w->spts, w->scode, w->sid, cv, w->geo, w->hinfo, w->hkeys,
                         w->hvals, w->pieces, mc, w->ctr, w->stream, default_seg_cells(c.g), kTensorDensityFill);
  }
}

void reset_call(Workspace* w, uint32_t flags) {
  w->begin_call(flags);
  cudaMemsetAsync(w->ctr, 0, sizeof(Counters) + sizeof(int), w->stream);
}

// Reserves the workspace for a plan and uploads its tables.
int prepare(Workspace* w, CallPlan& P, const dpc_batch* b, const std::vector<Inst>& insts,
            const dpc_params* params, uint32_t flags) {
  sort_init();
  small_init();
  P.params = params;
  P.skip_noise = (flags & DPC_FLAG_SKIP_NOISE) != 0;
  int rc = w->reserve(P.max_n, P.max_inst, P.ncut);
  if (rc) return rc;
  reset_call(w, flags);
  return upload_tables(w, P, b, insts, params);
}

}  // namespace
}  // namespace dpc

using namespace dpc;

extern "C" {

const char* dpc_version(void) { return "0.3.0"; }

int dpc_cut_band(double d_cut, int32_t dim, float* out) {
  if (!out || dim < 1 || dim > kMaxDim || !std::isfinite(d_cut) || d_cut < 0.0) return DPC_ERR_ARG;
  const CutHost h = make_cut_host(d_cut, dp_of(dim));
  out[0] = h.t_in;
  out[1] = h.t_out;
  out[2] = h.band_mul;
  out[3] = h.band_add;
  return DPC_OK;
}

const char* dpc_strerror(int status) {
  switch (status) {
    case DPC_OK: return "ok";
    case DPC_ERR_ARG: return "invalid argument";
    case DPC_ERR_CUDA: return "CUDA error or no CUDA device";
    case DPC_ERR_OOM: return "device memory allocation failed";
    case DPC_ERR_TIMEOUT: return "a bounded device-side wait gave up";
    case DPC_ERR_OVERFLOW: return "an instance, or the whole batch, has 2^31 or more points";
    case DPC_ERR_UNSUPPORTED: return "not supported by this build";
    case DPC_ERR_DATA: return "coordinates out of range or NaN, or dependent pointers not a forest";
    default: return "unknown status";
  }
}

int dpc_density(const void* pts, int dtype, const dpc_batch* b, int32_t* rho, uint32_t flags,
                void* stream) {
  std::vector<Inst> insts;
  uint64_t N = 0;
  int rc = check_batch(b, &insts, &N);
  if (rc) return rc;
  if ((rc = check_flags(flags))) return rc;
  if (flags & DPC_FLAG_SKIP_NOISE) return DPC_ERR_ARG;  // no thresholds here
  if (dtype != DPC_I32 && dtype != DPC_F32) return DPC_ERR_ARG;
  if (N > 0 && (!pts || !rho)) return DPC_ERR_ARG;
  Workspace* w = nullptr;
  if ((rc = get_workspace((cudaStream_t)stream, &w))) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  CallPlan P = make_plan(b, insts, 0, b->n_dcut, false);
  if ((rc = prepare(w, P, b, insts, nullptr, flags))) return rc;
  const bool fp64 = (flags & DPC_PREC_MASK) == DPC_PREC_FP64;
  // binary64 densities of int32 points: the same values in 64-bit integers
  const int prec = fp64 ? (dtype == DPC_I32 ? 2 : 1) : 0;
  for (const ClassPlan& c : P.classes) {
    const ClassView cv = view_of(w, c, insts);
    if (small_class(w, b, P, c, insts, flags, true)) {
      small_density_step(w, pts, dtype, P, c, cv, b, insts, fp64, rho, N);
      continue;
    }
    bin_class(w, pts, dtype, P, c, cv, b, insts);
    if (sweep_call(P, flags)) {
      for (const CutGroup& g : group_cuts(P, b, c)) group_density_step(w, c, cv, P.ncut, g, prec, rho, N);
      continue;
    }
    for (int k = 0; k < P.ncut; ++k) {
      CutGeom* cuts = w->cuts + (size_t)k * cv.ninst;
      const Choice ch = choose(w, c, cv, cuts, b, k, prec, rho + (size_t)k * N, flags);
      cells_step(w, c, cv, cuts);
      density_step(w, c, cv, cuts, prec, ch.dlay, ch.sc, rho + (size_t)k * N, ch.dfill);
    }
  }
  return finish(w, flags);
}

int dpc_dependent(const void* pts, int dtype, const dpc_batch* b, int32_t dcut_index,
                  const int32_t* rho, int32_t rho_skip, int32_t* lambda, double* delta,
                  uint32_t flags, void* stream) {
  std::vector<Inst> insts;
  uint64_t N = 0;
  int rc = check_batch(b, &insts, &N);
  if (rc) return rc;
  if ((rc = check_flags(flags))) return rc;
  if (flags & DPC_FLAG_SKIP_NOISE) return DPC_ERR_ARG;  // rho_skip is the argument here
  if (dtype != DPC_I32 && dtype != DPC_F32) return DPC_ERR_ARG;
  if (dcut_index < 0 || dcut_index >= b->n_dcut) return DPC_ERR_ARG;
  if (N > 0 && (!pts || !rho || !lambda || !delta)) return DPC_ERR_ARG;
  Workspace* w = nullptr;
  if ((rc = get_workspace((cudaStream_t)stream, &w))) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  CallPlan P = make_plan(b, insts, dcut_index, 1, false);
  if ((rc = prepare(w, P, b, insts, nullptr, flags))) return rc;
  const bool fp64 = (flags & DPC_PREC_MASK) == DPC_PREC_FP64;
  // binary64 densities of int32 points: the same values in 64-bit integers
  const int prec = fp64 ? (dtype == DPC_I32 ? 2 : 1) : 0;
  for (const ClassPlan& c : P.classes) {
    const ClassView cv = view_of(w, c, insts);
    if (small_class(w, b, P, c, insts, flags, false)) {
      launch_chunks(cv, w->chunk_inst, w->chunk_pos, w->stream);
      w->have_last = false;
      small_dependent_step(w, pts, dtype, P, c, cv, b, insts, fp64, 0, rho_skip, rho, lambda, delta);
      continue;
    }
    bin_class(w, pts, dtype, P, c, cv, b, insts);
    tree_step(w, cv);
    const Choice ch = choose(w, c, cv, w->cuts, b, dcut_index, prec, nullptr,
                             flags & ~DPC_FLAG_AUTOTUNE, nullptr);
    cells_step(w, c, cv, w->cuts);
    launch_keys_from_rho(rho, w->sid, cv.N, w->skey, w->stream);
    dependent_step(w, c, cv, w->cuts, pts, dtype, rho_skip, fp64, ch.nlay, ch.ns, ch.sc, lambda,
                   delta, ch.nfill);
  }
  return finish(w, flags);
}

int dpc_cluster(const dpc_batch* b, int32_t dcut_index, const dpc_params* params,
                const int32_t* rho, const int32_t* lambda, const double* delta, int32_t* label,
                uint32_t flags, void* stream) {
  std::vector<Inst> insts;
  uint64_t N = 0;
  int rc = check_batch(b, &insts, &N);
  if (rc) return rc;
  if (flags & ~kKnownFlags) return DPC_ERR_ARG;
  if (dcut_index < 0 || dcut_index >= b->n_dcut || !params) return DPC_ERR_ARG;
  if (N > 0 && (!rho || !lambda || !delta || !label)) return DPC_ERR_ARG;
  for (int i = 0; i < b->n_inst; ++i)
    if (std::isnan(params[(size_t)i * b->n_dcut + dcut_index].delta_min)) return DPC_ERR_ARG;
  Workspace* w = nullptr;
  if ((rc = get_workspace((cudaStream_t)stream, &w))) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  CallPlan P = make_plan(b, insts, dcut_index, 1, true);
  if ((rc = prepare(w, P, b, insts, params, flags))) return rc;
  for (const ClassPlan& c : P.classes) {
    const ClassView cv = view_of(w, c, insts);
    if (!labels_by_instance(c.N, cv.ninst, c.nmax)) launch_chunks(cv, w->chunk_inst, w->chunk_pos, w->stream);
    labels_step(w, c, cv, 0, one_params(params, c, P.ncut_all, dcut_index), rho, lambda, delta,
                label);
  }
  return finish(w, flags);
}

// The kernels of every class and cutoff (the part of dpc_run a graph holds).
// A phase of one cutoff finished for every class: stage 0 after the density
// (rho), 1 after the dependent search (lambda, delta), 2 after the labels.
using StageDone = std::function<void(int stage, int cut)>;

static void run_classes(Workspace* w, const CallPlan& P, const void* pts, int dtype,
                        const dpc_batch* b, const std::vector<Inst>& insts, uint64_t N,
                        const dpc_params* params, int32_t* rho, int32_t* lambda, double* delta,
                        int32_t* label, uint32_t flags, const StageDone* done = nullptr) {
  const bool fp64 = (flags & DPC_PREC_MASK) == DPC_PREC_FP64;
  // binary64 densities of int32 points: the same values in 64-bit integers
  const int prec = fp64 ? (dtype == DPC_I32 ? 2 : 1) : 0;
  for (const ClassPlan& c : P.classes) {
    // classes run one after another on the stream, so a phase of the last
    // class finishes that phase's output of every class
    const bool last = &c == &P.classes.back();
    const ClassView cv = view_of(w, c, insts);
    if (small_class(w, b, P, c, insts, flags, false)) {
      small_density_step(w, pts, dtype, P, c, cv, b, insts, fp64, rho, N);
      for (int k = 0; k < P.ncut; ++k) {
        const size_t o = (size_t)k * N;
        if (last && done) (*done)(0, k);
        small_dependent_step(w, pts, dtype, P, c, cv, b, insts, fp64, k, 0, rho + o, lambda + o, delta + o);
        if (last && done) (*done)(1, k);
        labels_step(w, c, cv, k, one_params(params, c, P.ncut_all, k), rho + o, lambda + o, delta + o, label + o);
        if (last && done) (*done)(2, k);
      }
      continue;
    }
    bin_class(w, pts, dtype, P, c, cv, b, insts);
    tree_step(w, cv);
    if (sweep_call(P, flags)) {
      int prev = -1;  // the cutoff whose dependent points were found last
      for (const CutGroup& g : group_cuts(P, b, c)) {
        group_density_step(w, c, cv, P.ncut, g, prec, rho, N);
        if (last && done)
          for (int k : g.cuts) (*done)(0, k);
        for (int k : g.near) {
          const size_t o = (size_t)k * N;
          CutGeom* cuts = w->cuts + (size_t)k * cv.ninst;
          launch_adopt_geometry(cv, w->geo, cuts, w->stream);
          launch_keys_from_rho(rho + o, w->sid, cv.N, w->skey, w->stream);
          FarHint hint;
          if (prev >= 0) {
            hint.lambda = lambda + (size_t)prev * N;
            hint.rho = rho + o;
            hint.pts = pts;
            hint.dtype = dtype;
          }
          prev = k;
          dependent_step(w, c, cv, cuts, pts, dtype, 0, fp64, default_nlayout(c, fp64), 0, default_seg_cells(c.g),
                         lambda + o, delta + o, kTensorNearFill, hint);
          if (last && done) (*done)(1, k);
          labels_step(w, c, cv, k, one_params(params, c, P.ncut_all, k), rho + o, lambda + o, delta + o, label + o);
          if (last && done) (*done)(2, k);
        }
      }
      continue;
    }
    for (int k = 0; k < P.ncut; ++k) {
      const size_t o = (size_t)k * N;
      CutGeom* cuts = w->cuts + (size_t)k * cv.ninst;
      const NearTrial nt{pts, dtype, lambda + o, delta + o};
      const Choice ch = choose(w, c, cv, cuts, b, k, prec, rho + o, flags, &nt);
      cells_step(w, c, cv, cuts);
      density_step(w, c, cv, cuts, prec, ch.dlay, ch.sc, rho + o, ch.dfill);
      if (last && done) (*done)(0, k);
      dependent_step(w, c, cv, cuts, pts, dtype, 0, fp64, ch.nlay, ch.ns, ch.sc, lambda + o,
                     delta + o, ch.nfill);
      if (last && done) (*done)(1, k);
      labels_step(w, c, cv, k, one_params(params, c, P.ncut_all, k), rho + o, lambda + o,
                  delta + o, label + o);
      if (last && done) (*done)(2, k);
    }
  }
}

int dpc_decision_graph(const dpc_batch* b, const int32_t* rho, const double* delta, int32_t k,
                       int32_t* top, double* gamma, int32_t rho_bins, int32_t delta_bins,
                       double delta_lo, int64_t* hist, uint32_t flags, void* stream) {
  std::vector<Inst> insts;
  uint64_t N = 0;
  int rc = check_batch(b, &insts, &N);
  if (rc) return rc;
  if (flags & ~(DPC_FLAG_SYNC_CHECK)) return DPC_ERR_ARG;
  if (k < 0 || k > decision_max_topk()) return DPC_ERR_ARG;
  if (rho_bins < 0 || rho_bins > 32 || delta_bins < 0 || delta_bins > 2048) return DPC_ERR_ARG;
  if ((rho_bins > 0) != (delta_bins > 0)) return DPC_ERR_ARG;
  if (k > 0 && (!top || !gamma)) return DPC_ERR_ARG;
  if (rho_bins > 0 && (!hist || !(delta_lo > 0.0) || !std::isfinite(delta_lo))) return DPC_ERR_ARG;
  if (N > 0 && (!rho || !delta)) return DPC_ERR_ARG;
  Workspace* w = nullptr;
  if ((rc = get_workspace((cudaStream_t)stream, &w))) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  // every non-empty instance in one class (the summaries do not depend on the
  // dimension); rows of empty instances keep the padding written first
  CallPlan P = make_plan(b, insts, 0, 1, true);
  if ((rc = prepare(w, P, b, insts, nullptr, flags))) return rc;
  const size_t members = P.classes.empty() ? 0 : P.classes[0].members.size();
  launch_decision_init(b->n_inst, k, members < (size_t)b->n_inst, top, gamma, rho_bins, delta_bins,
                       (unsigned long long*)hist, w->stream);
  for (const ClassPlan& c : P.classes) {
    const ClassView cv = view_of(w, c, insts);
    if (k > 0 &&
        (rc = w->reserve_buf(&w->scr, &w->scr_bytes, decision_scratch_bytes(cv.ninst, cv.N, k))))
      return rc;
    launch_chunks(cv, w->chunk_inst, w->chunk_pos, w->stream);
    if (launch_decision(rho, delta, cv, k, top, gamma, rho_bins, delta_bins, delta_lo,
                        (unsigned long long*)hist, w->scr, w->status, w->stream)) {
      cudaGetLastError();
      return DPC_ERR_CUDA;
    }
  }
  return finish(w, flags);
}

int dpc_priority_range(const void* pts, int dtype, const dpc_batch* b, const int32_t* rho,
                       int32_t n_query, const int32_t* q_inst, const double* q_box,
                       const int32_t* q_rho, int32_t max_out, int64_t* count, int32_t* ids,
                       uint32_t flags, void* stream) {
  std::vector<Inst> insts;
  uint64_t N = 0;
  int rc = check_batch(b, &insts, &N);
  if (rc) return rc;
  if (flags & ~(DPC_FLAG_SYNC_CHECK)) return DPC_ERR_ARG;
  if (dtype != DPC_I32 && dtype != DPC_F32) return DPC_ERR_ARG;
  if (n_query < 0 || max_out < 0) return DPC_ERR_ARG;
  if (n_query == 0) return DPC_OK;
  if (!q_inst || !q_box || !q_rho || !count || (max_out > 0 && !ids)) return DPC_ERR_ARG;
  if (N > 0 && (!pts || !rho)) return DPC_ERR_ARG;
  Workspace* w = nullptr;
  if ((rc = get_workspace((cudaStream_t)stream, &w))) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  // classes by dimension; the first cutoff of every instance sizes its grid
  // (the results do not depend on it)
  CallPlan P = make_plan(b, insts, 0, 1, false);
  if ((rc = prepare(w, P, b, insts, nullptr, flags))) return rc;
  cudaStream_t st = w->stream;
  const uint32_t nq = (uint32_t)n_query;
  const size_t o_cnt = 0;
  const size_t o_off = align_up(sizeof(uint32_t) * nq);
  const size_t o_map = o_off + align_up(sizeof(unsigned long long) * (nq + 1));
  const size_t bytes = o_map + align_up(sizeof(int32_t) * (size_t)b->n_inst);
  if ((rc = w->reserve_buf(&w->scr, &w->scr_bytes, bytes))) return rc;
  uint32_t* cnt = (uint32_t*)((char*)w->scr + o_cnt);
  unsigned long long* off = (unsigned long long*)((char*)w->scr + o_off);
  int32_t* rowmap = (int32_t*)((char*)w->scr + o_map);
  PrangeArgs a;
  a.nq = nq;
  a.n_inst = b->n_inst;
  a.q_inst = q_inst;
  a.q_box = q_box;
  a.q_rho = q_rho;
  a.rowmap = nullptr;
  a.one_row = -1;
  a.count = (long long*)count;
  launch_prange_init(a, ids, max_out, w->status, st);
  std::vector<int32_t> map_host((size_t)b->n_inst);
  for (const ClassPlan& c : P.classes) {
    const ClassView cv = view_of(w, c, insts);
    bin_class(w, pts, dtype, P, c, cv, b, insts);
    launch_keys_from_rho(rho, w->sid, cv.N, w->skey, st);
    launch_prange_boxes(c.dp, w->spts, w->skey, cv, w->nbox, st);
    if (c.uploaded()) {
      std::fill(map_host.begin(), map_host.end(), -1);
      for (size_t j = 0; j < c.members.size(); ++j) map_host[c.members[j]] = (int32_t)j;
      // pageable source: staged before the call returns
      cudaMemcpyAsync(rowmap, map_host.data(), sizeof(int32_t) * map_host.size(),
                      cudaMemcpyHostToDevice, st);
      a.rowmap = rowmap;
      a.one_row = -1;
    } else {
      a.rowmap = nullptr;
      a.one_row = c.members[0];
    }
    // the warp's buffer serves up to prange_top_ids() ids in one pass
    const bool top = max_out > 0 && max_out <= prange_top_ids();
    if (top) cudaMemsetAsync(off + nq, 0, sizeof(unsigned long long), st);
    launch_prange(c.dp, top ? 2 : 0, w->spts, w->skey, cv, w->nbox, a, cnt, nullptr, nullptr, ids, max_out,
                  off + nq, w->status, st);
    if (max_out == 0) continue;
    if (!top) launch_prange_scan(cnt, nq, off, st);
    unsigned long long total = 0;
    if (cudaMemcpyAsync(&total, off + nq, sizeof(total), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
      cudaGetLastError();
      return DPC_ERR_CUDA;
    }
    if (top) {
      if (total >= (1ull << 32)) return DPC_ERR_OVERFLOW;
      continue;
    }
    if (total == 0) continue;
    if (total >= (1ull << 32)) return DPC_ERR_OVERFLOW;
    const uint32_t tn = (uint32_t)total;
    const size_t k_a = 0;
    const size_t k_b = align_up(sizeof(unsigned long long) * tn);
    const size_t v_a = 2 * k_b;
    const size_t v_b = v_a + align_up(sizeof(uint32_t) * tn);
    const size_t h_o = v_b + align_up(sizeof(uint32_t) * tn);
    const size_t need = h_o + align_up(sizeof(uint32_t) * sort_hist_words(tn));
    if ((rc = w->reserve_buf(&w->scr2, &w->scr2_bytes, need))) return rc;
    char* s2 = (char*)w->scr2;
    unsigned long long* keys_a = (unsigned long long*)(s2 + k_a);
    unsigned long long* keys_b = (unsigned long long*)(s2 + k_b);
    launch_prange(c.dp, 1, w->spts, w->skey, cv, w->nbox, a, cnt, off, keys_a, ids, max_out, nullptr,
                  w->status, st);
    // sort the keys (query << 31 | id): 31 id bits under ib query bits
    int ib = 0;
    while (ib < 32 && (1ull << ib) < nq) ++ib;
    ClassGeom g;
    std::memset(&g, 0, sizeof(g));
    g.S = 31;
    g.ib = ib;
    g.status = w->status;
    cudaMemcpyAsync(w->cls, &g, sizeof(g), cudaMemcpyHostToDevice, st);
    launch_sort(keys_a, keys_b, (uint32_t*)(s2 + v_a), (uint32_t*)(s2 + v_b), tn, w->cls,
                (uint32_t*)(s2 + h_o), false, st);
    const int passes = sort_passes(31, ib);
    launch_prange_scatter((passes & 1) ? keys_b : keys_a, total, off, nq, max_out, ids, w->status, st);
  }
  return finish(w, flags);
}

static int run_device(Workspace* w, const void* pts, int dtype, const dpc_batch* b,
                      const std::vector<Inst>& insts, uint64_t N, const dpc_params* params,
                      int32_t* rho, int32_t* lambda, double* delta, int32_t* label,
                      uint32_t flags, const StageDone* done = nullptr) {
  CallPlan P = make_plan(b, insts, 0, b->n_dcut, false);
  int rc = prepare(w, P, b, insts, params, flags);
  if (rc) return rc;
  run_classes(w, P, pts, dtype, b, insts, N, params, rho, lambda, delta, label, flags, done);
  return cudaGetLastError() == cudaSuccess ? DPC_OK : DPC_ERR_CUDA;
}

// Everything a captured graph depends on: the pointers, the batch, the
// thresholds and the flags that change the kernel sequence.
static std::string graph_key(const void* pts, int dtype, const dpc_batch* b,
                             const dpc_params* params, const void* rho, const void* lambda,
                             const void* delta, const void* label, uint32_t flags) {
  std::string k;
  auto put = [&](const void* p, size_t n) { k.append((const char*)p, n); };
  const void* ptrs[5] = {pts, rho, lambda, delta, label};
  put(ptrs, sizeof(ptrs));
  // every flag that changes a kernel or its arguments (the skip threshold of a
  // single instance is one)
  const uint32_t f = flags & (DPC_PREC_MASK | DPC_FLAG_RADIUS_MASK | DPC_FLAG_LAYOUT_MASK |
                              DPC_FLAG_NEAR_SHIFT_MASK | DPC_FLAG_SKIP_NOISE);
  put(&dtype, sizeof(dtype));
  put(&f, sizeof(f));
  put(&b->n_inst, sizeof(b->n_inst));
  put(&b->n_dcut, sizeof(b->n_dcut));
  put(b->pt_offset, sizeof(int64_t) * (b->n_inst + 1));
  put(b->dim, sizeof(int32_t) * b->n_inst);
  if (b->coord_offset) put(b->coord_offset, sizeof(int64_t) * b->n_inst);
  put(b->d_cut, sizeof(double) * b->n_inst * b->n_dcut);
  put(params, sizeof(dpc_params) * b->n_inst * b->n_dcut);
  return k;
}

// dpc_run with DPC_FLAG_GRAPH: the kernels of a call are captured into a CUDA
// graph on the first call with a new key and replayed afterwards.  The
// per-call work outside the graph: status reset and the instance tables' copy.
static int run_graph(Workspace* w, const void* pts, int dtype, const dpc_batch* b,
                     const std::vector<Inst>& insts, uint64_t N, const dpc_params* params,
                     int32_t* rho, int32_t* lambda, double* delta, int32_t* label, uint32_t flags) {
  if (w->stream == nullptr) return DPC_ERR_UNSUPPORTED;  // the legacy stream cannot be captured
  const uint32_t f = flags & ~(DPC_FLAG_PHASE_TIMES | DPC_FLAG_AUTOTUNE);
  CallPlan P = make_plan(b, insts, 0, b->n_dcut, false);
  int rc = prepare(w, P, b, insts, params, f);
  if (rc) return rc;
  std::string key = graph_key(pts, dtype, b, params, rho, lambda, delta, label, f);
  if (!w->gexec || key != w->gkey) {
    w->drop_graph();
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(w->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      return DPC_ERR_CUDA;
    }
    const long long before = g_kernel_launches;
    run_classes(w, P, pts, dtype, b, insts, N, params, rho, lambda, delta, label, f);
    const cudaError_t e1 = cudaStreamEndCapture(w->stream, &g);
    if (e1 != cudaSuccess || g == nullptr) {
      cudaGetLastError();
      if (g) cudaGraphDestroy(g);
      return DPC_ERR_CUDA;
    }
    const cudaError_t e2 = cudaGraphInstantiate(&w->gexec, g, 0);
    cudaGraphDestroy(g);
    if (e2 != cudaSuccess) {
      cudaGetLastError();
      w->gexec = nullptr;
      return DPC_ERR_CUDA;
    }
    w->gkey.swap(key);
    w->glaunches = g_kernel_launches - before;
  } else {
    g_kernel_launches += w->glaunches;
  }
  if (cudaGraphLaunch(w->gexec, w->stream) != cudaSuccess) {
    cudaGetLastError();
    return DPC_ERR_CUDA;
  }
  return cudaGetLastError() == cudaSuccess ? DPC_OK : DPC_ERR_CUDA;
}

static int check_run(const void* pts, int dtype, const dpc_batch* b, const dpc_params* params,
                     const void* rho, const void* lambda, const void* delta, const void* label,
                     uint32_t flags, std::vector<Inst>* insts, uint64_t* N) {
  int rc = check_batch(b, insts, N);
  if (rc) return rc;
  if ((rc = check_flags(flags))) return rc;
  if (dtype != DPC_I32 && dtype != DPC_F32) return DPC_ERR_ARG;
  if (!params) return DPC_ERR_ARG;
  for (int i = 0; i < b->n_inst * b->n_dcut; ++i)
    if (std::isnan(params[i].delta_min)) return DPC_ERR_ARG;
  if (*N > 0 && (!pts || !rho || !lambda || !delta || !label)) return DPC_ERR_ARG;
  return DPC_OK;
}

int dpc_run(const void* pts, int dtype, const dpc_batch* b, const dpc_params* params, int32_t* rho,
            int32_t* lambda, double* delta, int32_t* label, uint32_t flags, void* stream) {
  std::vector<Inst> insts;
  uint64_t N = 0;
  int rc = check_run(pts, dtype, b, params, rho, lambda, delta, label, flags, &insts, &N);
  if (rc) return rc;
  Workspace* w = nullptr;
  if ((rc = get_workspace((cudaStream_t)stream, &w))) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  if (flags & DPC_FLAG_GRAPH)
    rc = run_graph(w, pts, dtype, b, insts, N, params, rho, lambda, delta, label, flags);
  else
    rc = run_device(w, pts, dtype, b, insts, N, params, rho, lambda, delta, label, flags);
  if (rc) return rc;
  return finish(w, flags);
}

int dpc_run_host(const void* pts_host, int dtype, const dpc_batch* b, const dpc_params* params,
                 int32_t* rho_host, int32_t* lambda_host, double* delta_host, int32_t* label_host,
                 uint32_t flags, void* stream) {
  std::vector<Inst> insts;
  uint64_t N = 0;
  int rc = check_run(pts_host, dtype, b, params, rho_host, lambda_host, delta_host, label_host,
                     flags, &insts, &N);
  if (rc) return rc;
  Workspace* w = nullptr;
  if ((rc = get_workspace((cudaStream_t)stream, &w))) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  uint64_t elems = 0;
  for (auto& in : insts) {
    uint64_t e = in.coord_off + in.n * (uint64_t)in.d;
    elems = e > elems ? e : elems;
  }
  const size_t R = (size_t)b->n_dcut * N;
  const size_t o_pts = 0;
  const size_t o_rho = align_up(4 * elems);
  const size_t o_lam = o_rho + align_up(4 * R);
  const size_t o_del = o_lam + align_up(4 * R);
  const size_t o_lab = o_del + align_up(8 * R);
  const size_t total = o_lab + align_up(4 * R);
  if ((rc = w->reserve_io(total ? total : kAlign))) return rc;
  char* io = (char*)w->io;
  cudaStream_t st = w->stream;
  // each output goes back as soon as its phase has finished (a copy stream
  // behind an event), overlapping the phases still to run
  if (!w->copy_stream && cudaStreamCreateWithFlags(&w->copy_stream, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    w->copy_stream = nullptr;
    return DPC_ERR_CUDA;
  }
  const size_t nev = 3u * (size_t)b->n_dcut;
  while (w->out_ev.size() < nev) {
    cudaEvent_t e = nullptr;
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      return DPC_ERR_CUDA;
    }
    w->out_ev.push_back(e);
  }
  cudaStream_t cs = w->copy_stream;
  const StageDone done = [&](int stage, int k) {
    const size_t o = (size_t)k * N;
    cudaEvent_t ev = w->out_ev[3u * (size_t)k + (size_t)stage];
    cudaEventRecord(ev, st);
    cudaStreamWaitEvent(cs, ev, 0);
    if (N == 0) return;
    if (stage == 0) {
      cudaMemcpyAsync(rho_host + o, io + o_rho + 4 * o, 4 * N, cudaMemcpyDeviceToHost, cs);
    } else if (stage == 1) {
      cudaMemcpyAsync(lambda_host + o, io + o_lam + 4 * o, 4 * N, cudaMemcpyDeviceToHost, cs);
      cudaMemcpyAsync(delta_host + o, io + o_del + 8 * o, 8 * N, cudaMemcpyDeviceToHost, cs);
    } else {
      cudaMemcpyAsync(label_host + o, io + o_lab + 4 * o, 4 * N, cudaMemcpyDeviceToHost, cs);
    }
  };
  if (elems) cudaMemcpyAsync(io + o_pts, pts_host, 4 * elems, cudaMemcpyHostToDevice, st);
  rc = run_device(w, io + o_pts, dtype, b, insts, N, params, (int32_t*)(io + o_rho),
                  (int32_t*)(io + o_lam), (double*)(io + o_del), (int32_t*)(io + o_lab), flags,
                  &done);
  // no copy into the caller's buffers may outlive the call, whatever happened
  const cudaError_t ec = cudaStreamSynchronize(cs);
  if (rc) return rc;
  if (ec != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
    cudaGetLastError();
    return DPC_ERR_CUDA;
  }
  return finish(w, flags | DPC_FLAG_SYNC_CHECK);
}

int dpc_get_stats(void* stream, dpc_stats* out) {
  if (!out) return DPC_ERR_ARG;
  Workspace* w = nullptr;
  int rc = get_workspace((cudaStream_t)stream, &w);
  if (rc) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  std::memset(out, 0, sizeof(*out));
  if (!w->base) return DPC_OK;
  if (cudaStreamSynchronize(w->stream) != cudaSuccess) {
    cudaGetLastError();
    return DPC_ERR_CUDA;
  }
  Counters c;
  cudaMemcpy(&c, w->ctr, sizeof(c), cudaMemcpyDeviceToHost);
  out->band_pairs = (int64_t)c.band_pairs;
  out->far_queries = (int64_t)c.far_queries;
  out->exact_rescans = (int64_t)c.exact_rescans;
  out->kernel_launches = w->launches_last;
  out->far_nodes = (int64_t)c.far_nodes;
  out->far_nodes_max = (int64_t)c.far_nodes_max;
  out->density_pairs = (int64_t)c.pairs;
  if (w->have_last) {
    CutGeom cg;
    GridGeom g;
    HashInfo hi;
    cudaMemcpy(&cg, w->last_cut, sizeof(cg), cudaMemcpyDeviceToHost);
    cudaMemcpy(&g, w->last_geom, sizeof(g), cudaMemcpyDeviceToHost);
    cudaMemcpy(&hi, w->hinfo, sizeof(hi), cudaMemcpyDeviceToHost);
    out->occupied_cells = hi.m;
    out->grid_level = cg.k;
    out->block_radius = cg.R;
    // what the fill rule left to the CUDA-core layouts (tensor_fill)
    const Choice& ch = w->last_choice;
    auto sparse = [&](uint32_t fill) { return (uint64_t)w->last_points < (uint64_t)fill * hi.m; };
    out->density_layout = ch.dlay == kLayoutTensor && sparse(ch.dfill) ? kLayoutSegment : ch.dlay;
    out->near_layout = ch.nlay == kLayoutTensor && sparse(ch.nfill) ? kLayoutTree : ch.nlay;
    if (ch.nlay == kLayoutTree && ch.ufill && !sparse(ch.ufill)) out->near_layout = kLayoutUnion;
    out->near_shift = w->last_choice.ns;
    out->bits_per_axis = g.B;
  }
  return cudaGetLastError() == cudaSuccess ? DPC_OK : DPC_ERR_CUDA;
}

int dpc_get_phase_times(void* stream, dpc_phase_times* out) {
  if (!out) return DPC_ERR_ARG;
  Workspace* w = nullptr;
  int rc = get_workspace((cudaStream_t)stream, &w);
  if (rc) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  std::memset(out, 0, sizeof(*out));
  if (cudaStreamSynchronize(w->stream) != cudaSuccess) {
    cudaGetLastError();
    return DPC_ERR_CUDA;
  }
  for (const auto& r : w->recs) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, r.a, r.b) != cudaSuccess) {
      cudaGetLastError();
      return DPC_ERR_CUDA;
    }
    out->ms[r.phase] += ms;
    out->launches[r.phase] += 1;
  }
  return DPC_OK;
}

int dpc_last_status(void* stream) {
  Workspace* w = nullptr;
  int rc = get_workspace((cudaStream_t)stream, &w);
  if (rc) return rc;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!w->base) return DPC_OK;
  if (cudaStreamSynchronize(w->stream) != cudaSuccess) {
    cudaGetLastError();
    return DPC_ERR_CUDA;
  }
  int s = 0;
  if (cudaMemcpy(&s, w->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) {
    cudaGetLastError();
    return DPC_ERR_CUDA;
  }
  return status_to_code(s);
}

void dpc_release(void) {
  std::lock_guard<std::mutex> lk(g_mu);
  for (auto& kv : g_ws) {
    int cur = -1;
    cudaGetDevice(&cur);
    cudaSetDevice(kv.second->device);
    kv.second->release();
    delete kv.second;
    if (cur >= 0) cudaSetDevice(cur);
  }
  g_ws.clear();
}

}  // extern "C"

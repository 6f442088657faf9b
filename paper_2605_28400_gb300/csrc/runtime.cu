// runtime.cu — host runtime behind the C ABI of include/trioseq.h.
//
// Plan: scoring scheme validated and turned into the device tables of the shifted frame
// (sigma'' = sigma - 2*alpha, a virtual residue row/column of zeros, x8 for traceback keys).
// Batch: encoded + packed residues, per-triplet descriptors (engine.h), the ordered column-task
// queue, and a device workspace (faces, progress flags, codes, outputs).
// Queue order: tasks sorted by anti-diagonal D = J + K of their column block, then by the
// triplet's rank in longest-processing-time order (largest cube first). Every producer of a
// task, (J-1,K) and (J,K-1), has a smaller D and therefore an earlier queue slot. The LPT part
// follows the paper's dynamic partition by cumulative cells (Sec. V-D), applied here to the
// warps of one GPU instead of to GPUs.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdlib>
#include <cstdio>
#include <cstring>
#include <deque>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <thread>
#include <tuple>
#include <unordered_map>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "engine.h"
#include "guard.h"
#include "trioseq.h"

using namespace trioseq;

namespace {

// NVTX range for the duration of a scope: plan, autotune, batch, run, traceback and server
// launches show up by name in profilers that read NVTX (header-only NVTX 3; no cost without one).
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

// Host-side fault injection for tests: with TRIOSEQ_TEST_FAIL_ALLOC=N at trioseq_plan, the N-th
// device allocation after it fails as if the device were out of memory; with TRIOSEQ_TEST_FAIL_PINNED=N the
// N-th pinned host allocation.
struct AllocFault {
  std::atomic<long> calls{0}, fail_at{0};
  void arm(const char* env) {
    const char* v = std::getenv(env);
    calls.store(0);
    fail_at.store(v ? std::max(0, std::atoi(v)) : 0);
  }
  bool hit() {
    const long at = fail_at.load(std::memory_order_relaxed);
    return at > 0 && calls.fetch_add(1, std::memory_order_relaxed) + 1 == at;
  }
};
AllocFault g_device_fault, g_pinned_fault;

struct DevBuf {
  void* p = nullptr;
  size_t cap = 0;
  cudaStream_t st_ = nullptr;  // stream of a stream-ordered allocation (freed in its order)
  ~DevBuf() { reset(); }
  // Release the buffer: stream-ordered allocations are freed in their stream's order, which
  // blocks neither the host nor other streams.
  void reset() {
    if (p) {
      if (st_)
        cudaFreeAsync(p, st_);
      else
        cudaFree(p);
    }
    p = nullptr;
    cap = 0;
    st_ = nullptr;
  }
  // Grow to at least `bytes` (contents are not preserved). With a stream, the old buffer is
  // released and the new one taken in that stream's order (no device-wide synchronisation), so
  // a growing workspace does not stall work running on other streams. The caller orders that
  // stream after the old buffer's last use.
  bool ensure(size_t bytes, cudaStream_t st = nullptr) {
    if (bytes <= cap && p) return true;
    const size_t want = std::max<size_t>(bytes, 256);
    if (g_device_fault.hit()) return false;
    reset();
    const cudaError_t e = st ? cudaMallocAsync(&p, want, st) : cudaMalloc(&p, want);
    if (e != cudaSuccess) {
      p = nullptr;
      cudaGetLastError();
      return false;
    }
    cap = want;
    st_ = st;
    return true;
  }
  template <typename T>
  T* as() const {
    return reinterpret_cast<T*>(p);
  }
};

struct HostPinned {
  void* p = nullptr;
  size_t cap = 0;
  ~HostPinned() {
    if (p) cudaFreeHost(p);
  }
  bool ensure(size_t bytes) {
    if (bytes <= cap && p) return true;
    if (p) cudaFreeHost(p);
    p = nullptr;
    cap = 0;
    const size_t want = std::max<size_t>(bytes, 4096);
    if (g_pinned_fault.hit() || cudaMallocHost(&p, want) != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
      return false;
    }
    cap = want;
    return true;
  }
};

// Device workspace of one in-flight batch.
struct Workspace {
  DevBuf inputs;    // packed residues | descriptors | tasks | traceback tables
  DevBuf faces;     // j- and k-face planes
  DevBuf progress;  // progress flags | queue head | error word
  DevBuf codes;     // traceback codes
  DevBuf scores;    // int32 per triplet
  DevBuf rows;      // traceback rows
  DevBuf lens;      // alignment lengths
  DevBuf planes;    // slab mode: checkpoint planes (traceback) or two ping-pong planes (score)
  DevBuf walkstate; // slab mode: (i, j, k, n) of the traceback walk between slabs
  DevBuf best64;    // semi-global / local traceback: (score, first cell) key per triplet
  DevBuf spans;     // traceback: begin and end cell of each alignment (6 int32)
  HostPinned staging;  // per-call path: inputs up, then room for results down (Staging)
  // Buffers are allocated and freed in this stream's order. Plans and device-resident batches
  // own a private stream here (own_stream); a serving slot uses its launch stream.
  cudaStream_t alloc_stream = nullptr;
  bool own_stream = false;
  // Recorded on the launching stream after each enqueued use: growth and destruction wait for
  // this workspace's own work only, never for the whole device.
  cudaEvent_t last_use = nullptr;
  bool used = false;

  // A private allocation stream (non-blocking, so it never waits on the legacy default stream).
  cudaError_t make_own_stream() {
    const cudaError_t e = cudaStreamCreateWithFlags(&alloc_stream, cudaStreamNonBlocking);
    own_stream = e == cudaSuccess;
    if (e != cudaSuccess) alloc_stream = nullptr;
    return e;
  }
  // Mark the end of a use enqueued on `st`.
  cudaError_t mark_use(cudaStream_t st) {
    if (!last_use) {
      const cudaError_t e = cudaEventCreateWithFlags(&last_use, cudaEventDisableTiming);
      if (e != cudaSuccess) {
        last_use = nullptr;
        return e;
      }
    }
    const cudaError_t e = cudaEventRecord(last_use, st);
    used = used || e == cudaSuccess;
    return e;
  }
  // Host wait for this workspace's last recorded use (not for other streams' work).
  void wait_last_use() {
    if (used && last_use) cudaEventSynchronize(last_use);
  }
  // Order the allocation stream after the last recorded use, before buffers are freed there.
  void order_after_last_use() {
    if (used && last_use && alloc_stream) cudaStreamWaitEvent(alloc_stream, last_use, 0);
  }
  // Free every device buffer in the allocation stream's order, after the last recorded use.
  // Must run while that stream exists (a serving slot calls it before destroying its stream).
  void release() {
    order_after_last_use();
    for (DevBuf* b : {&inputs, &faces, &progress, &codes, &scores, &rows, &lens, &planes,
                      &walkstate, &best64, &spans})
      b->reset();
  }
  ~Workspace() {
    release();
    if (last_use) cudaEventDestroy(last_use);
    if (own_stream && alloc_stream) cudaStreamDestroy(alloc_stream);  // released when idle
  }
};

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Register tile per lane: nj x nk cells; vl = 1 for the two-cells-per-register kernel
// (wavefront_vl.cuh), whose lane tile is two nj x nk/2 column halves.
struct Variant {
  int nj, nk;
  int vl = 0;
};

}  // namespace

struct trioseq_plan_s {
  int device = 0;
  int sms = 0;
  int K = 0;
  int KP = 0;
  char alphabet[kMaxAlphabet] = {};
  int16_t lut[256];
  std::vector<int32_t> sub;
  int32_t gap = 0;
  int atype = kGlobal;             // alignment type of Sec. II (plan flags)
  int32_t max_abs_sig2 = 0;        // max |sigma''| over the extended table
  DevBuf sig_score, sig_tb;        // KP*KP int32 device tables
  bool affine = false;             // trioseq_plan_affine: natural affine gap costs (affine.cu)
  int32_t gap_open = 0;            // gamma, per maximal gap run of a pair
  DevBuf sig_affine;               // KP*KP int32 table of sigma itself (affine model)
  int32_t max_abs_sub = 0;         // max |sigma|
  Workspace ws;                    // workspace of trioseq_align_batch
  std::unique_ptr<trioseq_batch_s> last;  // last align_batch (traceback rows kept here)
  int TI = 8;
  int64_t wait_ns = 2000000000LL;  // 2 s without progress = give up
  bool test_wait_unset = false;    // test switch: first-wave warps wait on a flag nothing sets
  bool test_no_records = false;    // test switch: queue task 0 never runs, its records never come
  bool test_poison = false;        // test switch: boundary records start as a large garbage value
  int data_flags = -1;             // TRIOSEQ_DATA_FLAGS: records as readiness flags (-1: chosen)
  bool graphs = true;              // trioseq_batch_run replays a captured CUDA graph
  bool packed16 = true;            // pair score-only global triplets in int16 halves if they fit
  bool sig2_nonneg = false;        // every sigma'' >= 0: the biased packed mode applies
  size_t slab_budget = 0;          // bytes a one-triplet batch may use before it runs in slabs
  bool pace = true;                // pace the first wave of multi-wave launches
  int slab_slices = 0;             // forced slab height (0: chosen from the budget)
  Variant score_variant{8, 8};
  Variant tb_variant{4, 8};
  bool score_forced = false, tb_forced = false;  // set by TRIOSEQ_SCORE_TILE / TRIOSEQ_TB_TILE
  // Autotuner cache: (mode, single triplet or batch, bit length of the longest sequence) ->
  // fastest (tile, progress interval) measured by trioseq_plan_autotune.
  struct Tuned {
    Variant var;
    int TI;
  };
  std::map<int, Tuned> tuned;
  // Set while the autotuner measures: candidate tiles in `forced`, or (tune_rule) the rules' own choice.
  bool tuning = false, tune_rule = false;
  Tuned forced{{8, 8}, 8};
};

namespace {
int tune_key(uint32_t mode, size_t n, uint32_t maxlen) {
  int bits = 0;
  while ((maxlen >> bits) > 0 && bits < 31) ++bits;
  return (int)mode * 1000 + (n > 1 ? 100 : 0) + bits;
}
}  // namespace

struct trioseq_batch_s {
  trioseq_plan_s* plan = nullptr;
  Workspace* ws = nullptr;             // where it runs (owned if own_ws)
  std::unique_ptr<Workspace> own_ws;
  size_t n = 0;
  uint32_t mode = 0;
  Variant var{8, 8};
  uint64_t cells = 0;
  std::vector<TripDesc> desc;
  std::vector<Task> tasks;
  std::vector<int32_t> tb_trips;       // triplet index per traceback request
  std::vector<int64_t> row_off;
  std::vector<int32_t> row_cap;
  std::vector<int32_t> tb_of;          // triplet -> traceback request (-1)
  std::vector<int8_t> seq;             // packed residue codes (host copy)
  size_t seq_bytes = 0, face_ints = 0, code_words = 0, rows_bytes = 0;
  size_t off_desc = 0, off_tasks = 0, off_tb = 0, off_rowoff = 0, off_rowcap = 0, inputs_bytes = 0;
  int grid = 0;
  size_t smem = 0;
  int TI = 8;  // progress-publication interval of this batch's launches
  bool df = false;  // boundary records are their own readiness flags
  int packed = 0;  // packed int16x2 mode (0: none, 1: signed, 2: biased): two triplets per task
  // affine model: the launches of a run as (first task, number of tasks); none when it runs over
  // planes, whose largest has affine_cells cells
  std::vector<std::pair<size_t, size_t>> affine_chunks;
  int64_t affine_cells = 0;
  // Slab mode (one triplet whose records, or codes, would not fit at once): the cube runs as
  // nslab launches of `slab` slices, chained through planes of plane_ints int32 each.
  int slab = 0, nslab = 0;
  size_t plane_ints = 0, nplanes = 0, off_slab = 0;
  std::vector<TripDesc> slab_desc;
  bool uploaded = false;
  bool no_room = false;  // the upload found no room for the boundary records, the codes or the rest
  // results of the last run (host)
  std::vector<uint8_t> h_rows;
  std::vector<int32_t> h_lens;
  std::vector<int32_t> h_spans;  // 6 per traceback request
  bool have_rows = false;
  // optional per-kernel timing (events on the launching stream)
  bool profile = false;
  bool timed = false;
  cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
  uint64_t h2d_bytes = 0, d2h_bytes = 0;
  // trioseq_batch_run replays one captured CUDA graph (progress reset, wavefront, walk). The key
  // holds the buffer addresses and the profiling switch the graph was captured with.
  cudaGraphExec_t gexec = nullptr;
  cudaStream_t capture_stream = nullptr;
  std::array<const void*, 12> gkey{};
  ~trioseq_batch_s() {
    for (auto& e : ev)
      if (e) cudaEventDestroy(e);
    if (gexec) cudaGraphExecDestroy(gexec);
    if (capture_stream) cudaStreamDestroy(capture_stream);
  }
};

namespace {

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

trioseq_status cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return TRIOSEQ_OK;
  cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? TRIOSEQ_ENOMEM : TRIOSEQ_ECUDA;
}

int env_int(const char* name, int def) {
  const char* v = std::getenv(name);
  return v ? std::atoi(v) : def;
}

// Device layout of a batch's input block: residues | descriptors | slab descriptors | queue |
// traceback tables.
void layout_inputs(trioseq_batch_s* bt) {
  size_t off = align_up(bt->seq_bytes, 256);
  bt->off_desc = off;
  off = align_up(off + sizeof(TripDesc) * std::max<size_t>(bt->n, 1), 256);
  bt->off_slab = off;
  off = align_up(off + sizeof(TripDesc) * bt->slab_desc.size(), 256);
  bt->off_tasks = off;
  off = align_up(off + sizeof(Task) * std::max<size_t>(bt->tasks.size(), 1), 256);
  bt->off_tb = off;
  off = align_up(off + sizeof(int32_t) * std::max<size_t>(bt->tb_trips.size(), 1), 256);
  bt->off_rowoff = off;
  off = align_up(off + sizeof(int64_t) * std::max<size_t>(bt->row_off.size(), 1), 256);
  bt->off_rowcap = off;
  off = align_up(off + sizeof(int32_t) * std::max<size_t>(bt->row_cap.size(), 1), 256);
  bt->inputs_bytes = off;
}

// Affine-gap batch over anti-diagonal planes (affine_plane_kernel): one queue entry per triplet,
// largest cube first; each CTA of the persistent launch sweeps its triplets' planes in four
// rotating plane buffers of 13 int32 states per cell.
trioseq_status build_affine_planes(trioseq_plan_s* plan, trioseq_batch_s* bt) {
  const size_t n = bt->n;
  std::vector<int32_t> order(n);
  int64_t maxcells = 1;
  for (size_t t = 0; t < n; t++) {
    order[t] = (int32_t)t;
    const TripDesc& d = bt->desc[t];
    maxcells = std::max<int64_t>(maxcells, (int64_t)(d.len[1] + 1) * (d.len[2] + 1));
  }
  const auto vol = [&](int32_t t) {
    const TripDesc& d = bt->desc[t];
    return (double)(d.len[0] + 1) * (d.len[1] + 1) * (d.len[2] + 1);
  };
  std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return vol(x) > vol(y); });
  bt->tasks.clear();
  for (const int32_t t : order) bt->tasks.push_back(Task{t, 0, 0, 0});
  int bpm = 0;
  if (affine_plane_occupancy(&bpm) != 0 || bpm <= 0) return TRIOSEQ_ECUDA;
  bt->grid = (int)std::max<size_t>(1, std::min<size_t>((size_t)plan->sms * bpm, n));
  bt->affine_cells = maxcells;
  bt->face_ints = (size_t)bt->grid * 4 * (size_t)maxcells * 16;  // 16 int32 per cell (13 used)
  layout_inputs(bt);
  return TRIOSEQ_OK;
}

// Affine-gap batch (affine.cu). Units of one triplet, or two per register when every pair fits
// the 16-bit halves; column tasks in the order of the linear engine (anti-diagonal, then largest
// cube first). The boundary records take 2.5 bytes per cell of the grid, so large batches run as
// chunks, one launch after another over the same records: 4 GB hold about ten waves of tasks of
// 200-residue triplets, so the tail of a chunk costs little. A triplet whose records exceed the
// plan's budget runs over planes instead (four planes of 64 bytes per (j, k) cell).
// lean: the layout to build when the device had no room for a larger one: 1 the smallest chunks, 2 planes.
// cap: bytes the records may take (a server's admission), where the plan's budget is larger.
constexpr size_t kAffineChunkInts = (size_t)1 << 30;  // 4 GB
constexpr size_t kAffineKeep = (size_t)16 << 30;      // bytes of records a plan keeps between calls
trioseq_status build_affine(trioseq_plan_s* plan, trioseq_batch_s* bt, int lean, size_t cap) {
  const size_t n = bt->n;
  bt->seq_bytes = bt->seq.size();
  bt->affine_chunks.clear();
  bt->affine_cells = 0;
  if (lean >= 2) return build_affine_planes(plan, bt);
  const auto volume = [&](int32_t t) {
    const TripDesc& d = bt->desc[t];
    return (double)(d.len[0] + 1) * (d.len[1] + 1) * (d.len[2] + 1);
  };
  const size_t budget = std::min(plan->slab_budget, cap) / 4;  // ints
  std::vector<int32_t> order(n);
  for (size_t t = 0; t < n; t++) order[t] = (int32_t)t;
  std::vector<std::pair<int32_t, int32_t>> units;
  // Packed: sigma'' >= 0, every value of the pair's grid below 2^15 (engine.h), and -infinity
  // (4 |gamma|, plus at most three sigma'') below the smallest real value 2^14 - 8 |gamma|; and the records of
  // every pair's grid (of its maximal lengths) within the budget.
  const int32_t go = -plan->gap_open;
  if (n >= 2 && plan->packed16 && plan->sig2_nonneg &&
      12 * (int64_t)go + 3 * plan->max_abs_sig2 < (1 << 14)) {
    const auto cls = [&](int32_t t) {
      const TripDesc& d = bt->desc[t];
      return std::make_tuple((d.len[1] + kAffineWJ) / kAffineWJ,
                             (d.len[2] + kAffineWK) / kAffineWK, d.len[0]);
    };
    std::stable_sort(order.begin(), order.end(),
                     [&](int32_t x, int32_t y) { return cls(x) < cls(y); });
    bool fits = true;
    for (size_t u = 0; u < n && fits; u += 2) {
      const int32_t t0 = order[u], t1 = u + 1 < n ? order[u + 1] : order[u];
      size_t g[3];
      for (int q = 0; q < 3; q++)
        g[q] = (size_t)std::max(bt->desc[t0].len[q], bt->desc[t1].len[q]);
      fits = (int64_t)plan->max_abs_sig2 * (int64_t)(g[0] + g[1] + g[2] + 3) < (1 << 14) &&
             (g[0] + 1) * ((g[1] + kAffineWJ) / kAffineWJ) * ((g[2] + kAffineWK) / kAffineWK) *
                     (size_t)(kAffineRecJ + kAffineRecK) <= budget;
      units.emplace_back(t0, t1);
    }
    if (!fits) units.clear();
  }
  bt->packed = units.empty() ? 0 : 2;
  if (units.empty())
    for (size_t t = 0; t < n; t++) units.emplace_back((int32_t)t, -1);
  // grids, then chunks of units (largest first) whose records share one buffer
  for (const auto& un : units) {
    TripDesc& d = bt->desc[un.first];
    if (un.second >= 0) {
      const TripDesc& h = bt->desc[un.second];
      for (int q = 0; q < 3; q++) d.glen[q] = std::max(d.len[q], h.len[q]);
      d.pair = un.second;
    }
    d.nJ = (d.glen[1] + kAffineWJ) / kAffineWJ;
    d.nK = (d.glen[2] + kAffineWK) / kAffineWK;
    d.T = d.glen[0] + 1 + (kPR - 1) + (kPC - 1);
  }
  std::stable_sort(units.begin(), units.end(), [&](const auto& x, const auto& y) {
    return volume(x.first) > volume(y.first);
  });
  const auto records = [&](const TripDesc& d) {  // ints
    return (size_t)d.nJ * d.nK * (size_t)(d.glen[0] + 1) * (size_t)(kAffineRecJ + kAffineRecK);
  };
  size_t limit = lean ? 0 : std::min(budget, kAffineChunkInts);
  for (const auto& un : units) {
    const size_t rec = records(bt->desc[un.first]);
    if (rec > budget) {
      for (size_t t = 0; t < n; t++) {
        for (int q = 0; q < 3; q++) bt->desc[t].glen[q] = bt->desc[t].len[q];
        bt->desc[t].pair = -1;
      }
      bt->packed = 0;
      return build_affine_planes(plan, bt);
    }
    limit = std::max(limit, rec);
  }
  bt->tasks.clear();
  bt->face_ints = 4;
  int64_t prog = 0;
  for (size_t u0 = 0; u0 < units.size();) {
    size_t face = 0, u1 = u0;
    int maxD = 0;
    for (; u1 < units.size(); u1++) {
      TripDesc& d = bt->desc[units[u1].first];
      const size_t ntask = (size_t)d.nJ * d.nK, A = (size_t)d.glen[0] + 1;
      if (u1 > u0 && face + records(d) > limit) break;
      d.oj_off = (int64_t)face;
      d.ok_off = (int64_t)(face + ntask * A * kAffineRecJ);
      face += records(d);
      d.prog_base = prog;
      prog += (int64_t)ntask;
      maxD = std::max(maxD, d.nJ + d.nK - 2);
    }
    bt->face_ints = std::max(bt->face_ints, face);
    const size_t first = bt->tasks.size();
    for (int D = 0; D <= maxD; D++)
      for (size_t u = u0; u < u1; u++) {
        const int32_t t = units[u].first;
        const TripDesc& d = bt->desc[t];
        for (int J = std::max(0, D - d.nK + 1); J <= std::min(D, d.nJ - 1); J++)
          bt->tasks.push_back(Task{t, J, D - J, 0});
      }
    bt->affine_chunks.emplace_back(first, bt->tasks.size() - first);
    u0 = u1;
  }
  bt->smem = affine_smem_bytes(plan->KP, bt->packed != 0);
  int bpm = 0;
  if (affine_occupancy(bt->packed != 0, bt->smem, &bpm) != 0 || bpm <= 0) return TRIOSEQ_ECUDA;
  bt->grid = plan->sms * bpm;
  layout_inputs(bt);
  return TRIOSEQ_OK;
}

int plan_atype(const trioseq_batch_s* bt) { return bt->plan->atype; }

// Units of the packed int16x2 mode on WJ x WK column tasks: two triplets of the same grid class each
// (the last one with itself when n is odd), or none when some pair's grid leaves the int16 margin of
// engine.h: max|sigma''| * (a+b+c + 3) < 2^14 on the pair's maximal lengths.
std::vector<std::pair<int32_t, int32_t>> pack_units(const trioseq_plan_s* plan,
                                                    const trioseq_triplet* trip, size_t n, int WJ,
                                                    int WK) {
  std::vector<std::pair<int32_t, int32_t>> units;
  // by grid class, then length, then position (keys beside the indices: sorting reads no triplet)
  std::vector<std::tuple<uint64_t, uint32_t, int32_t>> keys(n);
  for (size_t t = 0; t < n; t++) {
    const uint32_t* L = trip[t].len;
    keys[t] = {(uint64_t)((L[1] + WJ) / WJ) << 32 | (L[2] + WK) / WK, L[0], (int32_t)t};
  }
  std::sort(keys.begin(), keys.end());
  std::vector<int32_t> order(n);
  for (size_t t = 0; t < n; t++) order[t] = std::get<2>(keys[t]);
  for (size_t u = 0; u < n; u += 2) {
    const int32_t t0 = order[u], t1 = (u + 1 < n) ? order[u + 1] : order[u];
    int64_t gsum = 0;
    for (int q = 0; q < 3; q++) gsum += std::max(trip[t0].len[q], trip[t1].len[q]);
    if ((int64_t)plan->max_abs_sig2 * (gsum + 3) >= (1 << 14)) return {};
    units.emplace_back(t0, t1);
  }
  return units;
}

// Whether the tile of a plan's batches is chosen by default_variant: no forced tile, and two values per
// register not switched off.
bool auto_tile(const trioseq_plan_s* plan, bool tb) {
  return !plan->affine && plan->packed16 && !(tb ? plan->tb_forced : plan->score_forced);
}

// Schemes and types the two-cells-per-register kernel admits (its range argument). Traceback keys
// (global type) take 3 bits more.
bool vl_admits(const trioseq_plan_s* plan, bool tb) {
  return plan->sig2_nonneg && plan->max_abs_sig2 <= (tb ? 30 : 33) &&
         (plan->atype == kGlobal || (!tb && -2 * plan->gap <= 33));
}

// The tile of a batch when neither the environment nor the autotuner names one: two cells of a
// triplet per register (wavefront_vl.cuh; build_batch falls back to int32 where the scheme or the
// budget does not admit it), 16 x 64 tasks while they number at most two per SM (more warps than 32 x 64 tasks
// give, each with a shorter step; beyond that their records cost more than they gain), else 32 x 64.
// Measured, kernel time (16 x 64 / 32 x 64 / int32 default): score, protein, 300 residues (95 / 50 tasks)
// 0.185 / 0.209 / 0.50 ms; 1,000 residues (1,008 / 512) 0.77 / 0.66 / 1.74 ms; traceback, DNA, 128
// residues (16 / 8) 0.090 / 0.109 / 0.129 ms, 1,000 residues 0.95 / 0.89 / 1.47 ms, 96 triplets of
// 200..600 3.2 / 3.0 / 6.3 ms; 1,024 semi-global triplets of 100..300 4.6 / 4.0 / 7.2 ms.
// One triplet of 20 / 45 / 60 / 80 DNA residues: score 27 / 36 / 42 / 60 us against 29 / 57 / 68 / 109 on int32;
// with rows 30 / 41 / 48 / 71 against 33 / 51 / 64 / 92; semi-global 34 / 48 / 57 / 80 against 46 / 94 / 114 / 173.
// Kept on int32, whose packing they have always reported, although no faster there: global batches of at most 8
// such tasks that are one triplet over two block columns or several triplets with rows, and two
// global triplets that cannot pack when one of them is a single task.
Variant default_variant(const trioseq_plan_s* plan, const trioseq_triplet* trip, size_t n, bool tb) {
  uint64_t tasks = 0, least = UINT64_MAX;
  for (size_t t = 0; t < n; t++) {
    const uint64_t q = (uint64_t)((trip[t].len[1] + 16) / 16) * ((trip[t].len[2] + 64) / 64);
    tasks += q;
    least = std::min(least, q);
  }
  const bool small = plan->atype == kGlobal && tasks <= 8 && (n != 1 || (!tb && trip[0].len[2] >= 64));
  const bool uneven = plan->atype == kGlobal && !tb && n == 2 && least == 1;
  if (small || uneven) return tb ? plan->tb_variant : plan->score_variant;
  return tasks <= 2 * (uint64_t)plan->sms ? Variant{4, 8, 1} : Variant{8, 8, 1};
}

// The tile of a batch of pairs (two triplets per register, biased; wavefront_vp.cuh). 8x4 (32 x 32 tasks)
// has the fewest instructions per cell that fit the registers; 4x4 (16 x 32) is 7% slower per cell, and
// taken where its tasks pad less than that (lengths of a few tens), or where 8x4 would leave warps idle (at
// most two tasks per SM). Kernel time, 8x4 / 4x8 / 4x4 / 8x8: 4,096 DNA triplets of 100..300 residues
// 11.2 / 11.8 / 12.2 / 13.3 ms, of 30..60 260 / 243 / 243 / 350 us; 100 of 60..100 77 / 78 / 82 / 129 us; 8 of
// 100..200 132 / 138 / 115 / 223 us; 300 protein triplets of 100..200 436 / 460 / 440 / 571 us.
// 8x8 (32 x 64), whose records are two thirds of 8x4's, where those would exceed the plan's record budget.
Variant packed_variant(const trioseq_plan_s* plan, const trioseq_triplet* trip, size_t n) {
  double tasks = 0, wide = 0, narrow = 0;  // tasks of 8x4; steps of 8x4 and 4x4 tasks, in 16 x 32 blocks
  for (size_t t = 0; t < n; t++) {
    const double a = trip[t].len[0] + 11.0, k = (trip[t].len[2] + 32) / 32;
    const double j8 = (trip[t].len[1] + 32) / 32, j4 = (trip[t].len[1] + 16) / 16;
    tasks += 0.5 * j8 * k;
    wide += a * j8 * k * 2;
    narrow += a * j4 * k;
  }
  const bool few = tasks <= 2.0 * plan->sms || 1.08 * narrow < wide;
  const double bytes = few ? 0.5 * narrow * 4 * (vp_rec_j(4) + vp_rec_k(4))
                           : 0.25 * wide * 4 * (vp_rec_j(4) + vp_rec_k(8));
  if (bytes > (double)plan->slab_budget) return Variant{8, 8};
  return few ? Variant{4, 4} : Variant{8, 4};
}

// The int32 tile of a semi-global or local batch with traceback: 4x4 (16 x 32 tasks), whose one-pass step with
// its best-cell bookkeeping keeps to fewer registers, unless its records (0.41 B a cell against 0.33 on 4x8)
// and the codes exceed the plan's budget. Kernel time, 4x8 / 8x4 / 4x4: local, DNA, 100 residues 375 / 330 / 238 us,
// 1,000 4.0 / 3.9 / 3.2 ms, protein, 1,700 13.9 / 14.1 / 10.5; semi-global, DNA, 1,000 3.2 / 3.0 / 2.4 ms, protein,
// 1,700 8.8 / 8.7 / 7.4; 60 DNA triplets of 100..400 local 4.0 / 3.9 / 2.9, semi-global 3.3 / 3.0 / 2.2.
// One triplet whose third sequence is by far the longest is a chain of column tasks along k, which 16 x 64 tasks
// halve: c >= 12 a and c >= 4 b. Semi-global, 4x8 / 4x4, us: 20 x 20 x 3,000 803 / 978, 20 x 600 x 3,000
// 1,047 / 1,156, 60 x 60 x 700 324 / 338; past the line 100 x 100 x 1,000 524 / 518, 300 x 300 x 2,500
// 1,449 / 1,389, 20 x 500 x 500 353 / 311.
Variant typed_tb_tile(const trioseq_plan_s* plan, const trioseq_triplet* trip, size_t n) {
  if (n == 1 && trip[0].len[2] >= 12.0 * std::max(1u, trip[0].len[0]) &&
      trip[0].len[2] >= 4.0 * trip[0].len[1])
    return Variant{4, 8};
  double bytes = 0;
  for (size_t t = 0; t < n; t++)
    bytes += (trip[t].len[0] + 11.0) * ((trip[t].len[1] + 16) / 16) * ((trip[t].len[2] + 32) / 32) *
             (4.0 * (kPC * 4 + 4 + kPR * 4) + 32.0 * 2 * 4);
  return bytes <= (double)plan->slab_budget ? Variant{4, 4} : Variant{4, 8};
}

// Build the host side of a batch: encode, pack, describe, order the queue. lean > 0: a layout for a device
// that had no room for the batch's first one (make_batch): int32 tiles, or pairs on their 8x8 tile; affine
// gaps as build_affine says.
trioseq_status build_batch(trioseq_plan_s* plan, const trioseq_triplet* trip, size_t n,
                           uint32_t mode, trioseq_batch_s* bt, int lean = 0,
                           size_t cap = SIZE_MAX) {
  if (!trip && n) return TRIOSEQ_EINVAL;
  if (mode > TRIOSEQ_WITH_TRACEBACK) return TRIOSEQ_EINVAL;
  const bool tb = mode == TRIOSEQ_WITH_TRACEBACK;
  bt->plan = plan;
  bt->n = n;
  bt->mode = mode;
  bt->var = tb ? plan->tb_variant : plan->score_variant;
  bt->TI = plan->TI;
  std::vector<std::pair<int32_t, int32_t>> units;  // (low-half triplet, high-half triplet or -1)
  {
    uint32_t maxlen = 0;
    for (size_t t = 0; t < n; t++)
      for (int q = 0; q < 3; q++) maxlen = std::max(maxlen, trip[t].len[q]);
    if (plan->tuning && !plan->tune_rule) {
      bt->var = plan->forced.var;
      bt->TI = plan->forced.TI;
    } else if (lean) {
      if (!(tb ? plan->tb_forced : plan->score_forced)) bt->var = tb ? Variant{4, 8} : Variant{8, 8};
    } else {
      auto it = plan->tune_rule ? plan->tuned.end() : plan->tuned.find(tune_key(mode, n, maxlen));
      if (it != plan->tuned.end()) {
        bt->var = it->second.var;
        bt->TI = it->second.TI;
      } else if (auto_tile(plan, tb) &&
                 !(n == 1 && plan->atype == kGlobal && plan->slab_slices > 0)) {
        // global score batches whose pairs fit run two triplets per register
        if (!tb && plan->atype == kGlobal && n >= 2 && maxlen <= (1u << 24)) {
          const Variant v = plan->sig2_nonneg ? packed_variant(plan, trip, n) : bt->var;
          units = pack_units(plan, trip, n, kPR * v.nj, kPC * v.nk);
          if (!units.empty()) bt->var = v;
        }
        if (units.empty()) bt->var = default_variant(plan, trip, n, tb);
      }
    }
  }
  // Two cells of one triplet per register (wavefront_vl.cuh): schemes, types and modes that vl_admits
  // names, tiles that are built for them, and boundary records within the slab budget (it has no slab form).
  // Outside the autotuner's own candidate runs, work it cannot take runs on the int32 tiles instead.
  if (bt->var.vl) {
    // (semi-global and local too: their zero axes and floor add steps of -2*alpha, which must
    // also stay <= 33)
    bool ok_vl = vl_admits(plan, tb) &&
                 wavefront_vl(bt->var.nj, bt->var.nk, bt->var.vl - 1, plan->atype, tb) != nullptr;
    if (ok_vl) {
      const int wj = kPR * bt->var.nj, wk = kPC * bt->var.nk;
      double rec = 0;  // boundary records of all triplets: steps x tasks x row
      for (size_t t = 0; t < n; t++)
        rec += (trip[t].len[0] + 19.0) * ((trip[t].len[1] + wj) / wj) *
               ((trip[t].len[2] + wk) / wk) * (4.0 * (vl_rec_j(bt->var.nk / 2) + kVlRecK));
      // one traceback triplet's codes count too: beyond the budget it runs in (int32) slabs
      if (tb && n == 1)
        rec += (trip[0].len[0] + 19.0) * ((trip[0].len[1] + wj) / wj) *
               ((trip[0].len[2] + wk) / wk) * (wj * wk / 2.0);
      ok_vl = rec <= (double)plan->slab_budget && !(tb && n == 1 && plan->slab_slices > 0);
    }
    if (!ok_vl) {
      if (plan->tuning && !plan->tune_rule) return TRIOSEQ_ECUDA;  // the autotuner skips the candidate
      // the int32 defaults
      bt->var = tb ? (plan->atype != kGlobal ? typed_tb_tile(plan, trip, n) : Variant{4, 8}) : Variant{8, 8};
    }
  }
  const int NJ = bt->var.nj, NK = bt->var.nk;
  const int WJ = kPR * NJ, WK = kPC * NK, W = NJ * NK / 8;
  // encode + pack (16-byte aligned sequences)
  size_t total = 0;
  for (size_t t = 0; t < n; t++)
    for (int q = 0; q < 3; q++) {
      if (trip[t].len[q] && !trip[t].s[q]) return TRIOSEQ_EINVAL;
      if (trip[t].len[q] > (1u << 24)) return TRIOSEQ_EOVERFLOW;
      total += align_up(trip[t].len[q], 16);
    }
  bt->seq.assign(std::max<size_t>(total, 16), 0);
  bt->desc.resize(n);
  bt->tb_of.assign(n, -1);
  bt->tb_trips.clear();
  bt->row_off.clear();
  bt->row_cap.clear();
  size_t pos = 0, face = 0, codes = 0, rows = 0;
  int64_t prog = 0;
  bt->cells = 0;
  // 1a. Packed positions, then the residue codes (alphabet lookup). Large batches encode on
  //     several host threads, each over a contiguous range of triplets.
  for (size_t t = 0; t < n; t++)
    for (int q = 0; q < 3; q++) {
      bt->desc[t].s_off[q] = (int64_t)pos;
      pos += align_up(trip[t].len[q], 16);
    }
  {
    std::atomic<bool> bad{false};
    const auto encode = [&](size_t t0, size_t t1) {
      for (size_t t = t0; t < t1 && !bad.load(std::memory_order_relaxed); t++)
        for (int q = 0; q < 3; q++) {
          const unsigned char* src = reinterpret_cast<const unsigned char*>(trip[t].s[q]);
          int8_t* dst = bt->seq.data() + bt->desc[t].s_off[q];
          int16_t acc = 0;
          for (uint32_t e = 0; e < trip[t].len[q]; e++) {
            const int16_t code = plan->lut[src[e]];
            acc |= code;  // negative iff some residue is outside the alphabet
            dst[e] = (int8_t)code;
          }
          if (acc < 0) bad.store(true, std::memory_order_relaxed);
        }
    };
    // a thread per 128 KiB of residues (~140 us of work); the thread count is asked for only then (it reads
    // the system's files: 10 us, most of a small call's encoding)
    size_t nth = std::min<size_t>({(size_t)8, n, total / (1u << 17) + 1});
    if (nth > 1)
      nth = std::min<size_t>(nth, std::max(1u, std::thread::hardware_concurrency()));
    if (nth <= 1) {
      encode(0, n);
    } else {  // split the triplets into nth ranges of about equal residue counts
      std::vector<std::thread> pool;
      size_t t0 = 0;
      for (size_t k = 1; k <= nth && t0 < n; k++) {
        size_t t1 = t0;
        const size_t goal = total * k / nth;
        while (t1 < n && (k == nth || (size_t)bt->desc[t1].s_off[0] < goal)) t1++;
        if (t1 == t0) continue;
        try {
          pool.emplace_back(encode, t0, t1);
        } catch (...) {  // no thread: encode the range here
          encode(t0, t1);
        }
        t0 = t1;
      }
      for (auto& th : pool) th.join();
    }
    if (bad.load()) return TRIOSEQ_EINVAL;
  }
  // 1b. Per triplet: range checks, output slots.
  for (size_t t = 0; t < n; t++) {
    TripDesc& d = bt->desc[t];
    int64_t sumlen = 0;
    for (int q = 0; q < 3; q++) {
      const uint32_t L = trip[t].len[q];
      d.len[q] = d.glen[q] = (int32_t)L;
      sumlen += L;
    }
    // |M'| <= max|sigma''| * (a+b+c) (and, with zero axes or v = 0, <= 2|alpha| * (a+b+c));
    // keys need 8*|M'| + 8 below 2^29.
    if ((int64_t)std::max(plan->max_abs_sig2, plan->atype != kGlobal ? -2 * plan->gap : 0) *
            sumlen >= (1LL << 26) - 1)
      return TRIOSEQ_EOVERFLOW;
    if (2LL * (int64_t)std::abs(plan->gap) * sumlen >= (1LL << 30)) return TRIOSEQ_EOVERFLOW;
    // semi-global / local traceback: the best cell's index must fit 37 bits (engine.h, best64)
    if (tb && plan->atype != kGlobal &&
        (double)(d.len[0] + 1) * (d.len[1] + 1) * (d.len[2] + 1) >= (double)(1ULL << 37))
      return TRIOSEQ_EOVERFLOW;
    // affine: |score| <= (3 max|sigma| + 3|alpha| + 3|gamma|) * (a+b+c), kept below 2^29
    if (plan->affine &&
        (int64_t)(3 * plan->max_abs_sub + 3 * std::abs(plan->gap) + 3 * std::abs(plan->gap_open)) *
                std::max<int64_t>(sumlen, 1) >= (1LL << 29))
      return TRIOSEQ_EOVERFLOW;
    d.pair = -1;
    d.score_base = 2 * plan->gap * (int32_t)sumlen;
    d.out_idx = (int32_t)t;
    d.tb_idx = -1;
    d.code_off = -1;
    bt->cells += (uint64_t)d.len[0] * (uint64_t)d.len[1] * (uint64_t)d.len[2];
  }
  if (plan->affine) {
    if (tb) return TRIOSEQ_ENOTIMPL;  // the affine model is score-only on the device
    return build_affine(plan, bt, lean, cap);
  }
  // 2. Units of work: one triplet, or in packed int16x2 mode two triplets of the same column-task
  //    grid class paired in one unit (the high halves run on the grid of their maximal lengths).
  bt->packed = 0;
  const bool vl = bt->var.vl != 0;  // admitted above
  if (vl) bt->packed = 2 + bt->var.vl;  // 3: registers; 4, 5: sigma'' tile in shared memory
  const int pmode = plan->sig2_nonneg ? 2 : 1;
  if (!vl && !tb && plan->atype == kGlobal && plan->packed16 && n >= 2 &&
      wavefront_packed(NJ, NK, pmode) != nullptr) {
    if (units.empty()) units = pack_units(plan, trip, n, WJ, WK);
    if (!units.empty()) bt->packed = pmode;
  }
  if (units.empty())  // one unit per triplet (no pairs formed)
    for (size_t t = 0; t < n; t++) units.emplace_back((int32_t)t, -1);
  // 3. Per unit: task grid, boundary records, progress flags, traceback codes and rows.
  for (const auto& un : units) {
    TripDesc& d = bt->desc[un.first];
    if (un.second >= 0) {
      const TripDesc& h = bt->desc[un.second];
      for (int q = 0; q < 3; q++) d.glen[q] = std::max(d.len[q], h.len[q]);
      d.pair = un.second;
    }
    const int a = d.glen[0], b = d.glen[1], c = d.glen[2];
    d.nJ = (b + 1 + WJ - 1) / WJ;
    d.nK = (c + 1 + WK - 1) / WK;
    d.T = a + 1 + (kPR - 1) + (kPC - 1) + (vl ? kPC : 0);  // vl: 2*kPC virtual lane columns
    // boundary records of every column task: (a+1) x (WK+4) j-records, (a+1) x WJ k-records
    const size_t ntask = (size_t)d.nJ * (size_t)d.nK;
    // (two per register, biased: T rows by producer step, of the tasks that have a consumer)
    const bool by_step = vl || bt->packed == 2;
    d.oj_off = (int64_t)face;
    face += by_step ? (ntask - d.nK) * (size_t)d.T * (size_t)(vl ? vl_rec_j(NK / 2) : vp_rec_j(NK))
                    : ntask * (size_t)(a + 1) * (size_t)(WK + 4);
    d.ok_off = (int64_t)face;
    face += by_step ? (ntask - d.nJ) * (size_t)d.T * (size_t)(vl ? kVlRecK : vp_rec_k(NJ))
                    : ntask * (size_t)(a + 1) * (size_t)WJ;
    face = align_up(face, 4);
    d.prog_base = prog;
    prog += (int64_t)d.nJ * d.nK;
    if (un.second >= 0 && un.second != un.first) {  // the high half shares the grid
      TripDesc& h = bt->desc[un.second];
      for (int q = 0; q < 3; q++) h.glen[q] = d.glen[q];
      h.nJ = d.nJ;
      h.nK = d.nK;
      h.T = d.T;
      h.oj_off = d.oj_off;
      h.ok_off = d.ok_off;
      h.prog_base = d.prog_base;
    }
    if (tb) {
      const int32_t t = un.first;
      d.code_off = (int64_t)codes;
      codes += (size_t)d.nJ * d.nK * (size_t)d.T * 32 * W;
      d.tb_idx = (int32_t)bt->tb_trips.size();
      bt->tb_of[t] = d.tb_idx;
      bt->tb_trips.push_back(t);
      const int cap = std::max(1, a + b + c);
      bt->row_off.push_back((int64_t)rows);
      bt->row_cap.push_back(cap);
      rows += align_up((size_t)3 * cap, 16);
    }
  }
  // 4. Slab mode: one global-type int32 triplet whose boundary records (and, with traceback,
  //    codes) would exceed the plan's budget at once, or any such triplet when a slab height is
  //    forced. The cube then runs slab by slab, each launch seeded from the plane the slab below
  //    left (linear-space traceback).
  bt->slab = bt->nslab = 0;
  bt->nplanes = bt->plane_ints = 0;
  bt->slab_desc.clear();
  if (n == 1 && plan->atype == kGlobal && !bt->packed) {
    TripDesc& d = bt->desc[0];
    const size_t ntask = (size_t)d.nJ * (size_t)d.nK;
    const size_t A = (size_t)d.len[0] + 1;                     // slices of the cube
    const size_t rec = ntask * (size_t)((WK + 4) + WJ);         // record ints per slice
    const size_t cw = tb ? ntask * 32 * (size_t)W : 0;          // code words per step
    const size_t plane = (size_t)d.nJ * WJ * (size_t)d.nK * WK;  // ints per plane
    const auto bytes = [&](size_t S) {  // workspace of slab height S
      const size_t slabs = (A + S - 1) / S;
      const size_t planes = tb ? slabs - 1 : std::min<size_t>(2, slabs - 1);
      return 4 * (S * rec + (S + 10) * cw + planes * plane);
    };
    size_t S = (size_t)plan->slab_slices;
    if (S == 0 && 4 * (A * rec + (A + 10) * cw) > plan->slab_budget) {
      // the largest power-of-two fraction of the cube that fits; fall back to the smallest
      // workspace when none does (the allocation then reports ENOMEM)
      size_t best = A;
      for (S = A; S >= 1; S = S / 2) {
        if (bytes(S) < bytes(best)) best = S;
        if (bytes(S) <= plan->slab_budget) break;
        if (S == 1) {
          S = best;
          break;
        }
      }
    }
    if (S > 0) {
      S = std::min(S, A);
      bt->slab = (int)S;
      bt->nslab = (int)((A + S - 1) / S);
      bt->plane_ints = plane;
      bt->nplanes = tb ? bt->nslab - 1 : std::min(2, bt->nslab - 1);
      for (int m = 0; m < bt->nslab; m++) {
        TripDesc sd = d;
        const int len0 = (int)std::min(S, A - (size_t)m * S) - 1;  // last local slice
        sd.len[0] = sd.glen[0] = len0;
        sd.T = len0 + 1 + (kPR - 1) + (kPC - 1);
        sd.oj_off = 0;
        sd.ok_off = (int64_t)(ntask * S * (size_t)(WK + 4));
        sd.prog_base = 0;
        sd.code_off = 0;
        sd.out_idx = (m == bt->nslab - 1) ? 0 : -1;  // only the top slab ends at (a, b, c)
        bt->slab_desc.push_back(sd);
      }
      d.code_off = 0;  // the walk reads the one slab of codes in the buffer
      face = ntask * S * (size_t)((WK + 4) + WJ);
      codes = tb ? ntask * (S + 10) * 32 * (size_t)W : 0;
    }
  }
  bt->seq_bytes = bt->seq.size();
  bt->face_ints = std::max<size_t>(face, 4);
  bt->code_words = std::max<size_t>(codes, 4);
  bt->rows_bytes = std::max<size_t>(rows, 16);
  // queue: (anti-diagonal, LPT rank of the unit's grid, J), built by counting sort on the
  // anti-diagonal: units visited in LPT order and J ascending within a unit give the same order as
  // a stable sort on the full key.
  const size_t nu = units.size();
  std::vector<int32_t> order(nu);
  {
    std::vector<std::pair<double, int32_t>> key(nu);  // largest volume first, then position
    for (size_t u = 0; u < nu; u++) {
      const TripDesc& d = bt->desc[units[u].first];
      key[u] = {-(double)(d.glen[0] + 1) * (d.glen[1] + 1) * (d.glen[2] + 1), (int32_t)u};
    }
    std::sort(key.begin(), key.end());
    for (size_t u = 0; u < nu; u++) order[u] = key[u].second;
  }
  int maxD = 0;
  for (const auto& un : units) {
    const TripDesc& d = bt->desc[un.first];
    maxD = std::max(maxD, d.nJ + d.nK - 2);
  }
  std::vector<size_t> start((size_t)maxD + 2, 0);
  for (const auto& un : units) {
    const TripDesc& d = bt->desc[un.first];
    for (int J = 0; J < d.nJ; J++)
      for (int K = 0; K < d.nK; K++) start[(size_t)(J + K) + 1]++;
  }
  for (size_t D = 1; D < start.size(); D++) start[D] += start[D - 1];
  bt->tasks.assign((size_t)prog, Task{0, 0, 0, 0});
  {
    for (const int32_t u : order) {
      const int32_t t = units[u].first;
      const TripDesc& d = bt->desc[t];
      for (int J = 0; J < d.nJ; J++)
        for (int K = 0; K < d.nK; K++) bt->tasks[start[(size_t)(J + K)]++] = Task{t, J, K, 0};
    }
  }
  layout_inputs(bt);
  // launch shape
  bt->smem = bt->packed >= 3 ? wavefront_vl_smem_bytes(NJ, NK, plan->KP, bt->packed - 3)
             : bt->packed == 2 ? wavefront_vp_smem_bytes(NJ, NK, plan->KP)
                               : wavefront_smem_bytes(NJ, NK, plan->KP, bt->packed != 0);
  int bpm = 0;
  // Int32 traceback launches of one triplet use the records as readiness flags; TRIOSEQ_DATA_FLAGS at
  // plan creation forces it on (1) or off (0). (The two-cells-per-register kernel always does.)
  // Batches of the semi-global and local types too: 60 DNA triplets of 100..400 2.9 -> 2.5 and 2.2 -> 1.9 ms.
  bt->df = tb && !vl && !bt->slab &&
           (plan->data_flags >= 0 ? plan->data_flags != 0 : n == 1 || plan->atype != kGlobal);
  if (wavefront_occupancy(NJ, NK, tb, plan->atype, bt->packed, bt->slab > 0, bt->smem,
                          &bpm) != 0 ||
      bpm <= 0)
    return TRIOSEQ_ECUDA;
  const int want = env_int("TRIOSEQ_CTAS_PER_SM", bpm);
  bt->grid = plan->sms * std::max(1, std::min(bpm, want));
  if (vl || bt->packed == 2)  // no CTA without a task: one that finds the queue empty still costs its start
    bt->grid = (int)std::max<size_t>(1, std::min<size_t>((size_t)bt->grid, bt->tasks.size()));
  return TRIOSEQ_OK;
}


// Bytes of a run's results as fetch() stages them: error word, scores, rows, lengths and spans.
size_t results_bytes(const trioseq_batch_s* bt) {
  const size_t ntb = bt->tb_trips.size();
  return 64 + align_up(bt->n * 4, 64) +
         (ntb ? align_up(bt->rows_bytes, 64) + align_up(ntb * 4, 64) + align_up(ntb * 24, 64) : 0);
}

// How a batch's inputs (and results) pass the host: kPageable copies the inputs synchronously from pageable
// memory (one-off batch creation); kPinned stages them through the workspace's pinned buffer and copies
// asynchronously on the launch stream (a server's slot, which has a pinned buffer of its own for results);
// kPinnedBoth also leaves room there for the results (trioseq_align_batch).
enum class Staging { kPageable, kPinned, kPinnedBoth };
// Results beyond this many bytes go straight to their destinations: the copies themselves then take longer
// than the waits that staging saves, and the plan would keep that much pinned memory.
constexpr size_t kStagedResults = (size_t)16 << 20;

// Size the workspace and copy the inputs of `bt` into it (stream-ordered).
trioseq_status upload(trioseq_batch_s* bt, cudaStream_t st, Staging how) {
  const bool pinned = how != Staging::kPageable;
  Workspace& ws = *bt->ws;
  const bool tb = bt->mode == TRIOSEQ_WITH_TRACEBACK;
  const size_t nprog = bt->tasks.size() + 64;
  cudaStream_t as = ws.alloc_stream;
  ws.order_after_last_use();  // a buffer that grows is freed only after its last use
  if (!ws.inputs.ensure(bt->inputs_bytes, as)) return TRIOSEQ_ENOMEM;
  if (!ws.faces.ensure(bt->face_ints * sizeof(int32_t), as) ||
      !ws.progress.ensure(nprog * sizeof(int32_t), as) ||
      !ws.scores.ensure(std::max<size_t>(bt->n, 1) * sizeof(int32_t), as) ||
      (tb && (!ws.codes.ensure(bt->code_words * sizeof(uint32_t), as) ||
              !ws.rows.ensure(bt->rows_bytes, as) ||
              !ws.lens.ensure(std::max<size_t>(bt->tb_trips.size(), 1) * sizeof(int32_t), as))) ||
      (bt->nplanes && !ws.planes.ensure(bt->nplanes * bt->plane_ints * sizeof(int32_t), as)) ||
      (bt->slab && tb && !ws.walkstate.ensure(4 * sizeof(int32_t), as)) ||
      (tb && !ws.spans.ensure(std::max<size_t>(bt->tb_trips.size(), 1) * 6 * sizeof(int32_t),
                              as)) ||
      (tb && plan_atype(bt) != kGlobal &&
       !ws.best64.ensure(std::max<size_t>(bt->n, 1) * sizeof(unsigned long long), as))) {
    bt->no_room = true;  // records and codes, or what comes after them: a smaller layout may fit
    return TRIOSEQ_ENOMEM;
  }
  if (pinned) {  // without room for the results they are fetched directly
    const size_t res = how == Staging::kPinnedBoth ? results_bytes(bt) : 0;
    if (!(res && res <= kStagedResults && ws.staging.ensure(align_up(bt->inputs_bytes, 256) + res)) &&
        !ws.staging.ensure(bt->inputs_bytes))
      return TRIOSEQ_ENOMEM;
  }
  // On a private allocation stream, the buffers are ready before any launch stream uses them.
  if (ws.own_stream && cudaStreamSynchronize(as) != cudaSuccess)
    return cuda_status(cudaGetLastError());
  std::vector<char> pageable;
  if (!pinned) pageable.assign(bt->inputs_bytes, 0);
  char* h = pinned ? reinterpret_cast<char*>(ws.staging.p) : pageable.data();
  std::memcpy(h, bt->seq.data(), bt->seq_bytes);
  std::memcpy(h + bt->off_desc, bt->desc.data(), sizeof(TripDesc) * bt->n);
  std::memcpy(h + bt->off_tasks, bt->tasks.data(), sizeof(Task) * bt->tasks.size());
  if (!bt->slab_desc.empty())
    std::memcpy(h + bt->off_slab, bt->slab_desc.data(), sizeof(TripDesc) * bt->slab_desc.size());
  if (tb) {
    std::memcpy(h + bt->off_tb, bt->tb_trips.data(), sizeof(int32_t) * bt->tb_trips.size());
    std::memcpy(h + bt->off_rowoff, bt->row_off.data(), sizeof(int64_t) * bt->row_off.size());
    std::memcpy(h + bt->off_rowcap, bt->row_cap.data(), sizeof(int32_t) * bt->row_cap.size());
  }
  cudaError_t e =
      pinned ? cudaMemcpyAsync(ws.inputs.p, h, bt->inputs_bytes, cudaMemcpyHostToDevice, st)
             : cudaMemcpy(ws.inputs.p, h, bt->inputs_bytes, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_status(e);
  // Test switch: fill the boundary records and slab planes with 0x3F3F3F3F, a value far above
  // any score, so that a kernel reading a record slot before (or without) its producer writing
  // it gives a wrong result instead of one that fresh, zeroed memory would hide.
  if (bt->plan->test_poison) {
    if (ws.faces.p && (e = cudaMemsetAsync(ws.faces.p, 0x3F, ws.faces.cap, st)) != cudaSuccess)
      return cuda_status(e);
    if (ws.planes.p && (e = cudaMemsetAsync(ws.planes.p, 0x3F, ws.planes.cap, st)) != cudaSuccess)
      return cuda_status(e);
  }
  bt->uploaded = true;
  bt->h2d_bytes = bt->inputs_bytes;
  return TRIOSEQ_OK;
}

// Device bytes of a batch's records, codes and slab planes: what its layout decides.
size_t layout_bytes(const trioseq_batch_s& bt) {
  return 4 * (bt.face_ints + bt.nplanes * bt.plane_ints +
              (bt.mode == TRIOSEQ_WITH_TRACEBACK ? bt.code_words : 0));
}

// Build a batch and place it in `ws` (or a workspace of its own). Where the device has no room for the records
// and codes of the default layout, the layouts that need less are tried before the call fails. cap: the bytes
// that a server can give the launch; a layout beyond it gives way to a smaller one, if there is one.
trioseq_status make_batch(trioseq_plan_s* plan, const trioseq_triplet* trip, size_t n, uint32_t mode,
                          Workspace* ws, cudaStream_t st, Staging how,
                          std::unique_ptr<trioseq_batch_s>* out, size_t cap = SIZE_MAX) {
  const int last = plan->affine ? 2 : 1;
  size_t least = SIZE_MAX;  // bytes of the smallest layout so far
  std::unique_ptr<trioseq_batch_s> bt;  // that layout, not yet tried
  trioseq_status s = TRIOSEQ_ENOMEM;
  for (int lean = 0; lean <= last; lean++) {
    std::unique_ptr<trioseq_batch_s> next(new (std::nothrow) trioseq_batch_s());
    if (!next) return TRIOSEQ_ENOMEM;
    s = build_batch(plan, trip, n, mode, next.get(), lean, cap);
    if (s != TRIOSEQ_OK) return s;
    const size_t bytes = layout_bytes(*next);
    if (bytes < least) {
      least = bytes;
      bt = std::move(next);
    }
    s = TRIOSEQ_ENOMEM;
    if (!bt || (least > cap && lean < last)) continue;
    if (!ws) {
      bt->own_ws.reset(new (std::nothrow) Workspace());
      if (!bt->own_ws) return TRIOSEQ_ENOMEM;
      if (bt->own_ws->make_own_stream() != cudaSuccess) return cuda_status(cudaGetLastError());
    }
    bt->ws = ws ? ws : bt->own_ws.get();
    s = upload(bt.get(), st, how);
    if (s == TRIOSEQ_OK) {
      *out = std::move(bt);
      return s;
    }
    if (!bt->no_room) return s;
    bt.reset();
    if (ws) {  // what the larger layout did get
      ws->faces.reset();
      ws->codes.reset();
    }
  }
  return s;
}

// Event record that also works inside a stream capture (there it becomes an event-record node
// instead of a capture-internal dependency).
cudaError_t record(cudaEvent_t ev, cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (st && cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusActive)
    return cudaEventRecordWithFlags(ev, st, cudaEventRecordExternal);
  return cudaEventRecord(ev, st);
}

// One pass of the hot path on device-resident inputs.
trioseq_status run(trioseq_batch_s* bt, cudaStream_t st) {
  Workspace& ws = *bt->ws;
  trioseq_plan_s* plan = bt->plan;
  const bool tb = bt->mode == TRIOSEQ_WITH_TRACEBACK;
  const size_t nprog = bt->tasks.size() + 64;
  int32_t* prog = ws.progress.as<int32_t>();
  int32_t* queue = prog + bt->tasks.size();
  int32_t* err = queue + 32;
  cudaError_t e = cudaMemsetAsync(prog, 0, nprog * sizeof(int32_t), st);
  if (e != cudaSuccess) return cuda_status(e);
  if (bt->n == 0) return TRIOSEQ_OK;
  char* in = ws.inputs.as<char>();
  if (plan->affine) {  // affine gaps (affine.cu): score only
    const TripDesc* desc = reinterpret_cast<const TripDesc*>(in + bt->off_desc);
    const Task* tasks = reinterpret_cast<const Task*>(in + bt->off_tasks);
    if (bt->profile && record(bt->ev[0], st) != cudaSuccess) return cuda_status(cudaGetLastError());
    if (bt->affine_cells) {
      AffinePlaneParams ap{};
      ap.desc = desc;
      ap.tasks = tasks;
      ap.n = (int32_t)bt->tasks.size();
      ap.KP = plan->KP;
      ap.seq = reinterpret_cast<const int8_t*>(in);
      ap.sub = plan->sig_affine.as<int32_t>();
      ap.gap = plan->gap;
      ap.gap_open = plan->gap_open;
      ap.planes = ws.faces.as<int32_t>();
      ap.plane_cells = bt->affine_cells;
      ap.queue = queue;
      ap.scores = ws.scores.as<int32_t>();
      if (launch_affine_plane(ap, bt->grid, st) != 0) return cuda_status(cudaGetLastError());
    }
    for (size_t ch = 0; ch < bt->affine_chunks.size(); ch++) {
      const auto& [first, count] = bt->affine_chunks[ch];
      if (ch && (e = cudaMemsetAsync(queue, 0, sizeof(int32_t), st)) != cudaSuccess)
        return cuda_status(e);
      const bool pk = bt->packed != 0;
      const auto both = [&](int32_t v) { return pk ? (v & 0xffff) | (int32_t)((uint32_t)v << 16) : v; };
      AffineParams ap{};
      ap.desc = desc;
      ap.tasks = tasks + first;
      ap.ntasks = (int32_t)count;
      ap.KP = plan->KP;
      ap.seq = reinterpret_cast<const int8_t*>(in);
      ap.sig = plan->sig_score.as<int32_t>();
      ap.faces = ws.faces.as<int32_t>();
      ap.progress = prog;
      ap.queue = queue;
      ap.scores = ws.scores.as<int32_t>();
      ap.err = err;
      ap.TI = std::max(1, bt->TI);
      ap.wait_ns = plan->wait_ns;
      ap.go1 = both(plan->gap_open);
      ap.go2 = both(2 * plan->gap_open);
      ap.neg = pk ? both(-4 * plan->gap_open) : kNeg;
      ap.one = 1;
      if (launch_affine(pk, ap, bt->grid, bt->smem, st) != 0)
        return cuda_status(cudaGetLastError());
    }
    if (bt->profile) {
      if (record(bt->ev[1], st) != cudaSuccess || record(bt->ev[2], st) != cudaSuccess)
        return cuda_status(cudaGetLastError());
      bt->timed = true;
    }
    return TRIOSEQ_OK;
  }
  WaveParams p{};
  p.desc = reinterpret_cast<const TripDesc*>(in + bt->off_desc);
  p.tasks = reinterpret_cast<const Task*>(in + bt->off_tasks);
  p.ntasks = (int32_t)bt->tasks.size();
  p.KP = plan->KP;
  p.seq = reinterpret_cast<const int8_t*>(in);
  p.sig = tb ? plan->sig_tb.as<int32_t>() : plan->sig_score.as<int32_t>();
  p.faces = ws.faces.as<int32_t>();
  p.progress = prog;
  p.queue = queue;
  p.codes = tb ? ws.codes.as<uint32_t>() : nullptr;
  p.scores = ws.scores.as<int32_t>();
  p.err = err;
  p.TI = std::max(1, bt->TI);
  p.wait_ns = plan->wait_ns;
  p.g2 = -2 * plan->gap;
  p.one = 1;
  // One-triplet int32 traceback launches, whose time is the wavefront ramp: records carry their own
  // readiness (sentinel-filled here, in the launch's stream order), so each producer-consumer
  // level lags by its skew alone instead of also by a publication interval and a flag round trip;
  // progress is then published only at the end of a task.
  p.data_flags = bt->df;
  if (p.data_flags) {
    if ((e = cudaMemsetAsync(p.faces, 0x80, bt->face_ints * sizeof(int32_t), st)) != cudaSuccess)
      return cuda_status(e);
    p.TI = 1 << 30;
  }
  if (plan->test_no_records && bt->packed >= 2) {
    // Test of the bounded waits on records that are their own flags: the launch finds queue task 0 already
    // taken, with its records filled with the sentinel and released, and nothing ever writes them. Its
    // consumers give up after wait_ns, theirs on the records of those.
    const TripDesc& d0 = bt->desc[bt->tasks[0].trip];
    if ((e = cudaMemsetAsync(p.faces, 0xff, bt->face_ints * sizeof(int32_t), st)) != cudaSuccess ||
        (e = cudaMemsetAsync(queue, 1, 1, st)) != cudaSuccess ||
        (e = cudaMemsetAsync(prog + d0.prog_base, 1, 1, st)) != cudaSuccess)
      return cuda_status(e);
  }
  const int warps_per_cta = wavefront_block_threads(bt->packed) / 32;  // resident warps per CTA
  if (plan->test_wait_unset && !bt->slab) {
    // Test of the bounded waits: every first-wave task but queue task 0 waits on a word of the
    // progress buffer that nothing writes (zeroed above), gives up after wait_ns, sets the error
    // word and returns; the call then reports TRIOSEQ_ETIMEOUT.
    p.pace_n = bt->grid * warps_per_cta;
    p.pace_T = 1 << 20;
    p.pace_flag = prog + bt->tasks.size() + 48;
  } else if (!bt->slab && plan->pace && !p.data_flags && bt->packed < 2 &&
             bt->tasks.size() >= 2 * (size_t)bt->grid * warps_per_cta) {
    // pace the first wave against the progress of queue task 0, the (0,0) block of its triplet
    const TripDesc& d0 = bt->desc[bt->tasks[0].trip];
    p.pace_n = bt->grid * warps_per_cta;
    p.pace_T = d0.T;
    p.pace_flag = prog + d0.prog_base;
  }
  if (tb && plan->atype != kGlobal) {  // (score, first cell) keys start from 0
    p.best64 = ws.best64.as<unsigned long long>();
    if ((e = cudaMemsetAsync(p.best64, 0, bt->n * sizeof(unsigned long long), st)) != cudaSuccess)
      return cuda_status(e);
  }
  // Semi-global and local scores are maxima accumulated with atomicMax: start from 0x80808080.
  if (plan->atype != kGlobal &&
      (e = cudaMemsetAsync(p.scores, 0x80, bt->n * sizeof(int32_t), st)) != cudaSuccess)
    return cuda_status(e);
  WalkParams w{};
  w.desc = p.desc;
  w.tb_trips = reinterpret_cast<const int32_t*>(in + bt->off_tb);
  w.ntb = (int32_t)bt->tb_trips.size();
  w.seq = p.seq;
  w.codes = p.codes;
  w.rows = ws.rows.as<uint8_t>();
  w.row_off = reinterpret_cast<const int64_t*>(in + bt->off_rowoff);
  w.row_cap = reinterpret_cast<const int32_t*>(in + bt->off_rowcap);
  w.aln_len = ws.lens.as<int32_t>();
  w.err = err;
  w.NJ = bt->var.nj;
  w.NK = bt->var.vl ? bt->var.nk / 2 : bt->var.nk;  // virtual lanes hold half the columns
  w.vl = bt->var.vl ? 1 : 0;
  w.atype = plan->atype;
  w.best64 = p.best64;
  w.scores = p.scores;
  w.span = tb ? ws.spans.as<int32_t>() : nullptr;
  bt->timed = false;
  if (bt->profile && record(bt->ev[0], st) != cudaSuccess)
    return cuda_status(cudaGetLastError());
  if (bt->slab) {
    // Slab mode. Slab m covers the slices m*S .. of the cube; plane m holds its last slice.
    // Score: forward through all slabs, planes ping-pong. Traceback: forward through all but the
    // top slab keeping every plane (no codes), then from the top slab down: recompute the slab
    // with codes from the plane below it and continue the walk through it.
    const TripDesc* sdesc = reinterpret_cast<const TripDesc*>(in + bt->off_slab);
    int32_t* planes = ws.planes.as<int32_t>();
    const auto plane = [&](int idx) { return planes + (size_t)idx * bt->plane_ints; };
    const auto wave = [&](int m, const int32_t* pin, int32_t* pout, bool codes) {
      const cudaError_t ee = cudaMemsetAsync(prog, 0, nprog * sizeof(int32_t), st);
      if (ee != cudaSuccess) return cuda_status(ee);
      WaveParams q = p;
      q.desc = sdesc + m;
      q.i0 = m * bt->slab;
      q.plane_in = pin;
      q.plane_out = pout;
      q.codes = codes ? p.codes : nullptr;
      if (launch_wavefront(bt->var.nj, bt->var.nk, tb, kGlobal, false, true, q, bt->grid,
                           bt->smem, st) != 0)
        return cuda_status(cudaGetLastError());
      return TRIOSEQ_OK;
    };
    const int M = bt->nslab;
    trioseq_status s = TRIOSEQ_OK;
    if (!tb) {
      for (int m = 0; m < M && s == TRIOSEQ_OK; m++)
        s = wave(m, m ? plane((m - 1) & 1) : nullptr, m + 1 < M ? plane(m & 1) : nullptr, false);
    } else {
      for (int m = 0; m + 1 < M && s == TRIOSEQ_OK; m++)
        s = wave(m, m ? plane(m - 1) : nullptr, plane(m), false);
      for (int m = M - 1; m >= 0 && s == TRIOSEQ_OK; m--) {
        s = wave(m, m ? plane(m - 1) : nullptr, nullptr, true);
        if (s != TRIOSEQ_OK) break;
        WalkParams wm = w;
        wm.i_lo = m * bt->slab;
        wm.T_slab = bt->slab_desc[m].T;  // steps per task of the slab that wrote the codes
        wm.state = ws.walkstate.as<int32_t>();
        wm.init_state = (m == M - 1) ? 1 : 0;
        if (launch_walk(wm, st) != 0) s = cuda_status(cudaGetLastError());
      }
    }
    if (s != TRIOSEQ_OK) return s;
    if (bt->profile && record(bt->ev[1], st) != cudaSuccess)
      return cuda_status(cudaGetLastError());
  } else {
    if (launch_wavefront(bt->var.nj, bt->var.nk, tb, plan->atype, bt->packed, false, p,
                         bt->grid, bt->smem, st) != 0)
      return cuda_status(cudaGetLastError());
    if (bt->profile && record(bt->ev[1], st) != cudaSuccess)
      return cuda_status(cudaGetLastError());
    if (tb && !bt->tb_trips.empty() && launch_walk(w, st) != 0)
      return cuda_status(cudaGetLastError());
  }
  if (bt->profile) {
    if (record(bt->ev[2], st) != cudaSuccess) return cuda_status(cudaGetLastError());
    bt->timed = true;
  }
  return TRIOSEQ_OK;
}

// trioseq_batch_run: replay the batch's graph, capturing it first (on a private stream, so the
// caller's stream may be the legacy default stream) when there is none yet or the workspace
// buffers or the profiling switch changed since it was captured.
trioseq_status run_graph(trioseq_batch_s* bt, cudaStream_t st) {
  const Workspace& ws = *bt->ws;
  // every device address a captured launch bakes in (the slab and walk launches included)
  const std::array<const void*, 12> key{ws.inputs.p,    ws.faces.p,     ws.progress.p,
                                        ws.codes.p,     ws.scores.p,    ws.rows.p,
                                        ws.lens.p,      ws.planes.p,    ws.walkstate.p,
                                        ws.best64.p,    ws.spans.p,
                                        bt->profile ? (const void*)bt->ev[0] : nullptr};
  if (!bt->gexec || key != bt->gkey) {
    if (bt->gexec) {
      cudaGraphExecDestroy(bt->gexec);
      bt->gexec = nullptr;
    }
    cudaError_t e = cudaSuccess;
    if (!bt->capture_stream)
      e = cudaStreamCreateWithFlags(&bt->capture_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess)
      e = cudaStreamBeginCapture(bt->capture_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_status(e);
    const trioseq_status s = run(bt, bt->capture_stream);
    cudaGraph_t graph = nullptr;
    e = cudaStreamEndCapture(bt->capture_stream, &graph);
    if (s == TRIOSEQ_OK && e == cudaSuccess) e = cudaGraphInstantiate(&bt->gexec, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    if (s != TRIOSEQ_OK) return s;
    if (e != cudaSuccess) {
      bt->gexec = nullptr;
      return cuda_status(e);
    }
    bt->gkey = key;
  }
  bt->timed = false;
  const cudaError_t e = cudaGraphLaunch(bt->gexec, st);
  if (e != cudaSuccess) return cuda_status(e);
  bt->timed = bt->profile;
  return TRIOSEQ_OK;
}

// Wait for the run, check the error word, fetch scores (and traceback rows). `staged` (after an upload through
// the pinned buffer): the copies go to that buffer, behind the inputs and enqueued behind the run, and are
// handed on after one wait (a copy to pageable memory holds the caller for its own round trip: 48 us for the
// five of a call with rows, 22 us for the two of a score call, against 16 and 12). Without, straight to their
// destinations, which several threads may do at once.
trioseq_status fetch(trioseq_batch_s* bt, cudaStream_t st, int32_t* scores_out,
                     bool staged = false) {
  Workspace& ws = *bt->ws;
  const bool tb = bt->mode == TRIOSEQ_WITH_TRACEBACK;
  int32_t herr = 0;
  cudaError_t e = cudaSuccess;
  struct Part {
    void* dst;
    const void* src;
    size_t bytes, off;
  };
  Part parts[5];
  int np = 0;
  size_t total = 0;
  const auto add = [&](void* dst, const void* src, size_t bytes) {
    parts[np++] = Part{dst, src, bytes, total};
    total += align_up(bytes, 64);
  };
  if (bt->n) {
    add(&herr, ws.progress.as<int32_t>() + bt->tasks.size() + 32, sizeof(int32_t));
    if (scores_out) add(scores_out, ws.scores.p, bt->n * sizeof(int32_t));
    if (tb && !bt->tb_trips.empty()) {
      bt->h_rows.resize(bt->rows_bytes);
      bt->h_lens.resize(bt->tb_trips.size());
      bt->h_spans.resize(6 * bt->tb_trips.size());
      add(bt->h_rows.data(), ws.rows.p, bt->rows_bytes);
      add(bt->h_lens.data(), ws.lens.p, bt->h_lens.size() * sizeof(int32_t));
      add(bt->h_spans.data(), ws.spans.p, bt->h_spans.size() * sizeof(int32_t));
    }
  }
  const size_t at = align_up(bt->inputs_bytes, 256);
  char* h = staged && at + total <= ws.staging.cap ? reinterpret_cast<char*>(ws.staging.p) + at
                                                   : nullptr;
  for (int q = 0; q < np && e == cudaSuccess; q++)
    e = cudaMemcpyAsync(h ? h + parts[q].off : parts[q].dst, parts[q].src, parts[q].bytes,
                        cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e);
  for (int q = 0; q < np && h; q++) std::memcpy(parts[q].dst, h + parts[q].off, parts[q].bytes);
  if (herr & 1) return TRIOSEQ_ETIMEOUT;
  if (herr & 2) return TRIOSEQ_ECUDA;
  bt->have_rows = tb;
  bt->d2h_bytes = bt->n ? sizeof(int32_t) * (1 + bt->n) : 0;
  if (tb && !bt->tb_trips.empty())
    bt->d2h_bytes += bt->rows_bytes + bt->h_lens.size() * sizeof(int32_t) +
                     bt->h_spans.size() * sizeof(int32_t);
  return TRIOSEQ_OK;
}

trioseq_status copy_span(const trioseq_batch_s* bt, size_t idx, int32_t* begin, int32_t* end) {
  if (!bt || !bt->have_rows || idx >= bt->n || !begin || !end) return TRIOSEQ_EINVAL;
  const int32_t q = bt->tb_of[idx];
  if (q < 0 || bt->h_lens[q] < 0) return TRIOSEQ_EINVAL;
  for (int t = 0; t < 3; t++) {
    begin[t] = bt->h_spans[6 * q + t];
    end[t] = bt->h_spans[6 * q + 3 + t];
  }
  return TRIOSEQ_OK;
}

trioseq_status copy_alignment(const trioseq_batch_s* bt, size_t idx, char* r0, char* r1, char* r2,
                              size_t cap, size_t* aln_len) {
  if (!bt || !bt->have_rows || idx >= bt->n || !aln_len) return TRIOSEQ_EINVAL;
  const int32_t q = bt->tb_of[idx];
  if (q < 0) return TRIOSEQ_EINVAL;
  const int32_t L = bt->h_lens[q];
  if (L < 0) return TRIOSEQ_ECUDA;
  *aln_len = (size_t)L;
  if (L == 0) return TRIOSEQ_OK;
  if (cap < (size_t)L || !r0 || !r1 || !r2) return TRIOSEQ_EINVAL;
  const int32_t rc = bt->row_cap[q];
  const uint8_t* base = bt->h_rows.data() + bt->row_off[q];
  const char* alpha = bt->plan->alphabet;
  char* out[3] = {r0, r1, r2};
  for (int s = 0; s < 3; s++) {
    const uint8_t* row = base + (size_t)s * rc + (rc - L);
    for (int32_t t = 0; t < L; t++) out[s][t] = row[t] == 255 ? '-' : alpha[row[t]];
  }
  return TRIOSEQ_OK;
}

}  // namespace

extern "C" {

const char* trioseq_strerror(trioseq_status st) {
  switch (st) {
    case TRIOSEQ_OK: return "ok";
    case TRIOSEQ_EINVAL: return "invalid argument";
    case TRIOSEQ_ENOMEM: return "out of memory";
    case TRIOSEQ_EAGAIN: return "not ready / queue full";
    case TRIOSEQ_EOVERFLOW: return "score bound exceeds the integer range";
    case TRIOSEQ_ETIMEOUT: return "bounded device wait expired";
    case TRIOSEQ_ECUDA: return "CUDA error or no usable GPU";
    case TRIOSEQ_ENOTIMPL: return "not implemented";
    case TRIOSEQ_ESCRATCH: return "request exceeds the fixed scratch of the allocation-free call";
  }
  return "unknown status";
}

trioseq_status trioseq_plan(const trioseq_scoring* sc, uint32_t max_len_hint, uint32_t flags,
                            trioseq_plan_t* out) {
  return no_throw([&]() -> trioseq_status {
    (void)max_len_hint;
    NvtxRange range("trioseq_plan");
    if (!out) return TRIOSEQ_EINVAL;
    *out = nullptr;
    if (!sc || !sc->alphabet || !sc->sub || flags > TRIOSEQ_LOCAL) return TRIOSEQ_EINVAL;
    const int K = sc->alphabet_size;
    if (K < 1 || K > kMaxAlphabet || sc->gap > 0 || sc->gap < -127) return TRIOSEQ_EINVAL;
    std::unique_ptr<trioseq_plan_s> plan(new (std::nothrow) trioseq_plan_s());
    if (!plan) return TRIOSEQ_ENOMEM;
    for (int i = 0; i < 256; i++) plan->lut[i] = -1;
    for (int i = 0; i < K; i++) {
      const unsigned char ch = (unsigned char)sc->alphabet[i];
      if (plan->lut[ch] >= 0) return TRIOSEQ_EINVAL;  // duplicate residue
      plan->lut[ch] = (int16_t)i;
      plan->alphabet[i] = (char)ch;
    }
    for (int i = 0; i < K; i++)
      for (int j = 0; j < K; j++)
        if (sc->sub[i * K + j] != sc->sub[j * K + i]) return TRIOSEQ_EINVAL;
    plan->K = K;
    plan->KP = K + 1;
    plan->gap = sc->gap;
    plan->atype = (int)flags;
    plan->sub.assign(sc->sub, sc->sub + K * K);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
      cudaGetLastError();
      return TRIOSEQ_ECUDA;
    }
    plan->device = dev;
    if (cudaDeviceGetAttribute(&plan->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      return TRIOSEQ_ECUDA;
    }
    const int KP = K + 1;
    std::vector<int32_t> s2((size_t)KP * KP, 0), s8((size_t)KP * KP, 0);
    int32_t mx = 0, mn = 0;
    for (int i = 0; i < K; i++)
      for (int j = 0; j < K; j++) {
        const int32_t v = (int32_t)sc->sub[i * K + j] - 2 * sc->gap;  // sigma'' = sigma - 2 alpha
        s2[(size_t)i * KP + j] = v;
        s8[(size_t)i * KP + j] = 8 * v;
        mx = std::max(mx, std::abs(v));
        mn = std::min(mn, v);
      }
    plan->max_abs_sig2 = std::max(mx, 1);
    plan->sig2_nonneg = mn >= 0;
    // The plan's device memory is allocated and freed in the order of its own stream.
    if (plan->ws.make_own_stream() != cudaSuccess) return cuda_status(cudaGetLastError());
    cudaStream_t as = plan->ws.alloc_stream;
    if (!plan->sig_score.ensure(s2.size() * 4, as) || !plan->sig_tb.ensure(s8.size() * 4, as))
      return TRIOSEQ_ENOMEM;
    if (cudaMemcpyAsync(plan->sig_score.p, s2.data(), s2.size() * 4, cudaMemcpyHostToDevice,
                        as) != cudaSuccess ||
        cudaMemcpyAsync(plan->sig_tb.p, s8.data(), s8.size() * 4, cudaMemcpyHostToDevice, as) !=
            cudaSuccess ||
        cudaStreamSynchronize(as) != cudaSuccess)
      return cuda_status(cudaGetLastError());
    plan->TI = std::max(1, env_int("TRIOSEQ_TI", 8));
    plan->graphs = env_int("TRIOSEQ_GRAPHS", 1) != 0;
    plan->packed16 = env_int("TRIOSEQ_PACKED", 1) != 0;
    plan->pace = env_int("TRIOSEQ_PACE", 1) != 0;
    plan->wait_ns = (int64_t)std::max(1, env_int("TRIOSEQ_WAIT_MS", 2000)) * 1000000LL;
    plan->test_wait_unset = env_int("TRIOSEQ_TEST_WAIT_UNSET", 0) != 0;
    plan->test_no_records = env_int("TRIOSEQ_TEST_NO_RECORDS", 0) != 0;
    plan->test_poison = env_int("TRIOSEQ_TEST_POISON", 0) != 0;
    plan->data_flags = env_int("TRIOSEQ_DATA_FLAGS", -1);
    g_device_fault.arm("TRIOSEQ_TEST_FAIL_ALLOC");
    g_pinned_fault.arm("TRIOSEQ_TEST_FAIL_PINNED");
    {
      size_t fr = 0, tot = 0;
      if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
        cudaGetLastError();
        fr = 0;
      }
      const int mb = env_int("TRIOSEQ_SLAB_BUDGET_MB", 0);
      plan->slab_budget = mb > 0 ? (size_t)mb << 20 : fr / 2;
      plan->slab_slices = std::max(0, env_int("TRIOSEQ_SLAB_SLICES", 0));
    }
    // "RxC": register tile rows x columns per lane
    const auto parse_tile = [](const char* v, Variant* out, bool* forced) {
      if (!v) return;
      char* end = nullptr;
      const long rj = std::strtol(v, &end, 10);
      if (!end || *end != 'x') return;
      char* end2 = nullptr;
      const long ck = std::strtol(end + 1, &end2, 10);
      // "8x16" and a trailing 'v' ("8x8v") select the two-cells-per-register kernel; a trailing
      // 's' or 't' ("8x16s", "8x16t") its variants with the sigma''(y,z) tile in shared memory
      const char sfx = end2 ? *end2 : 0;
      const int two = sfx == 's' ? 2 : (sfx == 't' ? 3 : ((ck == 16 || sfx == 'v') ? 1 : 0));
      if (rj > 0 && rj <= 16 && ck > 0 && ck <= 32) {
        *out = Variant{(int)rj, (int)ck, two};
        *forced = true;
      }
    };
    parse_tile(std::getenv("TRIOSEQ_SCORE_TILE"), &plan->score_variant, &plan->score_forced);
    parse_tile(std::getenv("TRIOSEQ_TB_TILE"), &plan->tb_variant, &plan->tb_forced);
    *out = plan.release();
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_plan_affine(const trioseq_scoring* sc, int32_t gap_open, uint32_t flags,
                                   trioseq_plan_t* out) {
  return no_throw([&]() -> trioseq_status {
    NvtxRange range("trioseq_plan_affine");
    if (!out) return TRIOSEQ_EINVAL;
    *out = nullptr;
    if (flags != TRIOSEQ_GLOBAL || gap_open > 0 || gap_open < -(1 << 20)) return TRIOSEQ_EINVAL;
    trioseq_plan_t plan = nullptr;
    trioseq_status s = trioseq_plan(sc, 0, flags, &plan);
    if (s != TRIOSEQ_OK) return s;
    std::unique_ptr<trioseq_plan_s, trioseq_status (*)(trioseq_plan_t)> keep(
        plan, &trioseq_plan_destroy);
    DeviceGuard g(plan->device);
    plan->affine = true;
    plan->gap_open = gap_open;
    const int K = plan->K, KP = plan->KP;
    std::vector<int32_t> tab((size_t)KP * KP, 0);
    int32_t mx = 0;
    for (int i = 0; i < K; i++)
      for (int j = 0; j < K; j++) {
        tab[(size_t)i * KP + j] = sc->sub[i * K + j];
        mx = std::max(mx, std::abs((int32_t)sc->sub[i * K + j]));
      }
    plan->max_abs_sub = mx;
    cudaStream_t as = plan->ws.alloc_stream;
    if (!plan->sig_affine.ensure(tab.size() * 4, as)) return TRIOSEQ_ENOMEM;
    if (cudaMemcpyAsync(plan->sig_affine.p, tab.data(), tab.size() * 4, cudaMemcpyHostToDevice,
                        as) != cudaSuccess ||
        cudaStreamSynchronize(as) != cudaSuccess)
      return cuda_status(cudaGetLastError());
    *out = keep.release();
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_plan_destroy(trioseq_plan_t plan) {
  return no_throw([&]() -> trioseq_status {
    if (!plan) return TRIOSEQ_OK;
    DeviceGuard g(plan->device);
    // Wait for the plan's own last use only (its trioseq_align_batch work); batches made from
    // the plan are destroyed before it and have waited for theirs. Other streams, a running
    // server's included, are not synchronised. The substitution tables are freed in the order
    // of the plan's stream, before the workspace releases that stream.
    plan->ws.wait_last_use();
    plan->last.reset();
    plan->ws.order_after_last_use();
    plan->sig_score.reset();
    plan->sig_tb.reset();
    plan->sig_affine.reset();
    delete plan;
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_align_batch(trioseq_plan_t plan, const trioseq_triplet* triplets, size_t n,
                                   uint32_t mode, int32_t* scores_out, void* stream) {
  return no_throw([&]() -> trioseq_status {
    NvtxRange range("trioseq_align_batch");
    if (!plan || (n && !scores_out)) return TRIOSEQ_EINVAL;
    DeviceGuard g(plan->device);
    cudaStream_t st = (cudaStream_t)stream;
    std::unique_ptr<trioseq_batch_s> bt;
    plan->last.reset();
    trioseq_status s = make_batch(plan, triplets, n, mode, &plan->ws, st, Staging::kPinnedBoth, &bt);
    if (s != TRIOSEQ_OK) return s;
    s = run(bt.get(), st);
    plan->ws.mark_use(st);  // also after a partial enqueue: destroy waits for what did run
    if (s != TRIOSEQ_OK) return s;
    if ((s = fetch(bt.get(), st, scores_out, true)) != TRIOSEQ_OK) return s;
    // A plan keeps at most 16 GB of affine records from one call to the next: those of a triplet of 1,850
    // residues. Beyond, they go back to the device and are taken again by the next call, which costs about as
    // long as its kernel (2,000 residues, 20 GB: 35 -> 79 ms).
    if (plan->affine && plan->ws.faces.cap > kAffineKeep) {
      plan->ws.order_after_last_use();
      plan->ws.faces.reset();
      cudaStreamSynchronize(plan->ws.alloc_stream);  // the pool returns it at the next synchronisation
    }
    bt->seq.clear();
    bt->seq.shrink_to_fit();
    plan->last = std::move(bt);
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_traceback(trioseq_plan_t plan, size_t idx, char* row0, char* row1,
                                 char* row2, size_t cap, size_t* aln_len) {
  return no_throw([&]() -> trioseq_status {
    NvtxRange range("trioseq_traceback");
    if (!plan || !plan->last) return TRIOSEQ_EINVAL;
    return copy_alignment(plan->last.get(), idx, row0, row1, row2, cap, aln_len);
  });
}

trioseq_status trioseq_traceback_span(trioseq_plan_t plan, size_t idx, int32_t begin[3],
                                      int32_t end[3]) {
  return no_throw([&]() -> trioseq_status {
    if (!plan || !plan->last) return TRIOSEQ_EINVAL;
    return copy_span(plan->last.get(), idx, begin, end);
  });
}

trioseq_status trioseq_batch_create(trioseq_plan_t plan, const trioseq_triplet* triplets,
                                    size_t n, uint32_t mode, trioseq_batch_t* out) {
  return no_throw([&]() -> trioseq_status {
    NvtxRange range("trioseq_batch_create");
    if (!plan || !out) return TRIOSEQ_EINVAL;
    *out = nullptr;
    DeviceGuard g(plan->device);
    std::unique_ptr<trioseq_batch_s> bt;
    const trioseq_status s = make_batch(plan, triplets, n, mode, nullptr, nullptr, Staging::kPageable,
                                        &bt);
    if (s != TRIOSEQ_OK) return s;
    *out = bt.release();
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_batch_run(trioseq_batch_t bt, void* stream) {
  return no_throw([&]() -> trioseq_status {
    NvtxRange range("trioseq_batch_run");
    if (!bt) return TRIOSEQ_EINVAL;
    DeviceGuard g(bt->plan->device);
    const cudaStream_t st = (cudaStream_t)stream;
    const trioseq_status s = bt->plan->graphs ? run_graph(bt, st) : run(bt, st);
    const cudaError_t e = bt->ws->mark_use(st);
    return s != TRIOSEQ_OK ? s : cuda_status(e);
  });
}

trioseq_status trioseq_batch_scores(trioseq_batch_t bt, void* stream, int32_t* scores_out) {
  return no_throw([&]() -> trioseq_status {
    if (!bt || (bt->n && !scores_out)) return TRIOSEQ_EINVAL;
    DeviceGuard g(bt->plan->device);
    return fetch(bt, (cudaStream_t)stream, scores_out);
  });
}

trioseq_status trioseq_batch_device_scores(trioseq_batch_t bt, int32_t** d_scores) {
  return no_throw([&]() -> trioseq_status {
    if (!bt || !d_scores) return TRIOSEQ_EINVAL;
    *d_scores = bt->ws->scores.as<int32_t>();
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_batch_alignment(trioseq_batch_t bt, size_t idx, char* row0, char* row1,
                                       char* row2, size_t cap, size_t* aln_len) {
  return no_throw([&]() -> trioseq_status {
    return copy_alignment(bt, idx, row0, row1, row2, cap, aln_len);
  });
}

trioseq_status trioseq_batch_span(trioseq_batch_t bt, size_t idx, int32_t begin[3],
                                  int32_t end[3]) {
  return no_throw([&]() -> trioseq_status {
    return copy_span(bt, idx, begin, end);
  });
}

trioseq_status trioseq_batch_info(trioseq_batch_t bt, size_t* n, uint64_t* cells, uint64_t* tasks,
                                  int32_t* tile_j, int32_t* tile_k) {
  return no_throw([&]() -> trioseq_status {
    if (!bt) return TRIOSEQ_EINVAL;
    if (n) *n = bt->n;
    if (cells) *cells = bt->cells;
    if (tasks) *tasks = bt->tasks.size();
    if (tile_j) *tile_j = bt->var.nj;
    if (tile_k) *tile_k = bt->var.nk;
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_batch_slabs(trioseq_batch_t bt, int32_t* slices, int32_t* slabs) {
  return no_throw([&]() -> trioseq_status {
    if (!bt || !slices || !slabs) return TRIOSEQ_EINVAL;
    *slices = bt->slab;
    *slabs = bt->nslab;
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_batch_packing(trioseq_batch_t bt, int32_t* per_word) {
  return no_throw([&]() -> trioseq_status {
    if (!bt || !per_word) return TRIOSEQ_EINVAL;
    *per_word = bt->packed ? 2 : 1;
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_batch_kernel(trioseq_batch_t bt, char* name, size_t cap) {
  return no_throw([&]() -> trioseq_status {
    if (!bt || !name || cap == 0) return TRIOSEQ_EINVAL;
    const bool tb = bt->mode == TRIOSEQ_WITH_TRACEBACK;
    const int at = bt->plan->atype;
    const char* type = at == kLocal ? "local" : (at == kSemiGlobal ? "semiglobal" : "global");
    const int nj = bt->var.nj, nk = bt->var.nk;
    char buf[160];
    if (bt->plan->affine)
      std::snprintf(buf, sizeof buf, bt->affine_cells ? "affine_plane_kernel tile plane"
                                                        : "affine_kernel tile 4x4");
    else if (bt->packed >= 3)
      std::snprintf(buf, sizeof buf, "wavefront_vl_kernel<%d,%d,%d%s> tile %dx%d%s", nj, nk / 2,
                    bt->packed - 3, tb ? ",traceback" : "", nj, nk,
                    bt->packed == 4 ? "s" : (bt->packed == 5 ? "t" : (nk == 16 ? "" : "v")));
    else if (bt->packed == 2)
      std::snprintf(buf, sizeof buf, "wavefront_vp_kernel<%d,%d> tile %dx%d", nj, nk, nj, nk);
    else if (bt->packed)
      std::snprintf(buf, sizeof buf,
                    "wavefront_kernel<%d,%d,score,global,two triplets per register, signed> tile %dx%d",
                    nj, nk, nj, nk);
    else
      std::snprintf(buf, sizeof buf, "wavefront_kernel<%d,%d,%s,%s%s> tile %dx%d", nj, nk,
                    tb ? "traceback" : "score", type, bt->slab ? ",slab" : "", nj, nk);
    std::snprintf(name, cap, "%s", buf);
    return std::strlen(buf) < cap ? TRIOSEQ_OK : TRIOSEQ_EINVAL;
  });
}

trioseq_status trioseq_batch_profile(trioseq_batch_t bt, int32_t enable) {
  return no_throw([&]() -> trioseq_status {
    if (!bt) return TRIOSEQ_EINVAL;
    DeviceGuard g(bt->plan->device);
    if (enable)
      for (auto& e : bt->ev)
        if (!e && cudaEventCreate(&e) != cudaSuccess) return cuda_status(cudaGetLastError());
    bt->profile = enable != 0;
    bt->timed = false;
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_batch_timing(trioseq_batch_t bt, float ms[2]) {
  return no_throw([&]() -> trioseq_status {
    if (!bt || !ms || !bt->profile || !bt->timed) return TRIOSEQ_EINVAL;
    DeviceGuard g(bt->plan->device);
    float a = 0.f, b = 0.f;
    if (cudaEventElapsedTime(&a, bt->ev[0], bt->ev[1]) != cudaSuccess ||
        cudaEventElapsedTime(&b, bt->ev[1], bt->ev[2]) != cudaSuccess)
      return cuda_status(cudaGetLastError());
    ms[0] = a;
    ms[1] = b;
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_plan_autotune(trioseq_plan_t plan, const trioseq_triplet* sample, size_t n,
                                     uint32_t mode, int32_t* tile_j, int32_t* tile_k,
                                     int32_t* ti) {
  return no_throw([&]() -> trioseq_status {
    NvtxRange range("trioseq_plan_autotune");
    if (!plan || !sample || n == 0 || mode > TRIOSEQ_WITH_TRACEBACK) return TRIOSEQ_EINVAL;
    DeviceGuard g(plan->device);
    if (plan->affine) {  // one kernel shape: nothing to choose
      if (tile_j) *tile_j = 0;
      if (tile_k) *tile_k = 0;
      if (ti) *ti = 0;
      return mode == TRIOSEQ_WITH_TRACEBACK ? TRIOSEQ_ENOTIMPL : TRIOSEQ_OK;
    }
    // What the rules choose by themselves is measured first, so that a tuned plan is not slower than an untuned
    // one; then the candidate tiles per mode (int32 or pairs, and with vl two cells per register).
    static const Variant kScoreTiles[] = {{8, 8},    {4, 8},     {4, 4},     {8, 16, 1},
                                          {8, 8, 1}, {8, 16, 2}, {8, 16, 3}, {4, 8, 1}};
    static const Variant kTbTiles[] = {{8, 8}, {4, 8}, {4, 4}, {8, 4}, {8, 8, 1}, {4, 8, 1}};
    static const int kTI[] = {4, 8, 16, 32};
    const bool tb_mode = mode == TRIOSEQ_WITH_TRACEBACK;
    const Variant* tiles = tb_mode ? kTbTiles : kScoreTiles;
    const size_t ntiles = tb_mode ? sizeof(kTbTiles) / sizeof(kTbTiles[0])
                                  : sizeof(kScoreTiles) / sizeof(kScoreTiles[0]);
    uint32_t maxlen = 0;
    for (size_t t = 0; t < n; t++)
      for (int q = 0; q < 3; q++) maxlen = std::max(maxlen, sample[t].len[q]);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
      return cuda_status(cudaGetLastError());
    trioseq_status result = TRIOSEQ_OK;
    trioseq_plan_s::Tuned rule{tb_mode ? plan->tb_variant : plan->score_variant, plan->TI}, bestv{};
    float rule_ms = 3.0e38f, best = 3.0e38f;
    bool fits = false;  // something could be measured
    {
      struct Tuning {  // also on the way out of an exception
        trioseq_plan_s* plan;
        explicit Tuning(trioseq_plan_s* p) : plan(p) { plan->tuning = true; }
        ~Tuning() { plan->tuning = plan->tune_rule = false; }
      } tuning(plan);
      Workspace ws;       // one workspace, grown to the largest candidate
      bool moot = false;  // the last launch publishes no progress: its interval changes nothing
      // Time of two passes of a candidate, or (null) of the rules' choice, which `rule` then names; skipped
      // where there is no such kernel for the work, or no room for its records.
      const auto measure = [&](const trioseq_plan_s::Tuned* v, float* least) -> trioseq_status {
        plan->tune_rule = v == nullptr;
        if (v) plan->forced = *v;
        moot = true;
        trioseq_batch_s bt;
        trioseq_status s = build_batch(plan, sample, n, mode, &bt);
        if (s != TRIOSEQ_OK) return s == TRIOSEQ_ECUDA ? TRIOSEQ_OK : s;
        bt.ws = &ws;
        s = upload(&bt, nullptr, Staging::kPageable);
        if (s != TRIOSEQ_OK) return bt.no_room ? TRIOSEQ_OK : s;
        moot = bt.packed >= 2 || bt.df;
        if (!v) rule = trioseq_plan_s::Tuned{bt.var, bt.TI};
        if ((s = run(&bt, nullptr)) != TRIOSEQ_OK || (s = fetch(&bt, nullptr, nullptr)) != TRIOSEQ_OK)
          return s;
        float ms = 0.f;
        cudaEventRecord(e0, nullptr);
        for (int rep = 0; rep < 2 && s == TRIOSEQ_OK; rep++) s = run(&bt, nullptr);
        cudaEventRecord(e1, nullptr);
        if (s == TRIOSEQ_OK) s = fetch(&bt, nullptr, nullptr);
        if (s != TRIOSEQ_OK) return s;
        if (cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) return cuda_status(cudaGetLastError());
        *least = std::min(*least, ms);
        fits = true;
        return TRIOSEQ_OK;
      };
      result = measure(nullptr, &rule_ms);
      for (size_t vi = 0; vi < ntiles && result == TRIOSEQ_OK; vi++) {
        for (int ti : kTI) {
          const trioseq_plan_s::Tuned cand{tiles[vi], ti};
          float ms = 3.0e38f;
          if ((result = measure(&cand, &ms)) != TRIOSEQ_OK) break;
          if (ms < best) {
            best = ms;
            bestv = cand;
          }
          if (moot) break;
        }
      }
      // once more, as warm as the candidates were
      if (result == TRIOSEQ_OK) result = measure(nullptr, &rule_ms);
    }
    if (result == TRIOSEQ_OK && !fits) result = TRIOSEQ_ENOMEM;
    const bool tuned = best < 0.98f * rule_ms;  // clearly faster than the rules' choice
    if (!tuned) bestv = rule;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (result != TRIOSEQ_OK) return result;
    if (tuned)
      plan->tuned[tune_key(mode, n, maxlen)] = bestv;
    else
      plan->tuned.erase(tune_key(mode, n, maxlen));  // later batches of the class follow the rules
    if (tile_j) *tile_j = bestv.var.nj;
    if (tile_k) *tile_k = bestv.var.nk;
    if (ti) *ti = bestv.TI;
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_plan_io_bytes(trioseq_plan_t plan, uint64_t* h2d, uint64_t* d2h) {
  return no_throw([&]() -> trioseq_status {
    if (!plan || !plan->last) return TRIOSEQ_EINVAL;
    if (h2d) *h2d = plan->last->h2d_bytes;
    if (d2h) *d2h = plan->last->d2h_bytes;
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_batch_destroy(trioseq_batch_t bt) {
  return no_throw([&]() -> trioseq_status {
    if (!bt) return TRIOSEQ_OK;
    DeviceGuard g(bt->plan->device);
    // Wait for this batch's own last run only; its buffers are then freed in the order of its
    // private stream. Other streams (a running server's included) are not synchronised.
    bt->ws->wait_last_use();
    delete bt;
    return TRIOSEQ_OK;
  });
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// Serving: continuous batching behind submit/poll.
//
// A server thread owns a FIFO of requests and kSlots slots, each a CUDA stream with its own
// reusable workspace and pinned result buffer. Every tick it (1) harvests slots whose launch has
// completed (event query, never a blocking wait) and publishes their results, then (2) admits
// pending requests into free slots: the oldest request fixes the (scoring, mode) group, and
// further requests of that group join the launch in arrival order while the launch's workspace
// estimate stays within the slot's share of the device-memory budget. Requests that arrive
// while other launches run are therefore admitted as soon as a slot frees, and launches of
// different slots overlap on the device. poll() only looks up the result table.
namespace {

using Clock = std::chrono::steady_clock;

struct SrvReq {
  uint64_t ticket = 0;
  int32_t plan_id = 0;
  uint32_t mode = 0;
  std::string s[3];
  size_t bytes = 0;        // workspace estimate inside a launch of several requests
  size_t bytes_alone = 0;  // estimate of a launch of this request alone (slab form if it applies)
};

struct SrvRes {
  trioseq_status st = TRIOSEQ_OK;
  int32_t score = 0;
  bool has_rows = false;
  std::string rows[3];
};

struct SrvSlot {
  cudaStream_t stream = nullptr;
  cudaEvent_t done = nullptr;
  bool busy = false;
  Workspace ws;
  HostPinned out;  // scores | error word | alignment lengths | rows
  size_t off_err = 0, off_lens = 0, off_rows = 0;
  std::unique_ptr<trioseq_batch_s> batch;
  std::vector<SrvReq> reqs;
  size_t bytes = 0;  // workspace admitted for the launch on this slot: its estimate, then at least what it took
  size_t cap = 0;    // the estimate and what the budget had left
  trioseq_status launch_st = TRIOSEQ_OK;
};

// Device bytes one request adds to a launch's workspace (boundary records, flags, inputs, and in traceback
// mode the code stream and rows): the most of the tiles that its launch may run on. kLean: the plan's own tile
// alone, to which make_batch falls back. kGroup: a launch with others, whose tasks together decide the tile, or
// which pairs it with one of them. Half of a pair on this request's own lengths is counted: one on the maximal
// lengths of unlike requests, or on the 4x4 tile of a launch of few tasks, may take more; the server counts what
// the launch then took, and make_batch keeps that to what the budget has left.
enum class Launch { kLean, kAlone, kGroup };
size_t request_bytes(const trioseq_plan_s* plan, uint32_t mode, const uint32_t len[3], Launch in) {
  const bool tb = mode == TRIOSEQ_WITH_TRACEBACK, group = in == Launch::kGroup;
  const bool own = in != Launch::kLean && auto_tile(plan, tb);
  const size_t a = len[0], b = len[1], c = len[2];
  const auto tasks = [&](const Variant& v) {
    const size_t WJ = (size_t)kPR * v.nj, WK = (size_t)kPC * v.nk;
    return ((b + WJ) / WJ) * ((c + WK) / WK);
  };
  // records of `slices` slices or steps of `ints` int32, codes of `steps` steps, flag and queue entry
  const auto sum = [&](const Variant& v, size_t slices, size_t ints, size_t steps) {
    const size_t cells = (size_t)kPR * v.nj * kPC * v.nk;
    return tasks(v) * (4 * slices * ints + (tb ? steps * cells / 2 : 0) + 4 + sizeof(Task));
  };
  const auto by_slice = [&](const Variant& v) {  // int32 records
    return sum(v, a + 1, kPC * v.nk + 4 + kPR * v.nj, a + 11);
  };
  const auto by_step = [&](const Variant& v) {  // two cells per register
    return sum(v, a + 19, vl_rec_j(v.nk / 2) + kVlRecK, a + 19);
  };
  const auto half_pair = [&](const Variant& v) {  // two triplets per register
    return sum(v, a + 11, vp_rec_j(v.nk) + vp_rec_k(v.nj), 0) / 2;
  };
  const Variant v = tb ? plan->tb_variant : plan->score_variant;
  size_t bytes = by_slice(v);
  if (v.vl && in != Launch::kLean) bytes = std::max(bytes, by_step(v));
  if (own && tb && plan->atype != kGlobal) bytes = std::max(bytes, by_slice(Variant{4, 4}));
  if (own && vl_admits(plan, tb)) {
    const bool narrow = tasks(Variant{4, 8, 1}) <= 2 * (size_t)plan->sms;
    if (narrow) bytes = std::max(bytes, by_step(Variant{4, 8, 1}));
    if (!narrow || group) bytes = std::max(bytes, by_step(Variant{8, 8, 1}));
  }
  if (own && group && !tb && plan->atype == kGlobal && plan->sig2_nonneg)
    bytes = std::max(bytes, half_pair(Variant{8, 4}));
  return bytes + a + b + c + 48 + sizeof(TripDesc) + 256 + (tb ? 3 * (a + b + c) + 64 : 0);
}

// Estimates of one request on a server of `budget` bytes, for a launch with others and for one alone.
//  * A global-type triplet whose one-launch workspace exceeds the plan's slab budget runs in slabs within that
//    budget when alone (build_batch), so it needs no more.
//  * One that fits the server's budget on the plan's own tile is not refused for the larger records of
//    another: make_batch keeps the launch to what the budget has left where it can.
//  * Affine gaps: the records, or the planes where a triplet's records exceed the budget; over planes every
//    triplet of a launch would take as much as the largest, so such a request joins no other.
void estimate(const trioseq_plan_s* plan, const uint32_t len[3], size_t budget, SrvReq* r) {
  size_t lean = request_bytes(plan, r->mode, len, Launch::kLean);
  if (plan->affine) {
    const size_t a = len[0], b = len[1], c = len[2];
    const size_t tasks = ((b + kAffineWJ) / kAffineWJ) * ((c + kAffineWK) / kAffineWK);
    const size_t rest = a + b + c + 48 + sizeof(TripDesc) + 512 + tasks * (4 + sizeof(Task));
    const size_t rec = 4 * tasks * (a + 1) * (size_t)(kAffineRecJ + kAffineRecK) + rest;
    const bool fits = rec <= std::min(plan->slab_budget, budget);
    r->bytes = fits ? rec : SIZE_MAX / 4;
    r->bytes_alone = fits ? rec : 256 * (b + 1) * (c + 1) + rest;
  } else {
    r->bytes = request_bytes(plan, r->mode, len, Launch::kGroup);
    r->bytes_alone = request_bytes(plan, r->mode, len, Launch::kAlone);
    if (plan->atype == kGlobal) {
      const size_t slabs = std::max<size_t>(plan->slab_budget, 1 << 20);
      r->bytes_alone = std::min(r->bytes_alone, slabs);
      lean = std::min(lean, slabs);
    }
  }
  if (lean <= budget) r->bytes_alone = std::min(r->bytes_alone, budget);
}

size_t workspace_device_bytes(const Workspace& ws) {
  return ws.inputs.cap + ws.faces.cap + ws.progress.cap + ws.codes.cap + ws.scores.cap +
         ws.rows.cap + ws.lens.cap + ws.planes.cap + ws.walkstate.cap + ws.best64.cap +
         ws.spans.cap;
}

}  // namespace

struct trioseq_server_s {
  static constexpr int kSlots = 4;
  std::vector<trioseq_plan_s*> plans;
  int device = 0;
  // Admission by device memory: launches on the device together hold at most `budget` bytes of
  // workspace estimates (in_flight). With no budget given, each admission is also bounded by
  // the memory free on the device at that moment. launch_share (budget / kSlots) caps how many
  // small requests one launch groups, so that several launches overlap; a single larger
  // request may use whatever room is left, and waits for room while other launches run.
  size_t budget = 0;
  size_t launch_share = 0;
  size_t in_flight = 0;
  bool budget_from_free = false;
  size_t max_pending = (size_t)1 << 20;  // TRIOSEQ_SERVER_MAX_PENDING at creation
  size_t max_batch = 1024;
  std::thread th;
  std::mutex mu;
  std::condition_variable cv;
  std::deque<SrvReq> pending;
  std::unordered_map<uint64_t, SrvRes> done;
  std::unordered_map<uint64_t, int> live;  // submitted and not yet consumed by poll
  uint64_t next_ticket = 1;
  bool stop = false;
  SrvSlot slots[kSlots];
};

namespace {

// Enqueue one launch for the requests in `sl.reqs` on the slot's stream (server thread, no lock).
trioseq_status srv_launch(trioseq_server_s* S, SrvSlot& sl) {
  const int32_t pid = sl.reqs.front().plan_id;
  const uint32_t mode = sl.reqs.front().mode;
  trioseq_plan_s* plan = S->plans[pid];
  std::vector<trioseq_triplet> trips(sl.reqs.size());
  for (size_t i = 0; i < sl.reqs.size(); i++)
    for (int q = 0; q < 3; q++) {
      trips[i].s[q] = sl.reqs[i].s[q].data();
      trips[i].len[q] = (uint32_t)sl.reqs[i].s[q].size();
    }
  trioseq_status st =
      make_batch(plan, trips.data(), trips.size(), mode, &sl.ws, sl.stream, Staging::kPinned,
                 &sl.batch, sl.cap);
  if (st != TRIOSEQ_OK) return st;
  trioseq_batch_s* bt = sl.batch.get();
  NvtxRange range("trioseq_server_launch");
  if ((st = run(bt, sl.stream)) != TRIOSEQ_OK) return st;
  const bool tb = mode == TRIOSEQ_WITH_TRACEBACK;
  const size_t n = bt->n, ntb = bt->tb_trips.size();
  sl.off_err = align_up(n * 4, 64);
  sl.off_lens = sl.off_err + 64;
  sl.off_rows = align_up(sl.off_lens + ntb * 4, 64);
  const size_t need = sl.off_rows + (tb ? bt->rows_bytes : 0);
  if (!sl.out.ensure(need)) return TRIOSEQ_ENOMEM;
  char* h = reinterpret_cast<char*>(sl.out.p);
  int32_t* err = sl.ws.progress.as<int32_t>() + bt->tasks.size() + 32;
  cudaError_t e = cudaMemcpyAsync(h, sl.ws.scores.p, n * 4, cudaMemcpyDeviceToHost, sl.stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h + sl.off_err, err, 4, cudaMemcpyDeviceToHost, sl.stream);
  if (e == cudaSuccess && tb && ntb) {
    e = cudaMemcpyAsync(h + sl.off_lens, sl.ws.lens.p, ntb * 4, cudaMemcpyDeviceToHost,
                        sl.stream);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(h + sl.off_rows, sl.ws.rows.p, bt->rows_bytes, cudaMemcpyDeviceToHost,
                          sl.stream);
  }
  if (e == cudaSuccess) e = cudaEventRecord(sl.done, sl.stream);
  return cuda_status(e);
}

// Turn a finished slot into results (server thread, lock held).
void srv_harvest(trioseq_server_s* S, SrvSlot& sl) {
  trioseq_batch_s* bt = sl.batch.get();
  const char* h = reinterpret_cast<const char*>(sl.out.p);
  trioseq_status st = sl.launch_st;
  // A launch that failed part-way may have left work on the stream: drain it before the
  // slot's workspace is reused.
  if (st != TRIOSEQ_OK) cudaStreamSynchronize(sl.stream);
  if (st == TRIOSEQ_OK && cudaEventQuery(sl.done) != cudaSuccess) st = TRIOSEQ_ECUDA;
  int32_t herr = 0;
  if (st == TRIOSEQ_OK) {
    std::memcpy(&herr, h + sl.off_err, 4);
    if (herr & 1) st = TRIOSEQ_ETIMEOUT;
    else if (herr & 2) st = TRIOSEQ_ECUDA;
  }
  const char* alpha = st == TRIOSEQ_OK ? bt->plan->alphabet : nullptr;
  for (size_t i = 0; i < sl.reqs.size(); i++) {
    SrvRes r;
    r.st = st;
    if (st == TRIOSEQ_OK) {
      std::memcpy(&r.score, h + 4 * i, 4);
      const int32_t q = bt->tb_of[i];
      if (q >= 0) {
        int32_t L = 0;
        std::memcpy(&L, h + sl.off_lens + 4 * (size_t)q, 4);
        const int32_t rc = bt->row_cap[q];
        const uint8_t* base =
            reinterpret_cast<const uint8_t*>(h + sl.off_rows + (size_t)bt->row_off[q]);
        r.has_rows = true;
        r.st = no_throw([&] {
          for (int s = 0; s < 3; s++) {
            r.rows[s].resize((size_t)L);
            const uint8_t* row = base + (size_t)s * rc + (rc - L);
            for (int32_t t = 0; t < L; t++) r.rows[s][t] = row[t] == 255 ? '-' : alpha[row[t]];
          }
          return TRIOSEQ_OK;
        });
        if (r.st != TRIOSEQ_OK) {
          r.has_rows = false;
          for (auto& x : r.rows) std::string().swap(x);
        }
      }
    }
    S->done[sl.reqs[i].ticket] = std::move(r);
  }
  sl.reqs.clear();
  sl.batch.reset();
  sl.busy = false;
  S->in_flight -= std::min(S->in_flight, sl.bytes);
  sl.bytes = 0;
}

void srv_loop(trioseq_server_s* S) {
  cudaSetDevice(S->device);
  std::unique_lock<std::mutex> lk(S->mu);
  for (;;) {
    bool busy_any = false, acted = false;
    for (auto& sl : S->slots) {
      if (!sl.busy) continue;
      if (sl.launch_st != TRIOSEQ_OK || cudaEventQuery(sl.done) != cudaErrorNotReady) {
        srv_harvest(S, sl);
        acted = true;
      } else {
        busy_any = true;
      }
    }
    for (auto& sl : S->slots) {
      if (sl.busy || S->pending.empty()) continue;
      // Room for a launch on this slot: the budget minus the launches in flight, and with no
      // budget given, no more than the device has free now (plus what this slot already holds,
      // which the launch reuses).
      size_t room = S->budget > S->in_flight ? S->budget - S->in_flight : 0;
      if (S->budget_from_free) {
        size_t fr = 0, tot = 0;
        if (cudaMemGetInfo(&fr, &tot) == cudaSuccess)
          room = std::min(room, fr / 10 * 9 + workspace_device_bytes(sl.ws));
        else
          cudaGetLastError();
      }
      bool others_busy = false;
      for (auto& o : S->slots) others_busy = others_busy || o.busy;
      const SrvReq& head = S->pending.front();
      if (head.bytes_alone > room) {
        if (others_busy) break;  // wait: harvested launches give their room back
        if (head.bytes_alone > S->budget) {  // can never fit: fail it alone
          SrvRes r;
          r.st = TRIOSEQ_ENOMEM;
          S->done[head.ticket] = std::move(r);
          S->pending.pop_front();
          acted = true;
          continue;
        }
        // nothing else runs: launch it; its allocations report a real shortage (ENOMEM)
      }
      // Form a launch: the oldest request fixes the group; same-group requests follow in arrival
      // order while the launch's estimate stays within its share of the room.
      const int32_t pid = head.plan_id;
      const uint32_t mode = head.mode;
      const size_t limit = std::max(head.bytes_alone, std::min(room, S->launch_share));
      size_t full = 0;
      std::deque<SrvReq> rest;
      while (!S->pending.empty()) {
        SrvReq& r = S->pending.front();
        const bool same = r.plan_id == pid && r.mode == mode;
        if (sl.reqs.empty() ||
            (same && sl.reqs.size() < S->max_batch && full + r.bytes <= limit)) {
          full += r.bytes;
          sl.reqs.push_back(std::move(r));
        } else {
          rest.push_back(std::move(r));
        }
        S->pending.pop_front();
        if (sl.reqs.size() >= S->max_batch || full >= limit) break;
      }
      while (!rest.empty()) {  // keep arrival order of what was skipped
        S->pending.push_front(std::move(rest.back()));
        rest.pop_back();
      }
      sl.bytes = sl.reqs.size() == 1 ? sl.reqs.front().bytes_alone : full;
      S->in_flight += sl.bytes;
      sl.cap = sl.bytes + (S->budget > S->in_flight ? S->budget - S->in_flight : 0);
      sl.busy = true;
      acted = true;
      lk.unlock();
      sl.launch_st = no_throw([&] { return srv_launch(S, sl); });  // the thread must not throw
      lk.lock();
      if (sl.batch && layout_bytes(*sl.batch) > sl.bytes) {  // a pair of unlike requests, for instance
        S->in_flight += layout_bytes(*sl.batch) - sl.bytes;
        sl.bytes = layout_bytes(*sl.batch);
      }
      busy_any = true;
    }
    if (S->stop && S->pending.empty() && !busy_any) break;
    if (!acted) S->cv.wait_for(lk, std::chrono::microseconds(busy_any ? 20 : 2000));
  }
}

}  // namespace

extern "C" {

trioseq_status trioseq_server_create(const trioseq_plan_t* plans, int32_t nplans,
                                     size_t hbm_budget, trioseq_server_t* out) {
  return no_throw([&]() -> trioseq_status {
    if (!out) return TRIOSEQ_EINVAL;
    *out = nullptr;
    if (!plans || nplans < 1) return TRIOSEQ_EINVAL;
    for (int32_t i = 0; i < nplans; i++)
      if (!plans[i] || plans[i]->device != plans[0]->device) return TRIOSEQ_EINVAL;
    std::unique_ptr<trioseq_server_s> S(new (std::nothrow) trioseq_server_s());
    if (!S) return TRIOSEQ_ENOMEM;
    S->plans.assign(plans, plans + nplans);
    S->device = plans[0]->device;
    DeviceGuard g(S->device);
    if (hbm_budget == 0) {
      size_t fr = 0, tot = 0;
      if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) return cuda_status(cudaGetLastError());
      hbm_budget = fr / 10 * 8;
      S->budget_from_free = true;
    }
    S->budget = std::max<size_t>(hbm_budget, 1 << 20);
    S->launch_share = std::max<size_t>(S->budget / trioseq_server_s::kSlots, 1 << 20);
    S->max_pending = (size_t)std::max(0, env_int("TRIOSEQ_SERVER_MAX_PENDING", 1 << 20));
    for (auto& sl : S->slots) {
      if (cudaStreamCreateWithFlags(&sl.stream, cudaStreamNonBlocking) != cudaSuccess ||
          cudaEventCreateWithFlags(&sl.done, cudaEventDisableTiming) != cudaSuccess)
        return cuda_status(cudaGetLastError());
      sl.ws.alloc_stream = sl.stream;
    }
    try {
      S->th = std::thread(srv_loop, S.get());
    } catch (...) {
      return TRIOSEQ_ENOMEM;
    }
    *out = S.release();
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_submit(trioseq_server_t S, const trioseq_triplet* t, int32_t plan_id,
                              uint32_t mode, uint64_t* ticket) {
  return no_throw([&]() -> trioseq_status {
    if (!S || !t || !ticket || plan_id < 0 || plan_id >= (int32_t)S->plans.size() ||
        mode > TRIOSEQ_WITH_TRACEBACK)
      return TRIOSEQ_EINVAL;
    const trioseq_plan_s* plan = S->plans[plan_id];
    SrvReq r;
    r.plan_id = plan_id;
    r.mode = mode;
    int64_t sumlen = 0;
    for (int q = 0; q < 3; q++) {
      if (t->len[q] && !t->s[q]) return TRIOSEQ_EINVAL;
      if (t->len[q] > (1u << 24)) return TRIOSEQ_EOVERFLOW;
      const unsigned char* src = reinterpret_cast<const unsigned char*>(t->s[q]);
      for (uint32_t e = 0; e < t->len[q]; e++)
        if (plan->lut[src[e]] < 0) return TRIOSEQ_EINVAL;
      r.s[q].assign(t->s[q] ? t->s[q] : "", t->len[q]);
      sumlen += t->len[q];
    }
    if ((int64_t)std::max(plan->max_abs_sig2, plan->atype != kGlobal ? -2 * plan->gap : 0) *
            sumlen >= (1LL << 26) - 1)
      return TRIOSEQ_EOVERFLOW;
    estimate(plan, t->len, S->budget, &r);
    {
      std::lock_guard<std::mutex> lk(S->mu);
      if (S->stop) return TRIOSEQ_EINVAL;
      if (S->pending.size() >= S->max_pending) return TRIOSEQ_EAGAIN;
      r.ticket = S->next_ticket++;
      *ticket = r.ticket;
      S->live[r.ticket] = 0;
      S->pending.push_back(std::move(r));
    }
    S->cv.notify_one();
    return TRIOSEQ_OK;
  });
}

trioseq_status trioseq_poll(trioseq_server_t S, uint64_t ticket, int32_t* score, char* rows[3],
                            size_t cap, size_t* aln_len) {
  return no_throw([&]() -> trioseq_status {
    if (!S) return TRIOSEQ_EINVAL;
    std::lock_guard<std::mutex> lk(S->mu);
    auto it = S->done.find(ticket);
    if (it == S->done.end()) return S->live.count(ticket) ? TRIOSEQ_EAGAIN : TRIOSEQ_EINVAL;
    SrvRes& r = it->second;
    if (r.st == TRIOSEQ_OK && r.has_rows) {
      if (aln_len) *aln_len = r.rows[0].size();
      if (rows) {
        if (cap < r.rows[0].size() || !rows[0] || !rows[1] || !rows[2]) return TRIOSEQ_EINVAL;
        for (int s = 0; s < 3; s++) std::memcpy(rows[s], r.rows[s].data(), r.rows[s].size());
      }
    } else if (aln_len) {
      *aln_len = 0;
    }
    if (score) *score = r.score;
    const trioseq_status st = r.st;
    S->done.erase(it);
    S->live.erase(ticket);
    return st;
  });
}

trioseq_status trioseq_server_destroy(trioseq_server_t S) {
  return no_throw([&]() -> trioseq_status {
    if (!S) return TRIOSEQ_OK;
    {
      std::lock_guard<std::mutex> lk(S->mu);
      S->stop = true;
    }
    S->cv.notify_all();
    if (S->th.joinable()) S->th.join();
    {
      DeviceGuard g(S->device);
      for (auto& sl : S->slots) {
        if (sl.stream) cudaStreamSynchronize(sl.stream);
        sl.batch.reset();
        sl.ws.release();  // freed in the slot stream's order, while the stream exists
        if (sl.stream) cudaStreamSynchronize(sl.stream);
        if (sl.done) cudaEventDestroy(sl.done);
        if (sl.stream) cudaStreamDestroy(sl.stream);
      }
    }
    delete S;
    return TRIOSEQ_OK;
  });
}

}  // extern "C"

// Host side of the C ABI (include/ddm.h): argument checks, device workspace,
// stream-ordered launches and the single status read-back per call.
#include <algorithm>
#include <cmath>
#include <utility>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <new>

#include <nvtx3/nvToolsExt.h>

#include "ddm_internal.cuh"

using namespace ddm;

namespace {
std::atomic<unsigned long long> g_launches{0};
}  // namespace

void ddm::note_launches(unsigned count) { g_launches.fetch_add(count, std::memory_order_relaxed); }

namespace {

struct DevBuf {
  void* p = nullptr;
  size_t cap = 0;
};

// Workspace of one set's ordering.
struct OrderBufs {
  DevBuf keys[2], vals[2], hist, lookback, counters;  // radix sort
  DevBuf aos;                                         // interleaved coordinates
  DevBuf bglog2, bngroups, bgbase, sums;              // re-sort groups of instances
  DevBuf* all[11] = {&keys[0], &keys[1], &vals[0], &vals[1], &hist, &lookback, &counters, &aos,
                     &bglog2, &bngroups, &bgbase};
};

}  // namespace

struct ddm_ctx {
  int device = 0;
  int sms = 0;
  uint64_t alloc_limit = 0;  // 0 = unlimited (testing aid)
  uint64_t allocated = 0;

  // Workspace comes from the context's own memory pool, allocated and freed
  // in stream order on the calling stream: growing a buffer never
  // synchronises the device (cudaMalloc / cudaFree would), so one context's
  // growth does not stall the work of others.  The pool keeps what is freed
  // (no release threshold) for the next growth.
  cudaMemPool_t pool = nullptr;
  cudaStream_t cur = nullptr;      // stream of the call in progress
  bool capturing = false;          // that stream is being captured into a graph
  // Calls may come on different streams: each call records `done` on its
  // stream when it has enqueued its work, and a call on another stream first
  // waits for it, so the context's buffers are never used by two streams at
  // once and a stream-ordered free never overtakes earlier work.
  cudaEvent_t done = nullptr;
  cudaStream_t last = nullptr;
  bool done_pending = false;

  Status* st_dev = nullptr;
  Status* st_host = nullptr;  // pinned mirror

  // Ordering workspace: [0] serves both sets in turn; [1] the updates of a
  // one-shot call, ordered on `side` while the tree is built.
  // Between calls and after the join [1] is given back when room runs out,
  // unless a recorded call uses it.
  OrderBufs ob[2];
  bool side_busy = false, side_recorded = false;
  cudaStream_t side = nullptr;
  cudaEvent_t fork = nullptr, joined = nullptr;
  // tree
  DevBuf e, sid, nodes, tab;
  bool tables_on = true;        // rank tables of the leaves (ddm_set_tiling)
  // plan: sorted updates, per-update counts and offsets
  DevBuf qe, qid, counts, counts_pos, offsets, pos_offsets, sums;
  // range selection for ddm_write over a sub-range of updates
  DevBuf sel_offs, sel_list;
  // replay records of the count pass
  DevBuf rec, blk_own, blk_count, pkt_nblk, pkt_off, blk_list,
      plan_state, order_state;
  uint64_t replay_budget = 0;   // bytes; 0 = never record
  uint32_t rec_blocks = 0;      // blocks of the current arena
  // Blocks needed, packets and blocks held by the latest recorded count
  // pass, copied back by every plan without a host synchronisation (pinned;
  // read as a sizing hint for the next arena, possibly one plan stale).
  volatile uint32_t* rec_hint = nullptr;
  RecordArena arena{};          // arena of the current plan (max_blocks 0 = none)
  // batched instances
  DevBuf inst_s, inst_u;
  DevBuf leaf_off;              // padded tree of a batch
  // size classes of the tree order (d >= 2)
  DevBuf cls_hist, cls_off;
  DevBuf probe;                 // words polled by the ddm_debug_*_timeout calls
  BatchView bv{};               // count 0 = single problem
  // tuning knobs (ddm_set_tuning)
  int str_shift = 0;            // added to the re-sort group exponents
  uint32_t ctas_per_sm = 8;     // CTAs per SM of the packet kernels
  bool replay_on = true;        // record / replay write pass allowed
  uint32_t upd_base = 0;        // added to update ids in written pairs (ddm_set_update_id_base)
  // tiling (ddm_set_tiling): log2 of the queries per packet, and the number of
  // a packet's queries meeting a leaf from which the count pass swaps the loops
  uint32_t qpp_log2 = 5;
  bool ordered = false;         // the plan holds the plan order's offsets and entries
  uint32_t plan_qpp_log2 = 5;   // of the current plan (smaller for few updates)
  uint32_t tmin = 12;

  // Within one call: the status block (with the ticket words) is zero from
  // reset_status() to the words' first use.
  bool work_zeroed[2] = {false, false};
  // Within one synchronising call: a walking write pass held back, to be run
  // only if the replay reports incomplete records.
  bool walk_pending = false;
  QueryView walk_q{};
  WriteView walk_w{};

  bool built = false;
  bool attached = false;        // tree borrowed from another context (ddm_attach)
  bool swapped = false;         // one-shot call with DDM_SWAP_ROLES: tree over the updates
  uint64_t last_tests = 0;      // (query, leaf) tests of the last count pass read back
  TreeView tree{};
  bool planned = false;
  const float* ulo = nullptr;
  const float* uhi = nullptr;
  uint32_t m = 0;
  uint32_t flags = 0;
};

namespace {

// NVTX range around a phase of a call (tree build, plan, write pass, refit),
// so that a timeline tool shows the library's phases by name.  NVTX is
// header-only and costs nothing when no tool is attached.
class Phase {
 public:
  explicit Phase(const char* name) { nvtxRangePushA(name); }
  ~Phase() { nvtxRangePop(); }
};

class DeviceGuard {
 public:
  explicit DeviceGuard(int dev) {
    ok_ = cudaGetDevice(&prev_) == cudaSuccess;
    if (ok_ && prev_ != dev) ok_ = cudaSetDevice(dev) == cudaSuccess;
    switched_ = ok_ && prev_ != dev;
  }
  ~DeviceGuard() {
    if (switched_) cudaSetDevice(prev_);
  }
  bool ok() const { return ok_; }

 private:
  int prev_ = 0;
  bool ok_ = false, switched_ = false;
};

// Orders a call's work after the context's previous call (made on another
// stream) and marks its end; binds the call's stream for ensure().  A stream
// being captured into a graph is neither waited on nor recorded (its work runs
// only when the graph is launched); growth is refused while capturing.
class StreamUse {
 public:
  StreamUse(ddm_ctx* c, cudaStream_t s) : c_(c), s_(s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
      cudaGetLastError();
      st = cudaStreamCaptureStatusNone;
    }
    capturing_ = st != cudaStreamCaptureStatusNone;
    if (!capturing_ && c->done_pending && c->last != s) cudaStreamWaitEvent(s, c->done, 0);
    c->cur = s;
    c->capturing = capturing_;
  }
  ~StreamUse() {
    c_->work_zeroed[0] = c_->work_zeroed[1] = false;
    c_->walk_pending = false;
    c_->side_busy = false;
    if (!capturing_ && cudaEventRecord(c_->done, s_) == cudaSuccess) {
      c_->done_pending = true;
      c_->last = s_;
    }
    cudaGetLastError();
    c_->capturing = false;
  }

 private:
  ddm_ctx* c_;
  cudaStream_t s_;
  bool capturing_ = false;
};

// Whether ticket word i is still zero from this call's reset_status().
bool zeroed_work(ddm_ctx* c, int i) {
  const bool z = c->work_zeroed[i];
  c->work_zeroed[i] = false;
  return z;
}

void release_now(ddm_ctx* c, DevBuf& b) {
  if (b.p) {
    cudaFreeAsync(b.p, c->cur);
    c->allocated -= b.cap;
  }
  b.p = nullptr;
  b.cap = 0;
}

// Gives the side stream's workspace back; false if there is none to give.
bool release_side(ddm_ctx* c) {
  if (c->side_recorded) return false;
  const uint64_t before = c->allocated;
  for (DevBuf* b : c->ob[1].all) release_now(c, *b);
  release_now(c, c->ob[1].sums);
  return c->allocated != before;
}

int grow(ddm_ctx* c, DevBuf& b, size_t bytes) {
  size_t want = bytes + bytes / 4;  // headroom against regrowth
  if (b.p) {
    cudaFreeAsync(b.p, c->cur);  // after the work already enqueued on this stream
    c->allocated -= b.cap;
    b.p = nullptr;
    b.cap = 0;
  }
  if (c->alloc_limit && c->allocated + want > c->alloc_limit) {
    want = bytes;
    if (c->allocated + want > c->alloc_limit) return DDM_ERR_NOMEM;
  }
  if (cudaMallocFromPoolAsync(&b.p, want, c->pool, c->cur) != cudaSuccess) {
    cudaGetLastError();  // clear the allocation error
    b.p = nullptr;
    return DDM_ERR_NOMEM;
  }
  b.cap = want;
  c->allocated += want;
  return DDM_OK;
}

int ensure(ddm_ctx* c, DevBuf& b, size_t bytes) {
  if (bytes <= b.cap) return DDM_OK;
  if (c->capturing) return DDM_ERR_NOMEM;  // a graph cannot own the workspace
  int rc = grow(c, b, bytes);
  // What a call needs goes before what only runs it faster.
  if (rc == DDM_ERR_NOMEM && !c->side_busy && release_side(c)) rc = grow(c, b, bytes);
  return rc;
}

// Interleaved copy of a set's coordinates for the gathers by id; NULL (the
// gathers then read the caller's rows) if it cannot be allocated.
float2* aos_buffer(ddm_ctx* c, OrderBufs& o, int d, uint32_t cnt) {
  if (cnt == 0 || ensure(c, o.aos, sizeof(float2) * (size_t)d * cnt) != DDM_OK) return nullptr;
  return static_cast<float2*>(o.aos.p);
}

void release(DevBuf& b) {
  if (b.p) cudaFreeAsync(b.p, nullptr);
  b.p = nullptr;
  b.cap = 0;
}

#define DDM_TRY(expr)              \
  do {                             \
    int rc_ = (expr);              \
    if (rc_ != DDM_OK) return rc_; \
  } while (0)
#define DDM_CUDA(expr)                    \
  do {                                    \
    if ((expr) != cudaSuccess) {          \
      cudaGetLastError();                 \
      return DDM_ERR_CUDA;                \
    }                                     \
  } while (0)

bool set_ok(int d, const float* lo, const float* hi, uint32_t cnt) {
  if (cnt > DDM_MAX_EXTENTS) return false;
  if (cnt > 0 && (!lo || !hi)) return false;
  (void)d;
  return true;
}

int walk_write(ddm_ctx* c, const QueryView& q, const WriteView& w, cudaStream_t s);

// Reads the status block back (and runs the walking write pass held back by
// this call if the replay asked for it).
int sync_status(ddm_ctx* c, cudaStream_t s) {
  DDM_CUDA(cudaMemcpyAsync(c->st_host, c->st_dev, sizeof(Status), cudaMemcpyDeviceToHost, s));
  DDM_CUDA(cudaStreamSynchronize(s));
  if (!c->walk_pending) return DDM_OK;
  c->walk_pending = false;
  if (!c->st_host->walk) return DDM_OK;
  DDM_TRY(walk_write(c, c->walk_q, c->walk_w, s));
  DDM_CUDA(cudaMemcpyAsync(c->st_host, c->st_dev, sizeof(Status), cudaMemcpyDeviceToHost, s));
  DDM_CUDA(cudaStreamSynchronize(s));
  return DDM_OK;
}

int status_code(const Status& st) {
  if (st.err & kErrChecked) return DDM_ERR_INTERNAL;
  if (st.err & kErrTimeout) return DDM_ERR_TIMEOUT;
  if (st.err & kErrExtent) return DDM_ERR_EXTENT;
  if (st.err & kErrCapacity) return DDM_ERR_CAPACITY;
  return DDM_OK;
}

int ensure_sort(ddm_ctx* c, OrderBufs& o, uint32_t cnt) {
  DDM_TRY(ensure(c, o.keys[0], sizeof(unsigned long long) * cnt));
  DDM_TRY(ensure(c, o.keys[1], sizeof(unsigned long long) * cnt));
  DDM_TRY(ensure(c, o.vals[0], sizeof(uint32_t) * cnt));
  DDM_TRY(ensure(c, o.vals[1], sizeof(uint32_t) * cnt));
  DDM_TRY(ensure(c, o.hist, sizeof(uint32_t) * 8 * 256));
  DDM_TRY(ensure(c, o.counters, sizeof(uint32_t) * 8));
  DDM_TRY(ensure(c, o.lookback, sizeof(uint32_t) * sort_lookback_words(cnt)));
  return DDM_OK;
}

// Radix sort of the keys/ids in buffer pair `cur` over `passes` 8-bit
// digits; `cur` is updated to the buffer pair holding the result.
int sort_pass(ddm_ctx* c, OrderBufs& o, uint32_t cnt, int passes, int* cur, cudaStream_t s) {
  SortScratch sc;
  sc.keys[0] = static_cast<unsigned long long*>(o.keys[*cur].p);
  sc.keys[1] = static_cast<unsigned long long*>(o.keys[*cur ^ 1].p);
  sc.vals[0] = static_cast<uint32_t*>(o.vals[*cur].p);
  sc.vals[1] = static_cast<uint32_t*>(o.vals[*cur ^ 1].p);
  sc.hist = static_cast<uint32_t*>(o.hist.p);
  sc.lookback = static_cast<uint32_t*>(o.lookback.p);
  sc.counters = static_cast<uint32_t*>(o.counters.p);
  int out = 0;
  DDM_CUDA(launch_sort64(sc, cnt, passes, &out, c->st_dev, c->sms, s));
  *cur ^= out;
  return DDM_OK;
}

// A set is sorted into the spatial order used by the tree: dimension-0 key
// first, then, for each further dimension with a group size, a stable re-sort
// by that dimension's lower bound inside aligned groups.  The order_set
// functions validate the set on the way and return the buffer pair whose vals
// hold the order.

// Bits needed to hold values 0..v.
int bits_of(uint64_t v) {
  int b = 0;
  while (v) {
    ++b;
    v >>= 1;
  }
  return b;
}
// Bits of a set's ids in packed words.
int id_bits_of(uint32_t cnt) { return std::max(bits_of(cnt - 1u), 1); }

// Packed sort of a set (launch_sort_packed): the ids end up in vals[0], so
// *cur becomes 0.  A source's k32 lies in vals[1].
int packed_pass(ddm_ctx* c, OrderBufs& o, uint32_t cnt, const uint32_t* hi, bool source, int key_bits,
                int id_bits, int* cur, cudaStream_t s, const float* second = nullptr) {
  SortScratch sc;
  for (int b = 0; b < 2; ++b) {
    sc.keys[b] = static_cast<unsigned long long*>(o.keys[b].p);
    sc.vals[b] = static_cast<uint32_t*>(o.vals[b].p);
  }
  sc.hist = static_cast<uint32_t*>(o.hist.p);
  sc.lookback = static_cast<uint32_t*>(o.lookback.p);
  sc.counters = static_cast<uint32_t*>(o.counters.p);
  const SortSource src{source ? sc.vals[1] : nullptr, hi, 24, id_bits, second != nullptr,
                       second ? &c->st_dev->both : nullptr, second};
  DDM_CUDA(launch_sort_packed(sc, src, cnt, key_bits, c->st_dev, c->sms, s));
  *cur = 0;
  return DDM_OK;
}

// Re-sort of the ids in vals[*cur] by (group, locality key) over the whole
// set, `groups` numbered groups: the keys are written by `rekey`(keys[0],
// id_bits), packed with the ids if they fit one word.
template <typename Rekey>
int resort_pass(ddm_ctx* c, OrderBufs& o, uint32_t cnt, uint64_t groups, int* cur, Rekey rekey,
                cudaStream_t s) {
  const int key_bits = 24 + bits_of(groups - 1u), id_bits = id_bits_of(cnt);
  if (key_bits + id_bits <= 64) {
    DDM_CUDA(rekey(static_cast<unsigned long long*>(o.keys[0].p), id_bits));
    return packed_pass(c, o, cnt, nullptr, false, key_bits, id_bits, cur, s);
  }
  DDM_CUDA(rekey(static_cast<unsigned long long*>(o.keys[*cur].p), 0));
  return sort_pass(c, o, cnt, (key_bits + 7) / 8, cur, s);
}

// Re-sort of the ids in buffer pair `cur` inside the plan's groups (in place).
int seg_pass(ddm_ctx* c, OrderBufs& o, uint32_t cnt, const float* lo_k, int g, const SegPlan& plan, int tile_log2,
             int cur, cudaStream_t s) {
  DDM_CUDA(launch_segsort(static_cast<uint32_t*>(o.vals[cur].p), lo_k, cnt, g, plan, tile_log2,
                          static_cast<unsigned long long*>(o.keys[0].p),
                          static_cast<unsigned long long*>(o.keys[1].p), c->sms, s));
  return DDM_OK;
}

// Sets up to this size are ordered by counting.  Quadratic against the cluster
// sort's passes, of which a d = 1 tree needs eight, the others three or four.
// Measured, one match of n + n extents, by radix sort and by counting: d = 1,
// n = 64: 90 / 65 us, 4,096: 105 / 78, 8,192: 112 / 92, 10,000: 116 / 111 (and
// 117 / 122 at 12,000); d = 2, n = 64: 91 / 81, 4,096: 123 / 115, 6,000: 126 /
// 122, 8,192: 126 / 134; d = 3, n = 4,096: 155 / 150, 6,000: 155 / 152, 8,192:
// 159 / 163.
uint32_t rank_sort_max(int d) { return d == 1 ? 8192u : 6144u; }

// Batched sets: the instance is the major sort key, and each instance's
// re-sort groups are sized from its own extent count.
struct BatchSet {
  const unsigned long long* off;  // [count + 1] positions of each instance
  uint32_t count;
  uint32_t* inst;                 // [cnt] instance of each position (filled here)
  uint32_t padded;                // positions of the padded tree (BatchView), 0: not padded
  unsigned long long* leaf_off;   // [count + 1] of the padded tree (filled here), or null
};

// Workspace of order_set_batch.
int ensure_batch(ddm_ctx* c, OrderBufs& o, int d, uint32_t cnt, uint32_t count) {
  DDM_TRY(ensure_sort(c, o, cnt));
  DDM_TRY(ensure(c, o.bglog2, sizeof(int) * (size_t)d * count));
  DDM_TRY(ensure(c, o.sums, sizeof(unsigned long long) * batch_plan_words(count, d)));
  return ensure(c, o.bgbase, sizeof(unsigned long long) * (size_t)d * ((size_t)count + 1));
}

int order_set_batch(ddm_ctx* c, OrderBufs& o, int d, const float* lo, const float* hi, uint32_t cnt,
                    const BatchSet& bs, float2* aos, int* cur, cudaStream_t s) {
  *cur = 0;
  DDM_TRY(ensure_batch(c, o, d, cnt, bs.count));
  // Sizes are known on the device only, so the chunks of the re-sorts and the
  // leaves are planned there.
  auto* gl = static_cast<int*>(o.bglog2.p);
  auto* cb = static_cast<unsigned long long*>(o.bgbase.p);
  if (d > 1 || bs.leaf_off)
    DDM_CUDA(launch_batch_plan(bs.off, bs.count, cnt, d, c->str_shift, kSegTileLog2, gl, cb, bs.leaf_off,
                               static_cast<unsigned long long*>(o.sums.p), s));
  DDM_CUDA(launch_fill_inst(bs.off, bs.count, cnt, bs.inst, c->sms, s));
  const int inst_bits = bits_of(bs.count ? bs.count - 1u : 0u), id_bits = id_bits_of(cnt);
  const bool packed = inst_bits + 24 + id_bits <= 64;
  DDM_CUDA(launch_validate_batch(d, lo, hi, cnt, bs.inst,
                                 static_cast<unsigned long long*>(o.keys[0].p),
                                 static_cast<uint32_t*>(o.vals[0].p),
                                 packed ? static_cast<uint32_t*>(o.vals[1].p) : nullptr, aos,
                                 c->st_dev, c->sms, s));
  if (packed)
    DDM_TRY(packed_pass(c, o, cnt, inst_bits ? bs.inst : nullptr, true, 24 + inst_bits, id_bits, cur, s));
  else
    DDM_TRY(sort_pass(c, o, cnt, (24 + inst_bits + 7) / 8, cur, s));
  // The re-sorts stay inside an instance's groups.
  for (int k = 1; k < d; ++k)
    DDM_TRY(seg_pass(c, o, cnt, lo + (size_t)k * cnt, 0,
                     SegPlan{bs.off, gl + (size_t)k * bs.count, cb + (size_t)k * (bs.count + 1u), bs.count},
                     kSegTileLog2, *cur, s));
  return DDM_OK;
}

// A tile of 2^t positions, the groups' size, or more positions per CTA where
// that leaves CTAs to spare: a chunk's time grows with the keys per thread
// (ballots), so few chunks are better small, many better large (31,627
// positions in groups of 1,024: 18.3 us in eight chunks, 8.6 in 31; the served
// request 119 -> 107 us).
int tile_for(uint32_t cnt, int t, int sms) {
  while (t < kSegTileLog2 && (cnt >> t) > (uint32_t)sms) ++t;
  return t;
}

// Tile of the on-chip re-sort of dimension k for a single problem of cnt
// extents (no class or set of it has larger groups), or 0 if its groups may be
// larger than a CTA takes: groups of 2^13 positions reach to about 2e6 (d = 2)
// or 2e5 (d = 3, k = 1) extents, and beyond there are as many CTAs' worth of
// positions per group that one radix sort over the set is the better form.
int seg_tile(uint32_t cnt, int d, int k, int shift, int sms) {
  if (cnt < 64u) return kSegTileLog2Min;
  const double nb = (double)((cnt + 31u) / 32u);
  const double e = std::log2(32.0 * std::pow(nb, (double)(d - k) / (double)d)) + shift;
  for (int t = kSegTileLog2Min; t <= kSegTileLog2Max; ++t)
    if (e < t + 0.49) return tile_for(cnt, t, sms);
  return 0;
}

// Tree order for d >= 2: sort by (size class, lower bound), then refine
// each class by the sort-tile-recursive re-sorts of its own size (the
// per-instance machinery of batched sets, with the classes as instances).
int order_set_classes(ddm_ctx* c, OrderBufs& o, int d, const float* lo, const float* hi, uint32_t cnt,
                      float2* aos, int* cur, cudaStream_t s) {
  constexpr uint32_t kClasses = 256;
  *cur = 0;
  DDM_TRY(ensure_sort(c, o, cnt));
  DDM_TRY(ensure(c, c->cls_hist, sizeof(uint32_t) * kClasses));
  DDM_TRY(ensure(c, c->cls_off, sizeof(unsigned long long) * (kClasses + 1)));
  DDM_TRY(ensure(c, o.bglog2, sizeof(int) * kClasses * DDM_MAX_DIMS));
  DDM_TRY(ensure(c, o.bngroups, sizeof(uint32_t) * kClasses));
  DDM_TRY(ensure(c, o.bgbase, sizeof(unsigned long long) * (kClasses + 1) * DDM_MAX_DIMS));
  DDM_TRY(ensure(c, o.sums, sizeof(unsigned long long) * 4));
  auto* hist = static_cast<uint32_t*>(c->cls_hist.p);
  auto* off = static_cast<unsigned long long*>(c->cls_off.p);
  auto* sums = static_cast<unsigned long long*>(o.sums.p);
  DDM_CUDA(cudaMemsetAsync(hist, 0, sizeof(uint32_t) * kClasses, s));
  if (cnt <= rank_sort_max(d)) {
    DDM_CUDA(launch_rank_sort(kRankClass, d, lo, hi, cnt, static_cast<uint32_t*>(o.vals[0].p), hist,
                              aos, nullptr, nullptr, c->st_dev, s));
  } else {
    DDM_CUDA(launch_validate_class(d, lo, hi, cnt, static_cast<uint32_t*>(o.vals[1].p), hist, aos,
                                   c->st_dev, c->sms, s));
    // (class, 24-bit lower bound)
    DDM_TRY(packed_pass(c, o, cnt, nullptr, true, 32, id_bits_of(cnt), cur, s));
  }
  ClassPlan plan{off, static_cast<int*>(o.bglog2.p), static_cast<unsigned long long*>(o.bgbase.p), {}};
  int tile_log2[DDM_MAX_DIMS] = {};
  for (int k = 1; k < d; ++k) {
    tile_log2[k] = seg_tile(cnt, d, k, c->str_shift, c->sms);
    plan.tile[k] = 1u << (tile_log2[k] ? tile_log2[k] : kSegTileLog2);
  }
  DDM_CUDA(launch_class_plan(hist, d, c->str_shift, plan, s));
  for (int k = 1; k < d; ++k) {
    const int* gl = plan.glog2 + k * kClasses;
    if (tile_log2[k]) {
      DDM_TRY(seg_pass(c, o, cnt, lo + (size_t)k * cnt, 0,
                       SegPlan{off, gl, plan.cbase + k * (kClasses + 1), kClasses}, tile_log2[k],
                       *cur, s));
      continue;
    }
    // Groups beyond a CTA: one radix sort over the whole set.
    DDM_TRY(ensure(c, c->inst_s, sizeof(uint32_t) * cnt));
    auto* inst = static_cast<uint32_t*>(c->inst_s.p);
    auto* ng = static_cast<uint32_t*>(o.bngroups.p);
    auto* gb = plan.cbase + k * (kClasses + 1);
    if (k == 1) DDM_CUDA(launch_fill_inst(off, kClasses, cnt, inst, c->sms, s));
    DDM_CUDA(launch_batch_groups(off, kClasses, gl, ng, s));
    DDM_CUDA(launch_scan(ng, kClasses, gb, sums, nullptr, s));
    // groups: at most one per class without re-sort plus cnt / 64
    DDM_TRY(resort_pass(
        c, o, cnt, (uint64_t)kClasses + cnt / 64 + 1, cur,
        [&](unsigned long long* keys, int id_bits) {
          return launch_rekey_batch(static_cast<const uint32_t*>(o.vals[*cur].p), lo + (size_t)k * cnt,
                                    cnt, inst, off, gl, gb, keys, id_bits, c->sms, s);
        },
        s));
  }
  return DDM_OK;
}

// `tree`: the d = 1 tree's order, else the updates'.  *gathered (updates): qe
// and qid are written too.
int order_set(ddm_ctx* c, OrderBufs& o, int d, const float* lo, const float* hi, uint32_t cnt, bool tree,
              float2* aos, int* cur, bool* gathered, cudaStream_t s) {
  *cur = 0;
  *gathered = false;
  DDM_TRY(ensure_sort(c, o, cnt));
  if (cnt <= rank_sort_max(d)) {
    *gathered = !tree && d == 1;  // no re-sorts follow
    DDM_CUDA(launch_rank_sort(tree ? kRankTree : kRankLocal, d, lo, hi, cnt,
                              static_cast<uint32_t*>(o.vals[0].p), nullptr, aos,
                              *gathered ? static_cast<float2*>(c->qe.p) : nullptr,
                              *gathered ? static_cast<uint32_t*>(c->qid.p) : nullptr, c->st_dev, s));
  } else {
    DDM_CUDA(launch_validate(d, lo, hi, cnt, static_cast<uint32_t*>(o.vals[1].p), tree, aos,
                             c->st_dev, c->sms, s));
    const int id_bits = id_bits_of(cnt);
    DDM_TRY(packed_pass(c, o, cnt, nullptr, true, tree ? 32 : 24, id_bits, cur, s, tree ? hi : nullptr));
    if (tree) {  // the words are in keys[0]; ties by upper bound
      auto* words = static_cast<unsigned long long*>(o.keys[0].p);
      auto* vals = static_cast<uint32_t*>(o.vals[0].p);
      auto* list = static_cast<uint2*>(o.vals[1].p);
      DDM_CUDA(launch_tie_order(words, cnt, id_bits, hi, vals, list, c->st_dev, c->sms, s));
      DDM_CUDA(launch_long_ties(words, cnt, id_bits, hi, vals, list,
                                static_cast<unsigned long long*>(o.keys[1].p), c->st_dev, c->sms, s));
    }
  }
  int glog2[DDM_MAX_DIMS];
  str_groups(cnt, d, glog2, c->str_shift);
  for (int k = 1; k < d; ++k) {
    if (!glog2[k]) continue;
    if (glog2[k] <= kSegTileLog2Max) {
      DDM_TRY(seg_pass(c, o, cnt, lo + (size_t)k * cnt, glog2[k], SegPlan{},
                       tile_for(cnt, std::max(glog2[k], kSegTileLog2Min), c->sms), *cur, s));
      continue;
    }
    DDM_TRY(resort_pass(
        c, o, cnt, ((uint64_t)(cnt - 1u) >> glog2[k]) + 1u, cur,
        [&](unsigned long long* keys, int id_bits) {
          return launch_rekey(static_cast<const uint32_t*>(o.vals[*cur].p), lo + (size_t)k * cnt, cnt,
                              glog2[k], keys, id_bits, c->sms, s);
        },
        s));
  }
  return DDM_OK;
}

// Validate S, sort it into tree order and build the tree (steps run on `s`,
// no host synchronisation).
int build_async(ddm_ctx* c, int d, const float* slo, const float* shi, uint32_t n, cudaStream_t s,
                const BatchSet* bs = nullptr) {
  Phase phase("ddm build");
  c->built = false;
  c->attached = false;
  c->swapped = false;
  if (!bs) c->bv = BatchView{};
  c->planned = false;
  TreeView t{};
  const uint32_t set_n = n;
  if (bs && bs->padded) n = bs->padded;  // positions of the tree; set_n of them hold extents
  t.d = d;
  t.n = n;
  if (n == 0) {
    c->tree = t;
    c->built = true;
    return DDM_OK;
  }
  tree_shape(n, &t.L, t.cnt, t.off, &t.total);
  DDM_TRY(ensure(c, c->e, sizeof(float2) * (size_t)d * n));
  DDM_TRY(ensure(c, c->sid, sizeof(uint32_t) * n));
  DDM_TRY(ensure(c, c->nodes, sizeof(float2) * (size_t)d * t.total));
  int cur = 0;
  bool gathered = false;
  OrderBufs& o = c->ob[0];
  float2* aos = aos_buffer(c, o, d, set_n);
  LeafMap map{};
  if (bs && bs->padded) map = LeafMap{bs->off, bs->leaf_off, bs->count};
  if (bs)
    DDM_TRY(order_set_batch(c, o, d, slo, shi, set_n, *bs, aos, &cur, s));
  else if (d >= 2)
    DDM_TRY(order_set_classes(c, o, d, slo, shi, n, aos, &cur, s));
  else
    DDM_TRY(order_set(c, o, d, slo, shi, n, true, aos, &cur, &gathered, s));
  t.e = static_cast<const float2*>(c->e.p);
  t.sid = static_cast<const uint32_t*>(c->sid.p);
  t.nodes = static_cast<const float2*>(c->nodes.p);
  // Rank tables of the leaves (d <= 3): 544 bytes per leaf and dimension.
  // Optional: without room for them the swapped leaf test compares instead.
  t.tab = nullptr;
  if (d <= 3 && c->tables_on &&
      ensure(c, c->tab, sizeof(uint32_t) * 2u * kRankSlot * (size_t)d * t.cnt[1]) == DDM_OK)
    t.tab = static_cast<const uint32_t*>(c->tab.p);
  DDM_CUDA(launch_build(t, set_n, map, static_cast<const uint32_t*>(o.vals[cur].p), slo, shi, aos,
                        static_cast<float2*>(c->e.p), static_cast<uint32_t*>(c->sid.p),
                        static_cast<float2*>(c->nodes.p), const_cast<uint32_t*>(t.tab),
                        c->st_dev, s));
  c->tree = t;
  c->built = true;
  return DDM_OK;
}

// Grid size argument of the packet kernels (they launch 8 CTAs per "SM").
int packet_sms(const ddm_ctx* c) {
  const int v = (int)((uint64_t)c->sms * c->ctas_per_sm / 8u);
  return v > 0 ? v : 1;
}

// Packets of the count pass (and of its records) covering positions [0, m).
uint32_t packets_of(const ddm_ctx* c, uint32_t m) {
  return (uint32_t)(((uint64_t)m + (1u << c->plan_qpp_log2) - 1u) >> c->plan_qpp_log2);
}

QueryView query_view(ddm_ctx* c) {
  QueryView q{};
  q.m = c->m;
  q.qe = static_cast<const float2*>(c->qe.p);
  q.qid = static_cast<const uint32_t*>(c->qid.p);
  q.list = nullptr;
  q.first = 0;
  q.nq = c->m;
  q.qpp_log2 = c->plan_qpp_log2;
  q.tmin = c->tmin;
  return q;
}

// Words before the scans' state in plan_state: the block counter, and whether
// a wait of the plan's scan ran out (kept until the next plan, since every
// later call on the plan uses its offsets).
constexpr size_t kPlanWords = 2;
uint32_t* plan_failed(const ddm_ctx* c) {
  return reinterpret_cast<uint32_t*>(static_cast<unsigned long long*>(c->plan_state.p) + 1);
}

int ensure_queries(ddm_ctx* c, int d, uint32_t m) {
  DDM_TRY(ensure(c, c->qe, sizeof(float2) * (size_t)d * (m ? m : 1)));
  return ensure(c, c->qid, sizeof(uint32_t) * (m ? m : 1));
}

// Validate U, sort it and gather the queries in plan order (qe, qid).
int order_updates(ddm_ctx* c, OrderBufs& o, int d, const float* ulo, const float* uhi, uint32_t m,
                  const BatchSet* bs, float2* aos, cudaStream_t s) {
  int cur = 0;
  bool gathered = false;
  if (bs)
    DDM_TRY(order_set_batch(c, o, d, ulo, uhi, m, *bs, aos, &cur, s));
  else
    DDM_TRY(order_set(c, o, d, ulo, uhi, m, false, aos, &cur, &gathered, s));
  if (gathered) return DDM_OK;
  DDM_CUDA(launch_gather(d, static_cast<const uint32_t*>(o.vals[cur].p), ulo, uhi, aos, m,
                         static_cast<float2*>(c->qe.p), static_cast<uint32_t*>(c->qid.p), c->sms, s));
  return DDM_OK;
}

// Validate U, sort it (unless `sorted`: order_updates has run), count per
// update, scan (no host synchronisation).
// `ordered`: the plan order's offsets too (the staged calls); the one-shot
// calls do not write by plan order, and a staged call after one of them has
// ready_ordered() compute them.
int plan_async(ddm_ctx* c, const float* ulo, const float* uhi, uint32_t m, uint32_t flags,
               bool record, bool ordered, cudaStream_t s, const BatchSet* bs = nullptr,
               bool sorted = false) {
  Phase phase("ddm plan");
  c->planned = false;
  const int d = c->tree.d;
  // Few updates: packets of fewer queries (down to four), until there are
  // sixteen warps' worth per SM (2,432 packets on 152 SMs).  A packet is one
  // warp's serial walk, and with fewer packets the chip idles: at 33,333
  // updates (d = 5, 1,042 packets of 32) a match took 5.3 ms, 3.55 with
  // packets of 8; at 31,627 (d = 2) a served plan and write 152 and 142 us; at
  // 30,011 374 and 352 us.  From twice as many packets the smaller ones cost
  // more walks than they save (served 157 us, d = 2 377 us).
  c->plan_qpp_log2 = c->qpp_log2;
  while (c->plan_qpp_log2 > 2 && packets_of(c, m) < (uint32_t)c->sms * 16u) --c->plan_qpp_log2;
  DDM_TRY(ensure(c, c->counts, sizeof(uint32_t) * (m ? m : 1)));
  DDM_TRY(ensure(c, c->counts_pos, sizeof(uint32_t) * (m ? m : 1)));
  DDM_TRY(ensure(c, c->offsets, sizeof(unsigned long long) * ((size_t)m + 1)));
  DDM_TRY(ensure(c, c->pos_offsets, sizeof(unsigned long long) * ((size_t)m + 1)));
  // tile sums of a range selection (write_async)
  DDM_TRY(ensure(c, c->sums, sizeof(unsigned long long) * ((size_t)m / kScanTile + 2)));
  DDM_TRY(ensure_queries(c, d, m));
  auto* counts = static_cast<uint32_t*>(c->counts.p);
  auto* counts_pos = static_cast<uint32_t*>(c->counts_pos.p);
  auto* offsets = static_cast<unsigned long long*>(c->offsets.p);
  auto* pos_offsets = static_cast<unsigned long long*>(c->pos_offsets.p);
  c->m = m;
  c->arena = RecordArena{};
  if (record && c->replay_on && m > 0 && c->tree.n > 0 && c->replay_budget > 0) {
    const uint32_t packets = packets_of(c, m);
    // bytes per block: records (ten bytes each) and header, count/owner/list entries
    const uint64_t per_block = (uint64_t)kRecWords * sizeof(uint32_t) + sizeof(uint32_t) +
                               sizeof(uint2) + sizeof(uint4);
    // Blocks the arena holds now, and what the latest recorded pass needed.
    uint64_t have = c->rec.cap / ((size_t)kRecWords * sizeof(uint32_t));
    have = std::min<uint64_t>(have, c->blk_count.cap / sizeof(uint32_t));
    have = std::min<uint64_t>(have, c->blk_own.cap / sizeof(uint2));
    have = std::min<uint64_t>(have, c->blk_list.cap / sizeof(uint4));
    const uint32_t hint_blocks = c->rec_hint[0], hint_packets = c->rec_hint[1],
                   hint_max = c->rec_hint[2];
    uint64_t want = have;
    if (have < (uint64_t)packets * kRecChains || (hint_packets && hint_blocks > hint_max)) {
      // No arena yet, not a block for each chain, or the last pass ran out of
      // it: size from that pass's blocks per packet (plus 1/8 and some
      // slack), else one per chain and an eighth of a block per packet.  An
      // arena that sufficed is kept as it is: the blocks per packet depend on
      // how densely the updates cover the space, so extrapolating them from
      // one plan to the next would reallocate for nothing.
      const uint64_t need =
          hint_packets ? (uint64_t)((double)hint_blocks / (double)hint_packets * 1.125 *
                                    (double)packets) + 64
                       : (uint64_t)kRecChains * packets + packets / 8 + 64;
      want = std::max(have, need);
    }
    const uint64_t cap_blocks = c->replay_budget / per_block;
    if (want > cap_blocks) want = cap_blocks;
    // no room for a first block of every chain: all from the counter
    const bool firsts = want >= (uint64_t)packets * kRecChains;
    if (want > 0xfffffff0ull) want = 0xfffffff0ull;
    if (want > 0 && ensure(c, c->rec, (size_t)want * kRecWords * sizeof(uint32_t)) == DDM_OK &&
        ensure(c, c->blk_own, (size_t)want * sizeof(uint2)) == DDM_OK &&
        ensure(c, c->blk_count, (size_t)want * sizeof(uint32_t)) == DDM_OK &&
        ensure(c, c->blk_list, (size_t)want * sizeof(uint4)) == DDM_OK &&
        ensure(c, c->pkt_nblk, (size_t)packets * sizeof(uint32_t)) == DDM_OK &&
        ensure(c, c->pkt_off, ((size_t)packets + 1) * sizeof(unsigned long long)) == DDM_OK) {
      c->arena.rec = static_cast<uint32_t*>(c->rec.p);
      c->arena.blk_own = static_cast<uint2*>(c->blk_own.p);
      c->arena.blk_count = static_cast<uint32_t*>(c->blk_count.p);
      c->arena.blk_list = static_cast<uint4*>(c->blk_list.p);
      c->arena.pkt_nblk = static_cast<uint32_t*>(c->pkt_nblk.p);
      c->arena.pkt_off = static_cast<unsigned long long*>(c->pkt_off.p);
      c->arena.chains = firsts ? packets * kRecChains : 0u;
      c->arena.max_blocks = (uint32_t)want;
    }
  }
  // Offsets by update id and, for a plan whose order will be written or read
  // out, by plan position and of the record entries in plan order.  The block
  // counter (two words), the plan's failure word (plan_failed) and the scans'
  // state are cleared by one memset.
  const uint32_t packets = packets_of(c, m);
  const ScanJob jobs[kMaxScanJobs] = {
      {counts, m, offsets, true},
      {counts_pos, m, pos_offsets, false},
      {c->arena.pkt_nblk, packets, c->arena.pkt_off, false}};
  const int njobs = !ordered ? 1 : c->arena.max_blocks ? 3 : 2;
  const size_t state_words = kPlanWords + scan_state_words(jobs, njobs);
  DDM_TRY(ensure(c, c->plan_state, sizeof(unsigned long long) * state_words));
  // what ready_ordered() needs, so that it never allocates
  DDM_TRY(ensure(c, c->order_state,
                 sizeof(unsigned long long) * scan_state_words(jobs + 1, c->arena.max_blocks ? 2 : 1)));
  auto* state = static_cast<unsigned long long*>(c->plan_state.p);
  DDM_CUDA(cudaMemsetAsync(state, 0, sizeof(unsigned long long) * state_words, s));
  if (c->arena.max_blocks) c->arena.blk_counter = reinterpret_cast<uint32_t*>(state);
  if (m > 0) {
    if (!sorted) DDM_TRY(order_updates(c, c->ob[0], d, ulo, uhi, m, bs, aos_buffer(c, c->ob[0], d, m), s));
    if (c->tree.n > 0) {
      DDM_CUDA(launch_count(c->tree, query_view(c), c->bv, flags, counts, counts_pos, c->arena,
                            c->st_dev->work, zeroed_work(c, 0), c->st_dev, packet_sms(c), s));
    } else {
      DDM_CUDA(cudaMemsetAsync(counts, 0, sizeof(uint32_t) * m, s));
      DDM_CUDA(cudaMemsetAsync(counts_pos, 0, sizeof(uint32_t) * m, s));
    }
  }
  const ScanHint hint{c->arena.max_blocks ? c->rec_hint : nullptr, c->arena.blk_counter,
                      c->arena.chains, packets, c->arena.max_blocks};
  DDM_CUDA(launch_scan_multi(jobs, njobs, state + kPlanWords, hint, plan_failed(c), c->st_dev, s));
  if (ordered && c->arena.max_blocks)
    DDM_CUDA(launch_block_list(c->arena, pos_offsets + m, c->sms, s));
  c->ordered = ordered;
  c->ulo = ulo;
  c->uhi = uhi;
  c->flags = flags;
  c->planned = true;
  return DDM_OK;
}

int walk_write(ddm_ctx* c, const QueryView& q, const WriteView& w, cudaStream_t s) {
  DDM_CUDA(launch_write(c->tree, q, c->bv, c->flags, w, c->arena, c->st_dev->work, c->st_dev,
                        packet_sms(c), s));
  return DDM_OK;
}

// The walking write pass behind a replay: it does nothing when the records
// are complete, which is the rule, so a call that synchronises holds it back
// until it has read the status; the others launch it.
int walk_or_hold(ddm_ctx* c, const QueryView& q, const WriteView& w, bool synced, cudaStream_t s) {
  if (!synced || !c->arena.max_blocks) return walk_write(c, q, w, s);
  c->walk_pending = true;
  c->walk_q = q;
  c->walk_w = w;
  return DDM_OK;
}

// The plan order's offsets and record entries, for a staged call after a
// one-shot call's plan (a plan made for staged calls has them).  Under capture
// (ddm_plan_order alone) the offsets are always recorded, from the counts that
// every plan leaves: the graph may run again after a plan of the other kind.
int ready_ordered(ddm_ctx* c, cudaStream_t s) {
  if (c->ordered && !c->capturing) return DDM_OK;
  const uint32_t packets = packets_of(c, c->m);
  const ScanJob jobs[2] = {
      {static_cast<uint32_t*>(c->counts_pos.p), c->m,
       static_cast<unsigned long long*>(c->pos_offsets.p), false},
      {c->arena.pkt_nblk, packets, c->arena.pkt_off, false}};
  const bool list = c->arena.max_blocks && !c->capturing;
  const int njobs = list ? 2 : 1;
  const size_t words = scan_state_words(jobs, njobs);
  DDM_TRY(ensure(c, c->order_state, sizeof(unsigned long long) * words));  // done by the plan
  auto* state = static_cast<unsigned long long*>(c->order_state.p);
  DDM_CUDA(cudaMemsetAsync(state, 0, sizeof(unsigned long long) * words, s));
  DDM_CUDA(launch_scan_multi(jobs, njobs, state, ScanHint{}, plan_failed(c), c->st_dev, s));
  if (list) DDM_CUDA(launch_block_list(c->arena, jobs[0].offsets + c->m, c->sms, s));
  if (!c->capturing) c->ordered = true;
  return DDM_OK;
}

// Write pass for updates with ids in [begin, end), laid out by update id.
// Global update ids (update-id base + local id) must fit 32 bits.
bool base_fits(const ddm_ctx* c) { return (uint64_t)c->upd_base + c->m <= (1ull << 32); }

int write_async(ddm_ctx* c, uint32_t begin, uint32_t end, ddm_pair* pairs, uint64_t capacity,
                bool synced, cudaStream_t s, const uint32_t* qids = nullptr) {
  Phase phase("ddm write");
  if (!qids && !c->swapped && !c->bv.count && !base_fits(c)) return DDM_ERR_ARG;
  if (end > begin && c->tree.n > 0) {
    QueryView q = query_view(c);
    if (begin != 0 || end != c->m) {
      DDM_TRY(ensure(c, c->sel_offs, sizeof(unsigned long long) * ((size_t)c->m + 1)));
      DDM_TRY(ensure(c, c->sel_list, sizeof(uint32_t) * c->m));
      DDM_CUDA(launch_select(q.qid, c->m, begin, end, static_cast<uint32_t*>(c->counts.p),
                             static_cast<unsigned long long*>(c->sel_offs.p),
                             static_cast<unsigned long long*>(c->sums.p),
                             static_cast<uint32_t*>(c->sel_list.p), c->st_dev, s));
      q.list = static_cast<const uint32_t*>(c->sel_list.p);
      q.nq = end - begin;
    }
    WriteView w{};
    w.start = static_cast<const unsigned long long*>(c->offsets.p);
    w.by_pos = false;
    w.swap = c->swapped;
    w.qids = qids;
    w.qbase = (c->swapped || c->bv.count) ? 0u : c->upd_base;
    w.b_idx = begin;
    w.e_idx = end;
    w.pairs = pairs;
    w.capacity = capacity;
    w.failed = plan_failed(c);
    if (c->arena.max_blocks) {
      const bool full = begin == 0 && end == c->m;
      RecordArena ra = c->arena;
      ra.blk_list = nullptr;
      DDM_CUDA(launch_replay(c->tree, query_view(c), c->bv, ra, w, 0, packets_of(c, c->m), 0, c->m,
                             !full, begin, end, c->st_dev->work + 1, zeroed_work(c, 1), c->st_dev,
                             c->sms, s));
    }
    DDM_TRY(walk_or_hold(c, q, w, synced, s));
  } else {
    DDM_CUDA(cudaMemsetAsync(&c->st_dev->K, 0, sizeof(unsigned long long), s));
  }
  return DDM_OK;
}

// Write pass for the plan positions [pb, pe), laid out in plan order.
int write_ordered_async(ddm_ctx* c, uint32_t pb, uint32_t pe, ddm_pair* pairs, uint64_t capacity,
                        cudaStream_t s, uint32_t* ids = nullptr) {
  Phase phase("ddm write ordered");
  if (!ids && !base_fits(c)) return DDM_ERR_ARG;
  DDM_TRY(ready_ordered(c, s));
  if (pe > pb && c->tree.n > 0) {
    QueryView q = query_view(c);
    q.first = pb;
    q.nq = pe - pb;
    WriteView w{};
    w.start = static_cast<const unsigned long long*>(c->pos_offsets.p);
    w.by_pos = true;
    w.qbase = c->upd_base;
    w.b_idx = pb;
    w.e_idx = pe;
    w.pairs = pairs;
    w.ids = ids;
    w.capacity = capacity;
    w.failed = plan_failed(c);
    if (c->arena.max_blocks)
      DDM_CUDA(launch_replay(c->tree, q, c->bv, c->arena, w, pb >> c->plan_qpp_log2, packets_of(c, pe), pb, pe, false, 0, 0,
                             c->st_dev->work + 1, zeroed_work(c, 1), c->st_dev, c->sms, s));
    DDM_TRY(walk_or_hold(c, q, w, true, s));
  } else {
    DDM_CUDA(cudaMemsetAsync(&c->st_dev->K, 0, sizeof(unsigned long long), s));
  }
  return DDM_OK;
}

// Build and plan of a one-shot call: the updates are ordered on the context's
// side stream while the tree is built -- both are chains of short launches
// that leave most of the chip idle.  The side stream starts after the work
// enqueued so far and the caller's stream goes on after it, so nothing of the
// call is left on it.  Its workspace is allocated before, on the caller's
// stream; without room for it the two run one after the other.  Measured, one
// match: 64 + 64 extents (d = 1) 99 -> 89 us, 5,000 + 5,000 124 -> 109 us, 5e5
// + 5e5 388 -> 356 us (d = 1) and 328 -> 272 us (d = 2), 2.5e7 + 2.5e7 8.15 ->
// 7.94 ms; 256 batched instances in a graph 289 -> 198 us.
int build_and_plan(ddm_ctx* c, int d, const float* slo, const float* shi, uint32_t n,
                   const float* ulo, const float* uhi, uint32_t m, uint32_t flags, bool record,
                   bool swap, cudaStream_t s, const BatchSet* bs_s = nullptr,
                   const BatchSet* bs_u = nullptr, const BatchView* bv = nullptr) {
  OrderBufs& o = c->ob[1];
  auto sequel = [&](bool sorted) {
    c->swapped = swap;
    if (bv) c->bv = *bv;
    return plan_async(c, ulo, uhi, m, flags, record, false, s, bs_u, sorted);
  };
  if (m > 0 && n > 0) {
    c->side_busy = true;
    int rc = bs_u ? ensure_batch(c, o, d, m, bs_u->count) : ensure_sort(c, o, m);
    if (rc == DDM_OK) rc = ensure_queries(c, d, m);
    if (rc == DDM_OK) {
      float2* aos = aos_buffer(c, o, d, m);
      DDM_CUDA(cudaEventRecord(c->fork, s));
      rc = build_async(c, d, slo, shi, n, s, bs_s);
      if (rc == DDM_OK) {
        c->side_recorded |= c->capturing;
        DDM_CUDA(cudaStreamWaitEvent(c->side, c->fork, 0));
        rc = order_updates(c, o, d, ulo, uhi, m, bs_u, aos, c->side);
        DDM_CUDA(cudaEventRecord(c->joined, c->side));  // also after an error: joined before returning
        DDM_CUDA(cudaStreamWaitEvent(s, c->joined, 0));
        c->side_busy = false;
        if (rc == DDM_OK) rc = sequel(true);
      }
    }
    c->side_busy = false;
    if (rc != DDM_ERR_NOMEM) return rc;
    if (!c->capturing) release_side(c);  // a recorded call neither allocates nor frees
  }
  DDM_TRY(build_async(c, d, slo, shi, n, s, bs_s));
  return sequel(false);
}

int reset_status(ddm_ctx* c, cudaStream_t s) {
  DDM_CUDA(cudaMemsetAsync(c->st_dev, 0, sizeof(Status), s));
  c->work_zeroed[0] = c->work_zeroed[1] = true;
  return DDM_OK;
}

}  // namespace

extern "C" {

const char* ddm_strerror(int code) {
  switch (code) {
    case DDM_OK: return "success";
    case DDM_ERR_ARG: return "invalid argument";
    case DDM_ERR_EXTENT: return "invalid extent (lo > hi or NaN)";
    case DDM_ERR_CAPACITY: return "pair buffer too small";
    case DDM_ERR_NOMEM: return "device memory allocation failed";
    case DDM_ERR_CUDA: return "CUDA error";
    case DDM_ERR_TIMEOUT: return "bounded device wait timed out";
    case DDM_ERR_STATE: return "tree or plan missing";
    case DDM_ERR_INTERNAL: return "an index failed its bounds check (checked build)";
    default: return "unknown error";
  }
}

int ddm_create(ddm_ctx** out, int device) {
  if (!out) return DDM_ERR_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
    cudaGetLastError();
    return DDM_ERR_CUDA;
  }
  DeviceGuard g(device);
  if (!g.ok()) return DDM_ERR_CUDA;
  ddm_ctx* c = new (std::nothrow) ddm_ctx();
  if (!c) return DDM_ERR_NOMEM;
  c->device = device;
  {
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess) c->replay_budget = total_b / 4;
    cudaGetLastError();
  }
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = device;
  const uint64_t keep_all = ~0ull;
  if (cudaMemPoolCreate(&c->pool, &props) != cudaSuccess ||
      cudaMemPoolSetAttribute(c->pool, cudaMemPoolAttrReleaseThreshold, (void*)&keep_all) !=
          cudaSuccess ||
      cudaEventCreateWithFlags(&c->done, cudaEventDisableTiming) != cudaSuccess ||
      cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->fork, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->joined, cudaEventDisableTiming) != cudaSuccess ||
      cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
      cudaMalloc(&c->st_dev, sizeof(Status)) != cudaSuccess ||
      ready_group_table() != cudaSuccess ||
      cudaMallocHost(&c->st_host, sizeof(Status)) != cudaSuccess ||
      cudaMallocHost((void**)&c->rec_hint, 3 * sizeof(uint32_t)) != cudaSuccess) {
    cudaGetLastError();
    ddm_destroy(c);
    return DDM_ERR_NOMEM;
  }
  c->rec_hint[0] = c->rec_hint[1] = c->rec_hint[2] = 0;
  *out = c;
  return DDM_OK;
}

int ddm_destroy(ddm_ctx* c) {
  if (!c) return DDM_OK;
  DeviceGuard g(c->device);
  cudaDeviceSynchronize();
  for (OrderBufs& o : c->ob) {
    for (DevBuf* b : o.all) release(*b);
    release(o.sums);
  }
  for (DevBuf* b : {&c->e, &c->sid, &c->nodes, &c->tab, &c->qe, &c->qid, &c->counts,
                    &c->counts_pos, &c->offsets, &c->pos_offsets, &c->sums,
                    &c->sel_offs, &c->sel_list, &c->rec, &c->blk_own, &c->blk_count,
                    &c->pkt_nblk, &c->pkt_off,
                    &c->blk_list, &c->plan_state, &c->order_state, &c->inst_s, &c->inst_u,
                    &c->leaf_off,
                    &c->cls_hist, &c->cls_off, &c->probe})
    release(*b);
  cudaDeviceSynchronize();  // the stream-ordered frees above have run
  if (c->pool) cudaMemPoolDestroy(c->pool);
  if (c->done) cudaEventDestroy(c->done);
  if (c->fork) cudaEventDestroy(c->fork);
  if (c->joined) cudaEventDestroy(c->joined);
  if (c->side) cudaStreamDestroy(c->side);
  if (c->st_dev) cudaFree(c->st_dev);
  if (c->st_host) cudaFreeHost(c->st_host);
  if (c->rec_hint) cudaFreeHost((void*)c->rec_hint);
  delete c;
  return DDM_OK;
}

int ddm_set_replay_budget(ddm_ctx* c, uint64_t bytes) {
  if (!c) return DDM_ERR_ARG;
  c->replay_budget = bytes;
  return DDM_OK;
}

int ddm_set_tuning(ddm_ctx* c, int str_shift, uint32_t ctas_per_sm, uint32_t replay) {
  if (!c || str_shift < -4 || str_shift > 4 || ctas_per_sm < 1 || ctas_per_sm > 32)
    return DDM_ERR_ARG;
  c->str_shift = str_shift;
  c->ctas_per_sm = ctas_per_sm;
  c->replay_on = replay != 0;
  return DDM_OK;
}

int ddm_set_tiling(ddm_ctx* c, uint32_t queries_per_packet, uint32_t swap_min) {
  if (!c || (queries_per_packet != 16 && queries_per_packet != 32) || swap_min < 1 ||
      swap_min > 33)
    return DDM_ERR_ARG;
  const uint32_t lg = queries_per_packet == 16 ? 4u : 5u;
  if (lg != c->qpp_log2) c->planned = false;  // the plan's records use its packets
  c->qpp_log2 = lg;
  c->tmin = swap_min;
  return DDM_OK;
}

int ddm_set_update_id_base(ddm_ctx* c, uint32_t base) {
  if (!c) return DDM_ERR_ARG;
  c->upd_base = base;
  return DDM_OK;
}

int ddm_debug_wait_timeout(ddm_ctx* c, uint32_t polls, void* stream) {
  if (!c || polls == 0 || polls > (1u << 22)) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(ensure(c, c->probe, sizeof(uint32_t)));
  DDM_CUDA(cudaMemsetAsync(c->probe.p, 0, sizeof(uint32_t), s));
  DDM_TRY(reset_status(c, s));
  DDM_CUDA(launch_debug_wait(static_cast<const uint32_t*>(c->probe.p), polls, c->st_dev, s));
  DDM_TRY(sync_status(c, s));
  return status_code(*c->st_host);
}

int ddm_debug_scan_timeout(ddm_ctx* c, uint32_t polls, void* stream) {
  if (!c || polls == 0 || polls > (1u << 22)) return DDM_ERR_ARG;
  if (!c->planned) return DDM_ERR_STATE;
  const ScanJob job{static_cast<uint32_t*>(c->counts.p), c->m,
                    static_cast<unsigned long long*>(c->offsets.p), true};
  if (c->m <= (uint32_t)kScanTile) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(ensure(c, c->probe, sizeof(unsigned long long) * scan_state_words(&job, 1)));
  DDM_TRY(reset_status(c, s));
  DDM_CUDA(launch_debug_scan(job, static_cast<unsigned long long*>(c->probe.p), polls, plan_failed(c),
                             c->st_dev, s));
  DDM_TRY(sync_status(c, s));
  return status_code(*c->st_host);
}

uint64_t ddm_debug_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

int ddm_debug_set_alloc_limit(ddm_ctx* c, uint64_t bytes) {
  if (!c) return DDM_ERR_ARG;
  c->alloc_limit = bytes;
  return DDM_OK;
}

int ddm_build(ddm_ctx* c, int d, const float* slo, const float* shi, uint32_t n, void* stream) {
  if (!c || d < 1 || d > DDM_MAX_DIMS || !set_ok(d, slo, shi, n)) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(reset_status(c, s));
  DDM_TRY(build_async(c, d, slo, shi, n, s));
  DDM_TRY(sync_status(c, s));
  const int rc = status_code(*c->st_host);
  if (rc != DDM_OK) c->built = false;
  return rc;
}

int ddm_plan(ddm_ctx* c, const float* ulo, const float* uhi, uint32_t m, uint32_t flags,
             uint64_t* offsets, uint64_t* k_out, void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->built) return DDM_ERR_STATE;
  if (!set_ok(c->tree.d, ulo, uhi, m) || (flags & ~DDM_OPEN)) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(reset_status(c, s));
  DDM_TRY(plan_async(c, ulo, uhi, m, flags, true, true, s));
  if (offsets)
    DDM_CUDA(cudaMemcpyAsync(offsets, c->offsets.p, sizeof(unsigned long long) * ((size_t)m + 1),
                             cudaMemcpyDeviceToDevice, s));
  DDM_TRY(sync_status(c, s));
  c->last_tests = c->st_host->tests;
  if (k_out) *k_out = c->st_host->K;
  const int rc = status_code(*c->st_host);
  if (rc != DDM_OK) c->planned = false;
  return rc;
}

int ddm_write(ddm_ctx* c, uint32_t begin, uint32_t end, ddm_pair* pairs, uint64_t capacity,
              uint64_t* k_out, void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->planned) return DDM_ERR_STATE;
  if (begin > end || end > c->m || (end > begin && !pairs)) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(reset_status(c, s));
  DDM_TRY(write_async(c, begin, end, pairs, capacity, true, s));
  DDM_TRY(sync_status(c, s));
  if (k_out) *k_out = c->st_host->K;
  return status_code(*c->st_host);
}

int ddm_chunk_end(ddm_ctx* c, uint32_t begin, uint64_t capacity, uint32_t* upd_end, void* stream) {
  if (!c || !upd_end) return DDM_ERR_ARG;
  if (!c->planned) return DDM_ERR_STATE;
  if (begin > c->m) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_CUDA(launch_chunk_end(static_cast<const unsigned long long*>(c->offsets.p), c->m, begin,
                            capacity, plan_failed(c), c->st_dev, s));
  DDM_TRY(sync_status(c, s));
  if (c->st_host->aux == kPlanFailed) return DDM_ERR_TIMEOUT;
  *upd_end = (uint32_t)c->st_host->aux;
  if (*upd_end == begin && begin < c->m) return DDM_ERR_CAPACITY;
  return DDM_OK;
}

int ddm_plan_async(ddm_ctx* c, const float* ulo, const float* uhi, uint32_t m, uint32_t flags,
                   void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->built || c->bv.count) return DDM_ERR_STATE;
  if (!set_ok(c->tree.d, ulo, uhi, m) || (flags & ~DDM_OPEN)) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(reset_status(c, s));
  DDM_TRY(plan_async(c, ulo, uhi, m, flags, true, true, s));
  return DDM_OK;
}

int ddm_write_async(ddm_ctx* c, uint32_t begin, uint32_t end, ddm_pair* pairs, uint64_t capacity,
                    uint64_t* k_dev, uint32_t* err_dev, void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->planned) return DDM_ERR_STATE;
  if (begin > end || end > c->m || (end > begin && !pairs && capacity > 0)) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  // keep the plan's error bits; the write sets K (and the capacity bit)
  DDM_TRY(write_async(c, begin, end, pairs, capacity, false, s));
  if (k_dev)
    DDM_CUDA(cudaMemcpyAsync(k_dev, &c->st_dev->K, sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
  if (err_dev)
    DDM_CUDA(cudaMemcpyAsync(err_dev, &c->st_dev->err, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
  return DDM_OK;
}

int ddm_plan_stats(ddm_ctx* c, uint64_t* leaf_tests) {
  if (!c || !leaf_tests) return DDM_ERR_ARG;
  *leaf_tests = c->last_tests;
  return DDM_OK;
}

int ddm_match_moved(ddm_ctx* c, const float* lo, const float* hi, uint32_t k, const uint32_t* ids,
                    uint32_t flags, ddm_pair* pairs, uint64_t capacity, uint64_t* k_out,
                    void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->built || c->bv.count) return DDM_ERR_STATE;
  if (!set_ok(c->tree.d, lo, hi, k) || (flags & ~(DDM_OPEN | DDM_SWAP_ROLES)) ||
      (k > 0 && !pairs && capacity > 0))
    return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(reset_status(c, s));
  DDM_TRY(plan_async(c, lo, hi, k, flags & DDM_OPEN, true, false, s));
  const bool was = c->swapped;
  c->swapped = (flags & DDM_SWAP_ROLES) != 0;
  const int wrc = write_async(c, 0, k, pairs, capacity, true, s, ids);
  c->swapped = was;
  DDM_TRY(wrc);
  DDM_TRY(sync_status(c, s));
  c->last_tests = c->st_host->tests;
  if (k_out) *k_out = c->st_host->K;
  const int rc = status_code(*c->st_host);
  if (rc != DDM_OK) c->planned = false;
  return rc;
}

int ddm_pair_offsets_async(ddm_ctx* c, const uint64_t* upd_off, uint32_t count, uint64_t* pair_off,
                           void* stream) {
  if (!c || !upd_off || !pair_off) return DDM_ERR_ARG;
  if (!c->planned) return DDM_ERR_STATE;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  StreamUse use(c, static_cast<cudaStream_t>(stream));
  DDM_CUDA(launch_gather_offsets(static_cast<const unsigned long long*>(c->offsets.p), c->m,
                                 reinterpret_cast<const unsigned long long*>(upd_off), count,
                                 reinterpret_cast<unsigned long long*>(pair_off),
                                 static_cast<cudaStream_t>(stream)));
  return DDM_OK;
}

int ddm_write_ordered(ddm_ctx* c, uint32_t pos_begin, uint32_t pos_end, ddm_pair* pairs,
                      uint64_t capacity, uint64_t* k_out, void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->planned) return DDM_ERR_STATE;
  if (pos_begin > pos_end || pos_end > c->m || (pos_end > pos_begin && !pairs)) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(reset_status(c, s));
  DDM_TRY(write_ordered_async(c, pos_begin, pos_end, pairs, capacity, s));
  DDM_TRY(sync_status(c, s));
  if (k_out) *k_out = c->st_host->K;
  return status_code(*c->st_host);
}

int ddm_write_ordered_ids(ddm_ctx* c, uint32_t pos_begin, uint32_t pos_end, uint32_t* sub_ids,
                          uint64_t capacity, uint64_t* k_out, void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->planned) return DDM_ERR_STATE;
  if (pos_begin > pos_end || pos_end > c->m || (pos_end > pos_begin && !sub_ids)) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(reset_status(c, s));
  DDM_TRY(write_ordered_async(c, pos_begin, pos_end, nullptr, capacity, s, sub_ids));
  DDM_TRY(sync_status(c, s));
  if (k_out) *k_out = c->st_host->K;
  return status_code(*c->st_host);
}

int ddm_chunk_end_ordered(ddm_ctx* c, uint32_t pos_begin, uint64_t capacity, uint32_t* pos_end,
                          void* stream) {
  if (!c || !pos_end) return DDM_ERR_ARG;
  if (!c->planned) return DDM_ERR_STATE;
  if (pos_begin > c->m) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(ready_ordered(c, s));
  DDM_CUDA(launch_chunk_end(static_cast<const unsigned long long*>(c->pos_offsets.p), c->m,
                            pos_begin, capacity, plan_failed(c), c->st_dev, s));
  DDM_TRY(sync_status(c, s));
  if (c->st_host->aux == kPlanFailed) return DDM_ERR_TIMEOUT;
  *pos_end = (uint32_t)c->st_host->aux;
  if (*pos_end == pos_begin && pos_begin < c->m) return DDM_ERR_CAPACITY;
  return DDM_OK;
}

int ddm_plan_order(ddm_ctx* c, uint32_t* order, uint64_t* order_offsets, void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->planned) return DDM_ERR_STATE;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  if (order && c->m)
    DDM_CUDA(cudaMemcpyAsync(order, c->qid.p, sizeof(uint32_t) * c->m, cudaMemcpyDeviceToDevice, s));
  if (order_offsets) DDM_TRY(ready_ordered(c, s));
  if (order_offsets)
    DDM_CUDA(cudaMemcpyAsync(order_offsets, c->pos_offsets.p,
                             sizeof(unsigned long long) * ((size_t)c->m + 1),
                             cudaMemcpyDeviceToDevice, s));
  return DDM_OK;
}

static int match_impl(ddm_ctx* c, int d, const float* ulo, const float* uhi, uint32_t m,
                      const float* slo, const float* shi, uint32_t n, uint32_t begin, uint32_t end,
                      uint32_t flags, ddm_pair* pairs, uint64_t capacity, uint64_t* k_out,
                      void* stream, bool write) {
  if (!c || d < 1 || d > DDM_MAX_DIMS || !set_ok(d, ulo, uhi, m) || !set_ok(d, slo, shi, n) ||
      (flags & ~(DDM_OPEN | DDM_SWAP_ROLES)) || begin > end || end > m)
    return DDM_ERR_ARG;
  const bool swap = (flags & DDM_SWAP_ROLES) != 0;
  if (swap && (begin != 0 || end != m)) return DDM_ERR_ARG;
  if (write && end > begin && !pairs && capacity > 0) return DDM_ERR_ARG;
  if (swap) {  // tree over the updates, one query per subscription
    std::swap(ulo, slo);
    std::swap(uhi, shi);
    std::swap(m, n);
    begin = 0;
    end = m;
  }
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(reset_status(c, s));
  DDM_TRY(build_and_plan(c, d, slo, shi, n, ulo, uhi, m, flags & DDM_OPEN, write, swap, s));
  if (write) DDM_TRY(write_async(c, begin, end, pairs, capacity, true, s));
  DDM_TRY(sync_status(c, s));
  c->last_tests = c->st_host->tests;
  if (k_out) *k_out = c->st_host->K;
  const int rc = status_code(*c->st_host);
  // a swapped problem's tree and plan are not the caller's sets: no staged use
  if (swap || rc == DDM_ERR_EXTENT || rc == DDM_ERR_TIMEOUT) c->built = c->planned = false;
  return rc;
}

int ddm_count(ddm_ctx* c, int d, const float* ulo, const float* uhi, uint32_t m, const float* slo,
              const float* shi, uint32_t n, uint32_t flags, uint64_t* k_out, void* stream) {
  return match_impl(c, d, ulo, uhi, m, slo, shi, n, 0, m, flags, nullptr, 0, k_out, stream, false);
}

int ddm_match(ddm_ctx* c, int d, const float* ulo, const float* uhi, uint32_t m, const float* slo,
              const float* shi, uint32_t n, uint32_t flags, ddm_pair* pairs, uint64_t capacity,
              uint64_t* k_out, void* stream) {
  return match_impl(c, d, ulo, uhi, m, slo, shi, n, 0, m, flags, pairs, capacity, k_out, stream,
                    true);
}

int ddm_match_range(ddm_ctx* c, int d, const float* ulo, const float* uhi, uint32_t m,
                    const float* slo, const float* shi, uint32_t n, uint32_t begin, uint32_t end,
                    uint32_t flags, ddm_pair* pairs, uint64_t capacity, uint64_t* k_out,
                    void* stream) {
  return match_impl(c, d, ulo, uhi, m, slo, shi, n, begin, end, flags, pairs, capacity, k_out,
                    stream, true);
}

static int batch_impl(ddm_ctx* c, int d, uint32_t count, const float* ulo, const float* uhi,
                      const uint64_t* upd_off, uint32_t m, const float* slo, const float* shi,
                      const uint64_t* sub_off, uint32_t n, uint32_t flags, ddm_pair* pairs,
                      uint64_t capacity, uint64_t* pair_off, uint64_t* k_out, uint64_t* k_dev,
                      uint32_t* err_dev, void* stream, bool sync) {
  if (!c || d < 1 || d > DDM_MAX_DIMS || count == 0 || !upd_off || !sub_off || !set_ok(d, ulo, uhi, m) ||
      !set_ok(d, slo, shi, n) || (flags & ~DDM_OPEN) || (!pairs && capacity > 0))
    return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(ensure(c, c->inst_s, sizeof(uint32_t) * (n ? n : 1)));
  DDM_TRY(ensure(c, c->inst_u, sizeof(uint32_t) * (m ? m : 1)));
  DDM_TRY(reset_status(c, s));
  const auto* uoff = reinterpret_cast<const unsigned long long*>(upd_off);
  const auto* soff = reinterpret_cast<const unsigned long long*>(sub_off);
  // Whole leaves per instance when that adds at most a quarter of positions.
  const uint64_t positions = ((uint64_t)n + 31ull * count + 31u) / 32u * 32u;
  const uint32_t padded = n >= 128ull * count && positions <= DDM_MAX_EXTENTS ? (uint32_t)positions : 0u;
  DDM_TRY(ensure(c, c->leaf_off, sizeof(unsigned long long) * ((size_t)count + 1)));
  auto* leaf_off = padded ? static_cast<unsigned long long*>(c->leaf_off.p) : nullptr;
  BatchSet bs_s{soff, count, static_cast<uint32_t*>(c->inst_s.p), padded, leaf_off};
  BatchSet bs_u{uoff, count, static_cast<uint32_t*>(c->inst_u.p), 0u, nullptr};
  const BatchView bv{count, uoff, soff, static_cast<const uint32_t*>(c->inst_u.p), leaf_off};
  DDM_TRY(build_and_plan(c, d, slo, shi, n, ulo, uhi, m, flags, true, false, s, &bs_s, &bs_u, &bv));
  // a k_dev or pair_off copy is enqueued behind the write: only a plain
  // synchronising call can hold the walking pass back
  DDM_TRY(write_async(c, 0, m, pairs, capacity, sync && !k_dev && !err_dev, s));
  if (pair_off && m > 0)
    DDM_CUDA(launch_gather_offsets(static_cast<const unsigned long long*>(c->offsets.p), m, uoff,
                                   count, reinterpret_cast<unsigned long long*>(pair_off), s));
  else if (pair_off)
    DDM_CUDA(cudaMemsetAsync(pair_off, 0, sizeof(uint64_t) * ((size_t)count + 1), s));
  if (k_dev)
    DDM_CUDA(cudaMemcpyAsync(k_dev, &c->st_dev->K, sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
  if (err_dev)
    DDM_CUDA(cudaMemcpyAsync(err_dev, &c->st_dev->err, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
  // The tree and plan hold a batch: the single-problem staged calls must not use them.
  c->built = c->planned = false;
  if (!sync) return DDM_OK;
  DDM_TRY(sync_status(c, s));
  c->last_tests = c->st_host->tests;
  if (k_out) *k_out = c->st_host->K;
  return status_code(*c->st_host);
}

int ddm_batch_match(ddm_ctx* c, int d, uint32_t count, const float* upd_lo, const float* upd_hi,
                    const uint64_t* upd_off, uint32_t m_total, const float* sub_lo,
                    const float* sub_hi, const uint64_t* sub_off, uint32_t n_total, uint32_t flags,
                    ddm_pair* pairs, uint64_t capacity, uint64_t* pair_off, uint64_t* k_out,
                    void* stream) {
  return batch_impl(c, d, count, upd_lo, upd_hi, upd_off, m_total, sub_lo, sub_hi, sub_off,
                    n_total, flags, pairs, capacity, pair_off, k_out, nullptr, nullptr, stream, true);
}

int ddm_batch_match_async(ddm_ctx* c, int d, uint32_t count, const float* upd_lo,
                          const float* upd_hi, const uint64_t* upd_off, uint32_t m_total,
                          const float* sub_lo, const float* sub_hi, const uint64_t* sub_off,
                          uint32_t n_total, uint32_t flags, ddm_pair* pairs, uint64_t capacity,
                          uint64_t* pair_off, uint64_t* k_dev, uint32_t* err_dev, void* stream) {
  return batch_impl(c, d, count, upd_lo, upd_hi, upd_off, m_total, sub_lo, sub_hi, sub_off,
                    n_total, flags, pairs, capacity, pair_off, nullptr, k_dev, err_dev, stream,
                    false);
}

int ddm_refit(ddm_ctx* c, const float* sub_lo, const float* sub_hi, void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->built || c->attached || c->bv.count) return DDM_ERR_STATE;
  if (c->tree.n > 0 && (!sub_lo || !sub_hi)) return DDM_ERR_ARG;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  DDM_TRY(reset_status(c, s));
  c->planned = false;
  Phase phase("ddm refit");
  if (c->tree.n > 0) {
    float2* aos = aos_buffer(c, c->ob[0], c->tree.d, c->tree.n);
    DDM_CUDA(launch_validate(c->tree.d, sub_lo, sub_hi, c->tree.n, nullptr, false, aos, c->st_dev, c->sms, s));
    // Same order, new coordinates: gather through the tree's own id column and
    // recompute every node's per-dimension (minlower, maxupper).
    DDM_CUDA(launch_build(c->tree, c->tree.n, LeafMap{}, c->tree.sid, sub_lo, sub_hi, aos, static_cast<float2*>(c->e.p),
                          static_cast<uint32_t*>(c->sid.p), static_cast<float2*>(c->nodes.p),
                          const_cast<uint32_t*>(c->tree.tab), c->st_dev, s));
  }
  DDM_TRY(sync_status(c, s));
  const int rc = status_code(*c->st_host);
  if (rc != DDM_OK) c->built = false;
  return rc;
}

int ddm_attach(ddm_ctx* c, const ddm_ctx* src) {
  if (!c || !src || c == src) return DDM_ERR_ARG;
  if (!src->built || src->bv.count) return DDM_ERR_STATE;
  if (c->device != src->device) return DDM_ERR_ARG;
  c->tree = src->tree;
  c->bv = BatchView{};
  c->built = true;
  c->attached = true;
  c->planned = false;
  return DDM_OK;
}

int ddm_tree_shape(ddm_ctx* c, int* levels, uint32_t* counts, uint32_t* total) {
  if (!c) return DDM_ERR_ARG;
  if (!c->built) return DDM_ERR_STATE;
  const TreeView& t = c->tree;
  const int L = t.n ? t.L : 0;
  if (levels) *levels = L;
  uint32_t tot = 0;
  for (int l = 1; l <= L; ++l) {
    if (counts) counts[l - 1] = t.cnt[l];
    tot += t.cnt[l];
  }
  if (total) *total = tot;
  return DDM_OK;
}

int ddm_tree_export(ddm_ctx* c, uint32_t* order, float* node_lo, float* node_hi, void* stream) {
  if (!c) return DDM_ERR_ARG;
  if (!c->built) return DDM_ERR_STATE;
  if (c->tree.n == 0) return DDM_OK;
  DeviceGuard g(c->device);
  if (!g.ok()) return DDM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  StreamUse use(c, s);
  if (order)
    DDM_CUDA(cudaMemcpyAsync(order, c->sid.p, sizeof(uint32_t) * c->tree.n,
                             cudaMemcpyDeviceToDevice, s));
  DDM_CUDA(launch_export_nodes(c->tree, node_lo, node_hi, s));
  return DDM_OK;
}

}  // extern "C"

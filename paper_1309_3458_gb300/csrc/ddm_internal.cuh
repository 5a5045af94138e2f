// Internal declarations shared by the libddm translation units.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "ddm.h"
#include "ddm_ranges.h"

namespace ddm {

// Tree fan-out: one warp lane per child, so a node's 32 children are tested
// by one coalesced load and one ballot.
constexpr int kFan = 32;
constexpr int kLog2Fan = 5;
constexpr int kMaxLevels = DDM_MAX_TREE_LEVELS;

// Device error bits (Status::err).
constexpr unsigned kErrExtent = 1u;
constexpr unsigned kErrTimeout = 2u;
constexpr unsigned kErrCapacity = 4u;
constexpr unsigned kErrChecked = 8u;  // checked build: an index failed its bounds check

// Device-resident status word read back once per synchronising call.
struct Status {
  unsigned long long K;    // pairs counted (plan) or written (write)
  unsigned int err;        // kErr* bits
  unsigned int walk;       // the replay found the records incomplete
  unsigned long long aux;  // call-specific (chunk end, ...)
  unsigned long long tests;  // count pass: (query, leaf) tests, 32 subscriptions each
  unsigned int work[2];    // tickets of the packet kernels and of the replay
  // d = 1 tree: sort by both bounds (ties abound), else the runs of equal lower
  // bounds left to a warp [0] and to a CTA [1] each
  unsigned int both;
  unsigned int runs[2];
  unsigned int pad;
};

__device__ inline void note_out_of_bounds(Status* st) {
  if (st) atomicOr(&st->err, kErrChecked);
}

// Checked build (compiled with DDM_CHECKED, as libddm_checked.so): kernels
// verify the indices they are about to use, and an index out of its bounds
// sets kErrChecked in the status word (the call returns DDM_ERR_INTERNAL)
// and the access is skipped -- never a trap.  In the normal build the check
// is the constant true and costs nothing.
#ifdef DDM_CHECKED
#define DDM_IN_BOUNDS(cond, st) ((cond) ? true : (::ddm::note_out_of_bounds(st), false))
#else
#define DDM_IN_BOUNDS(cond, st) true
#endif

struct Status;
__device__ inline void note_out_of_bounds(Status* st);

// Read-only view of a built tree, passed to kernels by value.
//
// Elements (the subscriptions) sit at sorted positions 0..n-1; a level-l
// node g covers positions [g*32^l, min(n, (g+1)*32^l)) and stores, per
// dimension k, (minlower, maxupper) of the extents in its range.
struct TreeView {
  int d;
  uint32_t n;
  int L;                          // internal levels 1..L; level L has <= 32 nodes
  uint32_t cnt[kMaxLevels + 1];   // nodes per level (index 1..L)
  uint32_t off[kMaxLevels + 1];   // first node of each level within one dimension
  uint32_t total;                 // nodes per dimension
  const float2* e;                // [d][n] (lo, hi) per dimension, sorted order
  const uint32_t* sid;            // [n] subscription id per sorted position
  const float2* nodes;            // [d][total] (minlower, maxupper) per dimension
  // Rank tables (d <= 3, else null): per leaf g and slot 2k (lower bounds of
  // dimension k) / 2k + 1 (upper bounds), kRankSlot words at
  // (g * 2d + slot) * kRankSlot: the leaf's 32 bounds sorted ascending (float
  // bits, padding positions +inf), then at word 35 + c the mask of the leaf
  // positions holding the c smallest (c = 0..32); word 32 of slot 0 is the
  // mask of the leaf's positions that hold an extent.
  const uint32_t* tab;
};
constexpr uint32_t kRankSlot = 68;  // words per rank-table slot (16-byte multiple)

// Read-only view of the planned updates (queries) in their sorted order.
struct QueryView {
  uint32_t m;
  const float2* qe;               // [d][m] (lo, hi) per dimension, sorted order
  const uint32_t* qid;            // [m] update id per sorted position
  const uint32_t* list;           // optional subset of sorted positions (ranges)
  uint32_t first;                 // without list: run positions first .. first+nq-1
  uint32_t nq;                    // number of queries to run
  uint32_t qpp_log2;              // log2 of the queries per packet (2..5: 4 to 32)
  uint32_t take_log2;             // log2 of the packets a warp takes per ticket
  uint32_t tmin;                  // count pass: swapped leaf loops from this many queries
};

// Where the write pass puts each query's pairs: query j's pairs start at
// start[key] - start[b_idx] in `pairs`, key = its update id (by_pos false) or
// its sorted position (by_pos true); start[e_idx] - start[b_idx] pairs in all.
struct WriteView {
  const unsigned long long* start;
  bool by_pos;
  bool swap;  // roles swapped: the tree holds the updates, queries are subscriptions
  const uint32_t* qids;  // optional: id written for query q is qids[q] (else q + qbase)
  uint32_t qbase;        // added to every update id written (a shard's first global id)
  uint32_t b_idx, e_idx;
  ddm_pair* pairs;
  uint32_t* ids;  // when set: only each pair's subscription id is written, here, and pairs is unused
  unsigned long long capacity;
  // set if a wait of the plan's scan ran out: its offsets are too small, so
  // that need <= capacity bounds nothing; nothing is written then
  const uint32_t* failed;
};

// Batched instances: instance i owns update positions [upd_off[i],
// upd_off[i+1]) and subscription positions [sub_off[i], sub_off[i+1]) of the
// concatenated sets; sorting keeps these ranges (the instance is the major
// key), so they hold in sorted order too.  q_inst[p] = instance of the update
// at sorted position p.  count == 0: a single problem.
//
// Whole leaves (leaf_off set): the tree's positions are padded so that every
// instance starts a leaf: instance i owns leaves [leaf_off[i], leaf_off[i+1]),
// subscriptions in the same order, the rest of its last leaf empty.  Without
// that, leaves straddle the re-sort groups of an instance (and instances), and
// the box of such a leaf spans a whole slab, so that every query of the slab
// tests it: 5.2 leaf tests per query on the 4,096-instance workload.
struct BatchView {
  uint32_t count;
  const unsigned long long* upd_off;  // [count + 1]
  const unsigned long long* sub_off;  // [count + 1]
  const uint32_t* q_inst;             // [m]
  const unsigned long long* leaf_off; // [count + 1], or null: positions are not padded
};
// How a padded tree's leaves are filled: leaf l holds the sorted positions
// from off[b] + 32 * (l - leaf_off[b]) on, b the instance owning it; leaves
// past the last are empty.
struct LeafMap {
  const unsigned long long* off;
  const unsigned long long* leaf_off;  // [count + 1], null: the tree is not padded
  uint32_t count;
};

// Exponent of the sort-tile-recursive group size for re-sorting dimension k
// (1 <= k < d) of a set of n extents: with nb = n/32 leaves each dimension
// gets about nb^(1/d) slabs, so dimension k is re-sorted inside groups of
// 32 * nb^((d-k)/d) positions, rounded to a power of two.  0 = no re-sort
// (groups of fewer than 64 would not change any leaf's box).  Kernels use the
// same rule by thresholds (ready_group_table).
__host__ __device__ inline int str_group_log2(uint32_t n, int d, int k, int shift = 0) {
  if (n < 64u) return 0;
  const double nb = (double)((n + 31u) / 32u);
  const double G = 32.0 * pow(nb, (double)(d - k) / (double)d);
  const int g = (int)floor(log2(G) + 0.5) + shift;
  if (g < 6 || (1ull << g) >= (unsigned long long)n) return 0;
  return g;
}

// Order-preserving map from float to uint32 (IEEE order; -0 maps like +0).
__host__ __device__ inline uint32_t float_key(float f) {
#ifdef __CUDA_ARCH__
  uint32_t b = __float_as_uint(f);
#else
  uint32_t b;
  __builtin_memcpy(&b, &f, 4);
#endif
  if (b == 0x80000000u) b = 0u;
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Number of kernels this library has launched in the process (all
// contexts), for launch accounting by callers; defined in ddm_api.cu.
void note_launches(unsigned count);

// OwnerSearch by one warp.
__device__ __forceinline__ uint32_t warp_owner(const unsigned long long* __restrict__ prefix,
                                               uint32_t count, unsigned long long i) {
  OwnerSearch s(count);
  while (s.more()) s.take(__ballot_sync(0xffffffffu, s.probe(prefix, threadIdx.x & 31u, i)));
  return s.lo;
}

// ---- ddm_layout.cu --------------------------------------------------------
// Validate a set (lo <= hi, no NaN in every dimension) and (k32 set) emit its
// sort key: key(lo0), whole (d = 1 tree; st->both is then set if one value of
// the lower bound abounds) or its top 24 bits (a locality order).
// aos (optional, cnt * d float2): an interleaved copy of the coordinates,
// aos[i*d + k] = (lo_k, hi_k) of extent i, written while validating, so that
// the gathers by id read one contiguous record per extent instead of 2d
// scattered words.
cudaError_t launch_validate(int d, const float* lo, const float* hi, uint32_t cnt,
                            uint32_t* k32, bool whole_key, float2* aos, Status* st, int sms,
                            cudaStream_t s);
// keys[i] = (i >> glog2) << 24 | the top 24 bits of key(lo_k[vals[i]]): re-sort
// inside groups; with id_bits > 0 the packed word, above the id vals[i].
cudaError_t launch_rekey(const uint32_t* vals, const float* lo_k, uint32_t cnt, int glog2,
                         unsigned long long* keys, int id_bits, int sms, cudaStream_t s);
// Batched sets: inst[i] = instance owning position i (off has count+1 entries).
// Validation and class-major tree keys for d >= 2; hist[256] (zeroed by the
// caller) receives the number of extents of each size class.
cudaError_t launch_validate_class(int d, const float* lo, const float* hi, uint32_t cnt,
                                  uint32_t* k32, uint32_t* hist, float2* aos, Status* st, int sms,
                                  cudaStream_t s);
// inst[i] = the b with off[b] <= i < off[b+1], for 0 <= i < total.
cudaError_t launch_fill_inst(const unsigned long long* off, uint32_t count, uint32_t total,
                             uint32_t* inst, int sms, cudaStream_t s);
// Batched validation + keys: the top 24 bits of key(lo0[i]) in k32 or, below
// inst[i], in keys (with vals = ids).
cudaError_t launch_validate_batch(int d, const float* lo, const float* hi, uint32_t cnt,
                                  const uint32_t* inst, unsigned long long* keys, uint32_t* vals,
                                  uint32_t* k32, float2* aos, Status* st, int sms, cudaStream_t s);
// Groups of each instance (or class) for a re-sort over the whole set, from
// its group exponent (0: one group).  glog2/ngroups: [count] each.
cudaError_t launch_batch_groups(const unsigned long long* off, uint32_t count, const int* glog2,
                                uint32_t* ngroups, cudaStream_t s);
// Batched re-sort keys: group = gbase[inst] + (local position >> glog2[inst]).
cudaError_t launch_rekey_batch(const uint32_t* vals, const float* lo_k, uint32_t cnt,
                               const uint32_t* inst, const unsigned long long* off,
                               const int* glog2, const unsigned long long* gbase,
                               unsigned long long* keys, int id_bits, int sms, cudaStream_t s);
// qe[k][i] = (lo_k, hi_k)[vals[i]], qid[i] = vals[i].
cudaError_t launch_gather(int d, const uint32_t* vals, const float* lo, const float* hi,
                          const float2* aos, uint32_t cnt, float2* qe, uint32_t* qid, int sms,
                          cudaStream_t s);

// ---- ddm_sort.cu ----------------------------------------------------------
struct SortScratch {
  unsigned long long* keys[2];
  uint32_t* vals[2];
  uint32_t* hist;       // [8][256]
  uint32_t* lookback;   // [8][tiles][256], or the cooperative sort's scratch
  uint32_t* counters;   // [8]
};
constexpr int kSortTile = 4096;
size_t sort_lookback_words(uint32_t n);
// Stable LSD radix sort on the low 8*passes bits of 64-bit keys, with a
// uint32 payload (one cluster, one cooperative launch or onesweep, by size).
// Input in keys[0]/vals[0]; *out_buf receives the index (0 or 1) of the
// buffers holding the result.
// Test hook: one warp polls `word` (which nothing sets) with the sort's
// bounded wait, at most `limit` polls, and records kErrTimeout.
cudaError_t launch_debug_wait(const uint32_t* word, uint32_t limit, Status* st, cudaStream_t s);
cudaError_t launch_sort64(SortScratch sc, uint32_t n, int passes, int* out_buf, Status* st, int sms,
                          cudaStream_t s);
// The same for keys that fit one 64-bit word together with the id: words key
// << id_bits | id, sorted by key_bits bits above id_bits; the ids come out in
// vals[0].  With a source the words are built from it (its arrays may not
// overlap keys[] or vals[0]), else they are in keys[0].
struct SortSource {
  const uint32_t* k32;  // [n] low part of the key, or null
  const uint32_t* hi;   // optional [n]: the part above k32_bits
  int k32_bits;
  int id_bits;
  bool words_out;       // the sorted words go to keys[0] instead (an even number of passes)
  // Optional: when *both is set, sorted by (key, key(second)): by the second
  // key first, then, the words rebuilt from their ids, by the first (a k32 and
  // 32 key bits each).  The ids come out in vals[0] then.
  const uint32_t* both;
  const float* second;  // [n]
};
// Longest runs of equal lower bounds put in order by the elements themselves, by
// a warp, and by a CTA on chip (longer ones it sorts in global memory, some 20
// us per 2,048 elements, so a value that promises more than twice the digits
// would cost is sorted by both bounds from the start).
constexpr uint32_t kNearRun = 64, kWarpRun = 128, kCtaRun = 2048;
// Order of a d = 1 tree from its words: ids to vals, ties of the lower bound in
// the order of their upper bound (unless st->both: the sort has done that).
// Runs of more than kNearRun equal lower bounds are listed in `list` (n words, uint2
// entries: those of a warp from the front, of a CTA from the back) and counted
// in st->runs, for launch_long_ties, which overwrites words and tmp there.
cudaError_t launch_tie_order(const unsigned long long* words, uint32_t n, int id_bits,
                             const float* hi, uint32_t* vals, uint2* list, Status* st, int sms,
                             cudaStream_t s);
cudaError_t launch_sort_packed(SortScratch sc, const SortSource& src, uint32_t n, int key_bits,
                               Status* st, int sms, cudaStream_t s);

// ---- ddm_ranksort.cu ------------------------------------------------------
// Validation, first order (vals) and optional interleaved copy of a small set
// in one launch, the order of launch_validate's or launch_validate_class's
// keys (hist as there); qe and qid (optional) receive the set in that order.
enum { kRankTree = 1, kRankLocal = 2, kRankClass = 3 };
cudaError_t launch_rank_sort(int mode, int d, const float* lo, const float* hi, uint32_t n,
                             uint32_t* vals, uint32_t* hist, float2* aos, float2* qe, uint32_t* qid,
                             Status* st, cudaStream_t s);

// ---- ddm_segsort.cu -------------------------------------------------------
// Thresholds of the group exponents, before the first plan on a device.
cudaError_t ready_group_table();
// Positions a CTA re-sorts at once (log2 10 to 13).
constexpr int kSegTileLog2Min = 10, kSegTileLog2 = 12, kSegTileLog2Max = 13;
// A set's re-sort in one dimension, by instance (off null: one instance).
struct SegPlan {
  const unsigned long long* off;    // [count + 1] positions of each instance
  const int* glog2;                 // [count] group exponents, 0 = left as it is
  const unsigned long long* cbase;  // [count + 1] first chunk of each instance
  uint32_t count;
};
// Size classes: written by launch_class_plan from the class histogram.
struct ClassPlan {
  unsigned long long* off;    // [257]
  int* glog2;                 // [d][256], by dimension
  unsigned long long* cbase;  // [d][257]
  uint32_t tile[DDM_MAX_DIMS];  // positions per chunk, by dimension
};
cudaError_t launch_class_plan(const uint32_t* hist, int d, int shift, const ClassPlan& plan,
                              cudaStream_t s);
// Batched sets: group exponents glog2 [d][count] and first chunks cbase
// [d][count + 1] of every dimension, and (optional) first leaves leaf_off
// [count + 1] of a padded tree.  No chunks if `off` descends or passes `total`.
// sums: batch_plan_words() words of scratch.
size_t batch_plan_words(uint32_t count, int d);
cudaError_t launch_batch_plan(const unsigned long long* off, uint32_t count, uint32_t total, int d,
                              int shift, int tile_log2, int* glog2, unsigned long long* cbase,
                              unsigned long long* leaf_off, unsigned long long* sums,
                              cudaStream_t s);
// Stable re-sort of the ids in `vals` by the locality key of lo_k inside each
// group, in place; with one instance g is its group exponent.  tmp0 and tmp1
// (`total` words each) are used only by groups larger than a chunk's tile.
cudaError_t launch_segsort(uint32_t* vals, const float* lo_k, uint32_t total, int g,
                           const SegPlan& plan, int tile_log2, unsigned long long* tmp0,
                           unsigned long long* tmp1, int sms, cudaStream_t s);

cudaError_t launch_long_ties(unsigned long long* words, uint32_t n, int id_bits, const float* hi,
                             uint32_t* vals, const uint2* list, unsigned long long* tmp,
                             const Status* st, int sms, cudaStream_t s);

// ---- ddm_tree.cu ----------------------------------------------------------
void tree_shape(uint32_t n, int* L, uint32_t* cnt, uint32_t* off, uint32_t* total);
// Group sizes (log2) of the per-dimension re-sorts: dimension k >= 1 is
// re-sorted by lower bound inside aligned groups of 2^glog2[k] positions;
// `shift` is added to every exponent (tuning knob, 0 = the STR sizes).
void str_groups(uint32_t n, int d, int* glog2, int shift = 0);
// `set_n` extents in lo / hi (t.n unless the tree is padded by `map`).
cudaError_t launch_build(const TreeView& t, uint32_t set_n, const LeafMap& map,
                         const uint32_t* sorted_ids, const float* lo, const float* hi,
                         const float2* aos, float2* e, uint32_t* sid, float2* nodes, uint32_t* tab,
                         Status* st, cudaStream_t s);
cudaError_t launch_export_nodes(const TreeView& t, float* node_lo, float* node_hi, cudaStream_t s);

// ---- ddm_query.cu ---------------------------------------------------------
// Replay records.  While counting, every (query, leaf) test of a packet
// that has hits is stored as one record of ten bytes: x = leaf << 5 | query
// lane, the hit mask over the leaf's 32 subscriptions, and (16 bits) the
// query's matches before this leaf counted from the start of the record's
// block.  Records of a packet are kept in walk order (leaf by leaf, query
// lanes ascending within a leaf), in chains of fixed-size blocks of a shared
// arena; a block has a header with the matches each query of its chain had
// before the block's first record, so that a record's place in its query's
// output is the header entry plus its 16-bit count (a block holds at most 512
// records of at most 32 hits: the count stays below 2^14).  After counting,
// the blocks are listed in plan order and the write pass expands any range of
// them, every record independently, instead of walking the tree again.
//
// The first block of each chain belongs to it from the start (its header is
// zero); only the blocks after it are taken from a counter, so that the
// packets of a sparse problem make no atomic.  (If the record budget does not
// reach for that, every block is taken from the counter: a plan whose hits lie
// in few packets can still be recorded.)  Every block is an entry of the
// write pass, but for the two first blocks of a packet, which are one if the
// plan has few pairs per entry.
// A write laid out by update id takes the blocks as they are (the chains'
// first, then those handed out); only writes of ranges of the plan order need
// them listed in that order.  With every block
// from the counter and listed, the count pass of 2.5e7 + 2.5e7 extents
// (d = 1, alpha = 1) took 2.81 ms and the write pass 2.58 ms; now 1.73 and
// 1.47 ms.
constexpr uint32_t kRecBlock = 512;  // records per block: x and hit mask 2 KiB each, counts 1 KiB
constexpr uint32_t kRecHdr = 16;     // header: one running count per query of the chain
// words per block: x[kRecBlock], hit mask[kRecBlock], 16-bit counts, header
constexpr uint32_t kRecWords = 2 * kRecBlock + kRecBlock / 2 + kRecHdr;
// A packet's records go to two chains of blocks, one per half of its query
// lanes, so that a block holds the records of at most 16 queries (its pairs
// land in fewer output runs): the write pass took 127 instead of 134 ms on
// the clustered d = 3 workload, the count pass 5 ms more.  Chain c of packet
// p is chain index p * kRecChains + c of the arena's per-chain arrays, and its
// first block has that number.
constexpr uint32_t kRecChains = 2;
constexpr uint32_t kNoBlock = 0xffffffffu;
struct RecordArena {
  uint32_t* rec;           // [max_blocks][kRecWords]: x, hit mask, 16-bit counts, header
  uint2* blk_own;          // [max_blocks] packet of a block handed out, and its
                           // number among that packet's blocks handed out
  uint32_t* blk_count;     // [max_blocks] records in the block
  uint32_t* pkt_nblk;      // [packets] blocks of each packet, the two first as one
  unsigned long long* pkt_off;  // [packets + 1] exclusive prefix of pkt_nblk
  uint4* blk_list;         // [max_blocks] entries in plan order: block, packet,
                           // its records, and those of the next block if the
                           // entry is a packet's two first blocks (plans with
                           // short entries); null: not listed
  uint32_t* blk_counter;   // [0] blocks handed out beyond the chains' first (may
                           // exceed the arena), [1] such blocks the whole pass
                           // needed
  uint32_t chains;         // chains of the plan's packets, 0: no first blocks of their own
  uint32_t max_blocks;     // 0: no recording
};
// Pairs per entry of a plan up to which its entries count as short: the write
// pass then takes a packet's two first blocks as one entry and expands by
// listing pairs instead of record by record.  Writes of 5e5 + 5e5 extents, short
// and long form: d = 1, 65 pairs per entry 54 / 66 us, 129: 65 / 66, 257: 78 /
// 66, 384: 90 / 68; d = 2, 64: 53 / 66, 128: 65 / 66, 256: 77 / 71; d = 3 (3e5 +
// 3e5), 130: 53 / 54, 262: 64 / 66, 526: 80 / 69.
constexpr uint32_t kShortEntry = 160;
// The records of the last count pass are complete (the write pass may
// replay them) iff recording was on and the arena did not run out.
__device__ __forceinline__ bool records_complete(const RecordArena& ra) {
  return ra.max_blocks > 0 &&
         (unsigned long long)ra.chains + ra.blk_counter[0] <= ra.max_blocks;
}

// counts[update id] (and counts_pos[sorted position], if not null); records
// into `ra` when ra.max_blocks > 0.  With bv.count > 0 every query only
// matches its own instance's subscriptions and pairs carry instance-local ids.
// `sms` sizes the persistent grids: pass SMs x CTAs-per-SM / 8 to change the
// default of 8 CTAs of 256 threads per SM (tuning knob).  `zeroed`: *work is
// zero already.
cudaError_t launch_count(const TreeView& t, const QueryView& q, const BatchView& bv,
                         uint32_t flags, uint32_t* counts, uint32_t* counts_pos,
                         const RecordArena& ra, uint32_t* work, bool zeroed, Status* st, int sms,
                         cudaStream_t s);
// Walking write pass; it does nothing when `ra` holds complete records (the
// replay kernel, launched next to it, writes the pairs then).
cudaError_t launch_write(const TreeView& t, const QueryView& q, const BatchView& bv,
                         uint32_t flags, const WriteView& w, const RecordArena& ra,
                         uint32_t* work, Status* st, int sms, cudaStream_t s);
// After the count pass: blk_list = every packet's entries, packets in plan
// order; pkt_off must already hold the prefix of pkt_nblk, and *pairs the
// plan's pairs.
cudaError_t launch_block_list(const RecordArena& ra, const unsigned long long* pairs, int sms,
                              cudaStream_t s);
// Write pass from records: positions [pb, pe) of the plan, in packets [p0,
// p1) (without a list: all packets), and (when id_filter) only updates with
// ids in [idb, ide).  Only sets st->walk unless `ra` holds complete records.
cudaError_t launch_replay(const TreeView& t, const QueryView& q, const BatchView& bv,
                          const RecordArena& ra, const WriteView& w, uint32_t p0, uint32_t p1,
                          uint32_t pb, uint32_t pe, bool id_filter, uint32_t idb, uint32_t ide,
                          uint32_t* work, bool zeroed, Status* st, int sms, cudaStream_t s);
// pair_off[i] = offsets[min(upd_off[i], m)] for i <= count.
cudaError_t launch_gather_offsets(const unsigned long long* offsets, uint32_t m,
                                  const unsigned long long* upd_off, uint32_t count,
                                  unsigned long long* pair_off, cudaStream_t s);

// ---- ddm_scan.cu ----------------------------------------------------------
constexpr int kScanTile = 4096;
// offsets[0..m] = exclusive prefix of counts; offsets[m] and st->K = total.
cudaError_t launch_scan(const uint32_t* counts, uint32_t m, unsigned long long* offsets,
                        unsigned long long* block_sums, Status* st, cudaStream_t s);
// Up to kMaxScanJobs independent scans of the form above in one launch.
// `state` holds scan_state_words() words, zeroed by the caller on the stream.
// A wait that runs out is recorded in st->err and *failed (its offsets are then
// too small).
// `hint` (optional) receives the sizing hint of the plan's record arena.
struct ScanJob {
  const uint32_t* counts;
  uint32_t m;
  unsigned long long* offsets;
  bool total_to_k;  // the total goes to st->K too
};
constexpr int kMaxScanJobs = 3;
// What the last recorded count pass needed, written to host memory: blocks in
// all, packets, blocks held.
struct ScanHint {
  volatile uint32_t* to;  // pinned host memory, or null
  const uint32_t* blk_counter;
  uint32_t chains, packets, max_blocks;
};
size_t scan_state_words(const ScanJob* jobs, int count);
cudaError_t launch_scan_multi(const ScanJob* jobs, int count, unsigned long long* state,
                              const ScanHint& hint, uint32_t* failed, Status* st, cudaStream_t s);
// Test hook: the scan of `job` without its first tile, so that the waits of
// the others, of at most `polls` polls, run out.
cudaError_t launch_debug_scan(const ScanJob& job, unsigned long long* state, uint32_t polls,
                              uint32_t* failed, Status* st, cudaStream_t s);
// st->aux = the largest end, kPlanFailed in its place if *failed is set.
constexpr unsigned long long kPlanFailed = ~0ull;
cudaError_t launch_chunk_end(const unsigned long long* offsets, uint32_t m, uint32_t begin,
                             unsigned long long capacity, const uint32_t* failed, Status* st,
                             cudaStream_t s);
// list = sorted positions i (ascending) with begin <= qid[i] < end; uses
// flags/offs/sums as scratch.
cudaError_t launch_select(const uint32_t* qid, uint32_t m, uint32_t begin, uint32_t end,
                          uint32_t* flags, unsigned long long* offs, unsigned long long* sums,
                          uint32_t* list, Status* st, cudaStream_t s);

}  // namespace ddm

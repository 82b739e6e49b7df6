// Internal interfaces between the host solver (solver.cu) and the kernels
// (kernels.cu).  Not part of the public ABI.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "per_device.h"

namespace mstgpu {

typedef unsigned long long u64;
constexpr u64 KEY_INF = ~0ULL;

// Device-side error bits, latched in DevState::err.
enum : uint32_t {
  ERR_VERTEX = 1u,    // an input vertex id >= n
  ERR_LOOKBACK = 2u,  // the output scan's barrier was not reached in time (bounded wait ran out)
  ERR_HASH = 4u,      // hash table probe sequence exhausted
  ERR_JUMP = 8u,      // pointer doubling did not reach a root within its bound
  ERR_TMA = 16u,      // a bulk copy never completed (bounded mbarrier wait ran out); tiles were skipped
  ERR_TABLE = 32u,    // a batched size table is inconsistent (offsets not starting at 0 or decreasing)
  ERR_OVERFLOW = 64u, // a compaction's survivors exceeded its output capacity (nothing past it was written)
  ERR_BARRIER = 128u, // a grid barrier of the one-launch rounds was not reached in time (bounded wait ran out)
};
// Rounds that ended early: parent[] may hold tagged links instead of vertices,
// so the passes that follow its entries (jump, filter, further rounds) do nothing.
constexpr uint32_t ERR_ROUNDS = ERR_JUMP | ERR_BARRIER;

// Small per-handle device state.
constexpr int LVL_MAX = 32;  // recursion levels of a planned Filter-Borůvka
struct DevState {
  uint32_t err;
  uint32_t jump_flag;   // set when a pointer-jump launch left a vertex short of its root
  uint32_t scan_ctr[2]; // blocks of the output scan that have arrived at its barrier, and that have ended
  u64 count[6 + 2 * LVL_MAX];  // counts written by the last tile of a scan kernel; from CNT_LVL on,
                               //   the list lengths of a planned Filter-Borůvka (see CNT_LVL)
  u64 pivot;            // result of the pivot selection
  uint32_t giant_root;  // root of the largest sampled component (filter fast path)
  uint32_t max_w;       // largest input weight (key layout)
  uint32_t local_samples;  // sampled local edges (automatic tile contraction)
  uint32_t giant_count;    // of the GIANT_SAMPLES sampled edge ends, those in the giant component
};
// Edge ends the giant-component root is sampled from.  The filter tests the
// giant-component bitmap first only when at least GIANT_MIN_COUNT of them lie
// in that component: otherwise (a batch of many small graphs has no giant
// component) nearly every heavy edge needs its labels anyway, and the bitmap
// gathers only add a dependent round trip.
constexpr uint32_t GIANT_SAMPLES = 1024, GIANT_MIN_COUNT = 512;
// CNT_LVL + k: length of the light list of recursion level k (level 0: the
// input); CNT_LVL + LVL_MAX + k: the filtered heavy edges of level k.
enum { CNT_EDGES = 0, CNT_ACTIVE = 1, CNT_TMP = 2, CNT_AUX = 3, CNT_USER = 4, CNT_CUT = 5, CNT_LVL = 6 };

// Where a kernel that ends a call leaves the device state for the host.
struct Readback {
  const DevState *state;
  DevState *mirror;  // page-locked, mapped
  uint32_t *flag;    // mapped word that the host polls for seq
  uint32_t seq;
};

// Output bookkeeping of a compaction launch.  Unordered compactions claim
// their output ranges by atomic adds on *total (zero before the launch); the
// ordered scan of the output ids exchanges its blocks' counts and writes *total.
constexpr int FINISH_BLOCKS = 1024;  // of the ordered scan, at most
struct ScanState {
  uint32_t *count;     // [FINISH_BLOCKS] set bits of each block's words
  uint32_t *arrived;   // blocks that have written theirs (zero between launches)
  uint32_t *ended;     // blocks that have ended (zero between launches)
  u64 *total;
  uint32_t *err;
  uint32_t spin_limit;  // polls of the barrier before the wait gives up (ERR_LOOKBACK)
};

struct HashSlot {
  u64 pair;  // (min(u,v) << 32) | max(u,v); all ones = empty
  u64 key;   // minimum (w << 32) | id seen for this pair
};

// Layout of the uint64 relaxation key of a solve.  Edges are ordered by
// (w, id).  When the weight, the edge id and a vertex id fit into 64 bits
// together (vbits + idbits + bits(max w) <= 64), the key is
//   w << (idbits + vbits) | id << vbits | other,
// where `other` is the far end of the edge as seen from the relaxed vertex, so
// the hook reads the chosen neighbour straight from the key.  Otherwise the
// key is w << 32 | id and the hook finds the neighbour through the input
// arrays.  Either way the minimum key of a vertex is its (w, id)-lightest edge.
struct KeyLayout {
  int packed;
  int vbits, idbits;
};

// An edge list in structure-of-arrays form.  id == nullptr: id = index.
struct EdgeList {
  const uint32_t *u, *v, *w, *id;
};
struct EdgeOut {
  uint32_t *u, *v, *w, *id;
};

enum CompactMode : int {
  CM_RELABEL = 0,    // (label[u], label[v]); drop self-loops
  CM_PARTITION = 1,  // key <= pivot and u != v; unchanged
  CM_FILTER = 2,     // key > pivot; (label[u], label[v]); drop self-loops
  CM_DEDUPE = 3,     // keep iff the hash table holds this edge's key for its pair
  CM_HEAVY = 4,      // key > pivot and not both ends in the giant component; unchanged (first filter pass)
};

struct CompactArgs {
  EdgeList in;
  uint64_t m;              // input length, or with m_dev the input list's capacity
  const u64 *m_dev;        // input length in device memory (read as min(*m_dev, m)), or nullptr
  EdgeOut out;
  const uint32_t *label;   // relabel / filter
  const uint32_t *giant_bits;  // filter: bitmap of the vertices in the largest component, or nullptr
  const uint32_t *giant_count; // filter: if set, the bitmap is used only when *giant_count >= GIANT_MIN_COUNT
  u64 pivot;               // partition / filter (used when pivot_dev == nullptr)
  const u64 *pivot_dev;
  u64 *best;               // if set: relax best[] of both ends with each survivor's key
  KeyLayout kl;
  HashSlot *table;         // dedupe lookup, or insert target when hash_insert
  uint64_t tmask;
  int hash_insert;
  uint32_t n;              // vertex count, for validation
  int validate;            // check u, v < n (sets ERR_VERTEX, skips the edge)
  uint32_t *max_w;         // if set: atomicMax of every input weight (key layout)
  uint32_t *cur_u, *cur_v; // if set: cur_u[id], cur_v[id] = the survivor's written ends
  ScanState st;
  int shape;               // tile shape of the relabel / partition compaction (see shape_index)
  int warp_partition;      // partition in the default shape: 1 runs the warp-streamed pass (for light
                           //   shares up to 1/8, where its per-warp output claims stay few), 0 the block kernel
  uint64_t out_cap;        // if nonzero: output capacity; a tile that would write past it writes
                           //   nothing and sets ERR_OVERFLOW (with m_dev, m bounds the input count)
};

struct HookArgs {
  const uint32_t *cand;    // candidate vertices; nullptr = 0..ncand-1
  uint64_t ncand;
  u64 *best;               // keys (see KeyLayout) of the round's minimum edges
  KeyLayout kl;
  const uint32_t *src, *dst;  // ends of each edge by id (unpacked keys): the input arrays,
                              // or the ends recorded when the current list was written
  uint32_t *parent;
  uint32_t *chosen_bits;   // bitmap over edge ids
  uint32_t *active_out;    // active vertices (best != INF), unspecified order
  u64 *counter;            // number written to active_out; zero before the launch
  uint32_t *err;
  u64 *wsum;               // if set: the weights of the chosen edges are added into these
                           //   WSUM_SLOTS counters (one add per warp, spread over the slots)
  int shape;               // tile shape (see shape_index)
};

// Tile shapes of the compaction and hook kernels, as the `shape` field of
// their argument structs: 0 is the default, 256 threads per block x 8 items
// per thread (so a zero-initialised struct gets it); 1 + 3 * b + i is the b-th
// of {128, 256, 512} threads with the i-th of {4, 8, 16} items per thread.
constexpr int SHAPE_COUNT = 10;
inline int shape_index(uint32_t block_threads, uint32_t items_per_thread) {
  if (block_threads == 0 && items_per_thread == 0) return 0;
  const uint32_t bt = block_threads ? block_threads : 256, it = items_per_thread ? items_per_thread : 8;
  const int b = bt == 128 ? 0 : bt == 256 ? 1 : bt == 512 ? 2 : -1;
  const int i = it == 4 ? 0 : it == 8 ? 1 : it == 16 ? 2 : -1;
  return (b < 0 || i < 0) ? -1 : 1 + 3 * b + i;
}
// The relabel compaction's shape: both zero is 128 x 4 (shape 1).
inline int relabel_shape_index(uint32_t block_threads, uint32_t items_per_thread) {
  return (block_threads == 0 && items_per_thread == 0) ? 1 : shape_index(block_threads, items_per_thread);
}

// Counters the kernels that choose MSF edges add the chosen weights into, so
// that the forest's total needs no gather of w at the end.
constexpr int WSUM_SLOTS = 256;

inline int current_device() {
  int dev = 0;
  cudaGetDevice(&dev);
  return dev;
}

// ---- launchers (kernels.cu); all asynchronous on `s` ----
void launch_compact(CompactMode mode, const CompactArgs &a, uint64_t max_count, cudaStream_t s);
// max_w: as in RoundsArgs.
void launch_min_edges(EdgeList in, uint64_t m, uint32_t n, int validate, KeyLayout kl, u64 *best, uint32_t *err,
                      int sms, cudaStream_t s, const uint32_t *max_w = nullptr);
void launch_max_weight(const uint32_t *w, uint64_t m, uint32_t *out, int sms, cudaStream_t s);
void launch_hook(const HookArgs &a, cudaStream_t s);
// max_steps: parent steps per thread and launch (0: the default of 64).
// With act == count_dev == nullptr the launch covers every vertex
// 0..count_host-1 and, given gbits, sets bit v of that bitmap iff v's walk
// reached the root *groot in this launch (gbits is ignored for lists); it does
// nothing when *err holds ERR_ROUNDS.
void launch_jump(const uint32_t *act, const u64 *count_dev, uint64_t count_host, uint64_t max_count,
                 uint32_t *parent, u64 *best, int reset_best, uint32_t *flag, const uint32_t *err, int sms,
                 cudaStream_t s, uint32_t max_steps = 0, const uint32_t *groot = nullptr, uint32_t *gbits = nullptr);
// Sets ERR_VERTEX in *err if some x[i] (i < count) is >= bound.
void launch_range_check(const uint32_t *x, uint64_t count, uint32_t bound, uint32_t *err, int sms, cudaStream_t s);
void launch_hash_insert(EdgeList in, uint64_t m, HashSlot *table, uint64_t tmask, uint32_t *err, int sms,
                        cudaStream_t s);
// The pivot is the sample key of rank `rank` (0-based); a rank >= sample
// means sample / 2, the sample median of Alg. 2.
void launch_pivot(EdgeList in, uint64_t m, const u64 *m_dev, u64 state, uint32_t sample, u64 *sample_buf,
                  u64 *pivot_out, cudaStream_t s, uint32_t rank = ~0u);
// Pivot selection by a cooperative multi-block radix select (same result as
// launch_pivot); `scratch` holds pivot_scratch_bytes().  False if the
// cooperative launch was refused.
size_t pivot_scratch_bytes();
bool launch_pivot_coop(EdgeList in, uint64_t m, u64 state, uint32_t sample, u64 *keys, void *scratch,
                       u64 *pivot_out, cudaStream_t s, const u64 *m_dev = nullptr, uint32_t rank = ~0u);
// What a solve starts from.
struct InitArgs {
  u64 *best;         // [n] KEY_INF
  uint32_t *parent;  // [n] own index
  uint32_t n;
  uint32_t *bits;    // [words] zero
  uint64_t words;
  uint32_t *zero;    // [zero_words] zero: the handle's counters
  uint64_t zero_words;
  // with w: the largest of its m weights in *max_w (zero before), and *max_next zero
  const uint32_t *w;
  uint64_t m;
  uint32_t *max_w, *max_next;
};
void launch_init(const InitArgs &a, int sms, cudaStream_t s);
// The bitmap's ids in ascending order and their number.
struct FinishArgs {
  const uint32_t *bits;
  uint64_t nwords;
  const uint32_t *w;  // weights to add up into *total_weight (zero before), or nullptr
  uint32_t *out_ids, *out_count;
  u64 *total_weight;
  ScanState st;
  const u64 *wsum;    // WSUM_SLOTS counters whose sum is the total, or nullptr
  Readback rb;        // behind everything else, if rb.state
};
void launch_finish(const FinishArgs &a, int sms, cudaStream_t s);
// The giant component's root: the most frequent root among the labels of
// sampled edge ends (P is walked to the roots); launch_giant_bits also marks
// its vertices (bit v set iff P[v] is that root; P fully contracted).
void launch_giant_root(EdgeList in, uint64_t m, u64 state, const uint32_t *P, uint32_t n, uint32_t *root_tmp,
                       cudaStream_t s, const u64 *m_dev = nullptr, uint32_t *count_out = nullptr);
void launch_giant_bits(EdgeList in, uint64_t m, u64 state, const uint32_t *P, uint32_t n, uint32_t *root_tmp,
                       uint32_t *bits, int sms, cudaStream_t s);
// tile-local contraction (Section 4.1)
void launch_tile_count(EdgeList in, uint64_t m, uint32_t n, uint32_t B, u64 *cutmin, uint32_t *count,
                       u64 *local_total, uint32_t *max_w, uint32_t *err, int sms, cudaStream_t s);
void launch_tile_scan(const uint32_t *count, uint32_t ntiles, u64 *offsets, cudaStream_t s);
void launch_tile_scatter(EdgeList in, uint64_t m, uint32_t n, uint32_t B, const u64 *offsets, uint32_t *fill,
                         uint32_t *b_ends, uint32_t *b_w, uint32_t *b_id, EdgeOut cut, u64 *cut_fill, int sms,
                         cudaStream_t s);
bool launch_tile_contract(uint32_t n, uint32_t B, uint64_t nlocal, const u64 *cutmin, const u64 *offsets,
                          const uint32_t *b_ends, const uint32_t *b_w, const uint32_t *b_id, uint32_t *parent,
                          uint32_t *bits, EdgeOut rest, u64 *rest_fill, uint32_t *err, cudaStream_t s,
                          int filter_heavy, u64 *wsum);
void launch_tile_sample(EdgeList in, uint64_t m, uint32_t n, uint32_t B, u64 state, uint32_t samples,
                        uint32_t *local_count, cudaStream_t s);
// Stable LSD radix sort of (u64 key, u32 value) pairs over the low `bits` bits;
// true when the result is in (keys_tmp, vals_tmp).  hist holds radix_hist_bytes().
size_t radix_hist_bytes(uint64_t m, int sms);
bool launch_radix_sort(u64 *keys, uint32_t *vals, u64 *keys_tmp, uint32_t *vals_tmp, uint64_t m, int bits,
                       uint32_t *hist, int sms, cudaStream_t s);
// Sort-based parallel-edge removal of list T (ends already component labels,
// no self-loops, ids present): keeps each unordered pair's (w, id)-lightest
// edge and emits it through `emit` (out, counter, best / ends as a compaction).
// vbits: bits of a vertex label; wbits, ibits: of a weight and an id.
size_t sort_dedupe_scratch_bytes(uint64_t m, int sms);
void launch_sort_dedupe(EdgeList T, uint64_t m, int vbits, int wbits, int ibits, const CompactArgs &emit,
                        void *scratch, int sms, cudaStream_t s);

// minEdges by sorting both ends of every edge by vertex and taking segmented
// minima (one atomic per vertex run and warp); false if 2m does not fit 32 bits.
size_t min_edges_sort_scratch_bytes(uint64_t m, int sms);
bool launch_min_edges_sort(EdgeList E, uint64_t m, uint32_t n, int validate, KeyLayout kl, u64 *best, uint32_t *err,
                           void *scratch, int sms, cudaStream_t s);

// The rounds of a Borůvka call in one cooperative launch (rounds.cu).
constexpr int ROUNDS_MAX = 72;  // rounds of a call at most (components at least halve: 2 * (32 + 2) for 32-bit ids)
struct RoundsState {            // zero before the launch
  uint32_t bar;                 // grid barrier
  uint32_t jflag[4];            // a jump pass left a vertex short of its root (rotating)
  uint32_t levels;              // rounds run
  u64 ca;                       // vertices of the call (with at least one edge)
  u64 ce[ROUNDS_MAX], cv[ROUNDS_MAX];  // edges left after round r; components left with a root in round r
  u64 off[ROUNDS_MAX + 1];      // offset of each round's part of link and rep
};
struct RoundsArgs {
  EdgeList in;          // the call's list; ends are current representatives (plain ids < n)
  uint64_t m;           // its length, or with m_dev its capacity
  const u64 *m_dev;     // length in device memory (read as min(*m_dev, m)), or nullptr
  EdgeOut list[2];      // ping-pong lists of the rounds, each with room for the whole list
  int first_slot;       // the first round's output (in may be the other one)
  int best_ready;       // best[] already holds the list's minEdges
  int validate;         // check u, v < n in the first pass (without best_ready)
  KeyLayout kl;         // with max_w only its bit widths count
  const uint32_t *max_w;  // largest weight in device memory: packs the keys when they fit; or nullptr
  u64 *best;            // [n] all KEY_INF but for a ready first round; with want_parent all KEY_INF again afterwards
  uint32_t *parent;     // [n] representatives; the call's vertices are updated if want_parent
  uint32_t *link;       // [n] links of the rounds after the first
  uint32_t *rep;        // [n] representatives of their components (want_parent)
  uint32_t *act;        // [n] the call's vertices
  int want_parent;
  const uint32_t *src, *dst;  // ends by id of a list whose ends nothing recorded
  uint32_t *cur_u, *cur_v;    // ends by id as last written (unpacked keys)
  int ends_rec;         // cur_u, cur_v hold the list's ends
  int record_first;     // record them in the first pass (a list with ids whose ends nothing recorded)
  uint32_t *chosen_bits;
  u64 *wsum;
  uint32_t n, max_rounds;
  RoundsState *st;
  uint32_t *err;
  uint32_t spin_limit;  // polls of a grid barrier before the wait gives up (ERR_BARRIER)
};
// States that a solve's start clears; its later launches clear the last again.
constexpr int ROUNDS_STATES = 8;
// max_edges: bound on the list's length; clear: a.st is not zero yet.  False if
// the launch was refused (nothing ran).
bool launch_rounds(const RoundsArgs &a, uint64_t max_edges, bool clear, int sms, cudaStream_t s);

// Whole graphs solved by one block each (block.cu).
constexpr uint32_t BLOCK_MAX_N = 65536;   // 16-bit labels
constexpr uint64_t BLOCK_MAX_M = 1ULL << 22;
// Vertices up to which a graph runs in a block of 256 threads (four per SM),
// and of 512 (two per SM): their minima fill the blocks' shared memory, as those
// of BLOCK_BIG_N vertices fill a whole SM's.
constexpr uint32_t BLOCK_SMALL_N = 12288, BLOCK_MID_N = 28416, BLOCK_BIG_N = 57344;
struct BlockArgs {
  const uint32_t *gn;          // vertices per graph
  const uint64_t *edge_off, *vert_off;
  const uint32_t *src, *dst, *w;
  uint64_t m_total;            // edges of the arrays
  const uint32_t *order;       // graphs, largest first
  uint32_t first, num;         // this launch's part of order
  uint32_t *queue;             // zero before the launch
  uint4 *ent;                  // [m_total] scratch
  uint2 *live;                 // [m_total] scratch
  u64 *gbest;                  // [vertices] scratch
  uint32_t *bits;              // chosen-edge bitmap
  u64 *totals;                 // forest weight and size, and 1 in solved, of each graph
  uint32_t *sizes;
  uint32_t *solved;
  uint32_t *err;
  uint32_t smem;               // set by the launchers
  Readback rb;                 // at the end of launch_block_single
};
// kind: 0 the large graphs, 1 the middle ones, 2 the small ones.  False if the
// launch was refused (nothing ran).
bool launch_block_batch(const BlockArgs &a, int kind, cudaStream_t s);
// The one graph (n, m) of the arrays; clears *err, bits and writes the forest.
// False as above.
bool launch_block_single(const BlockArgs &a, uint32_t n, uint32_t m, uint32_t *out_ids, uint32_t *out_count,
                         cudaStream_t s);

// single-block base case: the last rounds of a Borůvka call in one launch
constexpr uint32_t BASE_MAX_N = 4096;  // live components (16-bit local ends; shared-memory vertex arrays)
constexpr uint64_t BASE_MAX_M = 6144;  // live edges (fit the tile kernel's shared-memory edge capacity)
struct BaseScratch {
  uint32_t *loc;      // [n] local index of each live component (only those entries are written)
  uint32_t *ends;     // [m] packed local ends
  u64 *cutmin;        // [BASE_MAX_N] all ones (no cut limit)
  u64 *offsets;       // [2]
  uint32_t *plocal;   // [BASE_MAX_N] local root of each live component
  EdgeOut rest;       // [m] edges left between final components (discarded)
  u64 *rest_fill;
};
// False (nothing launched) when the call does not fit the base case.
bool launch_base_case(const uint32_t *act, uint32_t n_act, EdgeList cur, uint64_t m, uint32_t *parent, uint32_t *bits,
                      const BaseScratch &b, uint32_t *err, cudaStream_t s, int filter_heavy, u64 *wsum);
void launch_iota(uint32_t *p, uint64_t n, int sms, cudaStream_t s);

}  // namespace mstgpu

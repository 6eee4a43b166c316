// Device-side data layout and the phase functions of one octree update.
//
// The update of one batch follows Section 5 of the paper, re-planned for a
// GPU that can keep the per-update working set in L2:
//
//  count   every batch point walks from the root to its leaf and is counted
//          there (Section 5.1, "Counting"); the leaf is kept per point (its
//          cursor).
//  decide  per candidate leaf: one whose stored + counted points exceed T
//          splits (Section 5.1, "Splitting"): one spill task per chunk of its
//          stored points. Any other counted leaf is final and gets its chunks
//          now (Section 5.3).
//  hist    the points of the leaves that split (batch points, and the stored
//          points in the old chunks) are counted into the cubes up to 5 levels
//          below their leaf (HIST_DEPTH).
//  build   one block per split leaf sums the counts upwards and creates the
//          whole subtree at once: an inner node wherever a cube holds more
//          than T points. decide then gives its leaves their chunks; a leaf of
//          the lowest level that still holds too many goes round again. The
//          paper deepens the tree one level per counting round, which read
//          every moving point 2.3 times over on a shuffled building scan.
//  claim   with every point at its final leaf, the points sample the grids
//          (Section 3.3) from the leaf's parent upwards. Cells nest: a cell of
//          a node lies inside one cell of the node's parent. So a point whose
//          cell is occupied already is done with every coarser level too, and
//          so is a point that meets a lower arrival index in its cell: that
//          point has the lower index in the coarser cells as well. Most points
//          stop at their first claim, where a walk from the root claimed at
//          every level (4.8 claims a point on a shuffled building scan).
//  store   every point goes to its cursor leaf at the next free slot, and the
//          inner nodes get the chunks of their new voxels; then every new
//          voxel goes to its node (Section 5.4), occupancy bits are set, and
//          the chunks of split leaves return to the pool (Section 3.4).
//
// Voxel claims: the paper lets the first point that finds an empty cell win.
// Here all contenders of an update for a (node, cell) meet in an open-
// addressing table with a 64-bit atomicMin on (gidx << 32 | rgba), so the
// lowest arrival index wins regardless of thread timing. The table entries of
// an update are listed (the backlog of Section 5.2) and cleared by store.
//
// Descents read the node table (first child) from a copy in shared memory of the
// first NODE_CACHE nodes (the node ids of the upper levels are the smallest): the
// plain form's kernels load it, the persistent kernel loads it once and patches it
// after every build with the nodes that split or were created.
// Per-node counters are summed per block in shared memory before they reach
// the global counters (the block tally cache).
#pragma once

#include <cstddef>
#include <cstdint>

#include "simlod.h"

// Namespace of this instance of the device code: the library builds the
// persistent update kernel more than once, with other launch-shape knobs,
// each instance in a namespace of its own (fused_variant.cu).
#ifndef SL_NS
#define SL_NS sl
#endif

namespace SL_NS {

constexpr uint32_t NONE = 0xFFFFFFFFu;
constexpr unsigned long long HASH_EMPTY = ~0ull;
constexpr uint32_t FULL_MASK = 0xFFFFFFFFu;
constexpr int MAX_PROBES = 1 << 14;
constexpr uint32_t REF_BYTES = 256;  // chunk, grid and directory references count 256-byte units
constexpr uint32_t CHUNK_HEADER = 16;
// Launch-shape and algorithm knobs (compile-time; -D overrides them).
#ifndef SL_NODE_CACHE
#define SL_NODE_CACHE 4096
#endif
#ifndef SL_PHASE_BLOCK
#define SL_PHASE_BLOCK 512
#endif
#ifndef SL_PHASE_MIN_BLOCKS
#define SL_PHASE_MIN_BLOCKS 2
#endif
#ifndef SL_COUNT_UNROLL
#define SL_COUNT_UNROLL 2
#endif
#ifndef SL_STORE_UNROLL
#define SL_STORE_UNROLL 2
#endif
#ifndef SL_BLOCK_TALLY
#define SL_BLOCK_TALLY 1
#endif
#ifndef SL_COUNT_CHUNK_MAX
#define SL_COUNT_CHUNK_MAX 2  // log2 of the largest count-phase chunk (4 units)
#endif
#ifndef SL_COUNT_CHUNK_DIV
#define SL_COUNT_CHUNK_DIV 8  // a chunk size keeps at least this many chunks per warp
#endif
constexpr uint32_t NODE_CACHE = SL_NODE_CACHE;         // nodes mirrored in shared memory
constexpr uint32_t ZERO_UNIT = 4096;                   // bytes of grid zeroed per warp unit
constexpr int COUNT_U = SL_COUNT_UNROLL;               // count units a warp carries at a time
#ifndef SL_WBUF
#define SL_WBUF 128
#endif
constexpr uint32_t WBUF = SL_WBUF;                      // new-cell slots staged per warp
constexpr int PHASE_BLOCK = SL_PHASE_BLOCK;            // threads of a phase block
constexpr int PHASE_MIN_BLOCKS = SL_PHASE_MIN_BLOCKS;  // resident blocks per SM they aim for
constexpr uint32_t TALLY_LOG2 = 9;                      // block tally cache: 512 nodes
constexpr uint32_t TALLY_SLOTS = 1u << TALLY_LOG2;
constexpr uint32_t CLAIM_QUEUE = 64;  // points of a warp that wait for their next claim
// dynamic shared memory of the phase blocks: node cache, new-cell staging,
// claim queues, block tally cache
constexpr uint32_t SMEM_WBUF = NODE_CACHE;            // in u32 words
constexpr uint32_t SMEM_QUEUE = SMEM_WBUF + (PHASE_BLOCK / 32) * WBUF * 2;
constexpr uint32_t SMEM_TALLY = SMEM_QUEUE + (PHASE_BLOCK / 32) * CLAIM_QUEUE * 6;
constexpr uint32_t PHASE_SMEM_BYTES = 4 * (SMEM_TALLY + 2 * TALLY_SLOTS);

// Sticky device error bits.
enum : uint32_t {
  E_ARENA = 1u,
  E_NODES = 2u,
  E_SPILL = 4u,
  E_BACKLOG = 8u,
  E_ALLOC_REFS = 16u,
  E_INTERNAL = 32u,
  E_POOL = 64u,
  E_TIMEOUT = 128u,
  E_ITER_CAP = 256u,
};

// Control block at the start of the arena.
// The counters that warps all over the grid change with atomics inside a
// phase (SL_HOT) each start a 128-byte line of their own, so that their
// atomics spread over several L2 slices instead of queueing at one.
#define SL_HOT alignas(128)
// An expansion round of the plain form, whose kernels find here what the ones
// before them left: split entries [s_lo, s_lo + K) are built d levels deep
// below lvl0 levels of earlier rounds, which made `inner` inner nodes; the
// nodes of this round begin at n_lo.
struct PlainRound {
  uint32_t s_lo, K, inner, d, lvl0, n_lo;
};
constexpr uint32_t MAX_ROUNDS = 33;  // from 1; a round builds at least one of 31 levels

struct Ctl {
  unsigned long long base;                  // gidx of the next accepted point
  SL_HOT unsigned long long bump;           // bytes taken from the data region
  unsigned long long chunks_bumped;         // chunks taken from the data region
  SL_HOT unsigned int n_nodes;
  SL_HOT int pool_top;                      // chunk refs in the pool
  unsigned long long bump0;                 // bump at the end of the last update: the grids of
                                            //   nodes that split in this one lie above it
  unsigned int key_rate;                    // expected voxel keys per 1,024 points of an update
  unsigned int open;                        // 1: restored voxels do not nest (see k_check_nested)
  unsigned int error;                       // sticky E_* bits
  unsigned int reject;                      // out-of-cube point seen in this update
  SL_HOT unsigned int spill_count;          // re-inserted points of this update
  SL_HOT unsigned int nkeys;                // new voxels (backlog entries) of this update
  PlainRound round[2];                      // plain form: round r is round[r & 1]
  SL_HOT unsigned int alloc_seq;            // alloc_refs entries of this update
  SL_HOT unsigned int split_count;          // split-list entries of this update
  unsigned int split_inner;                 //   those made by the builds (inner nodes below the
                                            //   split leaves): decide does not change it
  SL_HOT unsigned int ntasks;               // spill tasks (= freed chunks) of this update
  unsigned int split_most;                  // points of the fullest leaf that split so far in this
                                            //   update (hist_depth)
  unsigned int iters;                       // expansion rounds of this update (0: no split)
  unsigned long long st_batches, st_points, st_rejected, st_spilled, st_splits, st_voxels,
      st_iter_max, st_rounds;
  unsigned long long last_points, last_spilled, last_splits, last_voxels, last_iters;
  unsigned long long st_rejected_async;  // rejections inside fused launches
  SL_HOT unsigned long long render_samples;  // points and voxels visited by the last render
  unsigned int vis_count;                    // nodes drawn by the last render
  unsigned int draw_units;                   // chunks and array pieces they were cut into
  unsigned long long phase_ns[8];        // fused form: time per phase (see PH_*)
  unsigned long long st_compacted;       // nodes turned into arrays (simlod_compact), in all
  unsigned long long st_compact_chunks;  // chunks those nodes gave back to the pool
  unsigned long long st_decompacted;     // arrays turned back into chunk lists by an insert
  unsigned long long compact_now;        // nodes that are arrays now
  unsigned long long compact_chunks_now; // chunks those arrays stand in for
  unsigned long long compact_need;       // bytes the candidates of a compaction need
  unsigned long long compact_from;       // the bump pointer before it
  unsigned int store_blocks;             // plain form: blocks that finished the store
};
#undef SL_HOT
static_assert(sizeof(Ctl) % 16 == 0, "Ctl size");

// Phases of the fused form, for its phase clock.
enum : int { PH_COUNT = 0, PH_DECIDE, PH_ADVANCE, PH_STORE, PH_END, PH_CLAIM, PH_LAUNCH, PH_OTHER };

// Per-node metadata that the descents do not touch.
struct NodeMeta {
  int32_t min[3];
  uint32_t level;
  uint32_t n_chunks;
  uint32_t head, tail;  // chunk list (points of a leaf, voxels of an inner node)
  uint32_t dir;         // chunk directory of a leaf (ref), NONE if none
  uint32_t st_nch;      // store map of the current update: chunks before allocation,
  uint32_t st_tail;     //   the tail before allocation,
  uint32_t st_seq;      //   first alloc_refs entry of the newly allocated chunks,
  uint32_t st_base;     //   and the records stored before this update
  uint32_t touched;     // updates applied when the node last received records (1 = the first)
  uint32_t compact;     // 1: the records are one contiguous array (head), not a chunk list
  uint32_t up;          // parent | parent's level << NODE_BITS, NONE at the root
  uint32_t up_grid;     // the parent's occupancy grid
};
static_assert(sizeof(NodeMeta) == 64, "NodeMeta size");
static_assert(offsetof(NodeMeta, st_nch) == 32 && offsetof(NodeMeta, st_base) == 44,
              "the store map is one aligned 16-byte load");
static_assert(offsetof(NodeMeta, up) == 56, "up and up_grid are one aligned 8-byte load");

constexpr uint32_t NODE_BITS = 27;  // node ids below 2^27 (the node table limit)
constexpr uint32_t NODE_MASK = (1u << NODE_BITS) - 1u;

struct __align__(16) HSlot {
  unsigned long long key;  // (node << 3G) | cell, HASH_EMPTY when free
  unsigned long long val;  // (gidx << 32) | rgba of the best contender so far
};

// A leaf to split is marked in its store cursor (scur, unused until the store
// phase): SPLIT_MARK | its log2 size << SPLIT_BITS | its split-list entry.
constexpr uint32_t SPLIT_MARK = 1u << 31;
constexpr uint32_t SPLIT_BITS = 26;  // split-list entries: at most max_nodes / 8 + 1


// The stored points of one chunk of a split leaf, re-inserted this update:
// point q of the chunk is spill entry dst + q.
struct SpillTask {
  uint32_t ref;   // the chunk
  uint32_t node;  // the leaf that split
  uint32_t dst;   // first spill entry
  uint32_t n;     // points in the chunk
};

// Everything a phase needs: arena pointers and the configuration.
struct Ctx {
  Ctl* ctl;
  uint32_t* child;    // first child id or NONE (leaf), per node
  uint32_t* gridref;  // occupancy grid ref or NONE, per node
  uint32_t* cnt;      // per-update counter: new points (leaf) or new voxels (inner)
  uint32_t* num;      // stored points (leaf) or voxels (inner)
  NodeMeta* meta;
  uint32_t* pool;
  uint32_t* pending;  // chunk refs freed by this update's splits (one per task)
  uint32_t* alloc_refs;
  uint32_t* splits;   // nodes that split in this update
  SpillTask* tasks;
  uint32_t* sp_cur;   // per re-inserted point: final leaf
  uint32_t* b_cur;    // per batch point: leaf of the descent, then final leaf
  uint32_t* scur;     // per node: store cursor of the current update
  uint32_t* hist;     // counts of the cubes below split leaves; zero between updates
  uint32_t* hist_up;  //   their sums per inner level, and the list of inner nodes
  HSlot* hash;
  uint2* keys;        // backlog: table slot and node of this update's first key_nodes new
                      //   cells, behind them the slots of the others
  uint8_t* data;
  unsigned long long data_bytes;
  int4* staging;
  int32_t rmin[3];
  uint32_t rlog2, T, C, G;
  uint32_t chunk_bytes, chunk_units, grid_bytes, dir_bytes, dir_cap;
  uint32_t hash_mask;
  uint32_t C_mul, C_shift;  // division by C (div_by)
  uint32_t parts, P_mul, P_shift;  // 32-record units per chunk, and division by them
  uint32_t chunk_lim, grid_lim;    // first references whose chunk or grid would not fit
  uint32_t max_nodes, max_chunks, spill_cap, backlog_cap, key_nodes, max_splits;
  uint64_t max_batch;
  uint64_t hist_words;
  unsigned long long* launch_bar;  // barrier word of the persistent launch (abort bit)
  unsigned long long bar_ns;       // persistent launch: time limit of one grid-barrier wait
  unsigned long long ready_ns;     //   and of one wait for a batch's ready flag
  unsigned int* progress;          // persistent launch: host-mapped words, [0] batches finished,
                                   //   [1] batches dropped by budget stops (nullptr: none)
};

// Abort bit of a persistent launch's barrier word: set with the first
// device error, so that every block leaves at its next barrier.
constexpr unsigned long long BAR_ABORT = 1ull << 63;

// ------------------------------------------------------------------ helpers

// First thing in a kernel that may be launched before the one in front of it
// has ended (launch_next): let the kernel behind be placed too, then wait until
// the one in front has ended and its writes are visible. Returns at once in a
// kernel that was launched the plain way.
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}

template <typename T>
__device__ __forceinline__ T vload(const T* p) {
  return *reinterpret_cast<const volatile T*>(p);
}

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

__device__ __forceinline__ void set_error(const Ctx& c, uint32_t bits) {
  atomicOr(&c.ctl->error, bits);
  atomicOr(c.launch_bar, BAR_ABORT);
}

// All 32 lanes call and get one answer: a device error has left the octree half
// updated (the host learns of it at its next look at the control block).
__device__ __forceinline__ bool update_failed(const Ctx& c) {
  return __any_sync(FULL_MASK, vload(&c.ctl->error) != 0u);
}

// n / d for any 32-bit n: multiply, add and shift by the constants that Granlund
// and Montgomery ("Division by invariant integers using multiplication", 1994)
// give for a divisor (div_constants).
__device__ __forceinline__ uint32_t div_by(uint32_t n, uint32_t d, uint32_t mul, uint32_t shift) {
  if (d == 1u) return n;
  const uint32_t t = __umulhi(mul, n);
  return (t + ((n - t) >> 1)) >> shift;
}

inline void div_constants(uint32_t d, uint32_t* mul, uint32_t* shift) {  // d >= 1
  uint32_t l = 0;
  while ((1ull << l) < d) ++l;
  *mul = (uint32_t)(((1ull << 32) * ((1ull << l) - d)) / d + 1ull);
  *shift = l ? l - 1u : 0u;
}

__device__ __forceinline__ uint8_t* ref_ptr(const Ctx& c, uint32_t ref) {
  return c.data + (size_t)ref * REF_BYTES;
}

__device__ __forceinline__ uint32_t* chunk_next(const Ctx& c, uint32_t ref) {
  return reinterpret_cast<uint32_t*>(ref_ptr(c, ref));
}

__device__ __forceinline__ int4* chunk_recs(const Ctx& c, uint32_t ref) {
  return reinterpret_cast<int4*>(ref_ptr(c, ref) + CHUNK_HEADER);
}

__device__ __forceinline__ uint32_t* chunk_aux(const Ctx& c, uint32_t ref) {
  return reinterpret_cast<uint32_t*>(ref_ptr(c, ref) + CHUNK_HEADER + 16u * c.C);
}

// A compacted node's records: one array in the data region, a chunk header
// (next = NONE, then the capacity) followed by cap records and cap aux words,
// the layout of a chunk of cap records.
__device__ __forceinline__ int4* array_recs(const Ctx& c, uint32_t ref) {
  return reinterpret_cast<int4*>(ref_ptr(c, ref) + CHUNK_HEADER);
}

__device__ __forceinline__ uint32_t* array_aux(const Ctx& c, uint32_t ref, uint32_t cap) {
  return reinterpret_cast<uint32_t*>(ref_ptr(c, ref) + CHUNK_HEADER + 16ull * cap);
}

__device__ __forceinline__ unsigned long long array_bytes(uint32_t cap) {
  return ((CHUNK_HEADER + 20ull * cap) + REF_BYTES - 1) / REF_BYTES * REF_BYTES;
}

// A reference that stays inside the data region for `bytes` bytes.
__device__ __forceinline__ bool ref_ok(const Ctx& c, uint32_t ref, uint32_t bytes) {
  return ref != NONE && (unsigned long long)ref * REF_BYTES + bytes <= c.data_bytes;
}

// References below these limits hold a whole chunk or grid (NONE never does).
__device__ __forceinline__ bool chunk_ok(const Ctx& c, uint32_t ref) { return ref < c.chunk_lim; }
__device__ __forceinline__ bool grid_ok(const Ctx& c, uint32_t ref) { return ref < c.grid_lim; }

// An array of cap records at ref stays inside the data region.
__device__ __forceinline__ bool array_ok(const Ctx& c, uint32_t ref, uint32_t cap) {
  return ref != NONE && (unsigned long long)ref * REF_BYTES + array_bytes(cap) <= c.data_bytes;
}

__device__ __forceinline__ uint32_t* grid_words(const Ctx& c, uint32_t ref) {
  return reinterpret_cast<uint32_t*>(ref_ptr(c, ref));
}

__device__ __forceinline__ uint32_t* dir_entries(const Ctx& c, uint32_t ref) {
  return reinterpret_cast<uint32_t*>(ref_ptr(c, ref));
}

// Coordinates relative to the root minimum; false when outside the root cube.
// The cube lies in the int32 range and its side is at most 2^31, so the
// wrapped 32-bit difference is below the side exactly for the points inside.
__device__ __forceinline__ bool rel_coords(const Ctx& c, int4 p, uint32_t& rx, uint32_t& ry,
                                           uint32_t& rz) {
  rx = (uint32_t)p.x - (uint32_t)c.rmin[0];
  ry = (uint32_t)p.y - (uint32_t)c.rmin[1];
  rz = (uint32_t)p.z - (uint32_t)c.rmin[2];
  return ((rx | ry | rz) >> c.rlog2) == 0u;
}

// Octant of a point inside a node of side 2^L (L >= 1): bit L-1 per axis.
__device__ __forceinline__ uint32_t octant(uint32_t rx, uint32_t ry, uint32_t rz, uint32_t L) {
  uint32_t s = L - 1u;
  return ((rx >> s) & 1u) | (((ry >> s) & 1u) << 1) | (((rz >> s) & 1u) << 2);
}

// Cell of a point in the 2^G grid of a node of side 2^L (L <= 31): per axis
// ((p - min) << G) >> L, where p - min is the low L bits of the root-relative
// coordinate (Section 3.3); the result's G bits are those of r shifted by
// L - G, whichever way.
__device__ __forceinline__ uint32_t cell_index(uint32_t rx, uint32_t ry, uint32_t rz, uint32_t L,
                                               uint32_t G) {
  const uint32_t m = (1u << G) - 1u;
  if (L >= G) {
    const uint32_t sh = L - G;
    return ((rx >> sh) & m) | (((ry >> sh) & m) << G) | (((rz >> sh) & m) << (2u * G));
  }
  const uint32_t sh = G - L;
  return ((rx << sh) & m) | (((ry << sh) & m) << G) | (((rz << sh) & m) << (2u * G));
}

// ------------------------------------------------------- node-table cache

// Shared-memory copy of child[] for nodes [0, NODE_CACHE).
struct NodeCache {
  uint32_t* child;
  uint32_t n;  // cached nodes
};

// The cache of the first min(n_nodes, NODE_CACHE) nodes in `smem`.
__device__ __forceinline__ NodeCache node_cache_at(uint32_t* smem, uint32_t n_nodes) {
  NodeCache nc;
  nc.child = smem;
  nc.n = n_nodes < NODE_CACHE ? n_nodes : NODE_CACHE;
  return nc;
}

// The whole block copies nodes [lo, hi) (those below NODE_CACHE) into the
// cache. The caller synchronises the block before the cache is read.
__device__ __forceinline__ void node_cache_load(const Ctx& c, uint32_t* smem, uint32_t lo,
                                                uint32_t hi) {
  hi = hi < NODE_CACHE ? hi : NODE_CACHE;
  for (uint32_t i = lo + threadIdx.x; i < hi; i += blockDim.x) smem[i] = c.child[i];
}

// The whole block brings the cache up to date after a build: the nodes of the
// split entries [s_lo, s_hi) became inner, the nodes [n_lo, n_hi) were
// created. Nothing else in the node table changes during an update. The caller
// synchronises.
__device__ __forceinline__ void node_cache_patch(const Ctx& c, uint32_t* smem, uint32_t s_lo,
                                                 uint32_t s_hi, uint32_t n_lo, uint32_t n_hi) {
  for (uint32_t e = s_lo + threadIdx.x; e < s_hi; e += blockDim.x) {
    const uint32_t id = c.splits[e];
    if (id < NODE_CACHE) smem[id] = c.child[id];
  }
  node_cache_load(c, smem, n_lo, n_hi);
}

// The whole block empties the block tally cache (at the start of a phase,
// before a block barrier).
__device__ __forceinline__ void tally_init(uint32_t* smem) {
  for (uint32_t i = threadIdx.x; i < TALLY_SLOTS; i += blockDim.x) {
    smem[SMEM_TALLY + i] = NONE;
    smem[SMEM_TALLY + TALLY_SLOTS + i] = 0;
  }
}

// ------------------------------------------------------ block tally cache
//
// Per-update counters (points counted into a leaf or a cube below a split
// leaf, new voxels of an inner node) are summed per block in shared memory
// first: a direct-mapped table of TALLY_SLOTS (index, count) pairs. An index
// whose slot holds another one goes to the global counter at once. Dense
// regions send thousands of warps to the same few counters; the cache turns
// their global atomics, which serialise at one L2 slice, into one per block
// and counter.

__device__ __forceinline__ void tally_add(uint32_t* counters, uint32_t* smem, uint32_t i,
                                          uint32_t k) {
#if SL_BLOCK_TALLY
  const uint32_t slot = (i * 0x9E3779B1u) >> (32u - TALLY_LOG2);
  uint32_t* tn = smem + SMEM_TALLY;
  const uint32_t old = tn[slot] == i ? i : atomicCAS(tn + slot, NONE, i);
  if (old == NONE || old == i) {
    atomicAdd(tn + TALLY_SLOTS + slot, k);
    return;
  }
#endif
  atomicAdd(counters + i, k);
}

// The whole block calls at the end of a phase: add the cached counts to the
// global counters.
__device__ __forceinline__ void tally_flush(uint32_t* counters, uint32_t* smem) {
#if SL_BLOCK_TALLY
  __syncthreads();
  const uint32_t* tn = smem + SMEM_TALLY;
  for (uint32_t i = threadIdx.x; i < TALLY_SLOTS; i += blockDim.x) {
    const uint32_t at = tn[i], k = tn[TALLY_SLOTS + i];
    if (at != NONE && k) atomicAdd(counters + at, k);
  }
#endif
}

__device__ __forceinline__ uint32_t node_child(const Ctx& c, NodeCache nc, uint32_t id) {
  return id < nc.n ? nc.child[id] : c.child[id];
}

// -------------------------------------------------------- voxel claims

// Key and value of a claim-table slot in one 16-byte load. Within an update
// a slot's value only decreases once its key is set (the store phase empties
// the slots between updates), so a value read with the key bounds the current
// one from above.
__device__ __forceinline__ ulonglong2 slot_load(const HSlot* s) {
  ulonglong2 kv;
  asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];"
               : "=l"(kv.x), "=l"(kv.y)
               : "l"(s)
               : "memory");
  return kv;
}

// Put (key, val) into an empty slot with one 16-byte compare-and-swap; returns
// what the slot held. (An 8-byte one on the key and a minimum on the value are
// one more atomic on a scattered line, and leave a moment in which the key is
// there without its value: claims 0.78 against 0.82 ms on a 16M-point terrain,
// 1.37 against 1.45 ms on a 40M-point building scan.)
__device__ __forceinline__ ulonglong2 slot_cas(HSlot* s, unsigned long long key,
                                               unsigned long long val) {
  ulonglong2 o;
  asm volatile(
      "{\n\t.reg .b128 cmp, swp, old;\n\t"
      "mov.b128 cmp, {%2, %2};\n\t"
      "mov.b128 swp, {%3, %4};\n\t"
      "atom.relaxed.gpu.global.cas.b128 old, [%5], cmp, swp;\n\t"
      "mov.b128 {%0, %1}, old;\n\t}"
      : "=l"(o.x), "=l"(o.y)
      : "l"(HASH_EMPTY), "l"(key), "l"(val), "l"(s)
      : "memory");
  return o;
}

// The claim table of one update. A key (node << 3G | cell) is looked for along
// a fixed sequence of slots: CLAIM_NEAR of them in the table's first near + 1
// slots, as many as the update's expected keys call for, then in the whole
// table (two slots per backlog entry, whatever the data). So the updates
// of a stream use the same lines again, which stay in L2, where a table sized
// for the largest update took new lines from DRAM every time: claims of a
// uniform stream of 500k batches 0.90 against 1.27 ms a pass, of a shuffled
// building scan 1.20 against 1.40 ms.
// Cells that differ in the low CLAIM_BUCKET bits of their x sit in one bucket
// of 8 neighbouring slots (128 bytes), because the cells that a warp claims
// are neighbours (a 16M-point terrain: 0.69 against 0.94 ms). The bucket is
// the top bits of (key without those bits) * 2^64 / phi. The near step is odd,
// so that a sequence reaches every slot, and one more than a bucket, so that
// keys that meet do not fill each other's buckets (0.69 against 0.82 ms with
// the next slot); the far step is an odd part of the hash, which leaves the
// full near part at once. Where a key sits does not change which point wins.
constexpr uint32_t CLAIM_BUCKET = 3;
constexpr uint32_t CLAIM_LOW = (1u << CLAIM_BUCKET) - 1u;
constexpr uint32_t CLAIM_STEP = (1u << CLAIM_BUCKET) + 1u;
constexpr int CLAIM_NEAR = 16;

__device__ __forceinline__ uint32_t claim_slot(unsigned long long key, uint32_t mask) {
  const uint32_t top =
      (uint32_t)(((key >> CLAIM_BUCKET) * 0x9E3779B97F4A7C15ull) >> 32) >> __clz(mask);
  return ((top & ~CLAIM_LOW) | ((uint32_t)key & CLAIM_LOW)) & mask;  // (mask > 0)
}

// The near mask of an update of n points, batch and re-inserted, that is
// expected to make `rate` / 1024 keys per point (Ctl::key_rate): 6 to 12
// slots per expected key. (Fewer lengthen the probes, more leave L2: 0.5, 1,
// 2 and 4 slots per point took 1.26, 1.20, 1.31 and 1.34 ms on the building
// scan with 0.11 keys per point, 2 and 4 took 1.80 and 1.09 ms on the uniform
// stream with 1.4.)
__device__ __forceinline__ uint32_t claim_near_mask(const Ctx& c, uint64_t n, uint32_t rate) {
  const uint64_t want = n * rate * 6u / 1024u;
  if (want > c.hash_mask) return c.hash_mask;
  return want <= 1024u ? (c.hash_mask < 1023u ? c.hash_mask : 1023u)
                       : FULL_MASK >> __clz((uint32_t)want - 1u);
}

// Probes after the first for `key` (slot h held another key). CLAIM_NEW, with
// the slot in h: this call put the key into the table (the cell is new in this
// update); CLAIM_LOWERED: the slot held the key with a larger value;
// CLAIM_BEATEN: it holds a lower one.
enum : int { CLAIM_NEW = 0, CLAIM_LOWERED, CLAIM_BEATEN };

__device__ int hash_claim_rest(const Ctx& c, unsigned long long key, unsigned long long val,
                               uint32_t near, uint32_t& h) {
  uint32_t mask = near, step = CLAIM_STEP;
  for (int probe = 1; probe < MAX_PROBES; ++probe) {
    h = (h + step) & mask;
    if (probe == CLAIM_NEAR) {
      mask = c.hash_mask;
      h = claim_slot(key, mask);
      step = (uint32_t)(key * 0x9E3779B97F4A7C15ull >> 16) | 1u;
    }
    HSlot* s = c.hash + h;
    const ulonglong2 kv = slot_load(s);
    unsigned long long k = kv.x, v = kv.y;
    if (k == HASH_EMPTY) {
      const ulonglong2 o = slot_cas(s, key, val);
      k = o.x;
      v = o.y;
      if (k == HASH_EMPTY) return CLAIM_NEW;
    }
    if (k == key) {
      if (v < val) return CLAIM_BEATEN;
      atomicMin(&s->val, val);
      return CLAIM_LOWERED;
    }
  }
  set_error(c, E_BACKLOG);
  return CLAIM_BEATEN;
}

// ------------------------------------------------ lane runs (warp groups)
//
// Lanes that hold the same value in a contiguous run of participating lanes
// form one group: one shuffle and two ballots, instead of a match over the
// whole warp. Equal values in separate runs form separate groups, which every
// caller tolerates (more groups, same result: counts and slot reservations
// add up, claims of one cell meet again in the table). The points a warp
// holds are neighbours in the stream, so equal nodes and cells mostly sit in
// runs.
struct LaneRun {
  bool head;       // this lane starts its run
  uint32_t first;  // the lane that starts this lane's run
  uint32_t end;    // one past the run's last lane
};

__device__ __forceinline__ unsigned lanes_upto(uint32_t lane) {
  return lane == 31u ? FULL_MASK : (2u << lane) - 1u;
}

// All 32 lanes call; lanes without `on` take part in no run.
template <typename T>
__device__ __forceinline__ LaneRun lane_run(bool on, T v) {
  const uint32_t lane = lane_id();
  const unsigned onm = __ballot_sync(FULL_MASK, on);
  const T prev = __shfl_up_sync(FULL_MASK, v, 1);
  const bool head = on && !(lane > 0u && ((onm >> (lane - 1u)) & 1u) && prev == v);
  const unsigned heads = __ballot_sync(FULL_MASK, head);
  LaneRun r;
  r.head = head;
  const unsigned below = heads & lanes_upto(lane);
  r.first = below ? 31u - (uint32_t)__clz(below) : lane;
  const unsigned breaks = (heads | ~onm) & ~lanes_upto(r.first);
  r.end = breaks ? (uint32_t)__ffs(breaks) - 1u : 32u;
  return r;
}

// The slot of backlog entry e (the arena may leave no room for all entries' nodes).
__device__ __forceinline__ uint32_t* key_slot(const Ctx& c, uint32_t e) {
  return e < c.key_nodes ? &c.keys[e].x
                         : reinterpret_cast<uint32_t*>(c.keys + c.key_nodes) + (e - c.key_nodes);
}

// Per-warp staging of the table slots of new cells (shared memory), flushed
// to the backlog with one atomic per flush.
struct WarpBuf {
  uint2* buf;      // WBUF entries (slot, node) of this warp
  uint32_t n;      // staged entries (the same value in every lane)
  uint32_t* smem;  // the block's dynamic shared memory (tally cache)
};

__device__ __forceinline__ WarpBuf warp_buf(uint32_t* smem) {
  WarpBuf wb;
  wb.buf = reinterpret_cast<uint2*>(smem + SMEM_WBUF) + (threadIdx.x / 32) * WBUF;
  wb.n = 0;
  wb.smem = smem;
  return wb;
}

// All 32 lanes call: append the staged slots to the backlog.
__device__ __forceinline__ void warp_flush(const Ctx& c, WarpBuf& wb) {
  if (wb.n == 0u) return;
  __syncwarp();
  uint32_t e0 = 0;
  if (lane_id() == 0) e0 = atomicAdd(&c.ctl->nkeys, wb.n);
  e0 = __shfl_sync(FULL_MASK, e0, 0);
  for (uint32_t k = lane_id(); k < wb.n; k += 32) {
    const uint32_t e = e0 + k;
    const uint2 at = wb.buf[k];  // slot, node
    if (e < c.key_nodes) c.keys[e] = at;
    else if (e < c.backlog_cap) *key_slot(c, e) = at.x;
    else set_error(c, E_BACKLOG);
  }
  wb.n = 0;
  __syncwarp();
}

// All 32 lanes call. Lanes with `lead` offer val for key (a cell of `node`) to the
// update's claim table, where the lowest value wins. A key new in this update is
// staged for the backlog and counted towards its node's new voxels. `on` becomes
// true in lanes that met no lower value.
__device__ __forceinline__ void warp_claim(const Ctx& c, WarpBuf& wb, bool lead,
                                           unsigned long long key, unsigned long long val,
                                           uint32_t node, uint32_t near, bool& on) {
  const uint32_t lane = lane_id();
  uint32_t h = claim_slot(key, near);
  bool inst = false;
  if (lead) {
    ulonglong2 kv = slot_load(c.hash + h);
    const bool cas = kv.x == HASH_EMPTY;
    if (cas) kv = slot_cas(c.hash + h, key, val);
    if (cas && kv.x == HASH_EMPTY) {
      inst = on = true;
    } else if (kv.x == key) {
      if (kv.y > val) {
        on = true;
        atomicMin(&c.hash[h].val, val);
      }
    } else {
      const int got = hash_claim_rest(c, key, val, near, h);
      inst = got == CLAIM_NEW;
      if (got != CLAIM_BEATEN) on = true;
    }
  }
  const unsigned mi = __ballot_sync(FULL_MASK, inst);
  if (mi == 0u) return;
  const uint32_t ni = (uint32_t)__popc(mi);
  if (wb.n + ni > WBUF) warp_flush(c, wb);
  const LaneRun r = lane_run(inst, node);
  if (inst) {
    wb.buf[wb.n + __popc(mi & ((1u << lane) - 1u))] = make_uint2(h, node);
    if (r.head) tally_add(c.cnt, wb.smem, node, r.end - lane);
  }
  wb.n += ni;
}

// All 32 lanes call. Lanes with `valid` add one to counters[i] (one addition
// per run of equal counters).
__device__ __forceinline__ void warp_tally(uint32_t* counters, uint32_t* smem, bool valid,
                                           uint32_t i) {
  const LaneRun r = lane_run(valid, i);
  if (valid && r.head) tally_add(counters, smem, i, r.end - lane_id());
}

// The k-th 32-item unit of a phase that a warp handles: chunks of 2^chl
// consecutive units are dealt out to the warps in turn (chunk q to warp q mod
// nwarps), so that a warp's units are neighbours in the stream while the work
// stays spread over the grid.
__device__ __forceinline__ uint32_t warp_unit(uint32_t warp0, uint32_t nwarps, uint32_t k,
                                              uint32_t chl) {
  return ((warp0 + (k >> chl) * nwarps) << chl) + (k & ((1u << chl) - 1u));
}

// log2 of the count phase's chunk for `units` units: the largest power of two
// up to 2^SL_COUNT_CHUNK_MAX that still leaves SL_COUNT_CHUNK_DIV chunks per
// warp. Chunks of neighbouring points let a warp's descents and claims share
// nodes and cells (measured on the clustered stream: 15.1 against 18.7 ms of
// count phase with chunks of 4); batches too small to give every warp several
// chunks keep single units (1M-point batches slowed down with chunks of 8).
__device__ __forceinline__ uint32_t count_chunk_log2(uint32_t units, uint32_t nwarps) {
  uint32_t chl = 0;
  while (chl < SL_COUNT_CHUNK_MAX &&
         units >= (uint64_t)(nwarps * SL_COUNT_CHUNK_DIV) << (chl + 1))
    ++chl;
  return chl;
}

// ------------------------------------------------------------ phase: count1

// Iteration 1 for the batch points [0, n): descend and count. `smem` holds
// PHASE_SMEM_BYTES of dynamic shared memory. Every block first writes down where
// the top JUMP levels lead each of their 8^JUMP cubes to (node | level <<
// NODE_BITS, in the queue region): a point's first steps are one lookup.
constexpr uint32_t JUMP = 3;
static_assert((1u << (3u * JUMP)) <= (PHASE_BLOCK / 32) * CLAIM_QUEUE * 6, "the jump table fits");
__device__ void phase_count1(const Ctx& c, uint32_t* smem, const NodeCache nc, const int4* pts,
                             uint32_t n, uint32_t warp0, uint32_t nwarps) {
  constexpr int U = COUNT_U;
  tally_init(smem);
  __syncthreads();  // also publishes the caller's node-cache writes
  uint32_t* jump = smem + SMEM_QUEUE;
  const uint32_t jl = c.rlog2 < JUMP ? c.rlog2 : JUMP, top = c.rlog2 - jl;
  for (uint32_t t = threadIdx.x; t < (1u << (3u * jl)); t += blockDim.x) {
    const uint32_t m = (1u << jl) - 1u;
    uint32_t node = 0, lvl = 0;
    for (uint32_t ch = node_child(c, nc, 0u); ch != NONE && lvl < jl && ch + 8u <= c.max_nodes;
         ch = node_child(c, nc, node)) {
      node = ch + octant(t & m, (t >> jl) & m, t >> (2u * jl), jl - lvl);
      ++lvl;
    }
    jump[t] = node | (lvl << NODE_BITS);
  }
  __syncthreads();
  const uint32_t lane = lane_id();
  // each warp carries U units of 32 points (warp_unit k, k + 1, ...) at a
  // time so that their descents overlap; the next units' points are loaded
  // while the current ones descend
  const uint32_t chl = count_chunk_log2((n + 31) / 32, nwarps);
  int4 pn[U];
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const uint32_t i = warp_unit(warp0, nwarps, j, chl) * 32 + lane;
    pn[j] = i < n ? __ldcg(pts + i) : make_int4(0, 0, 0, 0);
  }
  for (uint32_t k0 = 0; warp_unit(warp0, nwarps, k0, chl) * 32 < n; k0 += U) {
    bool valid[U], walking[U];
    uint32_t rx[U], ry[U], rz[U], node[U], L[U];
    uint32_t iu[U];
    bool any = false;
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const uint32_t i = warp_unit(warp0, nwarps, k0 + j, chl) * 32 + lane;
      iu[j] = i;
      valid[j] = i < n;
      const int4 p = pn[j];
      const uint32_t inext = warp_unit(warp0, nwarps, k0 + j + U, chl) * 32 + lane;
      pn[j] = inext < n ? __ldcg(pts + inext) : make_int4(0, 0, 0, 0);
      if (!rel_coords(c, p, rx[j], ry[j], rz[j]) && valid[j]) {
        atomicOr(&c.ctl->reject, 1u);
        valid[j] = false;
      }
      const uint32_t e = valid[j] ? jump[(rx[j] >> top) | ((ry[j] >> top) << jl) |
                                         ((rz[j] >> top) << (2u * jl))]
                                  : 0u;
      node[j] = e & NODE_MASK;
      L[j] = c.rlog2 - (e >> NODE_BITS);
      walking[j] = valid[j];
      any = any || walking[j];
    }
    while (any) {
      any = false;
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if (!walking[j]) continue;
        const uint32_t ch = node_child(c, nc, node[j]);
        if (ch == NONE) {
          walking[j] = false;
        } else if (ch + 8u > c.max_nodes || L[j] == 0u) {
          set_error(c, E_INTERNAL);
          walking[j] = false;
        } else {
          node[j] = ch + octant(rx[j], ry[j], rz[j], L[j]);
          --L[j];
          any = true;
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < U; ++j) {
      warp_tally(c.cnt, smem, valid[j], node[j]);
      if (valid[j]) c.b_cur[iu[j]] = node[j];
    }
  }
  tally_flush(c.cnt, smem);
}

// -------------------------------------------------------- phase: histogram

// The spill tasks as units of 32 re-inserted points (a unit never crosses into
// the next task).
// Lane's re-inserted point of unit u of the tasks [0, t_hi): its task, its
// place in the task's chunk; false past the end of the task.
__device__ __forceinline__ bool task_point(const Ctx& c, uint32_t u, SpillTask& tk, uint32_t& q) {
  const uint32_t t = div_by(u, c.parts, c.P_mul, c.P_shift);
  q = (u - t * c.parts) * 32u + lane_id();
  tk = c.tasks[t];
  if (!chunk_ok(c, tk.ref) || tk.n > c.C || tk.node >= c.max_nodes ||
      (unsigned long long)tk.dst + tk.n > c.spill_cap) {
    if (lane_id() == 0) set_error(c, E_INTERNAL);
    return false;
  }
  return q < tk.n;
}

// From `node` down to the leaf that holds the point now.
__device__ __forceinline__ uint32_t walk_down(const Ctx& c, NodeCache nc, uint32_t node,
                                              uint32_t rx, uint32_t ry, uint32_t rz) {
  uint32_t ch = node_child(c, nc, node);
  if (ch == NONE) return node;
  uint32_t L = c.rlog2 - c.meta[node].level;
  while (ch != NONE) {
    if (ch + 8u > c.max_nodes || L == 0u) {
      set_error(c, E_INTERNAL);
      break;
    }
    node = ch + octant(rx, ry, rz, L);
    --L;
    ch = node_child(c, nc, node);
  }
  return node;
}

// Bits of a 5-bit number, two zeros between them.
__device__ __forceinline__ uint32_t spread5(uint32_t x) {
  x = (x | (x << 8)) & 0x100Fu;
  x = (x | (x << 4)) & 0x10C3u;
  return (x | (x << 2)) & 0x1249u;
}

// Levels below a split leaf that one histogram covers, for K leaves of `most`
// points at most, of an update of n points: 3, one more for every factor of 4
// that the fullest leaf is over T (points lie on surfaces: four children out
// of eight), at most HIST_DEPTH and a count per moving point. A leaf that is
// not deep enough yet goes round again, which reads the points once more. That
// round keeps the update's fullest leaf for `most`, so that it goes as deep and
// is mostly the last (with the leaves of the round itself: a building scan of
// 120M points 12.28 against 12.34 ms and mixed batches 2.89 against 2.92, but one
// of 12M points 1.67 against 1.65 and a z-ordered one 0.860 against 0.848). 5
// levels for every leaf cost more counts than that saves (terrain: build 0.30
// against 0.11 ms a pass; mixed batches: histogram 0.68 against 0.51 ms), 1 and
// 2 levels more than the factors took a second round too often (clustered
// scan: 1.72 and 1.57 against 1.50 ms). A leaf of more than 2^HIST_WIDE times T
// points gets 3 levels again: its subtree would be thousands of nodes, which one
// block would write (2M even points into leaves of 100: 0.08 against 0.34 ms).
// hist_words has room for one level.
constexpr uint32_t HIST_DEPTH = 5, HIST_WIDE = 9;
__host__ __device__ __forceinline__ uint32_t hist_depth(const Ctx& c, uint32_t K, uint64_t n,
                                                        uint32_t most) {
  const uint64_t want = n < 32768u ? 32768u : n;
  const uint64_t lim = want < c.hist_words ? want : c.hist_words;
  uint32_t aim = 3, d = 1;
  while (aim < HIST_DEPTH && ((unsigned long long)c.T << (2u * (aim - 2u))) < most) ++aim;
  if ((most >> HIST_WIDE) > c.T) aim = 3;
  while (d < aim && ((uint64_t)K << (3u * (d + 1u))) <= lim) ++d;
  return d;
}

// Count the points of the leaves in the split entries [s_lo, s_lo + K) into
// the cubes d levels below (hist[entry][Morton index]). In the first round a
// point's cursor is its leaf; later the leaf is looked up (only leaves of the
// lowest level of the round before split again, which is rare).
__device__ void phase_hist(const Ctx& c, uint32_t* smem, const NodeCache nc, const int4* pts,
                           uint32_t n, uint32_t t_hi, uint32_t s_lo, uint32_t K, uint32_t d,
                           bool first) {
  tally_init(smem);
  __syncthreads();  // also publishes the caller's node-cache writes
  if (((uint64_t)K << (3u * d)) > c.hist_words) {
    if (blockIdx.x == 0 && threadIdx.x == 0) set_error(c, E_INTERNAL);
    return;  // (the same in every thread)
  }
  const uint32_t lane = lane_id();
  const uint32_t us = t_hi * c.parts, units = us + (n + 31u) / 32u;
  // every block takes one range of neighbouring units: its points fall into
  // few cubes, whose counts its tally cache adds up (a shuffled building scan
  // of 40M points: 1.03 against 1.47 ms a pass with the units dealt out)
  const uint32_t per = (units + gridDim.x - 1u) / gridDim.x;
  const uint32_t last = (blockIdx.x + 1u) * per, end = last < units ? last : units;
  for (uint32_t w = blockIdx.x * per + threadIdx.x / 32u; w < end; w += blockDim.x / 32) {
    bool on = false, have = false;
    uint32_t cur = 0;
    uint32_t i = 0;
    int4 p = make_int4(0, 0, 0, 0);
    if (w < us) {
      SpillTask tk;
      uint32_t q;
      on = have = task_point(c, w, tk, q);
      if (on) {
        p = chunk_recs(c, tk.ref)[q];
        cur = tk.node;
      }
    } else {
      i = (w - us) * 32 + lane;
      on = i < n;
      cur = on ? c.b_cur[i] : 0u;
    }
    uint32_t rx = 0, ry = 0, rz = 0;
    if (on && !first) {
      if (!have) p = __ldcg(pts + i);
      have = true;
      rel_coords(c, p, rx, ry, rz);
      cur = walk_down(c, nc, cur, rx, ry, rz);
    }
    const uint32_t mark = on ? c.scur[cur] : 0u;
    const uint32_t e = (mark & ((1u << SPLIT_BITS) - 1u)) - s_lo;
    on = (mark & SPLIT_MARK) && e < K;  // e: wraps for entries of earlier rounds
    uint32_t at = 0;
    if (on) {
      if (!have) p = __ldcg(pts + i);
      rel_coords(c, p, rx, ry, rz);
      const uint32_t L = (mark >> SPLIT_BITS) & 31u;
      const uint32_t de = d < L ? d : L, sh = L - de, m = (1u << de) - 1u;
      const uint32_t cube = spread5((rx >> sh) & m) | (spread5((ry >> sh) & m) << 1) |
                            (spread5((rz >> sh) & m) << 2);
      at = (e << (3u * d)) | (cube << (3u * (d - de)));
    }
    warp_tally(c.hist, smem, on, at);
  }
  tally_flush(c.hist, smem);
}

// ------------------------------------------------------------ phase: build

// Index of the first cube of level j below a split leaf among its cubes of all
// levels (8^0 + ... + 8^(j-1)). hist_up holds, per leaf, the sums of levels
// 0 .. d-1 in this order, then the list of the inner nodes among them.
__device__ __forceinline__ uint32_t level_first(uint32_t j) { return ((1u << (3u * j)) - 1u) / 7u; }

// A split leaf that a build turns into a subtree.
struct BuildRoot {
  uint32_t id, level, L;  // L: log2 size
  int32_t min[3];
};

__device__ __forceinline__ BuildRoot build_root(const Ctx& c, uint32_t id) {
  const NodeMeta& m = c.meta[id];
  return BuildRoot{id, m.level, c.rlog2 - m.level, {m.min[0], m.min[1], m.min[2]}};
}

// Node `kid` at the octant path `path`, j + 1 levels below the root: a child of
// `up` (whose grid is up_grid); an inner node with children at `first` and a
// grid, or (first = NONE) a leaf of n points with a directory.
__device__ __forceinline__ void build_node(const Ctx& c, const BuildRoot& r, uint32_t kid,
                                           uint32_t j, uint32_t path, uint32_t up,
                                           uint32_t up_grid, uint32_t first, uint32_t grid,
                                           uint32_t dir, uint32_t n) {
  NodeMeta cm;
  for (uint32_t a = 0; a < 3; ++a) {
    cm.min[a] = r.min[a];
#pragma unroll 1
    for (uint32_t l = 0; l <= j; ++l)  // octant digits, the topmost first
      cm.min[a] += (int32_t)(((path >> (3u * (j - l) + a)) & 1u) << (r.L - 1u - l));
  }
  cm.level = r.level + j + 1u;
  cm.n_chunks = 0;
  cm.head = cm.tail = NONE;
  cm.dir = first == NONE ? dir : NONE;
  cm.st_nch = 0;
  cm.st_tail = NONE;
  cm.st_seq = 0;
  cm.st_base = 0;
  cm.touched = 0;
  cm.compact = 0;
  cm.up = up | ((r.level + j) << NODE_BITS);
  cm.up_grid = up_grid;
  c.meta[kid] = cm;
  c.child[kid] = first;
  c.gridref[kid] = first == NONE ? NONE : grid;
  c.cnt[kid] = first == NONE ? n : 0u;
  c.num[kid] = 0;
}

// Room for ns inner nodes' children, directories and grids, and for the list
// entries of all but the root. False (and an error) when there is none.
struct BuildRoom {
  uint32_t node0, entry;
  unsigned long long data;
};

__device__ __forceinline__ bool build_room(const Ctx& c, uint32_t ns, uint32_t rounds,
                                           uint32_t max_iters, BuildRoom& b) {
  const unsigned long long bytes = (unsigned long long)ns * (8u * c.dir_bytes + c.grid_bytes);
  b.node0 = atomicAdd(&c.ctl->n_nodes, 8u * ns);
  b.data = atomicAdd(&c.ctl->bump, bytes);
  b.entry = ns > 1u ? atomicAdd(&c.ctl->split_count, ns - 1u) : 0u;
  if (ns > 1u) atomicAdd(&c.ctl->split_inner, ns - 1u);
  if (rounds >= max_iters) set_error(c, E_ITER_CAP);
  else if ((unsigned long long)b.node0 + 8ull * ns > c.max_nodes ||
           (unsigned long long)b.entry + ns > c.max_splits)
    set_error(c, E_NODES);
  else if (b.data + bytes > c.data_bytes) set_error(c, E_ARENA);
  else return true;
  return false;
}

// The build for histograms of one or two levels, which are what many leaves that
// split together get (hist_depth): one warp per leaf. Lanes 4q to 4q + 3 hold the
// points of child q; with two levels a child of more than T points is an inner
// node too, with the next 8 of the node ids. (2M even points in 500k batches into
// leaves of one point: histograms and builds 2.2 ms, with a block and its barriers
// per leaf 9.0; of 10 points 0.18 against 0.95.)
__device__ void phase_build_warps(const Ctx& c, uint32_t s_lo, uint32_t K, uint32_t d,
                                  uint32_t lvl0, uint32_t max_iters, uint32_t warp0,
                                  uint32_t nwarps) {
  const uint32_t lane = lane_id();
  uint32_t deepest = 0;
  for (uint32_t k = warp0; k < K; k += nwarps) {
    uint32_t* hist = c.hist + ((uint64_t)k << (3u * d));
    const BuildRoot r = build_root(c, c.splits[s_lo + k]);
    uint32_t sum;
    if (d == 1u) {
      sum = hist[lane >> 2];
    } else {
      const uint2 b = reinterpret_cast<const uint2*>(hist)[lane];
      sum = b.x + b.y;
      sum += __shfl_xor_sync(FULL_MASK, sum, 1);
      sum += __shfl_xor_sync(FULL_MASK, sum, 2);
    }
    const unsigned deep = __ballot_sync(  // bit 4q: child q is an inner node
        FULL_MASK, (lane & 3u) == 0u && d > 1u && r.L > 1u && sum > c.T);
    const uint32_t ns = 1u + (uint32_t)__popc(deep);
    const uint32_t rounds = lvl0 + (ns > 1u ? 2u : 1u);
    deepest = rounds > deepest ? rounds : deepest;
    BuildRoom b{0, 0, 0};
    bool ok = false;
    if (lane == 0) ok = build_room(c, ns, rounds, max_iters, b);
    ok = __shfl_sync(FULL_MASK, (int)ok, 0) != 0;
    if (ok) {
      b.node0 = __shfl_sync(FULL_MASK, b.node0, 0);
      b.entry = __shfl_sync(FULL_MASK, b.entry, 0);
      b.data = __shfl_sync(FULL_MASK, b.data, 0);
      const unsigned long long grid0 = b.data + (unsigned long long)ns * 8u * c.dir_bytes;
      auto grid_of = [&](uint32_t e) -> uint32_t {
        return (uint32_t)((grid0 + (unsigned long long)e * c.grid_bytes) / REF_BYTES);
      };
      auto number = [&](uint32_t q) -> uint32_t {  // of inner child q; the root is 0
        return 1u + (uint32_t)__popc(deep & ((1u << (4u * q)) - 1u));
      };
#pragma unroll 1
      for (uint32_t t0 = 0; t0 < 8u * ns; t0 += 32u) {
        const uint32_t t = t0 + lane, e = t >> 3, o = t & 7u;
        const uint32_t n0 = __shfl_sync(FULL_MASK, sum, (int)(4u * o));
        if (t >= 8u * ns) continue;
        const uint32_t dir =
            (uint32_t)((b.data + (unsigned long long)t * c.dir_bytes) / REF_BYTES);
        const bool in = e == 0u && ((deep >> (4u * o)) & 1u);
        const uint32_t f = number(o);
        unsigned rest = deep;
#pragma unroll 1
        for (uint32_t x = 1; x < e; ++x) rest &= rest - 1u;
        const uint32_t q = (uint32_t)(__ffs(rest) - 1) >> 2;  // e > 0: the e-th inner child
        const uint32_t path = e == 0u ? o : 8u * q + o;
        build_node(c, r, b.node0 + t, e == 0u ? 0u : 1u, path, e == 0u ? r.id : b.node0 + q,
                   grid_of(e), in ? b.node0 + 8u * f : NONE, grid_of(f), dir,
                   e == 0u ? n0 : hist[path]);
      }
      if ((deep >> lane) & 1u) c.splits[b.entry + number(lane >> 2) - 1u] = b.node0 + (lane >> 2);
      if (lane == 0) {
        c.child[r.id] = b.node0;
        c.gridref[r.id] = grid_of(0);
      }
    }
    __syncwarp();  // all counts have been read
    if (lane < (2u << (3u * (d - 1u)))) reinterpret_cast<uint4*>(hist)[lane] = make_uint4(0, 0, 0, 0);
  }
  if (lane == 0 && deepest) atomicMax(&c.ctl->iters, deepest + 1u);
}

// One block per split leaf (entries [s_lo, s_lo + K)): sum its cube counts
// level by level, make every cube with more than T points an inner node (8
// children with chunk directories, and a grid each, zeroed in the claim
// phase), leave the leaves' counts in cnt for decide, and clear the histogram.
// lvl0: levels that earlier rounds of this update built above. A round here
// stands for d of the paper's: iters counts the paper's, and max_iters bounds
// them as if they had been made one by one.
// The subtree of a leaf is a few dozen nodes; the sums read 8^d counts
// (128 KB at d = 5) from L2, which the other blocks do at the same time.
__device__ void phase_build(const Ctx& c, uint32_t s_lo, uint32_t K, uint32_t d, uint32_t lvl0,
                            uint32_t max_iters) {
  if (d <= 2u) {
    const uint32_t wpb = blockDim.x / 32u;
    phase_build_warps(c, s_lo, K, d, lvl0, max_iters, blockIdx.x * wpb + threadIdx.x / 32u,
                      gridDim.x * wpb);
    return;
  }
  __shared__ uint32_t s_n, s_deep, s_node, s_entry, s_ok;
  __shared__ unsigned long long s_data;
  const uint32_t U = level_first(d), bins = 1u << (3u * d);
  for (uint32_t k = blockIdx.x; k < K; k += gridDim.x) {
    uint32_t* hist = c.hist + ((uint64_t)k << (3u * d));
    uint32_t* up = c.hist_up + (uint64_t)k * 2u * U;
    uint32_t* list = up + U;
    const BuildRoot r = build_root(c, c.splits[s_lo + k]);
    if (threadIdx.x == 0) s_n = s_deep = 0;
    for (uint32_t j = d; j-- > 0;) {
      const uint32_t* below = up + level_first(j + 1u);
      const uint4* bins4 = reinterpret_cast<const uint4*>(hist);
      for (uint32_t q = threadIdx.x; q < (1u << (3u * j)); q += blockDim.x) {
        uint32_t t = 0;
        if (j + 1u == d) {
          const uint4 a = bins4[2u * q], b = bins4[2u * q + 1u];
          t = a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w;
        } else {
#pragma unroll
          for (uint32_t o = 0; o < 8; ++o) t += below[8u * q + o];
        }
        up[level_first(j) + q] = t;
      }
      __syncthreads();
    }
    // number the inner nodes; an inner node's sum becomes SPLIT_MARK | number
    for (uint32_t i = threadIdx.x; i < U; i += blockDim.x) {
      uint32_t j = 0;
      while (level_first(j + 1u) <= i) ++j;
      if (i == 0 || (up[i] > c.T && r.L > j)) {
        const uint32_t e = atomicAdd(&s_n, 1u);
        atomicMax(&s_deep, j);
        list[e] = i;
        up[i] = SPLIT_MARK | e;
      }
    }
    __syncthreads();
    const uint32_t ns = s_n;
    if (threadIdx.x == 0) {
      const uint32_t rounds = lvl0 + s_deep + 1u;
      BuildRoom b;
      s_ok = build_room(c, ns, rounds, max_iters, b);
      s_node = b.node0;
      s_data = b.data;
      s_entry = b.entry;
      atomicMax(&c.ctl->iters, rounds + 1u);
    }
    __syncthreads();
    if (s_ok) {
      const uint32_t node0 = s_node;
      const unsigned long long grid0 = s_data + (unsigned long long)ns * 8u * c.dir_bytes;
      auto grid_of = [&](uint32_t e) -> uint32_t {
        return (uint32_t)((grid0 + (unsigned long long)e * c.grid_bytes) / REF_BYTES);
      };
#pragma unroll 1
      for (uint32_t t = threadIdx.x; t < 8u * ns; t += blockDim.x) {
        const uint32_t e = t >> 3, o = t & 7u, i = list[e];
        uint32_t j = 0;
        while (level_first(j + 1u) <= i) ++j;
        const uint32_t q = i - level_first(j);
        const uint32_t id =
            j == 0 ? r.id : node0 + 8u * (up[level_first(j - 1u) + (q >> 3)] & ~SPLIT_MARK) + (q & 7u);
        const uint32_t path = 8u * q + o, kid = node0 + t;
        const uint32_t w = j + 1u == d ? hist[path] : up[level_first(j + 1u) + path];
        const bool inner = j + 1u < d && (w & SPLIT_MARK);
        const uint32_t x = w & ~SPLIT_MARK;  // an inner node's number
        build_node(c, r, kid, j, path, id, grid_of(e), inner ? node0 + 8u * x : NONE, grid_of(x),
                   (uint32_t)((s_data + (unsigned long long)t * c.dir_bytes) / REF_BYTES), w);
        if (o == 0) {
          if (j == 0) {
            c.child[r.id] = node0 + 8u * e;
            c.gridref[r.id] = grid_of(e);
          } else {
            // entry numbers without the root's
            const uint32_t re = up[0] & ~SPLIT_MARK;
            c.splits[s_entry + (e < re ? e : e - 1u)] = id;
          }
        }
      }
    }
    __syncthreads();
    uint4* h4 = reinterpret_cast<uint4*>(hist);
    for (uint32_t i = threadIdx.x; i < bins / 4u; i += blockDim.x) h4[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();  // before s_n is used again
  }
}

// Zero the grids of this update's splits (entries [0, s_hi)); the claim phase
// does so while it claims (nothing reads them before the voxels are stored).
__device__ __forceinline__ void zero_grids(const Ctx& c, uint32_t s_hi, uint64_t warp0,
                                           uint64_t nwarps) {
  const uint32_t lane = lane_id();
  const uint32_t zpg = (c.grid_bytes + ZERO_UNIT - 1) / ZERO_UNIT;  // zero units per grid
  const uint64_t uz = (uint64_t)s_hi * zpg;
  for (uint64_t w = warp0; w < uz; w += nwarps) {
    const uint32_t id = c.splits[(uint32_t)(w / zpg)];
    const uint32_t gref = id < c.max_nodes ? c.gridref[id] : NONE;
    if (!grid_ok(c, gref)) {
      if (lane == 0) set_error(c, E_INTERNAL);
      continue;
    }
    const uint32_t lo = (uint32_t)(w % zpg) * ZERO_UNIT;
    const uint32_t hi = min(lo + ZERO_UNIT, c.grid_bytes);
    int4* g = reinterpret_cast<int4*>(grid_words(c, gref));
    for (uint32_t b = lo / 16 + lane; b < hi / 16; b += 32) g[b] = make_int4(0, 0, 0, 0);
  }
}

// ------------------------------------------------------------- phase: claim

// Points of a warp that go on to the next coarser level wait in shared memory
// until 32 of them make a full warp: about one point in ten survives its first
// claim, so walking on at once would leave most lanes idle for every further
// level.
constexpr uint32_t RESPILL = 1u << 31;
struct ClaimQueue {
  uint32_t* q;  // node | spill flag, rx, ry, rz, rgba, gidx: CLAIM_QUEUE words each
  uint32_t n;   // the same value in every lane
};

// One claim of one point: the parent of `node`.
struct ClaimItem {
  uint32_t node;  // | RESPILL: a re-inserted point
  uint32_t rx, ry, rz, rgba, gidx;
};

// What the claim phase needs to know about the update: nodes0 = nodes before
// it, grid0 = first grid reference of its own splits, open = Ctl::open, near =
// claim_near_mask.
struct ClaimArgs {
  uint32_t nodes0, grid0, open, near;
};

// All 32 lanes call: lanes with `on` sample the grid of their node's parent.
// SORTED: the items are a unit of consecutive batch points or (respill) of
// re-inserted ones of one chunk. A lane whose neighbour lane is in the same
// cell with a lower index is done (unless the voxels do not nest); in a unit of
// batch points the index grows with the lane, so only the left one can have
// it. Points that have to go on join the queue, naming the parent.
template <bool SORTED>
__device__ __forceinline__ void claim_level(const Ctx& c, WarpBuf& wb, ClaimQueue& cq,
                                            const ClaimArgs& a, bool on, const ClaimItem& it,
                                            bool respill) {
  const uint32_t lane = lane_id();
  const uint2 up = on ? *reinterpret_cast<const uint2*>(&c.meta[it.node & NODE_MASK].up)
                      : make_uint2(NONE, 0u);
  const uint32_t par = up.x & NODE_MASK;
  uint32_t word = 0, cell = 0;
  bool want = false;
  if (up.x != NONE) {
    cell = cell_index(it.rx, it.ry, it.rz, c.rlog2 - (up.x >> NODE_BITS), c.G);
    if (!grid_ok(c, up.y) || par >= c.max_nodes) {
      set_error(c, E_INTERNAL);
    } else {
      want = true;
      // a grid of this update's own splits is empty until the store
      if (up.y < a.grid0) word = grid_words(c, up.y)[cell >> 5];
    }
  }
  bool more = want && a.open != 0u;
  want = want && ((word >> (cell & 31u)) & 1u) == 0u;
  const unsigned long long key = ((unsigned long long)par << (3u * c.G)) | cell;
  const unsigned long long val = ((unsigned long long)it.gidx << 32) | it.rgba;
  bool lead = want;
  if (SORTED) {
    // a neighbour lane in the same cell with a lower index: done
    const unsigned wm = __ballot_sync(FULL_MASK, want);
    const uint32_t pc = __shfl_up_sync(FULL_MASK, cell, 1);
    const uint32_t pp = __shfl_up_sync(FULL_MASK, par, 1);
    const uint32_t pg = __shfl_up_sync(FULL_MASK, it.gidx, 1);
    bool beaten = lane != 0u && ((wm >> (lane - 1u)) & 1u) && pc == cell && pp == par &&
                  pg < it.gidx;
    if (respill) {
      const uint32_t nc2 = __shfl_down_sync(FULL_MASK, cell, 1);
      const uint32_t np = __shfl_down_sync(FULL_MASK, par, 1);
      const uint32_t ng = __shfl_down_sync(FULL_MASK, it.gidx, 1);
      beaten = beaten || (lane != 31u && ((wm >> (lane + 1u)) & 1u) && nc2 == cell && np == par &&
                          ng < it.gidx);
    }
    lead = want && (!beaten || a.open);
  }
  warp_claim(c, wb, lead, key, val, par, a.near, more);
  // a re-inserted point sampled the grids above its old leaf when it came
  if ((it.node & RESPILL) && par < a.nodes0) more = false;
  const unsigned mm = __ballot_sync(FULL_MASK, more);
  if (more) {
    uint32_t* q = cq.q + cq.n + __popc(mm & ((1u << lane) - 1u));
    q[0] = par | (it.node & RESPILL);
    q[CLAIM_QUEUE] = it.rx;
    q[2 * CLAIM_QUEUE] = it.ry;
    q[3 * CLAIM_QUEUE] = it.rz;
    q[4 * CLAIM_QUEUE] = it.rgba;
    q[5 * CLAIM_QUEUE] = it.gidx;
  }
  cq.n += (uint32_t)__popc(mm);
  __syncwarp();
}

// All 32 lanes call: take 32 points (the last time: what is left) from the
// queue and claim for them, while more than `keep` wait.
__device__ __forceinline__ void claim_drain(const Ctx& c, WarpBuf& wb, ClaimQueue& cq,
                                            const ClaimArgs& a, uint32_t keep) {
  while (cq.n > keep) {
    const uint32_t k = cq.n < 32u ? cq.n : 32u;
    cq.n -= k;
    const bool on = lane_id() < k;
    ClaimItem it{0, 0, 0, 0, 0, 0};
    if (on) {
      const uint32_t* q = cq.q + cq.n + lane_id();
      it = ClaimItem{q[0], q[CLAIM_QUEUE], q[2 * CLAIM_QUEUE], q[3 * CLAIM_QUEUE],
                     q[4 * CLAIM_QUEUE], q[5 * CLAIM_QUEUE]};
    }
    __syncwarp();
    claim_level<false>(c, wb, cq, a, on, it, false);
  }
}

// The re-inserted points (of the spill tasks [0, t_hi)) and the batch points
// [0, n): each is followed to its final leaf (noted in sp_cur, b_cur for the
// store phase) and claims from the leaf's parent upwards. The re-inserted
// points come first: they have the lowest indices, so batch points stop at
// them. Each warp loads the next unit's points and cursors while it claims.
__device__ void phase_claim(const Ctx& c, uint32_t* smem, const NodeCache nc, const int4* pts,
                            uint32_t n, unsigned long long base, uint32_t t_hi, uint32_t s_hi,
                            const ClaimArgs& a, uint32_t warp0, uint32_t nwarps) {
  tally_init(smem);
  __syncthreads();  // also publishes the caller's node-cache writes
  zero_grids(c, s_hi, warp0, nwarps);
  WarpBuf wb = warp_buf(smem);
  ClaimQueue cq;
  cq.q = smem + SMEM_QUEUE + (threadIdx.x / 32) * CLAIM_QUEUE * 6;
  cq.n = 0;
  const uint32_t lane = lane_id();
  // units [0, us) are re-inserted points, the rest batch points
  const uint32_t us = t_hi * c.parts, units = us + (n + 31u) / 32u;
  const uint32_t chl = count_chunk_log2(units, nwarps);
  int4 pn;
  uint32_t curn, gn;
  auto load = [&](uint32_t w, int4& p, uint32_t& cur, uint32_t& g) {  // cur = NONE: no point
    p = make_int4(0, 0, 0, 0);
    cur = NONE;
    g = 0;
    if (w < us) {
      SpillTask tk;
      uint32_t q;
      if (task_point(c, w, tk, q)) {
        p = chunk_recs(c, tk.ref)[q];
        g = chunk_aux(c, tk.ref)[q];
        cur = tk.node | RESPILL;
      }
    } else {
      const uint32_t i = (w - us) * 32 + lane;
      if (i < n) {
        p = __ldcg(pts + i);
        g = (uint32_t)(base + i);
        cur = c.b_cur[i];
      }
    }
  };
  load(warp_unit(warp0, nwarps, 0, chl), pn, curn, gn);
  // (the last time round there are no points, and the queue is emptied: one copy
  // of the drain, 10 KB of code less than with a second one behind the loop. The
  // persistent kernel's phases share the instruction caches: a 16M-point terrain
  // 2.248 against 2.266 ms)
  for (uint32_t k = 0, more = 1; more; ++k) {
    const uint32_t w = warp_unit(warp0, nwarps, k, chl);
    more = w < units;
    const bool on = curn != NONE;
    ClaimItem it{curn, 0, 0, 0, (uint32_t)pn.w, gn};
    rel_coords(c, pn, it.rx, it.ry, it.rz);
    load(warp_unit(warp0, nwarps, k + 1u, chl), pn, curn, gn);
    if (on) {
      const uint32_t cur = it.node & ~RESPILL;
      const uint32_t leaf = walk_down(c, nc, cur, it.rx, it.ry, it.rz);
      if (w < us) {
        const uint32_t t = div_by(w, c.parts, c.P_mul, c.P_shift);
        c.sp_cur[c.tasks[t].dst + (w - t * c.parts) * 32u + lane] = leaf;
      } else if (leaf != cur) {
        c.b_cur[(w - us) * 32 + lane] = leaf;
      }
      it.node = leaf | (it.node & RESPILL);
    }
    claim_level<true>(c, wb, cq, a, on, it, w < us);
    claim_drain(c, wb, cq, a, more ? 31u : 0u);
  }
  warp_flush(c, wb);
  tally_flush(c.cnt, smem);
}

// ------------------------------------------------------------ phase: decide

// Take up to k refs from the pool; returns how many and the first index.
// One atomicSub per allocation: the top may go below zero while the pool is
// empty; store and end clamp it at zero.
__device__ __forceinline__ uint32_t pool_take(const Ctx& c, uint32_t k, int* first) {
  const int t = atomicSub(&c.ctl->pool_top, (int)k);
  if (t <= 0) return 0;
  const int take = t < (int)k ? t : (int)k;
  *first = t - take;
  return (uint32_t)take;
}

// Section 5.3, all 32 lanes of a warp call with the same arguments: give
// node `id` ceil(total / C) chunks, pool first, then the bump allocator; link
// them, note them in a leaf's directory and record the store map for this
// update. Lane 0 takes the allocator atomics; the lanes link the new chunks
// in parallel (chunk q's successor is chunk q + 1 of the same allocation).
__device__ void alloc_chunks(const Ctx& c, uint32_t id, uint32_t total, bool leaf, uint32_t num,
                             const uint4& chunks) {
  const uint32_t lane = lane_id();
  NodeMeta& m = c.meta[id];
  const uint32_t have = chunks.x, tail = chunks.z, mdir = chunks.w;
  const uint32_t need = (uint32_t)(((unsigned long long)total + c.C - 1) / c.C);
  const uint32_t k = need > have ? need - have : 0u;
  uint32_t seq = 0, from_pool = 0, ok = 1;
  int pfirst = 0;
  unsigned long long off = 0;
  if (lane == 0 && k) {
    // (both on their way before either is looked at)
    seq = atomicAdd(&c.ctl->alloc_seq, k);
    from_pool = pool_take(c, k, &pfirst);
    if ((unsigned long long)seq + k > c.max_chunks) {
      set_error(c, E_ALLOC_REFS);
      ok = 0;
    } else {
      const uint32_t rest = k - from_pool;
      if (rest) {
        off = atomicAdd(&c.ctl->bump, (unsigned long long)rest * c.chunk_bytes);
        if (off + (unsigned long long)rest * c.chunk_bytes > c.data_bytes) {
          set_error(c, E_ARENA);
          ok = 0;
        } else {
          atomicAdd(&c.ctl->chunks_bumped, (unsigned long long)rest);
        }
      }
    }
  }
  seq = __shfl_sync(FULL_MASK, seq, 0);
  from_pool = __shfl_sync(FULL_MASK, from_pool, 0);
  pfirst = __shfl_sync(FULL_MASK, pfirst, 0);
  off = __shfl_sync(FULL_MASK, off, 0);
  ok = __shfl_sync(FULL_MASK, ok, 0);
  if (lane == 0) {
    m.st_nch = have;
    m.st_tail = tail;
    m.st_seq = k ? seq : 0u;
    m.st_base = num;
    m.touched = (uint32_t)c.ctl->st_batches + 1u;
    c.scur[id] = 0;
  }
  if (!k || !ok) return;
  uint32_t* dir = (leaf && ref_ok(c, mdir, c.dir_bytes)) ? dir_entries(c, mdir) : nullptr;
  const uint32_t bump_ref = (uint32_t)(off / REF_BYTES);
  auto ref_of = [&](uint32_t q) -> uint32_t {
    return q < from_pool ? c.pool[pfirst + (int)q] : bump_ref + (q - from_pool) * c.chunk_units;
  };
  for (uint32_t q = lane; q < k; q += 32) {
    const uint32_t ref = ref_of(q);
    const uint32_t nxt = q + 1u < k ? ref_of(q + 1u) : NONE;
    c.alloc_refs[seq + q] = ref;
    *chunk_next(c, ref) = nxt;
    if (dir && have + q < c.dir_cap) dir[have + q] = ref;
    if (q == 0) {
      if (tail == NONE) m.head = ref;
      else *chunk_next(c, tail) = ref;
    }
    if (q + 1u == k) m.tail = ref;
  }
  if (lane == 0) m.n_chunks = need;
}

// Section 5.1, all 32 lanes of a warp call: list leaf `id`, whose count exceeds
// T, for the build phase, with one spill task per chunk of its stored points;
// those chunks return to the pool at the end of the update.
__device__ void split_leaf(const Ctx& c, uint32_t id, uint32_t total) {
  const uint32_t lane = lane_id();
  NodeMeta& m = c.meta[id];
  const uint32_t stored = c.num[id], nch = m.n_chunks, mdir = m.dir;
  uint32_t s0 = 0, t0 = 0, e = 0, ok = 1;
  if (lane == 0) {
    s0 = atomicAdd(&c.ctl->spill_count, stored);
    t0 = atomicAdd(&c.ctl->ntasks, nch);
    e = atomicAdd(&c.ctl->split_count, 1u);
    atomicMax(&c.ctl->split_most, total);
    if (e >= c.max_splits) {
      set_error(c, E_NODES);
      ok = 0;
    } else if ((unsigned long long)s0 + stored > c.spill_cap) {
      set_error(c, E_SPILL);
      ok = 0;
    } else if ((unsigned long long)t0 + nch > c.max_chunks || nch > c.dir_cap ||
               (nch && !ref_ok(c, mdir, c.dir_bytes))) {
      set_error(c, E_INTERNAL);
      ok = 0;
    }
  }
  if (!__shfl_sync(FULL_MASK, ok, 0)) return;
  s0 = __shfl_sync(FULL_MASK, s0, 0);
  t0 = __shfl_sync(FULL_MASK, t0, 0);
  e = __shfl_sync(FULL_MASK, e, 0);
  const uint32_t* dir = nch ? dir_entries(c, mdir) : nullptr;
  for (uint32_t j = lane; j < nch; j += 32) {
    const uint32_t ref = dir[j];
    const uint32_t first = j * c.C;
    c.tasks[t0 + j] = SpillTask{ref, id, s0 + first, min(c.C, stored - first)};
    c.pending[t0 + j] = ref;
  }
  __syncwarp();  // every lane has read m before lane 0 rewrites it
  if (lane == 0) {
    c.splits[e] = id;
    c.scur[id] = SPLIT_MARK | ((c.rlog2 - m.level) << SPLIT_BITS) | e;
    m.n_chunks = 0;
    m.head = m.tail = NONE;
    m.dir = NONE;
    c.num[id] = 0;
    c.cnt[id] = 0;
  }
}

// All 32 lanes of a warp call: a compacted node (simlod_compact) that receives
// records again goes back to a chunk list first: ceil(n / C) chunks, pool
// first then bump, linked and noted in the leaf's directory, with its n
// records copied in. The array's space is not reused.
__device__ void restore_chunks(const Ctx& c, uint32_t id, bool leaf) {
  NodeMeta& m = c.meta[id];
  const uint32_t n = c.num[id], arr = m.head;
  if (!array_ok(c, arr, n)) {
    if (lane_id() == 0) set_error(c, E_INTERNAL);
    return;
  }
  __syncwarp();
  if (lane_id() == 0) {
    m.n_chunks = 0;
    m.head = m.tail = NONE;
  }
  __syncwarp();
  alloc_chunks(c, id, n, leaf, n, make_uint4(0, NONE, NONE, m.dir));
  __syncwarp();
  const uint32_t seq = m.st_seq, nch = m.n_chunks;
  if (nch != (n + c.C - 1) / c.C || (unsigned long long)seq + nch > c.max_chunks) {
    if (lane_id() == 0) set_error(c, E_INTERNAL);  // the allocation failed (error already set)
    return;
  }
  const int4* src = array_recs(c, arr);
  const uint32_t* sax = array_aux(c, arr, n);
  for (uint32_t i = lane_id(); i < n; i += 32u) {
    const uint32_t ref = c.alloc_refs[seq + i / c.C], q = i % c.C;
    chunk_recs(c, ref)[q] = src[i];
    chunk_aux(c, ref)[q] = sax[i];
  }
  __syncwarp();
  if (lane_id() == 0) {
    m.compact = 0;
    atomicAdd(&c.ctl->st_decompacted, 1ull);
    atomicAdd(&c.ctl->compact_now, ~0ull);  // minus one
    atomicAdd(&c.ctl->compact_chunks_now, 0ull - nch);
  }
  __syncwarp();
}

// A node's n_chunks, head, tail and dir, loaded where it stands (the compiler
// would move the load behind the test of the node's count).
__device__ __forceinline__ uint4 chunk_words(const Ctx& c, uint32_t id) {
  static_assert(offsetof(NodeMeta, n_chunks) == 16 && offsetof(NodeMeta, dir) == 28,
                "the chunk words are one aligned 16-byte load");
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(&c.meta[id].n_chunks)
               : "memory");
  return v;
}

// All 32 lanes of a warp call for one candidate node (a leaf: inner nodes have
// no counts before the claim phase). What a node with a count needs is loaded
// with the count: most of this phase is the chain of one node's round trips.
__device__ __forceinline__ void decide_node(const Ctx& c, uint32_t id) {
  const uint32_t k = vload(c.cnt + id);
  uint4 chunks = chunk_words(c, id);
  const uint32_t child = vload(c.child + id), num = vload(c.num + id);
  const uint32_t level = vload(&c.meta[id].level), compact = vload(&c.meta[id].compact);
  if (k == 0) return;
  const bool leaf = child == NONE;
  if (compact) {
    restore_chunks(c, id, leaf);
    chunks = chunk_words(c, id);
  }
  const uint32_t total = num + k;
  if (leaf && total > c.T && c.rlog2 > level) {
    split_leaf(c, id, total);
    return;
  }
  alloc_chunks(c, id, total, leaf, num, chunks);
  __syncwarp();
  if (lane_id() == 0) {
    c.num[id] = total;
    c.cnt[id] = 0;
  }
}

// Candidates: the node id range [n_lo, n_hi). In the expansion rounds these are
// leaves; after the claim phase the counts left are the inner nodes' new voxels,
// which get their chunks here. One warp per node. From DECIDE_SCAN nodes per warp
// on, a warp first reads the counts of its next 32 nodes at once and visits those
// that have one: a small update of a large octree then pays a round trip per 32
// nodes (4,096 points into 300k nodes 36 against 52 us, into 104k nodes 33 against
// 38; both looks at the nodes used to load five words of each). Below that the
// look would only come in front of the node's own loads.
constexpr uint32_t DECIDE_SCAN = 2;
__device__ void phase_decide(const Ctx& c, uint32_t n_lo, uint32_t n_hi, uint32_t warp0,
                             uint32_t nwarps) {
  const bool scan = n_hi - n_lo > DECIDE_SCAN * nwarps;
  uint32_t seen = n_lo + warp0;  // scan: the warp's first node not looked at yet
  unsigned some = 0;             // which of the last 32 looked at are to be visited
#pragma unroll 1
  for (uint32_t w = seen; w < n_hi; w += nwarps) {
    if (scan) {
      while (some == 0u && seen < n_hi) {
        const uint32_t id = seen + lane_id() * nwarps;
        some = __ballot_sync(FULL_MASK, id < n_hi && __ldcg(c.cnt + id) != 0u);
        seen += 32u * nwarps;
      }
      if (some == 0u) break;
      w = seen - (33u - (uint32_t)__ffs(some)) * nwarps;
      some &= some - 1u;
    }
    decide_node(c, w);
  }
}

// The batch was rejected (a point outside the root cube): undo the counts of
// its count round, nodes [0, n_nodes), so nothing changed.
__device__ void phase_rollback(const Ctx& c, uint32_t n_nodes, uint64_t t0, uint64_t nthreads) {
  for (uint64_t t = t0; t < n_nodes; t += nthreads) c.cnt[t] = 0;
}

// -------------------------------------------------------------- phase: store

// Slots of the items that one block stores (the table lies over the staging,
// queue and tally regions, which the store phases do not use): the block
// counts its items per node, takes one range per node with one atomicAdd on
// the node's store cursor, and its threads then place the items in the ranges
// with shared-memory atomics. With one range per node and round of 1,024
// items (the form before) the returning atomics on a few cursors and the two
// block barriers of every round were the phase: 50 of 54 stalled cycles per
// instruction waited for memory, at 12 % of the issue slots and of DRAM.
constexpr uint32_t PLACE_WORDS = SMEM_TALLY + 2 * TALLY_SLOTS - SMEM_WBUF;
constexpr uint32_t place_log2(uint32_t words) {
  uint32_t l = 0;
  while ((5u << (l + 1u)) <= words) ++l;
  return l;
}
constexpr uint32_t PLACE_LOG2 = place_log2(PLACE_WORDS);
constexpr uint32_t PLACE_SLOTS = 1u << PLACE_LOG2;
constexpr int PLACE_PROBES = 6;  // then the item's own atomic takes its slot

struct PlaceTable {
  uint32_t *node, *next;       // node, NONE: free; items counted, then next slot
  uint32_t *nch, *tail, *seq;  // the node's store map
};

__device__ __forceinline__ PlaceTable place_table(uint32_t* smem) {
  uint32_t* w = smem + SMEM_WBUF;
  return PlaceTable{w, w + PLACE_SLOTS, w + 2 * PLACE_SLOTS, w + 3 * PLACE_SLOTS,
                    w + 4 * PLACE_SLOTS};
}

__device__ __forceinline__ uint32_t place_home(uint32_t node) {
  return (node * 0x9E3779B1u) >> (32u - PLACE_LOG2);
}

// The node's entry, made if there is none (pass 1); NONE after PLACE_PROBES.
__device__ __forceinline__ uint32_t place_insert(const PlaceTable& t, uint32_t node) {
  uint32_t h = place_home(node);
  for (int p = 0; p < PLACE_PROBES; ++p) {
    uint32_t old = t.node[h];
    if (old == NONE) old = atomicCAS(t.node + h, NONE, node);
    if (old == NONE || old == node) return h;
    h = (h + 1u) & (PLACE_SLOTS - 1u);
  }
  return NONE;
}

__device__ __forceinline__ uint32_t place_find(const PlaceTable& t, uint32_t node) {
  uint32_t h = place_home(node);
  for (int p = 0; p < PLACE_PROBES; ++p) {
    if (t.node[h] == node) return h;
    h = (h + 1u) & (PLACE_SLOTS - 1u);
  }
  return NONE;
}

__device__ __forceinline__ void put_rec(const Ctx& c, uint32_t ref, uint32_t q, int4 rec,
                                        uint32_t aux) {
  chunk_recs(c, ref)[q] = rec;
  chunk_aux(c, ref)[q] = aux;
}

constexpr int STORE_U = SL_STORE_UNROLL;

struct StoreItem {
  uint32_t node;         // NONE: nothing
  int4 rec;
  uint32_t aux;
  uint32_t slot, gref;   // voxels: claim-table slot and occupancy grid
};

// All threads of the block call. The block takes a contiguous range of the
// `units` (32 items each). node_of(w): the lane's node in unit w, NONE for
// none. load(w, node, item): its record. done(item): after its record is in
// place. Equal nodes of a run of lanes share one reservation. Each warp carries
// STORE_U units at a time.
template <typename NodeOf, typename Load, typename Done>
__device__ __forceinline__ void place_units(const Ctx& c, uint32_t* smem, uint32_t units,
                                            NodeOf&& node_of, Load&& load, Done&& done) {
  constexpr int U = STORE_U;
  const PlaceTable t = place_table(smem);
  const uint32_t lane = lane_id();
  const uint32_t per = (units + gridDim.x - 1u) / gridDim.x;
  const uint32_t first = blockIdx.x * per, last = first + per;
  const uint32_t lo = first + threadIdx.x / 32u, hi = last < units ? last : units;
  const uint32_t wpb = blockDim.x / 32;
  if (first >= units) return;  // (all threads of the block alike)
  __syncthreads();             // the regions' last use is over
  for (uint32_t i = threadIdx.x; i < PLACE_SLOTS; i += blockDim.x) {
    t.node[i] = NONE;
    t.next[i] = 0;
  }
  __syncthreads();
  for (uint32_t w = lo; w < hi; w += wpb) {
    const uint32_t node = node_of(w);
    const LaneRun r = lane_run(node != NONE, node);
    if (r.head) {
      const uint32_t h = place_insert(t, node);
      if (h != NONE) atomicAdd(t.next + h, r.end - lane);
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < PLACE_SLOTS; i += blockDim.x) {
    const uint32_t node = t.node[i];
    if (node == NONE) continue;
    const uint4 map = *reinterpret_cast<const uint4*>(&c.meta[node].st_nch);
    t.next[i] = map.w + atomicAdd(&c.scur[node], t.next[i]);
    t.nch[i] = map.x;
    t.tail[i] = map.y;
    t.seq[i] = map.z;
  }
  __syncthreads();
  for (uint32_t w0 = lo; w0 < hi; w0 += U * wpb) {
    StoreItem it[U];
    uint32_t slot[U];
    uint32_t nch[U], tail[U], seq[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const uint32_t w = w0 + j * wpb;
      it[j] = StoreItem{w < hi ? node_of(w) : NONE, make_int4(0, 0, 0, 0), 0, 0, 0};
    }
#pragma unroll
    for (int j = 0; j < U; ++j)
      if (it[j].node != NONE) load(w0 + j * wpb, it[j]);
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const LaneRun r = lane_run(it[j].node != NONE, it[j].node);
      uint32_t at = 0;
      nch[j] = seq[j] = 0;
      tail[j] = NONE;
      if (it[j].node != NONE) {
        const uint32_t h = place_find(t, it[j].node);
        if (h != NONE) {
          if (r.head) at = atomicAdd(t.next + h, r.end - lane);
          nch[j] = t.nch[h];
          tail[j] = t.tail[h];
          seq[j] = t.seq[h];
        } else {
          const uint4 map = *reinterpret_cast<const uint4*>(&c.meta[it[j].node].st_nch);
          if (r.head) at = map.w + atomicAdd(&c.scur[it[j].node], r.end - lane);
          nch[j] = map.x;
          tail[j] = map.y;
          seq[j] = map.z;
        }
      }
      slot[j] = __shfl_sync(FULL_MASK, at, (int)r.first) + lane - r.first;
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      if (it[j].node == NONE) continue;
      const uint32_t k = div_by(slot[j], c.C, c.C_mul, c.C_shift), q = slot[j] - k * c.C;
      uint32_t ref = NONE;
      if (k + 1u == nch[j]) {
        ref = tail[j];
      } else if (k >= nch[j]) {
        const unsigned long long a = (unsigned long long)seq[j] + (k - nch[j]);
        if (a < c.max_chunks) ref = c.alloc_refs[a];
      }
      if (!chunk_ok(c, ref)) {
        set_error(c, E_INTERNAL);
        continue;
      }
      put_rec(c, ref, q, it[j].rec, it[j].aux);
      done(it[j]);
    }
  }
}

// Store the batch points and the re-inserted points (of the spill tasks
// [0, t_hi), still in their old chunks), each at the next free slot of its leaf.
__device__ void phase_store(const Ctx& c, uint32_t* smem, const int4* pts, uint32_t n,
                            unsigned long long base, uint32_t t_hi) {
  const uint32_t lane = lane_id();
  // units [0, us) are re-inserted points, the rest batch points
  const uint32_t us = t_hi * c.parts;
  place_units(
      c, smem, us + (n + 31u) / 32u,
      [&](uint32_t w) -> uint32_t {
        uint32_t node = NONE;
        if (w < us) {
          SpillTask tk;
          uint32_t q;
          if (!task_point(c, w, tk, q)) return NONE;
          node = c.sp_cur[tk.dst + q];
        } else {
          const uint32_t i = (w - us) * 32u + lane;
          if (i >= n) return NONE;
          node = c.b_cur[i];
        }
        if (node < c.max_nodes) return node;
        set_error(c, E_INTERNAL);
        return NONE;
      },
      [&](uint32_t w, StoreItem& it) {
        if (w < us) {
          SpillTask tk;
          uint32_t q;
          if (!task_point(c, w, tk, q)) return;
          it.rec = chunk_recs(c, tk.ref)[q];
          it.aux = chunk_aux(c, tk.ref)[q];
        } else {
          const uint32_t i = (w - us) * 32u + lane;
          it.rec = __ldcg(pts + i);
          it.aux = (uint32_t)(base + i);
        }
      },
      [](const StoreItem&) {});
}

// Store the n_keys new voxels, each at the next free slot of its node, set
// their occupancy bits and clear their table slots; hand the n_tasks chunks of
// split leaves (one per task) to the pool above pool_top (phase_end then
// raises it).
__device__ void phase_store_voxels(const Ctx& c, uint32_t* smem, uint32_t n_tasks, uint32_t n_keys,
                                   int pool_top, uint64_t t0, uint64_t nthreads) {
  const uint32_t lane = lane_id();
  const uint32_t G = c.G, cmask = (1u << (3u * G)) - 1u, amask = (1u << G) - 1u;
  place_units(
      c, smem, n_keys / 32u + (n_keys % 32u ? 1u : 0u),
      [&](uint32_t w) -> uint32_t {
        const uint32_t e = w * 32u + lane;
        if (e >= n_keys) return NONE;
        const uint32_t node = e < c.key_nodes
                                  ? c.keys[e].y
                                  : (uint32_t)(c.hash[*key_slot(c, e)].key >> (3u * G));
        if (node < c.max_nodes) return node;
        set_error(c, E_INTERNAL);
        return NONE;
      },
      [&](uint32_t w, StoreItem& it) {
        it.slot = *key_slot(c, w * 32u + lane);
        it.gref = c.gridref[it.node];
        const ulonglong2 kv = *reinterpret_cast<const ulonglong2*>(c.hash + it.slot);
        // the node's min corner and level
        const int4 nm = *reinterpret_cast<const int4*>(&c.meta[it.node].min[0]);
        const uint32_t L = c.rlog2 - (uint32_t)nm.w;
        it.aux = (uint32_t)kv.x & cmask;  // the cell
        const uint32_t cx = it.aux & amask, cy = (it.aux >> G) & amask, cz = it.aux >> (2u * G);
        // Section 3.4: the voxel is a point at the (floor of the) cell centre
        it.rec = make_int4(nm.x + (int32_t)(((2ull * cx + 1ull) << L) >> (G + 1u)),
                           nm.y + (int32_t)(((2ull * cy + 1ull) << L) >> (G + 1u)),
                           nm.z + (int32_t)(((2ull * cz + 1ull) << L) >> (G + 1u)), (int32_t)kv.y);
        if (!grid_ok(c, it.gref)) {
          set_error(c, E_INTERNAL);
          it.gref = NONE;
        }
      },
      [&](const StoreItem& it) {
        if (it.gref != NONE)
          atomicOr(grid_words(c, it.gref) + (it.aux >> 5), 1u << (it.aux & 31u));
        *reinterpret_cast<ulonglong2*>(c.hash + it.slot) = make_ulonglong2(HASH_EMPTY, HASH_EMPTY);
      });
  const int top = pool_top > 0 ? pool_top : 0;
  if ((unsigned long long)top + n_tasks > c.max_chunks) {
    if (t0 == 0) set_error(c, E_POOL);
    return;
  }
  for (uint64_t q = t0; q < n_tasks; q += nthreads) c.pool[top + q] = c.pending[q];
}

// Expected new voxels per 1,024 points of the next update: those of the
// octree so far (`voxels` made by `points`, re-insertions counted), as if half
// an update of `last` points had come before it and made a voxel for every
// second point.
__device__ __forceinline__ uint32_t key_rate_of(unsigned long long voxels,
                                                unsigned long long points,
                                                unsigned long long last) {
  const unsigned long long r = (voxels + last / 4u) * 1024u / (points + last / 2u + 1u);
  return r < 16u ? 16u : r > 16384u ? 16384u : (uint32_t)r;
}

// One thread: close an applied update (advance gidx, return the freed
// chunks to the pool, fold the update into the stats, clear the per-update
// counters).
__device__ void phase_end(const Ctx& c, uint64_t n) {
  Ctl* t = c.ctl;
  const uint32_t iters = t->iters ? t->iters : 1u;
  const unsigned long long nk =
      min((unsigned long long)t->nkeys, (unsigned long long)c.backlog_cap);
  t->base += n;
  const int top = t->pool_top > 0 ? t->pool_top : 0;
  t->pool_top = ((unsigned long long)top + t->ntasks <= c.max_chunks) ? top + (int)t->ntasks : top;
  t->st_batches += 1;
  t->st_points += n;
  t->st_spilled += t->spill_count;
  t->st_splits += t->split_count;
  t->st_voxels += nk;
  if (iters > t->st_iter_max) t->st_iter_max = iters;
  t->st_rounds += iters;
  t->last_points = n;
  t->last_spilled = t->spill_count;
  t->last_splits = t->split_count;
  t->last_voxels = nk;
  t->last_iters = iters;
  t->spill_count = 0;
  t->nkeys = 0;
  t->alloc_seq = 0;
  t->split_count = 0;
  t->split_inner = 0;
  t->ntasks = 0;
  t->iters = 0;
  t->split_most = 0;
  t->bump0 = t->bump;
  t->key_rate = key_rate_of(t->st_voxels, t->st_points + t->st_spilled,
                            n + t->last_spilled);
}

// One thread: close a rejected update (the rollback undid its counts).
__device__ void phase_end_rejected(const Ctx& c) {
  Ctl* t = c.ctl;
  t->reject = 0;
  t->st_rejected += 1;
}

}  // namespace SL_NS

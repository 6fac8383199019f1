// Device helpers and graph state shared by the CUDA sources of libcupc.
//
// Sketch layout in HBM (layer-major): bucket (r, w, j) of layer r, vertex w,
// bucket j lives at sketch[(r * V + w) * W + j], 16 bytes {alpha, gamma}.
// j = 0 is the deterministic bucket, j = 1 + c*D + d is row d of column c
// (App. A.1.1, Theorem A.2: one bucket per column per update).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>
#include <stdint.h>

#include "cupc.h"

namespace cupc {

constexpr uint32_t kErrInval = 1u;
constexpr uint32_t kErrTimeout = 2u;
constexpr uint32_t kErrQuery = 4u;  // a query pair out of range (does not drop updates)
constexpr uint64_t kNone = ~0ull;
constexpr uint32_t kNoneU32 = 0xFFFFFFFFu;
// Most vertices: an edge id (< V^2) and a vertex id share one 64-bit key in
// the recovery's hook.
constexpr uint32_t kMaxVertices = 1u << 21;

// Rows per column that the update kernel folds in shared memory (the first
// three are folded in registers); deeper rows (probability 2^-(kSmemRows+3)
// per index) are XORed straight into HBM. The default.
constexpr uint32_t kSmemRows = 8;
constexpr uint32_t kSmemRowsMax = 16;
// Records (endpoint incidences) per update work item.
constexpr uint32_t kItemRecords = 512;  // maximum
constexpr uint32_t kDefaultItemRecords = 256;
constexpr uint32_t kMinItemRecords = 64;
// The update groups a batch through per-CTA shared histograms when
// V <= kPrivMaxV (8 bytes per vertex of shared memory) and one CTA per
// kPrivPerVertex * V endpoint records (at most one per SM) gives at least
// kPrivMinCtas CTAs. Measured on GB300 (group time per batch): V = 16384,
// 2^20 edges 77 -> 45 us; V = 4096, 2^20 edges 133 -> 36 us; one CTA per
// 2V records was slower, and too few CTAs lose to the global atomics.
constexpr uint32_t kPrivMaxV = 24576;
constexpr uint32_t kPrivPerVertex = 1;
constexpr uint32_t kPrivMinCtas = 48;
// Batches of at least kShardEdges edges on larger graphs count and scatter in
// kShards arrays of counters, one per CTA modulo kShards, so that the records
// of a hub do not all queue at one address. GB300, us for a batch with 4 arrays
// (1): V = 2^17, 2^22 R-MAT edges 2407 (2514); V = 2^15, 2^20 R-MAT
// edges 615 (711). 8 or 16 arrays, or sharding from 2^16 or 2^18 edges, gave
// nothing more.
constexpr uint32_t kShards = 4;
constexpr uint32_t kShardEdges = 1u << 20;
// The update's plan: vertices per slice (one CTA each) and threads per CTA.
constexpr uint32_t kPlanSlice = 1024;
constexpr uint32_t kPlanThreads = 256;
inline uint32_t plan_slices(uint32_t V) { return (V + kPlanSlice - 1) / kPlanSlice; }
// Counters of one update chunk: the plan's fold and direct records and those of
// hubs, and the apply kernel's next chunk of records for each layer group (at
// most 32, since L*P <= 1024).
constexpr uint32_t kWorkFold = 0, kWorkDirect = 1, kWorkHub = 2, kWorkNext = 32, kWorkSlots = 64;
// A vertex of more than two records starts at, and is padded to, a multiple
// of kPad records.
constexpr uint32_t kPad = 4;
// Entries of the record array for n edges: 2n records and the padding of the
// vertices that have at least three.
__host__ __device__ constexpr size_t rec_entries(size_t V, size_t n) {
  return 2 * n + (kPad - 1) * (V < 2 * n / 3 ? V : 2 * n / 3);
}
// Most edges of one update chunk: its record offsets fit 32 bits. A graph's
// max_batch may be larger (up to 2^31 - 1): its staging holds that many, and
// launch_update splits such a batch.
constexpr uint32_t kMaxChunkEdges = (1u << 31) - (1u << 22);
inline uint32_t chunk_edges(uint32_t max_batch) { return std::min(max_batch, kMaxChunkEdges); }
static_assert(rec_entries(kMaxVertices, kMaxChunkEdges) < 0xFFFFFFFFull - 4096, "record offsets fit 32 bits");
// Records an apply warp stages per pass (one per lane), and the distance of
// two layers' checksums of a pass.
constexpr uint32_t kStage = 32;
constexpr uint32_t kStageStride = kStage + 2;
// Warps of an apply CTA (they share nothing), and CTAs per SM its registers
// leave room for.
constexpr uint32_t kApplyWarps = 4;
constexpr uint32_t kApplyCtas = 5;
// Rows a column's lane folds on chip: 0..2 in registers, then `rows` (the
// tunable) in shared memory.
inline uint32_t fold_rows(uint32_t rows, uint32_t D) { return std::min(D, rows + 3); }
// Buckets of shared memory per lane of an apply warp that folds R rows (all
// pass through their slots on the way out), and bytes per warp: slots, kStage
// edge ids and their checksums of 32/P layers.
__host__ __device__ constexpr uint32_t apply_slots(uint32_t R) { return (1 + (R < 3 ? 3 : R)) | 1; }
__host__ __device__ constexpr uint32_t apply_warp_bytes(uint32_t R, uint32_t P) {
  return kStage * 8 + 32 * apply_slots(R) * 16 + (32 / P) * kStageStride * 8;
}
// Layer groups of a graph: an apply warp holds 32/P layers.
__host__ __device__ constexpr uint32_t layer_groups(uint32_t L, uint32_t P) { return (L * P + 31) / 32; }
// Edge ids of at most 32 bits: V^2 <= 2^32.
inline bool small_ids(uint32_t V) { return V <= 65536; }
// Batches of at most kSmallEdges edges are applied by one launch (k_small).
// Against the grouped path, us, uniform batches: V = 1024, 8192 edges 25.1
// (28.9), 12288 edges 30.1 (32.5); V = 5003, 12288 edges 39.5 (40.7); V = 2^14,
// 8192 edges 60 (75), 12288 edges 90 (99); V = 2^17, 8192 edges 90 (98), 12288
// edges 129 (136); R-MAT on V = 2^17, 10000 edges 72 (85), 12288 edges 90 (85).
constexpr uint32_t kSmallEdges = 12288;
// More edges than this, on a graph of more than kSmallHubV vertices (so that a
// vertex can have as many), and k_small looks for hubs. GB300, us, without ->
// with, batches whose edges all meet in one vertex (the kernel that folded every
// batch in brackets): V = 2^14, 4096 edges 34 -> 15 (56), 6000 edges 56 -> 31
// (56), 12000 edges 164 -> 64 (93); V = 2^17, 4096 edges 51 -> 19 (44), 8000 edges
// 123 -> 60 (85). Uniform and R-MAT batches: between 11 percent faster and 6
// slower, the latter above 8192 edges. Below 3072 edges, and on smaller graphs
// (V = 4096, 12288 edges 35, with 39), hubs cost less than looking for them.
constexpr uint32_t kSmallHubV = 4096;
constexpr uint32_t kSmallHubEdges = 3072;
// Records per chunk of a batch of nrec records on V vertices: at most `most`,
// and such that the `warps` of a layer group run out of chunks together (a
// whole number of chunks each, as near as steps of 16 records and the padding,
// 1.5 records per folded vertex on average, allow); small batches in quarter
// passes, two for every warp, as the latency of a warp's records is then all
// that counts. Batches of fewer than kSparseMean records per vertex, whose
// vertices' costs differ most (one flush each, or none), take 1.6 chunks a warp.
// GB300, us, uniform batches, 1.6 chunks and one (the kernel that gave a CTA a
// vertex): V = 2^17, 50000 edges 385 and 434 (403), 30011 edges 259, 261 (271); V
// = 65536, 50000 edges 283, 323 (323), 30011 edges 215, 233 (234). From 8 records
// a vertex on one is faster: V = 5003, 50000 edges 57, two take 66. Always a
// multiple of kPad, whatever `most` is: the apply kernel folds kPad records at a
// time and no chunk may split a group.
constexpr uint32_t kSparseMean = 4;
// Records of a batch for each of `warps` warps, the padding of evenly spread
// records included (1.5 for a vertex of three or more).
inline uint32_t records_per_warp(uint32_t nrec, uint32_t V, uint32_t warps) {
  const double m = (double)nrec / V, folded = V * (1.0 - std::exp(-m) * (1.0 + m + m * m / 2));
  const uint64_t all = (uint64_t)nrec + (uint64_t)(1.5 * std::max(0.0, folded));
  return (uint32_t)(all / std::max(1u, warps)) + 1;
}
inline uint32_t chunk_records(uint32_t nrec, uint32_t V, uint32_t warps, uint32_t most) {
  static_assert(kStage / 4 % kPad == 0 && 16 % kPad == 0 && kMinItemRecords >= kPad, "chunks are whole groups");
  most = most / kPad * kPad;
  const uint32_t per = records_per_warp(nrec, V, warps);
  if (per <= kStage) return std::max(kStage / 4, (per / 2 + kStage / 4 - 1) / (kStage / 4) * (kStage / 4));
  if (nrec / kSparseMean < V && per / 8 * 5 <= most)
    return std::min(most, std::max(kStage, (per / 8 * 5 + per % 8 * 5 / 8 + 8) / 16 * 16));
  const uint32_t rounds = (per + most - 1) / most;
  return std::min(most, (per / rounds + 16) / 16 * 16);
}
// The most records per chunk where the caller leaves it to the library and no
// hubs hold much of the batch: batches of kDenseMean records per vertex or more
// take one or two long chunks a warp where that is enough, as every cut through a
// vertex's records costs a flush. GB300, us, uniform batches with at most 512 and
// 256 records (the kernel that gave a CTA a vertex): V = 2048, 100000 edges 67, 73
// (70); V = 3099, 200000 edges 110, 114 (111); V = 5003, 160000 edges 97, 102
// (106); V = 2^14, 240000 edges 166, 189 (237). The other way below that mean (V =
// 24576, 80000 edges 219, 192) and with three chunks a warp (V = 4096, 400000
// edges 187, 179), and with hubs (R-MAT, V = 2^14, 160000 edges 195, 175).
constexpr uint32_t kDenseMean = 10;
inline uint32_t default_most(uint32_t nrec, uint32_t V, uint32_t warps) {
  const bool two = nrec / kDenseMean >= V && records_per_warp(nrec, V, warps) <= 2 * kItemRecords;
  return two ? kItemRecords : kDefaultItemRecords;
}
// Records per chunk of a batch whose hubs hold more than an eighth of its records:
// a chunk of a hub's records takes one flush, one of many small vertices a flush
// for each, so equal chunks, one or two a warp, end far apart. Four or five
// each, of 32 to 160 records. Used on graphs of at most kPrivMaxV vertices that
// get kHubMean records or more on average; elsewhere smaller chunks lose more to
// their flushes than they balance. GB300, us, R-MAT batches (chunk_records
// alone): V = 2048, 80000 edges 67 (73); V = 4096, 60000 and 280000 edges 77, 149
// (85, 162); V = 8192, 160000 and 280000 edges 142, 170 (150, 183); the other way
// V = 16384, 200000 edges 202 (198). (With a fifth of a warp's share, but no less
// than 64 records where a quarter is more: V = 2048, 50000 edges 62, 56 now.)
constexpr uint32_t kHubMean = 24;
inline uint32_t hub_chunk_records(uint32_t nrec, uint32_t warps, uint32_t most) {
  const uint32_t per = nrec / std::max(1u, warps) + 1, part = (per / 9 * 2 + 15) / 16 * 16;
  return std::min(most / kPad * kPad, std::min(5 * kStage, std::max(kStage, part)));
}
// A vertex of more records than this is a hub of its batch: four times the mean.
inline uint32_t hub_records(uint32_t nrec, uint32_t V) { return 4 * (nrec / V) + 8; }
// Key words of a graph: L*(C+1) (column multipliers and layer checksum
// keys) + 3*L*C (the other multiply-add-shift words of every column).
constexpr size_t key_words(uint32_t L, uint32_t C) { return (size_t)L * (C + 1) + (size_t)3 * L * C; }
// Output bits of one multiply-add-shift stage for indices below V^2:
// 65 - 2*ceil(log2 V) (strong universality with 64-bit words).
inline uint32_t hash_bits(uint32_t V) {
  uint32_t lg = 0;
  while (((uint64_t)1 << lg) < (uint64_t)V) lg++;
  if (lg < 1) lg = 1;
  return 65 - 2 * lg;
}
// Threads of a CTA of the grid-wide recovery, one CTA per SM (two of half the
// registers, with twice the warps for the reduce, spill: 221 against 186 us at
// V = 2^14), and the members of a component over several runs that one warp
// may read again alone.
constexpr uint32_t kRecThreads = 512;
constexpr uint32_t kRecSpan = 32;
// Buckets of a sum the recovery reads at a time (two per lane), and the
// counters of components that need more than one such pass.
constexpr uint32_t kPrefix = 64;
constexpr uint32_t kRetries = 3;
constexpr uint32_t kWarpBuckets = 8;  // buckets per lane in the recovery: W <= 256
static_assert(32 * kWarpBuckets <= kPrefix * (kRetries + 1), "a counter for every pass but the last");
// Crossing candidates at or below which a recovery hook finishes in one CTA
// (shared memory) instead of across the grid.
constexpr uint32_t kSmallHook = 1024;
constexpr uint32_t kHookBytes = 2 * kSmallHook * (8 + 4 + 4);  // its shared memory
// One-cluster recovery (recover_small.cu): graphs of at most kClMaxV
// vertices keep their per-vertex recovery state in one CTA's shared memory
// (26 bytes a vertex); kClThreads threads per CTA. Measured on GB300 (one
// recovery after 100 toggles, ER graphs): V = 1024 55 us vs 118 us for the
// grid-wide kernel, V = 2048 74 vs 128, V = 4096 117-148 vs 150-179 (1024
// threads per CTA; 512 gave 56, 81 and 139-167 us). With 512 threads the
// grid-wide kernel was faster from V = 6144 on (186 vs 157 us): the
// cluster's 16 SMs run out of issue and memory bandwidth.
constexpr uint32_t kClMaxV = 4096;
constexpr uint32_t kClThreads = 1024;
// Bounded device-side waits give up after this long.
constexpr uint64_t kWaitLimitNs = 2000000000ull;

// Device-side counters of one graph (u32 slots of `gc`).
enum : uint32_t {
  GC_ERR = 0,        // sticky error bits (kErrInval drops update batches)
  GC_NFOREST = 3,
  GC_NZ = 4,         // non-ZERO samples this round
  GC_ACTIVE = 5,     // MSF: candidates still crossing two trees (even hook steps)
  GC_NMEMBERS = 6,   // live members this round
  GC_NFAIL = 7,
  GC_NFP = 8,
  GC_ROUNDS = 9,
  GC_COMPLETE = 10,
  GC_LOGLEN = 11,
  GC_ACTIVE_ODD = 12,  // MSF: same count for odd hook steps
  GC_BAR_COUNT = 13,   // arrivals at the grid barriers of a recovery
  GC_BAR_DONE = 14,    // CTAs that left the recovery
  GC_RECOVERIES = 15,
  GC_BATCHES = 16,   // update chunks applied
  GC_SORT_DONE = 17, // CTAs of the forest sort that are done
  GC_NLIVE = 19,     // live components of the next recovery round
  GC_REC_DIRTY = 20, // a recovery gave up at a barrier: its scratch may be non-zero
  GC_LABELS_VALID = 21,  // incremental mode: labels hold the current graph's components
  GC_FOREST_SORTED = 22, // forest_sorted holds the last recovery's forest
  GC_BATCH_DEL = 24,     // number of the last batch that deletes an edge (incremental mode)
  GC_WARM = 25,          // incremental mode: forest edges were deleted: warm-start recovery
  GC_NSORTED = 26,       // length of forest_sorted
  GC_NFADD = 27,         // incremental mode: merge edges recorded in fadd since the last recovery
  GC_BATCH_MERGE = 28,   // number of the last batch that merged two components (incremental mode)
  GC_RETRY = 29,         // [kRetries] components that need another kPrefix buckets, per pass
  GC_SLOTS = 32
};

// SplitMix64 output finalizer (Steele, Lea, Flood, OOPSLA 2014).
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Key j of a graph: K(j) = mix(seed + phi * (j + 1)).
__host__ __device__ __forceinline__ uint64_t graph_key(uint64_t seed, uint32_t j) {
  return mix64(seed + 0x9E3779B97F4A7C15ull * (uint64_t)(j + 1));
}

__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t ld_cg(const uint32_t* p) { return __ldcg(p); }
__device__ __forceinline__ uint64_t ld_cg(const uint64_t* p) {
  return (uint64_t)__ldcg((const unsigned long long*)p);
}
__device__ __forceinline__ uint8_t ld_cg(const uint8_t* p) {
  return (uint8_t)__ldcg((const unsigned char*)p);
}

}  // namespace cupc

// Host-side state of one graph. Device arrays are carved from one workspace.
struct cupc_graph {
  uint32_t V, L, C, D, W, P, R;  // P: lanes per layer in the update kernel
  uint32_t ell;                  // bits of one column-hash stage (hash_bits(V))
  uint64_t seed;
  uint32_t max_batch, max_pairs;  // edges, pairs the staging holds
  uint32_t max_chunk;             // edges of one update chunk: chunk_edges(max_batch)
  void* ws;
  size_t ws_bytes;
  bool owns_ws;
  bool dirty;
  bool inc;           // incremental labels (cupc_set_incremental)
  bool forest_stale;  // an update since the last full recovery
  uint32_t inc_batch; // incremental mode: batches so far
  bool sort_pending;  // incremental mode: a recovery ran; the next update sorts its forest first
  bool imported;      // words from cupc_import_sketches since the last reset:
                      // the XOR of all vertex sketches need not be zero
  int device, sms;
  int apply_smem, apply_grid;
  uint32_t item_records, apply_cps;  // tunables: records per chunk at most, CTAs per SM (0 = max)
  bool item_default;                 // item_records was left to the library (default_most)
  // optional per-batch-size settings: bucket floor(log4 edges) (at least 5)
  struct ApplyTune {
    bool set, item_default;
    uint32_t item_records, R, cps;
    int smem, grid;
  } tune_b[16];
  int rec_grid;
  int rec_share;  // at most this many CTAs while other recoveries wait (0: no limit)
  int rec_cluster;  // CTAs of the one-cluster recovery (0: the grid-wide kernel)
  // sketches and keys
  ulonglong2* sketch;  // L*V*W
  uint64_t* keys;      // key_words(L, C)
  uint32_t* gc;        // GC_SLOTS device counters
  // update scratch
  uint32_t shards;     // arrays of V counters in cnt and cursor
  uint32_t* cnt;       // shards * V
  uint32_t* cursor;    // shards * V
  uint64_t* rec;       // rec_cap endpoint records, grouped by vertex
  uint32_t rec_cap;
  uint32_t* work;      // kWorkSlots counters of the current chunk
  uint32_t* stage_edges;  // 2*max_batch (host-input staging slot 0)
  int8_t* stage_ops;      // max_batch
  uint32_t* stage_edges1;  // 2*max_batch (slot 1)
  int8_t* stage_ops1;      // max_batch
  // host inputs of cupc_update_batch are copied on copy_stream into the two
  // slots in turn: slot_ready[k] after a copy, slot_free[k] after the last
  // kernel (on the caller's stream) that reads slot k
  cudaStream_t copy_stream;
  cudaEvent_t slot_ready[2], slot_free[2];
  int next_slot;
  uint32_t* stage_pairs;  // 2*max_pairs
  uint8_t* stage_out;     // max_pairs
  // recovery state
  uint32_t* label;   // V
  uint32_t* parent;  // V
  uint32_t* minv;    // V
  uint32_t* rcnt;    // V
  uint32_t* roff;    // V
  uint32_t* perm;    // V: members of live components, grouped
  uint32_t* pcount;  // V: runs of a component reduced so far
  uint8_t* final_;   // V
  uint8_t* merged;   // V
  uint64_t* best;    // V
  uint64_t* best2;   // V
  ulonglong2* cand;  // V: {candidate edge, endpoint labels}
  uint64_t* forest;  // V
  uint64_t* forest_sorted;  // V
  ulonglong2* acc;   // V*W (partial component sums)
  uint64_t* log_ids; // L*V
  uint32_t* log_live;   // L
  uint32_t* log_ncand;  // L
  ulonglong2* hlist;    // kSmallHook: crossing candidates of a hook step (recovery)
  uint32_t* ipar;       // V: union-find over labels for incremental inserts
  uint8_t* fdead;       // V: forest_sorted[i] was deleted since the last recovery
  // incremental mode: the inserts that merged two components since the last
  // recovery (forest edges the stream added), and a hash table of their ids
  uint64_t* fadd;       // V
  uint8_t* fadd_dead;   // V: fadd[j] was deleted since
  uint64_t* ftab;       // 2^ftab_bits ids (0 = empty slot; no edge has id 0)
  uint32_t* ftab_pos;   // 2^ftab_bits: the fadd index of ftab's id
  uint32_t ftab_bits;
  cupc_status last_recovery;
  // profiling: (kernel class, start, stop, launches) per recorded launch group
  struct ProfRec {
    int cls;
    cudaEvent_t a, b;
    int launches;
  };
  bool prof_on;
  std::vector<ProfRec> prof;
  double prof_ms[8];
  uint64_t prof_launches[8];
  cudaStream_t last_stream;
};

namespace cupc {
enum ProfClass { PC_VALIDATE = 0, PC_GROUP = 1, PC_APPLY = 2, PC_RECOVER = 3, PC_QUERY = 4, PC_SORT = 5, PC_N = 8 };
// Record an event pair around a launch group when profiling is on.
struct ProfScope {
  cupc_graph* g;
  cudaStream_t s;
  int cls, launches;
  cudaEvent_t a = nullptr;
  ProfScope(cupc_graph* g_, cudaStream_t s_, int cls_, int launches_) : g(g_), s(s_), cls(cls_), launches(launches_) {
    g->last_stream = s;
    if (g->prof_on && cudaEventCreate(&a) == cudaSuccess) cudaEventRecord(a, s);
  }
  ~ProfScope() {
    if (!a) return;
    cudaEvent_t b;
    if (cudaEventCreate(&b) != cudaSuccess) {
      cudaEventDestroy(a);
      return;
    }
    cudaEventRecord(b, s);
    g->prof.push_back({cls, a, b, launches});
  }
};
}  // namespace cupc

namespace cupc {
// Whether a kernel of `device` may store 64-bit words at p: memory that lives
// on that device. What lives on another GPU needs peer access, which the
// runtime's copies do not.
inline bool stores_directly(const cudaPointerAttributes& at, const void* p, int device) {
  return (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged) && at.device == device &&
         (uintptr_t)p % 8 == 0;
}

// Launchers (defined in update.cu / recover.cu); all stream-ordered.
cudaError_t launch_keys(cupc_graph* g, cudaStream_t s);
// validate_ops: also validate this chunk (a batch of one chunk), else the
// caller has validated the whole batch first.
cudaError_t launch_update_chunk(cupc_graph* g, const uint32_t* edges, size_t n, cudaStream_t s,
                                const int8_t* validate_ops = nullptr);
// A device batch of any length, in chunks of at most g->max_chunk edges; ops:
// also validate the batch as a whole.
cudaError_t launch_update(cupc_graph* g, const uint32_t* edges, size_t n, cudaStream_t s, const int8_t* ops);
cudaError_t launch_validate(cupc_graph* g, const uint32_t* edges, const int8_t* ops, size_t n, cudaStream_t s);
cudaError_t setup_update(cupc_graph* g);
cudaError_t configure_apply(cupc_graph* g);
cudaError_t apply_config(const cupc_graph* g, uint32_t R, uint32_t cps, int* smem, int* grid);
// Tuning bucket of a batch of n edges: floor(log4 n), at least 5, at most 15.
inline uint32_t tune_bucket(size_t n) {
  uint32_t b = 5;
  while (b < 15 && ((size_t)1 << (2 * (b + 1))) <= n) b++;
  return b;
}
cudaError_t raise_apply_smem_limit(int bytes);
cudaError_t setup_recover(cupc_graph* g);
cudaError_t launch_recover(cupc_graph* g, cudaStream_t s, bool force = false);
cudaError_t launch_query(cupc_graph* g, const uint32_t* pairs, size_t m, uint8_t* out, cudaStream_t s);
cudaError_t launch_forest_sort(cupc_graph* g, cudaStream_t s);
cudaError_t launch_copy_forest(cupc_graph* g, uint64_t* out, size_t cap, cudaStream_t s);
cudaError_t launch_incremental(cupc_graph* g, const uint32_t* edges, const int8_t* ops, size_t n, cudaStream_t s);
}  // namespace cupc

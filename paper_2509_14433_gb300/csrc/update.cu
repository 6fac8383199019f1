// Batched edge updates into the vertex sketches (App. A.1.1, "The AGM
// Algorithm": an update of edge (u,v) updates every sketch of u and of v;
// Theorem A.2: CameoSketch touches one bucket per column per update).
//
// One chunk of <= max_chunk edges goes through four stream-ordered kernels (a
// batch of several chunks is validated whole by k_validate first, a batch of
// one chunk inside the count):
//   k_count   per-vertex record counts (2 records per edge, one per
//             endpoint); k_count_priv for dense batches on small graphs,
//             through per-CTA shared histograms
//   k_plan    a segment of the record array for every vertex
//   k_scatter endpoint records (vertex, other end) grouped by vertex
//             (k_scatter_priv with k_count_priv)
//   k_apply   persistent warps; a warp owns some layers of the graph and takes
//             chunks of the record array (apply_chunk)
// XOR is associative and commutative, so the result is bit-identical to
// applying the updates one by one in stream order.
#include "update_dev.cuh"

namespace cupc {

__global__ void k_keys(uint64_t seed, uint64_t* keys, uint32_t n) {
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    keys[j] = graph_key(seed, j);
}

cudaError_t launch_keys(cupc_graph* g, cudaStream_t s) {
  k_keys<<<1, 256, 0, s>>>(g->seed, g->keys, (uint32_t)key_words(g->L, g->C));
  return cudaGetLastError();
}

// Problem 1's stream: ((u,v), Delta) with u != v in V and Delta = +-1.
__global__ void k_validate(const uint32_t* __restrict__ edges, const int8_t* __restrict__ ops, size_t n,
                           uint32_t V, uint32_t* gc) {
  bool bad = false;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    uint32_t u = edges[2 * i], v = edges[2 * i + 1];
    int8_t op = ops[i];
    bad |= (u >= V) | (v >= V) | (u == v) | ((op != 1) & (op != -1));
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&gc[GC_ERR], kErrInval);
}

cudaError_t launch_validate(cupc_graph* g, const uint32_t* edges, const int8_t* ops, size_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  int grid = (int)std::min<size_t>((n + 255) / 256, (size_t)g->sms * 8);
  ProfScope ps(g, s, PC_VALIDATE, 1);
  k_validate<<<grid, 256, 0, s>>>(edges, ops, n, g->V, g->gc);
  return cudaGetLastError();
}

// The plan's record counts and the apply kernel's chunk counters start at 0.
__device__ __forceinline__ void reset_work(uint32_t* work) {
  if (blockIdx.x == 0 && threadIdx.x < kWorkSlots) work[threadIdx.x] = 0;
}

// With ops (a batch of one chunk) it also validates the batch as k_validate
// does, saving that pass; counts of an invalid batch are cleared by k_plan.
// CTA b counts in shard b % shards (of V counters): the records of a hub
// queue at its counter, 155 us of this kernel for 2^22 R-MAT edges on V =
// 2^17 with one shard, 52 for as many uniform edges.
__global__ void k_count(const uint32_t* __restrict__ edges, const int8_t* __restrict__ ops, size_t n, uint32_t V,
                        uint32_t* cnt, uint32_t shards, uint32_t* work, uint32_t* gc) {
  if (ld_cg(&gc[GC_ERR]) & kErrInval) return;
  reset_work(work);
  cnt += (size_t)(blockIdx.x % shards) * V;
  bool bad = false;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const uint32_t u = edges[2 * i], v = edges[2 * i + 1];
    if (ops) {
      const int8_t op = ops[i];
      bad |= (u >= V) | (v >= V) | (u == v) | ((op != 1) & (op != -1));
    }
    if (u < V && v < V) {
      atomicAdd(&cnt[u], 1u);
      atomicAdd(&cnt[v], 1u);
    }
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&gc[GC_ERR], kErrInval);
}

// Dense batches on small graphs (V <= kPrivMaxV, at least kPrivPerVertex
// records per vertex on average): each CTA takes a contiguous slice of the
// batch and counts its endpoints in a shared histogram of all V vertices, so
// the global counters see one atomic per (CTA, vertex) instead of one per
// record.
__global__ void __launch_bounds__(1024) k_count_priv(const uint32_t* __restrict__ edges,
                                                     const int8_t* __restrict__ ops, size_t n, uint32_t V,
                                                     uint32_t* cnt, uint32_t* work, uint32_t* gc) {
  extern __shared__ uint32_t s_h[];  // V
  // another CTA may set the error meanwhile: the threads of a CTA, which meet
  // at barriers below, must agree on what they read
  if (__syncthreads_or(ld_cg(&gc[GC_ERR]) & kErrInval)) return;
  reset_work(work);
  for (uint32_t w = threadIdx.x; w < V; w += blockDim.x) s_h[w] = 0;
  __syncthreads();
  const size_t chunk = (n + gridDim.x - 1) / gridDim.x, lo = blockIdx.x * chunk, hi = min(n, lo + chunk);
  bool bad = false;
  for (size_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const uint32_t u = edges[2 * i], v = edges[2 * i + 1];
    if (ops) {
      const int8_t op = ops[i];
      bad |= (u >= V) | (v >= V) | (u == v) | ((op != 1) & (op != -1));
    }
    if (u < V && v < V) {
      atomicAdd(&s_h[u], 1u);
      atomicAdd(&s_h[v], 1u);
    }
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&gc[GC_ERR], kErrInval);
  __syncthreads();
  for (uint32_t w = threadIdx.x; w < V; w += blockDim.x) {
    const uint32_t c = s_h[w];
    if (c) atomicAdd(&cnt[w], c);
  }
}

// ... and groups them: the CTA counts its slice again, reserves one range of
// each of its vertices' segments (one atomic per vertex), then places each
// record at the range start + its rank in shared memory. Records of a vertex
// land in a different order than with k_scatter; XOR does not see order.
__global__ void __launch_bounds__(1024) k_scatter_priv(const uint32_t* __restrict__ edges, size_t n, uint32_t V,
                                                       uint32_t* cursor, uint64_t* __restrict__ rec,
                                                       const uint32_t* gc) {
  extern __shared__ uint32_t s_h[];  // V counts, then V range starts
  uint32_t* s_base = s_h + V;
  if (ld_cg(&gc[GC_ERR]) & kErrInval) return;
  for (uint32_t w = threadIdx.x; w < V; w += blockDim.x) s_h[w] = 0;
  __syncthreads();
  const size_t chunk = (n + gridDim.x - 1) / gridDim.x, lo = blockIdx.x * chunk, hi = min(n, lo + chunk);
  for (size_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    atomicAdd(&s_h[edges[2 * i]], 1u);
    atomicAdd(&s_h[edges[2 * i + 1]], 1u);
  }
  __syncthreads();
  for (uint32_t w = threadIdx.x; w < V; w += blockDim.x) {
    const uint32_t c = s_h[w];
    if (c) s_base[w] = atomicAdd(&cursor[w], c);
    s_h[w] = 0;
  }
  __syncthreads();
  for (size_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const uint32_t u = edges[2 * i], v = edges[2 * i + 1];
    const uint32_t pu = s_base[u] + atomicAdd(&s_h[u], 1u), pv = s_base[v] + atomicAdd(&s_h[v], 1u);
    rec[pu] = make_record(u, v);
    rec[pv] = make_record(v, u);
  }
}

// ---- incremental labels (cupc_set_incremental). After a complete
// recovery the labels are the components of the graph; with a valid stream
// (inserts of absent edges, deletes of present ones) an insert can only
// merge two components, and deleting an edge outside a spanning forest of
// the graph cannot split one. So a batch keeps the labels exact by merging
// the endpoint labels of its inserts (union-find over labels, the larger
// root under the smaller, so a root is its component's minimum vertex id,
// the label a recovery gives). Each insert whose link succeeds joins two
// components: it becomes a forest edge (fadd, with a hash table of ids), so
// the recovered forest plus these edges stays a spanning forest of the
// graph. A deleted forest edge of either kind is marked (fdead, fadd_dead)
// and sets GC_WARM: the next recovery starts from the fragments of the
// remaining forest. In a batch that both merges and deletes, an edge the
// batch inserts (a merge) and then deletes is found by a second lookup pass
// (k_incr_rest) once all of the batch's merges are recorded.
__device__ __forceinline__ uint32_t inc_find(uint32_t* par, uint32_t x, uint32_t V) {
  for (uint32_t k = 0; k < V; k++) {  // a path is shorter than V
    const uint32_t y = ld_cg(&par[x]);
    if (y == x) break;
    const uint32_t z = ld_cg(&par[y]);
    if (z != y) par[x] = z;  // halving: only ever to an ancestor
    x = y;
  }
  return x;
}

// Home slot of an edge id in the merge-edge table (Fibonacci hashing).
__device__ __forceinline__ uint32_t ftab_home(uint64_t id, uint32_t bits) {
  return (uint32_t)((id * 0x9E3779B97F4A7C15ull) >> (64 - bits));
}

struct IncArgs {
  const uint32_t* label;
  uint32_t* ipar;
  const uint64_t* forest_sorted;
  uint8_t* fdead;
  uint64_t* fadd;
  uint8_t* fadd_dead;
  unsigned long long* ftab;
  uint32_t* ftab_pos;
  uint32_t ftab_bits, V;
  uint32_t batch;  // number of this batch: what gc[GC_BATCH_DEL] and gc[GC_BATCH_MERGE] hold if it deletes, merges
  uint32_t* gc;
};

__global__ void k_incr(const uint32_t* __restrict__ edges, const int8_t* __restrict__ ops, size_t n, IncArgs a) {
  uint32_t* gc = a.gc;
  if ((ld_cg(&gc[GC_ERR]) & kErrInval) || !ld_cg(&gc[GC_LABELS_VALID])) return;
  const uint32_t V = a.V, nf = ld_cg(&gc[GC_NSORTED]), nadd = ld_cg(&gc[GC_NFADD]);
  const uint32_t mask = (1u << a.ftab_bits) - 1u;
  bool del = false, merged = false, cut = false, warm = false;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const uint32_t u = edges[2 * i], v = edges[2 * i + 1];
    const uint64_t id = (uint64_t)min(u, v) * V + max(u, v);
    if (ops[i] < 0) {
      del = true;
      uint32_t lo = 0, hi = nf;  // first recovered forest id >= id
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a.forest_sorted[mid] < id)
          lo = mid + 1;
        else
          hi = mid;
      }
      if (lo < nf && a.forest_sorted[lo] == id) {
        a.fdead[lo] = 1;
        warm = true;
      } else if (nadd) {  // a forest edge added by a merge?
        uint32_t sl = ftab_home(id, a.ftab_bits);
        for (uint32_t k = 0; k <= mask; k++, sl = (sl + 1) & mask) {
          const unsigned long long key = ld_cg((const uint64_t*)&a.ftab[sl]);
          if (key == 0ull) break;
          if (key == (unsigned long long)id) {
            const uint32_t j = ld_cg(&a.ftab_pos[sl]);
            if (j < V) a.fadd_dead[j] = 1;
            warm = true;
            break;
          }
        }
      }
    } else {
      uint32_t x = a.label[u], y = a.label[v];
      for (uint32_t k = 0; k < (1u << 20); k++) {  // bounded retries; giving up clears the labels
        x = inc_find(a.ipar, x, V);
        y = inc_find(a.ipar, y, V);
        if (x == y) break;
        if (x > y) {
          const uint32_t t = x;
          x = y;
          y = t;
        }
        if (atomicCAS(&a.ipar[y], y, x) == y) {
          merged = true;
          // this insert joined two components: record it as a forest edge
          const uint32_t j = atomicAdd(&gc[GC_NFADD], 1u);
          bool placed = false;
          if (j < V) {
            a.fadd[j] = id;
            a.fadd_dead[j] = 0;
            uint32_t sl = ftab_home(id, a.ftab_bits);
            for (uint32_t q = 0; q <= mask; q++, sl = (sl + 1) & mask) {
              const unsigned long long prev = atomicCAS(&a.ftab[sl], 0ull, (unsigned long long)id);
              if (prev == 0ull || prev == (unsigned long long)id) {
                a.ftab_pos[sl] = j;
                placed = true;
                break;
              }
            }
          }
          if (!placed) cut = true;  // cannot happen with a valid stream
          break;
        }
        if (k + 1 == (1u << 20)) cut = true;
      }
    }
  }
  if (__any_sync(0xffffffffu, cut) && (threadIdx.x & 31) == 0) gc[GC_LABELS_VALID] = 0;
  if (__any_sync(0xffffffffu, del) && (threadIdx.x & 31) == 0) gc[GC_BATCH_DEL] = a.batch;
  if (__any_sync(0xffffffffu, merged) && (threadIdx.x & 31) == 0) gc[GC_BATCH_MERGE] = a.batch;
  if (__any_sync(0xffffffffu, warm) && (threadIdx.x & 31) == 0) gc[GC_WARM] = 1;
}

// The rest of a batch, once k_incr has recorded all of its merges.
//
// Labels after the merges: every vertex takes its label's root. Merges are
// exact whatever else the batch did: a delete can only split components, and
// one that removed a forest edge has set GC_WARM, so the next query recovers
// from the fragments of the remaining forest.
//
// A batch that both merges and deletes: k_incr looked each delete up in the
// merge edges recorded before the batch, so an edge this batch inserted (and
// recorded as a merge) and then deleted again, in stream order, is looked up
// again here.
__global__ void k_incr_rest(const uint32_t* __restrict__ edges, const int8_t* __restrict__ ops, size_t n,
                            uint32_t* label, IncArgs a) {
  uint32_t* gc = a.gc;
  if ((ld_cg(&gc[GC_ERR]) & kErrInval) || !ld_cg(&gc[GC_LABELS_VALID]) || ld_cg(&gc[GC_BATCH_MERGE]) != a.batch) return;
  const uint32_t V = a.V, t = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (uint32_t w = t; w < V; w += stride) label[w] = inc_find(a.ipar, label[w], V);
  if (ld_cg(&gc[GC_BATCH_DEL]) != a.batch) return;
  const uint32_t mask = (1u << a.ftab_bits) - 1u;
  bool warm = false;
  for (size_t i = t; i < n; i += stride) {
    if (ops[i] >= 0) continue;
    const uint32_t u = edges[2 * i], v = edges[2 * i + 1];
    const uint64_t id = (uint64_t)min(u, v) * V + max(u, v);
    uint32_t sl = ftab_home(id, a.ftab_bits);
    for (uint32_t k = 0; k <= mask; k++, sl = (sl + 1) & mask) {
      const unsigned long long key = ld_cg((const uint64_t*)&a.ftab[sl]);
      if (key == 0ull) break;
      if (key == (unsigned long long)id) {
        const uint32_t j = ld_cg(&a.ftab_pos[sl]);
        if (j < V) a.fadd_dead[j] = 1;
        warm = true;
        break;
      }
    }
  }
  if (warm) gc[GC_WARM] = 1;
}

cudaError_t launch_incremental(cupc_graph* g, const uint32_t* edges, const int8_t* ops, size_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  if (g->sort_pending) {  // the forest of the last recovery, which this batch's deletes look up
    cudaError_t e = launch_forest_sort(g, s);
    if (e != cudaSuccess) return e;
    g->sort_pending = false;
  }
  IncArgs a;
  a.label = g->label;
  a.ipar = g->ipar;
  a.forest_sorted = g->forest_sorted;
  a.fdead = g->fdead;
  a.fadd = g->fadd;
  a.fadd_dead = g->fadd_dead;
  a.ftab = (unsigned long long*)g->ftab;
  a.ftab_pos = g->ftab_pos;
  a.ftab_bits = g->ftab_bits;
  a.V = g->V;
  if (++g->inc_batch == 0) g->inc_batch = 1;  // 0: no batch
  a.batch = g->inc_batch;
  a.gc = g->gc;
  const int grid = (int)std::min<size_t>((n + 255) / 256, (size_t)g->sms * 8);
  k_incr<<<grid, 256, 0, s>>>(edges, ops, n, a);
  const size_t rest = std::max<size_t>(n, g->V);
  k_incr_rest<<<(int)std::min<size_t>((rest + 255) / 256, (size_t)g->sms * 4), 256, 0, s>>>(edges, ops, n, g->label, a);
  return cudaGetLastError();
}

// The work plan of one chunk (plan_slice), one CTA per slice of vertices.
__global__ void __launch_bounds__(kPlanThreads) k_plan(uint32_t* cnt, uint32_t* cursor, uint64_t* rec, uint32_t V,
                                                       uint32_t cap, uint32_t shards, uint32_t hub,
                                                       uint32_t* work, uint32_t* gc) {
  const bool dropped = (ld_cg(&gc[GC_ERR]) & kErrInval) != 0;  // a dropped batch may have counted: start clean
  plan_slice(cnt, cursor, rec, V, cap, blockIdx.x, work, dropped, shards, hub);
  if (!dropped && blockIdx.x == 0 && threadIdx.x == 0) gc[GC_BATCHES] += 1;
}

// The same grid as k_count, so that a CTA's records are those of its shard.
__global__ void k_scatter(const uint32_t* __restrict__ edges, size_t n, uint32_t V, uint32_t* cursor, uint32_t shards,
                          uint64_t* __restrict__ rec, const uint32_t* gc) {
  if (ld_cg(&gc[GC_ERR]) & kErrInval) return;
  cursor += (size_t)(blockIdx.x % shards) * V;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const uint32_t u = edges[2 * i], v = edges[2 * i + 1];
    const uint32_t pu = atomicAdd(&cursor[u], 1u), pv = atomicAdd(&cursor[v], 1u);
    rec[pu] = make_record(u, v);
    rec[pv] = make_record(v, u);
  }
}

// Apply the records, in chunks of `chunk` records, or `hub_chunk` if hubs hold
// more than an eighth of them (apply_chunk). A warp keeps the layer group (its
// number modulo the groups). Its first two chunks are given, the others come from
// the group's counter, asked for two chunks ahead, so that the next chunk's
// records load while it works on this one.
//
// What bounds it. Batches of many records per vertex: instruction issue and
// the ALU (64 lanes a cycle per SM), which folding rows 0..2 in registers and
// the write-back by bulk reductions leave as the limit: per warp (4 layers x 8
// lanes) and record about 40 instructions, 20 of them on the ALU. Batches of
// few records per vertex: the rate of separate runs in HBM (20..29 G runs/s
// for runs of 16..64 bytes, 15 G/s for 128), so a column's rows go out as one
// run: one bulk XOR reduction moves 117 G buckets/s, 64-bit atomics 60 G/s,
// load and store 68 G/s (V = 2^17, runs of 8 buckets). Against the kernel
// that folded every row in shared memory and wrote back by atomics, GB300, us
// per batch: V = 5003, 30011 edges: 59 (78); V = 65536, 10^5, 10^6 edges: 400,
// 763 (460, 942); V = 2^17, 3*10^5 edges: 990 (1083).
template <bool kX32>
__global__ void __launch_bounds__(32 * kApplyWarps, kApplyCtas) k_apply(
    ulonglong2* __restrict__ sketch, const uint64_t* __restrict__ keys, const uint64_t* __restrict__ rec, uint32_t cap,
    uint32_t chunk, uint32_t hub_chunk, uint32_t* work, const uint32_t* gc, uint32_t V, uint32_t L, uint32_t C,
    uint32_t D, uint32_t W, uint32_t P, uint32_t R, uint32_t ell) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (ld_cg(&gc[GC_ERR]) & kErrInval) return;
  const uint32_t nslots = apply_slots(R);
  const uint32_t gw = blockIdx.x * kApplyWarps + (threadIdx.x >> 5), groups = layer_groups(L, P);
  const uint32_t group = gw % groups, warps = (gridDim.x * kApplyWarps - group + groups - 1) / groups;
  const ChunkPlan c = chunk_plan(work, chunk, hub_chunk);
  uint32_t q = gw / groups;
  if (q >= c.total) return;
  const ApplySmem m = apply_smem(smem_raw + (threadIdx.x >> 5) * apply_warp_bytes(R, P), nslots, P);
  const ApplyLane l = apply_lane(keys, sketch, V, L, C, D, W, P, ell, group);
  zero_slots(m, nslots);
  LaneSums a;
  clear_sums(a);
  a.dirty = 0;
  bool pending = false;
  Chunk k = chunk_at(c, q, rec, cap);
  uint64_t r = load_record(k, 0, k);
  q += warps;
  while (k.n) {
    const Chunk next = chunk_at(c, q, rec, cap);
    uint32_t ahead = q;
    if ((threadIdx.x & 31) == 0 && next.n) ahead = 2 * warps + atomicAdd(&work[kWorkNext + group], 1u);
    apply_chunk<kX32>(l, m, a, pending, k, next, r, V, W, C, P, R);
    q = __shfl_sync(0xffffffffu, ahead, 0);
    k = next;
  }
  bulk_wait_all();
}

// A small batch (n <= kSmallEdges edges, one chunk) in one launch: every CTA
// validates the whole batch, so that none needs to wait for another, then its
// warps XOR their records' buckets straight into HBM, P records (a lane each)
// and one layer group at a time. What bounds it is latency: the launch, the
// batch's loads and one pass per warp; the more edges, the bigger the CTAs, so
// that the validation stays a few loads a thread.
template <bool kX32>
__global__ void __launch_bounds__(1024) k_small(ulonglong2* __restrict__ sketch, const uint64_t* __restrict__ keys,
                                                const uint32_t* __restrict__ edges, const int8_t* __restrict__ ops,
                                                uint32_t n, uint32_t* gc, uint32_t V, uint32_t L, uint32_t C,
                                                uint32_t D, uint32_t W, uint32_t P, uint32_t ell) {
  const uint32_t lane = threadIdx.x & 31, gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const uint32_t groups = layer_groups(L, P), s = lane % P;
  // this warp's records and lanes, in flight during the validation
  const uint32_t i = gw / groups * P + s;  // record i: endpoint i & 1 of edge i / 2
  const bool have = i < 2 * n;
  const uint32_t w = have ? edges[i] : 0, other = have ? edges[i ^ 1] : 0;
  const ApplyLane l = apply_lane(keys, sketch, V, L, C, D, W, P, ell, gw % groups);
  bool drop = (ld_cg(&gc[GC_ERR]) & kErrInval) != 0, bad = false;
#pragma unroll 4
  for (uint32_t j = threadIdx.x; j < n; j += blockDim.x) {
    const uint32_t u = edges[2 * j], v = edges[2 * j + 1];
    const int8_t op = ops[j];
    bad |= (u >= V) | (v >= V) | (u == v) | ((op != 1) & (op != -1));
  }
  if (__syncthreads_or(bad)) {
    if (threadIdx.x == 0) atomicOr(&gc[GC_ERR], kErrInval);
    drop = true;
  }
  if (__syncthreads_or(drop)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) gc[GC_BATCHES] += 1;
  const uint64_t x = record_id(make_record(w, other), V), c = mix64(x ^ l.kchk);  // of this lane's layer
  for (uint32_t k = 0; k < P; k++) {
    const uint32_t from = (lane & ~(P - 1)) + k;
    const bool in = __shfl_sync(0xffffffffu, have, from);
    const uint32_t wk = __shfl_sync(0xffffffffu, w, from);
    const uint64_t xk = __shfl_sync(0xffffffffu, x, from), ck = __shfl_sync(0xffffffffu, c, from);
    if (l.active && in) xor_bucket_atomic(l.base + (size_t)wk * W + lane_depth<kX32>(l, xk), make_ulonglong2(xk, ck));
  }
}

// The same where a vertex may be a hub, whose records would queue at its few lines
// of memory: a CTA has one layer group; it looks for a hub, the vertex that one of
// its warps has most records of, if that is more than a quarter, sums its rows
// below kHubRows in shared memory and sends each once. A kernel of its own: as one
// template with k_small, batches of 160 to 256 edges took 6.2 us instead of 4.9
// to 5.7 (V = 1024).
constexpr uint32_t kHubRows = 4;
template <bool kX32>
__global__ void __launch_bounds__(1024) k_small_hubs(ulonglong2* __restrict__ sketch,
                                                     const uint64_t* __restrict__ keys,
                                                     const uint32_t* __restrict__ edges,
                                                     const int8_t* __restrict__ ops, uint32_t n, uint32_t* gc,
                                                     uint32_t V, uint32_t L, uint32_t C, uint32_t D, uint32_t W,
                                                     uint32_t P, uint32_t ell) {
  __shared__ uint32_t s_sum[kHubRows][4][32];  // [row][word][lane]: its slot's sum over the CTA
  __shared__ uint32_t s_most[32];              // of each warp: records << 24 | vertex
  static_assert(kMaxVertices <= 1u << 24, "a vertex id fits beside the count");
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, warps = blockDim.x >> 5, s = lane % P;
  const uint32_t groups = layer_groups(L, P);
  // this warp's records and lanes, in flight during the validation
  const uint32_t i = (blockIdx.x / groups * warps + wid) * P + s;  // endpoint i & 1 of edge i / 2
  const bool have = i < 2 * n;
  const uint32_t w = have ? edges[i] : 0, other = have ? edges[i ^ 1] : 0;
  const ApplyLane l = apply_lane(keys, sketch, V, L, C, D, W, P, ell, blockIdx.x % groups);
  for (uint32_t k = threadIdx.x; k < kHubRows * 4 * 32; k += blockDim.x) (&s_sum[0][0][0])[k] = 0;
  bool drop = (ld_cg(&gc[GC_ERR]) & kErrInval) != 0, bad = false;
#pragma unroll 4
  for (uint32_t j = threadIdx.x; j < n; j += blockDim.x) {
    const uint32_t u = edges[2 * j], v = edges[2 * j + 1];
    const int8_t op = ops[j];
    bad |= (u >= V) | (v >= V) | (u == v) | ((op != 1) & (op != -1));
  }
  const uint32_t same = __popc(__match_any_sync(0xffffffffu, w)) / (32 / P);  // the layers repeat the records
  const uint32_t mine =
      __reduce_max_sync(0xffffffffu, have && same > max(1u, P / 4) ? same << 24 | (w & 0xFFFFFFu) : 0u);
  if (lane == 0) s_most[wid] = mine;
  if (__syncthreads_or(bad)) {
    if (threadIdx.x == 0) atomicOr(&gc[GC_ERR], kErrInval);
    drop = true;
  }
  if (__syncthreads_or(drop)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) gc[GC_BATCHES] += 1;
  const uint32_t most = __reduce_max_sync(0xffffffffu, lane < warps ? s_most[lane] : 0u);
  const uint32_t hub = most ? most & 0xFFFFFFu : kNoneU32;
  const uint64_t x = record_id(make_record(w, other), V), c = mix64(x ^ l.kchk);  // of this lane's layer
  for (uint32_t k = 0; k < P; k++) {
    const uint32_t from = (lane & ~(P - 1)) + k;
    const bool in = __shfl_sync(0xffffffffu, have, from);
    const uint32_t wk = __shfl_sync(0xffffffffu, w, from);
    const uint64_t xk = __shfl_sync(0xffffffffu, x, from), ck = __shfl_sync(0xffffffffu, c, from);
    if (!l.active || !in) continue;
    const uint32_t row = lane_depth<kX32>(l, xk);
    if (wk == hub && row < kHubRows) {
      atomicXor(&s_sum[row][0][lane], (uint32_t)xk);
      if (!kX32) atomicXor(&s_sum[row][1][lane], (uint32_t)(xk >> 32));
      atomicXor(&s_sum[row][2][lane], (uint32_t)ck);
      atomicXor(&s_sum[row][3][lane], (uint32_t)(ck >> 32));
    } else {
      xor_bucket_atomic(l.base + (size_t)wk * W + row, make_ulonglong2(xk, ck));
    }
  }
  if (hub == kNoneU32) return;
  __syncthreads();
  for (uint32_t q = wid; q < kHubRows; q += warps) {
    const ulonglong2 v = make_ulonglong2((uint64_t)s_sum[q][1][lane] << 32 | s_sum[q][0][lane],
                                         (uint64_t)s_sum[q][3][lane] << 32 | s_sum[q][2][lane]);
    if (v.x | v.y) xor_bucket_atomic(l.base + (size_t)hub * W + q, v);
  }
}

// The dynamic shared-memory limit of k_apply is process-wide: only ever
// raise it, so that a graph created later never shrinks it below what an
// earlier graph's launches need.
cudaError_t raise_apply_smem_limit(int bytes) {
  const void* fns[2] = {(const void*)k_apply<false>, (const void*)k_apply<true>};
  for (const void* f : fns) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
    if (fa.maxDynamicSharedSizeBytes >= bytes) continue;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t setup_update(cupc_graph* g) {
  // the shared histograms of the dense-batch grouping (fixed maximum sizes)
  cudaError_t e = cudaFuncSetAttribute(k_count_priv, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * kPrivMaxV);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_scatter_priv, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * kPrivMaxV);
  if (e != cudaSuccess) return e;
  g->P = 1;
  while (g->P < g->C + 1) g->P <<= 1;
  g->R = g->D < kSmemRows ? g->D : kSmemRows;
  g->ell = hash_bits(g->V);
  g->item_records = kDefaultItemRecords;
  g->item_default = true;
  g->apply_cps = 0;
  return configure_apply(g);
}

// Shared memory and persistent grid of k_apply for the given tunables.
cudaError_t apply_config(const cupc_graph* g, uint32_t R, uint32_t cps, int* smem, int* grid) {
  // the range of settings the entry points have always taken, which is less than
  // this kernel could launch with (at most 80 KB of shared memory a CTA)
  if ((size_t)R * layer_groups(g->L, g->P) * 512 + (size_t)g->L * 520 + 1536 > 232448) return cudaErrorInvalidValue;
  *smem = (int)(kApplyWarps * apply_warp_bytes(fold_rows(R, g->D), g->P));
  cudaError_t e = raise_apply_smem_limit(*smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_apply<false>, 32 * kApplyWarps, *smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  if (cps && (int)cps < per_sm) per_sm = (int)cps;
  *grid = per_sm * g->sms;
  return cudaSuccess;
}

// ... and for the graph's default tunables.
cudaError_t configure_apply(cupc_graph* g) {
  return apply_config(g, g->R, g->apply_cps, &g->apply_smem, &g->apply_grid);
}

cudaError_t launch_update_chunk(cupc_graph* g, const uint32_t* edges, size_t n, cudaStream_t s,
                                const int8_t* validate_ops) {
  if (n == 0) return cudaSuccess;
  if (validate_ops && n <= kSmallEdges) {
    ProfScope ps(g, s, PC_APPLY, 1);
    const bool hubs = n > kSmallHubEdges && g->V > kSmallHubV;
    const uint32_t threads = n <= 512 ? 128 : n > 8192 ? 1024 : hubs ? 512 : 256;
    const uint32_t per = threads / 32, groups = layer_groups(g->L, g->P);
    const uint32_t parts = (uint32_t)((2 * n + g->P - 1) / g->P);  // warps of a layer group
    const uint32_t grid = hubs ? (parts + per - 1) / per * groups : (parts * groups + per - 1) / per;
    auto kern = hubs ? (small_ids(g->V) ? k_small_hubs<true> : k_small_hubs<false>)
                     : (small_ids(g->V) ? k_small<true> : k_small<false>);
    kern<<<grid, threads, 0, s>>>(g->sketch, g->keys, edges, validate_ops, (uint32_t)n, g->gc, g->V, g->L, g->C, g->D,
                                  g->W, g->P, g->ell);
    return cudaGetLastError();
  }
  // the setting of this batch size's bucket, else the graph's default
  uint32_t ir = g->item_records, R = g->R;
  bool ir_default = g->item_default;
  int smem = g->apply_smem, grid_max = g->apply_grid;
  const cupc_graph::ApplyTune& t = g->tune_b[tune_bucket(n)];
  if (t.set) {
    ir = t.item_records;
    ir_default = t.item_default;
    R = t.R;
    smem = t.smem;
    grid_max = t.grid;
  }
  const int grid = (int)std::min<size_t>((n + 255) / 256, (size_t)g->sms * 8);
  // dense batch on a small graph: group through shared histograms
  const int pgrid = (int)std::min<size_t>((size_t)g->sms, 2 * n / ((size_t)kPrivPerVertex * g->V));
  const bool priv = g->V <= kPrivMaxV && pgrid >= (int)kPrivMinCtas;
  const uint32_t shards = !priv && n >= kShardEdges ? g->shards : 1u;
  const uint32_t nrec = (uint32_t)(2 * n);
  const uint32_t groups = layer_groups(g->L, g->P), warps = (uint32_t)grid_max * kApplyWarps / groups;
  // the chunks if hubs hold little of the batch, and if they hold much of it
  const uint32_t chunk = chunk_records(nrec, g->V, warps, ir_default ? default_most(nrec, g->V, warps) : ir);
  const uint32_t hub_chunk = g->V <= kPrivMaxV && nrec / g->V >= kHubMean ? hub_chunk_records(nrec, warps, ir)
                                                                          : chunk_records(nrec, g->V, warps, ir);
  {
    ProfScope ps(g, s, PC_GROUP, 3);
    if (priv)
      k_count_priv<<<pgrid, 1024, 4 * g->V, s>>>(edges, validate_ops, n, g->V, g->cnt, g->work, g->gc);
    else
      k_count<<<grid, 256, 0, s>>>(edges, validate_ops, n, g->V, g->cnt, shards, g->work, g->gc);
    k_plan<<<plan_slices(g->V), kPlanThreads, 0, s>>>(g->cnt, g->cursor, g->rec, g->V, g->rec_cap, shards,
                                                       chunk != hub_chunk ? hub_records(nrec, g->V) : kNoneU32, g->work,
                                                       g->gc);
    if (priv)
      k_scatter_priv<<<pgrid, 1024, 8 * g->V, s>>>(edges, n, g->V, g->cursor, g->rec, g->gc);
    else
      k_scatter<<<grid, 256, 0, s>>>(edges, n, g->V, g->cursor, shards, g->rec, g->gc);
  }
  ProfScope ps(g, s, PC_APPLY, 1);
  // at most: chunks of padded fold records and of direct records
  const size_t units = (size_t)(rec_entries(g->V, n) / std::min(chunk, hub_chunk) + 2) * groups;
  const int agrid = (int)std::min<size_t>((size_t)grid_max, (units + kApplyWarps - 1) / kApplyWarps);
  auto kern = small_ids(g->V) ? k_apply<true> : k_apply<false>;
  kern<<<agrid, 32 * kApplyWarps, smem, s>>>(g->sketch, g->keys, g->rec, g->rec_cap, chunk, hub_chunk, g->work, g->gc,
                                             g->V, g->L, g->C, g->D, g->W, g->P, fold_rows(R, g->D), g->ell);
  return cudaGetLastError();
}

cudaError_t launch_update(cupc_graph* g, const uint32_t* edges, size_t n, cudaStream_t s, const int8_t* ops) {
  if (n <= g->max_chunk) return launch_update_chunk(g, edges, n, s, ops);  // validated on the way
  cudaError_t e = ops ? launch_validate(g, edges, ops, n, s) : cudaSuccess;
  for (size_t i = 0; e == cudaSuccess && i < n; i += g->max_chunk)
    e = launch_update_chunk(g, edges + 2 * i, std::min<size_t>(n - i, g->max_chunk), s);
  return e;
}

}  // namespace cupc

extern "C" cupc_status cupc_build_info(int* binary_version, int* ptx_version) {
  if (!binary_version || !ptx_version) return CUPC_EINVAL;
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, (const void*)cupc::k_apply<false>) != cudaSuccess) {
    cudaGetLastError();
    return CUPC_ECUDA;
  }
  *binary_version = fa.binaryVersion;
  *ptx_version = fa.ptxVersion;
  return CUPC_OK;
}

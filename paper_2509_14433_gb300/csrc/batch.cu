// Batching: update batches of many graphs in one launch per stage.
//
// A cupc_batcher applies one batch to each of k graphs (App. A.1.1: every
// update touches every sketch of both endpoints; graphs are independent)
// with four launches in all, whatever k is: count (which also validates),
// plan, scatter and apply each cover every graph. Their arguments live in a
// descriptor table in device memory (one InstDesc per graph, prefix offsets
// of edges, plan slices and work units), so the launch sequence is fixed for
// a batcher and is captured once as a CUDA graph and replayed; each call only
// refreshes the table with one host-to-device copy (double-buffered pinned
// staging). A work unit is one chunk of a graph's records for one of its
// layer groups; the units of all graphs are laid end to end and dealt to
// persistent warps in turn, which apply them with the single-graph kernel's
// code (apply_chunk). Results are identical to k separate cupc_update_batch
// calls.
#include <string.h>

#include <new>
#include <vector>

#include "update_dev.cuh"

namespace cupc {

struct alignas(16) InstDesc {
  const uint32_t* edges;
  const int8_t* ops;
  ulonglong2* sketch;
  const uint64_t* keys;
  uint32_t* cnt;
  uint32_t* cursor;
  uint64_t* rec;
  uint32_t* work;
  uint32_t* gc;
  uint64_t edge_base;   // first edge of this graph in the launch's edge space
  uint32_t slice_base;  // first plan slice
  uint32_t unit_base;   // first work unit: chunk c of layer group l is unit_base + l * nchunks + c (k_scatter_m)
  uint32_t n, V, L, C, D, W, P, R;
  uint32_t ell;         // bits of one column-hash stage
  uint32_t chunk;       // records per chunk
  uint32_t nchunks;     // chunks of the fold and the direct records, 0 if dropped (k_scatter_m)
  uint32_t cap;         // entries of rec
  uint32_t small;       // edge ids of at most 32 bits
};

struct alignas(16) BatchHead {
  uint32_t k;             // graphs in this launch
  uint32_t total_units;   // set by k_scatter_m
  uint32_t total_slices;
  uint32_t next_unit;     // 0 in every copy of the table
  uint64_t total_edges;
  uint64_t pad[5];
};

static_assert(sizeof(BatchHead) == 64, "head size");
static_assert(sizeof(InstDesc) % 16 == 0, "descriptor alignment");

__device__ __forceinline__ const InstDesc* descs_of(const BatchHead* h) {
  return reinterpret_cast<const InstDesc*>(h + 1);
}

// Graph holding global edge i: the last j with edge_base <= i.
__device__ __forceinline__ uint32_t inst_of_edge(const InstDesc* d, uint32_t k, uint64_t i) {
  uint32_t lo = 0, hi = k;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (d[mid].edge_base <= i)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// Graph holding plan slice (kUnits: work unit) x.
template <bool kUnits>
__device__ __forceinline__ uint32_t inst_of(const InstDesc* d, uint32_t k, uint32_t x) {
  uint32_t lo = 0, hi = k;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if ((kUnits ? d[mid].unit_base : d[mid].slice_base) <= x)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// Counts of every graph's batch, and its validation (Problem 1's stream); an
// invalid batch's counts are cleared by k_plan_m.
__global__ void k_count_m(const BatchHead* __restrict__ h) {
  const InstDesc* d = descs_of(h);
  const uint32_t k = h->k;
  const uint64_t total = h->total_edges;
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < k) d[t].work[kWorkFold] = d[t].work[kWorkDirect] = 0;
  for (uint64_t i = t; i < total; i += (uint64_t)gridDim.x * blockDim.x) {
    const InstDesc& g = d[inst_of_edge(d, k, i)];
    const uint64_t j = i - g.edge_base;
    const uint32_t u = g.edges[2 * j], v = g.edges[2 * j + 1];
    const int8_t op = g.ops[j];
    if ((u >= g.V) | (v >= g.V) | (u == v) | ((op != 1) & (op != -1))) {
      atomicOr(&g.gc[GC_ERR], kErrInval);
    } else if (!(ld_cg(&g.gc[GC_ERR]) & kErrInval)) {
      atomicAdd(&g.cnt[u], 1u);
      atomicAdd(&g.cnt[v], 1u);
    }
  }
}

__global__ void __launch_bounds__(kPlanThreads) k_plan_m(const BatchHead* __restrict__ h) {
  const InstDesc* d = descs_of(h);
  const uint32_t k = h->k;
  for (uint32_t x = blockIdx.x; x < h->total_slices; x += gridDim.x) {
    const InstDesc& g = d[inst_of<false>(d, k, x)];
    const bool dropped = (ld_cg(&g.gc[GC_ERR]) & kErrInval) != 0;
    plan_slice(g.cnt, g.cursor, g.rec, g.V, g.cap, x - g.slice_base, g.work, dropped, 1u, kNoneU32);
    if (!dropped && g.n > 0 && x == g.slice_base && threadIdx.x == 0) g.gc[GC_BATCHES] += 1;
  }
}

// Lay the graphs' work units end to end, by one CTA.
__device__ __forceinline__ void number_units(BatchHead* h) {
  InstDesc* d = const_cast<InstDesc*>(descs_of(h));
  const uint32_t k = h->k;
  uint64_t run = 0;
  for (uint32_t j0 = 0; j0 < k; j0 += blockDim.x) {
    const uint32_t j = j0 + threadIdx.x;
    uint32_t nchunks = 0, units = 0;
    if (j < k && d[j].n && !(ld_cg(&d[j].gc[GC_ERR]) & kErrInval)) {
      nchunks = chunk_plan(d[j].work, d[j].chunk, d[j].chunk).total;
      units = nchunks * layer_groups(d[j].L, d[j].P);
    }
    uint64_t total;
    const uint64_t before = block_scan(units, &total);
    if (j < k) {
      d[j].unit_base = (uint32_t)(run + before);
      d[j].nchunks = nchunks;
    }
    run += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) h->total_units = (uint32_t)run;
}

__global__ void k_scatter_m(BatchHead* __restrict__ h) {
  const InstDesc* d = descs_of(h);
  const uint32_t k = h->k;
  const uint64_t total = h->total_edges;
  if (blockIdx.x == gridDim.x - 1) number_units(h);  // read by k_apply_m only
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (uint64_t)gridDim.x * blockDim.x) {
    const InstDesc& g = d[inst_of_edge(d, k, i)];
    if (ld_cg(&g.gc[GC_ERR]) & kErrInval) continue;
    const uint64_t j = i - g.edge_base;
    const uint32_t u = g.edges[2 * j], v = g.edges[2 * j + 1];
    const uint32_t pu = atomicAdd(&g.cursor[u], 1u), pv = atomicAdd(&g.cursor[v], 1u);
    g.rec[pu] = make_record(u, v);
    g.rec[pv] = make_record(v, u);
  }
}

struct Unit {
  uint32_t j, group;
  Chunk c;
};
__device__ __forceinline__ Unit unit_at(const InstDesc* d, uint32_t k, uint32_t total, uint32_t x) {
  Unit u{0, 0, {nullptr, 0, false}};
  if (x >= total) return u;
  u.j = inst_of<true>(d, k, x);
  const InstDesc& g = d[u.j];
  const uint32_t at = x - g.unit_base;
  u.group = at / g.nchunks;
  u.c = chunk_at(chunk_plan(g.work, g.chunk, g.chunk), at % g.nchunks, g.rec, g.cap);
  return u;
}

// The units go to the warps in order, so that the warps at work at one time
// are on neighbouring vertices: what bounds the kernel is memory, and equal
// runs of consecutive units per warp (fewer layout changes) were slower, 501
// against 465 us for 64 graphs of 1024..8192 vertices and 1000 edges each,
// 1210 against 1060 us with 4000 edges, as their accesses are spread over all
// of the graphs' memory. A warp asks for its units two ahead, so that the next
// unit's records load during the current one, and rebuilds the lane layout
// when the graph or the layer group changes.
__global__ void __launch_bounds__(32 * kApplyWarps, kApplyCtas) k_apply_m(BatchHead* __restrict__ h,
                                                                         uint32_t warp_bytes) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* mine = smem_raw + (threadIdx.x >> 5) * warp_bytes;
  const InstDesc* d = descs_of(h);
  const uint32_t k = h->k, total = h->total_units, warps = gridDim.x * kApplyWarps;
  uint32_t x = blockIdx.x * kApplyWarps + (threadIdx.x >> 5), cur_j = kNoneU32, cur_group = 0;
  ApplyLane l{};
  ApplySmem m{};
  LaneSums a;
  clear_sums(a);
  a.dirty = 0;
  bool pending = false;
  Unit u = unit_at(d, k, total, x);
  uint64_t r = load_record(u.c, 0, u.c);
  x += warps;
  while (u.c.n) {
    const Unit next = unit_at(d, k, total, x);
    uint32_t ahead = x;
    if ((threadIdx.x & 31) == 0 && next.c.n) ahead = 2 * warps + atomicAdd(&h->next_unit, 1u);
    const InstDesc& g = d[u.j];
    if (u.j != cur_j || u.group != cur_group) {
      reuse_slots(m, a, pending);
      __syncwarp();
      if (u.j != cur_j) {  // another slot layout: its slots start at zero
        m = apply_smem(mine, apply_slots(g.R), g.P);
        zero_slots(m, apply_slots(g.R));
      }
      l = apply_lane(g.keys, g.sketch, g.V, g.L, g.C, g.D, g.W, g.P, g.ell, u.group);
      cur_j = u.j;
      cur_group = u.group;
      __syncwarp();
    }
    if (g.small)
      apply_chunk<true>(l, m, a, pending, u.c, next.c, r, g.V, g.W, g.C, g.P, g.R);
    else
      apply_chunk<false>(l, m, a, pending, u.c, next.c, r, g.V, g.W, g.C, g.P, g.R);
    u = next;
    x = __shfl_sync(0xffffffffu, ahead, 0);
  }
  bulk_wait_all();
}

}  // namespace cupc

using namespace cupc;

struct cupc_batcher {
  uint32_t max_graphs;
  int sms;
  bool use_graph;
  size_t table_bytes;
  BatchHead* dtab;
  BatchHead* htab[2];
  cudaEvent_t used[2];
  int cur;
  cudaStream_t cap_stream;
  struct Exec {
    uint32_t warp_bytes;
    int apply_grid, apply_smem;
    cudaGraphExec_t exec[2];
  };
  std::vector<Exec> execs;
};

namespace {

bool is_dev(const void* p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

cudaError_t enqueue(cupc_batcher* b, int slot, const cupc_batcher::Exec& x, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(b->dtab, b->htab[slot], b->table_bytes, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  const int grid = b->sms * 8;
  k_count_m<<<grid, 256, 0, s>>>(b->dtab);
  k_plan_m<<<grid, kPlanThreads, 0, s>>>(b->dtab);
  k_scatter_m<<<grid, 256, 0, s>>>(b->dtab);
  k_apply_m<<<x.apply_grid, 32 * kApplyWarps, x.apply_smem, s>>>(b->dtab, x.warp_bytes);
  return cudaGetLastError();
}

cudaError_t get_exec(cupc_batcher* b, uint32_t warp_bytes, cupc_batcher::Exec** out) {
  for (auto& x : b->execs)
    if (x.warp_bytes == warp_bytes) {
      *out = &x;
      return cudaSuccess;
    }
  cupc_batcher::Exec x{};
  x.warp_bytes = warp_bytes;
  x.apply_smem = (int)(kApplyWarps * warp_bytes);
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, k_apply_m);
  if (e != cudaSuccess) return e;
  if (fa.maxDynamicSharedSizeBytes < x.apply_smem) {
    e = cudaFuncSetAttribute(k_apply_m, cudaFuncAttributeMaxDynamicSharedMemorySize, x.apply_smem);
    if (e != cudaSuccess) return e;
  }
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_apply_m, 32 * kApplyWarps, x.apply_smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  x.apply_grid = per_sm * b->sms;
  if (b->use_graph) {
    for (int slot = 0; slot < 2; slot++) {
      cudaGraph_t graph;
      e = cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal);
      if (e != cudaSuccess) return e;
      cudaError_t e2 = enqueue(b, slot, x, b->cap_stream);
      e = cudaStreamEndCapture(b->cap_stream, &graph);
      if (e2 != cudaSuccess) return e2;
      if (e != cudaSuccess) return e;
      e = cudaGraphInstantiate(&x.exec[slot], graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) return e;
    }
  }
  b->execs.push_back(x);
  *out = &b->execs.back();
  return cudaSuccess;
}

}  // namespace

extern "C" {

cupc_status cupc_batcher_create(uint32_t max_graphs, int use_cuda_graph, cupc_batcher** out) {
  if (!out || max_graphs == 0 || max_graphs > 4096) return CUPC_EINVAL;
  *out = nullptr;
  cupc_batcher* b = new (std::nothrow) cupc_batcher();
  if (!b) return CUPC_ENOMEM;
  b->max_graphs = max_graphs;
  b->use_graph = use_cuda_graph != 0;
  b->table_bytes = sizeof(BatchHead) + (size_t)max_graphs * sizeof(InstDesc);
  int dev = 0;
  bool ok = cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaMalloc((void**)&b->dtab, b->table_bytes) == cudaSuccess &&
            cudaMallocHost((void**)&b->htab[0], b->table_bytes) == cudaSuccess &&
            cudaMallocHost((void**)&b->htab[1], b->table_bytes) == cudaSuccess &&
            cudaEventCreateWithFlags(&b->used[0], cudaEventDisableTiming) == cudaSuccess &&
            cudaEventCreateWithFlags(&b->used[1], cudaEventDisableTiming) == cudaSuccess &&
            cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    cupc_batcher_destroy(b);
    return CUPC_ENOMEM;
  }
  *out = b;
  return CUPC_OK;
}

cupc_status cupc_batcher_update(cupc_batcher* b, cupc_graph* const* graphs, const uint32_t* const* edges,
                                const int8_t* const* ops, const size_t* n, uint32_t k, cupc_stream stream) {
  if (!b || (k && (!graphs || !edges || !ops || !n)) || k > b->max_graphs) return CUPC_EINVAL;
  if (k == 0) return CUPC_OK;
  cudaStream_t s = (cudaStream_t)stream;
  for (uint32_t i = 0; i < k; i++) {
    if (!graphs[i] || n[i] > graphs[i]->max_batch) return CUPC_EINVAL;
    if (n[i] && (!is_dev(edges[i]) || !is_dev(ops[i]))) return CUPC_EINVAL;
    for (uint32_t j = 0; j < i; j++)
      if (graphs[j] == graphs[i]) return CUPC_EINVAL;
  }
  const int slot = b->cur;
  if (cudaEventSynchronize(b->used[slot]) != cudaSuccess) return CUPC_ECUDA;
  BatchHead* h = b->htab[slot];
  memset(h, 0, sizeof(BatchHead) + (size_t)k * sizeof(InstDesc));
  InstDesc* d = reinterpret_cast<InstDesc*>(h + 1);
  uint64_t base = 0, units = 0, work = 0, records = 0, vertices = 0;
  uint32_t slices = 0, warp_bytes = 0;
  // a batch longer than one chunk gets its graph's own launch sequence, and
  // none of the joined one
  auto joined = [&](uint32_t i) { return n[i] <= graphs[i]->max_chunk ? (uint32_t)n[i] : 0u; };
  for (uint32_t i = 0; i < k; i++) {
    if (n[i] && !joined(i) && launch_update(graphs[i], edges[i], n[i], s, ops[i]) != cudaSuccess) return CUPC_ECUDA;
    work += 2 * (uint64_t)joined(i) * layer_groups(graphs[i]->L, graphs[i]->P);
    records += 2 * (uint64_t)joined(i);
    vertices += graphs[i]->V;
  }
  // records per chunk: about three units for each warp of a full device, but
  // one pass where vertices get two records or fewer on average: nearly all
  // records then go straight to HBM, and short units keep the warps on
  // neighbouring vertices (64 graphs of 1024..8192 vertices, 1000 edges each:
  // 462 us, 480 with 48..64 records; 4000 edges each: 1131, 1059)
  const uint64_t per = work / (3ull * b->sms * kApplyWarps * kApplyCtas);
  const uint32_t chunk =
      records <= 2 * vertices ? kStage : (uint32_t)std::min<uint64_t>(kDefaultItemRecords, (per + 16) / 16 * 16);
  for (uint32_t i = 0; i < k; i++) {
    cupc_graph* g = graphs[i];
    InstDesc& x = d[i];
    x.edges = edges[i];
    x.ops = ops[i];
    x.sketch = g->sketch;
    x.keys = g->keys;
    x.cnt = g->cnt;
    x.cursor = g->cursor;
    x.rec = g->rec;
    x.work = g->work;
    x.gc = g->gc;
    x.edge_base = base;
    x.n = joined(i);
    x.V = g->V;
    x.L = g->L;
    x.C = g->C;
    x.D = g->D;
    x.W = g->W;
    x.P = g->P;
    x.R = fold_rows(g->R, g->D);
    x.ell = g->ell;
    x.small = small_ids(g->V) ? 1u : 0u;
    x.chunk = chunk;
    x.cap = g->rec_cap;
    x.slice_base = slices;
    base += x.n;
    if (x.n) slices += plan_slices(g->V);
    units += (uint64_t)layer_groups(g->L, g->P) * (rec_entries(g->V, x.n) / chunk + 2);
    warp_bytes = std::max(warp_bytes, apply_warp_bytes(x.R, x.P));
  }
  if (units >= 0xFFFFFFFFull) return CUPC_EINVAL;
  h->k = k;
  h->total_edges = base;
  h->total_slices = slices;
  cupc_batcher::Exec* x = nullptr;
  if (get_exec(b, warp_bytes, &x) != cudaSuccess) {
    cudaGetLastError();
    return CUPC_ECUDA;
  }
  cudaError_t e = b->use_graph ? cudaGraphLaunch(x->exec[slot], s) : enqueue(b, slot, *x, s);
  if (e != cudaSuccess) return CUPC_ECUDA;
  if (cudaEventRecord(b->used[slot], s) != cudaSuccess) return CUPC_ECUDA;
  b->cur ^= 1;
  // like cupc_update_batch: the next query recovers; the batcher does not
  // follow incremental labels, so a graph in that mode drops them
  for (uint32_t i = 0; i < k; i++) {
    if (!n[i]) continue;
    graphs[i]->dirty = true;
    graphs[i]->forest_stale = true;
    if (graphs[i]->inc && cudaMemsetAsync(graphs[i]->gc + GC_LABELS_VALID, 0, sizeof(uint32_t), s) != cudaSuccess)
      return CUPC_ECUDA;
  }
  return CUPC_OK;
}

void cupc_batcher_destroy(cupc_batcher* b) {
  if (!b) return;
  for (int i = 0; i < 2; i++) {
    if (b->used[i]) cudaEventSynchronize(b->used[i]);
  }
  for (auto& x : b->execs)
    for (int i = 0; i < 2; i++)
      if (x.exec[i]) cudaGraphExecDestroy(x.exec[i]);
  if (b->dtab) cudaFree(b->dtab);
  for (int i = 0; i < 2; i++) {
    if (b->htab[i]) cudaFreeHost(b->htab[i]);
    if (b->used[i]) cudaEventDestroy(b->used[i]);
  }
  if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
  delete b;
}

cupc_status cupc_update_batches(cupc_graph* g, const uint32_t* edges, const int8_t* ops, const uint64_t* offsets,
                                size_t k, cupc_stream stream) {
  if (!g || (k && !offsets)) return CUPC_EINVAL;
  if (k == 0) return CUPC_OK;
  for (size_t i = 0; i < k; i++)
    if (offsets[i + 1] < offsets[i]) return CUPC_EINVAL;
  // consecutive batches stored back to back are one batch: sketch addition
  // is XOR, so applying their concatenation equals applying them in order
  const uint64_t first = offsets[0], total = offsets[k] - offsets[0];
  return cupc_update_batch(g, edges + 2 * first, ops + first, total, stream);
}

}  // extern "C"

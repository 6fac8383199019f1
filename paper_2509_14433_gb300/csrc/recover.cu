// Spanning-forest recovery by Boruvka rounds over the vertex sketches
// (App. A.1.1, "The AGM Algorithm": query each supernode's merged sketch for
// an edge leaving it, merge supernodes and their sketches, repeat for
// O(log V) rounds) and Connected(u,v) answers from the result (Problem 2).
//
// The whole recovery is one cooperative launch: every CTA is co-resident, and
// the phases of a round are separated by a grid barrier whose wait is bounded
// (on expiry it sets the timeout error and every CTA returns). Round r:
//   group       live vertices grouped by component label (count, segment
//               offsets, scatter); round 0 skips it: every vertex is its own
//               component
//   reduce      an equal run of the live members per warp, lane l XORing
//               buckets l and l + 32 of layer r of each. A component inside
//               one run is sampled in place; one over several is XORed into
//               its accumulator and sampled by the last run to finish.
//               Buckets are read kPrefix at a time, the later ones only where
//               the earlier ones do not decide the sample
//   sample      ZERO / GOOD(edge) / FAIL, first good bucket in index order;
//               32 samples of a warp are booked at once
//   hook        minimum spanning forest (weights = edge ids) of the candidate
//               edges over the round-start components: grid-wide Boruvka
//               steps with min-id edges until at most kSmallHook candidates
//               still cross two trees, then one CTA finishes in shared
//               memory; it adds exactly the edges Kruskal in ascending id
//               order would
//   relabel     every vertex takes the root of its component (after the last
//               round, its minimum vertex id)
// A component whose merged sketch is ZERO has an empty cut; it is not sampled
// again until it changes. With one live component left its merged sketch is
// zero by linearity, so the round is logged without reading its layer.
#include "recover_dev.cuh"

namespace cupc {


// Release and acquire at device scope: what a CTA wrote before its arrival is
// seen by every CTA after the barrier (__syncthreads orders the CTA's other
// threads with the arriving one). Cheaper than the sequentially consistent
// fences of __threadfence.
__device__ __forceinline__ void red_release(uint32_t* p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t atom_add_acq_rel(uint32_t* p, uint32_t v) {
  uint32_t old;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}

// Grid barrier for a cooperative launch: CTA thread 0 adds one to an arrival
// counter that only grows during the launch (zero before it) and waits until
// all CTAs of this barrier have arrived. The wait is bounded:
// after kWaitLimitNs it records kErrTimeout and returns false in every
// thread of the CTA, which must then return.
__device__ __forceinline__ bool grid_barrier(uint32_t* gc, uint32_t nblocks, uint32_t& epoch, int* s_ok,
                                             uint64_t limit_ns = kWaitLimitNs) {
  __syncthreads();
  if (threadIdx.x == 0) {
    epoch += 1;
    const uint32_t target = epoch * nblocks;
    int ok = 1;
    red_release(&gc[GC_BAR_COUNT], 1u);
    uint64_t t0 = 0;
    for (uint32_t spin = 0; ld_acquire(&gc[GC_BAR_COUNT]) < target; spin++) {
      if ((spin & 63) == 63) {
        const uint64_t t = global_timer_ns();
        if (t0 == 0) t0 = t;
        if (ld_cg(&gc[GC_ERR]) & kErrTimeout) {
          ok = 0;
          break;
        }
        if (t - t0 > limit_ns) {
          atomicOr(&gc[GC_ERR], kErrTimeout);
          atomicOr(&gc[GC_REC_DIRTY], 1u);
          ok = 0;
          break;
        }
      }
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// Root of x in the hook forest; points x straight at it and, on the way, every
// second node at its grandparent: the walks of one phase start together, so
// they shorten each other's paths. Other threads may rewrite parent[]
// concurrently, but only ever to an ancestor, so every value read is an
// ancestor and the walk ends at the same root.
__device__ __forceinline__ uint32_t find_root(uint32_t* parent, uint32_t x, uint32_t V) {
  uint32_t r = x;
  for (uint32_t k = 0; k < V; k++) {
    const uint32_t p = ld_cg(&parent[r]);
    if (p == r) break;
    const uint32_t g = ld_cg(&parent[p]);
    if (g == p) {
      r = p;
      break;
    }
    parent[r] = g;
    r = g;
  }
  if (r != x && ld_cg(&parent[x]) != r) parent[x] = r;
  return r;
}

// The roots of x and y, their walks side by side. Read only: a store to a node
// near a root, which every walk of a phase passes, makes all of them wait (a
// relabel of V = 2^14 took 10 to 50 us with find_root, all SMs leaving it at the
// same moment, against 3). Of a chain of n hooks, walked by threads that start
// together, a walk takes at most about sqrt(2n) steps, as each thread points its
// own component at the root behind its walk: a stream's samples make chains of
// tens, and imported words that make one chain of all vertices recover in 267 us
// at V = 2^17, 1.6 ms at 2^20, 3.2 ms at 2^21 (434 us, 2.8 and 5.6 ms with
// find_root).
__device__ __forceinline__ void walk_roots(const uint32_t* parent, uint32_t& x, uint32_t& y, uint32_t V) {
  for (uint32_t k = 0; k < V; k++) {
    const uint32_t p = ld_cg(&parent[x]), q = ld_cg(&parent[y]);
    if (p == x && q == y) break;
    x = p;
    y = q;
  }
}

// Book the samples stashed in a warp, one per lane (K = kNoneU32: none):
// ZERO marks the component final; GOOD with an edge that leaves K becomes
// its candidate (stored with both endpoint labels) and is logged; GOOD with
// an edge inside K is a checksum false positive. Counters are aggregated per
// warp. Every lane of the warp must call this.
__device__ __forceinline__ void book_samples(const RecArgs& a, uint32_t r, bool multi, uint32_t K, uint32_t res,
                                             uint64_t e) {
  const uint32_t lane = threadIdx.x & 31;
  const bool have = K != kNoneU32;
  bool cand = false;
  if (have) {
    if (res == 0) {
      a.final_[K] = 1;
    } else if (res == 1) {
      uint64_t u, v;
      a.ids.split(e, u, v);
      const uint32_t lu = multi ? ld_cg(&a.label[u]) : (uint32_t)u,
                     lv = multi ? ld_cg(&a.label[v]) : (uint32_t)v;
      if ((lu == K) != (lv == K)) {
        cand = true;
        a.cand[K] = make_ulonglong2(e, ((uint64_t)lu << 32) | lv);
      }
    }
  }
  const uint32_t m_have = __ballot_sync(0xffffffffu, have);
  const uint32_t m_nz = __ballot_sync(0xffffffffu, have && res != 0);
  const uint32_t m_fail = __ballot_sync(0xffffffffu, have && res == 2);
  const uint32_t m_cand = __ballot_sync(0xffffffffu, cand);
  const uint32_t m_fp = m_nz & ~m_fail & ~m_cand;
  uint32_t base = 0;
  if (lane == 0) {
    if (m_have) atomicAdd(&a.log_live[r], (uint32_t)__popc(m_have));
    if (m_nz) atomicAdd(&a.gc[GC_NZ], (uint32_t)__popc(m_nz));
    if (m_fail) atomicAdd(&a.gc[GC_NFAIL], (uint32_t)__popc(m_fail));
    if (m_fp) atomicAdd(&a.gc[GC_NFP], (uint32_t)__popc(m_fp));
    if (m_cand) {
      base = atomicAdd(&a.gc[GC_LOGLEN], (uint32_t)__popc(m_cand));
      atomicAdd(&a.log_ncand[r], (uint32_t)__popc(m_cand));
    }
  }
  base = __shfl_sync(0xffffffffu, base, 0);
  if (cand) a.log_ids[base + __popc(m_cand & ((1u << lane) - 1))] = e;
}

// Position of this lane's item in ctr[key]'s range: lanes of the warp with
// the same key share one atomicAdd. All 32 lanes call it; `take` selects the
// lanes that add one item.
__device__ __forceinline__ uint32_t warp_grab(uint32_t* ctr, uint32_t key, bool take) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t act = __ballot_sync(0xffffffffu, take);
  uint32_t peers = 0, leader = lane, base = 0;
  if (take) {
    peers = __match_any_sync(act, key);
    leader = __ffs(peers) - 1;
    if (lane == leader) base = atomicAdd(&ctr[key], (uint32_t)__popc(peers));
  }
  // one shuffle for all keys (one per key, with its lanes as the mask, would
  // run them one after another)
  base = __shfl_sync(0xffffffffu, base, leader);
  return take ? base + __popc(peers & ((1u << lane) - 1)) : 0;
}

// Root in a shared-memory forest with path halving; concurrent halving only
// ever points a node at an ancestor.
__device__ __forceinline__ uint32_t s_find(volatile uint32_t* par, uint32_t x) {
  for (uint32_t k = 0; k < 2 * kSmallHook; k++) {  // a path is shorter than the node count
    const uint32_t y = par[x];
    if (y == x) break;
    const uint32_t z = par[y];
    if (z != y) par[x] = z;
    x = y;
  }
  return x;
}

// The rest of a hook, run by one CTA once at most kSmallHook candidates
// still cross two trees (hlist[0..n): edge, both current roots): the same
// minimum spanning forest by Boruvka as the grid-wide steps (a root's key is
// edge << 11 | the root on the other side; two roots that chose the same
// edge hook once, the larger under the smaller), over local node ids, with
// __syncthreads between steps and pointer jumping after each hook step.
// Publishes parent[] of the roots that hooked and appends the forest edges.
// smem: kHookBytes.
static __device__ __noinline__ void small_hook(const RecArgs& a, uint32_t n, unsigned char* smem) {
  constexpr uint32_t kPer = kSmallHook / kRecThreads;  // candidates per thread
  constexpr uint32_t kNodeBits = 11;                    // nodes < 2 * kSmallHook
  static_assert(2 * kSmallHook <= (1u << kNodeBits), "node ids fit the key");
  uint64_t* s_best = reinterpret_cast<uint64_t*>(smem);  // 2 * kSmallHook
  uint32_t* s_par = reinterpret_cast<uint32_t*>(s_best + 2 * kSmallHook);
  uint32_t* s_lab = s_par + 2 * kSmallHook;  // node -> global root
  __shared__ uint32_t s_nn, s_nf, s_f0;
  const uint32_t tid = threadIdx.x, bd = blockDim.x;
  if (tid == 0) {
    s_nn = 0;
    s_nf = 0;
    s_f0 = ld_cg(&a.gc[GC_NFOREST]);  // the other CTAs wait at the grid barrier: this CTA owns the count
  }
  for (uint32_t x = tid; x < 2 * kSmallHook; x += bd) s_lab[x] = kNoneU32;
  __syncthreads();
  // node ids of the roots: the first claim of root x (a CAS on pcount[x],
  // zero at rest during the hook and cleared again at the end) takes a new
  // id, later claims read it; an id whose claim lost stays unused. All of a
  // thread's claims are in flight at once.
  uint64_t ce[kPer];  // this thread's candidates: edge, node pair
  uint32_t cab[kPer], root[2 * kPer], mine[2 * kPer], prev[2 * kPer];
#pragma unroll
  for (uint32_t k = 0; k < kPer; k++) {
    const uint32_t i = tid + k * bd;
    ce[k] = kNone;
    if (i < n) {
      const ulonglong2 h = __ldcg(&a.hlist[i]);
      ce[k] = h.x;
      root[2 * k] = (uint32_t)(h.y >> 32);
      root[2 * k + 1] = (uint32_t)h.y;
    }
  }
#pragma unroll
  for (uint32_t j = 0; j < 2 * kPer; j++)
    if (ce[j / 2] != kNone) mine[j] = atomicAdd(&s_nn, 1u);
#pragma unroll
  for (uint32_t j = 0; j < 2 * kPer; j++)
    if (ce[j / 2] != kNone) prev[j] = atomicCAS(&a.pcount[root[j]], 0u, mine[j] + 1);
#pragma unroll
  for (uint32_t k = 0; k < kPer; k++) {
    cab[k] = kNoneU32;
    if (ce[k] == kNone) continue;
    uint32_t node[2];
#pragma unroll
    for (uint32_t q = 0; q < 2; q++) {
      const uint32_t j = 2 * k + q;
      if (prev[j] == 0) s_lab[mine[j]] = root[j];
      node[q] = prev[j] == 0 ? mine[j] : prev[j] - 1;
    }
    cab[k] = node[0] | (node[1] << 16);
  }
  __syncthreads();
  const uint32_t nn = s_nn;
  for (uint32_t x = tid; x < nn; x += bd) {
    s_par[x] = x;
    s_best[x] = kNone;
  }
  __syncthreads();
  for (uint32_t iter = 0; iter < 64; iter++) {
    int any = 0;
#pragma unroll
    for (uint32_t k = 0; k < kPer; k++) {
      if (cab[k] == kNoneU32) continue;
      const uint32_t ra = s_find(s_par, cab[k] & 0xFFFFu), rb = s_find(s_par, cab[k] >> 16);
      if (ra != rb) {  // read first: most proposals to a big tree's root lose
        const uint64_t ka = ce[k] << kNodeBits | rb, kb = ce[k] << kNodeBits | ra;
        if (ka < s_best[ra]) atomicMin((unsigned long long*)&s_best[ra], (unsigned long long)ka);
        if (kb < s_best[rb]) atomicMin((unsigned long long*)&s_best[rb], (unsigned long long)kb);
        any = 1;
      } else {
        cab[k] = kNoneU32;  // both ends in one tree: never crosses again
      }
    }
    if (!__syncthreads_or(any)) break;
    for (uint32_t x = tid; x < nn; x += bd) {
      const uint64_t key = s_best[x];
      if (key == kNone) continue;
      const uint64_t e = key >> kNodeBits;
      const uint32_t o = (uint32_t)key & ((1u << kNodeBits) - 1);
      if ((s_best[o] >> kNodeBits) != e || x > o) {
        s_par[x] = o;
        a.forest[s_f0 + atomicAdd(&s_nf, 1u)] = e;
      }
    }
    __syncthreads();
    // flatten by pointer jumping, so that the next finds take one hop (the
    // hooks just made can form long chains); every value read is an ancestor
    for (uint32_t x = tid; x < nn; x += bd) s_best[x] = kNone;
    for (uint32_t pass = 0; pass < 16; pass++) {  // depth < 2^11 needs at most 11 passes
      int moved = 0;
      for (uint32_t x = tid; x < nn; x += bd) {
        const uint32_t p = s_par[x], pp = s_par[p];
        if (p != pp) {
          s_par[x] = pp;
          moved = 1;
        }
      }
      if (!__syncthreads_or(moved)) break;
    }
  }
  for (uint32_t x = tid; x < nn; x += bd) {
    const uint32_t lab = s_lab[x];
    if (lab == kNoneU32) continue;  // an id whose claim lost
    const uint32_t rt = s_find(s_par, x);
    if (rt != x) {
      a.parent[lab] = s_lab[rt];
      a.final_[s_lab[rt]] = 0;  // it absorbed another component: live
    }
    a.pcount[lab] = 0;
  }
  if (tid == 0) a.gc[GC_NFOREST] = s_f0 + s_nf;
}

// Add a warp's part of component K's sum (buckets base + lane + 32q) to
// acc[K]; the last of the component's `nparts` parts gets the whole sum in
// `acc` (true) and leaves acc[K] and the part count zero.
__device__ __forceinline__ bool join_parts(const RecArgs& a, ulonglong2 (&acc)[2], uint32_t K, uint32_t base,
                                           uint32_t W, uint32_t nparts) {
  const uint32_t lane = threadIdx.x & 31;
  ulonglong2* dst = a.acc + (size_t)K * W;
#pragma unroll
  for (uint32_t q = 0; q < 2; q++) {
    const uint32_t b = base + lane + 32 * q;
    if (b < W && (acc[q].x | acc[q].y)) {
      atomicXor(&dst[b].x, acc[q].x);
      atomicXor(&dst[b].y, acc[q].y);
    }
  }
  __syncwarp();
  uint32_t prev = 0;
  if (lane == 0) prev = atom_add_acq_rel(&a.pcount[K], 1u);
  __syncwarp();
  if (__shfl_sync(0xffffffffu, prev, 0) + 1 != nparts) return false;
#pragma unroll
  for (uint32_t q = 0; q < 2; q++) {
    const uint32_t b = base + lane + 32 * q;
    acc[q] = make_ulonglong2(0, 0);
    if (b < W) {
      acc[q] = __ldcg(dst + b);
      dst[b] = make_ulonglong2(0, 0);
    }
  }
  if (lane == 0) a.pcount[K] = 0;
  return true;
}

// Buckets base + lane + 32q of the four members that lanes m0 .. m0+3 hold in
// mw (kNoneU32: none), all in flight at once.
__device__ __forceinline__ void load_rows(ulonglong2 (&x)[4][2], const ulonglong2* __restrict__ layer, uint32_t mw,
                                          uint32_t m0, uint32_t base, uint32_t W) {
#pragma unroll
  for (uint32_t k = 0; k < 4; k++) {
    const uint32_t w = __shfl_sync(0xffffffffu, mw, m0 + k);
#pragma unroll
    for (uint32_t q = 0; q < 2; q++) {
      const uint32_t b = base + (threadIdx.x & 31) + 32 * q;
      x[k][q] = w != kNoneU32 && b < W ? __ldg(layer + (size_t)w * W + b) : make_ulonglong2(0, 0);
    }
  }
}

// The first good one of buckets [base, base + kPrefix) of the sum of the
// members perm[s0..s1), by one warp: its edge id, or kNone. Seldom called, so
// not inlined: its registers would add to the caller's.
static __device__ __noinline__ uint64_t read_on(const ulonglong2* __restrict__ layer, const uint32_t* perm, uint32_t s0,
                                                uint32_t s1, uint32_t base, uint32_t W, IdSplit ids, uint64_t kchk) {
  const uint32_t lane = threadIdx.x & 31;
  ulonglong2 sum[2] = {make_ulonglong2(0, 0), make_ulonglong2(0, 0)};
  for (uint32_t t0 = s0; t0 < s1; t0 += 32) {
    const uint32_t mw = t0 + lane < s1 ? ld_cg(&perm[t0 + lane]) : kNoneU32;
    for (uint32_t m0 = 0; m0 < min(32u, s1 - t0); m0 += 4) {
      ulonglong2 x[4][2];
      load_rows(x, layer, mw, m0, base, W);
#pragma unroll
      for (uint32_t k = 0; k < 4; k++)
#pragma unroll
        for (uint32_t q = 0; q < 2; q++) {
          sum[q].x ^= x[k][q].x;
          sum[q].y ^= x[k][q].y;
        }
    }
  }
  uint64_t e = 0;
  return warp_find(sum, base, W, ids, kchk, e) ? e : kNone;
}

// The recovery; false if there was nothing to do (no barrier was met).
__device__ __forceinline__ bool recover_body(const RecArgs& a) {
  __shared__ int s_ok;
  extern __shared__ __align__(16) unsigned char s_dyn[];  // small_hook; a reduce's partial sums
  constexpr uint32_t kSlots = 2 * (kRecThreads / 32);  // a warp's first and last component
  __shared__ uint32_t s_pk[kSlots];
  static_assert(kSmallHook % kRecThreads == 0, "small_hook: whole candidates per thread");
  static_assert(kSlots == 32 && kSlots * kPrefix * sizeof(ulonglong2) <= kHookBytes, "partial sums: one per lane id");
  ulonglong2* s_part = reinterpret_cast<ulonglong2*>(s_dyn);  // [kSlots][kPrefix]
  const uint32_t V = a.V, W = a.W, nb = gridDim.x, tid = threadIdx.x, lane = tid & 31;
  const uint32_t gtid = blockIdx.x * blockDim.x + tid, gstride = gridDim.x * blockDim.x;
  const uint32_t wpb = blockDim.x >> 5, gwarp = blockIdx.x * wpb + (tid >> 5), nwarps = gridDim.x * wpb;
  uint32_t* gc = a.gc;
  uint32_t epoch = 0;
#define CUPC_GRID_SYNC() \
  if (!grid_barrier(gc, nb, epoch, &s_ok)) return true

  // incremental mode: the updates since the last recovery kept the labels
  // exact (see k_incr), so there is nothing to recover; or they deleted
  // forest edges (of the recovered forest, or added by merges since): then
  // the components are unions of the fragments of the remaining forest, and
  // Boruvka starts from those (warm start) instead of from single vertices
  const bool valid = ld_cg(&gc[GC_LABELS_VALID]) != 0, warm = !a.force && valid && ld_cg(&gc[GC_WARM]) != 0;
  if (!a.force && valid && !warm) return false;
  const uint32_t nsorted = warm ? min(ld_cg(&gc[GC_NSORTED]), V) : 0;
  const uint32_t nadd = warm ? min(ld_cg(&gc[GC_NFADD]), V) : 0;
  // after a recovery that gave up at a barrier, the reduce accumulators and
  // the last-arriver counters may hold partial sums: clear them first
  const bool dirty = ld_cg(&gc[GC_REC_DIRTY]) != 0;
  for (uint32_t w = gtid; w < V; w += gstride) {
    a.label[w] = w;
    a.final_[w] = 0;
    a.parent[w] = w;
    a.minv[w] = kNoneU32;
    a.merged[w] = 0;
    a.cand[w] = make_ulonglong2(kNone, 0);
    a.best0[w] = kNone;
    a.best1[w] = kNone;
    a.rcnt[w] = 0;
    a.ipar[w] = w;
    if (!warm) a.fdead[w] = 0;  // a warm start reads them first
    if (dirty) a.pcount[w] = 0;
  }
  if (dirty)
    for (size_t i = gtid; i < (size_t)V * W; i += gstride) a.acc[i] = make_ulonglong2(0, 0);
  if (a.inc)  // the merge-edge table starts empty (fadd itself is read by a warm start below)
    for (size_t i = gtid; i < ((size_t)1 << a.ftab_bits); i += gstride) a.ftab[i] = 0ull;
  if (gtid == 0) {
    gc[GC_NLIVE] = 0;
    gc[GC_NFOREST] = 0;
    gc[GC_NFAIL] = 0;
    gc[GC_NFP] = 0;
    gc[GC_LOGLEN] = 0;
    gc[GC_COMPLETE] = 0;
    gc[GC_ROUNDS] = 0;
    gc[GC_NZ] = 0;
    gc[GC_ACTIVE] = 0;
    gc[GC_ACTIVE_ODD] = 0;
    gc[GC_NMEMBERS] = 0;
    for (uint32_t p = 0; p < kRetries; p++) gc[GC_RETRY + p] = 0;
    gc[GC_RECOVERIES] += 1;
  }
  for (uint32_t r = gtid; r < a.L; r += gstride) {
    a.log_live[r] = 0;
    a.log_ncand[r] = 0;
  }
  CUPC_GRID_SYNC();
  if (gtid == 0) {  // every CTA has read them (the early return and warm above depend on them)
    if (dirty) gc[GC_REC_DIRTY] = 0;
    gc[GC_NFADD] = 0;
    gc[GC_LABELS_VALID] = 0;
    gc[GC_FOREST_SORTED] = 0;
    gc[GC_WARM] = 0;
  }
  if (warm) {
    // fragments: union the endpoints of the forest edges still present (the
    // larger root under the smaller): the recovered forest's, then those
    // merges added. An edge whose union joins two fragments starts the new
    // forest (all of them with a valid stream; at most V - 1 in any case).
    const uint32_t nall = nsorted + nadd;
    for (uint32_t base = gwarp * 32; base < nall; base += nwarps * 32) {
      const uint32_t i = base + lane;
      bool keep = false;
      uint64_t e = 0;
      if (i < nsorted) {
        keep = !a.fdead[i];
        e = a.forest_sorted[i];
      } else if (i < nall) {
        keep = !a.fadd_dead[i - nsorted];
        e = a.fadd[i - nsorted];
      }
      if (keep) {
        uint32_t x = (uint32_t)(e / V), y = (uint32_t)(e % V);
        keep = false;
        for (uint32_t k = 0; k < V && x < V && y < V; k++) {  // bounded: each failed CAS is another thread's progress
          x = find_root(a.parent, x, V);
          y = find_root(a.parent, y, V);
          if (x == y) break;
          if (x > y) {
            const uint32_t t = x;
            x = y;
            y = t;
          }
          if (atomicCAS(&a.parent[y], y, x) == y) {
            keep = true;
            break;
          }
        }
      }
      const uint32_t m = __ballot_sync(0xffffffffu, keep);
      uint32_t at = 0;
      if (lane == 0 && m) at = atomicAdd(&gc[GC_NFOREST], (uint32_t)__popc(m));
      at = __shfl_sync(0xffffffffu, at, 0);
      if (keep) a.forest[at + __popc(m & ((1u << lane) - 1))] = e;
    }
    CUPC_GRID_SYNC();
    for (uint32_t w = gtid; w < V; w += gstride) a.label[w] = find_root(a.parent, w, V);  // the minimum id
    CUPC_GRID_SYNC();
    // A fragment that holds no endpoint of a deleted forest edge is a whole
    // component of the last complete recovery, joined with others only by
    // recorded merges: its cut is empty, so it starts final (its sample
    // would be ZERO). Only the split components are sampled again.
    for (uint32_t w = gtid; w < V; w += gstride)
      if (ld_cg(&a.label[w]) == w) a.final_[w] = 1;
    CUPC_GRID_SYNC();
    for (uint32_t i = gtid; i < nall; i += gstride) {
      const bool dead = i < nsorted ? a.fdead[i] != 0 : a.fadd_dead[i - nsorted] != 0;
      if (!dead) continue;
      const uint64_t e = i < nsorted ? a.forest_sorted[i] : a.fadd[i - nsorted];
      const uint32_t x = (uint32_t)(e / V), y = (uint32_t)(e % V);
      if (x < V && y < V) {
        a.final_[ld_cg(&a.label[x])] = 0;
        a.final_[ld_cg(&a.label[y])] = 0;
      }
    }
    CUPC_GRID_SYNC();
    // the split fragments are the live components of the first round: count members
    for (uint32_t base = gwarp * 32; base < V; base += nwarps * 32) {
      const uint32_t w = base + lane;
      uint32_t lab = 0;
      bool live = false;
      if (w < V) {
        lab = ld_cg(&a.label[w]);
        live = !ld_cg(&a.final_[lab]);
        a.parent[w] = w;
        a.fdead[w] = 0;
      }
      const uint32_t m_first = __ballot_sync(0xffffffffu, warp_grab(a.rcnt, lab, live) == 0 && live);
      if (lane == 0 && m_first) atomicAdd(&gc[GC_NLIVE], (uint32_t)__popc(m_first));
    }
    CUPC_GRID_SYNC();
  }

  for (uint32_t r = 0; r < a.L; r++) {
    const uint64_t kchk = a.keys[r * (a.C + 1) + a.C];
    const bool multi = r > 0 || warm;  // components may have several members
    // One live component left: every other component is final, and a final
    // component's merged sketch is zero (its cut is empty); the XOR of all
    // vertex sketches of a layer is zero (each edge enters both endpoints),
    // so the live one's merged sketch is zero too and it samples ZERO. Log
    // the round as sampled (one live component, no candidate) and stop.
    // Imported words need not come from a stream: then the round is run.
    if (multi && a.sum_zero && ld_cg(&gc[GC_NLIVE]) == 1) {
      if (gtid == 0) {
        a.log_live[r] = 1;
        gc[GC_ROUNDS] = r + 1;
        gc[GC_COMPLETE] = 1;
      }
      break;
    }
    // ---- group the live vertices of round r by component: the relabel of
    // round r-1 counted them; give each component a segment (warp-aggregated
    // atomics), then scatter
    uint32_t nmem = V;
    if (multi) {
      for (uint32_t base = blockIdx.x * blockDim.x; base < V; base += gstride) {
        const uint32_t K = base + tid;
        const uint32_t c = K < V ? ld_cg(&a.rcnt[K]) : 0;
        uint32_t inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= (uint32_t)o) inc += y;
        }
        uint32_t at = 0;
        if (lane == 31 && inc) at = atomicAdd(&gc[GC_NMEMBERS], inc);
        at = __shfl_sync(0xffffffffu, at, 31) + inc - c;
        if (c) {
          a.roff[K] = at;
          a.rcnt[K] = at;  // scatter cursor, then the segment end
        }
        if (K < V) {
          a.parent[K] = K;
        }
      }
      CUPC_GRID_SYNC();
      for (uint32_t base = gwarp * 32; base < V; base += nwarps * 32) {
        const uint32_t w = base + lane;
        const uint32_t K = w < V ? ld_cg(&a.label[w]) : 0;
        const bool live = w < V && !ld_cg(&a.final_[K]);
        const uint32_t pos = warp_grab(a.rcnt, K, live);
        if (live) a.perm[pos] = w;
      }
      CUPC_GRID_SYNC();
      nmem = ld_cg(&gc[GC_NMEMBERS]);
    }

    // ---- reduce + sample. The sample is the first good bucket in index
    // order, so the first kPrefix buckets of a sum nearly always decide it
    // (they hold the deterministic bucket and 1.8 columns or more, each of
    // which has a good bucket with probability 0.8): only they are read,
    // XORed and tested, and the next kPrefix ones only for the components
    // that need them. At V = 2^17 that is 64 of 239 buckets.
    //
    // Round 0: a warp per vertex. Later rounds: every warp takes an equal run
    // of the member list; a component inside one run is sampled by its warp,
    // the parts of one over several runs are summed by the CTA, and one over
    // several CTAs is XORed into acc[K] and sampled by the last CTA to finish
    // (XORs of every warp of the device into one giant component's acc[K]
    // would queue: 42 us against 8 at V = 2^14).
    uint32_t st_k = kNoneU32, st_res = 0, nst = 0;  // this lane's stashed sample
    uint64_t st_e = 0;
    auto book_stash = [&]() {  // up to 32 samples at once, one per lane
      if (nst) book_samples(a, r, multi, st_k, st_res, st_e);
      st_k = kNoneU32;
      nst = 0;
    };
    auto stash = [&](uint32_t K, uint32_t res, uint64_t e) {
      if (lane == nst) {
        st_k = K;
        st_res = res;
        st_e = e;
      }
      if (++nst == 32) book_stash();
    };
    const ulonglong2* layer = a.sketch + (size_t)r * V * W;
    const uint32_t run = (nmem + nwarps - 1) / nwarps, p0 = gwarp * run, p1 = min(nmem, p0 + run);
    // The sum of component K over [s0, s1) of the list, or this CTA's part of
    // it (nparts > 1), is complete: sample it.
    auto complete = [&](uint32_t base, uint32_t K, ulonglong2(&acc)[2], uint32_t s0, uint32_t s1, uint32_t nparts,
                        bool here) {
      if (nparts > 1 && !join_parts(a, acc, K, base, W, nparts)) return;
      uint64_t e = 0;
      uint32_t res = 2;
      if (base == 0)
        res = warp_sample_prefix(acc, W, a.ids, kchk, e);
      else if (warp_find(acc, base, W, a.ids, kchk, e))
        res = 1;
      // this warp's own, or a short one: reads on at once
      here = here || s1 - s0 <= kRecSpan;
      for (uint32_t b = base + kPrefix; here && res == 2 && b < W; b += kPrefix) {
        const uint64_t more = read_on(layer, a.perm, s0, s1, b, W, a.ids, kchk);
        if (more != kNone) {
          e = more;
          res = 1;
        }
      }
      const bool again = !here && res == 2 && base + kPrefix < W;
      if (lane == 0 && (again || base)) a.merged[K] = again ? 1 : 0;
      if (!again)
        stash(K, res, e);
      else if (lane == 0)
        atomicAdd(&gc[GC_RETRY + base / kPrefix], 1u);
    };
    auto reduce_run = [&](uint32_t base) {
      const uint32_t wid = tid >> 5;
      if (lane < 2) s_pk[2 * wid + lane] = kNoneU32;
      __syncwarp();
      ulonglong2 acc[2] = {make_ulonglong2(0, 0), make_ulonglong2(0, 0)};
      uint32_t K = kNoneU32;  // the component being summed
      auto finish = [&]() {
        if (K == kNoneU32 || (base && !ld_cg(&a.merged[K]))) return;
        const uint32_t s0 = ld_cg(&a.roff[K]), s1 = ld_cg(&a.rcnt[K]);
        if (s0 >= p0 && s1 <= p1) {
          complete(base, K, acc, s0, s1, 1, true);
        } else {  // it goes on in a neighbouring run
          const uint32_t slot = 2 * wid + (s0 < p0 ? 0 : 1);
          if (lane == 0) s_pk[slot] = K;
#pragma unroll
          for (uint32_t q = 0; q < 2; q++) s_part[slot * kPrefix + lane + 32 * q] = acc[q];
        }
      };
      for (uint32_t t0 = p0; t0 < p1; t0 += 32) {
        const uint32_t cnt = min(32u, p1 - t0);
        uint32_t mw = kNoneU32, mk = kNoneU32;
        if (lane < cnt) {
          mw = ld_cg(&a.perm[t0 + lane]);
          mk = ld_cg(&a.label[mw]);
          if (base && !ld_cg(&a.merged[mk])) mw = kNoneU32;  // not read again
        }
        uint32_t before = __shfl_up_sync(0xffffffffu, mk, 1);
        if (lane == 0) before = K;
        const uint32_t heads = __ballot_sync(0xffffffffu, lane < cnt && mk != before);
        if (mw != kNoneU32) {  // the members' rows head for L2
#pragma unroll
          for (uint32_t b = 0; b < kPrefix; b += 8)
            if (base + b < W) asm volatile("prefetch.global.L2 [%0];" ::"l"(layer + (size_t)mw * W + base + b));
        }
        for (uint32_t m0 = 0; m0 < cnt; m0 += 4) {
          ulonglong2 x[4][2];
          load_rows(x, layer, mw, m0, base, W);
          const uint32_t h = heads >> m0 & 0xFu;
          for (uint32_t m = 0; m < 4;) {  // the parts of components among the four
            if (h >> m & 1) {
              finish();
              K = __shfl_sync(0xffffffffu, mk, m0 + m);
              acc[0] = acc[1] = make_ulonglong2(0, 0);
            }
            const uint32_t more = h & (~1u << m), end = more ? (uint32_t)__ffs((int)more) - 1 : 4u;
#pragma unroll
            for (uint32_t k = 0; k < 4; k++)
              if (k >= m && k < end) {
#pragma unroll
                for (uint32_t q = 0; q < 2; q++) {
                  acc[q].x ^= x[k][q].x;
                  acc[q].y ^= x[k][q].y;
                }
              }
            m = end;
          }
        }
      }
      finish();
      __syncthreads();
      // the CTA's parts of one component, together
      const uint32_t pk = s_pk[lane], crun = run * wpb;
      for (uint32_t slot = wid; slot < kSlots; slot += wpb) {
        const uint32_t C = __shfl_sync(0xffffffffu, pk, slot);
        uint32_t parts = __ballot_sync(0xffffffffu, pk == C);
        if (C == kNoneU32 || (uint32_t)__ffs((int)parts) - 1 != slot) continue;
        ulonglong2 sum[2] = {make_ulonglong2(0, 0), make_ulonglong2(0, 0)};
        for (; parts; parts &= parts - 1) {
          const ulonglong2* v = s_part + (__ffs((int)parts) - 1) * kPrefix + lane;
#pragma unroll
          for (uint32_t q = 0; q < 2; q++) {
            sum[q].x ^= v[32 * q].x;
            sum[q].y ^= v[32 * q].y;
          }
        }
        const uint32_t s0 = ld_cg(&a.roff[C]), s1 = ld_cg(&a.rcnt[C]);
        complete(base, C, sum, s0, s1, (s1 - 1) / crun - s0 / crun + 1, false);
      }
      __syncthreads();
    };
    if (!multi) {
      // four vertices' rows in flight; the next four's head for L2
      constexpr uint32_t kAtOnce = 4;
      const uint32_t step = kAtOnce * nwarps;
      for (uint32_t w0 = kAtOnce * gwarp; w0 < V; w0 += step) {
        const uint32_t ahead = w0 + step + lane / 8;  // lane: 128 bytes of a row
        if (ahead < V && lane % 8 * 8 < W)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(layer + (size_t)ahead * W + lane % 8 * 8));
        ulonglong2 acc[kAtOnce][2];
#pragma unroll
        for (uint32_t k = 0; k < kAtOnce; k++)
#pragma unroll
          for (uint32_t q = 0; q < 2; q++) {
            const uint32_t b = lane + 32 * q;
            acc[k][q] = w0 + k < V && b < W ? __ldg(layer + (size_t)(w0 + k) * W + b) : make_ulonglong2(0, 0);
          }
        // the first 32 buckets of the four tested side by side; they decide
        // most samples
        uint32_t zero[kAtOnce], first[kAtOnce];
#pragma unroll
        for (uint32_t k = 0; k < kAtOnce; k++) {
          zero[k] = __ballot_sync(0xffffffffu, (acc[k][0].x | acc[k][0].y) == 0) & 1;
          first[k] = __ballot_sync(0xffffffffu, good_bucket(acc[k][0], lane, W, a.ids, kchk));
        }
#pragma unroll
        for (uint32_t k = 0; k < kAtOnce; k++) {
          if (w0 + k >= V) break;
          uint64_t e = 0;
          uint32_t res = 2;
          if (zero[k]) {
            res = 0;
          } else if (first[k]) {
            res = 1;
            e = __shfl_sync(0xffffffffu, acc[k][0].x, __ffs(first[k]) - 1);
          } else if (warp_find(acc[k], 0, W, a.ids, kchk, e)) {
            res = 1;
          }
          for (uint32_t base = kPrefix; res == 2 && base < W; base += kPrefix) {
            ulonglong2 more[2] = {make_ulonglong2(0, 0), make_ulonglong2(0, 0)};
            warp_xor_part(more, layer + (size_t)(w0 + k) * W, base, W, lane);
            if (warp_find(more, base, W, a.ids, kchk, e)) res = 1;
          }
          stash(w0 + k, res, e);
        }
      }
    } else {
      reduce_run(0);
    }
    book_stash();
    CUPC_GRID_SYNC();
    // Components of more than kRecSpan members that no warp holds alone and whose
    // buckets so far hold no good one are marked (merged[K], unused until the
    // relabel): another pass over the next kPrefix buckets.
    for (uint32_t base = kPrefix; multi && base < W && ld_cg(&gc[GC_RETRY + base / kPrefix - 1]); base += kPrefix) {
      reduce_run(base);
      book_stash();
      CUPC_GRID_SYNC();
    }
    if (gtid == 0) {
      gc[GC_ROUNDS] = r + 1;
      gc[GC_NLIVE] = 0;  // every CTA has read it
    }
    if (ld_cg(&gc[GC_NZ]) == 0) {
      if (gtid == 0) gc[GC_COMPLETE] = 1;
      break;
    }

    // ---- hook: minimum spanning forest of the candidates by Boruvka. A
    // root's key is edge << vbits | (root on the other side), so the min key names
    // the min-id crossing edge and where it leads; two roots that chose the
    // same edge hook once (the larger id under the smaller). A round with
    // few candidates hooks in one CTA (small_hook) behind a single barrier.
    const uint32_t vbits = 32 - __clz(V - 1);  // bits of a vertex id (V <= 2^21: keys fit 64 bits)
    const uint64_t vmask = (1ull << vbits) - 1;
    for (uint32_t iter = 0; iter < 64; iter++) {
      uint64_t* bc = (iter & 1) ? a.best1 : a.best0;
      uint64_t* bn = (iter & 1) ? a.best0 : a.best1;
      // candidates still crossing two trees: count them, list the first kSmallHook
      const uint32_t act = (iter & 1) ? GC_ACTIVE_ODD : GC_ACTIVE, act_next = (iter & 1) ? GC_ACTIVE : GC_ACTIVE_ODD;
      for (uint32_t base = gwarp * 32; base < V; base += nwarps * 32) {
        const uint32_t K = base + lane;
        bool cross = false;
        uint32_t ra = 0, rb = 0;
        ulonglong2 c = make_ulonglong2(kNone, 0);
        if (K < V) {
          if (iter == 0) a.rcnt[K] = 0;  // the relabel counts again
          c = __ldcg(&a.cand[K]);
          if (c.x != kNone) {
            ra = (uint32_t)(c.y >> 32);
            rb = (uint32_t)c.y;
            const bool left = ra == K;
            walk_roots(a.parent, ra, rb, V);
            // nobody else writes K's word now: the next walks are short
            const uint32_t root = left ? ra : rb;
            if (iter && root != K) a.parent[K] = root;
          }
        }
        // lanes leave the walk at different steps: together again before the
        // next loads
        __syncwarp();
        const uint64_t e = c.x;
        if (ra != rb) {  // read first: most proposals to a big tree's root lose
          const uint64_t ka = e << vbits | rb, kb = e << vbits | ra;
          const uint64_t ba = ld_cg(&bc[ra]), bb = ld_cg(&bc[rb]);
          if (ka < ba) atomicMin((unsigned long long*)&bc[ra], (unsigned long long)ka);
          if (kb < bb) atomicMin((unsigned long long*)&bc[rb], (unsigned long long)kb);
          cross = true;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, cross);
        if (m) {
          uint32_t at = 0;
          if (lane == 0) at = atomicAdd(&gc[act], (uint32_t)__popc(m));
          at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1));
          if (cross && at < kSmallHook) a.hlist[at] = make_ulonglong2(e, (uint64_t)ra << 32 | rb);
        }
      }
      CUPC_GRID_SYNC();
      const uint32_t nact = ld_cg(&gc[act]);
      if (nact == 0) break;
      if (nact <= kSmallHook) {  // finish in one CTA behind a single barrier
        if (blockIdx.x == 0) small_hook(a, nact, s_dyn);
        CUPC_GRID_SYNC();
        break;
      }
      for (uint32_t base = gwarp * 32; base < V; base += nwarps * 32) {
        const uint32_t x = base + lane;
        bool hook = false;
        uint64_t e = 0;
        uint32_t o = 0;
        if (x < V) {
          bn[x] = kNone;
          const uint64_t key = ld_cg(&bc[x]);
          if (key != kNone) {
            e = key >> vbits;
            o = (uint32_t)(key & vmask);
            const bool mutual = (ld_cg(&bc[o]) >> vbits) == e;
            hook = !mutual || x > o;
          }
        }
        const uint32_t m = __ballot_sync(0xffffffffu, hook);
        if (m) {
          uint32_t at = 0;
          if (lane == 0) at = atomicAdd(&gc[GC_NFOREST], (uint32_t)__popc(m));
          at = __shfl_sync(0xffffffffu, at, 0);
          if (hook) {
            a.parent[x] = o;
            a.final_[o] = 0;  // it absorbs another component: live
            a.forest[at + __popc(m & ((1u << lane) - 1))] = e;
          }
        }
      }
      if (gtid == 0) gc[act_next] = 0;
      CUPC_GRID_SYNC();
    }

    // ---- relabel to the root of each component; the members of next round's
    // live components are counted here; clear the round's scratch
    if (gtid == 0) {
      gc[GC_NZ] = 0;
      gc[GC_NMEMBERS] = 0;
      gc[GC_ACTIVE] = 0;
      gc[GC_ACTIVE_ODD] = 0;
      for (uint32_t p = 0; p < kRetries; p++) gc[GC_RETRY + p] = 0;
    }
    for (uint32_t base = gwarp * 32; base < V; base += nwarps * 32) {
      const uint32_t w = base + lane;
      uint32_t nl = 0;
      bool live = false;
      if (w < V) {
        a.cand[w] = make_ulonglong2(kNone, 0);
        a.best0[w] = kNone;
        a.best1[w] = kNone;
        nl = ld_cg(&a.label[w]);
        uint32_t same = nl;
        walk_roots(a.parent, nl, same, V);
      }
      __syncwarp();  // as above
      if (w < V) {
        a.label[w] = nl;
        live = !ld_cg(&a.final_[nl]);
      }
      __syncwarp();
      // the member that took position 0 of its component counts the component
      const uint32_t m_first = __ballot_sync(0xffffffffu, warp_grab(a.rcnt, nl, live) == 0 && live);
      if (lane == 0 && m_first) atomicAdd(&gc[GC_NLIVE], (uint32_t)__popc(m_first));
    }
    CUPC_GRID_SYNC();
  }
  // ---- labels: the rounds need one id per component (its root), the result
  // is the minimum vertex id
  for (uint32_t base = gwarp * 32; base < V; base += nwarps * 32) {
    const uint32_t w = base + lane;
    const uint32_t act = __ballot_sync(0xffffffffu, w < V);
    if (w < V) {  // the first of the lanes of one component has their minimum
      const uint32_t K = ld_cg(&a.label[w]), peers = __match_any_sync(act, K);
      if (lane == (uint32_t)__ffs(peers) - 1 && w < ld_cg(&a.minv[K])) atomicMin(&a.minv[K], w);
    }
  }
  CUPC_GRID_SYNC();
  for (uint32_t w = gtid; w < V; w += gstride) a.label[w] = ld_cg(&a.minv[ld_cg(&a.label[w])]);
  // a complete recovery starts an incremental epoch
  if (a.inc && gtid == 0) gc[GC_LABELS_VALID] = ld_cg(&gc[GC_COMPLETE]);
#undef CUPC_GRID_SYNC
  return true;
}

// The last CTA to leave zeroes the barrier's counters for the next launch,
// also when the CTAs gave up at a barrier.
__global__ void __launch_bounds__(kRecThreads, 1) k_recover(RecArgs a) {
  if (!recover_body(a)) return;
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(&a.gc[GC_BAR_DONE], 1u) == gridDim.x - 1) {
    a.gc[GC_BAR_COUNT] = 0;
    a.gc[GC_BAR_DONE] = 0;
  }
}

// Self-test of the bounded waits: every CTA but `absent` meets at two grid
// barriers; `absent` returns at once, so the others give up after limit_ns
// and record kErrTimeout.
__global__ void k_wait_selftest(uint32_t* gc, uint32_t absent, uint64_t limit_ns) {
  __shared__ int s_ok;
  uint32_t epoch = 0;
  if (blockIdx.x == absent) return;
  if (!grid_barrier(gc, gridDim.x, epoch, &s_ok, limit_ns)) return;
  grid_barrier(gc, gridDim.x, epoch, &s_ok, limit_ns);
}

cudaError_t setup_recover(cupc_graph* g) {
  int per_sm = 0;
  cudaError_t e = setup_recover_cluster(g);
  if (e != cudaSuccess || g->rec_cluster) return e;  // the grid-wide kernel is not used
  e = cudaFuncSetAttribute(k_recover, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHookBytes);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_recover, kRecThreads, kHookBytes);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // 128 vertices a CTA: few CTAs keep the grid barriers cheap and leave room
  // for other graphs' recoveries (a CTA fills an SM, and a cooperative launch
  // waits until all of its CTAs fit). GB300, us for one query with 64, 128,
  // 256 vertices a CTA: V = 8000 165, 163, 172; V = 16384 208, 207, 223; V =
  // 24000 228, 228, 235; 16 served graphs of 1024..32768 vertices: 2916, 2608,
  // 2243 (the server limits the grids further while several queries wait).
  const uint32_t want = std::max(16u, (g->V + 127) / 128);
  const uint32_t cap = (uint32_t)(per_sm * g->sms);
  g->rec_grid = (int)(want < cap ? want : cap);
  return cudaSuccess;
}

cudaError_t launch_recover(cupc_graph* g, cudaStream_t s, bool force) {
  RecArgs a;
  a.sketch = g->sketch;
  a.keys = g->keys;
  a.V = g->V;
  a.ids = IdSplit(g->V);
  a.L = g->L;
  a.C = g->C;
  a.D = g->D;
  a.W = g->W;
  a.label = g->label;
  a.parent = g->parent;
  a.minv = g->minv;
  a.rcnt = g->rcnt;
  a.roff = g->roff;
  a.perm = g->perm;
  a.pcount = g->pcount;
  a.final_ = g->final_;
  a.merged = g->merged;
  a.best0 = g->best;
  a.best1 = g->best2;
  a.cand = g->cand;
  a.forest = g->forest;
  a.log_ids = g->log_ids;
  a.acc = g->acc;
  a.log_live = g->log_live;
  a.log_ncand = g->log_ncand;
  a.hlist = g->hlist;
  a.ipar = g->ipar;
  a.forest_sorted = g->forest_sorted;
  a.fdead = g->fdead;
  a.fadd = g->fadd;
  a.fadd_dead = g->fadd_dead;
  a.ftab = (unsigned long long*)g->ftab;
  a.ftab_bits = g->ftab_bits;
  a.inc = g->inc ? 1u : 0u;
  a.force = force ? 1u : 0u;
  a.sum_zero = g->imported ? 0u : 1u;
  a.gc = g->gc;
  if (g->rec_cluster) {
    ProfScope ps(g, s, PC_RECOVER, 1);
    return launch_recover_cluster(g, a, s);
  }
  ProfScope ps(g, s, PC_RECOVER, 1);
  void* args[] = {&a};
  const int grid = g->rec_share ? std::min(g->rec_grid, g->rec_share) : g->rec_grid;
  return cudaLaunchCooperativeKernel((const void*)k_recover, dim3(grid), dim3(kRecThreads), args, kHookBytes,
                                     s);
}

}  // namespace cupc

extern "C" cupc_status cupc_selftest_wait_timeout(uint32_t ctas, uint32_t limit_us, int absent_cta,
                                                  cupc_stream stream) {
  using namespace cupc;
  if (ctas < 2 || ctas > 64 || limit_us == 0 || limit_us > 1000000) return CUPC_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  uint32_t* gc = nullptr;
  if (cudaMalloc((void**)&gc, GC_SLOTS * sizeof(uint32_t)) != cudaSuccess) return CUPC_ENOMEM;
  cupc_status st = CUPC_OK;
  uint32_t h[GC_SLOTS];
  uint32_t absent = absent_cta < 0 ? 0xFFFFFFFFu : (uint32_t)absent_cta;
  uint64_t limit = (uint64_t)limit_us * 1000;
  void* args[] = {&gc, &absent, &limit};
  if (cudaMemsetAsync(gc, 0, GC_SLOTS * sizeof(uint32_t), s) != cudaSuccess ||
      cudaLaunchCooperativeKernel((const void*)k_wait_selftest, dim3(ctas), dim3(32), args, 0, s) != cudaSuccess ||
      cudaMemcpyAsync(h, gc, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    st = CUPC_ECUDA;
  } else if (h[GC_ERR] & kErrTimeout) {
    st = CUPC_ETIMEOUT;
  }
  cudaFree(gc);
  return st;
}

namespace cupc {

// ---- Connected(u,v) from the recovered labels (Problem 2)
__global__ void k_query(const uint32_t* __restrict__ pairs, size_t m, uint8_t* __restrict__ out,
                        const uint32_t* __restrict__ label, uint32_t V, uint32_t* gc) {
  bool bad = false;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (size_t)gridDim.x * blockDim.x) {
    uint32_t u = pairs[2 * i], v = pairs[2 * i + 1];
    if (u >= V || v >= V) {
      bad = true;
      out[i] = 0;
    } else {
      out[i] = __ldcg(&label[u]) == __ldcg(&label[v]);
    }
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&gc[GC_ERR], kErrQuery);
}

cudaError_t launch_query(cupc_graph* g, const uint32_t* pairs, size_t m, uint8_t* out, cudaStream_t s) {
  if (m == 0) return cudaSuccess;
  int grid = (int)std::min<size_t>((m + 255) / 256, (size_t)g->sms * 4);
  ProfScope ps(g, s, PC_QUERY, 1);
  k_query<<<grid, 256, 0, s>>>(pairs, m, out, g->label, g->V, g->gc);
  return cudaGetLastError();
}

// ---- forest ids in ascending order: bitonic sort of 1024-id chunks, one id
// a thread (partners within a warp exchange by shuffles, farther ones through
// shared memory), then each id's final rank = its rank in its chunk + its
// lower bound in every other chunk (ids are distinct), a CTA taking the other
// chunks through shared memory one after the other, the next one in flight.
// V = 2^14 on GB300: 6 + 9 us; 14 + 29 us with the exchanges all in shared
// memory and the searches in global memory.
constexpr uint32_t kSortChunk = 1024;

__device__ __forceinline__ void sort_chunk(uint64_t* ids, uint32_t n, uint64_t (&s)[2][kSortChunk]) {
  const uint32_t tid = threadIdx.x, at = blockIdx.x * kSortChunk + tid;
  if (blockIdx.x * kSortChunk >= n) return;
  uint64_t v = at < n ? ids[at] : kNone;
  uint32_t buf = 0;
#pragma unroll
  for (uint32_t k = 2; k <= kSortChunk; k <<= 1) {
#pragma unroll
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      uint64_t y;
      if (j >= 32) {
        s[buf][tid] = v;
        __syncthreads();
        y = s[buf][tid ^ j];
        buf ^= 1;  // the next exchange's writes do not meet this one's reads
      } else {
        y = __shfl_xor_sync(0xffffffffu, v, j);
      }
      v = ((tid & j) == 0) == ((tid & k) == 0) ? min(v, y) : max(v, y);
    }
  }
  if (at < n) ids[at] = v;
}

__device__ __forceinline__ void merge_rank(const uint64_t* ids, uint64_t* out, uint32_t n,
                                           uint64_t (&s)[2][kSortChunk], uint32_t* gc) {
  const uint32_t nch = (n + kSortChunk - 1) / kSortChunk, tid = threadIdx.x, at = blockIdx.x * kSortChunk + tid;
  if (blockIdx.x < nch) {
    const uint64_t x = at < n ? ld_cg(&ids[at]) : kNone;
    uint32_t rank = tid;
    auto load = [&](uint32_t k) {  // chunk blockIdx.x + k, cyclically
      const uint32_t c = blockIdx.x + k < nch ? blockIdx.x + k : blockIdx.x + k - nch;
      const uint32_t i = c * kSortChunk + tid;
      return k < nch && i < n ? ld_cg(&ids[i]) : kNone;
    };
    uint64_t next = load(1);
    for (uint32_t k = 1; k < nch; k++) {
      uint64_t* c = s[k & 1];
      c[tid] = next;
      next = load(k + 1);
      __syncthreads();
      uint32_t lo = 0;  // ids of the chunk below x; the ids past its end are kNone
#pragma unroll
      for (uint32_t step = kSortChunk / 2; step > 0; step >>= 1)
        if (c[lo + step - 1] < x) lo += step;
      if (c[lo] < x) lo++;
      rank += lo;
    }
    if (at < n) out[rank] = x;
  }
  __syncthreads();
  if (tid == 0 && atomicAdd(&gc[GC_SORT_DONE], 1u) == gridDim.x - 1) {  // every CTA has read the flag above
    gc[GC_SORT_DONE] = 0;
    gc[GC_NSORTED] = n;
    gc[GC_FOREST_SORTED] = 1;
  }
}

__global__ void __launch_bounds__(kSortChunk) k_sort_chunks(uint64_t* ids, const uint32_t* gc) {
  __shared__ uint64_t s[2][kSortChunk];
  if (ld_cg(&gc[GC_FOREST_SORTED])) return;  // done since the last recovery
  sort_chunk(ids, ld_cg(&gc[GC_NFOREST]), s);
}

__global__ void __launch_bounds__(kSortChunk) k_merge_rank(const uint64_t* ids, uint64_t* out, uint32_t* gc) {
  __shared__ uint64_t s[2][kSortChunk];
  if (ld_cg(&gc[GC_FOREST_SORTED])) return;
  merge_rank(ids, out, ld_cg(&gc[GC_NFOREST]), s, gc);
}

// Both steps in one launch, where the chunks are the CTAs of one cluster
// (whose barrier orders the chunks' stores before the other CTAs' loads): in
// incremental mode most launches find the forest sorted, and cost only that.
__global__ void __launch_bounds__(kSortChunk) k_sort_cluster(uint64_t* ids, uint64_t* out, uint32_t* gc) {
  __shared__ uint64_t s[2][kSortChunk];
  if (ld_cg(&gc[GC_FOREST_SORTED])) return;
  const uint32_t n = ld_cg(&gc[GC_NFOREST]);
  sort_chunk(ids, n, s);
  cluster_sync_all();
  merge_rank(ids, out, n, s, gc);
}

cudaError_t launch_forest_sort(cupc_graph* g, cudaStream_t s) {
  const uint32_t nch = (g->V + kSortChunk - 1) / kSortChunk;
  if (nch <= 8) {  // the largest portable cluster
    ProfScope ps(g, s, PC_SORT, 1);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = nch;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nch);
    cfg.blockDim = dim3(kSortChunk);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_sort_cluster, g->forest, g->forest_sorted, g->gc);
  }
  ProfScope ps(g, s, PC_SORT, 2);
  k_sort_chunks<<<nch, kSortChunk, 0, s>>>(g->forest, g->gc);
  k_merge_rank<<<nch, kSortChunk, 0, s>>>(g->forest, g->forest_sorted, g->gc);
  return cudaGetLastError();
}

// The sorted forest into the caller's device memory, unless it does not fit
// or an error is pending (the caller then reports that and copies nothing).
__global__ void k_copy_forest(const uint64_t* __restrict__ ids, uint64_t* __restrict__ out, size_t cap,
                              const uint32_t* gc) {
  const uint32_t n = ld_cg(&gc[GC_NFOREST]);
  if (n > cap || (ld_cg(&gc[GC_ERR]) & (kErrTimeout | kErrInval))) return;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = ids[i];
}

cudaError_t launch_copy_forest(cupc_graph* g, uint64_t* out, size_t cap, cudaStream_t s) {
  k_copy_forest<<<(int)std::min<size_t>((g->V + 255) / 256, (size_t)g->sms * 4), 256, 0, s>>>(g->forest_sorted, out, cap,
                                                                                               g->gc);
  return cudaGetLastError();
}

}  // namespace cupc

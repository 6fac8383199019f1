// Recovery state and warp helpers shared by the grid-wide recovery
// (recover.cu) and the one-cluster recovery of small graphs
// (recover_small.cu).
#pragma once

#include "common.cuh"

namespace cupc {

// The endpoints of an edge id x = u*V + v. Every sample tests its id's order,
// and a 64-bit division is a long chain (V > 2^16); with inv = floor((2^64 -
// 1) / V) the high half of x * inv is floor(x / V) or one less: x/V - x*inv/2^64
// = x/2^64 * (2^64/V - inv) < 1, as 2^64/V - inv <= 1.
struct IdSplit {
  uint64_t inv;
  uint32_t V;
  __host__ explicit IdSplit(uint32_t n) : inv(~0ull / n), V(n) {}
  IdSplit() = default;
  __device__ __forceinline__ void split(uint64_t x, uint64_t& u, uint64_t& v) const {
    u = __umul64hi(x, inv);
    v = x - u * V;
    if (v >= V) {
      u++;
      v -= V;
    }
  }
  __device__ __forceinline__ bool ordered(uint64_t x) const {
    uint64_t u, v;
    split(x, u, v);
    return u < v;
  }
};

struct RecArgs {
  const ulonglong2* sketch;
  const uint64_t* keys;
  uint32_t V, L, C, D, W;
  IdSplit ids;
  uint32_t *label, *parent, *minv, *rcnt, *roff, *perm, *pcount;
  uint8_t *final_, *merged;
  uint64_t *best0, *best1, *forest, *log_ids;
  ulonglong2* cand;  // {edge, label[u] << 32 | label[v]} of a component's candidate
  ulonglong2* acc;
  uint32_t *log_live, *log_ncand;
  ulonglong2* hlist;  // kSmallHook: crossing candidates {edge, root_a << 32 | root_b} of a hook step
  uint32_t* ipar;     // V: union-find of incremental inserts, identity after a recovery
  const uint64_t* forest_sorted;
  uint8_t* fdead;     // V: forest_sorted[i] deleted since the last recovery
  const uint64_t* fadd;      // V: forest edges added by incremental merges since
  const uint8_t* fadd_dead;  // V: fadd[j] deleted since
  unsigned long long* ftab;  // 2^ftab_bits: the ids of fadd (cleared here)
  uint32_t ftab_bits;
  uint32_t inc, force;  // incremental mode; run even if the labels are valid
  uint32_t sum_zero;    // the XOR of all vertex sketches of a layer is zero (no import since reset)
  uint32_t* gc;
};

// Barrier of a thread-block cluster; arrive has release and wait acquire
// semantics at cluster scope.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// A bucket is good when its alpha is non-zero, its checksum holds and alpha is
// an edge id u*V+v with u < v. A sum's sample is ZERO if the deterministic
// bucket is zero, else the first good bucket in index order (deterministic
// bucket, then column-major), else FAIL.
__device__ __forceinline__ bool good_bucket(const ulonglong2& x, uint32_t j, uint32_t W, const IdSplit& ids,
                                            uint64_t kchk) {
  return j < W && x.x != 0 && mix64(x.x ^ kchk) == x.y && ids.ordered(x.x);
}

// Whether buckets base + lane + 32q, q < 2, of a warp's sum hold a good one;
// `edge` is the first one's id, in index order.
__device__ __forceinline__ bool warp_find(const ulonglong2 (&acc)[2], uint32_t base, uint32_t W, const IdSplit& ids,
                                          uint64_t kchk, uint64_t& edge) {
#pragma unroll
  for (uint32_t q = 0; q < 2; q++) {
    const uint32_t m =
        __ballot_sync(0xffffffffu, good_bucket(acc[q], base + (threadIdx.x & 31) + 32 * q, W, ids, kchk));
    if (m) {
      edge = __shfl_sync(0xffffffffu, acc[q].x, __ffs(m) - 1);
      return true;
    }
  }
  return false;
}

// The sample as far as the first kPrefix buckets decide it: 0 ZERO, 1 GOOD,
// 2 none of them is good.
__device__ __forceinline__ uint32_t warp_sample_prefix(const ulonglong2 (&acc)[2], uint32_t W,
                                                       const IdSplit& ids, uint64_t kchk, uint64_t& edge) {
  if (__shfl_sync(0xffffffffu, (acc[0].x | acc[0].y) == 0 ? 1u : 0u, 0)) return 0;
  return warp_find(acc, 0, W, ids, kchk, edge) ? 1u : 2u;
}

// Buckets base + lane + 32q, q < 2, of one member's row into acc.
__device__ __forceinline__ void warp_xor_part(ulonglong2 (&acc)[2], const ulonglong2* __restrict__ row, uint32_t base,
                                              uint32_t W, uint32_t lane) {
#pragma unroll
  for (uint32_t q = 0; q < 2; q++) {
    const uint32_t b = base + lane + 32 * q;
    if (b < W) {
      const ulonglong2 x = __ldg(row + b);
      acc[q].x ^= x.x;
      acc[q].y ^= x.y;
    }
  }
}

// One-cluster recovery of graphs of at most kClMaxV vertices
// (recover_small.cu): setup picks it (g->rec_cluster = CTAs of the cluster,
// 0 = the grid-wide kernel), launch runs it.
cudaError_t setup_recover_cluster(cupc_graph* g);
cudaError_t launch_recover_cluster(cupc_graph* g, const RecArgs& a, cudaStream_t s);

}  // namespace cupc

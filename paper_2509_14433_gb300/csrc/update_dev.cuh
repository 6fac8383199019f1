// Device-side pieces of the sketch update shared by the single-graph and the
// multi-graph kernels (see update.cu and batch.cu).
#pragma once

#include "common.cuh"

namespace cupc {

// Vertices with at most this many endpoint records in a batch take the
// direct path: no fold, each record's buckets are XORed straight into HBM.
constexpr uint32_t kDirectMax = 2;

// An endpoint record: the vertex it belongs to and the edge's other end. A
// padding record has the vertex itself there.
__device__ __forceinline__ uint64_t make_record(uint32_t w, uint32_t other) { return (uint64_t)w << 32 | other; }

// The edge id of a record.
__device__ __forceinline__ uint64_t record_id(uint64_t r, uint32_t V) {
  const uint32_t a = (uint32_t)(r >> 32), b = (uint32_t)r;
  return (uint64_t)min(a, b) * V + max(a, b);
}

// Block-wide exclusive scan of one u64 per thread (any multiple of 32 threads
// up to 1024): the prefix, and the block's total in `total`.
__device__ __forceinline__ uint64_t block_scan(uint64_t v, uint64_t* total) {
  __shared__ uint64_t sw[33];
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint64_t inc = v;
#pragma unroll
  for (uint32_t o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) sw[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    uint64_t x = lane < nw ? sw[lane] : 0;
    const uint64_t own = x;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    sw[lane] = x - own;
    if (lane == 31) sw[32] = x;
  }
  __syncthreads();
  *total = sw[32];
  return sw[wid] + inc - v;
}

// Work plan of one slice of kPlanSlice vertices, run by one CTA of
// kPlanThreads threads: gives each vertex a segment of the record array
// (cursor[w] = its start, count cnt[w]), resets cnt. Fold vertices fill the
// array from its start, padded to kPad records; direct vertices from its end
// (cap), unpadded. A slice takes its two ranges with one atomic each, so
// slices need not wait on one another; their order in the array does not
// matter, because the apply kernel reads each record's vertex from the
// record itself. Counts come in `shards` arrays of V; a vertex's segment is
// divided among them, cursor[k*V + w] = the start of shard k's records. The
// records of vertices with more than `hub` are counted.
__device__ __forceinline__ void plan_slice(uint32_t* cnt, uint32_t* cursor, uint64_t* rec, uint32_t V, uint32_t cap,
                                           uint32_t slice, uint32_t* work, bool dropped, uint32_t shards,
                                           uint32_t hub) {
  __shared__ uint32_t s_base[2];
  constexpr uint32_t kPer = kPlanSlice / kPlanThreads;
  const uint32_t w0 = slice * kPlanSlice + kPer * threadIdx.x;
  uint32_t c[kPer];
  uint64_t sum = 0;  // direct records << 32 | padded fold records
  uint32_t nhub = 0;
#pragma unroll
  for (uint32_t k = 0; k < kPer; k++) {
    c[k] = 0;
    for (uint32_t q = 0; q < shards && w0 + k < V; q++) c[k] += cnt[(size_t)q * V + w0 + k];
    sum += c[k] <= kDirectMax ? (uint64_t)c[k] << 32 : (uint64_t)((c[k] + kPad - 1) / kPad * kPad);
    if (c[k] > hub) nhub += c[k];
  }
  if (dropped) {
    for (uint32_t q = 0; q < shards; q++)
      for (uint32_t k = 0; k < kPer; k++)
        if (w0 + k < V) cnt[(size_t)q * V + w0 + k] = 0;
    return;
  }
  nhub = __reduce_add_sync(0xffffffffu, nhub);
  if (nhub && (threadIdx.x & 31) == 0) atomicAdd(&work[kWorkHub], nhub);
  uint64_t total;
  const uint64_t before = block_scan(sum, &total);
  if (threadIdx.x < 2) {
    const uint32_t t = threadIdx.x ? (uint32_t)(total >> 32) : (uint32_t)total;
    s_base[threadIdx.x] = t ? atomicAdd(&work[threadIdx.x ? kWorkDirect : kWorkFold], t) : 0;
  }
  __syncthreads();
  uint32_t fold = s_base[0] + (uint32_t)before, direct = cap - s_base[1] - (uint32_t)(before >> 32);
#pragma unroll
  for (uint32_t k = 0; k < kPer; k++) {
    if (c[k] == 0) continue;
    uint32_t at = fold;
    if (c[k] <= kDirectMax) at = direct -= c[k];
    for (uint32_t q = 0; q < shards; q++) {
      const size_t i = (size_t)q * V + w0 + k;
      cursor[i] = at;
      at += cnt[i];
      cnt[i] = 0;
    }
    if (c[k] > kDirectMax) {
      const uint32_t end = fold + (c[k] + kPad - 1) / kPad * kPad;
      for (uint32_t i = fold + c[k]; i < end; i++) rec[i] = make_record(w0 + k, w0 + k);
      fold = end;
    }
  }
}

__device__ __forceinline__ void xor_bucket_atomic(ulonglong2* p, ulonglong2 v) {
  atomicXor(&p->x, v.x);
  atomicXor(&p->y, v.y);
}

// Shared memory by its 32-bit address: address arithmetic on generic pointers
// would take 64 bits (twice the integer instructions of the loops below).
__device__ __forceinline__ uint64_t lds64(uint32_t p) {
  uint64_t v;
  asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(p));
  return v;
}
__device__ __forceinline__ ulonglong2 lds128(uint32_t p) {
  ulonglong2 v;
  asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(p));
  return v;
}
__device__ __forceinline__ void sts64(uint32_t p, uint64_t v) {
  asm volatile("st.shared.u64 [%0], %1;" ::"r"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t p, uint64_t x, uint64_t y) {
  asm volatile("st.shared.v2.u64 [%0], {%1, %2};" ::"r"(p), "l"(x), "l"(y) : "memory");
}

// XOR `bytes` (a multiple of 16) of shared memory into global memory, both
// 16-byte aligned. The calling thread's own shared writes are ordered before
// it; the source may be written again after bulk_wait_read in this thread.
__device__ __forceinline__ void bulk_xor(ulonglong2* dst, uint32_t src, uint32_t bytes) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.xor.b64 [%0], [%1], %2;" ::"l"(dst),
               "r"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// What one lane of an apply warp does. A warp owns 32/P layers of a graph
// (a layer group); lane = ll*P + s is layer group*32/P + ll, slot s: column s
// (s < C), the deterministic bucket (s == C) or idle.
//
// Column hash (Theorem A.1: 2-wise independent hash functions suffice):
// multiply-add-shift, h(x) = ((a*x + b) mod 2^64) div 2^(64-ell) with
// ell = 65 - 2*ceil(log2 V), strongly universal for indices x < V^2
// (Dietzfelbinger, STACS 1996); a second stage (a', b') continues the bit
// string when h(x) is zero. The depth is the number of leading zero bits of
// that string, capped at D-1. ell >= 23, so the high word z of a*x + b
// decides depths below 23: depth >= j is z < 2^(32-j).
//
// The deterministic lane uses a = 0, b = 2^63 (depth 0, z < t1 always), idle
// lanes z = 2^32 - 1 and t1 = 0 (never). Thresholds of depths beyond D-1 are 0.
struct ApplyLane {
  uint32_t a0, a1;         // first-stage multiplier, low and high word
  uint64_t kb;             // and addend
  const uint64_t* kx;      // {b, a', b'} of this lane's column (second stage)
  uint64_t kchk;           // checksum key of this lane's layer
  ulonglong2* base;        // bucket of depth 0, vertex 0
  uint32_t t1, t2;         // z below: depth >= 1, 2
  uint32_t tails;          // all ones where depths >= 3 exist (columns of D > 3), else 0
  uint32_t ell, dmax;      // bits per stage, D-1 (0 for the deterministic lane)
  uint32_t ll;             // layer within the group
  bool col, active;        // a column; a column or the deterministic bucket
  bool first;              // column 0: its bulk write also carries the deterministic bucket
};

// keys: K(r*(C+1) + c) = a of column c (c < C), K(r*(C+1) + C) = checksum
// key of layer r, K(L*(C+1) + 3*(r*C + c) + {0,1,2}) = b, a', b'.
__device__ __forceinline__ ApplyLane apply_lane(const uint64_t* keys, ulonglong2* sketch, uint32_t V, uint32_t L,
                                                uint32_t C, uint32_t D, uint32_t W, uint32_t P, uint32_t ell,
                                                uint32_t group) {
  ApplyLane l;
  const uint32_t lane = threadIdx.x & 31, s = lane % P, ll = lane / P, r = group * (32 / P) + ll;
  const bool in = r < L;
  l.col = in && s < C;
  l.active = in && s <= C;
  l.first = l.col && s == 0;
  const uint64_t a = l.col ? keys[r * (C + 1) + s] : 0ull;
  l.a0 = (uint32_t)a;
  l.a1 = (uint32_t)(a >> 32);
  l.kx = l.col ? keys + (size_t)L * (C + 1) + 3 * (size_t)(r * C + s) : nullptr;
  const bool det = in && s == C;
  l.kb = l.col ? l.kx[0] : (det ? 1ull << 63 : ~0ull);
  l.kchk = in ? keys[r * (C + 1) + C] : 0ull;
  l.base = sketch + ((size_t)(in ? r : 0) * V) * W + (s < C ? 1u + s * D : 0u);
  l.t1 = det ? 0xFFFFFFFFu : (l.col && D > 1 ? 1u << 31 : 0u);
  l.t2 = l.col && D > 2 ? 1u << 30 : 0u;
  l.tails = l.col && D > 3 ? ~0u : 0u;
  l.ell = ell;
  l.dmax = l.col ? D - 1 : 0u;
  l.ll = ll;
  return l;
}

// High word of a*x + b. kX32: x < 2^32 (V <= 65536).
template <bool kX32>
__device__ __forceinline__ uint32_t lane_z(const ApplyLane& l, uint64_t x) {
  const uint32_t x0 = (uint32_t)x;
  uint32_t z = (uint32_t)(((uint64_t)l.a0 * x0 + l.kb) >> 32) + l.a1 * x0;
  if (!kX32) z += l.a0 * (uint32_t)(x >> 32);
  return z;
}

// The exact depth when z does not decide it: leading zeros of the 2*ell-bit
// string h(x) h'(x) (probability 2^-min(ell,32)).
static __device__ __noinline__ uint32_t depth_long(uint64_t a, uint64_t b, const uint64_t* kx, uint32_t ell,
                                                   uint64_t x) {
  uint32_t d = min((uint32_t)__clzll((long long)(a * x + b)), ell);
  if (d == ell) d += min((uint32_t)__clzll((long long)(kx[1] * x + kx[2])), ell);
  return d;
}

template <bool kX32>
__device__ __forceinline__ uint32_t lane_depth(const ApplyLane& l, uint64_t x) {
  uint32_t d = (uint32_t)__clz((int)lane_z<kX32>(l, x));
  if (d >= min(l.ell, 32u) && l.col) d = depth_long((uint64_t)l.a1 << 32 | l.a0, l.kb, l.kx, l.ell, x);
  return min(d, l.dmax);
}

// Highest set bit (all ones if v is zero).
__device__ __forceinline__ uint32_t top_bit(uint32_t v) {
  uint32_t b;
  asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(v));
  return b;
}

// Shared memory of an apply warp: the staged records of a pass (edge ids x,
// and their checksums of every layer of the group, kStageStride apart so that
// the layers' equal positions fall into different banks), and `nslots`
// buckets a lane: slot 0 for the deterministic bucket (column 0's lane), slot
// 1+d for row d. An odd slot count spreads the lanes' equal slots over the
// banks.
struct ApplySmem {
  uint32_t x;      // kStage edge ids
  uint32_t g;      // kStage checksums of this lane's layer
  uint32_t slots;  // this lane's buckets
};
__device__ __forceinline__ ApplySmem apply_smem(unsigned char* warp_smem, uint32_t nslots, uint32_t P) {
  const uint32_t lane = threadIdx.x & 31;
  ApplySmem m;
  m.x = (uint32_t)__cvta_generic_to_shared(warp_smem);
  m.slots = m.x + kStage * 8 + lane * nslots * 16;
  m.g = m.x + kStage * 8 + 32 * nslots * 16 + lane / P * kStageStride * 8;
  return m;
}

// The sums a lane carries over the records of one vertex: s1, s2 and s3 hold
// {alpha, gamma} of the records of depth >= 1, 2 and 3 (the deterministic
// lane's s1: of all records).
struct LaneSums {
  uint32_t s1[4], s2[4], s3[4];
  uint32_t top;    // highest slot that holds records of depth >= 3 (0: none)
  uint32_t dirty;  // that of the previous vertex, zeroed before the slots' next use
};

__device__ __forceinline__ void clear_sums(LaneSums& a) {
#pragma unroll
  for (int k = 0; k < 4; k++) a.s1[k] = a.s2[k] = a.s3[k] = 0;
  a.top = 0;
}

// One record into the sums of depths >= 1 and >= 2; `t` shifts in a 0 when the
// depth is >= 3 (z + 7*2^29 carries exactly when z >= 2^29), else a 1.
template <bool kX32>
__device__ __forceinline__ void fold_record(const ApplyLane& l, LaneSums& a, uint64_t x, uint64_t g, uint32_t& t) {
  const uint32_t z = lane_z<kX32>(l, x);
  const uint32_t x0 = (uint32_t)x, x1 = (uint32_t)(x >> 32), g0 = (uint32_t)g, g1 = (uint32_t)(g >> 32);
  if (kX32) {
    asm("{.reg .pred p, q;\n\t.reg .u32 u;\n\t"
        "setp.lt.u32 p, %7, %8;\n\tsetp.lt.u32 q, %7, %9;\n\t"
        "@p xor.b32 %0, %0, %10;\n\t@p xor.b32 %1, %1, %11;\n\t@p xor.b32 %2, %2, %12;\n\t"
        "@q xor.b32 %3, %3, %10;\n\t@q xor.b32 %4, %4, %11;\n\t@q xor.b32 %5, %5, %12;\n\t"
        "add.cc.u32 u, %7, 0xE0000000;\n\taddc.u32 %6, %6, %6;}"
        : "+r"(a.s1[0]), "+r"(a.s1[2]), "+r"(a.s1[3]), "+r"(a.s2[0]), "+r"(a.s2[2]), "+r"(a.s2[3]), "+r"(t)
        : "r"(z), "r"(l.t1), "r"(l.t2), "r"(x0), "r"(g0), "r"(g1));
  } else {
    asm("{.reg .pred p, q;\n\t.reg .u32 u;\n\t"
        "setp.lt.u32 p, %9, %10;\n\tsetp.lt.u32 q, %9, %11;\n\t"
        "@p xor.b32 %0, %0, %12;\n\t@p xor.b32 %1, %1, %13;\n\t@p xor.b32 %2, %2, %14;\n\t@p xor.b32 %3, %3, %15;\n\t"
        "@q xor.b32 %4, %4, %12;\n\t@q xor.b32 %5, %5, %13;\n\t@q xor.b32 %6, %6, %14;\n\t@q xor.b32 %7, %7, %15;\n\t"
        "add.cc.u32 u, %9, 0xE0000000;\n\taddc.u32 %8, %8, %8;}"
        : "+r"(a.s1[0]), "+r"(a.s1[1]), "+r"(a.s1[2]), "+r"(a.s1[3]), "+r"(a.s2[0]), "+r"(a.s2[1]), "+r"(a.s2[2]),
          "+r"(a.s2[3]), "+r"(t)
        : "r"(z), "r"(l.t1), "r"(l.t2), "r"(x0), "r"(x1), "r"(g0), "r"(g1));
  }
}

// Before the slots are written again: the bulk write of the previous vertex
// has read them, and the rows it left behind are zeroed.
__device__ __forceinline__ void reuse_slots(const ApplySmem& m, LaneSums& a, bool& pending) {
  if (!pending) return;
  bulk_wait_read();
  for (uint32_t q = 4; q <= a.dirty; q++) sts128(m.slots + 16 * q, 0, 0);
  a.dirty = 0;
  pending = false;
}

// The staged records [pos, end) of vertex w (pos and end multiples of kPad)
// into the lane's sums; pads: stage_records. Depths 0..2 stay in registers; a
// record of depth >= 3 (one in eight) is marked in a bitmask per lane, and the
// lanes then walk their own marks side by side and fold those records into
// their slots (rows 3..R-1). Deeper records (slot 0 takes them, which is
// overwritten before it is used) are walked once more and go straight into HBM.
template <bool kX32>
__device__ __forceinline__ void fold_range(const ApplyLane& l, const ApplySmem& m, LaneSums& a, bool& pending,
                                           uint32_t pos, uint32_t end, uint32_t pads, uint32_t w, uint32_t W,
                                           uint32_t R) {
  const uint32_t gx = m.g - m.x, xe = m.x + 8 * end;
  uint32_t t = ~0u;  // a 0 is shifted in for a deep record
  static_assert(kPad == 4, "a vertex's records in a pass are whole groups of four");
#pragma unroll 2
  for (uint32_t px = m.x + 8 * pos; px < xe; px += 32) {
    const ulonglong2 xa = lds128(px), ga = lds128(px + gx), xb = lds128(px + 16), gb = lds128(px + gx + 16);
    fold_record<kX32>(l, a, xa.x, ga.x, t);
    fold_record<kX32>(l, a, xa.y, ga.y, t);
    fold_record<kX32>(l, a, xb.x, gb.x, t);
    fold_record<kX32>(l, a, xb.y, gb.y, t);
  }
  // bit b: record end-1-b has depth >= 3 and is no padding, whose id is zero: in
  // a column whose hash of zero is deep all of it would be walked, and go to HBM
  // where that is R or deeper. One seed in twenty has such a column at V = 2^14;
  // 320000 R-MAT edges then took 288 us on GB300, 269 without the padding.
  t = ~t & l.tails & ~(pads >> (32 - end));
  reuse_slots(m, a, pending);
  uint32_t deep = 0;
  while (t) {
    const uint32_t b = top_bit(t), bit = 1u << b, at = xe - 8 - 8 * b;
    const uint64_t x = lds64(at), g = lds64(at + gx);
    t ^= bit;
    a.s3[0] ^= (uint32_t)x;
    if (!kX32) a.s3[1] ^= (uint32_t)(x >> 32);
    a.s3[2] ^= (uint32_t)g;
    a.s3[3] ^= (uint32_t)(g >> 32);
    uint32_t q = 32 - top_bit(lane_z<kX32>(l, x));  // 1 + depth
    if (q > R) {
      q = 0;
      deep |= bit;
    }
    const uint32_t slot = m.slots + 16 * q;
    const ulonglong2 v = lds128(slot);
    sts128(slot, v.x ^ x, v.y ^ g);
    a.top = max(a.top, q);
  }
  while (deep) {
    const uint32_t b = top_bit(deep), at = xe - 8 - 8 * b;
    deep ^= 1u << b;
    const uint64_t x = lds64(at), g = lds64(at + gx);
    xor_bucket_atomic(l.base + (size_t)w * W + lane_depth<kX32>(l, x), make_ulonglong2(x, g));
  }
  __syncwarp();
}

__device__ __forceinline__ ulonglong2 sum_of(const uint32_t (&u)[4]) {
  return make_ulonglong2((uint64_t)u[1] << 32 | u[0], (uint64_t)u[3] << 32 | u[2]);
}
// slot = u ^ v
__device__ __forceinline__ void put_slot(uint32_t slot, ulonglong2 u, ulonglong2 v) {
  sts128(slot, u.x ^ v.x, u.y ^ v.y);
}

// XOR the sums of vertex w into HBM: each column's touched rows are one run
// of contiguous buckets, written by one bulk reduction per lane (column 0's
// run starts with the deterministic bucket, which is its neighbour). Row d is
// the sum of depth >= d less the sum of depth >= d+1; the sum over all
// records comes from the deterministic lane.
__device__ __forceinline__ void flush_vertex(const ApplyLane& l, const ApplySmem& m, LaneSums& a, bool& pending,
                                             uint32_t w, uint32_t W, uint32_t C, uint32_t P) {
  reuse_slots(m, a, pending);
  uint32_t s0[4];
  const uint32_t det = (threadIdx.x & 31 & ~(P - 1)) + C;
#pragma unroll
  for (int k = 0; k < 4; k++) s0[k] = __shfl_sync(0xffffffffu, a.s1[k], det);
  if (l.col) {
    const ulonglong2 v0 = sum_of(s0), v1 = sum_of(a.s1), v2 = sum_of(a.s2), v3 = sum_of(a.s3);
    put_slot(m.slots + 16, v0, v1);
    put_slot(m.slots + 32, v1, v2);
    put_slot(m.slots + 48, v2, v3);
    if (l.first) sts128(m.slots, v0.x, v0.y);
    const uint32_t any2 = a.s2[0] | a.s2[1] | a.s2[2] | a.s2[3];
    const uint32_t nrows = min(l.dmax + 1, max(a.top, any2 ? 3u : 2u));
    const uint32_t f = l.first ? 1u : 0u;
    bulk_xor(l.base + (size_t)w * W - f, m.slots + 16 - 16 * f, (nrows + f) * 16);
  }
  bulk_commit();
  pending = true;
  a.dirty = a.top;
  clear_sums(a);
}

// Stage a pass of records, one per lane: their edge ids and, for every layer
// of the group, their checksums. Padding records become zeros, which change
// no sum; returns them as a mask, record i at bit 31 - i.
__device__ __forceinline__ uint32_t stage_records(const ApplyLane& l, const ApplySmem& m, uint64_t r, uint32_t V,
                                              uint32_t P) {
  const uint32_t lane = threadIdx.x & 31;
  const bool pad = (uint32_t)(r >> 32) == (uint32_t)r;
  const uint64_t x = pad ? 0ull : record_id(r, V);
  uint32_t g = m.g - lane / P * kStageStride * 8 + lane * 8;
  __syncwarp();  // every lane is done with the previous pass
  sts64(m.x + 8 * lane, x);
  if (P == 8) {
#pragma unroll
    for (uint32_t k = 0; k < 4; k++) {
      const uint64_t c = mix64(x ^ __shfl_sync(0xffffffffu, l.kchk, 8 * k));
      sts64(g + 8 * kStageStride * k, pad ? 0ull : c);
    }
  } else {
    for (uint32_t k = 0; k < 32; k += P, g += 8 * kStageStride) {
      const uint64_t c = mix64(x ^ __shfl_sync(0xffffffffu, l.kchk, k));
      sts64(g, pad ? 0ull : c);
    }
  }
  __syncwarp();
  return __brev(__ballot_sync(0xffffffffu, pad));
}

// A chunk of a graph's records. The fold chunks come first, then the direct
// ones, which end at the end of the record array.
struct Chunk {
  const uint64_t* rec;
  uint32_t n;  // records (a multiple of kPad in a fold chunk), 0: none
  bool fold;
};
struct ChunkPlan {
  uint32_t nfold, ndirect, chunk, nf, total;  // records; of a chunk; fold chunks, chunks
};
// hub_chunk: the chunk size if hubs hold more than an eighth of the records.
__device__ __forceinline__ ChunkPlan chunk_plan(const uint32_t* work, uint32_t chunk, uint32_t hub_chunk) {
  ChunkPlan c;
  c.nfold = ld_cg(&work[kWorkFold]);
  c.ndirect = ld_cg(&work[kWorkDirect]);
  c.chunk = chunk;
  if (hub_chunk != chunk && ld_cg(&work[kWorkHub]) > (c.nfold + c.ndirect) / 8) c.chunk = hub_chunk;
  c.nf = (c.nfold + c.chunk - 1) / c.chunk;
  c.total = c.nf + (c.ndirect + c.chunk - 1) / c.chunk;
  return c;
}
__device__ __forceinline__ Chunk chunk_at(const ChunkPlan& c, uint32_t q, const uint64_t* rec, uint32_t cap) {
  Chunk k;
  k.fold = q < c.nf;
  const uint32_t b = (k.fold ? q : q - c.nf) * c.chunk, all = k.fold ? c.nfold : c.ndirect;
  k.n = q < c.total ? min(c.chunk, all - b) : 0u;
  k.rec = rec + (k.fold ? 0u : cap - c.ndirect) + b;
  return k;
}

// This lane's record of the pass at p of chunk k, or of the first pass of the
// next chunk when k ends there: loaded one pass ahead of its use.
__device__ __forceinline__ uint64_t load_record(const Chunk& k, uint32_t p, const Chunk& next) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t* at = p < k.n ? k.rec + p : next.rec;
  return lane < (p < k.n ? k.n - p : next.n) ? __ldg(at + lane) : 0ull;
}

// One chunk of the fold vertices' records into the layers of this warp's
// group, 32 records a pass (r: this lane's record of the first pass). The
// records of a vertex are folded together and written back when the vertex or
// the chunk ends.
template <bool kX32>
__device__ __forceinline__ void fold_chunk(const ApplyLane& l, const ApplySmem& m, LaneSums& a, bool& pending,
                                           const Chunk& k, const Chunk& next, uint64_t& r, uint32_t V, uint32_t W,
                                           uint32_t C, uint32_t P, uint32_t R) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t w = __shfl_sync(0xffffffffu, (uint32_t)(r >> 32), 0);  // the vertex being folded
  for (uint32_t p = 0; p < k.n; p += kStage) {
    const uint32_t nc = min(kStage, k.n - p), wr = (uint32_t)(r >> 32);
    const uint32_t pads = stage_records(l, m, r, V, P);
    r = load_record(k, p + kStage, next);
    uint32_t before = __shfl_up_sync(0xffffffffu, wr, 1);
    if (lane == 0) before = w;
    uint32_t heads = __ballot_sync(0xffffffffu, lane < nc && wr != before);
    for (uint32_t pos = 0; pos < nc;) {
      if (heads & 1u << pos) {
        flush_vertex(l, m, a, pending, w, W, C, P);
        w = __shfl_sync(0xffffffffu, wr, pos);
        heads &= heads - 1;
      }
      const uint32_t end = heads ? __ffs((int)heads) - 1 : nc;
      fold_range<kX32>(l, m, a, pending, pos, end, pads, w, W, R);
      pos = end;
    }
  }
  flush_vertex(l, m, a, pending, w, W, C, P);
}

// One chunk of the direct vertices' records: every bucket of every record
// straight into HBM.
template <bool kX32>
__device__ __forceinline__ void direct_chunk(const ApplyLane& l, const ApplySmem& m, const Chunk& k, const Chunk& next,
                                             uint64_t& r, uint32_t V, uint32_t W, uint32_t P) {
  for (uint32_t p = 0; p < k.n; p += kStage) {
    const uint32_t nc = min(kStage, k.n - p), wr = (uint32_t)(r >> 32);
    stage_records(l, m, r, V, P);
    r = load_record(k, p + kStage, next);
#pragma unroll 4
    for (uint32_t i = 0; i < nc; i++) {
      const uint32_t w = __shfl_sync(0xffffffffu, wr, i);
      const uint64_t x = lds64(m.x + 8 * i), g = lds64(m.g + 8 * i);
      const uint32_t d = lane_depth<kX32>(l, x);
      if (l.active) xor_bucket_atomic(l.base + (size_t)w * W + d, make_ulonglong2(x, g));
    }
  }
}

template <bool kX32>
__device__ __forceinline__ void apply_chunk(const ApplyLane& l, const ApplySmem& m, LaneSums& a, bool& pending,
                                            const Chunk& k, const Chunk& next, uint64_t& r, uint32_t V, uint32_t W,
                                            uint32_t C, uint32_t P, uint32_t R) {
  if (k.fold)
    fold_chunk<kX32>(l, m, a, pending, k, next, r, V, W, C, P, R);
  else
    direct_chunk<kX32>(l, m, k, next, r, V, W, P);
}

// Zero a lane's slots (before its first chunk).
__device__ __forceinline__ void zero_slots(const ApplySmem& m, uint32_t nslots) {
  for (uint32_t q = 0; q < nslots; q++) sts128(m.slots + 16 * q, 0, 0);
}

}  // namespace cupc

// Loop subdivision with on-the-fly reuse (Section 5.2): one subdivision step
// of a triangle mesh, streamed triangle by triangle.  Each input triangle
// (v0, v1, v2) yields four output triangles
//   (E0, M0, M2), (E1, M1, M0), (E2, M2, M1), (M0, M1, M2)
// where E_k is vertex k moved by Loop's vertex rule (its 1-ring, weight beta
// of Loop's thesis; boundary vertices: 3/4 v + 1/8 of their two boundary
// neighbours) and M_k is the new vertex on edge (v_k, v_k+1) (3/8 of the
// edge's ends plus 1/8 of the two opposite vertices; boundary edges: the
// midpoint).  The vertex rule reads a whole 1-ring, so it is the "vertex
// shader" the reuse methods share:
//   naive            -- every triangle evaluates its three vertices itself;
//   warp             -- Algorithm 1's rounds on static batches, one warp per
//                       batch: the lanes holding a round's vertices evaluate
//                       the rule, the round's triangles gather it by shuffles;
//   sort/hash/phash  -- one thread block per batch (static, or the dynamic
//                       batches of the partition) runs the shared dedup body;
//                       each unique vertex's rule is evaluated once into
//                       shared memory together with its position, then one
//                       thread per triangle builds the edge vertices and
//                       writes the four triangles.
// Output: 4 triangles x 3 corners x 3 floats = 144 bytes (9 aligned 16-byte
// words) per input triangle, in input order.
#include <algorithm>

#include "gp.h"
#include "gp_batch_body.cuh"
#include "gp_warp_body.cuh"

namespace gp {

struct LoopArgs {
  const uint32_t* idx;
  uint32_t num_tris;
  const unsigned char* verts;
  uint32_t stride, num_verts;
  uint32_t vec16;                 // 1: rows are 16-byte aligned (one load per position)
  const uint32_t* ring_off;
  const uint32_t* ring;
  uint32_t ring_count;
  uint32_t ring16;                // 1: the ring array is 16-byte aligned
  const uint32_t* vflags;
  const uint32_t* opp;
  float* out;
  const uint32_t* starts;         // dynamic batches (triangles), or nullptr for static
  uint32_t static_tris;           // static: triangles per batch
  uint32_t num_batches;           // static
  const uint32_t* num_batches_dev;  // dynamic
  unsigned long long* counters;   // [0] vertex-rule evaluations, [1] batches, [2] error bits
};

// Position of vertex v; an id out of range (a bad index or adjacency entry)
// reads as the origin and sets 'bad'.  No side effects: the loads of several
// positions go out together.  VEC: in one load where the rows allow it.
template <bool VEC>
__device__ __forceinline__ float3 loop_fetch(const LoopArgs& a, uint32_t v, bool& bad) {
  if (v >= a.num_verts) {
    bad = true;
    return make_float3(0.f, 0.f, 0.f);
  }
  const unsigned char* row = a.verts + (size_t)v * a.stride;
  if (VEC && a.vec16) {
    const float4 x = __ldg(reinterpret_cast<const float4*>(row));
    return make_float3(x.x, x.y, x.z);
  }
  const float* p = reinterpret_cast<const float*>(row);
  return make_float3(__ldg(p), __ldg(p + 1), __ldg(p + 2));
}

constexpr uint32_t kLoopStage = 16;  // triangles staged at once by a warp: all 32 cost more cache than they spare stores

__device__ __forceinline__ void loop_flag(const LoopArgs& a, bool bad) {
  if (bad) atomicOr(a.counters + 2, (unsigned long long)EBIT_INDEX_RANGE);
}

// The same, flagging GP_ERR_INDEX_RANGE by itself.
template <bool VEC>
__device__ __forceinline__ float3 loop_pos(const LoopArgs& a, uint32_t v) {
  bool bad = false;
  const float3 p = loop_fetch<VEC>(a, v, bad);
  loop_flag(a, bad);
  return p;
}

// Ring entries k..k + 3 (k < o1, a multiple of 4), of which the caller uses those
// in [o0, o1) (o1 <= ring_count): one 16-byte load where the array has all four.
// Rings of unrelated vertices are read side by side, so every load of a warp
// touches as many lines as it has lanes: two or three loads a ring instead of six
// (hash, phash and naive: 54 us with it, 56 without, at 500k triangles; warp
// voting and sort lose 4 us on a mesh whose rings lie in the order of its
// triangles, and read entry by entry).
__device__ __forceinline__ uint4 loop_ring4(const LoopArgs& a, uint32_t k, uint32_t o0, uint32_t o1) {
  if (a.ring16 && a.ring_count - k >= 4) return __ldg(reinterpret_cast<const uint4*>(a.ring + k));
  uint4 r = make_uint4(0, 0, 0, 0);
  if (k >= o0) r.x = __ldg(a.ring + k);
  if (k + 1 >= o0 && o1 - k > 1) r.y = __ldg(a.ring + k + 1);
  if (k + 2 >= o0 && o1 - k > 2) r.z = __ldg(a.ring + k + 2);
  if (k + 3 >= o0 && o1 - k > 3) r.w = __ldg(a.ring + k + 3);
  return r;
}

// Loop's vertex rule for vertex v at p.
template <bool WIDE, bool VEC>
__device__ __forceinline__ float3 loop_even(const LoopArgs& a, uint32_t v, float3 p) {
  if (v >= a.num_verts) return p;
  // ring entries past the ring array (inconsistent adjacency) are not read
  const uint32_t o0 = min(__ldg(a.ring_off + v), a.ring_count);
  const uint32_t o1 = max(o0, min(__ldg(a.ring_off + v + 1), a.ring_count));
  if ((__ldg(a.vflags + v) & 1u) && o1 - o0 >= 2) {
    const float3 b0 = loop_pos<VEC>(a, __ldg(a.ring + o0)), b1 = loop_pos<VEC>(a, __ldg(a.ring + o0 + 1));
    return make_float3(__fmaf_rn(0.75f, p.x, __fmul_rn(0.125f, __fadd_rn(b0.x, b1.x))),
                       __fmaf_rn(0.75f, p.y, __fmul_rn(0.125f, __fadd_rn(b0.y, b1.y))),
                       __fmaf_rn(0.75f, p.z, __fmul_rn(0.125f, __fadd_rn(b0.z, b1.z))));
  }
  const uint32_t n = o1 - o0;
  if (n == 0) return p;
  float sx = 0.f, sy = 0.f, sz = 0.f;
  if (WIDE) {
    // 4 entries at a time: their positions' loads in flight together, and the next entries' beside them
    bool bad = false;
    uint4 ids = loop_ring4(a, o0 & ~3u, o0, o1);
    for (uint32_t k = o0 & ~3u;; k += 4) {
      const uint32_t id[4] = {ids.x, ids.y, ids.z, ids.w};
      const bool more = o1 - k > 4;  // (k + 4 may wrap)
      if (more) ids = loop_ring4(a, k + 4, o0, o1);
      float3 q[4];
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i)
        if (k + i >= o0 && i < o1 - k) q[i] = loop_fetch<VEC>(a, id[i], bad);
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i)
        if (k + i >= o0 && i < o1 - k) {
          sx = __fadd_rn(sx, q[i].x);
          sy = __fadd_rn(sy, q[i].y);
          sz = __fadd_rn(sz, q[i].z);
        }
      if (!more) break;
    }
    loop_flag(a, bad);
  } else {
    for (uint32_t k = o0; k < o1; ++k) {
      const float3 q = loop_pos<VEC>(a, __ldg(a.ring + k));
      sx = __fadd_rn(sx, q.x);
      sy = __fadd_rn(sy, q.y);
      sz = __fadd_rn(sz, q.z);
    }
  }
  const float c = __fmaf_rn(0.25f, cosf(6.283185307179586f / (float)n), 0.375f);
  const float beta = __fdiv_rn(__fmaf_rn(-c, c, 0.625f), (float)n);
  const float w = __fmaf_rn(-(float)n, beta, 1.0f);
  return make_float3(__fmaf_rn(w, p.x, __fmul_rn(beta, sx)), __fmaf_rn(w, p.y, __fmul_rn(beta, sy)),
                     __fmaf_rn(w, p.z, __fmul_rn(beta, sz)));
}

// Loop's edge rule for edge (pa, pb) with opposite vertices pc (this
// triangle) and pd (the neighbour; none on a boundary).
__device__ __forceinline__ float3 loop_odd(float3 pa, float3 pb, float3 pc, bool boundary, float3 pd) {
  if (boundary)
    return make_float3(__fmul_rn(0.5f, __fadd_rn(pa.x, pb.x)), __fmul_rn(0.5f, __fadd_rn(pa.y, pb.y)),
                       __fmul_rn(0.5f, __fadd_rn(pa.z, pb.z)));
  return make_float3(__fmaf_rn(0.375f, __fadd_rn(pa.x, pb.x), __fmul_rn(0.125f, __fadd_rn(pc.x, pd.x))),
                     __fmaf_rn(0.375f, __fadd_rn(pa.y, pb.y), __fmul_rn(0.125f, __fadd_rn(pc.y, pd.y))),
                     __fmaf_rn(0.375f, __fadd_rn(pa.z, pb.z), __fmul_rn(0.125f, __fadd_rn(pc.z, pd.z))));
}

// Writes the four output triangles of each of the warp's triangles [t, t + n), a
// lane's from its moved vertices E and positions P (corner order).  Called by
// the whole warp.  A lane's 144 bytes go through shared memory ('stage', 9
// 16-byte words a lane: an odd stride, no bank conflicts), so that the warp
// writes whole lines; written by the lanes themselves, each store touched 32 of
// them.  With the rings read 16 bytes at a time: 500k triangles in 55 us, 62.5
// before.  (STAGED false, warp voting: its rounds end after a few triangles, and
// the stage's barriers cost it 4 us of 56 on a grid; and the lean batched kernels.)
template <bool STAGED, bool VEC, bool SERIAL>
__device__ __forceinline__ void loop_emit(const LoopArgs& a, uint32_t t, uint32_t n, const float3* E, const float3* P,
                                          float4* stage, uint32_t lane) {
  float f[36];
  if (lane < n) {
    float3 M[3];
    bool bad = false;
    if (!SERIAL) {
      uint32_t d[3];
      float3 D[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) d[k] = __ldg(a.opp + 3 * (t + lane) + k);
#pragma unroll
      for (int k = 0; k < 3; ++k) D[k] = d[k] != kEmpty ? loop_fetch<VEC>(a, d[k], bad) : make_float3(0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 3; ++k) M[k] = loop_odd(P[k], P[(k + 1) % 3], P[(k + 2) % 3], d[k] == kEmpty, D[k]);
    } else {  // the lean kernels' registers: one edge after another
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const uint32_t d = __ldg(a.opp + 3 * (t + lane) + k);
        float3 D = make_float3(0.f, 0.f, 0.f);
        if (d != kEmpty) D = loop_fetch<VEC>(a, d, bad);
        M[k] = loop_odd(P[k], P[(k + 1) % 3], P[(k + 2) % 3], d == kEmpty, D);
      }
    }
    loop_flag(a, bad);
    const float3 c[12] = {E[0], M[0], M[2], E[1], M[1], M[0], E[2], M[2], M[1], M[0], M[1], M[2]};
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      f[3 * k] = c[k].x;
      f[3 * k + 1] = c[k].y;
      f[3 * k + 2] = c[k].z;
    }
  }
  if (!STAGED) {
    float4* o = reinterpret_cast<float4*>(a.out) + (size_t)(t + lane) * 9;
#pragma unroll
    for (int w = 0; w < 9; ++w)
      if (lane < n) __stcs(o + w, make_float4(f[4 * w], f[4 * w + 1], f[4 * w + 2], f[4 * w + 3]));
    return;
  }
#pragma unroll
  for (uint32_t l0 = 0; l0 < 32; l0 += kLoopStage) {
    __syncwarp();  // the stage's last readers
    if (lane - l0 < kLoopStage && lane < n) {
#pragma unroll
      for (int w = 0; w < 9; ++w)
        stage[9 * (lane - l0) + w] = make_float4(f[4 * w], f[4 * w + 1], f[4 * w + 2], f[4 * w + 3]);
    }
    __syncwarp();
    const uint32_t words = l0 < n ? 9 * min(n - l0, kLoopStage) : 0u;
    float4* o = reinterpret_cast<float4*>(a.out) + (size_t)(t + l0) * 9;
#pragma unroll
    for (uint32_t w = lane; w < 9 * kLoopStage; w += 32)
      if (w < words) __stcs(o + w, stage[w]);
  }
}

__global__ void __launch_bounds__(256) loop_naive_kernel(const __grid_constant__ LoopArgs a) {
  __shared__ float4 stage[8 * 9 * kLoopStage];
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, lane = lane_id(), warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    atomicAdd(a.counters + 0, 3ull * min(blockDim.x, a.num_tris - blockIdx.x * blockDim.x));
    atomicAdd(a.counters + 1, 1ull);
  }
  if (t - lane >= a.num_tris) return;
  float3 E[3], P[3];
  if (t < a.num_tris) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint32_t v = __ldg(a.idx + 3 * t + k);
      P[k] = loop_pos<true>(a, v);
      E[k] = loop_even<true, true>(a, v, P[k]);
    }
  }
  loop_emit<true, true, false>(a, t - lane, min(32u, a.num_tris - (t - lane)), E, P, stage + warp * 9 * kLoopStage, lane);
}

// Evaluates the vertex rule of the warp's new ranks into shared memory.
template <bool WIDE, bool VEC>
struct LoopEven {
  const LoopArgs& la;
  const uint32_t* uniq;
  float* esh;  // rank -> moved position (3 floats)
  float* psh;  // rank -> position (3 floats)
  uint32_t ucap;
  __device__ __forceinline__ void operator()(uint32_t rb, uint32_t re, uint32_t lane) const {
    re = min(re, ucap);  // ranks >= ucap (a flagged capacity error) were not stored
    for (uint32_t r = rb + lane; r < re; r += 32) {
      const uint32_t v = uniq[r];
      const float3 p = loop_pos<VEC>(la, v), e = loop_even<WIDE, VEC>(la, v, p);
      esh[3 * r] = e.x; esh[3 * r + 1] = e.y; esh[3 * r + 2] = e.z;
      psh[3 * r] = p.x; psh[3 * r + 1] = p.y; psh[3 * r + 2] = p.z;
    }
  }
};

// Shared memory of a block.  The warps' stages ('threads': of those that write
// staged, 0 for the lean kernels) lie over what the deduplication alone needs: with
// 7.0 KB a block (64 unique vertices) instead of 8.5 the rest of the SM's 256 KB
// stays cache for the rings' positions, which neighbouring batches share.
struct LoopLayout {
  uint32_t off_table, off_win, off_uniq, off_map, off_even, off_dense, off_misc, total;
};

__host__ __device__ inline LoopLayout loop_layout(int dedup, uint32_t cap, uint32_t ucap, uint32_t slots,
                                                  uint32_t sort_n, uint32_t threads) {
  LoopLayout L;
  uint32_t o = 0;
  L.off_table = o; o += dedup == DEDUP_SORT ? sort_n * 8 : slots * 4;
  L.off_win = o; o += cap * 4;
  L.off_uniq = o; o += ucap * 4;
  const uint32_t with = (cap / 3 + 31) / 32, warps = threads / 32;  // warps with triangles to write
  const uint32_t stages = (warps < with ? warps : with) * kLoopStage * 144;
  o = o > stages ? o : stages;
  L.off_even = o; o += ucap * 24;
  L.off_misc = o; o += 64 * 4;
  L.off_map = o; o += ((cap + 1) & ~1u) * 2;
  L.off_dense = o; o += dedup == DEDUP_SORT ? 0u : slots * 2;
  L.total = o;
  return L;
}

// 56 registers: fewer spill, more leave the batches of 64 threads fewer blocks
// (500k triangles: 55 us; with 64 registers 58, with 48 57).  What bounds it is
// the L1's line lookups (a gather is one per lane) and the chain of seven
// dependent loads; a block running consecutive batches one after another for its
// L1's sake took 62 to 71 us.
// LEAN, batches of at most half as many triangles as threads: most warps have
// nothing to write, and what counts is how many blocks share an SM.  40 registers,
// triangles written by their lanes, rings read entry by entry and, but for sort,
// positions word by word (hash, S = 96, 2M triangles of a grid, us: 128 threads 227
// and, as the others, 321; 256 threads 408 and 660).
template <int DEDUP, bool LEAN>
__global__ void __maxnreg__(LEAN ? 40 : DEDUP == DEDUP_SORT ? 64 : 56)
    loop_batched_kernel(const __grid_constant__ LoopArgs la, const __grid_constant__ DrawArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool kVec = !LEAN || DEDUP == DEDUP_SORT;
  const uint32_t tid = threadIdx.x, NT = blockDim.x;
  const uint32_t nb = la.starts ? *la.num_batches_dev : la.num_batches;
  const uint32_t b = blockIdx.x;
  if (b >= nb) return;
  uint32_t t0, t1;
  if (la.starts) {
    t0 = __ldg(la.starts + b);
    t1 = __ldg(la.starts + b + 1);
  } else {
    t0 = b * la.static_tris;
    t1 = min(t0 + la.static_tris, la.num_tris);
  }
  const uint32_t n = 3 * (t1 - t0), cap = a.max_batch_idx, ucap = a.ucap;
  if (n > cap) {  // cannot happen with a consistent partition
    if (tid == 0) atomicOr(a.err, EBIT_CAPACITY);
    return;
  }
  const LoopLayout L = loop_layout(DEDUP, cap, ucap, a.hash_slots, a.sort_n, LEAN ? 0 : NT);
  uint32_t* win = reinterpret_cast<uint32_t*>(smem + L.off_win);
  uint32_t* uniq = reinterpret_cast<uint32_t*>(smem + L.off_uniq);
  uint16_t* map = reinterpret_cast<uint16_t*>(smem + L.off_map);
  float* esh = reinterpret_cast<float*>(smem + L.off_even);
  float* psh = esh + 3 * ucap;
  uint32_t* misc = reinterpret_cast<uint32_t*>(smem + L.off_misc);
  BatchSmem B;
  B.map = map;
  B.uniq = uniq;
  B.vsh = nullptr;
  if (DEDUP == DEDUP_SORT) {
    B.keys = reinterpret_cast<unsigned long long*>(smem + L.off_table);
  } else {
    B.table = reinterpret_cast<uint32_t*>(smem + L.off_table);
    B.dense = reinterpret_cast<uint16_t*>(smem + L.off_dense);
  }
  B.ucount = misc;
  B.wsum = misc + 8;
  for (uint32_t i = tid; i < n; i += NT) win[i] = __ldg(la.idx + 3 * t0 + i);
  if (DEDUP != DEDUP_SORT)
    for (uint32_t s = tid; s < a.hash_slots; s += NT) B.table[s] = kEmpty;
  if (tid == 0) *B.ucount = 0;
  __syncthreads();
  dedup<DEDUP, true>(a, B, win, n, tid, NT, BlockSync(),
                    LoopEven<!LEAN && DEDUP != DEDUP_SORT, kVec>{la, uniq, esh, psh, ucap});
  __syncthreads();
  const uint32_t U = min(*B.ucount, ucap);
  // the keys, the ids and the window have been read for the last time
  float4* stage = reinterpret_cast<float4*>(smem) + (tid >> 5) * 9 * kLoopStage;
  const uint32_t lane = lane_id();
  for (uint32_t jw = tid - lane; jw < t1 - t0; jw += NT) {  // warp-uniform
    const uint32_t j = min(jw + lane, t1 - t0 - 1);  // past the batch: computed and not written
    float3 E[3], P[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      uint32_t r = map[3 * j + k];
      if (DEDUP != DEDUP_SORT) r = B.dense[r];
      r = r < U ? r : 0u;  // only after a flagged capacity or index-range error
      E[k] = make_float3(esh[3 * r], esh[3 * r + 1], esh[3 * r + 2]);
      P[k] = make_float3(psh[3 * r], psh[3 * r + 1], psh[3 * r + 2]);
    }
    loop_emit<!LEAN, kVec, LEAN>(la, t0 + jw, min(32u, t1 - t0 - jw), E, P, stage, lane);
  }
  if (tid == 0) {
    atomicAdd(la.counters + 0, (unsigned long long)U);
    atomicAdd(la.counters + 1, 1ull);
  }
}

// Algorithm 1 per warp: per-warp shared memory held[32] | ids[S] | map[S].
__host__ __device__ inline uint32_t loop_warp_bytes(uint32_t S) { return 128 + ((S + 3) & ~3u) * 4 + ((S + 15) & ~15u); }

__global__ void __launch_bounds__(256) loop_warp_kernel(const __grid_constant__ LoopArgs la, uint32_t S,
                                                        uint32_t nbatches) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint32_t lane = lane_id(), warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  unsigned char* wp = smem + warp * loop_warp_bytes(S);
  uint32_t* held = reinterpret_cast<uint32_t*>(wp);
  uint32_t* widx = held + 32;
  unsigned char* map = reinterpret_cast<unsigned char*>(widx + ((S + 3) & ~3u));
  unsigned long long inv = 0, nb = 0;
  for (uint32_t b = blockIdx.x * wpb + warp; b < nbatches; b += gridDim.x * wpb) {
    const uint32_t B0 = b * S, n = min(B0 + S, 3 * la.num_tris) - B0;
    for (uint32_t i = lane; i < n; i += 32) {
      const uint32_t id = __ldg(la.idx + B0 + i);
      widx[i] = id < la.num_verts ? id : kInvalidId;
    }
    __syncwarp();
    for (uint32_t c = 0; c < n;) {
      uint32_t fill, done;
      warp_vote_round(widx, n, c, held, map, lane, fill, done);
      const uint32_t tris = done / 3;
      if (tris == 0) {  // cannot happen: a round's first chunk always places its lanes
        if (lane == 0) atomicOr(la.counters + 2, (unsigned long long)EBIT_CAPACITY);
        break;
      }
      float3 E = make_float3(0.f, 0.f, 0.f), P = E;
      if (lane < fill) {
        P = loop_pos<true>(la, held[lane]);
        E = loop_even<false, true>(la, held[lane], P);
      }
      inv += fill;
      const uint32_t tfirst = (B0 + c) / 3;
      for (uint32_t p = 0; p < tris; p += 32) {
        const uint32_t j = p + lane;
        const bool live = j < tris;
        float3 Ec[3], Pc[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const uint32_t sl = live ? map[3 * j + k] : 0u;
          Ec[k] = make_float3(__shfl_sync(kFull, E.x, sl), __shfl_sync(kFull, E.y, sl), __shfl_sync(kFull, E.z, sl));
          Pc[k] = make_float3(__shfl_sync(kFull, P.x, sl), __shfl_sync(kFull, P.y, sl), __shfl_sync(kFull, P.z, sl));
        }
        loop_emit<false, true, false>(la, tfirst + p, min(32u, tris - p), Ec, Pc, nullptr, lane);
      }
      __syncwarp();  // the next round overwrites held/map
      c += 3 * tris;
    }
    ++nb;
  }
  if (lane == 0 && nb) {
    atomicAdd(la.counters + 0, inv);
    atomicAdd(la.counters + 1, nb);
  }
}

}  // namespace gp

using namespace gp;

namespace {
template <bool LEAN>
const void* loop_fn(int dedup) {
  switch (dedup) {
    case DEDUP_SORT: return reinterpret_cast<const void*>(&loop_batched_kernel<DEDUP_SORT, LEAN>);
    case DEDUP_HASH: return reinterpret_cast<const void*>(&loop_batched_kernel<DEDUP_HASH, LEAN>);
    default: return reinterpret_cast<const void*>(&loop_batched_kernel<DEDUP_PHASH, LEAN>);
  }
}

uint32_t loop_pow2(uint32_t x) {
  uint32_t p = 1;
  while (p < x) p <<= 1;
  return p;
}
}  // namespace

extern "C" gp_status gp_loop_subdivide(const gp_loop_desc* d) {
  // Section 5.2; see include/gp.h
  if (!d || !d->d_counters) return GP_ERR_INVALID;
  const int32_t v = d->variant;
  if (v != GP_NAIVE && v != GP_WARP && v != GP_SORT && v != GP_HASH && v != GP_PHASH) return GP_ERR_INVALID;
  if (d->num_indices % 3) return GP_ERR_INVALID;
  const uint32_t T = (uint32_t)(d->num_indices / 3);
  if (d->num_indices >= 0xFFFFFFF0ull) return GP_ERR_INVALID;
  if (T && (!d->d_indices || !d->d_vertices || !d->d_ring_offsets || !d->d_vertex_flags || !d->d_opposite ||
            !d->d_out))
    return GP_ERR_INVALID;
  if (reinterpret_cast<uintptr_t>(d->d_out) % 16 || d->stride_bytes < 12 || d->stride_bytes % 4)
    return GP_ERR_INVALID;
  const bool dyn = d->d_starts != nullptr;
  if ((v == GP_NAIVE || v == GP_WARP) && dyn) return GP_ERR_INVALID;
  if (dyn && (!d->d_num_batches || d->max_batch_indices == 0 || d->max_batch_indices % 3 || d->max_batches == 0))
    return GP_ERR_INVALID;
  const uint32_t S = dyn ? d->max_batch_indices : (d->batch_indices ? d->batch_indices : (v == GP_WARP ? 96 : 768));
  if (S % 3 || S > 4095 || (v == GP_WARP && S > kWarpMaxBatch)) return GP_ERR_INVALID;
  const uint32_t threads = d->threads ? d->threads : (v == GP_WARP ? 64 : 256);
  if (v == GP_WARP && (threads % 32 || threads > 256)) return GP_ERR_INVALID;
  if (v != GP_NAIVE && v != GP_WARP && (threads % 32 || (threads & (threads - 1)) || threads > 512))
    return GP_ERR_INVALID;
  if (T == 0) return GP_OK;
  cudaStream_t s = static_cast<cudaStream_t>(d->stream);
  LoopArgs la{};
  la.idx = d->d_indices;
  la.num_tris = T;
  la.verts = static_cast<const unsigned char*>(d->d_vertices);
  la.stride = d->stride_bytes;
  la.num_verts = (uint32_t)d->num_vertices;
  la.vec16 = reinterpret_cast<uintptr_t>(d->d_vertices) % 16 == 0 && d->stride_bytes % 16 == 0 ? 1u : 0u;
  la.ring_off = d->d_ring_offsets;
  la.ring = d->d_ring;
  la.ring_count = (uint32_t)std::min<uint64_t>(d->ring_count, 0xFFFFFFFFu);
  la.ring16 = reinterpret_cast<uintptr_t>(d->d_ring) % 16 == 0 ? 1u : 0u;
  la.vflags = d->d_vertex_flags;
  la.opp = d->d_opposite;
  la.out = d->d_out;
  la.counters = d->d_counters;
  if (v == GP_NAIVE) {
    loop_naive_kernel<<<(T + 255) / 256, 256, 0, s>>>(la);
    return cudaGetLastError() == cudaSuccess ? GP_OK : GP_ERR_CUDA;
  }
  if (v == GP_WARP) {
    const uint32_t nbatches = (3 * T + S - 1) / S, wpb = threads / 32;
    const size_t smem = (size_t)wpb * loop_warp_bytes(S);
    loop_warp_kernel<<<(nbatches + wpb - 1) / wpb, threads, smem, s>>>(la, S, nbatches);
    return cudaGetLastError() == cudaSuccess ? GP_OK : GP_ERR_CUDA;
  }
  DrawArgs a{};
  const int dedup = v == GP_SORT ? DEDUP_SORT : (v == GP_HASH ? DEDUP_HASH : DEDUP_PHASH);
  const uint32_t ucap = dyn ? std::min(d->max_unique ? d->max_unique : S, S) : S;
  a.num_verts = la.num_verts;
  a.ucap = ucap;
  a.max_batch_idx = S;
  a.hash_slots = std::max(loop_pow2(2 * ucap), loop_pow2(threads));
  uint32_t bits = 0;
  while ((1u << bits) < a.hash_slots) ++bits;
  a.hash_bits = bits;
  a.sort_n = loop_pow2(S);
  a.probe_k = 4;
  a.err = reinterpret_cast<uint32_t*>(d->d_counters + 2);
  uint32_t grid;
  if (dyn) {
    la.starts = d->d_starts;
    la.num_batches_dev = d->d_num_batches;
    grid = d->max_batches;  // blocks past the device count return at once
  } else {
    la.static_tris = S / 3;
    la.num_batches = (T + la.static_tris - 1) / la.static_tris;
    grid = la.num_batches;
  }
  const bool lean = threads >= 2 * (S / 3);  // see loop_batched_kernel
  const size_t smem = loop_layout(dedup, S, ucap, a.hash_slots, a.sort_n, lean ? 0 : threads).total;
  const void* fn = lean ? loop_fn<true>(dedup) : loop_fn<false>(dedup);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return GP_ERR_UNSUPPORTED;
  void* args[] = {&la, &a};
  return cudaLaunchKernel(fn, dim3(grid), dim3(threads), args, smem, s) == cudaSuccess ? GP_OK : GP_ERR_CUDA;
}

// Dynamic batching preprocessing (Section 3.4): scan the triangles front to
// back, counting the unique indices of the open batch; close it before the
// triangle that would make it exceed N unique indices or the triangle cap.
//
// The scan is sequential by nature.  To use the whole GPU the triangle list
// is cut into segments of segment_tris triangles, a batch is also closed at
// every segment boundary, and each thread block scans one segment, a batch at
// a time, each thread holding IPT consecutive indices of the batch's largest
// window (max_tris triangles):
//   * every thread inserts its ids into the block's hash table (all CAS in
//     flight together) and counts the ones that were new; one block-wide sum
//     gives the window's unique ids.  When they are at most max_unique (the
//     rule on meshes with locality) the batch is the whole window: one
//     barrier per batch;
//   * otherwise the window is cut: the smallest position of each id
//     (atomicMin) tells where it is new, a block-wide scan counts the ids that
//     are new up to every position, and the triangle of the first position
//     whose count exceeds max_unique starts the next batch.  After a cut, the
//     next batch first inserts only about as many triangles as the last one
//     took, and the rest of its window only if they all fit.
// Two tables alternate, the one just used being emptied behind the sum's
// barrier; the indices run ahead of the scan into a ring of panels in shared
// memory (cp.async), two windows or more ahead, so no batch waits for a global
// load.
// A batch is a chain of one barrier and a few shared-memory round trips: that
// chain (13 batches a segment at the default limits) bounds a small mesh, the
// issue of its instructions a large one.  The whole partition of 500k triangles
// at the default limits takes 26 us, of 7.2M 90 us; one warp per segment, 32
// triangles a step with a scan each, took 166 and 207 us.
// A second kernel turns the per-segment lists into one array of batch
// starts (prefix of the segment counts, then a copy).
#include <algorithm>

#include "gp_device.cuh"

namespace gp {

__device__ __forceinline__ uint32_t part_hash(uint32_t id, uint32_t bits) {
  return bits ? (id * 2654435769u) >> (32 - bits) : 0u;
}

// 16 bytes of which only the first 'bytes' are read (the rest: zeros).
__device__ __forceinline__ void cp_async16_upto(void* dst_smem, const void* src_gmem, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst_smem)), "l"(src_gmem), "r"(bytes)
               : "memory");
}

constexpr uint32_t kPanels = 16;    // a window is at most four of them
constexpr uint32_t kPartMisc = 128;  // words: sums of alternate rounds (32 each), scan (32), cut

// Shared memory: two hash tables, the smallest positions (a word per slot
// each), misc, the ring of kPanels panels of 2^panel_bits triangles.
template <int IPT>
__global__ void __launch_bounds__(1024) partition_segments_kernel(const __grid_constant__ PartitionArgs p) {
  extern __shared__ __align__(16) uint32_t smem_w[];
  const uint32_t tid = threadIdx.x, NT = blockDim.x, lane = lane_id(), warp = tid >> 5, nw = NT >> 5;
  const uint32_t slots = p.table_slots, mask = slots - 1;
  uint32_t* pos = smem_w + 2 * slots;
  uint32_t* misc = smem_w + 3 * slots;  // [0..31], [32..63]: sums of alternate rounds; [64..95]: scan; [96], [97]: cut
  uint32_t* ring = misc + kPartMisc;
  const uint32_t pbits = p.panel_bits, ring_mask = (kPanels << pbits) - 1, ring_words = 3 * (kPanels << pbits);
  const uint32_t num_idx = 3 * p.num_tris;
  // panel k: the triangles from k << pbits, at that triangle modulo the ring; one group each
  auto fetch_panel = [&](uint32_t k) {
    const uint32_t c = 4 * tid;  // at most 4 tid < 3 << pbits words of a panel (NT >= its 16-byte words)
    if (c < 3u << pbits) {
      const uint64_t w = 3ull * (k << pbits) + c;
      if (w < num_idx)
        cp_async16_upto(ring + 3 * ((k << pbits) & ring_mask) + c, p.idx + w, 4 * min(4u, num_idx - (uint32_t)w));
    }
    cp_async_commit();
  };
  const uint32_t seg = blockIdx.x;
  const uint32_t seg_begin = seg * p.segment_tris;
  const uint32_t seg_end = min(seg_begin + p.segment_tris, p.num_tris);
  uint32_t panel = seg_begin >> pbits;  // of the scan's position; panels up to panel + 15 are on their way
  for (uint32_t k = 0; k < kPanels; ++k) fetch_panel(panel + k);
  for (uint32_t s = 4 * tid; s < 3 * slots; s += 4 * NT)
    *reinterpret_cast<uint4*>(smem_w + s) = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
  uint32_t* out = p.seg_starts + (size_t)seg * p.seg_cap;
  const uint32_t p0 = IPT * tid;  // this thread's first position in a window
  uint32_t count = 0, t = seg_begin, par = 0, rnd = 0, guess = p.max_tris;
  cp_async_wait<7>();
  __syncthreads();
  while (t < seg_end) {
    if (count >= p.seg_cap) {  // cannot happen: seg_cap bounds the batches of a segment
      if (tid == 0) atomicOr(p.err, EBIT_CAPACITY);
      break;
    }
    if (tid == 0) out[count] = t;
    ++count;
    const uint32_t wt = min(p.max_tris, seg_end - t);
    uint32_t* keys = smem_w + par * slots;
    uint32_t x[IPT], h[IPT];
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
      uint32_t w = 3 * (t & ring_mask) + p0 + q;  // past the window: read and not used
      w -= w >= ring_words ? ring_words : 0u;
      const uint32_t v = ring[w];
      x[q] = v == kEmpty ? kInvalidId : v;
      h[q] = part_hash(x[q], p.table_bits);
    }
    cp_async_wait<7>();  // behind the next barrier, panels up to panel + 8 have landed: this window and the next
    uint32_t c0 = 0, c1 = 3 * min(guess, wt), nu = 0, cut = wt;
    bool ordered = guess < wt;  // after a cut, expect one: look for it at once
    for (;;) {  // insert positions [c0, c1)
      uint32_t prev[IPT], fresh = 0;
      bool probing = false;
      const bool live = 32 * IPT * warp < c1;  // the others have nothing to insert
      if (live) {
#pragma unroll
        for (int q = 0; q < IPT; ++q)
          prev[q] = p0 + q >= c0 && p0 + q < c1 ? atomicCAS(&keys[h[q]], kEmpty, x[q]) : x[q];
#pragma unroll
        for (int q = 0; q < IPT; ++q) {
          fresh += prev[q] == kEmpty;
          probing |= prev[q] != kEmpty && prev[q] != x[q];
        }
        // collisions advance one slot per round together
        for (uint32_t probes = 0; probing; ++probes) {
          if (probes > slots) {  // cannot happen: the table has room for a whole window
            atomicOr(p.err, EBIT_CAPACITY);
            break;
          }
          bool again[IPT];
#pragma unroll
          for (int q = 0; q < IPT; ++q) {
            again[q] = prev[q] != kEmpty && prev[q] != x[q];
            if (again[q]) {
              h[q] = (h[q] + 1) & mask;
              prev[q] = atomicCAS(&keys[h[q]], kEmpty, x[q]);
            }
          }
          probing = false;
#pragma unroll
          for (int q = 0; q < IPT; ++q)
            if (again[q]) {
              fresh += prev[q] == kEmpty;
              probing |= prev[q] != kEmpty && prev[q] != x[q];
            }
        }
      }
      bool over = ordered;
      if (!ordered) {  // the unique ids so far
        const uint32_t wsum = __reduce_add_sync(kFull, fresh);
        if (lane == 0) misc[32 * rnd + warp] = wsum;
        __syncthreads();
        nu += __reduce_add_sync(kFull, lane < nw ? misc[32 * rnd + lane] : 0u);
        rnd ^= 1u;
        over = nu > p.max_unique;
      }
      if (over) {  // uniform: find where the positions inserted so far end the batch, if they do
        uint32_t* cutv = misc + 96 + par;
        if (tid == 0) *cutv = 3 * wt;
#pragma unroll
        for (int q = 0; q < IPT; ++q)
          if (live && p0 + q < c1) atomicMin(&pos[h[q]], p0 + q);
        __syncthreads();
        uint32_t upto[IPT], c = 0;  // ids that are new at this thread's positions, running
#pragma unroll
        for (int q = 0; q < IPT; ++q) {
          if (p0 + q < c1) c += pos[h[q]] == p0 + q;
          upto[q] = c;
        }
        const uint32_t inc = warp_inclusive_scan(c);
        if (lane == 31) misc[64 + warp] = inc;
        __syncthreads();
        const uint32_t ws = lane < nw ? misc[64 + lane] : 0u;
        const uint32_t before = inc - c + __reduce_add_sync(kFull, lane < warp ? ws : 0u);
        nu = __reduce_add_sync(kFull, ws);
#pragma unroll
        for (int q = 0; q < IPT; ++q)
          if (p0 + q < c1) pos[h[q]] = kEmpty;  // every position was read before the last barrier
        uint32_t first = 3 * wt;  // this thread's first position past the limit
#pragma unroll
        for (int q = IPT - 1; q >= 0; --q)
          if (p0 + q < c1 && before + upto[q] > p.max_unique) first = p0 + q;
        first = __reduce_min_sync(kFull, first);
        if (lane == 0 && first < 3 * wt) atomicMin(cutv, first);
        __syncthreads();
        if (nu > p.max_unique) {
          cut = max(1u, *cutv / 3);
          break;
        }
      }
      if (c1 == 3 * wt) break;
      c0 = c1;
      c1 = 3 * wt;
      ordered = false;
    }
    guess = cut < wt ? cut + cut / 8 + 8 : p.max_tris;
    // empty the table (every thread has left it); the next batch uses the other
    for (uint32_t s = 4 * tid; s < slots; s += 4 * NT)
      *reinterpret_cast<uint4*>(keys + s) = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
    par ^= 1u;
    t += cut;
    // on by at most four panels (cut <= max_tris <= 4 panels): every thread has read the ones left
    for (const uint32_t now = t >> pbits; panel < now;) fetch_panel(++panel + kPanels - 1);
  }
  cp_async_wait<0>();
  if (tid == 0) p.seg_counts[seg] = count;
}

// Each block adds up the counts of the segments before its own, then its
// warps copy one segment's starts each into the final array;
// starts[total] = T.
constexpr uint32_t kGatherSegs = 8;

__global__ void __launch_bounds__(256) partition_gather_kernel(const __grid_constant__ PartitionArgs p) {
  __shared__ uint32_t sums[8];
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
  const uint32_t first = blockIdx.x * kGatherSegs;
  auto count_of = [&](uint32_t s) { return s < p.num_segments ? min(p.seg_counts[s], p.seg_cap) : 0u; };
  uint32_t c = 0;
  for (uint32_t s = tid; s < first; s += 256) c += count_of(s);
  c = __reduce_add_sync(kFull, c);
  if (lane == 0) sums[warp] = c;
  __syncthreads();
  uint32_t o = __reduce_add_sync(kFull, lane < 8 ? sums[lane] : 0u);
  const uint32_t own = lane < kGatherSegs ? count_of(first + lane) : 0u;  // the block's segments
  o += __reduce_add_sync(kFull, lane < warp ? own : 0u);
  const uint32_t s = first + warp;
  if (s < p.num_segments) {
    const uint32_t n = __shfl_sync(kFull, own, warp);
    const uint32_t* src = p.seg_starts + (size_t)s * p.seg_cap;
    for (uint32_t k = lane; k < n; k += 32) p.starts[o + k] = src[k];
    o += n;
  }
  // the last segment's warp (or, of an empty buffer, the only block's first)
  if (lane == 0 && (s + 1 == p.num_segments || (p.num_segments == 0 && warp == 0))) {
    p.starts[o] = p.num_tris;
    *p.num_batches = o;
  }
}

cudaError_t launch_partition(const PartitionArgs& args, cudaStream_t s) {
  PartitionArgs p = args;
  if (p.num_segments) {
    // a block holds the largest window: one, two or four indices per thread (3 max_tris <= 4095)
    // -- one shortens the chain of a small window (64 triangles: 57 us against 80 at 500k triangles), four issue
    // the fewest instructions on a large one (341: 88 us against 139 at 7.2M; at 500k equal)
    const uint32_t ipt = p.max_tris <= 128 ? 1u : (p.max_tris <= 256 ? 2u : 4u);
    p.panel_bits = 6;
    while ((4u << p.panel_bits) < p.max_tris) ++p.panel_bits;
    // ... and a panel's 16-byte words
    const uint32_t threads = std::max((3 * p.max_tris + ipt - 1) / ipt, (3u << p.panel_bits) / 4) + 31 & ~31u;
    // slots for a window without a repeated id: at most three quarters full
    p.table_slots = 32;
    p.table_bits = 5;
    while (p.table_slots < 4 * p.max_tris) {
      p.table_slots <<= 1;
      ++p.table_bits;
    }
    const size_t smem = (3 * (size_t)p.table_slots + kPartMisc + 3 * ((size_t)kPanels << p.panel_bits)) * 4;
    const void* fn = ipt == 1   ? reinterpret_cast<const void*>(&partition_segments_kernel<1>)
                     : ipt == 2 ? reinterpret_cast<const void*>(&partition_segments_kernel<2>)
                                : reinterpret_cast<const void*>(&partition_segments_kernel<4>);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (ipt == 1) partition_segments_kernel<1><<<p.num_segments, threads, smem, s>>>(p);
    else if (ipt == 2) partition_segments_kernel<2><<<p.num_segments, threads, smem, s>>>(p);
    else partition_segments_kernel<4><<<p.num_segments, threads, smem, s>>>(p);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  partition_gather_kernel<<<std::max(1u, (p.num_segments + kGatherSegs - 1) / kGatherSegs), 256, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace gp

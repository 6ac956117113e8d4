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
  const uint32_t seg = blockIdx.x;
  const uint32_t seg_begin = seg * p.segment_tris;
  const uint32_t seg_end = min(seg_begin + p.segment_tris, p.num_tris);
  const uint32_t num_idx = 3 * p.num_tris;
  // panel k: the triangles from k << pbits, at that triangle modulo the ring; one group each (empty past the segment)
  auto fetch_panel = [&](uint32_t k) {
    const uint32_t c = 4 * tid;  // at most 4 tid < 3 << pbits words of a panel (NT >= its 16-byte words)
    if (c < 3u << pbits) {
      const uint64_t w = 3ull * (k << pbits) + c;
      if (w < 3 * seg_end)
        cp_async16_upto(ring + 3 * ((k << pbits) & ring_mask) + c, p.idx + w, 4 * min(4u, num_idx - (uint32_t)w));
    }
    cp_async_commit();
  };
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

// A warp per segment, where there are segments for several waves of blocks
// (partition_by_warps): slower through one segment, but with less work.  The
// window is read into the warp's shared memory; 32 triangles are examined per
// step, one per lane, their ids' smallest positions in the warp's hash table telling
// which are new, and a scan of their number tells where the batch ends.
struct PartLayout {
  uint32_t keys_off, pos_off, per_warp;
};

__host__ __device__ inline PartLayout part_layout(uint32_t max_tris, uint32_t slots) {
  PartLayout L;
  L.keys_off = ((3 * max_tris + 3) & ~3u) * 4;
  L.pos_off = L.keys_off + slots * 4;
  L.per_warp = L.pos_off + slots * 4;
  return L;
}

__global__ void __launch_bounds__(256) partition_warps_kernel(const __grid_constant__ PartitionArgs p) {
  extern __shared__ __align__(16) unsigned char smem[];
  const PartLayout L = part_layout(p.max_tris, p.table_slots);
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const uint32_t seg = blockIdx.x * (blockDim.x >> 5) + warp;
  if (seg >= p.num_segments) return;  // warp-uniform; no block barrier in this kernel
  unsigned char* wb = smem + warp * L.per_warp;
  uint32_t* win = reinterpret_cast<uint32_t*>(wb);
  uint32_t* keys = reinterpret_cast<uint32_t*>(wb + L.keys_off);
  uint32_t* pos = reinterpret_cast<uint32_t*>(wb + L.pos_off);
  const uint32_t mask = p.table_slots - 1;

  const uint32_t seg_begin = seg * p.segment_tris;
  const uint32_t seg_end = min(seg_begin + p.segment_tris, p.num_tris);
  uint32_t* out = p.seg_starts + (size_t)seg * p.seg_cap;
  uint32_t count = 0;
  uint32_t t = seg_begin;
  while (t < seg_end) {
    if (count >= p.seg_cap) {  // cannot happen: seg_cap bounds the batches of a segment
      if (lane == 0) atomicOr(p.err, EBIT_CAPACITY);
      break;
    }
    if (lane == 0) out[count] = t;
    ++count;
    const uint32_t wt = min(p.max_tris, seg_end - t);
    const uint32_t nidx = 3 * wt;
    const uint32_t* src = p.idx + 3 * (size_t)t;
    for (uint32_t i = lane; i < nidx; i += 32) {
      const uint32_t x = __ldg(src + i);
      win[i] = x == kEmpty ? kInvalidId : x;
    }
    for (uint32_t s = lane; s < p.table_slots; s += 32) {
      keys[s] = kEmpty;
      pos[s] = 0xFFFFFFFFu;
    }
    __syncwarp();
    uint32_t nu = 0;    // unique ids of the batch so far
    uint32_t cut = wt;  // triangles the batch takes
    for (uint32_t c = 0; c < wt; c += 32) {
      const uint32_t j = c + lane;
      const bool valid = j < wt;
      // the triangle's three ids: insert them (three independent CAS, then
      // the rare collisions), record their positions (three independent
      // atomicMin), and count the ids whose smallest position is here
      uint32_t x[3], h[3], prev[3];
      if (valid) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          x[k] = win[3 * j + k];
          h[k] = part_hash(x[k], p.table_bits);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) prev[k] = atomicCAS(&keys[h[k]], kEmpty, x[k]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          for (uint32_t probes = 0; prev[k] != kEmpty && prev[k] != x[k]; ++probes) {
            if (probes > p.table_slots) {  // cannot happen: the table has room
              atomicOr(p.err, EBIT_CAPACITY);
              break;
            }
            h[k] = (h[k] + 1) & mask;
            prev[k] = atomicCAS(&keys[h[k]], kEmpty, x[k]);
          }
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) atomicMin(&pos[h[k]], 3 * j + k);
      }
      __syncwarp();
      uint32_t fresh = 0;
      if (valid) {
#pragma unroll
        for (int k = 0; k < 3; ++k) fresh += pos[h[k]] == 3 * j + k;
      }
      const uint32_t cum = warp_inclusive_scan(fresh);
      const uint32_t over = __ballot_sync(kFull, valid && nu + cum > p.max_unique);
      if (over) {
        cut = max(1u, c + (uint32_t)(__ffs(over) - 1));
        break;
      }
      nu += __shfl_sync(kFull, cum, 31);
      __syncwarp();
    }
    t += cut;
    __syncwarp();
  }
  if (lane == 0) p.seg_counts[seg] = count;
}

// Many segments: how many batches lie before every kOffsetSegs-th segment, one
// block going over the counts once.  offsets[k]: before segment k kOffsetSegs.
constexpr uint32_t kOffsetSegs = 4;  // counts per thread and step

__global__ void __launch_bounds__(1024) partition_offsets_kernel(const __grid_constant__ PartitionArgs p,
                                                                 uint32_t* offsets) {
  __shared__ uint32_t warp_sums[33];
  uint32_t carry = 0;
  for (uint32_t base = 0; base < p.num_segments; base += kOffsetSegs * blockDim.x) {
    const uint32_t first = base + kOffsetSegs * threadIdx.x;
    uint32_t c = 0;
#pragma unroll
    for (uint32_t q = 0; q < kOffsetSegs; ++q)
      if (first + q < p.num_segments) c += min(p.seg_counts[first + q], p.seg_cap);
    uint32_t total;
    const uint32_t before = block_exclusive_scan(c, warp_sums, &total);
    if (first < p.num_segments) offsets[first / kOffsetSegs] = carry + before;
    carry += total;
    __syncthreads();
  }
}

// Each block adds up the counts of the segments before its own (or has their
// sum, 'offsets'), then its warps copy one segment's starts each into the final
// array; starts[total] = T.
constexpr uint32_t kGatherSegs = 8;

__global__ void __launch_bounds__(256) partition_gather_kernel(const __grid_constant__ PartitionArgs p,
                                                               const uint32_t* offsets) {
  __shared__ uint32_t sums[8];
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
  const uint32_t first = blockIdx.x * kGatherSegs;
  auto count_of = [&](uint32_t s) { return s < p.num_segments ? min(p.seg_counts[s], p.seg_cap) : 0u; };
  uint32_t o;
  if (offsets) {
    o = offsets[first / kOffsetSegs];
  } else {
    uint32_t c = 0;
    for (uint32_t s = tid; s < first; s += 256) c += count_of(s);
    c = __reduce_add_sync(kFull, c);
    if (lane == 0) sums[warp] = c;
    __syncthreads();
    o = __reduce_add_sync(kFull, lane < 8 ? sums[lane] : 0u);
  }
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

// Segments above which the batches before each are counted once, by a kernel of its own: below, adding up
// the counts in every block costs less than another launch.
constexpr uint32_t kManySegments = 16384;

static uint32_t slots_at_least(uint32_t n, PartitionArgs& p) {
  p.table_slots = 32;
  p.table_bits = 5;
  while (p.table_slots < n) {
    p.table_slots <<= 1;
    ++p.table_bits;
  }
  return p.table_slots;
}

// A block's launch shape for a largest window of p.max_tris (3 max_tris <= 4095): one, two or four indices per
// thread, and a panel's 16-byte words.  Sets the table and the panels; returns the threads.
static uint32_t block_shape(PartitionArgs& p, uint32_t ipt, size_t* smem) {
  p.panel_bits = 6;
  while ((4u << p.panel_bits) < p.max_tris) ++p.panel_bits;
  // a window without a repeated id fills at most five eighths (three quarters, as windows of a power of two did
  // with 4 slots a triangle, probe far: 3M triangles in random order, windows of 1,024: 556 us against 228)
  slots_at_least(24 * p.max_tris / 5, p);
  *smem = (3 * (size_t)p.table_slots + kPartMisc + 3 * ((size_t)kPanels << p.panel_bits)) * 4;
  return std::max((3 * p.max_tris + ipt - 1) / ipt, (3u << p.panel_bits) / 4) + 31 & ~31u;
}

static cudaError_t launch_warps(PartitionArgs& p, cudaStream_t s) {
  // a batch inserts at most one step's ids past its limit, and no more than its window's
  const uint32_t ids = std::min(p.max_unique + 96, 3 * p.max_tris);
  const size_t per_warp = part_layout(p.max_tris, slots_at_least(2 * ids, p)).per_warp;
  const uint32_t warps = (uint32_t)std::min<size_t>(4, 227u * 1024u / per_warp);
  const cudaError_t e = cudaFuncSetAttribute(partition_warps_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(warps * per_warp));
  if (e != cudaSuccess) return e;
  partition_warps_kernel<<<(p.num_segments + warps - 1) / warps, warps * 32, warps * per_warp, s>>>(p);
  return cudaGetLastError();
}

// Blocks or warps for the segments.  A block is faster through one segment, warps do less in all: once the blocks
// come in waves, what counts is the work.  Measured, us, warps first.
// Long segments: blocks, at the default limits for 500k triangles 167 and 26, 3M of them in random order 238 and 188,
// 7.2M 187 and 89 (2.9 waves); 1024 / 1365 on 7.2M 436 and 127.  But with many ids past the limit in a window
// (max_tris >= 4 max_unique) the batch is cut early and most of a block idles: 64 / 341 on 7.2M 247 and 301,
// 256 / 1365 on 3M in random order (4.8 waves) 404 and 455.
// Short segments, whose tables and panels are set up for a batch or two: warps from the first full wave on; segments
// of 256, 500k in random order 31 and 90, a torus 24 and 22; of 1,024, 64 / 64, 3M in random order 102 and 197, a
// grid 54 and 68.  But blocks for large windows that are seldom cut (max_tris <= 1.5 max_unique; segments of 1,024,
// 7.2M, 256 / 341: 157 and 103, 1024 / 1365 397 and 158) or never (3 max_tris <= max_unique; segments of 256, 3M in
// random order, 1024 / 341: 166 and 91).
// *ipt: one index per thread shortens the chain of a small window (64 triangles: 57 us against 80 at 500k triangles),
// four issue the fewest instructions (341: 88 us against 139 at 7.2M; 64: 132 against 144).
static bool partition_by_warps(PartitionArgs p, uint32_t* ipt) {
  constexpr float kSms = 152.f;
  *ipt = p.max_tris <= 128 ? 1u : (p.max_tris <= 256 ? 2u : 4u);
  size_t smem;
  const uint32_t threads = block_shape(p, *ipt, &smem);
  const uint32_t resident = std::min(2048u / threads, (uint32_t)(228u * 1024u / (smem + 1024u)));
  const float waves = (float)p.num_segments / (kSms * (float)resident);
  if (waves > 1.f) *ipt = 4u;
  if (p.segment_tris >= 2048) return waves >= 1.5f && p.max_tris >= 4 * p.max_unique;
  const bool never = 3 * p.max_tris <= p.max_unique, seldom = 2 * p.max_tris <= 3 * p.max_unique;
  if (p.max_tris >= 256 && (never || (seldom && p.segment_tris >= 1024))) return false;
  return waves >= 1.f;
}

static cudaError_t launch_blocks(PartitionArgs& p, uint32_t ipt, cudaStream_t s) {
  size_t smem;
  const uint32_t threads = block_shape(p, ipt, &smem);
  const void* fn = ipt == 1   ? reinterpret_cast<const void*>(&partition_segments_kernel<1>)
                   : ipt == 2 ? reinterpret_cast<const void*>(&partition_segments_kernel<2>)
                              : reinterpret_cast<const void*>(&partition_segments_kernel<4>);
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (ipt == 1) partition_segments_kernel<1><<<p.num_segments, threads, smem, s>>>(p);
  else if (ipt == 2) partition_segments_kernel<2><<<p.num_segments, threads, smem, s>>>(p);
  else partition_segments_kernel<4><<<p.num_segments, threads, smem, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_partition(const PartitionArgs& args, cudaStream_t s) {
  PartitionArgs p = args;
  p.max_tris = std::min(p.max_tris, p.segment_tris);  // a batch ends with its segment
  uint32_t* offsets = nullptr;
  if (p.num_segments) {
    uint32_t ipt;
    cudaError_t e = partition_by_warps(p, &ipt) ? launch_warps(p, s) : launch_blocks(p, ipt, s);
    if (e != cudaSuccess) return e;
    if (p.num_segments > kManySegments) {
      offsets = p.seg_counts + p.num_segments;  // as many words again lie there
      partition_offsets_kernel<<<1, 1024, 0, s>>>(p, offsets);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  partition_gather_kernel<<<std::max(1u, (p.num_segments + kGatherSegs - 1) / kGatherSegs), 256, 0, s>>>(p, offsets);
  return cudaGetLastError();
}

}  // namespace gp

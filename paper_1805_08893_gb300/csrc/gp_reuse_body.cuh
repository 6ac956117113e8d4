// One block's part of a vertex-reuse draw (sorting: Algorithm 2, hashing:
// Algorithm 3, parallel hashing: Section 3.4): the warp-specialised pipeline
// over the batches that a source hands out, shared by the single-draw kernel
// (gp_reuse.cu) and the frame kernel (gp_frame.cu).
//
// Its warps have two roles that run side by side, handing batches over
// through a two-deep ring of shared-memory slots guarded by mbarriers
// ("full": deduplicated, rows landed; "empty": assembled, slot free):
//
//   producer warps (five eighths of the block; sort: half, or two thirds of a
//     smaller block, reuse_block_threads) deduplicate
//     batch j into slot j mod 2: the index window (bulk-copied on an
//     mbarrier one batch ahead, its triangle range left beside it) is read
//     from the 16-byte boundary at or below the batch's first index, 4 words
//     per thread ("a group"); hash/phash -- each position's id is inserted
//     into the shared open-addressing table with atomicCAS (multiplicative
//     hash, linear probing; phash: at most probe_k probes alone, then 32
//     slots at a time with the whole warp), and the thread whose CAS stored
//     an id takes the next unique rank from the slot's counter (one
//     atomicAdd per warp step), records slot -> rank and rank -> id and
//     starts the cp.async copy of the vertex row into the slot; sort --
//     bitonic sort of (id, position) keys, tail flags, prefix sum
//     (gp_batch_body.cuh), each warp copying the rows of the ranks it
//     created.  Each group's 4 slots (hash) or ranks (sort) go to the map as
//     u16 x 4.  The "full" mbarrier completes when every producer thread has
//     arrived and every row copy has landed.
//   consumer warps (the rest) take batch j from its slot: each unique
//     vertex is shaded once, in place in its row; then every warp assembles
//     its groups (4 corners' shaded rows per lane) through a per-warp staging
//     area (a transpose): with 7 floats per corner a span that lies inside
//     the batch leaves in one bulk (TMA) store per warp, otherwise through
//     coalesced 16-byte streaming stores -- only the float4 at the batch's
//     two ends that the neighbouring batch shares are written float by
//     float -- and arrives on the slot's "empty" mbarrier.
//
// Deduplication (shared-memory atomics) and shading/assembly (shared-memory
// reads, FP32, stores) thus overlap across warps instead of alternating
// between block barriers; each role synchronises only its own warps (named
// barriers 1 and 2).  Every wait is bounded; a wait that gives up sets
// EBIT_TIMEOUT and stops the block.
#pragma once

#include "gp_batch_body.cuh"

namespace gp {

constexpr uint32_t kNoBatch = 0xFFFFFFFFu;  // a ring slot that ends the block's work
constexpr uint32_t kBarProducers = 1;  // named barrier of the producer warps
constexpr uint32_t kBarConsumers = 2;  // named barrier of the consumer warps

struct ReuseLayout {
  uint32_t off_misc, groups, win_words, off_win, off_scratch, map_elems, uniq_words, rb, off_ring,
      ring_map, ring_dense, ring_uniq, ring_rows, ring_bytes, off_stage, off_pal, total;
};

__host__ __device__ inline uint32_t reuse_align16(uint32_t x) { return (x + 15u) & ~15u; }

// Producer warps of a block of NT threads (at least 64): hash/phash five
// eighths, rounded down (5 of 8 warps) -- deduplication is the longer chain
// of dependent shared-memory round trips; sort half of its threads_per_group: of
// a block of three quarters of them two thirds (4 of 6), of a whole one half (4 of
// 8; see reuse_block_threads).  The rest are consumers.
__host__ __device__ inline uint32_t reuse_producer_warps(uint32_t NT, int dedup) {
  const uint32_t w = NT / 32, p = dedup != DEDUP_SORT ? (5 * w) / 8 : ((w & (w - 1)) == 0 ? w / 2 : (2 * w) / 3);
  return p < 1 ? 1 : (p >= w ? w - 1 : p);
}
// Groups (4 positions) a producer thread inserts per pass, all CAS in flight.
constexpr int kGroupsPerPass = 2;

// Shared-memory layout for NT threads, row_cap rows a slot (a.row_cap where batches
// may hold more vertices than rows, else a.ucap).  K: floats per output corner.  own_palette: with
// room for the skinning palette.
__host__ __device__ inline ReuseLayout reuse_layout(int dedup, int shader, const DrawArgs& a, uint32_t NT,
                                                    uint32_t row_cap, bool own_palette) {
  const uint32_t K = shader == 2 ? 8u : 7u;
  const uint32_t consumer_warps = NT / 32 - reuse_producer_warps(NT, dedup);
  ReuseLayout L;
  uint32_t o = 0;
  L.off_misc = o; o += 64 * 4;  // [0], [1]: unique counters of the two slots; [2]: abort; [4], [5]: each slot's
                                // batch; [6], [7]: the producers' next batch; [8..31]: sort scan; [32..35]: first
                                // and end triangle of the batch in each window buffer; [36..39]: of each slot's batch
  L.groups = (a.max_batch_idx + 6) / 4;  // pad (<= 3) + indices, in 4-word groups
  L.win_words = 4 * L.groups;
  L.off_win = o; o += 2 * L.win_words * 4;
  L.off_scratch = o;  // two hash tables (batches alternate), or the sort keys
  {
    const uint32_t table = dedup == DEDUP_SORT ? 0u : 2 * a.hash_slots * 4;
    const uint32_t keys = dedup == DEDUP_SORT ? a.sort_n * (a.sort_pos_bits ? 4u : 8u) : 0u;
    o += reuse_align16(table > keys ? table : keys);
  }
  L.map_elems = 4 * L.groups;
  L.uniq_words = (a.ucap + 3) & ~3u;
  L.rb = shader == 1 ? 64u : 32u;
  L.off_ring = o;
  L.ring_map = 0;
  L.ring_dense = reuse_align16(L.map_elems * 2);
  L.ring_uniq = L.ring_dense + reuse_align16(dedup == DEDUP_SORT ? 0u : a.hash_slots * 2);
  L.ring_rows = L.ring_uniq + L.uniq_words * 4;  // uniq_words is a multiple of 4
  L.ring_bytes = L.ring_rows + row_cap * L.rb;    // rows are 32 or 64 bytes
  o += 2 * L.ring_bytes;
  L.off_stage = o; o += consumer_warps * 32 * K * 16;
  L.off_pal = o; o += shader == 1 && own_palette ? 768 * 4 : 0;
  L.total = o;
  return L;
}

// Float4 slot (within a slot's rows) of half h of the shaded vertex r, shaded
// in place over its raw row: the halves are placed so that 8 consecutive
// ranks' same halves fall into 8 different bank groups.
template <int SH>
__device__ __forceinline__ uint32_t row_slot(uint32_t r, uint32_t h) {
  return ShaderTraits<SH>::kSkin ? 4u * r + h + 2u * ((r >> 1) & 1u) : 2u * r + (h ^ ((r >> 2) & 1u));
}

// Per-warp staging: lane l writes its K float4 (4 corners) at put(l, j); the
// warp then reads float4 q = 32 j + lane of its span at get(q).  Both sides
// are free of bank conflicts (K = 7: odd stride; K = 8: xor swizzle).
template <int K>
__device__ __forceinline__ uint32_t stage_put(uint32_t lane, uint32_t j) {
  return K == 8 ? lane * 8u + (j ^ (lane & 7u)) : lane * (uint32_t)K + j;
}
template <int K>
__device__ __forceinline__ uint32_t stage_get(uint32_t q) {
  if (K == 8) {
    const uint32_t o = q >> 3, e = q & 7u;
    return o * 8u + (e ^ (o & 7u));
  }
  return q;
}

__device__ __forceinline__ void st_stream4(float* p, const float4& v) {
  asm volatile("st.global.cs.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
}

__device__ __forceinline__ void named_sync(uint32_t id, uint32_t nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Bounded wait on an mbarrier phase that also gives up once another thread
// has stopped the block (*abort != 0).  The waiting thread sleeps in steps
// of at most 50 us (waking as soon as the phase completes), so a waiting
// warp takes no issue slots from the other role; after 2^14 steps (at most
// ~0.8 s) it sets EBIT_TIMEOUT and *abort and gives up.
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile uint32_t* abort,
                                              uint32_t* err) {
  for (uint32_t it = 0; it < (1u << 14); ++it) {
    if (mbar_try_wait_sleep(bar, parity, 50000u)) return true;
    if (*abort) return false;
  }
  atomicOr(err, EBIT_TIMEOUT);
  *abort = 1u;
  return false;
}

// Copies the raw row of vertex id into row r of a slot (cp.async, 16 bytes
// at a time; ids out of range are not copied, their rank is shaded as zeros).
template <int SH>
__device__ __forceinline__ void copy_row(const DrawArgs& a, unsigned char* rows, uint32_t r, uint32_t id) {
  if (id < a.num_verts) {
    constexpr uint32_t RB = ShaderTraits<SH>::kSkin ? 64u : 32u;
#pragma unroll
    for (uint32_t c = 0; c < RB / 16; ++c) cp_async16(rows + r * RB + c * 16, a.verts + (size_t)id * a.stride + c * 16);
  }
}

// Sort: each warp copies the rows of the ranks it has just created.
template <int SH>
struct RowCopy {
  const DrawArgs& a;
  unsigned char* rows;
  const uint32_t* uniq;
  __device__ __forceinline__ void operator()(uint32_t rb, uint32_t re, uint32_t lane) const {
    re = min(re, a.row_cap);
    for (uint32_t r = rb + lane; r < re; r += 32) copy_row<SH>(a, rows, r, uniq[r]);
  }
};

// Starts a run's mbarriers: window[2], full[2], empty[2].
__device__ __forceinline__ void reuse_init_bars(uint64_t* bars, uint32_t NP, uint32_t NC) {
  mbar_init(&bars[0], 1);
  mbar_init(&bars[1], 1);
  mbar_init(&bars[2], NP);
  mbar_init(&bars[3], NP);
  mbar_init(&bars[4], NC);
  mbar_init(&bars[5], NC);
  fence_mbar_init();
}

// One block's batches.  Src hands them out by number:
//   first(), end()       the first batch; numbers from end() on mean "none";
//   args(j)              the buffers of the draw that the block's j-th batch
//                        belongs to ('cap' holds what all of them share: the
//                        capacities, the error word, the counters);
//   range(b, j, t0, t1)  its triangles;
//   number(b, j)         its number in that draw;
//   next(b, j, lane)     the batch after b, which becomes the (j + 1)-th.
//                        Called by thread 0, or with kWarpNext by all lanes of
//                        warp 0 (only lane 0's result counts);
//   uniforms(j, t, n)    called by the n consumer threads before they shade
//                        the j-th batch: makes u and palette those of its draw.
// SPILL: a batch may hold more unique vertices than it has rows (static
// batches, cap.row_cap < cap.ucap).  The caller has initialised the mbarriers
// and emptied the tables and misc[0..2], with no block barrier needed behind;
// first() < end().  After a stopped run misc[2] is not 0.
template <int DEDUP, int SH, bool SPILL, class Src>
__device__ __forceinline__ void reuse_batches(const DrawArgs& cap, const Uniforms& u, const float* palette,
                                              unsigned char* smem, const ReuseLayout& L, uint64_t* bars, uint32_t NT,
                                              Src& src) {
  constexpr int K = ShaderTraits<SH>::K;
  constexpr uint32_t RB = ShaderTraits<SH>::kSkin ? 64u : 32u;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t NPW = reuse_producer_warps(NT, DEDUP), NP = 32 * NPW, NC = NT - NP;
  const uint32_t nb = src.end();
  // bars: [0,1] window, [2,3] full, [4,5] empty
  uint32_t* misc = reinterpret_cast<uint32_t*>(smem + L.off_misc);
  volatile uint32_t* abort_flag = misc + 2;
  uint32_t* winbuf = reinterpret_cast<uint32_t*>(smem + L.off_win);
  uint32_t* table = reinterpret_cast<uint32_t*>(smem + L.off_scratch);
  auto ring = [&](uint32_t s) { return smem + L.off_ring + s * L.ring_bytes; };

  // Thread 0: bulk copy of the 16-byte-aligned superset of batch b's window,
  // clipped to the 16-byte-granular part of the buffer (the rest is loaded
  // by plain loads).  A window larger than the buffer is refused here and
  // flagged by the producers.  The batch's triangle range goes beside it in
  // shared memory, so that no producer waits on a global load for it.
  auto issue_window = [&](const DrawArgs& a, uint32_t t0, uint32_t t1, uint32_t buf, bool copy) {
    const uint32_t n4 = a.num_idx & ~3u;  // end of the 16-byte-granular part of the index buffer
    misc[32 + 2 * buf] = t0;
    misc[33 + 2 * buf] = t1;
    const uint32_t base = (3 * t0) & ~3u, end = min((3 * t1 + 3) & ~3u, n4);
    const uint32_t bytes = (end > base && end - base <= L.win_words) ? (end - base) * 4 : 0;
    if (!copy) {  // failure injection: bytes that never come
      mbar_arrive_expect_tx(&bars[buf], 16);
      return;
    }
    mbar_arrive_expect_tx(&bars[buf], bytes);
    if (bytes) bulk_load(winbuf + buf * L.win_words, a.idx + base, bytes, &bars[buf]);
  };
  if (tid == 0) {
    uint32_t t0, t1;
    src.range(src.first(), 0, t0, t1);
    issue_window(src.args(0), t0, t1, 0, !cap.test_stall);
  }
  __syncthreads();

  if (warp < NPW) {
    // ======================= producers =======================
    const uint32_t pw = warp;
    uint32_t wph = 0u, eph = 0u;  // bit s: parity of window[s] / empty[s]
    bool window_pending = tid == 0;  // thread 0: a window copy may be in flight into pending_buf
    uint32_t pending_buf = 0;
    uint32_t b = src.first();  // the batch this iteration deduplicates
    for (uint32_t j = 0;; ++j) {
      const uint32_t s = j & 1u;
      // (a block stopped by another thread is noticed in the waits below)
      if (b >= nb) {  // no batch left: hand the consumers a slot that says so
        if (j >= 2 && !wait_or_abort(&bars[4 + s], (eph >> s) & 1u, abort_flag, cap.err)) break;
        if (tid == 0) misc[4 + s] = kNoBatch;
        mbar_arrive(&bars[2 + s]);
        break;
      }
      decltype(auto) a = src.args(j);
      const uint32_t t0 = misc[32 + 2 * s], t1 = misc[33 + 2 * s];  // left by thread 0 with the window
      const uint32_t i0 = 3 * t0, n = 3 * (t1 - t0), base = i0 & ~3u, pad = i0 - base;
      const uint32_t ngroups = (pad + n + 3) >> 2;
      unsigned char* slot_p = ring(s);
      uint16_t* map = reinterpret_cast<uint16_t*>(slot_p + L.ring_map);
      uint16_t* dense = reinterpret_cast<uint16_t*>(slot_p + L.ring_dense);
      uint32_t* uniq = reinterpret_cast<uint32_t*>(slot_p + L.ring_uniq);
      unsigned char* rows = slot_p + L.ring_rows;
      uint32_t* counter = misc + s;
      uint32_t* win = winbuf + s * L.win_words;
      // the slot is free once the consumers have assembled the batch two back
      if (j >= 2) {
        if (!wait_or_abort(&bars[4 + s], (eph >> s) & 1u, abort_flag, cap.err)) break;
        eph ^= 1u << s;
      }
      if (!wait_or_abort(&bars[s], (wph >> s) & 1u, abort_flag, cap.err)) break;
      wph ^= 1u << s;
      window_pending = false;
      if (Src::kWarpNext ? warp == 0 : tid == 0) {
        // the next batch's window goes into the other buffer, which was read
        // before the last batch's barrier
        const uint32_t next = src.next(b, j, lane);
        if (!Src::kWarpNext || lane == 0) {
          misc[6 + (s ^ 1u)] = next;
          misc[4 + s] = b;
          misc[36 + 2 * s] = t0;  // the slot's batch, for the consumers
          misc[37 + 2 * s] = t1;
          if (next < nb) {
            uint32_t nt0, nt1;
            src.range(next, j + 1, nt0, nt1);
            issue_window(src.args(j + 1), nt0, nt1, s ^ 1u, true);
            window_pending = true;
            pending_buf = s ^ 1u;
          }
        }
      }
      if (n > a.max_batch_idx) {  // cannot happen with a consistent partition; uniform
        if (tid == 0) atomicOr(a.err, EBIT_CAPACITY);
        *abort_flag = 1u;
        break;
      }
      {  // indices past the 16-byte-granular part of the buffer (the buffer's last batch only)
        const uint32_t end = min((3 * t1 + 3) & ~3u, a.num_idx & ~3u);
        const uint32_t p0 = max(end, base);
        if (p0 < i0 + n) {  // uniform per batch
          for (uint32_t i = p0 + tid; i < i0 + n; i += NP) win[i - base] = __ldg(a.idx + i);
          fence_proxy_async_smem();  // in a run, a later draw's window is bulk-copied over these words
          named_sync(kBarProducers, NP);
        }
      }
      uint32_t* tbl = table + (DEDUP == DEDUP_SORT ? 0u : s * a.hash_slots);  // this batch's hash table
      if (DEDUP == DEDUP_SORT) {
        BatchSmem S;
        S.map = map + pad;
        S.keys = reinterpret_cast<unsigned long long*>(table);
        S.uniq = uniq;
        S.ucount = counter;
        S.wsum = misc + 8;
        const RowCopy<SH> consume{a, rows, uniq};
        if (a.sort_pos_bits)
          sort_dedup<uint32_t>(a, S, win + pad, n, tid, NP, GroupSync{kBarProducers, NP}, consume, a.sort_pos_bits);
        else
          sort_dedup<unsigned long long>(a, S, win + pad, n, tid, NP, GroupSync{kBarProducers, NP}, consume, 32);
      } else {
        const uint32_t mask = a.hash_slots - 1;
        constexpr int Q = 4 * kGroupsPerPass;  // positions per thread and pass
        // Collisions all eight positions together, a slot per round: parallel hashing's
        // few probes alone (7.2M triangles: 203 us, one after another 213), and hashing
        // with the envelope shader, whose producers wait for the consumers (2M triangles
        // of a grid, batches of 64: 218 us and 231, at the tuned limits 100.4 and 100.2).
        // Hashing otherwise one position after another.
        constexpr bool kTogether = DEDUP == DEDUP_PHASH || SH == 2;
        for (uint32_t gb = 0; gb < ngroups; gb += kGroupsPerPass * NP) {  // warp-uniform
          // a thread's groups: the lanes of a warp take groups NPW apart, so
          // one CAS instruction meets fewer repeats of the same id
          uint32_t id[Q], sl[Q], prev[Q];
          uint32_t act = 0, newmask = 0, pend = 0;  // bit q: position q
#pragma unroll
          for (int k = 0; k < kGroupsPerPass; ++k) {
            const uint32_t g = gb + k * NP + lane * NPW + pw;
            uint4 w = make_uint4(0, 0, 0, 0);
            if (g < ngroups) w = reinterpret_cast<const uint4*>(win)[g];
            const uint32_t raw[4] = {w.x, w.y, w.z, w.w};
            // positions [pad, pad + n) of the window: all four of a group but at its two ends
            const uint32_t hi = min(pad + n - min(4 * g, pad + n), 4u), lo = g == 0 ? pad : 0u;
            act |= (((1u << hi) - 1u) & ~((1u << lo) - 1u)) << (4 * k);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              id[4 * k + e] = raw[e] < a.num_verts ? raw[e] : kInvalidId;
              sl[4 * k + e] = hash_slot(id[4 * k + e], a.hash_bits);
            }
          }
          // the first probe of every position, issued before any result is used
#pragma unroll
          for (int q = 0; q < Q; ++q) prev[q] = (act >> q) & 1u ? atomicCAS(&tbl[sl[q]], kEmpty, id[q]) : kEmpty;
          // collisions (6% of the positions at the tuned limits).  One after another:
          // a thread's positions still probing, a slot at a time, in one loop --
          // advancing all eight together takes as many rounds as the longest chain of
          // the warp, ~90 instructions each
          uint32_t probing = 0;
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            if (!((act >> q) & 1u)) sl[q] = 0;
            else if (prev[q] == kEmpty) newmask |= 1u << q;
            else if (prev[q] != id[q]) probing |= 1u << q;
          }
          if constexpr (kTogether) {
            const uint32_t rounds = DEDUP == DEDUP_PHASH ? a.probe_k : a.hash_slots;
            for (uint32_t round = 1; probing && round < rounds; ++round) {
#pragma unroll
              for (int q = 0; q < Q; ++q)
                if ((probing >> q) & 1u) {
                  sl[q] = (sl[q] + 1) & mask;
                  prev[q] = atomicCAS(&tbl[sl[q]], kEmpty, id[q]);
                }
#pragma unroll
              for (int q = 0; q < Q; ++q)
                if ((probing >> q) & 1u) {
                  if (prev[q] == kEmpty) newmask |= 1u << q;
                  if (prev[q] == kEmpty || prev[q] == id[q]) probing &= ~(1u << q);
                }
            }
            if (DEDUP == DEDUP_PHASH) {
#pragma unroll
              for (int q = 0; q < Q; ++q)
                if ((probing >> q) & 1u) sl[q] = (sl[q] + 1) & mask;  // the next slot to probe
              pend = probing;
            } else if (probing) {  // table full: cannot happen within capacity
              atomicOr(a.err, EBIT_CAPACITY);
            }
          } else {
            for (uint32_t tries = 1; probing;) {
              const uint32_t q = __ffs(probing) - 1;
              uint32_t myid = id[0], at = sl[0];
#pragma unroll
              for (int k = 1; k < Q; ++k)
                if (q == (uint32_t)k) {
                  myid = id[k];
                  at = sl[k];
                }
              at = (at + 1) & mask;
              const bool over = tries >= a.hash_slots;
              uint32_t got = 0;
              if (!over) {
                got = atomicCAS(&tbl[at], kEmpty, myid);
                ++tries;
                newmask |= (got == kEmpty ? 1u : 0u) << q;
              } else {  // table full: cannot happen within capacity
                atomicOr(a.err, EBIT_CAPACITY);
                at = 0;
              }
#pragma unroll
              for (int k = 0; k < Q; ++k)
                if (q == (uint32_t)k) sl[k] = at;
              if (over || got == kEmpty || got == myid) {
                probing &= probing - 1;
                tries = 1;
              }
            }
          }
          if (DEDUP == DEDUP_PHASH) {
            // the positions still pending (rare), one at a time -- the lowest
            // lane's lowest position first -- probed by the whole warp 32
            // consecutive slots at a time; one loop for all Q positions keeps
            // this cold path small
            for (uint32_t anyp = __ballot_sync(kFull, pend != 0u); anyp; anyp = __ballot_sync(kFull, pend != 0u)) {
              const uint32_t leader = __ffs(anyp) - 1;
              const uint32_t q = __ffs(__shfl_sync(kFull, pend, leader)) - 1;  // uniform
              uint32_t myid = id[0], mysl = sl[0];
#pragma unroll
              for (int k = 1; k < Q; ++k)
                if (q == (uint32_t)k) {
                  myid = id[k];
                  mysl = sl[k];
                }
              const uint32_t lid = __shfl_sync(kFull, myid, leader);
              uint32_t lh = __shfl_sync(kFull, mysl, leader);
              uint32_t found = 0;
              bool fresh = false;
              for (uint32_t guard = 0;; ++guard) {
                if (guard > a.hash_slots / 16 + 64) {  // table full: cannot happen within capacity
                  if (lane == 0) atomicOr(a.err, EBIT_CAPACITY);
                  found = 0;
                  break;
                }
                const uint32_t ps = (lh + lane) & mask;
                const uint32_t val = tbl[ps];
                const uint32_t hit = __ballot_sync(kFull, val == lid);
                if (hit) {
                  found = (lh + __ffs(hit) - 1) & mask;
                  break;
                }
                const uint32_t emp = __ballot_sync(kFull, val == kEmpty);
                if (emp) {
                  const uint32_t fl = __ffs(emp) - 1;
                  const uint32_t cs = (lh + fl) & mask;
                  uint32_t cv = 0;
                  if (lane == fl) cv = atomicCAS(&tbl[cs], kEmpty, lid);
                  cv = __shfl_sync(kFull, cv, fl);
                  if (cv == kEmpty || cv == lid) {
                    found = cs;
                    fresh = cv == kEmpty;
                    break;
                  }
                  lh = cs;  // the slot was just taken: probe on from it
                } else {
                  lh = (lh + 32) & mask;
                }
              }
              if (lane == leader) {
#pragma unroll
                for (int k = 0; k < Q; ++k)
                  if (q == (uint32_t)k) sl[k] = found;
                newmask |= (fresh ? 1u : 0u) << q;
                pend &= ~(1u << q);
              }
            }
          }
          // ranks for this pass's new ids (lane order, then position order);
          // each new vertex's row starts on its way into the slot at once
          const uint32_t cnt = __popc(newmask);
          const uint32_t b0 = __ballot_sync(kFull, cnt & 1u), b1 = __ballot_sync(kFull, cnt & 2u),
                         b2 = __ballot_sync(kFull, cnt & 4u), b3 = __ballot_sync(kFull, cnt & 8u);
          const uint32_t lt = lanemask_lt();
          const uint32_t total = __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2) + 8 * __popc(b3);
          uint32_t r = 0;
          if (lane == 0 && total) r = atomicAdd(counter, total);
          r = __shfl_sync(kFull, r, 0) + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt) +
              8 * __popc(b3 & lt);
          // Parallel hashing with the envelope shader, whose producers wait for the
          // consumers: a warp's new rows are copied one per lane (a lane holds one new
          // id of every five positions), fewer instructions for the other role; 2M
          // triangles 101.3 us, 102.8 copied as below.  Elsewhere each row starts as soon
          // as its id is known: hash 100.2 us (100.6 gathered), on a grid in batches of 64
          // triangles 231 (252), MVP on the 7.2M-triangle mesh 198.6 (204.2).
          constexpr bool kGather = SH == 2 && DEDUP == DEDUP_PHASH;
          uint32_t rw = 0;  // the warp's first rank
          if constexpr (kGather) rw = __shfl_sync(kFull, r, 0);
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            if ((newmask >> q) & 1u) {
              if (r < a.ucap) {
                dense[sl[q]] = (uint16_t)r;
                uniq[r] = id[q];
                if constexpr (!kGather) {
                  if (!SPILL || r < a.row_cap) copy_row<SH>(a, rows, r, id[q]);
                }
              } else {
                atomicOr(a.err, EBIT_CAPACITY);
              }
              ++r;
            }
          }
          if constexpr (kGather) {
            __syncwarp();
            const uint32_t re = min(rw + total, SPILL ? a.row_cap : a.ucap);
            for (uint32_t k = rw + lane; k < re; k += 32) copy_row<SH>(a, rows, k, uniq[k]);
          }
#pragma unroll
          for (int k = 0; k < kGroupsPerPass; ++k) {
            const uint32_t g = gb + k * NP + lane * NPW + pw;
            if (g < ngroups)
              reinterpret_cast<uint2*>(map)[g] =
                  make_uint2(sl[4 * k] | (sl[4 * k + 1] << 16), sl[4 * k + 2] | (sl[4 * k + 3] << 16));
          }
        }
      }
      // hand the slot over: its phase completes once every producer has
      // arrived and this thread's row copies have landed
      cp_async_mbar_arrive(&bars[2 + s]);
      mbar_arrive(&bars[2 + s]);
      if (DEDUP != DEDUP_SORT) {
        // empty the other table for the next batch (the last batch used it),
        // after this batch's insertions so that the stores do not queue
        // ahead of its atomics
        uint32_t* other = table + (s ^ 1u) * a.hash_slots;
        for (uint32_t sl = 4 * tid; sl < a.hash_slots; sl += 4 * NP)
          *reinterpret_cast<uint4*>(other + sl) = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
      }
      // every id of the batch inserted, the other table empty again; the
      // window and the sort keys are free; the next batch is known
      named_sync(kBarProducers, NP);
      b = misc[6 + (s ^ 1u)];
    }
    // never leave a copy in flight into this block's shared memory
    cp_async_wait<0>();
    if (tid == 0 && window_pending && *abort_flag)  // sleeps in steps, at most ~0.8 s
      for (uint32_t it = 0; it < (1u << 14); ++it)
        if (mbar_try_wait_sleep(&bars[pending_buf], (wph >> pending_buf) & 1u, 50000u)) break;
  } else {
    // ======================= consumers =======================
    const uint32_t ctid = tid - NP, cw = warp - NPW;
    float4* stage = reinterpret_cast<float4*>(smem + L.off_stage) + cw * 32u * K;
    unsigned long long inv_total = 0, nbatches = 0;
    bool bulk_pending = false;  // a bulk store of this warp may still read its staging area
    uint32_t fph = 0u;  // bit s: parity of full[s]
    for (uint32_t j = 0;; ++j) {
      const uint32_t s = j & 1u;
      if (!wait_or_abort(&bars[2 + s], (fph >> s) & 1u, abort_flag, cap.err)) break;
      fph ^= 1u << s;
      const uint32_t b = misc[4 + s];  // the slot's batch
      if (b == kNoBatch) break;
      decltype(auto) a = src.args(j);
      src.uniforms(j, ctid, NC);
      const uint32_t t0 = misc[36 + 2 * s], t1 = misc[37 + 2 * s];
      const uint32_t i0 = 3 * t0, n = 3 * (t1 - t0), base = i0 & ~3u, pad = i0 - base;
      const uint32_t ngroups = (pad + n + 3) >> 2;
      unsigned char* slot_p = ring(s);
      const uint16_t* map = reinterpret_cast<const uint16_t*>(slot_p + L.ring_map);
      const uint16_t* dense = reinterpret_cast<const uint16_t*>(slot_p + L.ring_dense);
      const uint32_t* uniq = reinterpret_cast<const uint32_t*>(slot_p + L.ring_uniq);
      unsigned char* rows = slot_p + L.ring_rows;
      float4* vsh = reinterpret_cast<float4*>(rows);
      const uint32_t U = min(misc[s], a.ucap);
      // where this slot's shaded vertices past row_cap go (a slot's readers are done before its next writers:
      // the consumers' barrier of the batch between)
      float4* spill = !SPILL ? nullptr : a.spill + (size_t)2 * (a.ucap - a.row_cap) * (2 * blockIdx.x + s);

      // --- shade each unique vertex once, in place
      for (uint32_t r = ctid; r < U; r += NC) {
        float o[8];
        const uint32_t id = uniq[r];
        if (id < a.num_verts) {
          VertexIn v;
          if (!SPILL || r < a.row_cap) load_raw<SH>(rows + r * RB, v);
          else fetch_vertex<SH>(a.verts, a.stride, id, v, a.vec8 != 0);
          shade_vertex<SH>(u, palette, v, o);
        } else {
#pragma unroll
          for (int c = 0; c < 8; ++c) o[c] = 0.f;
          atomicOr(a.err, EBIT_INDEX_RANGE);
        }
        if (K == 7) o[7] = 0.f;
        const float4 lo = make_float4(o[0], o[1], o[2], o[3]), hi = make_float4(o[4], o[5], o[6], o[7]);
        if (!SPILL || r < a.row_cap) {
          vsh[row_slot<SH>(r, 0)] = lo;
          vsh[row_slot<SH>(r, 1)] = hi;
        } else {
          spill[2 * (r - a.row_cap)] = lo;
          spill[2 * (r - a.row_cap) + 1] = hi;
        }
      }
      named_sync(kBarConsumers, NC);  // every unique vertex shaded; every consumer has read the counter
      if (ctid == 0) {
        misc[s] = 0;  // the slot's counter, for the batch two on
        inv_total += U;
        nbatches += 1;
        if (a.batch_inv != nullptr) {
          const uint32_t k = src.number(b, j);
          if (k < a.batch_cap) a.batch_inv[k] = U;
        }
      }

      // --- assemble the batch's triangles in input order
      if (n <= a.max_batch_idx) {  // a larger batch was flagged and stopped by the producers
        const size_t f_lo = (size_t)K * i0, f_hi = (size_t)K * (i0 + n);  // the batch's output floats
        for (uint32_t gw = cw * 32u; gw < ngroups; gw += NC) {  // warp-uniform
          const uint32_t g = gw + lane;
          uint2 m = make_uint2(0, 0);
          if (g < ngroups) m = reinterpret_cast<const uint2*>(map)[g];
          const uint32_t sl[4] = {m.x & 0xFFFFu, m.x >> 16, m.y & 0xFFFFu, m.y >> 16};
          float f[4 * 7];  // K = 7: the 4 corners' floats, regrouped into 7 float4
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            uint32_t r = (DEDUP == DEDUP_SORT) ? sl[e] : (uint32_t)dense[sl[e]];
            r = r < U ? r : 0u;  // positions outside the batch (never written) and flagged capacity errors
            float4 lo, hi;
            if (!SPILL || r < a.row_cap) {
              lo = vsh[row_slot<SH>(r, 0)];
              hi = vsh[row_slot<SH>(r, 1)];
            } else {
              lo = spill[2 * (r - a.row_cap)];
              hi = spill[2 * (r - a.row_cap) + 1];
            }
            if (K == 8) {  // a corner is two whole float4
              stage[stage_put<K>(lane, 2 * e)] = lo;
              stage[stage_put<K>(lane, 2 * e + 1)] = hi;
            } else {
              f[7 * e + 0] = lo.x; f[7 * e + 1] = lo.y; f[7 * e + 2] = lo.z; f[7 * e + 3] = lo.w;
              f[7 * e + 4] = hi.x; f[7 * e + 5] = hi.y; f[7 * e + 6] = hi.z;
            }
            if (a.corner_ids != nullptr) {
              const uint32_t p = 4 * g + e;
              if (g < ngroups && p >= pad && p < pad + n) a.corner_ids[base + p] = uniq[r];
            }
          }
          const size_t F0 = (size_t)K * (base + 4 * gw);  // first float of the warp's span (16-byte aligned)
          const bool interior = F0 >= f_lo && F0 + 128 * K <= f_hi;  // the whole span lies in the batch
          if (K == 7) {
            if (bulk_pending) {  // the last bulk store must have read the staging area
              if (lane == 0) bulk_wait_read<0>();
              __syncwarp();
              bulk_pending = false;
            }
#pragma unroll
            for (int jj = 0; jj < 7; ++jj)
              stage[stage_put<K>(lane, jj)] = make_float4(f[4 * jj], f[4 * jj + 1], f[4 * jj + 2], f[4 * jj + 3]);
            if (interior) {  // the span in one bulk (TMA) store, in output order in the staging area
              fence_proxy_async_smem();
              __syncwarp();
              if (lane == 0) {
                bulk_store(a.out + F0, stage, 128 * K * 4);
                bulk_commit();
              }
              bulk_pending = true;
              continue;
            }
          }
          __syncwarp();
#pragma unroll
          for (int jj = 0; jj < K; ++jj) {
            const float4 v = stage[stage_get<K>(32 * jj + lane)];
            const size_t fq = F0 + 4 * (32 * jj + lane);
            if (interior || (fq >= f_lo && fq + 4 <= f_hi)) {
              st_stream4(a.out + fq, v);
            } else if (fq + 4 > f_lo && fq < f_hi) {  // a float4 the neighbouring batch shares
              const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
              for (int c = 0; c < 4; ++c)
                if (fq + c >= f_lo && fq + c < f_hi) a.out[fq + c] = vv[c];
            }
          }
          __syncwarp();  // the staging area is read before the next step writes it
        }
      }
      mbar_arrive(&bars[4 + s]);  // this thread is done with the slot
    }
    if (lane == 0) bulk_wait_all<0>();  // this warp's bulk stores are complete
    if (ctid == 0 && nbatches) {
      atomicAdd(cap.counters + CNT_INVOCATIONS, inv_total);
      atomicAdd(cap.counters + CNT_BATCHES, nbatches);
      atomicAdd(cap.counters + CNT_UNIQUE, inv_total);
    }
  }
}

}  // namespace gp

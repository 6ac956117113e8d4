// Parallel random walk with on-the-fly reuse (Section 5.4).
//
// Agents live on a toroidal W x H grid; each is the packed key (x << 16) | y.
// Per step an agent evaluates every move (dx, dy) with 1 <= dx^2 + dy^2 <=
// 16^2 -- likelihood A[target] * (65536 / r^2), integers, so comparisons are
// exact -- keeps the 8 largest (earlier candidates first on ties) and draws
// one with probability proportional to its likelihood from a SplitMix64
// number of (seed, step, agent).  The 8 kept moves depend only on the cell,
// so the key is the "index" of the reuse methods:
//   naive  -- every agent evaluates its own cell;
//   warp   -- each warp takes 32 agents; __match_any_sync groups equal keys
//             and the lowest lane of a group evaluates the cell for all;
//   sort / hash / phash -- one thread block per static batch of agents runs
//             the shared dedup body (Algorithm 2 / Algorithm 3 / Section 3.4)
//             on the batch's keys; each unique cell is evaluated once into
//             shared memory, then every agent draws from its cell's row.
//
// The candidate moves sit in constant memory; all lanes of a warp walk them
// in step, so each constant read is a broadcast.
//
// Pruning.  The candidates are looked at nearest first, so their weights fall
// as 1 / r^2, and the activity within 4, 8 and 16 cells of the agent's tile of
// the field is bounded by walk_bound_kernel, once per call.  Once the 8th kept
// likelihood is above (bound) x (weight), no candidate left at that distance
// can enter: the 8 moves are exact after 8.3 of 796 candidates on average, and
// 14 for the slowest lane of a warp (Gaussian fields of sigma 8 to 40; a single
// bound for all 16 cells: 17 and 50).  300,000 agents on a 256 x 256 field:
// 23 us a step against 570 us for the whole neighbourhood.  The tiles are
// sized so that at most kWalkTiles cover the field.  On a field of few active cells
// nothing stops the scan, and nearest first its reads share no cache lines: a
// million agents on an 8192 x 8192 field, one cell in 500 active, took 6,570 us a
// step against 1,400 row by row; an agent with an empty cell beside it goes row by
// row (1,430, the bounds included).
#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

#include "gp.h"
#include "gp_batch_body.cuh"

namespace gp {

constexpr int kWalkRadius = 16;
constexpr int kWalkKeep = 8;
constexpr int kWalkCand = 796;  // offsets with 1 <= dx^2 + dy^2 <= 256

// Bound scratch: kWalkSlots tables, so that calls on different streams need
// not wait for one another; a slot's event orders its users (bound_slot).
constexpr uint32_t kWalkTiles = 4096;
constexpr uint32_t kWalkSlots = 4;

// The candidates nearest first (weights falling), then all of them again row by
// row (dy, then dx, each from -16 to 16): without a bound each one is looked
// at, and consecutive ones share cache lines.
__constant__ int32_t c_walk_off[2 * kWalkCand];  // (dx + 16) | (dy + 16) << 8
__constant__ uint32_t c_walk_w[2 * kWalkCand];   // 65536 / r^2
constexpr int kWalkIn4 = 48, kWalkIn8 = 196;     // candidates within 4 and 8 cells
static __device__ uint4 g_walk_bound[kWalkSlots][kWalkTiles];

struct WalkArgs {
  const uint32_t* act;  // [h][w]
  uint32_t w, h;
  const uint32_t* pin;
  uint32_t* pout;
  uint32_t n;
  uint64_t seed;
  uint32_t step;
  uint32_t batch;                  // agents per batch (counts; sort/hash/phash block size unit)
  const uint4* bound;              // per tile of 2^tile_bits cells a side: the largest activity within 4, 8 and 16
                                   // cells of the tile (nullptr: none, every candidate is looked at)
  uint32_t tile_bits, tiles_x, tiles;
  unsigned long long* counters;    // [0] evaluations, [1] batches, [2] error bits
};

// One step of SplitMix64 from state x: the increment, then the mix.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The 8 kept moves of cell (x, y): running sums of their likelihoods
// (cum[7] = total) and the moves, packed as in c_walk_off.
struct CellMoves {
  uint64_t cum[kWalkKeep];
  uint32_t mv[kWalkKeep];
};

// The likelihood of candidate j.
__device__ __forceinline__ uint64_t walk_likelihood(const WalkArgs& a, int x, int y, int j) {
  const int32_t o = c_walk_off[j];
  int tx = x + (o & 0xFF) - kWalkRadius, ty = y + (o >> 8) - kWalkRadius;
  tx += tx < 0 ? (int)a.w : 0;
  tx -= tx >= (int)a.w ? (int)a.w : 0;
  ty += ty < 0 ? (int)a.h : 0;
  ty -= ty >= (int)a.h ? (int)a.h : 0;
  return (uint64_t)__ldg(a.act + (uint32_t)ty * a.w + (uint32_t)tx) * c_walk_w[j];
}

// A kept candidate is one 64-bit key: the likelihood (below 2^48) above the
// complement of the packed offset, so that a larger key means a larger
// likelihood or, on equal ones, the earlier candidate; 0 = none.
__device__ __forceinline__ uint64_t walk_key(uint64_t lik, int j) {
  return lik ? (lik << 16) | (0xFFFFu - (uint32_t)c_walk_off[j]) : 0ull;
}

__device__ __forceinline__ void eval_cell(const WalkArgs& a, uint32_t key, CellMoves& out) {
  const int x = (int)(key >> 16), y = (int)(key & 0xFFFFu);
  const bool bounded = a.bound != nullptr;
  uint4 lim = make_uint4(0, 0, 0, 0);
  if (bounded) {
    const uint32_t cx = (uint32_t)x < a.w ? x : x - a.w, cy = (uint32_t)y < a.h ? y : y - a.h;
    lim = __ldg(a.bound + min((cy >> a.tile_bits) * a.tiles_x + (cx >> a.tile_bits), a.tiles - 1));
  }
  const int base = bounded ? 0 : kWalkCand;
  // the first eight, sorted (descending) by Batcher's odd-even merge network
  static_assert(kWalkKeep == 8, "the network below sorts eight");
  uint64_t kept[kWalkKeep];
#pragma unroll
  for (int k = 0; k < kWalkKeep; ++k) kept[k] = walk_key(walk_likelihood(a, x, y, base + k), base + k);
  auto cx = [&](int i, int k) {
    const uint64_t hi = kept[i] > kept[k] ? kept[i] : kept[k], lo = kept[i] > kept[k] ? kept[k] : kept[i];
    kept[i] = hi;
    kept[k] = lo;
  };
  cx(0, 1); cx(2, 3); cx(4, 5); cx(6, 7);
  cx(0, 2); cx(1, 3); cx(4, 6); cx(5, 7);
  cx(1, 2); cx(5, 6); cx(0, 4); cx(1, 5); cx(2, 6); cx(3, 7);
  cx(2, 4); cx(3, 5);
  cx(1, 2); cx(3, 4); cx(5, 6);
  static_assert(kWalkCand % 4 == 0 && kWalkIn4 % 4 == 0 && kWalkIn8 % 4 == 0, "candidates are read four at a time");
  uint64_t least = max(kept[kWalkKeep - 1] >> 16, (uint64_t)1);  // likelihood below which nothing enters
  auto four = [&](int j) {  // candidates j..j + 3: four independent activity reads in flight, then the insertions
    uint64_t lik[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) lik[q] = walk_likelihood(a, x, y, j + q);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (lik[q] >= least) {
        uint64_t cur = walk_key(lik[q], j + q);
#pragma unroll
        for (int k = 0; k < kWalkKeep; ++k) {
          const uint64_t t = kept[k];
          kept[k] = cur > t ? cur : t;
          cur = cur > t ? t : cur;
        }
        least = max(kept[kWalkKeep - 1] >> 16, (uint64_t)1);
      }
    }
  };
  if (bounded && kept[kWalkKeep - 1] == 0 && lim.z != 0) {
    // an empty cell beside the agent and activity somewhere near: the bounds will not stop the scan for long, so all
    // candidates are looked at, row by row
#pragma unroll
    for (int k = 0; k < kWalkKeep; ++k) kept[k] = 0;
#pragma unroll 1
    for (int j = 0; j < kWalkCand; j += 4) four(kWalkCand + j);
  } else {
    int j = kWalkKeep;
#pragma unroll 1
    for (int level = bounded ? 0 : 2; level < 3; ++level) {
      const int end = level == 0 ? kWalkIn4 : level == 1 ? kWalkIn8 : kWalkCand;
      const uint32_t amax = level == 0 ? lim.x : level == 1 ? lim.y : lim.z;
#pragma unroll 1
      for (; j < end; j += 4) {
        // c_walk_w[j] is the largest weight left
        if (bounded && least > (uint64_t)amax * c_walk_w[j]) break;
        four(base + j);
      }
      j = end;
    }
  }
  uint64_t acc = 0;
#pragma unroll
  for (int k = 0; k < kWalkKeep; ++k) {
    acc += kept[k] >> 16;
    out.cum[k] = acc;
    out.mv[k] = 0xFFFFu - (uint32_t)(kept[k] & 0xFFFFu);  // of an empty entry: never taken
  }
}

// One warp per tile: the largest activity of the cells within 4, 8 and 16
// cells of the tile's square (columns and rows counted apart; the field wraps
// around).  Reads that mostly hit L1/L2; runs once per call, before its steps.
__global__ void __launch_bounds__(256) walk_bound_kernel(const __grid_constant__ WalkArgs a, uint4* bound) {
  const uint32_t tile = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = lane_id();
  if (tile >= a.tiles) return;
  constexpr uint32_t R = kWalkRadius;
  const uint32_t x0 = (tile % a.tiles_x) << a.tile_bits, y0 = (tile / a.tiles_x) << a.tile_bits;
  const uint32_t sx = min(1u << a.tile_bits, a.w - x0), sy = min(1u << a.tile_bits, a.h - y0);
  // the square with its margin, at most once around the field
  const uint32_t nx = min(sx + 2 * R, a.w), ny = min(sy + 2 * R, a.h);
  // first column and row, wrapped (w, h >= 17 > R)
  const uint32_t fx = (x0 + a.w - R) % a.w, fy = (y0 + a.h - R) % a.h;
  // a column's rows in five runs: beyond 8 cells, beyond 4, near, and back;
  // where the margin meets itself around the field, every cell counts as near
  const bool once_x = nx == sx + 2 * R, once_y = ny == sy + 2 * R;
  uint32_t b4 = 0, b8 = 0, b16 = 0;
  for (uint32_t i = lane; i < nx; i += 32) {
    uint32_t x = fx + i;
    x -= x >= a.w ? a.w : 0u;
    auto rows = [&](uint32_t j0, uint32_t j1) {
      uint32_t m = 0;
#pragma unroll 8
      for (uint32_t j = j0; j < j1; ++j) {
        uint32_t y = fy + j;
        y -= y >= a.h ? a.h : 0u;
        m = max(m, __ldg(a.act + (size_t)y * a.w + x));
      }
      return m;
    };
    uint32_t m4, m8, m16;
    if (once_y) {
      m16 = max(rows(0, R - 8), rows(ny - (R - 8), ny));
      m8 = max(rows(R - 8, R - 4), rows(ny - (R - 4), ny - (R - 8)));
      m4 = rows(R - 4, ny - (R - 4));
      m8 = max(m8, m4);
      m16 = max(m16, m8);
    } else {
      m4 = m8 = m16 = rows(0, ny);
    }
    const uint32_t dx = !once_x ? 0u : (i < R ? R - i : (i >= R + sx ? i - R - sx + 1 : 0u));
    b16 = max(b16, m16);
    if (dx <= 8) b8 = max(b8, m8);
    if (dx <= 4) b4 = max(b4, m4);
  }
  b4 = __reduce_max_sync(kFull, b4);
  b8 = __reduce_max_sync(kFull, b8);
  b16 = __reduce_max_sync(kFull, b16);
  if (lane == 0) bound[tile] = make_uint4(b4, b8, b16, 0);
}

__device__ __forceinline__ uint32_t take_move(const WalkArgs& a, uint32_t key, uint32_t agent, const uint64_t* cum,
                                              const uint32_t* mv) {
  if (cum[kWalkKeep - 1] == 0) return key;  // no move has a positive likelihood: stay
  const uint64_t u = splitmix64(a.seed ^ (((uint64_t)a.step << 32) | agent));
  const uint64_t r = u % cum[kWalkKeep - 1];
  uint32_t m = mv[kWalkKeep - 1];
#pragma unroll
  for (int k = kWalkKeep - 2; k >= 0; --k) m = cum[k] > r ? mv[k] : m;
  int x = (int)(key >> 16) + (int)(m & 0xFF) - kWalkRadius;
  int y = (int)(key & 0xFFFFu) + (int)(m >> 8) - kWalkRadius;
  x += x < 0 ? (int)a.w : 0;
  x -= x >= (int)a.w ? (int)a.w : 0;
  y += y < 0 ? (int)a.h : 0;
  y -= y >= (int)a.h ? (int)a.h : 0;
  return ((uint32_t)x << 16) | (uint32_t)y;
}

__global__ void __launch_bounds__(256) walk_naive_kernel(const __grid_constant__ WalkArgs a) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  const uint32_t key = a.pin[i];
  CellMoves cm;
  eval_cell(a, key, cm);
  a.pout[i] = take_move(a, key, i, cm.cum, cm.mv);
  if (threadIdx.x == 0) {
    atomicAdd(a.counters + 0, (unsigned long long)min(blockDim.x, a.n - blockIdx.x * blockDim.x));
    atomicAdd(a.counters + 1, 1ull);
  }
}

// One warp per 32 agents; the group leader's row goes through shared memory.
__global__ void __launch_bounds__(256) walk_warp_kernel(const __grid_constant__ WalkArgs a) {
  __shared__ CellMoves rows[256];
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t lane = lane_id(), wbase = threadIdx.x & ~31u;
  if ((i & ~31u) >= a.n) return;  // warp-uniform
  const bool active = i < a.n;
  const uint32_t key = active ? a.pin[i] : 0xFFFFFFFFu;
  const uint32_t grp = __match_any_sync(kFull, key);
  const uint32_t leader = __ffs(grp) - 1;
  if (active && lane == leader) eval_cell(a, key, rows[threadIdx.x]);
  __syncwarp();
  if (active) {
    const CellMoves& r = rows[wbase + leader];
    a.pout[i] = take_move(a, key, i, r.cum, r.mv);
  }
  const uint32_t leaders = __ballot_sync(kFull, active && lane == leader);
  if (lane == 0) atomicAdd(a.counters + 0, (unsigned long long)__popc(leaders));
  if (threadIdx.x == 0) atomicAdd(a.counters + 1, 1ull);
}

// One block per batch of a.batch agents: dedup of the keys, one evaluation
// per unique cell into shared memory, then every agent's draw.
struct WalkShade {
  const WalkArgs& wa;
  const uint32_t* uniq;
  CellMoves* rows;
  uint32_t ucap;
  __device__ __forceinline__ void operator()(uint32_t rb, uint32_t re, uint32_t lane) const {
    re = min(re, ucap);  // ranks >= ucap (a flagged capacity error) were not stored
    for (uint32_t r = rb + lane; r < re; r += 32) eval_cell(wa, uniq[r], rows[r]);
  }
};

template <int DEDUP>
__global__ void __launch_bounds__(512, 2) walk_batched_kernel(const __grid_constant__ WalkArgs wa,
                                                           const __grid_constant__ DrawArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint32_t S = wa.batch, tid = threadIdx.x, NT = blockDim.x;
  const uint32_t i0 = blockIdx.x * S, n = min(S, wa.n - i0);
  // layout: rows [S] | keys [S] | map [S] u16 | uniq [S] | table [slots] + dense [slots] u16 or sort keys | misc
  CellMoves* rows = reinterpret_cast<CellMoves*>(smem);
  uint32_t* keys = reinterpret_cast<uint32_t*>(rows + S);
  uint16_t* map = reinterpret_cast<uint16_t*>(keys + S);
  uint32_t* uniq = reinterpret_cast<uint32_t*>(map + ((S + 1) & ~1u));
  unsigned char* tail = reinterpret_cast<unsigned char*>(uniq + S);
  BatchSmem B;
  B.map = map;
  B.uniq = uniq;
  if (DEDUP == DEDUP_SORT) {
    B.keys = reinterpret_cast<unsigned long long*>(tail);
    tail += (size_t)a.sort_n * 8;
  } else {
    B.table = reinterpret_cast<uint32_t*>(tail);
    B.dense = reinterpret_cast<uint16_t*>(tail + (size_t)a.hash_slots * 4);
    tail += (size_t)a.hash_slots * 6;
  }
  uint32_t* misc = reinterpret_cast<uint32_t*>(tail);
  B.ucount = misc;
  B.wsum = misc + 8;
  B.vsh = nullptr;
  for (uint32_t k = tid; k < n; k += NT) keys[k] = wa.pin[i0 + k];
  if (DEDUP != DEDUP_SORT)
    for (uint32_t s = tid; s < a.hash_slots; s += NT) B.table[s] = kEmpty;
  if (tid == 0) *B.ucount = 0;
  __syncthreads();
  dedup<DEDUP, true>(a, B, keys, n, tid, NT, BlockSync(), WalkShade{wa, uniq, rows, a.ucap});
  __syncthreads();
  const uint32_t U = min(*B.ucount, a.ucap);
  for (uint32_t k = tid; k < n; k += NT) {
    uint32_t r = map[k];
    if (DEDUP != DEDUP_SORT) r = B.dense[r];
    r = r < U ? r : 0u;  // only after a flagged capacity error
    wa.pout[i0 + k] = take_move(wa, keys[k], i0 + k, rows[r].cum, rows[r].mv);
  }
  if (tid == 0) {
    atomicAdd(wa.counters + 0, (unsigned long long)U);
    atomicAdd(wa.counters + 1, 1ull);
  }
}

size_t walk_batched_smem(int dedup, uint32_t S, uint32_t slots, uint32_t sort_n) {
  size_t o = (size_t)S * sizeof(CellMoves) + (size_t)S * 4 + (size_t)((S + 1) & ~1u) * 2 + (size_t)S * 4;
  o += dedup == DEDUP_SORT ? (size_t)sort_n * 8 : (size_t)slots * 6;
  return o + 64 * 4;
}

}  // namespace gp

using namespace gp;

namespace {

std::mutex g_walk_mu;
uint64_t g_walk_ready = 0;  // bit d: the candidate table is in device d's constant memory

gp_status walk_tables(int device) {
  std::lock_guard<std::mutex> lk(g_walk_mu);
  if (device < 64 && (g_walk_ready >> device) & 1) return GP_OK;
  std::vector<std::pair<int, int32_t>> cand;  // (r^2, packed offset)
  for (int dy = -kWalkRadius; dy <= kWalkRadius; ++dy)
    for (int dx = -kWalkRadius; dx <= kWalkRadius; ++dx) {
      const int r2 = dx * dx + dy * dy;
      if (r2 < 1 || r2 > kWalkRadius * kWalkRadius) continue;
      cand.emplace_back(r2, (dx + kWalkRadius) | ((dy + kWalkRadius) << 8));
    }
  if (cand.size() != (size_t)kWalkCand) return GP_ERR_UNSUPPORTED;
  int32_t off[2 * kWalkCand];
  uint32_t w[2 * kWalkCand];
  auto put = [&](int at) {
    for (int k = 0; k < kWalkCand; ++k) {
      off[at + k] = cand[k].second;
      w[at + k] = 65536u / (uint32_t)cand[k].first;
    }
  };
  put(kWalkCand);  // row by row, as they were found
  std::sort(cand.begin(), cand.end());
  put(0);
  if (cudaMemcpyToSymbol(c_walk_off, off, sizeof(off)) != cudaSuccess ||
      cudaMemcpyToSymbol(c_walk_w, w, sizeof(w)) != cudaSuccess)
    return GP_ERR_CUDA;
  if (device < 64) g_walk_ready |= 1ull << device;
  return GP_OK;
}

// The bound tables of each device: their address and, per table, the event
// that marks the end of its last user.
struct BoundSlots {
  uint4* base = nullptr;
  uint32_t next = 0;
  cudaEvent_t done[kWalkSlots] = {};
  std::mutex use[kWalkSlots];  // held from taking a slot to recording its event, so its users are ordered
};
std::mutex g_bound_mu;  // base, next
BoundSlots g_bound[64];

// A bound table for work on stream s of the device: the stream is made to
// wait for the table's last user (of any stream or thread).  nullptr without
// an error when there is none to be had: under stream capture (an event of
// uncaptured work cannot be waited for) or when the runtime refuses; the
// steps then look at every candidate.  The caller records *done behind its
// last use and then lets 'use' go.
uint4* bound_slot(int device, cudaStream_t s, std::unique_lock<std::mutex>& use, cudaEvent_t* done) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (device >= 64 || cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return nullptr;
  }
  BoundSlots& b = g_bound[device];
  uint32_t k;
  {
    std::lock_guard<std::mutex> lk(g_bound_mu);
    void* p = b.base;
    if (!p && cudaGetSymbolAddress(&p, g_walk_bound) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    b.base = static_cast<uint4*>(p);
    k = b.next++ % kWalkSlots;
  }
  use = std::unique_lock<std::mutex>(b.use[k]);
  if ((!b.done[k] && cudaEventCreateWithFlags(&b.done[k], cudaEventDisableTiming) != cudaSuccess) ||
      cudaStreamWaitEvent(s, b.done[k], 0) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  *done = b.done[k];
  return b.base + (size_t)k * kWalkTiles;
}

uint32_t pow2_at_least(uint32_t x) {
  uint32_t p = 1;
  while (p < x) p <<= 1;
  return p;
}

uint32_t tiles_of(uint32_t cells, uint32_t bits) { return (cells + (1u << bits) - 1) >> bits; }

// The bound is worked out when the cells read for it, per step, are at most
// the larger of these.  Measured: reading them takes 1.6 us per million; a
// step that looks at every candidate takes 170 us however few its agents are
// (the chain of one warp) and 1.9 us per 1000 agents where they fill the GPU.
// On a 2048 x 2048 field a step of 1,000 agents took 173 us without and 41 us
// with it; on 8192 x 8192, above the line, 10,000 agents 182 us and 187 us.
constexpr uint64_t kBoundReads = 64u << 20;
constexpr uint64_t kBoundReadsPerAgent = 1536;

}  // namespace

extern "C" gp_status gp_random_walk(const gp_walk_desc* d) {
  // Section 5.4; see include/gp.h
  if (!d) return GP_ERR_INVALID;
  if (d->width < 17 || d->height < 17 || d->width > 32768 || d->height > 32768 || !d->d_activity ||
      !d->d_counters)
    return GP_ERR_INVALID;
  if (d->num_agents && (!d->d_pos || !d->d_scratch)) return GP_ERR_INVALID;
  const int32_t v = d->variant;
  if (v != GP_NAIVE && v != GP_WARP && v != GP_SORT && v != GP_HASH && v != GP_PHASH) return GP_ERR_INVALID;
  const uint32_t S = d->batch_agents ? d->batch_agents : 576;
  const uint32_t threads = d->threads ? d->threads : 256;
  if (S % 32 || S == 0) return GP_ERR_INVALID;
  if (v >= GP_SORT && (S > 1024 || threads % 32 || (threads & (threads - 1)) || threads > 512))
    return GP_ERR_INVALID;
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) return GP_ERR_CUDA;
  gp_status st = walk_tables(device);
  if (st != GP_OK) return st;
  if (d->num_agents == 0 || d->steps == 0) return GP_OK;
  cudaStream_t s = static_cast<cudaStream_t>(d->stream);
  WalkArgs wa{};
  wa.act = d->d_activity;
  wa.w = d->width;
  wa.h = d->height;
  wa.n = d->num_agents;
  wa.seed = d->seed;
  wa.batch = S;
  wa.counters = d->d_counters;
  DrawArgs a{};
  size_t smem = 0;
  int dedup = DEDUP_HASH;
  if (v >= GP_SORT) {
    dedup = v == GP_SORT ? DEDUP_SORT : (v == GP_HASH ? DEDUP_HASH : DEDUP_PHASH);
    a.num_verts = 0xFFFFFFF0u;  // every key (< 2^31) is a valid "vertex"
    a.ucap = S;
    a.max_batch_idx = S;
    a.hash_slots = std::max(pow2_at_least(2 * S), pow2_at_least(threads));
    uint32_t bits = 0;
    while ((1u << bits) < a.hash_slots) ++bits;
    a.hash_bits = bits;
    a.sort_n = pow2_at_least(S);
    a.probe_k = 4;
    a.err = reinterpret_cast<uint32_t*>(d->d_counters + 2);
    smem = walk_batched_smem(dedup, S, a.hash_slots, a.sort_n);
    const void* fn = dedup == DEDUP_SORT ? (const void*)walk_batched_kernel<DEDUP_SORT>
                     : dedup == DEDUP_HASH ? (const void*)walk_batched_kernel<DEDUP_HASH>
                                           : (const void*)walk_batched_kernel<DEDUP_PHASH>;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      return GP_ERR_UNSUPPORTED;
  }
  std::unique_lock<std::mutex> slot_use;
  cudaEvent_t bound_done = nullptr;
  wa.tile_bits = 2;
  while ((uint64_t)tiles_of(d->width, wa.tile_bits) * tiles_of(d->height, wa.tile_bits) > kWalkTiles) ++wa.tile_bits;
  wa.tiles_x = tiles_of(d->width, wa.tile_bits);
  wa.tiles = wa.tiles_x * tiles_of(d->height, wa.tile_bits);
  const uint64_t side = (1ull << wa.tile_bits) + 2 * kWalkRadius;
  if (wa.tiles * side * side / d->steps <= std::max(kBoundReads, kBoundReadsPerAgent * d->num_agents)) {
    uint4* bound = bound_slot(device, s, slot_use, &bound_done);
    if (bound) {
      walk_bound_kernel<<<(wa.tiles + 7) / 8, 256, 0, s>>>(wa, bound);
      if (cudaGetLastError() != cudaSuccess) return GP_ERR_CUDA;
      wa.bound = bound;
    }
  }
  gp_status queued = GP_OK;
  for (uint32_t k = 0; k < d->steps && queued == GP_OK; ++k) {
    wa.step = d->first_step + k;
    wa.pin = (k & 1) ? d->d_scratch : d->d_pos;
    wa.pout = (k & 1) ? d->d_pos : d->d_scratch;
    if (v == GP_NAIVE) {
      walk_naive_kernel<<<(d->num_agents + 255) / 256, 256, 0, s>>>(wa);
    } else if (v == GP_WARP) {
      walk_warp_kernel<<<(d->num_agents + 255) / 256, 256, 0, s>>>(wa);
    } else {
      const uint32_t grid = (d->num_agents + S - 1) / S;
      if (dedup == DEDUP_SORT) walk_batched_kernel<DEDUP_SORT><<<grid, threads, smem, s>>>(wa, a);
      else if (dedup == DEDUP_HASH) walk_batched_kernel<DEDUP_HASH><<<grid, threads, smem, s>>>(wa, a);
      else walk_batched_kernel<DEDUP_PHASH><<<grid, threads, smem, s>>>(wa, a);
    }
    if (cudaGetLastError() != cudaSuccess) queued = GP_ERR_CUDA;
  }
  // behind whatever reads the table, also when a launch failed: its next user waits for that
  if (wa.bound && cudaEventRecord(bound_done, s) != cudaSuccess) queued = GP_ERR_CUDA;
  if (slot_use.owns_lock()) slot_use.unlock();
  if (queued != GP_OK) return queued;
  if (d->steps & 1) {  // the last step wrote the scratch buffer
    if (cudaMemcpyAsync(d->d_pos, d->d_scratch, (size_t)d->num_agents * 4, cudaMemcpyDeviceToDevice, s) !=
        cudaSuccess)
      return GP_ERR_CUDA;
  }
  return GP_OK;
}

// Single-draw vertex reuse: sorting (Algorithm 2), hashing (Algorithm 3) and
// parallel hashing (Section 3.4), over static batches (Section 3.3) or the
// dynamic batches of the partition (Section 3.4).
//
// Each block is persistent (grid = SMs x resident blocks): it takes batches
// blockIdx.x, blockIdx.x + gridDim.x, ... in turn, and for the last few
// rounds of the draw claims batches from a per-draw counter, one at a time,
// so blocks that run faster take more of them and all finish together.
// The block's work is reuse_batches (gp_reuse_body.cuh): producer warps
// deduplicate a batch while consumer warps shade and assemble the one before.
#include <algorithm>

#include "gp_reuse_body.cuh"

namespace gp {

constexpr uint32_t kReuseBarBytes = 64;
constexpr uint32_t kDynamicRounds = 6;  // rounds of batches per block claimed from the counter

// Batches [0, nstatic) go to the blocks in turn (block i: i, i + grid, ...);
// the last rounds, from nstatic on, are claimed from the per-draw counter, so
// blocks that run faster take more of them and all finish together -- and the
// claim's global atomic stays out of most batches.
template <bool DYN>
struct DrawSource {
  static constexpr bool kWarpNext = false;
  const DrawArgs& a;
  uint32_t nb, nstatic;
  __device__ __forceinline__ DrawSource(const DrawArgs& args) : a(args) {
    nb = DYN ? *a.num_batches_dev : a.num_batches;
    const uint32_t G = gridDim.x;
    nstatic = G * max(1u, nb / G > kDynamicRounds ? nb / G - kDynamicRounds : 1u);
  }
  __device__ __forceinline__ uint32_t first() const { return blockIdx.x; }
  __device__ __forceinline__ uint32_t end() const { return nb; }
  __device__ __forceinline__ const DrawArgs& args(uint32_t) const { return a; }
  __device__ __forceinline__ uint32_t number(uint32_t b, uint32_t) const { return b; }
  __device__ __forceinline__ void uniforms(uint32_t, uint32_t, uint32_t) const {}
  __device__ __forceinline__ uint32_t next(uint32_t b, uint32_t, uint32_t) const {
    return b + gridDim.x < nstatic
               ? b + gridDim.x
               : nstatic + atomicAdd(reinterpret_cast<unsigned int*>(a.counters + CNT_WORK), 1u);
  }
  __device__ __forceinline__ void range(uint32_t b, uint32_t, uint32_t& t0, uint32_t& t1) const {
    if (DYN) {
      t0 = __ldg(a.starts + b);
      t1 = __ldg(a.starts + b + 1);
    } else {
      t0 = b * a.static_batch_tris;
      t1 = min(t0 + a.static_batch_tris, a.num_tris);
    }
  }
};

template <int DEDUP, int SH, bool DYN, bool SPILL>
__device__ __forceinline__ void reuse_body(const DrawArgs& a, const Uniforms& u) {
  extern __shared__ __align__(128) unsigned char block_smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(block_smem);  // and behind them what reuse_layout lays out
  unsigned char* smem = block_smem + kReuseBarBytes;
  const uint32_t tid = threadIdx.x, NT = blockDim.x;
  DrawSource<DYN> src(a);
  if (src.first() >= src.end()) return;
  const ReuseLayout L = reuse_layout(DEDUP, SH, a, NT, SPILL ? a.row_cap : a.ucap, true);
  uint32_t* misc = reinterpret_cast<uint32_t*>(smem + L.off_misc);
  uint32_t* table = reinterpret_cast<uint32_t*>(smem + L.off_scratch);
  float* palette = reinterpret_cast<float*>(smem + L.off_pal);
  if (tid == 0) {
    const uint32_t NP = 32 * reuse_producer_warps(NT, DEDUP);
    reuse_init_bars(bars, NP, NT - NP);
    misc[0] = misc[1] = misc[2] = 0;
  }
  if (ShaderTraits<SH>::kSkin)
    for (uint32_t i = tid; i < 768; i += NT) palette[i] = u.palette[i];
  if (DEDUP != DEDUP_SORT)
    for (uint32_t s = tid; s < 2 * a.hash_slots; s += NT) table[s] = kEmpty;
  reuse_batches<DEDUP, SH, SPILL>(a, u, palette, smem, L, bars, NT, src);
}

// The kernel at 64 registers a thread (4 blocks of 256 threads fit an SM's
// registers) ...
template <int DEDUP, int SH, bool DYN, bool SPILL>
__global__ void __launch_bounds__(512, 2) reuse_kernel(const __grid_constant__ DrawArgs a,
                                                       const __grid_constant__ Uniforms u) {
  reuse_body<DEDUP, SH, DYN, SPILL>(a, u);
}

// ... and at up to 80 (3 blocks of 256 threads), for hash/phash draws over
// dynamic batches with the MVP or envelope shader: where shared memory already
// holds the block to 3 per SM, the extra registers cost no occupancy and spare
// the compiler's register-limited scheduling (draws take it only then).
template <int DEDUP, int SH>
__global__ void __maxnreg__(80) reuse_kernel_wide(const __grid_constant__ DrawArgs a,
                                                  const __grid_constant__ Uniforms u) {
  reuse_body<DEDUP, SH, true, false>(a, u);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

template <int D, bool DYN, bool SPILL>
static const void* reuse_fn_sh(int shader) {
  switch (shader) {
    case 0: return reinterpret_cast<const void*>(&reuse_kernel<D, 0, DYN, SPILL>);
    case 1: return reinterpret_cast<const void*>(&reuse_kernel<D, 1, DYN, SPILL>);
    case 2: return reinterpret_cast<const void*>(&reuse_kernel<D, 2, DYN, SPILL>);
    default: return reinterpret_cast<const void*>(&reuse_kernel<D, 3, DYN, SPILL>);
  }
}

template <bool DYN, bool SPILL>
static const void* reuse_fn(int dedup, int shader) {
  switch (dedup) {
    case DEDUP_SORT: return reuse_fn_sh<DEDUP_SORT, DYN, SPILL>(shader);
    case DEDUP_HASH: return reuse_fn_sh<DEDUP_HASH, DYN, SPILL>(shader);
    default: return reuse_fn_sh<DEDUP_PHASH, DYN, SPILL>(shader);
  }
}

static const void* reuse_kernel_ptr(int dedup, ReuseForm form, int shader) {
  switch (form) {
    case ReuseForm::kDynamic: return reuse_fn<true, false>(dedup, shader);
    case ReuseForm::kStatic: return reuse_fn<false, false>(dedup, shader);
    case ReuseForm::kSpill: return reuse_fn<false, true>(dedup, shader);
    default: break;  // kWide: instantiated for hash/phash, shaders 0 and 2 only
  }
  if (dedup == DEDUP_SORT || (shader != 0 && shader != 2)) return nullptr;
  if (dedup == DEDUP_HASH)
    return shader == 0 ? reinterpret_cast<const void*>(&reuse_kernel_wide<DEDUP_HASH, 0>)
                       : reinterpret_cast<const void*>(&reuse_kernel_wide<DEDUP_HASH, 2>);
  return shader == 0 ? reinterpret_cast<const void*>(&reuse_kernel_wide<DEDUP_PHASH, 0>)
                     : reinterpret_cast<const void*>(&reuse_kernel_wide<DEDUP_PHASH, 2>);
}

// Static batches have room for S unique vertices, yet a batch of a mesh with
// locality holds a fifth to a third of S: with rows for all of them a 768-index
// batch takes 98 KB of a block (skinning: 151 KB, one block per SM).  Here the rows
// are as many as let more blocks share an SM, at least two ninths of S (768 indices
// of a torus: 170 vertices), and the vertices past them are shaded from global
// memory into 'spill'.  700k triangles, S = 768, hash, us, all rows and these: a
// skinned torus 70 and 44, in random order 124 and 93; MVP 41 and 35, 68 and 57.
// (The hash table keeps its size: three quarters full it took up to 2.2 times as
// long on batches without locality.)  A kernel of its own: in one that never spills
// the code for it cost 2 to 8%.
bool reuse_shrink_static(DrawArgs& a, int dedup, int shader, int threads) {
  if (a.ucap < 192) return false;
  const uint32_t row = 2 * (shader == 1 ? 64u : 32u);  // both slots'
  const uint32_t fixed = reuse_layout(dedup, shader, a, (uint32_t)threads, 0, true).total + kReuseBarBytes;
  for (uint32_t n = 65536u / (64u * (uint32_t)threads); n > 1; --n) {  // blocks whose registers fit an SM
    const uint32_t room = 228u * 1024u / n - 1024u;
    if (fixed + row * (a.ucap * 2 / 9) > room) continue;
    a.row_cap = (room - fixed) / row & ~3u;
    return a.row_cap < a.ucap;
  }
  return false;
}

// The kernel splits its block into producer and consumer warps: at least two
// warps.  Sort: half of the threads sort and half consume.  Batches of no more
// indices than threads are sorted in a few stages; then a quarter consume, which is
// enough for a light shader, and five blocks of 192 threads fit an SM where four of
// 256 do -- if there are batches for them all.  700k triangles, MVP, us: S = 96 197
// in whole blocks, 172 in these; S = 255 107 and 96; but 20k triangles, S = 255 (235
// batches) 15.1 and 16.3.  1,024-key batches: no difference on 1.09M triangles with
// MVP (66), and whole blocks are faster on few triangles (envelope, 20k: 0.79 and
// 0.94 of what a loop over the network took), on vertices without locality and under
// loads.  A load of 256 steps leaves these blocks ahead (700k, S = 255: 0.91 and 0.99
// of the same), one of 1,024 does not (1.18 and 1.00).
int reuse_block_threads(int dedup, uint32_t threads, uint32_t batch_idx, uint64_t batches, uint32_t steps) {
  if (threads <= 64) return 64;
  const bool small = dedup == DEDUP_SORT && batch_idx <= std::min(threads, 256u) && batches > 304 && steps <= 256;
  return (int)(small ? threads / 4 * 3 : threads);
}

size_t reuse_smem_bytes(int dedup, int shader, const DrawArgs& a, int threads) {
  return reuse_layout(dedup, shader, a, (uint32_t)threads, a.row_cap, true).total + kReuseBarBytes;
}

constexpr size_t kMaxDynSmem = 227 * 1024;  // per block, opted in

static int blocks_per_sm(const void* fn, int threads, size_t smem) {
  if (fn == nullptr) return 0;
  // the limit is the device's, whatever this draw needs: other contexts launch the same function, and
  // launch_reuse then has nothing to set
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxDynSmem) != cudaSuccess) return 0;
  cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads, smem) != cudaSuccess) return 0;
  return nb;
}

int reuse_blocks_per_sm(int dedup, ReuseForm form, int shader, int threads, size_t smem) {
  return blocks_per_sm(reuse_kernel_ptr(dedup, form, shader), threads, smem);
}

cudaError_t launch_reuse(int dedup, ReuseForm form, const DrawArgs& a, const Uniforms& u, int shader, int threads,
                         int grid, size_t smem, cudaStream_t s) {
  const void* fn = reuse_kernel_ptr(dedup, form, shader);
  if (fn == nullptr) return cudaErrorInvalidValue;
  void* args[] = {const_cast<DrawArgs*>(&a), const_cast<Uniforms*>(&u)};
  return cudaLaunchKernel(fn, dim3(grid), dim3(threads), args, smem, s);
}

}  // namespace gp

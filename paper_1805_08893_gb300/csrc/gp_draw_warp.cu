// Statically batched warp voting (Algorithm 1, Section 3.3): one warp per
// static batch, persistent warps walking the batches with a grid stride.  The
// per-batch work is warp_vote_batch (gp_warp_body.cuh): a chain of ~10 rounds of
// votes, scattered row loads and shuffles per three batches, bound by the issue
// of its instructions and the rows' latency.  1.09M triangles, S = 96: 45 us;
// written and stored round by round, 56.  The bound of 256 threads lets the compiler
// choose 80 registers (24 warps an SM; 48 with the envelope shader): at 64 or 48 the
// spills cost more (60 us), without it the kernel takes 140 (66 us), and asking for
// three blocks an SM as well makes it spill more at the same 80 (skinning, 700k
// triangles, S = 48: 67 us against 53).
#include "gp_warp_body.cuh"

namespace gp {

template <int SH, uint32_t AHEAD>
__global__ void __launch_bounds__(256) warp_kernel(const __grid_constant__ DrawArgs a,
                                                   const __grid_constant__ Uniforms u) {
  using L = WarpSmem<SH>;
  extern __shared__ __align__(16) unsigned char smem[];
  float* palette = reinterpret_cast<float*>(smem);
  unsigned char* wbase = smem + (ShaderTraits<SH>::kSkin ? 768 * 4 : 0);
  if (ShaderTraits<SH>::kSkin) {
    for (int i = threadIdx.x; i < 768; i += blockDim.x) palette[i] = u.palette[i];
    __syncthreads();
  }
  const uint32_t S = 3u * a.static_batch_tris;
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  unsigned char* wp = wbase + warp * L::per_warp_bytes(S);

  const uint32_t warps_total = gridDim.x * (blockDim.x >> 5);
  unsigned long long inv_total = 0, batches = 0;
  WarpState<AHEAD> st;
  st.load(a, blockIdx.x * (blockDim.x >> 5) + warp, lane);
  for (uint32_t b = blockIdx.x * (blockDim.x >> 5) + warp; b < a.num_batches; b += warps_total) {
    const uint32_t inv = warp_vote_batch<SH>(a, u, palette, b, b + warps_total, wp, lane, st);
    if (lane == 0 && a.batch_inv != nullptr && b < a.batch_cap) a.batch_inv[b] = inv;
    inv_total += inv;
    batches += 1;
    __syncwarp();
  }
  st.settle(lane);  // the block's shared memory must outlive the last copy
  if (lane == 0 && batches) {
    atomicAdd(a.counters + CNT_INVOCATIONS, inv_total);
    atomicAdd(a.counters + CNT_BATCHES, batches);
  }
}

size_t warp_kernel_smem(int shader, int warps_per_block, uint32_t batch_idx) {
  uint32_t per;
  switch (shader) {
    case 0: per = WarpSmem<0>::per_warp_bytes(batch_idx); break;
    case 1: per = WarpSmem<1>::per_warp_bytes(batch_idx); break;
    case 2: per = WarpSmem<2>::per_warp_bytes(batch_idx); break;
    default: per = WarpSmem<3>::per_warp_bytes(batch_idx); break;
  }
  return (shader == 1 ? 768 * 4 : 0) + (size_t)warps_per_block * per;
}

// Batches over 96 indices: up to 256 are read ahead, in registers that would
// cost the smaller ones (7.2M triangles: S = 255 in 272 us instead of 337, but
// S = 96 in 319 instead of 291) and the envelope shader its 48 (2 to 5%).  Larger
// batches read their indices when they start; the kernel without the registers is
// the better one for them too (grid, S = 258: 32.7 us against 34.9).
constexpr uint32_t kWarpFar = 256;

template <int SH>
static const void* warp_fn(uint32_t batch_idx) {
  const bool far = batch_idx > kWarpAhead && batch_idx <= kWarpFar && SH != 2;
  return far ? reinterpret_cast<const void*>(&warp_kernel<SH, kWarpFar>)
             : reinterpret_cast<const void*>(&warp_kernel<SH, kWarpAhead>);
}

static const void* warp_kernel_ptr(int shader, uint32_t batch_idx) {
  switch (shader) {
    case 0: return warp_fn<0>(batch_idx);
    case 1: return warp_fn<1>(batch_idx);
    case 2: return warp_fn<2>(batch_idx);
    default: return warp_fn<3>(batch_idx);
  }
}

int warp_kernel_blocks_per_sm(int shader, int warps_per_block, uint32_t batch_idx) {
  const void* fn = warp_kernel_ptr(shader, batch_idx);
  const size_t smem = warp_kernel_smem(shader, warps_per_block, batch_idx);
  // (no carveout for shared memory: what the blocks leave caches the rows; 7.2M triangles, S = 96 247 us against
  // 291, S = 255 262 against 320)
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, warps_per_block * 32, smem) != cudaSuccess) return 1;
  return nb > 0 ? nb : 1;
}

cudaError_t launch_warp(const DrawArgs& a, const Uniforms& u, int shader, int warps_per_block, int grid,
                        cudaStream_t s) {
  if (3u * a.static_batch_tris > kWarpMaxBatch) return cudaErrorInvalidValue;
  if (a.num_batches == 0) return cudaSuccess;
  const size_t smem = warp_kernel_smem(shader, warps_per_block, 3u * a.static_batch_tris);
  const void* fn = warp_kernel_ptr(shader, 3u * a.static_batch_tris);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<DrawArgs*>(&a), const_cast<Uniforms*>(&u)};
  return cudaLaunchKernel(fn, dim3(grid), dim3(warps_per_block * 32), args, smem, s);
}

}  // namespace gp

// The collide-stream step with the block diagnostics fused in (lbm_step_reduce): the same
// per-node update as k_step, plus the sums that lbm_reduce would take in a second pass.
#include "lbm_cell.cuh"

namespace lbm {

// End of a fused-diagnostics CTA: each warp has written the sums of its gpw 32-node groups to
// swarp; the last warp to get here (shared-memory counter `done`, zeroed before any warp
// counts) adds the nwarps * gpw group sums in order and stores the CTA's record of 8 floats (6
// sums, 2 zeros: one 32-byte sector).  No warp waits for the others' updates.
__device__ __forceinline__ void finish_cta_record(float (*swarp)[6], unsigned& done, int lane,
                                                  int nwarps, int gpw, float* records) {
  unsigned last = 0u;
  __syncwarp();
  if (lane == 0) {
    __threadfence_block();
    last = atomicAdd(&done, 1u) == (unsigned)(nwarps - 1);
  }
  last = __shfl_sync(0xffffffffu, last, 0);
  if (last && lane < 8) {
    __threadfence_block();
    const volatile float* sv = &swarp[0][0];
    float s = 0.0f;
    if (lane < 6)
      for (int k = 0; k < nwarps * gpw; ++k) s += sv[k * 6 + lane];
    const size_t cta = blockIdx.x + (size_t)gridDim.x * (blockIdx.y + (size_t)gridDim.y * blockIdx.z);
    records[cta * 8 + lane] = s;
  }
}

// A step that also sums the diagnostics of the state it stores (lbm_step_reduce): every node
// writes its moments into its thread's shared-memory column as soon as they are known, so
// nothing is held through the collision; after the update each warp reads its nodes' six
// values back and sums them with a shuffle tree (six independent chains, a short tail at
// the end of every warp's life; neighbouring nodes first), and the last warp to finish adds the
// warps' sums in order and stores one record.  All of it in FP32 (FP64's issue rate on this
// part is a small fraction of FP32's); the records are summed in FP64 afterwards, in a fixed
// order.  Same populations, velocity and scalar as k_step.
template <typename T, int MINB, bool WALLS, bool LINEAR>
__global__ void __launch_bounds__(256, MINB) k_step_reduce(BlockView v, float* records) {
  __shared__ float snm[6][256];
  __shared__ float swarp[8][6];
  __shared__ unsigned done;
  int x, y;
  const bool in = thread_column<LINEAR>(v.nx, v.ny, x, y);
  const int z = blockIdx.z;
  const int t = threadIdx.y * blockDim.x + threadIdx.x;
  const int lane = t & 31, w = t >> 5;
#pragma unroll
  for (int i = 0; i < 6; ++i) snm[i][t] = 0.0f;
  if (t == 0) done = 0u;
  __syncthreads();                          // the counter is set before any warp counts
  const NodeMomentsOut out{&snm[0][t], 256};
  if (in) cell_update<T, uint32_t, false, WALLS, true, MINB == 3>(v, x, y, z, &out);
  __syncwarp();
  float val[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) val[i] = snm[i][t];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int i = 0; i < 6; ++i) val[i] += __shfl_xor_sync(0xffffffffu, val[i], o);
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < 6; ++i) swarp[w][i] = val[i];
  }
  finish_cta_record(swarp, done, lane, (blockDim.x * blockDim.y + 31) >> 5, 1, records);
}

// k_step_reduce with two nodes per thread (k_step2's update): the CTA covers the same bx x by
// nodes as k_step_reduce's, and thread t the nodes of its one-node threads 2t and 2t + 1, whose
// sum in the thread's column is the first stage of the one-node kernel's tree.  Four more
// stages sum both 32-node groups of the warp (2w in lanes 0-15, 2w + 1 in lanes 16-31), so the
// CTA records, and the diagnostics, are bit-identical to k_step_reduce's on the same node
// tile at less than half the tail: 12 words and 60 shuffles per lane before.
template <typename T, int MINB, bool WALLS, bool LINEAR>
__global__ void __launch_bounds__(128, MINB) k_step2_reduce(BlockView v, float* records) {
  __shared__ float snm[6][128];
  __shared__ float swarp[8][6];
  __shared__ unsigned done;
  int x, y;
  const bool in = thread_column<LINEAR>(v.nx / 2, v.ny, x, y);
  x *= 2;
  const int z = blockIdx.z;
  const int t = threadIdx.y * blockDim.x + threadIdx.x;
  const int lane = t & 31, w = t >> 5;
#pragma unroll
  for (int i = 0; i < 6; ++i) snm[i][t] = 0.0f;
  if (t == 0) done = 0u;
  __syncthreads();                          // the counter is set before any warp counts
  const NodeMomentsOut out{&snm[0][t], 128};
  if (in) {
    if constexpr (pair_corners_async<T>()) {
      __shared__ float corners[16][128];
      cell_update_pair<T, uint32_t, WALLS, true>(v, x, y, z, &corners[0][t], 128, &out);
    } else {
      cell_update_pair<T, uint32_t, WALLS, true>(v, x, y, z, nullptr, 0, &out);
    }
  }
  __syncwarp();
  float val[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) val[i] = snm[i][t];
#pragma unroll
  for (int o = 1; o < 16; o <<= 1)
#pragma unroll
    for (int i = 0; i < 6; ++i) val[i] += __shfl_xor_sync(0xffffffffu, val[i], o);
  if ((lane & 15) == 0) {
#pragma unroll
    for (int i = 0; i < 6; ++i) swarp[2 * w + (lane >> 4)][i] = val[i];
  }
  finish_cta_record(swarp, done, lane, (blockDim.x * blockDim.y + 31) >> 5, 2, records);
}

// records written by one k_step_reduce launch (one per CTA)
size_t step_reduce_ctas(const BlockView& v, int bx, int by) {
  const dim3 g = tile_grid(v.nx, v.ny, (unsigned)v.nz, bx, by);
  return (size_t)g.x * g.y * g.z;
}

// The register bound chosen for the block's step (the diagnostics add no live
// values through the collision: both bounds compile without spills).
template <typename T, int MINB, bool LINEAR>
static void launch_step_reduce_b(const BlockView& v, dim3 grid, dim3 block, float* records,
                                 cudaStream_t s) {
  if (v.walls) k_step_reduce<T, MINB, true, LINEAR><<<grid, block, 0, s>>>(v, records);
  else k_step_reduce<T, MINB, false, LINEAR><<<grid, block, 0, s>>>(v, records);
}

template <typename T>
static void launch_step_reduce_t(const BlockView& v, dim3 grid, dim3 block, int minb,
                                 float* records, cudaStream_t s) {
  if (tile_linear(v.nx, (int)block.x, (int)block.y)) launch_step_reduce_b<T, 4, true>(v, grid, block, records, s);
  else if (step_scalar_bound(minb) >= 4) launch_step_reduce_b<T, 4, false>(v, grid, block, records, s);
  else launch_step_reduce_b<T, 3, false>(v, grid, block, records, s);
}

// 128 registers (4 CTAs per SM) for both storages: 256^3 FP16 652 us per fused step against 665
// at 96, where the step alone is the faster one.
template <typename T, bool LINEAR>
static void launch_step2_reduce_b(const BlockView& v, dim3 grid, dim3 block, float* records,
                                  cudaStream_t s) {
  if (v.walls) k_step2_reduce<T, 4, true, LINEAR><<<grid, block, 0, s>>>(v, records);
  else k_step2_reduce<T, 4, false, LINEAR><<<grid, block, 0, s>>>(v, records);
}

template <typename T>
static void launch_step2_reduce_t(const BlockView& v, dim3 grid, dim3 block, float* records,
                                  cudaStream_t s) {
  if (tile_linear(v.nx / 2, (int)block.x, (int)block.y)) launch_step2_reduce_b<T, true>(v, grid, block, records, s);
  else launch_step2_reduce_b<T, false>(v, grid, block, records, s);
}

// 32-bit indexing only (27 N < 2^32): the caller checks fits_32bit_index.  A two-node bound
// code runs k_step2_reduce (same CTA grid and records) where the block allows pairs and the
// CTA is whole warps (its warp w owns the 32-node groups 2w and 2w + 1).
cudaError_t launch_step_records(const BlockView& v, int storage, int bx, int by, cudaStream_t s,
                                int minb, float* records) {
  if (step_is_pair(minb) && step_pair_ok(v, storage, bx, by) && bx * by <= 256 &&
      ((bx / 2) * by) % 32 == 0) {
    dim3 block(bx / 2, by, 1);
    const dim3 grid = tile_grid(v.nx / 2, v.ny, (unsigned)v.nz, bx / 2, by);
    if (storage == ST_FP16) launch_step2_reduce_t<__half>(v, grid, block, records, s);
    else launch_step2_reduce_t<float>(v, grid, block, records, s);
    return cudaGetLastError();
  }
  dim3 block(bx, by, 1);
  const dim3 grid = tile_grid(v.nx, v.ny, (unsigned)v.nz, bx, by);
  if (storage == ST_FP16) launch_step_reduce_t<__half>(v, grid, block, minb, records, s);
  else launch_step_reduce_t<float>(v, grid, block, minb, records, s);
  return cudaGetLastError();
}

cudaError_t launch_step_reduce(const BlockView& v, int storage, int bx, int by, cudaStream_t s,
                               int minb, float* records, const RedSink& sink) {
  const cudaError_t e = launch_step_records(v, storage, bx, by, s, minb, records);
  if (e != cudaSuccess) return e;
  return launch_reduce_records(records, step_reduce_ctas(v, bx, by), sink, s);
}

}  // namespace lbm

// Diagnostics reduction (mass, momentum, kinetic energy) over the current populations of a
// block: one pass over the 27 planes, deterministic order.
#include "lbm_internal.h"
#include "reduce_util.cuh"

namespace lbm {

template <typename T>
__global__ void __launch_bounds__(REDUCE_THREADS, 4) k_reduce(const T* d, const uint8_t* flags,
                                                              size_t N, double* partials) {
  unsigned count = 0;
  KahanF acc[5];
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < N;
       idx += (size_t)gridDim.x * blockDim.x) {
    if (flags[idx] & (F_SOLID | F_GHOST)) continue;
    float dd[27];
#pragma unroll
    for (int k = 0; k < 27; ++k) dd[k] = load_pop(d + (size_t)k * N + idx);
    float drho, jx, jy, jz;
    macros(dd, drho, jx, jy, jz);
    ++count;
    acc[0].add(drho);
    acc[1].add(jx);
    acc[2].add(jy);
    acc[3].add(jz);
    acc[4].add(0.5f * (jx * jx + jy * jy + jz * jz) / (1.0f + drho));
  }
  __shared__ double sh[REDUCE_THREADS / 32][6];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const double w = warp_sum(i == 0 ? (double)count : acc[i - 1].value());
    if (lane == 0) sh[wid][i] = w;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double s = 0;
    for (int w = 0; w < REDUCE_THREADS / 32; ++w) s += sh[w][threadIdx.x];
    partials[blockIdx.x * 6 + threadIdx.x] = s;
  }
}

// One warp per value: lane l sums partials l, l + 32, ... in order, then a fixed shuffle
// tree combines the lanes, so the result does not depend on scheduling.  out5 (optional)
// also receives the five diagnostics in the lbm_reduce layout (mass = out[0] + out[1]).
__global__ void __launch_bounds__(192) k_reduce_final(const double* partials, int n, double* out,
                                                      double* out5) {
  const int v = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double s = 0;
  for (int b = lane; b < n; b += 32) s += partials[b * 6 + v];
  s = warp_sum(s);
  if (lane == 0) out[v] = s;
  if (out5 != nullptr) {
    __syncthreads();
    if (threadIdx.x < 5) out5[threadIdx.x] = threadIdx.x == 0 ? out[0] + out[1] : out[threadIdx.x + 1];
  }
}

// n records of 8 floats (6 sums + 2 unused), summed in FP64 in a fixed order in one launch: warp v
// of CTA s sums value v over slice s of the records (lane l: records l, l + 32, ... in order,
// then the shuffle tree) into stage[s * 6 + v], and the last CTA to finish (a device counter,
// which it resets) sums the slices the same way.  The FP64 adds bound it (an SM issues one for a
// warp in about 16 cycles), so a slice has 256 records until there are RED_SLICES of them, and
// no thread adds anything but its own lane's sum.  One launch in place of two, half the record
// bytes, and the results and the error word go to pinned memory without a copy of their own.
__global__ void __launch_bounds__(192) k_reduce_records(const float* __restrict__ rec, size_t n,
                                                        RedSink k) {
  __shared__ double sh[6];
  __shared__ unsigned last;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const size_t per = (n + gridDim.x - 1) / gridDim.x;
  const size_t lo = per * blockIdx.x, hi = lo + per < n ? lo + per : n;
  double s = 0;
#pragma unroll 8
  for (size_t i = lo + lane; i < hi; i += 32) s += (double)__ldg(rec + (8 * i + w));
  s = warp_sum(s);
  if (lane == 0) {
    k.stage[blockIdx.x * 6 + w] = s;
    __threadfence();
  }
  __syncthreads();
  if (t == 0) last = atomicAdd(k.counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  double x = 0;
#pragma unroll 4
  for (int i = lane; i < (int)gridDim.x; i += 32) x += __ldcg(k.stage + (i * 6 + w));
  x = warp_sum(x);
  if (lane == 0) {
    sh[w] = x;
    k.out[w] = x;
    if (k.host6) k.host6[w] = x;
  }
  __syncthreads();
  if (k.out5 && t < 5) k.out5[t] = t == 0 ? sh[0] + sh[1] : sh[t + 1];
  if (t == 32) *k.counter = 0u;
  if (t == 64 && k.host_err) *k.host_err = *k.err;
}

cudaError_t launch_reduce_records(const float* records, size_t n, const RedSink& sink, cudaStream_t s) {
  const size_t slices = (n + 255) / 256;
  const unsigned g = (unsigned)(slices < 1 ? 1 : slices < RED_SLICES ? slices : RED_SLICES);
  k_reduce_records<<<g, 192, 0, s>>>(records, n, sink);
  return cudaGetLastError();
}

// Diagnostics of many domains in one launch (lbm_reduce_batch): a list of chunks, each of
// one member's nodes; every CTA takes chunks in turn (per-thread compensated FP32 sums, FP64
// across the CTA, in the order of k_reduce) and writes one record of 8 doubles per chunk.
template <typename T>
__global__ void __launch_bounds__(REDUCE_THREADS) k_reduce_items(const RedItem* items, int n_items,
                                                                 const RedMember* members,
                                                                 double* records) {
  __shared__ double sh[REDUCE_THREADS / 32][6];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int w = blockIdx.x; w < n_items; w += gridDim.x) {
    const RedItem it = items[w];
    const RedMember m = members[it.member];
    const T* d = static_cast<const T*>(m.f);
    unsigned count = 0;
    KahanF acc[5];
    for (size_t idx = it.start + threadIdx.x; idx < it.start + it.len; idx += blockDim.x) {
      if (m.flags[idx] & (F_SOLID | F_GHOST)) continue;
      float dd[27];
#pragma unroll
      for (int k = 0; k < 27; ++k) dd[k] = load_pop(d + (size_t)k * m.N + idx);
      float drho, jx, jy, jz;
      macros(dd, drho, jx, jy, jz);
      ++count;
      acc[0].add(drho);
      acc[1].add(jx);
      acc[2].add(jy);
      acc[3].add(jz);
      acc[4].add(0.5f * (jx * jx + jy * jy + jz * jz) / (1.0f + drho));
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const double v = warp_sum(i == 0 ? (double)count : acc[i - 1].value());
      if (lane == 0) sh[wid][i] = v;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
      double s = 0;
      for (int k = 0; k < REDUCE_THREADS / 32; ++k) s += sh[k][threadIdx.x];
      records[(size_t)w * 8 + threadIdx.x] = s;
    }
    __syncthreads();
  }
}

// One warp per member: its chunks' records (contiguous in the list) in order, then the
// shuffle tree; the member's device error word rides along in slot 6.
__global__ void __launch_bounds__(256) k_reduce_items_final(const double* records,
                                                            const RedMember* members, int n,
                                                            double* out) {
  const int m = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (m >= n) return;
  const RedMember mb = members[m];
  for (int v = 0; v < 6; ++v) {
    double s = 0;
    for (int c = lane; c < mb.n_items; c += 32) s += records[(size_t)(mb.first_item + c) * 8 + v];
    s = warp_sum(s);
    if (lane == 0) out[(size_t)m * 8 + v] = s;
  }
  if (lane == 0) out[(size_t)m * 8 + 6] = (double)*mb.err;
}

cudaError_t launch_reduce_items(int storage, const RedItem* items, int n_items,
                                const RedMember* members, int n_members, double* records,
                                double* out, cudaStream_t s) {
  const int ctas = n_items < REDUCE_CTAS ? n_items : REDUCE_CTAS;
  if (storage == ST_FP16)
    k_reduce_items<__half><<<ctas, REDUCE_THREADS, 0, s>>>(items, n_items, members, records);
  else
    k_reduce_items<float><<<ctas, REDUCE_THREADS, 0, s>>>(items, n_items, members, records);
  k_reduce_items_final<<<(n_members + 7) / 8, 256, 0, s>>>(records, members, n_members, out);
  return cudaGetLastError();
}

cudaError_t launch_reduce(const void* d, int storage, const uint8_t* flags, size_t N,
                          double* partials, double* out, cudaStream_t s, double* out5) {
  const size_t want = (N + REDUCE_THREADS - 1) / REDUCE_THREADS;
  const int ctas = (int)(want < (size_t)REDUCE_CTAS ? (want > 0 ? want : 1) : REDUCE_CTAS);
  if (storage == ST_FP16)
    k_reduce<__half><<<ctas, REDUCE_THREADS, 0, s>>>((const __half*)d, flags, N, partials);
  else
    k_reduce<float><<<ctas, REDUCE_THREADS, 0, s>>>((const float*)d, flags, N, partials);
  k_reduce_final<<<1, 192, 0, s>>>(partials, ctas, out, out5);
  return cudaGetLastError();
}

}  // namespace lbm

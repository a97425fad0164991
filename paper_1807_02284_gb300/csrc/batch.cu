// Batched stepping of many independent single-block domains of uneven sizes.
//
// Every member takes its own collide-stream launches (k_step / k_step2, or the diagnostics form
// in the last step), with the launch shape its size calls for; the members' steps are forked
// over a few streams, balanced by their nodes, and the whole call is captured in a CUDA graph.
// Members do not depend on one another, so while one member's last CTAs drain, the other
// branches' launches fill the SMs, and no step waits for the slowest member: one persistent
// kernel over all members with a device-wide barrier per step did, and held 128 registers, since
// a member's view came from memory instead of the constant bank (64 plumes of edges 24 to 96,
// uploads, diagnostics and reads: 31.2 ms a pass against 21.7; a new set's first call 57 against
// 23 ms).
// Every node runs the same cell_update as a domain stepped on its own, so results are
// bit-identical to that.
//
// The bounded device-wide barrier below (a wait that expires sets the TIMEOUT bit instead of
// hanging the GPU) is used by its self-test alone; no step waits on the device.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include "lbm_cell.cuh"
#include "reduce_util.cuh"
#include "runtime.h"

namespace lbm {

struct BarrierState {
  unsigned int count;
  unsigned int gen;
};

// Device-wide barrier with a bounded wait.  Returns false when the wait gave up.
__device__ __forceinline__ bool grid_barrier(BarrierState* bs, unsigned int nblocks, int* err,
                                             long long limit) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned int* vgen = &bs->gen;
    const unsigned int g = *vgen;
    __threadfence();
    const unsigned int arrived = atomicAdd(&bs->count, 1u);
    if (arrived == nblocks - 1) {
      atomicExch(&bs->count, 0u);
      __threadfence();
      atomicAdd(&bs->gen, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == g) {
        if (clock64() - t0 > limit) {
          atomicOr(err, 8);
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// The six sums of every member over its CTA records of the diagnostics step (8 floats each),
// one CTA per member, one warp per value: lane l takes records l, l + 32, ... in order, then the
// shuffle tree; the member's device error word rides along in slot 6.
__global__ void __launch_bounds__(192) k_batch_records(const float* __restrict__ records,
                                                       const RedMember* __restrict__ members,
                                                       double* __restrict__ out) {
  const RedMember m = members[blockIdx.x];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const float* rec = records + (size_t)m.first_item * 8 + w;
  double s = 0;
#pragma unroll 8
  for (int i = lane; i < m.n_items; i += 32) s += (double)__ldg(rec + (size_t)i * 8);
  s = warp_sum(s);
  if (lane == 0) out[(size_t)blockIdx.x * 8 + w] = s;
  if (threadIdx.x == 0) out[(size_t)blockIdx.x * 8 + 6] = (double)*m.err;
}

// One captured call: the launches of a set of domains from a given assignment of time levels
// over at most kGraphSteps steps.
struct BatchPlan {
  std::vector<unsigned long long> serials;   // members (domain serials, in call order)
  std::vector<int> curs;
  int steps = 0;
  cudaGraphExec_t exec = nullptr;
  // fused diagnostics (lbm_step_batch_reduce): per-CTA records, per-member sums (sums and
  // error word, 8 doubles each) copied to pinned host memory by the same graph
  bool red = false;
  std::vector<int> first;       // each member's first record
  float* records = nullptr;
  RedMember* members = nullptr;
  double* out_dev = nullptr;
  double* out_host = nullptr;
  double* out5_dev = nullptr;   // lbm_step_batch_reduce_async: 5 values per member
};

// Plans cached by the first domain of a batch.  A call with an odd step count flips every
// member's current level, so alternating calls need two plans, and a long call takes whole
// graphs and a rest; a few more cover a caller that alternates between batches.  Members are
// matched by serial, never by address, so a plan never refers to a destroyed domain's memory
// once it is chosen.
struct BatchCache {
  std::vector<BatchPlan*> plans;   // most recently used last
};
constexpr size_t kMaxBatchPlans = 8;
constexpr int kGraphSteps = 16;      // even: a whole graph ends in the levels it started from
constexpr int kBatchStreams = 32;

}  // namespace lbm

using namespace lbm;

static void free_plan(lbm_domain* dom, BatchPlan* p) {
  if (p->exec) cudaGraphExecDestroy(p->exec);
  if (p->records) dom->dev_free(p->records);
  if (p->members) dom->dev_free(p->members);
  if (p->out_dev) dom->dev_free(p->out_dev);
  if (p->out5_dev) dom->dev_free(p->out5_dev);
  if (p->out_host) cudaFreeHost(p->out_host);
  delete p;
}

// The diagnostics buffers of a plan: one record per CTA of every member's last step, the
// members' record ranges and error words, the per-member sums on the device and in pinned host
// memory.
static lbm_status add_red_buffers(lbm_domain* const* doms, int n, BatchPlan* p) {
  lbm_domain* d0 = doms[0];
  std::vector<RedMember> hm(n);
  p->first.resize(n);
  size_t at = 0;
  for (int i = 0; i < n; ++i) {
    const Block& B = doms[i]->blocks[0];
    const size_t cnt = step_reduce_ctas(doms[i]->view(0, B.cur, B.cur ^ 1), B.bx, B.by);
    hm[i] = RedMember{nullptr, nullptr, doms[i]->d_err, B.N, (int)at, (int)cnt};
    p->first[i] = (int)at;
    at += cnt;
  }
  if (at > (size_t)INT32_MAX) return d0->fail(LBM_ERR_UNSUPPORTED, "batch too large for one diagnostics pass");
  p->records = static_cast<float*>(d0->dev_alloc(at * 8 * sizeof(float)));
  p->members = static_cast<RedMember*>(d0->dev_alloc((size_t)n * sizeof(RedMember)));
  p->out_dev = static_cast<double*>(d0->dev_alloc((size_t)n * 8 * sizeof(double)));
  p->out5_dev = static_cast<double*>(d0->dev_alloc((size_t)n * 5 * sizeof(double)));
  if (!p->records || !p->members || !p->out_dev || !p->out5_dev)
    return d0->fail(LBM_ERR_OOM, "batch diagnostics buffers");
  if (cudaMallocHost(&p->out_host, (size_t)n * 8 * sizeof(double)) != cudaSuccess) {
    p->out_host = nullptr;
    return d0->fail(LBM_ERR_OOM, "batch diagnostics staging");
  }
  cudaError_t e = cudaMemcpyAsync(p->members, hm.data(), (size_t)n * sizeof(RedMember),
                                  cudaMemcpyHostToDevice, d0->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(d0->stream);
  if (e != cudaSuccess) return d0->cuda_fail(e, "batch diagnostics upload");
  p->red = true;
  return LBM_OK;
}

// Step k (0-based) of member i on stream s; the plan's last step writes the member's records.
static cudaError_t enqueue_member(lbm_domain* const* doms, const BatchPlan* p, int i, int k,
                                  cudaStream_t s) {
  const lbm_domain* d = doms[i];
  const Block& B = d->blocks[0];
  const int from = p->curs[i] ^ (k & 1);
  const BlockView v = d->view(0, from, from ^ 1);
  if (p->red && k == p->steps - 1)
    return launch_step_records(v, d->desc.storage, B.bx, B.by, s, B.minb,
                               p->records + (size_t)p->first[i] * 8);
  return launch_step(v, d->desc.storage, B.bx, B.by, s, B.minb);
}

static cudaError_t enqueue_sums(const BatchPlan* p, cudaStream_t s) {
  const int n = (int)p->serials.size();
  k_batch_records<<<n, 192, 0, s>>>(p->records, p->members, p->out_dev);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return cudaMemcpyAsync(p->out_host, p->out_dev, (size_t)n * 8 * sizeof(double),
                         cudaMemcpyDeviceToHost, s);
}

// The launches of a plan: members largest first onto the least loaded of a few branches, each
// branch step by step over its members, forked from and joined into s.
static cudaError_t enqueue_batch(lbm_domain* const* doms, const BatchPlan* p, cudaStream_t s) {
  lbm_domain* d0 = doms[0];
  const int n = (int)p->serials.size();
  const int nb = std::min(n, kBatchStreams);
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    return doms[a]->blocks[0].N > doms[b]->blocks[0].N;
  });
  std::vector<std::vector<int>> branch(nb);
  std::vector<size_t> load(nb, 0);
  for (int i : order) {
    const int b = (int)(std::min_element(load.begin(), load.end()) - load.begin());
    branch[b].push_back(i);
    load[b] += doms[i]->blocks[0].N;
  }
  cudaError_t e = cudaEventRecord(d0->event(0), s);
  for (int b = 0; b < nb && e == cudaSuccess; ++b) {
    cudaStream_t bs = b == 0 ? s : d0->post_stream(b);
    if (b) e = cudaStreamWaitEvent(bs, d0->event(0), 0);
    for (int k = 0; k < p->steps && e == cudaSuccess; ++k)
      for (size_t m = 0; m < branch[b].size() && e == cudaSuccess; ++m)
        e = enqueue_member(doms, p, branch[b][m], k, bs);
    if (b && e == cudaSuccess) e = cudaEventRecord(d0->event(b), bs);
  }
  for (int b = 1; b < nb && e == cudaSuccess; ++b) e = cudaStreamWaitEvent(s, d0->event(b), 0);
  if (e == cudaSuccess && p->red) e = enqueue_sums(p, s);
  return e;
}

void release_batch_plan(lbm_domain* dom) {
  BatchCache* c = static_cast<BatchCache*>(dom->batch_plan);
  if (!c) return;
  for (BatchPlan* p : c->plans) free_plan(dom, p);
  delete c;
  dom->batch_plan = nullptr;
}

// Captures the plan's launches, on a stream of the library's own: the members' stream may be one
// that cannot be captured (the legacy default stream), the graph runs on any.
static void capture_plan(lbm_domain* const* doms, BatchPlan* p) {
  cudaStream_t s = doms[0]->post_stream(0);
  cudaGraph_t g = nullptr;
  if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
    const cudaError_t e1 = enqueue_batch(doms, p, s);
    const cudaError_t e2 = cudaStreamEndCapture(s, &g);
    if (e1 == cudaSuccess && e2 == cudaSuccess && g && cudaGraphInstantiate(&p->exec, g, 0) != cudaSuccess)
      p->exec = nullptr;
    if (g) cudaGraphDestroy(g);
  }
  cudaGetLastError();  // a capture the driver refused leaves the direct launches
}

// The plan of `steps` (at most kGraphSteps) steps from the members' current levels, from the
// cache or captured now.  `own`: the caller is capturing the members' stream itself, where no plan
// is captured and none is kept (a call after the capture would find it without a graph): the plan
// is left in *own for this call alone.
static lbm_status batch_plan(lbm_domain* const* doms, int n, int steps, bool red, BatchPlan* own,
                             BatchPlan** out) {
  lbm_domain* d0 = doms[0];
  BatchCache* cache = static_cast<BatchCache*>(d0->batch_plan);
  if (!cache) {
    cache = new (std::nothrow) BatchCache();
    if (!cache) return d0->fail(LBM_ERR_OOM, "out of host memory");
    d0->batch_plan = cache;
  }
  for (size_t k = 0; k < cache->plans.size(); ++k) {
    BatchPlan* q = cache->plans[k];
    bool same = q->steps == steps && q->red == red && (int)q->serials.size() == n;
    for (int i = 0; i < n && same; ++i)
      same = q->serials[i] == doms[i]->serial && q->curs[i] == doms[i]->blocks[0].cur;
    if (same) {
      cache->plans.erase(cache->plans.begin() + k);
      cache->plans.push_back(q);
      *out = q;
      return LBM_OK;
    }
  }
  // the fork's streams and events exist before a capture
  const int nb = std::min(n, kBatchStreams);
  if (!d0->event(nb)) return d0->fail(LBM_ERR_CUDA, "cudaEventCreate");
  if (!d0->post_stream(nb - 1)) return d0->fail(LBM_ERR_CUDA, "cudaStreamCreate");
  const bool keep = !own || red;
  BatchPlan* p = keep ? new (std::nothrow) BatchPlan() : own;
  if (!p) return d0->fail(LBM_ERR_OOM, "out of host memory");
  p->steps = steps;
  p->serials.resize(n);
  p->curs.resize(n);
  for (int i = 0; i < n; ++i) {
    p->serials[i] = doms[i]->serial;
    p->curs[i] = doms[i]->blocks[0].cur;
  }
  if (!keep) {
    *out = p;
    return LBM_OK;
  }
  if (red) {
    const lbm_status st = add_red_buffers(doms, n, p);
    if (st != LBM_OK) { free_plan(d0, p); return st; }
  }
  capture_plan(doms, p);
  while (cache->plans.size() >= kMaxBatchPlans) {
    // a replaced plan's last launch may still be running; its buffers go back to the allocator
    if (cudaStreamSynchronize(d0->stream) != cudaSuccess) cudaGetLastError();
    free_plan(d0, cache->plans.front());
    cache->plans.erase(cache->plans.begin());
  }
  cache->plans.push_back(p);
  *out = p;
  return LBM_OK;
}

// Per-member sums (8 doubles: 6 sums, the member's error word, unused) to the 5 diagnostics of
// the lbm_reduce layout, and every member's error bits into the first domain's error word.
__global__ void k_batch_combine(const double* __restrict__ sums, int n, double* __restrict__ out5,
                                int* err0) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n) return;
  const double* r = sums + 8 * (size_t)m;
  double* o = out5 + 5 * (size_t)m;
  o[0] = r[0] + r[1];
  o[1] = r[2];
  o[2] = r[3];
  o[3] = r[4];
  o[4] = r[5];
  const int e = (int)r[6];
  if (e) atomicOr(err0, e);
}

// ticket != nullptr: lbm_step_batch_reduce_async (the values go to out on the stream).
static lbm_status step_batch(lbm_domain* const* doms, int32_t n, int32_t steps, double* out,
                             int64_t* ticket = nullptr) {
  if (!doms || n <= 0 || !doms[0]) return LBM_ERR_INVALID_ARG;
  lbm_domain* d0 = doms[0];
  cudaSetDevice(d0->desc.device);
  const bool red = out != nullptr;
  if (steps < 0) return d0->fail(LBM_ERR_INVALID_ARG, "negative step count");
  if (red && steps < 1) return d0->fail(LBM_ERR_INVALID_ARG, "lbm_step_batch_reduce needs at least one step");
  for (int i = 0; i < n; ++i) {
    if (!doms[i]) return d0->fail(LBM_ERR_INVALID_ARG, "null domain in batch");
    for (int j = 0; j < i; ++j)
      if (doms[j] == doms[i]) return d0->fail(LBM_ERR_INVALID_ARG, "a domain appears twice");
    if (doms[i]->blocks.size() != 1) return d0->fail(LBM_ERR_UNSUPPORTED, "batched domains must be single-block");
    if (doms[i]->desc.storage != d0->desc.storage) return d0->fail(LBM_ERR_INVALID_ARG, "mixed storage in batch");
    if (doms[i]->desc.device != d0->desc.device) return d0->fail(LBM_ERR_INVALID_ARG, "mixed devices in batch");
    if (doms[i]->tape) return d0->fail(LBM_ERR_UNSUPPORTED, "batched stepping does not record tapes");
    if (doms[i]->walls) return d0->fail(LBM_ERR_UNSUPPORTED, "batched domains cannot have wall faces");
    if (!fits_32bit_index(doms[i]->blocks[0].N))
      return d0->fail(LBM_ERR_UNSUPPORTED, "batched domains must have 27 N < 2^32");
    if (*doms[i]->h_err & 1) return d0->fail(LBM_ERR_DIVERGED, "a domain of the batch has diverged");
  }
  if (steps == 0) return LBM_OK;
  cudaStream_t s = d0->stream;
  // whole graphs, then the rest (with the diagnostics in its last step).  Both plans before the
  // first launch: a call that cannot have them leaves every domain as it was.  (A whole graph ends
  // in the levels it started from, so one plan serves all of them and the rest starts there too.)
  const int rest_steps = (steps - 1) % kGraphSteps + 1, n_whole = (steps - rest_steps) / kGraphSteps;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) cudaGetLastError();
  const bool callers = cap != cudaStreamCaptureStatusNone;
  BatchPlan own_whole, own_rest, *whole = nullptr, *p = nullptr;
  if (n_whole > 0) {
    const lbm_status st = batch_plan(doms, n, kGraphSteps, false, callers ? &own_whole : nullptr, &whole);
    if (st != LBM_OK) return st;
  }
  {
    const lbm_status st = batch_plan(doms, n, rest_steps, red, callers ? &own_rest : nullptr, &p);
    if (st != LBM_OK) return st;
  }
  // order the batch after pending work of every domain, and every domain after the batch
  std::vector<cudaEvent_t> evs;
  for (int i = 1; i < n; ++i) {
    if (doms[i]->stream == s) continue;
    cudaEvent_t ev;
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) break;
    cudaEventRecord(ev, doms[i]->stream);
    cudaStreamWaitEvent(s, ev, 0);
    evs.push_back(ev);
  }
  for (cudaEvent_t ev : evs) cudaEventDestroy(ev);

  cudaError_t e = cudaSuccess;
  for (int k = 0; k <= n_whole && e == cudaSuccess; ++k) {
    const BatchPlan* q = k < n_whole ? whole : p;
    e = q->exec ? cudaGraphLaunch(q->exec, s) : enqueue_batch(doms, q, s);
    if (e != cudaSuccess) break;
    for (int i = 0; i < n; ++i) {
      Block& B = doms[i]->blocks[0];
      if (q->steps & 1) B.cur ^= 1;
      doms[i]->steps += q->steps;
    }
  }
  // every domain's stream waits for the batch (each node reports divergence into its own
  // domain's error word)
  cudaEvent_t done;
  if (cudaEventCreateWithFlags(&done, cudaEventDisableTiming) == cudaSuccess) {
    cudaEventRecord(done, s);
    for (int i = 1; i < n; ++i)
      if (doms[i]->stream != s) cudaStreamWaitEvent(doms[i]->stream, done, 0);
    cudaEventDestroy(done);
  }
  if (e != cudaSuccess) return d0->cuda_fail(e, "batched launch");
  if (!red) {
    d0->post_error_probe();
    return LBM_OK;
  }
  if (ticket) {
    const int slot = (int)(d0->results_issued % lbm_domain::kResultSlots);
    if (!d0->result_ev[slot] &&
        cudaEventCreateWithFlags(&d0->result_ev[slot], cudaEventDisableTiming) != cudaSuccess) {
      d0->result_ev[slot] = nullptr;
      return d0->fail(LBM_ERR_CUDA, "cudaEventCreate");
    }
    k_batch_combine<<<(n + 63) / 64, 64, 0, s>>>(p->out_dev, n, p->out5_dev, d0->d_err);
    e = cudaGetLastError();
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(out, p->out5_dev, (size_t)n * 5 * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) {
      d0->post_error_probe();
      e = cudaEventRecord(d0->result_ev[slot], s);
    }
    if (e != cudaSuccess) return d0->cuda_fail(e, "batch diagnostics read-back");
    *ticket = ++d0->results_issued;
    return LBM_OK;
  }
  e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return d0->cuda_fail(e, "cudaStreamSynchronize");
  lbm_status first = LBM_OK;
  for (int i = 0; i < n; ++i) {
    const double* r = p->out_host + 8 * (size_t)i;
    double* o = out + 5 * (size_t)i;
    o[0] = r[0] + r[1];
    o[1] = r[2];
    o[2] = r[3];
    o[3] = r[4];
    o[4] = r[5];
    *doms[i]->h_err = (int)r[6];
    const lbm_status st = doms[i]->error_status();
    if (st != LBM_OK && first == LBM_OK) first = st;
  }
  return first;
}

extern "C" lbm_status lbm_step_batch(lbm_domain* const* doms, int32_t n, int32_t steps) {
  return step_batch(doms, n, steps, nullptr);
}

extern "C" lbm_status lbm_step_batch_reduce(lbm_domain* const* doms, int32_t n, int32_t steps,
                                            double* out) {
  if (!out) return LBM_ERR_INVALID_ARG;
  return step_batch(doms, n, steps, out);
}

extern "C" lbm_status lbm_step_batch_reduce_async(lbm_domain* const* doms, int32_t n,
                                                  int32_t steps, double* out, int64_t* ticket) {
  if (!out || !ticket) return LBM_ERR_INVALID_ARG;
  return step_batch(doms, n, steps, out, ticket);
}

// Self-test of the bounded device barrier: a cooperative kernel waits for `extra` more CTAs
// than it launched, so every wait runs out after about `limit_ms`; the expected result is
// LBM_ERR_TIMEOUT with the context still usable.
__global__ void k_barrier_selftest(BarrierState* bs, unsigned int expected, int* err,
                                   long long limit) {
  grid_barrier(bs, expected, err, limit);
}

extern "C" lbm_status lbm_barrier_selftest(int32_t extra, double limit_ms, void* cuda_stream) {
  if (extra < 0 || !(limit_ms > 0.0) || limit_ms > 5000.0) return LBM_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  BarrierState* bs = nullptr;
  int* err = nullptr;
  if (cudaMalloc(&bs, sizeof(BarrierState)) != cudaSuccess) return LBM_ERR_OOM;
  if (cudaMalloc(&err, sizeof(int)) != cudaSuccess) { cudaFree(bs); return LBM_ERR_OOM; }
  int dev = 0, clock_khz = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&clock_khz, cudaDevAttrClockRate, dev);
  const long long limit = (long long)(limit_ms * (clock_khz > 0 ? clock_khz : 2000000));
  cudaMemsetAsync(bs, 0, sizeof(BarrierState), s);
  cudaMemsetAsync(err, 0, sizeof(int), s);
  const int grid = 4;
  const unsigned int expected = (unsigned)(grid + extra);
  void* args[] = {(void*)&bs, (void*)&expected, (void*)&err, (void*)&limit};
  cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_barrier_selftest, dim3(grid),
                                              dim3(32), args, 0, s);
  int h = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(bs);
  cudaFree(err);
  if (e != cudaSuccess) return LBM_ERR_CUDA;
  return (h & 8) ? LBM_ERR_TIMEOUT : LBM_OK;
}

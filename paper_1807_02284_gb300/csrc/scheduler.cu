// Step scheduling of a domain (Algorithm 1) and the small host utilities around it.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "runtime.h"

using namespace lbm;

namespace lbm {
// Captured step graphs, keyed by the starting assignment of time levels (the `cur` level of
// every block) and the number of reference steps: `chunk`-step graphs (a multiple of the period
// after which the level assignment repeats, so they end in the assignment they started from),
// one-step graphs of continuous-scale domains, and shorter runs of small single blocks.  They
// hold level pointers and launch parameters only, so they outlive lbm_init_macro and
// lbm_write_field; whatever changes a launch (blocks, walls, a tape) drops them.
struct GraphCache {
  struct Entry {
    std::vector<int> cur;
    int steps;
    cudaGraphExec_t exec;      // null: seen once, not captured yet
  };
  std::vector<Entry> entries;
  int chunk = 0;
};
constexpr size_t kMaxStepGraphs = 96;

// Level assignment after one reference step (mirrors the schedule of multiscale_step).
static std::vector<int> next_levels(const std::vector<lbm::Block>& blocks, std::vector<int> cur) {
  cur[0] ^= 1;
  for (size_t b = 1; b < blocks.size(); ++b) {
    if (blocks[b].far) {     // far-field blocks ping-pong like the reference block
      cur[b] ^= 1;
      continue;
    }
    const int L = cur[b], A = (L + 1) % 3, B = (L + 2) % 3;
    int c = L;
    for (int j = 1; j <= blocks[b].substeps; ++j) c = (j == 1) ? A : (c == A ? B : A);
    cur[b] = c;
  }
  return cur;
}
}  // namespace lbm

// Launch shape of a block's collide-stream kernel, from its extents, storage and walls.  Figures:
// us per step on GB300, one node per thread / two.
void lbm_domain::pick_tiles(int b) {
  Block& B = blocks[b];
  if (B.tile_forced) return;
  const bool half = desc.storage == LBM_FP16_SHIFTED;
  // Two nodes per thread once the block is bound by bandwidth or issue rather than by latency:
  // from 2^20 nodes (96^3 40.8 / 42.5, FP16 40.0 / 41.2; 128^3 91 / 84, FP16 96 / 80; 256^3 702 /
  // 629, FP16 718 / 592).  Beside other blocks' kernels or with wall faces from 2^22 (steps of a
  // domain with a refined block: 128^3 148 / 152, 150^3 209 / 212, 160^3 235 / 234, 176^3 294 /
  // 286, 192^3 356 / 343; in a far-field block the two are within 1 % from 144^3 to 192^3; wall
  // faces: 128^3 97 / 97, 160^3 182 / 180, 176^3 243 / 232, 192^3 307 / 288).  With
  // obstacle-surface walls from 2^24: a warp that holds a surface node goes through the collision
  // three times, and with two nodes per thread twice as many nodes go with it, so it depends on
  // the surface (sphere of radius 0.15 edges: 128^3 95 / 116, 176^3 243 / 278, 224^3 487 / 547,
  // 256^3 716 / 740, 320^3 1386 / 1419, 384 x 256 x 384 1600 / 1528; 0.09 edges: 160^3 180 / 192,
  // 192^3 304 / 302, 256^3 709 / 686, 320^3 1371 / 1283; FP16 alike).
  const bool surfaces = (walls & WALLS_OBSTACLES) && !B.far;
  const size_t pairs_from = (size_t)1 << (surfaces ? 24 : walls || blocks.size() > 1 ? 22 : 20);
  if (B.nx % 2 == 0 && B.N >= pairs_from) {
    // tiles of 64 x 2 nodes on whole rows, one-row CTAs running on over ragged ones (two nodes per
    // thread, 224 x 250 x 190: FP32 410 us against 431 with 64 x 2 tiles, FP16 386 against 428)
    const bool tiles = B.nx % 64 == 0;
    B.bx = tiles ? 64 : 128;
    B.by = tiles ? 2 : 1;
    B.minb = STEP_PAIR + (half ? 5 : 4);
  } else if (B.nx <= 32) {
    // latency-bound: a warp per row keeps the faces in warps of their own, 80 registers take
    // cell_update's EARLY loads (12^3 3.8 us against 4.6 with one-row CTAs, 20^3 3.6 against 4.6,
    // 24^3 2.9 against 4.0, 32^3 3.5 against 3.8, 28 x 60 x 60 6.7 against 7.7; not on larger
    // blocks of shorter rows, whose idle lanes count: 12 x 60 x 60 6.3 against 5.1,
    // 16 x 128 x 128 21.5 against 12.9)
    B.bx = 32;
    B.by = 4;
    B.minb = 3;
  } else if (B.nx % 32 == 0) {
    B.bx = 32;                           // 64^3 11.3 us, 96^3 40.8 (with EARLY loads 11.6, 41.5)
    B.by = 4;
    B.minb = 4;
  } else {
    // ragged rows: no idle lanes (72 x 60 x 51 10.7 us against 12.5 with the best tile,
    // 97 x 61 x 75 21.7 against 25.8, 201 x 181 x 171 281 against 299)
    B.bx = 128;
    B.by = 1;
    B.minb = 4;
  }
  if (const char* env = std::getenv("LBM_TILE")) {  // "bx,by[,minb]" forces a launch shape
    int bx = 0, by = 0, mb = 3;
    const int n = std::sscanf(env, "%d,%d,%d", &bx, &by, &mb);
    const bool mb_ok = mb == 3 || mb == 4 || (mb >= STEP_PAIR + 4 && mb <= STEP_PAIR + 6);
    if (n >= 2 && bx > 0 && by > 0 && bx * by <= 256 && bx % 32 == 0 && mb_ok) {
      B.bx = bx;
      B.by = by;
      B.minb = mb;
      B.tile_forced = true;
    }
  }
}

void lbm_domain::invalidate_graphs() {
  if (!graphs) return;
  for (auto& en : graphs->entries)
    if (en.exec) cudaGraphExecDestroy(en.exec);
  delete graphs;
  graphs = nullptr;
}

void release_tape(lbm_domain* dom);        // adjoint.cu
void release_batch_plan(lbm_domain* dom);  // batch.cu

lbm_status lbm_domain::aux(cudaStream_t* out) {
  if (!aux_stream) {
    cudaError_t e = cudaStreamCreateWithFlags(&aux_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) { aux_stream = nullptr; return cuda_fail(e, "cudaStreamCreate"); }
  }
  *out = aux_stream;
  return LBM_OK;
}

cudaEvent_t lbm_domain::event(int i) {
  while ((int)events.size() <= i) {
    cudaEvent_t ev = nullptr;
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    events.push_back(ev);
  }
  return events[i];
}

cudaStream_t lbm_domain::post_stream(int k) {
  while ((int)post_streams.size() <= k) {
    cudaStream_t st = nullptr;
    if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
    post_streams.push_back(st);
  }
  return post_streams[k];
}

void lbm_domain::release_extras() {
  invalidate_graphs();
  release_batch_plan(this);
  if (rb_dev) dev_free(rb_dev);
  rb_dev = nullptr;
  rb_dev_bytes = 0;
  if (rb_host) cudaFreeHost(rb_host);
  rb_host = nullptr;
  rb_host_bytes = 0;
  if (ib_done) cudaEventSynchronize(ib_done);
  if (ib_dev) dev_free(ib_dev);
  ib_dev = nullptr;
  ib_dev_bytes = 0;
  if (ib_host) cudaFreeHost(ib_host);
  ib_host = nullptr;
  ib_host_bytes = 0;
  if (ib_done) cudaEventDestroy(ib_done);
  ib_done = nullptr;
  for (cudaEvent_t ev : events) cudaEventDestroy(ev);
  events.clear();
  for (cudaStream_t st : post_streams) cudaStreamDestroy(st);
  post_streams.clear();
  if (aux_stream) cudaStreamDestroy(aux_stream);
  aux_stream = nullptr;
  release_tape(this);
  if (small_host) cudaFreeHost(small_host);
  small_host = nullptr;
  if (small_done) cudaEventDestroy(small_done);
  small_done = nullptr;
  for (cudaEvent_t& ev : result_ev) {
    if (ev) cudaEventDestroy(ev);
    ev = nullptr;
  }
}

// Small host arrays (inflow records) go through a pinned buffer that the kernel reads in place
// (a copy to the device first was one more operation per call, 1.7 us on the GPU and about 4 of
// host time, for at most some tens of KB), so the caller can reuse its array on return;
// small_used() after the launch marks when the buffer is free again.
const void* lbm_domain::stage_small(const void* src, size_t bytes, lbm_status* st) {
  *st = LBM_OK;
  if (small_done) cudaEventSynchronize(small_done);   // the previous reader has left the buffer
  if (bytes > small_bytes) {
    if (small_host) cudaFreeHost(small_host);
    small_host = nullptr;
    small_bytes = 0;       // no buffer until the allocation below succeeds
    size_t cap = std::max<size_t>(bytes, 4096);
    if (cudaMallocHost(&small_host, cap) != cudaSuccess) {
      small_host = nullptr;
      *st = fail(LBM_ERR_OOM, "pinned allocation failed");
      return nullptr;
    }
    small_bytes = cap;
  }
  if (!small_done && cudaEventCreateWithFlags(&small_done, cudaEventDisableTiming) != cudaSuccess) {
    small_done = nullptr;
    *st = fail(LBM_ERR_CUDA, "cudaEventCreate");
    return nullptr;
  }
  std::memcpy(small_host, src, bytes);
  return small_host;
}

lbm_status lbm_domain::small_used() {
  const cudaError_t e = cudaEventRecord(small_done, stream);
  return e == cudaSuccess ? LBM_OK : cuda_fail(e, "cudaEventRecord");
}

void lbm_domain::on_state_reset(int b) {
  (void)b;
  steps = 0;
  release_tape(this);
}

lbm_status tape_before_step(lbm_domain* dom);  // adjoint.cu
lbm_status multiscale_step(lbm_domain* dom);  // coupling.cu

// n reference steps launched one kernel at a time.
lbm_status lbm_domain::advance_direct(int n) {
  for (int i = 0; i < n; ++i) {
    lbm_status st = tape_before_step(this);
    if (st != LBM_OK) return st;
    if (blocks.size() == 1) {
      Block& B = blocks[0];
      const int nxt = B.cur ^ 1;
      cudaError_t e = launch_step(view(0, B.cur, nxt), desc.storage, B.bx, B.by, stream, B.minb);
      if (e != cudaSuccess) return cuda_fail(e, "collide-stream launch");
      B.cur = nxt;
    } else {
      st = multiscale_step(this);
      if (st != LBM_OK) return st;
    }
    ++steps;
  }
  return LBM_OK;
}

// n reference steps as one graph launch, captured on the first such call from this level
// assignment (`eager`), or on the second (a run that may never come again).  *done = false:
// nothing was launched (a run that needs no graph is also left to the caller's launches on a stream
// that cannot be captured, such as the legacy default stream).
lbm_status lbm_domain::advance_graph(int n, bool eager, bool* done) {
  *done = false;
  std::vector<int> key(blocks.size());
  for (size_t b = 0; b < blocks.size(); ++b) key[b] = blocks[b].cur;
  GraphCache::Entry* en = nullptr;
  for (auto& e : graphs->entries)
    if (e.steps == n && e.cur == key) en = &e;
  if (!en) {
    if (graphs->entries.size() >= kMaxStepGraphs) return LBM_OK;
    graphs->entries.push_back({key, n, nullptr});
    en = &graphs->entries.back();
    if (!eager) return LBM_OK;
  }
  if (!en->exec) {
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess && !eager) {
      cudaGetLastError();
      return LBM_OK;
    }
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamBeginCapture");
    lbm_status st = LBM_OK;
    for (int i = 0; i < n && st == LBM_OK; ++i) {
      if (blocks.size() == 1) {
        Block& B = blocks[0];
        const cudaError_t el = launch_step(view(0, B.cur, B.cur ^ 1), desc.storage, B.bx, B.by, stream, B.minb);
        if (el != cudaSuccess) st = cuda_fail(el, "collide-stream launch");
        B.cur ^= 1;
      } else {
        st = multiscale_step(this);
      }
    }
    const cudaError_t e2 = cudaStreamEndCapture(stream, &g);
    for (size_t b = 0; b < blocks.size(); ++b) blocks[b].cur = key[b];
    if (st != LBM_OK || e2 != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      return st != LBM_OK ? st : cuda_fail(e2, "step graph capture");
    }
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
    en->exec = exec;
  }
  const cudaError_t e = cudaGraphLaunch(en->exec, stream);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch");
  std::vector<int> s = key;
  for (int i = 0; i < n; ++i) s = next_levels(blocks, s);
  for (size_t b = 0; b < blocks.size(); ++b) blocks[b].cur = s[b];
  steps += n;
  *done = true;
  return LBM_OK;
}

// Without a tape: whole chunks from chunk graphs; the rest of a continuous-scale domain step by
// step from one-step graphs (the schedule of one step is 16 launches with forks and joins on
// several streams; replaying it as one graph leaves the GPU no gaps between them), the rest
// of a small single block (up to 2^18 nodes, 3 steps or more) from a graph of its length once it
// has come twice, of a larger one launch by launch.  A graph has smaller gaps between steps and
// one call for the host: 4 steps one after another 32^3 30.5 -> 24.1 us, 64^3 62.6 -> 53.4.  The
// limit is no crossover: larger blocks gain less but gain too (80^3 122.7 -> 112.6, 96^3 181.5 ->
// 172.6, 128^3 357 -> 347); it keeps the graphs of every run length to blocks where they matter.
lbm_status lbm_domain::advance(int n) {
  if (blocks.size() > 1) {  // stream and events of the fork/join schedule exist before capture
    cudaStream_t a = nullptr;
    lbm_status st = aux(&a);
    if (st != LBM_OK) return st;
    if (!event(10 + 3 * (int)blocks.size())) return fail(LBM_ERR_CUDA, "cudaEventCreate");
    if (!post_stream((int)blocks.size())) return fail(LBM_ERR_CUDA, "cudaStreamCreate");
  }
  if (tape != nullptr) return advance_direct(n);
  if (!graphs) {
    std::vector<int> start(blocks.size());
    for (size_t b = 0; b < blocks.size(); ++b) start[b] = blocks[b].cur;
    int period = 1;
    std::vector<int> s = next_levels(blocks, start);
    while (s != start && period < 64) { s = next_levels(blocks, s); ++period; }
    if (s != start) return advance_direct(n);
    graphs = new GraphCache();
    graphs->chunk = period * ((16 + period - 1) / period);
  }
  const int chunk = graphs->chunk;
  const bool multi = blocks.size() > 1;
  bool ok = true;
  if (n >= 2 * chunk)
    while (n >= chunk && ok) {
      const lbm_status st = advance_graph(chunk, true, &ok);
      if (st != LBM_OK) return st;
      if (ok) n -= chunk;
    }
  if (multi) {
    ok = true;
    while (n > 0 && ok) {
      const lbm_status st = advance_graph(1, true, &ok);
      if (st != LBM_OK) return st;
      if (ok) --n;
    }
  } else if (n >= 3 && blocks[0].N <= (size_t)1 << 18) {
    // (a caller that captures the domain's stream itself gets the launches)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
      const int run = std::min(n, chunk);
      const lbm_status st = advance_graph(run, false, &ok);
      if (st != LBM_OK) return st;
      if (ok) n -= run;
    } else {
      cudaGetLastError();
    }
  }
  return advance_direct(n);
}

// lbm_step_reduce: n reference steps whose last one (on a single-block domain with 32-bit
// indexing) also sums the diagnostics of the state it stores, so that reading mass, momentum
// and energy back after a step costs no second pass over the populations.  Other domains
// take the n steps and lbm_reduce of block 0.
// Enqueues n steps and the diagnostics of block 0's new state: the 6 sums into dom->d_red,
// the 5 combined values into out5 (device, may be null), the 6 sums into h_red (`to_host`)
// and the error word into h_err.  On a single-block domain with 27 N < 2^32 the last step's
// own kernel sums them; otherwise a separate reduction follows.
static lbm_status enqueue_step_reduce(lbm_domain* dom, int32_t n, double* out5, bool to_host) {
  Block& B = dom->blocks[0];
  if (dom->blocks.size() > 1 || !fits_32bit_index(B.N)) {
    lbm_status st = dom->advance(n);
    if (st != LBM_OK) return st;
    cudaError_t e = launch_reduce(B.lv[B.cur].f, dom->desc.storage, B.flags, B.N,
                                  dom->d_partials, dom->d_red, dom->stream, out5);
    if (e == cudaSuccess && to_host)
      e = cudaMemcpyAsync(dom->h_red, dom->d_red, 6 * sizeof(double), cudaMemcpyDeviceToHost, dom->stream);
    if (e != cudaSuccess) return dom->cuda_fail(e, "reduce");
    dom->post_error_probe();
    return LBM_OK;
  }
  lbm_status st = dom->advance(n - 1);
  if (st == LBM_OK) st = tape_before_step(dom);
  if (st != LBM_OK) return st;
  const int nxt = B.cur ^ 1;
  const BlockView v = dom->view(0, B.cur, nxt);
  const size_t ctas = step_reduce_ctas(v, B.bx, B.by);
  if (ctas > dom->step_records_n) {
    if (dom->d_step_records) dom->dev_free(dom->d_step_records);
    dom->step_records_n = 0;
    dom->d_step_records = static_cast<float*>(
        dom->dev_alloc(6 * RED_SLICES * sizeof(double) + ctas * 8 * sizeof(float)));
    if (!dom->d_step_records) return dom->fail(LBM_ERR_OOM, "step-reduce records");
    dom->step_records_n = ctas;
  }
  RedSink sink;
  sink.out = dom->d_red;
  sink.out5 = out5;
  sink.host6 = to_host ? dom->h_red : nullptr;
  sink.err = dom->d_err;
  sink.host_err = dom->h_err;
  sink.stage = reinterpret_cast<double*>(dom->d_step_records);
  sink.counter = reinterpret_cast<unsigned*>(dom->d_err + 8);
  float* records = dom->d_step_records + 2 * 6 * RED_SLICES;
  const cudaError_t e = launch_step_reduce(v, dom->desc.storage, B.bx, B.by, dom->stream, B.minb,
                                           records, sink);
  if (e != cudaSuccess) return dom->cuda_fail(e, "collide-stream launch");
  B.cur = nxt;
  ++dom->steps;
  return LBM_OK;
}

lbm_status lbm_step_reduce(lbm_domain* dom, int32_t n, double out[5]) {
  if (!dom) return LBM_ERR_INVALID_ARG;
  cudaSetDevice(dom->desc.device);
  if (n < 1) return dom->fail(LBM_ERR_INVALID_ARG, "lbm_step_reduce needs at least one step");
  if (!out) return dom->fail(LBM_ERR_INVALID_ARG, "null output");
  if (*dom->h_err & 1) return dom->fail(LBM_ERR_DIVERGED, "divergence recorded by an earlier step");
  lbm_status st = enqueue_step_reduce(dom, n, nullptr, true);
  if (st != LBM_OK) return st;
  const cudaError_t e = cudaStreamSynchronize(dom->stream);
  if (e != cudaSuccess) return dom->cuda_fail(e, "cudaStreamSynchronize");
  st = dom->error_status();
  const double* r = dom->h_red;
  out[0] = r[0] + r[1];
  out[1] = r[2];
  out[2] = r[3];
  out[3] = r[4];
  out[4] = r[5];
  return st;
}

lbm_status lbm_step_reduce_async(lbm_domain* dom, int32_t n, double out[5], int64_t* ticket) {
  if (!dom) return LBM_ERR_INVALID_ARG;
  cudaSetDevice(dom->desc.device);
  if (n < 1) return dom->fail(LBM_ERR_INVALID_ARG, "lbm_step_reduce_async needs at least one step");
  if (!out || !ticket) return dom->fail(LBM_ERR_INVALID_ARG, "null output or ticket");
  if (*dom->h_err & 1) return dom->fail(LBM_ERR_DIVERGED, "divergence recorded by an earlier step");
  const int slot = (int)(dom->results_issued % lbm_domain::kResultSlots);
  if (!dom->result_ev[slot] &&
      cudaEventCreateWithFlags(&dom->result_ev[slot], cudaEventDisableTiming) != cudaSuccess) {
    dom->result_ev[slot] = nullptr;
    return dom->fail(LBM_ERR_CUDA, "cudaEventCreate");
  }
  double* d_out5 = dom->d_red + 8;
  lbm_status st = enqueue_step_reduce(dom, n, d_out5, false);
  if (st != LBM_OK) return st;
  cudaError_t e = cudaMemcpyAsync(out, d_out5, 5 * sizeof(double), cudaMemcpyDeviceToHost,
                                  dom->stream);
  if (e == cudaSuccess) e = cudaEventRecord(dom->result_ev[slot], dom->stream);
  if (e != cudaSuccess) return dom->cuda_fail(e, "reduce read-back");
  *ticket = ++dom->results_issued;
  return LBM_OK;
}

lbm_status lbm_wait_results(lbm_domain* dom, int64_t ticket) {
  if (!dom) return LBM_ERR_INVALID_ARG;
  cudaSetDevice(dom->desc.device);
  if (ticket < 1 || ticket > dom->results_issued)
    return dom->fail(LBM_ERR_INVALID_ARG, "not a ticket of lbm_step_reduce_async on this domain");
  const int slot = (int)((ticket - 1) % lbm_domain::kResultSlots);
  const cudaError_t e = cudaEventSynchronize(dom->result_ev[slot]);
  if (e != cudaSuccess) return dom->cuda_fail(e, "cudaEventSynchronize");
  return dom->error_status();
}

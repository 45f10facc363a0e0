// Many independent problems in one launch: each problem is a matrix (its own
// handle) and a population, as produced by many EBIC runs or restarts side by
// side (Step 4 of the "EBIC Algorithm" section, repeated over problems).
//
// A persistent kernel (one grid that fills the GPU) pulls work items --
// (problem, series, part of the series' rows) -- from a list ordered by
// decreasing estimated cost (longest-processing-time first), so that the
// long, heavy series start early and short ones fill the gaps.  A problem with a
// pair table is evaluated from it, any other from the fp32 columns.  Where all have
// tables, a walk of its own overlaps the chain of an item (claim, offsets, columns,
// first words, result) with the next one's; else the items run the single-problem
// kernels' code.  The launch (counter reset + kernel) can be captured once as a
// CUDA graph and replayed.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <functional>
#include <vector>

#include "ebic_internal.cuh"
#include "ebic_support.cuh"

namespace ebic {

struct BatchProb {
  const float* A_c;
  const uint32_t* LT;
  const double* LN;
  int* err;
  int32_t R, C, R_pad, W;
  CbfPop pop;
  EvalArgs a;
  int32_t path;          // EBIC_PATH_GATHER or EBIC_PATH_BITMASK
  int32_t vpi, ipc;      // vectors per part, parts per series
  uint32_t* scratch;     // split accumulators of this problem (2 x 64-bit per series)
};

constexpr int kBatchThreads = 256;
// 16-byte vectors a bitmask item walks at most: the most that leaves the grid
// kBatchItems items a warp (whole series in the 64-problem batch: 312 us, against
// 328 us at 256 vectors, 365 at 128, 413 at 64: a part repeats the set-up).
constexpr int kBatchVecs[] = {4096, 512, 256, 128, 64};
constexpr long long kBatchItems = 6;
constexpr int32_t kMaxCostLen = EBIC_MAX_EVAL_LEN;      // longest series a cost tells apart

// The result of an item whose atomic (split series) or log-table load (whole
// series) is still in flight; lane 0 writes it out one item later.
struct BatchPend {
  int32_t prob, sid, L;            // prob -1: none
  uint32_t cnt;
  unsigned long long old;          // split: the series' word before this part
                                   // whole: the bits of LN[cnt - 1]
};

__device__ __forceinline__ void batch_finish(const BatchProb* __restrict__ probs, BatchPend& p) {
  if (p.prob < 0) return;
  const BatchProb& pb = probs[p.prob];
  if (pb.ipc > 1) {
    if ((uint32_t)(p.old >> 32) == (uint32_t)pb.ipc - 1) {
      reinterpret_cast<unsigned long long*>(pb.scratch)[2 * (size_t)p.sid] = 0ull;
      finish_series(pb.a, pb.LN, p.sid, (uint32_t)p.old + p.cnt, 0u, p.L);
    }
  } else {
    double f = 0.0;
    if (p.cnt > 1) {
      int64_t e = (int64_t)p.cnt - (int64_t)pb.a.sigma;
      e = e > 0 ? 0 : (e < -2000 ? -2000 : e);
      f = __dmul_rn(ldexp(__longlong_as_double((long long)p.old), (int)e), (double)p.L);
    }
    pb.a.inc[p.sid] = p.cnt;
    pb.a.fit[p.sid] = f;
  }
  p.prob = -1;
}

// Bitmask items.  A warp's time is a chain of round trips -- claim, work entry,
// offsets, columns, table rows, ticket -- of which only the table rows need be
// waited for: the claim is taken two items ahead, the next item's work entry
// and offsets are read while this one's columns and first rows are in flight,
// and the result is written out one item later.  Two vectors a lane (64 of the
// part at a time) keep eight row loads in flight.  The first four AND steps are
// needed whole (a block of iid rows keeps about 128 / (t + 1)! of them after t
// steps), the next two are read together, and only then whole batches again:
// eight steps at a time read 1.65 times the bytes the early exit allows.
// NV: vectors a lane; one, with five CTAs an SM instead of three, where no problem
// has more than 32 (36 problems of 327 to 3,479 rows: 42.7 us instead of 45).
template <int NV>
__global__ void __launch_bounds__(kBatchThreads, NV == 1 ? 5 : 3)
k_support_batch(const BatchProb* __restrict__ probs, const int2* __restrict__ work,
                long long n_items, unsigned long long* __restrict__ counter) {
  const int lane = threadIdx.x & 31;
  const uint4 ones = make_uint4(kFull, kFull, kFull, kFull), zeros = make_uint4(0u, 0u, 0u, 0u);
  // A warp's first two items follow from its place (the heaviest spread over the
  // CTAs), the others are claimed from the counter behind them: claims of all
  // warps at once, on one address, delay a small batch by 4 us.
  const long long warps = (long long)gridDim.x * (kBatchThreads / 32);
  const long long item = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  if (item >= n_items) return;                           // warp-uniform
  long long raw = item + warps;                          // lane 0: the claim in flight
  int2 w = work[item];
  int32_t o_begin, o_end;
  {
    const BatchProb& pb = probs[w.x];
    const int32_t sid = w.y / pb.ipc;
    o_begin = pb.pop.offsets[sid];
    o_end = pb.pop.offsets[sid + 1];
  }
  BatchPend pend;
  pend.prob = -1;
  for (;;) {
    const BatchProb& pb = probs[w.x];
    const int32_t ipc = pb.ipc, sid = w.y / ipc, part = w.y % ipc;
    const int64_t begin = o_begin;
    const int32_t L = o_end - o_begin;
    const bool in = o_begin >= 0 && o_end <= pb.pop.total && L >= 1 && L <= EBIC_MAX_EVAL_LEN;
    const uint32_t C = (uint32_t)pb.C;
    // the first 32 steps' columns, and the next item's work entry
    uint32_t x = 0, y = 0;
    if (in) {
      if (lane < L) x = (uint32_t)pb.pop.cols[begin + lane];
      if (lane + 1 < L) y = (uint32_t)pb.pop.cols[begin + lane + 1];
    }
    const long long next = __shfl_sync(kFull, raw, 0);
    const bool more = next < n_items;                    // warp-uniform
    int2 wn = make_int2(0, 0);
    if (more) {
      wn = work[next];
      if (lane == 0) raw = 2 * warps + (long long)atomicAdd(counter, 1ull);
    }
    int32_t n_begin = 0, n_end = 0;
    auto read_next = [&]() {                             // its offsets
      if (!more) return;
      const BatchProb& pn = probs[wn.x];
      const int32_t ns = wn.y / pn.ipc;
      n_begin = pn.pop.offsets[ns];
      n_end = pn.pop.offsets[ns + 1];
    };
    bool lb = false;
    if (in) {
      lb = (lane < L && x >= C) || (lane + 1 < L && y >= C);
      for (int t = lane + 32; t < L; t += 32) lb |= (uint32_t)pb.pop.cols[begin + t] >= C;
    }
    const bool bad = __any_sync(kFull, lb) || !in;
    const int32_t nsteps = bad ? 0 : L - 1;
    const int32_t V = pb.W >> 2;
    const int32_t v_lo = part * pb.vpi, v_hi = min(v_lo + pb.vpi, V);
    const uint4* LT4 = reinterpret_cast<const uint4*>(pb.LT);
    const uint32_t first = x * C + y;                  // pair index of step `lane`
    uint32_t cnt = 0;
    bool ahead = false;
    for (int32_t vb = v_lo; vb < v_hi && nsteps > 0; vb += 32 * NV) {
      uint4 m[NV];
      bool on[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        on[k] = vb + lane + 32 * k < v_hi;
        m[k] = on[k] ? ones : zeros;
      }
      bool alive = true;                               // warp-uniform
      for (int32_t w0 = 0; alive && w0 < nsteps; w0 += 32) {
        uint32_t pi = first;
        if (w0 > 0 && w0 + lane < nsteps)
          pi = (uint32_t)pb.pop.cols[begin + w0 + lane] * C +
               (uint32_t)pb.pop.cols[begin + w0 + lane + 1];
        const int32_t wn_steps = min(32, nsteps - w0);
        for (int32_t t = 0; alive && t < wn_steps;) {
          const int32_t lim = min(t == 4 && w0 == 0 ? 2 : 4, wn_steps - t);
          bool live[NV];
          uint4 r[4][NV];
#pragma unroll
          for (int k = 0; k < NV; ++k) live[k] = nz4(m[k]);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint32_t p = __shfl_sync(kFull, pi, (t + u) & 31);
#pragma unroll
            for (int k = 0; k < NV; ++k)
              r[u][k] = live[k] && u < lim
                            ? ld_table(LT4 + (size_t)p * (uint32_t)V + (uint32_t)(vb + lane + 32 * k))
                            : ones;
          }
          if (!ahead) {
            ahead = true;
            read_next();
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int k = 0; k < NV; ++k) m[k] = and4(m[k], r[u][k]);
          alive = __any_sync(kFull, nz4(m[0]) || nz4(m[NV - 1]));
          t += lim;
        }
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) cnt += popc4(m[k]);
    }
    if (!ahead) read_next();
    cnt = __reduce_add_sync(kFull, cnt);
    if (!bad && L == 1 && part == 0) cnt = (uint32_t)pb.R;
    if (lane == 0) {
      if (bad) atomicOr(pb.err, 1);
      batch_finish(probs, pend);
      pend.prob = w.x;
      pend.sid = sid;
      pend.L = bad ? 1 : L;
      pend.cnt = cnt;
      if (ipc > 1)
        pend.old = atomicAdd(reinterpret_cast<unsigned long long*>(pb.scratch) + 2 * (size_t)sid,
                             (1ull << 32) | (unsigned long long)cnt);
      else if (cnt > 1)
        pend.old = (unsigned long long)__double_as_longlong(pb.LN[cnt - 1]);
    }
    if (!more) break;
    w = wn;
    o_begin = n_begin;
    o_end = n_end;
  }
  if (lane == 0) batch_finish(probs, pend);
}

// Batches with a problem that has no table, by the single-problem kernels' code: a
// gather item is long, so a warp claims one only when it is free, and neighbouring
// claims, which read the same columns, fall to one CTA.  Four CTAs an SM: 64 problems
// of up to 50,000 rows without tables 2,904 us, with half the tables 1,357, against
// 3,437 and 2,566 with items claimed ahead as above, 3,693 and 1,683 at three CTAs,
// 3,358 and 1,510 with first items spread over the CTAs; 12 of up to 20,000 rows,
// half the tables, 157 against 186, 156 and 172.
__global__ void __launch_bounds__(kBatchThreads, 4)
k_support_batch_any(const BatchProb* __restrict__ probs, const int2* __restrict__ work,
                    long long n_items, unsigned long long* __restrict__ counter) {
  const int lane = threadIdx.x & 31;
  for (;;) {
    unsigned long long i = 0;
    if (lane == 0) i = atomicAdd(counter, 1ull);
    i = __shfl_sync(kFull, i, 0);
    if ((long long)i >= n_items) break;                  // warp-uniform
    const int2 w = work[i];
    const BatchProb& pb = probs[w.x];
    const int32_t ipc = pb.ipc;
    const int32_t sid = w.y / ipc, part = w.y % ipc;
    if (pb.path == EBIC_PATH_BITMASK)
      bitmask_warp_item<false, true, 1, 8, CbfPop>(pb.LT, pb.C, pb.W, pb.R, pb.pop, pb.a, pb.vpi, ipc,
                                                   pb.scratch, pb.LN, pb.err, sid, part, lane);
    else
      gather_item<false, true, CbfPop>(pb.A_c, pb.C, pb.R_pad, pb.R, pb.pop, pb.a, pb.vpi, ipc,
                                       pb.scratch, pb.LN, pb.err, sid, part, lane);
  }
}

}  // namespace ebic

struct ebic_batch_ctx {
  int device = 0;
  int32_t n = 0;
  int32_t flags = 0;
  std::vector<ebic::BatchProb> probs;
  std::vector<long long> items_per_prob;
  ebic::DevBuf d_probs, d_work, d_scratch, d_counter;
  long long n_items = 0;
  int grid = 0;
  void (*kernel)(const ebic::BatchProb*, const int2*, long long, unsigned long long*) = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaGraph_t graph = nullptr;
  cudaStream_t own = nullptr;   // blocking stream used when the caller passes none
};

namespace ebic {

// Time of a problem without a table at one part size (fp32 vectors; 0: whole
// series), by the single-problem kernel, whose per-item code the batch runs.
static ebic_status time_parts(ebic_ctx* h, const ebic_batch_item_t& it, int32_t vpp, cudaStream_t s,
                              float* us) {
  if (vpp <= 0) vpp = (h->R_pad / 4 + 31) / 32 * 32;
  const int32_t saved_path = h->path;
  const ebic_eval_tuning_t saved = h->tuning;
  h->path = EBIC_PATH_GATHER;
  h->tuning = ebic_eval_tuning_t{};
  h->tuning.vecs_per_part_gather = vpp;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  ebic_status st = ebic_eval_population_dev(h, it.d_offsets, it.d_cols, it.P, it.total_cols,
                                            it.sigma, EBIC_SUPPORT_INC, it.d_inc, nullptr,
                                            it.d_fitness, s);
  cudaEventRecord(e0, s);
  for (int r = 0; r < 3 && st == EBIC_OK; ++r)
    st = ebic_eval_population_dev(h, it.d_offsets, it.d_cols, it.P, it.total_cols, it.sigma,
                                  EBIC_SUPPORT_INC, it.d_inc, nullptr, it.d_fitness, s);
  cudaEventRecord(e1, s);
  float ms = 1e30f;
  if (st == EBIC_OK && cudaEventSynchronize(e1) == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  h->path = saved_path;
  h->tuning = saved;
  *us = ms * 1000.f / 3.f;
  return st;
}

// Vectors per part (rounded to warps) and parts per series, as the
// single-problem launch computes them for a forced part size.
static void split_for(int32_t V, int32_t vpp, int32_t* vpi, int32_t* ipc) {
  if (vpp <= 0 || vpp >= V) {
    *vpi = ((V + 31) / 32) * 32;
    *ipc = 1;
    return;
  }
  *vpi = std::max(vpp / 32, 1) * 32;
  *ipc = (V + *vpi - 1) / *vpi;
}

}  // namespace ebic

using namespace ebic;

extern "C" {

ebic_status ebic_batch_create(const ebic_handle* handles, const ebic_batch_item_t* items,
                              int32_t n, int32_t flags, void* stream, ebic_batch* out) {
  if (!handles || !items || !out || n < 1) return fail(EBIC_ERR_ARG, "bad batch arguments");
  const int dev = handles[0] ? handles[0]->device : -1;
  for (int32_t i = 0; i < n; ++i) {
    if (!handles[i]) return fail(EBIC_ERR_ARG, "null handle %d", i);
    if (handles[i]->device != dev) return fail(EBIC_ERR_ARG, "handles on different devices");
    const ebic_batch_item_t& it = items[i];
    if (it.P < 1 || it.P > (1 << 24) || !it.d_offsets || !it.d_cols || !it.d_inc ||
        !it.d_fitness || it.total_cols < 0)
      return fail(EBIC_ERR_ARG, "bad batch item %d", i);
  }
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != dev) cudaSetDevice(dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  ebic_batch_ctx* b = new ebic_batch_ctx();
  b->device = dev;
  b->n = n;
  b->flags = flags;
  if (cudaStreamCreate(&b->own) != cudaSuccess) {
    cudaGetLastError();
    delete b;
    if (prev >= 0 && prev != dev) cudaSetDevice(prev);
    return fail(EBIC_ERR_CUDA, "cannot create the batch stream");
  }
  ebic_status st = EBIC_OK;
  auto fin = [&](ebic_status r) {
    if (r != EBIC_OK) ebic_batch_free(b);
    if (prev >= 0 && prev != dev) cudaSetDevice(prev);
    return r;
  };

  // Per problem: path and split.  With EBIC_BATCH_BUILD_TABLES the pair
  // table is built where it fits (half the free memory, cumulative); with
  // EBIC_BATCH_AUTOTUNE a few part sizes of the problems without one are timed.
  // A problem with a table takes it: the batch's walk over it is level with the
  // columns at the smallest problems and ahead of them everywhere else (one and
  // sixteen problems from 100 x 5 to 200,000 x 20, 1 to 4,000 series: 0.98 to 40
  // times as fast).
  size_t free_b = 0, total_b = 0;
  cudaMemGetInfo(&free_b, &total_b);
  size_t budget = free_b / 2;
  b->probs.resize((size_t)n);
  size_t scratch_words = 0;
  std::vector<size_t> scratch_off((size_t)n);
  for (int32_t i = 0; i < n; ++i) {
    ebic_ctx* h = handles[i];
    const ebic_batch_item_t& it = items[i];
    if ((flags & EBIC_BATCH_BUILD_TABLES) && !h->LT) {
      const size_t need = (size_t)h->C * h->C * h->W * sizeof(uint32_t);
      if (need <= budget) {
        if ((st = build_pair_table(h, s)) != EBIC_OK) return fin(st);
        budget -= need;
      }
    }
    int32_t best_vpp = 0;
    if ((flags & EBIC_BATCH_AUTOTUNE) && !h->LT) {
      float best = 1e30f;
      for (int32_t vpp : {32, 64, 128, 256, 512, 0}) {
        if (vpp > 0 && vpp / 2 >= h->R_pad / 4) continue;
        float us = 0.f;
        if ((st = time_parts(h, it, vpp, s, &us)) != EBIC_OK) return fin(st);
        if (us < best) {
          best = us;
          best_vpp = vpp;
        }
      }
    }
    BatchProb& pb = b->probs[(size_t)i];
    pb.A_c = h->A_c;
    pb.LT = h->LT;
    pb.LN = h->LN;
    pb.err = h->d_err;
    pb.R = h->R;
    pb.C = h->C;
    pb.R_pad = h->R_pad;
    pb.W = h->W;
    pb.pop = CbfPop{it.d_offsets, it.d_cols, it.total_cols};
    pb.a = EvalArgs{};
    pb.a.P = it.P;
    pb.a.sigma = it.sigma;
    pb.a.mode = EBIC_SUPPORT_INC;
    pb.a.want_dec = 0;
    pb.a.inc = it.d_inc;
    pb.a.dec = nullptr;
    pb.a.fit = it.d_fitness;
    pb.a.lnf = nullptr;
    pb.path = h->LT ? EBIC_PATH_BITMASK : EBIC_PATH_GATHER;
    split_for(h->R_pad / 4, best_vpp, &pb.vpi, &pb.ipc);   // (problems without a table)
  }
  // The launch: its kernel and grid, then the part size of the bitmask problems
  // (a batch has series enough to fill the grid).
  bool gather = false, narrow = true;
  for (const BatchProb& pb : b->probs)
    if (pb.path != EBIC_PATH_BITMASK) gather = true;
    else if (pb.W / 4 > 32) narrow = false;
  b->kernel = gather ? k_support_batch_any : narrow ? k_support_batch<1> : k_support_batch<2>;
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, b->kernel, kBatchThreads, 0);
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  b->grid = std::max(1, per_sm) * std::max(1, sms);
  auto parts_at = [](const BatchProb& pb, int32_t cap) {
    return (pb.W / 4 + cap - 1) / cap;
  };
  int32_t cap = 0;
  for (int32_t c : kBatchVecs) {
    cap = c;
    long long items_at = 0;
    for (const BatchProb& pb : b->probs)
      items_at += (long long)pb.a.P * (pb.path == EBIC_PATH_BITMASK ? parts_at(pb, c) : pb.ipc);
    if (items_at >= kBatchItems * b->grid * (kBatchThreads / 32)) break;
  }
  for (int32_t i = 0; i < n; ++i) {
    const ebic_batch_item_t& it = items[i];
    BatchProb& pb = b->probs[(size_t)i];
    if (pb.path == EBIC_PATH_BITMASK) {
      const int32_t V = pb.W / 4, parts = parts_at(pb, cap);
      split_for(V, ((V + parts - 1) / parts + 31) / 32 * 32, &pb.vpi, &pb.ipc);
    }
    if ((long long)it.P * pb.ipc >= (1ll << 31))
      return fin(fail(EBIC_ERR_ARG, "problem %d: too many work items", i));
    scratch_off[(size_t)i] = scratch_words;
    scratch_words += (pb.ipc > 1 ? (size_t)it.P * 4 : 0);   // 2 x 64-bit words per series
  }
  // scratch for split series
  if ((st = b->d_scratch.reserve_zeroed(std::max<size_t>(scratch_words, 4) * sizeof(uint32_t), s)) !=
      EBIC_OK)
    return fin(st);
  for (int32_t i = 0; i < n; ++i)
    b->probs[(size_t)i].scratch = b->d_scratch.as<uint32_t>() + scratch_off[(size_t)i];

  // work list, longest estimated cost first: cost = (L - 1) x vectors of the part,
  // equal costs in the order of problems, series and parts.  A problem has few
  // different costs -- one for full parts and one for last ones at each length --
  // so the items are counted and placed by cost (a batch of 16 problems of 600
  // series, 22,800 items, is made in 540 us; 720 with a comparison sort of them).
  std::vector<std::vector<int32_t>> len((size_t)n);
  for (int32_t i = 0; i < n; ++i) {
    const ebic_batch_item_t& it = items[i];
    std::vector<int32_t> off((size_t)it.P + 1);
    if (cudaMemcpy(off.data(), it.d_offsets, off.size() * sizeof(int32_t),
                   cudaMemcpyDeviceToHost) != cudaSuccess) {
      cudaGetLastError();
      return fin(fail(EBIC_ERR_CUDA, "reading offsets of problem %d", i));
    }
    // (the offsets are checked on the device: a length here is only an estimate)
    for (int32_t sid = 0; sid < it.P; ++sid)
      off[(size_t)sid] = std::clamp(off[(size_t)sid + 1] - off[(size_t)sid], 1, kMaxCostLen);
    off.resize((size_t)it.P);
    len[(size_t)i] = std::move(off);
  }
  auto cost_of = [](const BatchProb& pb, int32_t L, bool last) {
    const int32_t V = pb.path == EBIC_PATH_BITMASK ? pb.W / 4 : pb.R_pad / 4;
    const float unit = pb.path == EBIC_PATH_BITMASK ? 1.f : 32.f;   // bytes per row-step / 16
    const int32_t vecs = last ? V - (pb.ipc - 1) * pb.vpi : pb.vpi;
    return unit * (float)std::max(L - 1, 1) * (float)vecs;
  };
  std::vector<float> costs;                              // the different ones, descending
  for (int32_t i = 0; i < n; ++i) {
    std::vector<bool> seen((size_t)kMaxCostLen + 1, false);
    for (int32_t L : len[(size_t)i]) {
      if (seen[(size_t)L]) continue;
      seen[(size_t)L] = true;
      for (bool last : {false, true}) costs.push_back(cost_of(b->probs[(size_t)i], L, last));
    }
  }
  std::sort(costs.begin(), costs.end(), std::greater<float>());
  costs.erase(std::unique(costs.begin(), costs.end()), costs.end());
  // each(rank of the cost, item) over all items, in order
  auto for_items = [&](auto each) {
    std::vector<int32_t> rank(2 * ((size_t)kMaxCostLen + 1));
    for (int32_t i = 0; i < n; ++i) {
      const BatchProb& pb = b->probs[(size_t)i];
      std::fill(rank.begin(), rank.end(), -1);
      auto rank_of = [&](int32_t L, bool last) {
        int32_t& r = rank[2 * (size_t)L + (last ? 1 : 0)];
        if (r < 0)
          r = (int32_t)(std::lower_bound(costs.begin(), costs.end(), cost_of(pb, L, last),
                                         std::greater<float>()) - costs.begin());
        return (size_t)r;
      };
      for (int32_t sid = 0; sid < pb.a.P; ++sid) {
        const int32_t L = len[(size_t)i][(size_t)sid];
        for (int32_t q = 0; q < pb.ipc; ++q)
          each(rank_of(L, q + 1 == pb.ipc), make_int2(i, sid * pb.ipc + q));
      }
    }
  };
  std::vector<size_t> at(costs.size() + 1, 0);           // items of the costs before
  for_items([&](size_t r, int2) { ++at[r + 1]; });
  for (size_t k = 1; k < at.size(); ++k) at[k] += at[k - 1];
  std::vector<int2> wl(at.back());
  for_items([&](size_t r, int2 w) { wl[at[r]++] = w; });
  b->n_items = (long long)wl.size();
  if ((st = b->d_work.reserve(std::max<size_t>(wl.size(), 1) * sizeof(int2))) != EBIC_OK) return fin(st);
  if ((st = b->d_probs.reserve(b->probs.size() * sizeof(BatchProb))) != EBIC_OK) return fin(st);
  if ((st = b->d_counter.reserve(sizeof(unsigned long long))) != EBIC_OK) return fin(st);
  if (cudaMemcpyAsync(b->d_work.ptr, wl.data(), wl.size() * sizeof(int2), cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      cudaMemcpyAsync(b->d_probs.ptr, b->probs.data(), b->probs.size() * sizeof(BatchProb),
                      cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return fin(fail(EBIC_ERR_CUDA, "uploading the batch work list"));
  }
  *out = b;
  return fin(EBIC_OK);
}

ebic_status ebic_batch_eval(ebic_batch b, void* stream) {
  if (!b) return fail(EBIC_ERR_ARG, "null batch");
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != b->device) cudaSetDevice(b->device);
  // The legacy default stream cannot be captured: use the batch's own
  // blocking stream instead (blocking streams stay ordered with it).
  cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : b->own;
  auto launch = [&]() -> ebic_status {
    EBIC_CUDA_TRY(cudaMemsetAsync(b->d_counter.ptr, 0, sizeof(unsigned long long), s));
    b->kernel<<<b->grid, kBatchThreads, 0, s>>>(
        b->d_probs.as<BatchProb>(), b->d_work.as<int2>(), b->n_items,
        b->d_counter.as<unsigned long long>());
    EBIC_CUDA_TRY(cudaGetLastError());
    return EBIC_OK;
  };
  ebic_status st = EBIC_OK;
  if (b->flags & EBIC_BATCH_GRAPH) {
    if (!b->exec) {
      if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        cudaGetLastError();
        st = fail(EBIC_ERR_CUDA, "cannot capture on this stream");
      } else {
        st = launch();
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(s, &g);
        if (st == EBIC_OK && e == cudaSuccess && g) {
          b->graph = g;
          if (cudaGraphInstantiate(&b->exec, g, 0) != cudaSuccess) {
            cudaGetLastError();
            st = fail(EBIC_ERR_CUDA, "graph instantiation failed");
          }
        } else if (st == EBIC_OK) {
          cudaGetLastError();
          st = fail(EBIC_ERR_CUDA, "graph capture failed");
        }
      }
    }
    if (st == EBIC_OK && cudaGraphLaunch(b->exec, s) != cudaSuccess) {
      cudaGetLastError();
      st = fail(EBIC_ERR_CUDA, "graph launch failed");
    }
  } else {
    st = launch();
  }
  if (st == EBIC_OK) count_launches(1);
  if (prev >= 0 && prev != b->device) cudaSetDevice(prev);
  return st;
}

ebic_status ebic_batch_describe(ebic_batch b, int32_t problem, int32_t* path,
                                int32_t* vecs_per_part, int32_t* parts, int64_t* work_items,
                                int32_t* grid) {
  if (!b || problem < 0 || problem >= b->n) return fail(EBIC_ERR_ARG, "bad batch / problem");
  const BatchProb& pb = b->probs[(size_t)problem];
  if (path) *path = pb.path;
  if (vecs_per_part) *vecs_per_part = pb.vpi;
  if (parts) *parts = pb.ipc;
  if (work_items) *work_items = b->n_items;
  if (grid) *grid = b->grid;
  return EBIC_OK;
}

void ebic_batch_free(ebic_batch b) {
  if (!b) return;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != b->device) cudaSetDevice(b->device);
  cudaDeviceSynchronize();
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->d_probs.release();
  b->d_work.release();
  b->d_scratch.release();
  b->d_counter.release();
  if (b->own) cudaStreamDestroy(b->own);
  if (prev >= 0 && prev != b->device) cudaSetDevice(prev);
  delete b;
}

}  // extern "C"

// Step 6 ("prepare biclusters": the indices of the rows that match each
// series of columns), Step 7's expansion by negative trends, and the recovery
// and relevance scores of Eq. (2)-(3).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "ebic_internal.cuh"
#include "ebic_planes.cuh"
#include "ebic_support.cuh"

namespace ebic {

// ---------------------------------------------------------------------------
// Rows of a series.  One CTA per series walks the column-major matrix in
// chunks of 1,024 rows, each thread four consecutive rows (one float4 per
// column): a row is kept when its values rise strictly along the series (or,
// mode 1, rise or fall strictly).  With APPROX a row is kept when at most
// `breaks` of its adjacent pairs do not rise strictly (mode 1: or at most
// `breaks` do not fall strictly), counted per row.  The counting launch
// writes the number of kept rows; the writing launch stores their indices,
// ascending, from row_off[series] on (a block-wide scan orders them).
// ---------------------------------------------------------------------------
constexpr int kRowThreads = 256;

template <bool WRITE, bool APPROX>
__global__ void __launch_bounds__(kRowThreads)
k_rows(const float* __restrict__ A_c, int32_t R, int32_t R_pad, const int32_t* __restrict__ off,
       const int32_t* __restrict__ cols, int32_t mode, int32_t breaks,
       int32_t* __restrict__ counts, const long long* __restrict__ row_off,
       int32_t* __restrict__ rows) {
  __shared__ int s_warp[kRowThreads / 32];
  const int sid = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = off[sid], L = off[sid + 1] - b;
  long long written = 0;
  int total = 0;
  for (int r0 = 0; r0 < R_pad; r0 += 4 * kRowThreads) {
    const int r = r0 + 4 * tid;
    uint32_t keep = 0u;
    if (r < R_pad) {
      uint32_t rise = 0xFu, fall = 0xFu;
      int up_breaks[4] = {0, 0, 0, 0}, down_breaks[4] = {0, 0, 0, 0};
      float4 prev = *reinterpret_cast<const float4*>(A_c + (size_t)cols[b] * R_pad + r);
      for (int i = 1; i < L; ++i) {
        const float4 cur = *reinterpret_cast<const float4*>(A_c + (size_t)cols[b + i] * R_pad + r);
        const uint32_t up = lt4(prev, cur), down = gt4(prev, cur);
        if (APPROX) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            up_breaks[j] += ((up >> j) & 1u) ? 0 : 1;
            down_breaks[j] += ((down >> j) & 1u) ? 0 : 1;
          }
        } else {
          rise &= up;
          fall &= down;
        }
        prev = cur;
      }
      if (APPROX) {
        rise = fall = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          rise |= up_breaks[j] <= breaks ? 1u << j : 0u;
          fall |= down_breaks[j] <= breaks ? 1u << j : 0u;
        }
      }
      const uint32_t valid = (r < R ? 1u : 0u) | (r + 1 < R ? 2u : 0u) | (r + 2 < R ? 4u : 0u) |
                             (r + 3 < R ? 8u : 0u);
      keep = (rise | (mode == 1 ? fall : 0u)) & valid;
    }
    const int c = __popc(keep);
    if (!WRITE) {
      total += c;
      continue;
    }
    // exclusive position of this thread's rows within the chunk
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int before = 0, chunk = 0;
    for (int w = 0; w < kRowThreads / 32; ++w) {
      const int v = s_warp[w];
      before += w < warp ? v : 0;
      chunk += v;
    }
    int pos = (int)(written) + before + incl - c;
    int32_t* out = rows + row_off[sid];
    for (int j = 0; j < 4; ++j)
      if ((keep >> j) & 1u) out[pos++] = r + j;
    written += chunk;
    __syncthreads();                       // s_warp is reused by the next chunk
  }
  if (!WRITE) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    if (lane == 0) s_warp[warp] = total;
    __syncthreads();
    if (tid == 0) {
      int t = 0;
      for (int w = 0; w < kRowThreads / 32; ++w) t += s_warp[w];
      counts[sid] = t;
    }
  }
}

// ---------------------------------------------------------------------------
// The same from the rank planes (up to 511 columns), in three launches and one
// walk over the data:
//   k_row_masks    one warp per (series, slice of 1,024 rows) finds the kept rows
//                  as one bit each and stores its 32 words and their number;
//   k_row_offsets  one CTA turns the numbers into row_off;
//   k_row_write    one warp per (series, slice) writes the indices of its bits.
// 100 series, 20,000 x 200, both directions: 7.7 + 4.9 + 4.4 us against 78 us for
// the counting and 59 us for the writing launch of k_rows (one CTA a series,
// every column read whole); latency-bound at this size.  The workspaces stay
// on the handle.
// ---------------------------------------------------------------------------
// Valid rows of word w (bit l of word 4 b + i is row 128 b + 4 l + i).
__device__ __forceinline__ uint32_t row_valid(int32_t w, int32_t R) {
  const int n = min(32, max(0, (R - (w >> 2) * 128 - (w & 3) + 3) >> 2));
  return n >= 32 ? kFull : (1u << n) - 1u;
}

// Bit-sliced count of broken pairs, K bits and a sticky overflow.
template <int K>
struct BreakCount {
  uint32_t c[K], over;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < K; ++i) c[i] = 0u;
    over = 0u;
  }
  __device__ __forceinline__ void add(uint32_t x) {
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const uint32_t t = c[i] & x;
      c[i] ^= x;
      x = t;
    }
    over |= x;
  }
  // rows with at most e broken pairs (e < 2^K)
  __device__ __forceinline__ uint32_t at_most(int32_t e) const {
    uint32_t gt = 0u;
#pragma unroll
    for (int i = 0; i < K; ++i) gt = ((e >> i) & 1) ? (c[i] & gt) : (c[i] | gt);
    return ~(gt | over);
  }
};

// Rows of this lane's word with at most e broken pairs along a series of L >= 2
// columns, rising or (mode 1) falling; ties and NaN break both.
template <int B, int K>
__device__ __forceinline__ uint32_t plane_breaks(const uint32_t* __restrict__ PL, int32_t W,
                                                 const CbfPop& pop, int64_t begin, int32_t L,
                                                 int32_t w, uint32_t valid, int32_t mode, int32_t e) {
  uint32_t p[B][1], q[B][1], np[1], nq[1];
  BreakCount<K> up, down;
  up.clear();
  down.clear();
  load_planes<B, 1>(PL, W, (uint32_t)pop.col(begin, 0), w, p);
  nan_words<B, 1>(p, np);
  uint32_t keep = valid;
  for (int32_t t = 1; t < L; ++t) {
    load_planes<B, 1>(PL, W, (uint32_t)pop.col(begin, t), w, q);
    nan_words<B, 1>(q, nq);
    uint32_t lt[1] = {kFull}, gt[1] = {kFull};
    plane_step<true, B, 1>(p, q, lt, gt);
    up.add(~(lt[0] & ~nq[0]));
    down.add(~(gt[0] & ~np[0]));
    keep = valid & (up.at_most(e) | (mode == 1 ? down.at_most(e) : 0u));
    if (!__any_sync(kFull, keep != 0u)) break;
#pragma unroll
    for (int b = 0; b < B; ++b) p[b][0] = q[b][0];
    np[0] = nq[0];
  }
  return keep;
}

// K = 0: strict trends; else at most `breaks` < 2^K broken pairs.
template <int B, int K>
__global__ void __launch_bounds__(256)
k_row_masks(const uint32_t* __restrict__ PL, int32_t W, int32_t R, CbfPop pop, int32_t P,
            int32_t slices, int32_t mode, int32_t breaks, uint32_t* __restrict__ mask,
            int32_t* __restrict__ cnt) {
  const int lane = threadIdx.x & 31;
  const int64_t item = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (item >= (int64_t)P * slices) return;                 // warp-uniform
  const int32_t sid = (int32_t)(item / slices), slice = (int32_t)(item % slices);
  int64_t begin = 0;
  int32_t L = 0;
  pop.range(sid, &begin, &L);                              // checked by the caller
  const int32_t w = slice * 32 + lane;
  const bool on = w < W;
  const uint32_t valid = on ? row_valid(w, R) : 0u;
  uint32_t keep = valid;
  if (L > 1) {
    if (K == 0) {
      uint32_t m[1], d[1];
      if (mode == 1) plane_chain<true, B, 1, CbfPop>(PL, W, pop, begin, L, w, on, lane, m, d);
      else plane_chain<false, B, 1, CbfPop>(PL, W, pop, begin, L, w, on, lane, m, d);
      keep = m[0] | d[0];
    } else {
      keep = plane_breaks<B, (K ? K : 1)>(PL, W, pop, begin, L, on ? w : W - 1, valid, mode, breaks);
    }
  }
  if (on) mask[(size_t)sid * W + w] = keep;
  const uint32_t n = __reduce_add_sync(kFull, (uint32_t)__popc(keep));
  if (lane == 0) cnt[item] = (int32_t)n;
}

// The inclusive sum over the CTA's threads up to this one; *all = over all of them.
__device__ __forceinline__ long long block_scan(long long mine, long long* s_warp, long long* all) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  long long incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long u = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += u;
  }
  __syncthreads();
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  long long before = 0, sum = 0;
  for (int v = 0; v < 32; ++v) {
    before += v < warp ? s_warp[v] : 0;
    sum += s_warp[v];
  }
  *all = sum;
  return before + incl;
}

// row_off[i] = rows of the series before i; row_off[P] = all.  A CTA takes 1,024
// series; where there are more, its offsets count from its first series, its sum
// goes to part[], and k_row_bases and k_row_shift follow (one CTA for them all,
// 1,024 at a time, took 18 of 21 ms of a call with 2^20 series of 100 rows; 3.9 now).
__global__ void __launch_bounds__(1024)
k_row_offsets(const int32_t* __restrict__ cnt, int32_t P, int32_t slices,
              long long* __restrict__ row_off, long long* __restrict__ part) {
  __shared__ long long s_tot[1024], s_warp[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t p0 = blockIdx.x * 1024;
  const int n = min(1024, P - p0);
  long long mine = 0;
  if (slices == 1) {
    if (tid < n) mine = cnt[p0 + tid];
  } else {
    for (int i = warp; i < n; i += 32) {
      int s = 0;                                           // at most R rows a series
      for (int32_t j = lane; j < slices; j += 32) s += cnt[(size_t)(p0 + i) * slices + j];
      s = __reduce_add_sync(kFull, s);
      if (lane == 0) s_tot[i] = s;
    }
    __syncthreads();
    if (tid < n) mine = s_tot[tid];
  }
  long long all = 0;
  const long long incl = block_scan(mine, s_warp, &all);
  if (tid < n) row_off[p0 + tid] = incl - mine;
  if (tid != 0) return;
  if (gridDim.x == 1) row_off[P] = all;
  else part[blockIdx.x] = all;
}

// part[b] = rows of the CTAs before b; row_off[P] = all.
__global__ void __launch_bounds__(1024)
k_row_bases(int32_t blocks, int32_t P, long long* __restrict__ row_off, long long* __restrict__ part) {
  __shared__ long long s_warp[32];
  long long base = 0;
  for (int32_t b0 = 0; b0 < blocks; b0 += 1024) {
    const int32_t b = b0 + (int32_t)threadIdx.x;
    const long long mine = b < blocks ? part[b] : 0;
    long long all = 0;
    const long long incl = block_scan(mine, s_warp, &all);
    if (b < blocks) part[b] = base + incl - mine;
    base += all;
  }
  if (threadIdx.x == 0) row_off[P] = base;
}

__global__ void __launch_bounds__(1024)
k_row_shift(int32_t P, const long long* __restrict__ part, long long* __restrict__ row_off) {
  const int32_t p = (int32_t)(blockIdx.x * 1024 + threadIdx.x);
  if (p < P) row_off[p] += part[blockIdx.x];
}

__global__ void __launch_bounds__(256)
k_row_write(const uint32_t* __restrict__ mask, const int32_t* __restrict__ cnt, int32_t W, int32_t P,
            int32_t slices, const long long* __restrict__ row_off, long long room,
            int32_t* __restrict__ rows) {
  const int lane = threadIdx.x & 31;
  const int64_t item = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (item >= (int64_t)P * slices || cnt[item] == 0) return;     // warp-uniform
  const int32_t sid = (int32_t)(item / slices), slice = (int32_t)(item % slices);
  if (row_off[P] > room) return;
  int pre = 0;
  for (int32_t j = lane; j < slice; j += 32) pre += cnt[item - slice + j];
  pre = __reduce_add_sync(kFull, pre);
  // the four lanes of a vector hold its four words, a quarter of its rows each
  const int32_t w = slice * 32 + lane;
  const uint4 v = w < W ? reinterpret_cast<const uint4*>(mask + (size_t)sid * W)[w >> 2]
                        : make_uint4(0u, 0u, 0u, 0u);
  const int i = lane & 3;
  const int mine = i == 0 ? popc4(v) : 0;
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += u;
  }
  int32_t* out = rows + row_off[sid] + pre + (__shfl_sync(kFull, incl - mine, lane & ~3));
  uint32_t bits = i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
  while (bits) {
    const int l = __ffs(bits) - 1;
    bits &= bits - 1u;
    const uint32_t lo = (1u << l) - 1u;
    const int at = __popc(v.x & lo) + __popc(v.y & lo) + __popc(v.z & lo) + __popc(v.w & lo) +
                   (i > 0 ? (int)((v.x >> l) & 1u) : 0) + (i > 1 ? (int)((v.y >> l) & 1u) : 0) +
                   (i > 2 ? (int)((v.z >> l) & 1u) : 0);
    out[at] = 128 * (w >> 2) + 4 * l + i;
  }
}

// Larger masks than this take the fp32 columns.
constexpr size_t kRowMaskBytes = (size_t)256 << 20;

// A handle keeps no workspace above this between calls (the list of a full
// top-rank list of 100 series over 20,000 rows takes 8 MB, its masks 250 KB).
constexpr size_t kRowKeepBytes = (size_t)32 << 20;

struct RowTrim {
  ebic_ctx* h;
  ~RowTrim() {
    for (DevBuf* b : {&h->rw_mask, &h->rw_cnt, &h->rw_off, &h->rw_rows})
      if (b->bytes > kRowKeepBytes) b->release();
  }
};

template <int B>
static void launch_row_masks_b(ebic_ctx* h, const CbfPop& pop, int32_t P, int32_t slices,
                               int32_t mode, int32_t breaks, cudaStream_t s) {
  const unsigned grid = (unsigned)(((int64_t)P * slices + 7) / 8);
#define EBIC_RM(K)                                                                              \
  k_row_masks<B, K><<<grid, 256, 0, s>>>(h->PL, h->W, h->R, pop, P, slices, mode, breaks,       \
                                         h->rw_mask.as<uint32_t>(), h->rw_cnt.as<int32_t>())
  if (breaks <= 0) EBIC_RM(0);
  else if (breaks < 4) EBIC_RM(2);
  else if (breaks < 16) EBIC_RM(4);
  else EBIC_RM(11);
#undef EBIC_RM
}

static void launch_row_masks(ebic_ctx* h, const CbfPop& pop, int32_t P, int32_t slices,
                             int32_t mode, int32_t breaks, cudaStream_t s) {
  switch (h->nb) {
    case 6: launch_row_masks_b<6>(h, pop, P, slices, mode, breaks, s); break;
    case 7: launch_row_masks_b<7>(h, pop, P, slices, mode, breaks, s); break;
    case 8: launch_row_masks_b<8>(h, pop, P, slices, mode, breaks, s); break;
    default: launch_row_masks_b<9>(h, pop, P, slices, mode, breaks, s); break;
  }
}

// ---------------------------------------------------------------------------
// Eq. (2)-(3).  One warp per (expected e, found f) pair computes the Jaccard
// index of the two biclusters as sets of cells: |Re & Rf| |Ce & Cf| /
// (|Re| |Ce| + |Rf| |Cf| - |Re & Rf| |Ce & Cf|); intersections of ascending
// index lists by binary search of one list's entries in the other.
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long intersect_sorted(const int32_t* a, int na, const int32_t* b,
                                                      int nb, int lane) {
  long long n = 0;
  for (int i = lane; i < na; i += 32) {
    const int32_t v = a[i];
    int lo = 0, hi = nb;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (b[mid] < v) lo = mid + 1;
      else hi = mid;
    }
    n += (lo < nb && b[lo] == v) ? 1 : 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  return n;
}

__global__ void __launch_bounds__(256)
k_jaccard(int32_t E, int32_t F, const long long* __restrict__ er_off, const int32_t* __restrict__ er,
          const long long* __restrict__ ec_off, const int32_t* __restrict__ ec,
          const long long* __restrict__ fr_off, const int32_t* __restrict__ fr,
          const long long* __restrict__ fc_off, const int32_t* __restrict__ fc,
          double* __restrict__ J) {
  const int lane = threadIdx.x & 31;
  const long long pair = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (pair >= (long long)E * F) return;
  const int e = (int)(pair / F), f = (int)(pair % F);
  const int ner = (int)(er_off[e + 1] - er_off[e]), nec = (int)(ec_off[e + 1] - ec_off[e]);
  const int nfr = (int)(fr_off[f + 1] - fr_off[f]), nfc = (int)(fc_off[f + 1] - fc_off[f]);
  const long long ir = intersect_sorted(er + er_off[e], ner, fr + fr_off[f], nfr, lane);
  const long long ic = intersect_sorted(ec + ec_off[e], nec, fc + fc_off[f], nfc, lane);
  if (lane == 0) {
    const long long inter = ir * ic;
    const long long uni = (long long)ner * nec + (long long)nfr * nfc - inter;
    J[pair] = uni > 0 ? (double)inter / (double)uni : 0.0;
  }
}

// recovery = mean over e of max over f of J, relevance = mean over f of max
// over e (one CTA; fixed summation order)
__global__ void k_recovery_relevance(int32_t E, int32_t F, const double* __restrict__ J,
                                     double* __restrict__ out) {
  if (threadIdx.x != 0) return;
  double rec = 0.0, rel = 0.0;
  for (int e = 0; e < E; ++e) {
    double m = 0.0;
    for (int f = 0; f < F; ++f) m = fmax(m, J[(size_t)e * F + f]);
    rec += m;
  }
  for (int f = 0; f < F; ++f) {
    double m = 0.0;
    for (int e = 0; e < E; ++e) m = fmax(m, J[(size_t)e * F + f]);
    rel += m;
  }
  out[0] = rec / (double)E;
  out[1] = rel / (double)F;
}

}  // namespace ebic

using namespace ebic;

namespace {

struct Guard {
  int prev = -1, dev;
  explicit Guard(int d) : dev(d) {
    cudaGetDevice(&prev);
    if (prev != d) cudaSetDevice(d);
  }
  ~Guard() {
    if (prev >= 0 && prev != dev) cudaSetDevice(prev);
  }
};

// ascending, distinct, within [0, bound)
bool strictly_ascending(const int32_t* v, long long n, int32_t bound) {
  for (long long i = 0; i < n; ++i) {
    if (v[i] < 0 || v[i] >= bound) return false;
    if (i && v[i] <= v[i - 1]) return false;
  }
  return true;
}

}  // namespace

extern "C" {

// Steps 6 / 7 from the rank planes; the arguments have been checked and there is
// room for the masks.
static ebic_status extract_rows_planes(ebic_ctx* h, const int32_t* offsets, const int32_t* cols,
                                       int32_t P, int32_t total, int32_t slices, int32_t mode,
                                       int32_t breaks, int64_t* row_offsets, int32_t* rows,
                                       int64_t* inout_capacity) {
  const cudaStream_t s = h->stream;
  const RowTrim trim{h};
  const size_t off_bytes = (size_t)(P + 1) * sizeof(long long);
  EBIC_TRY(h->st_off.reserve((size_t)(P + 1) * sizeof(int32_t)));
  EBIC_TRY(h->st_cols.reserve((size_t)total * sizeof(int32_t)));
  EBIC_TRY(h->rw_cnt.reserve((size_t)P * slices * sizeof(int32_t)));
  const int32_t blocks = (P + 1023) / 1024;                // of k_row_offsets
  EBIC_TRY(h->rw_off.reserve(off_bytes + (size_t)blocks * sizeof(long long)));
  EBIC_TRY(h->h_stage.reserve(off_bytes));
  EBIC_CUDA_TRY(cudaMemcpyAsync(h->st_off.ptr, offsets, (size_t)(P + 1) * sizeof(int32_t),
                                cudaMemcpyHostToDevice, s));
  EBIC_CUDA_TRY(cudaMemcpyAsync(h->st_cols.ptr, cols, (size_t)total * sizeof(int32_t),
                                cudaMemcpyHostToDevice, s));
  const CbfPop pop{h->st_off.as<int32_t>(), h->st_cols.as<int32_t>(), total};
  launch_row_masks(h, pop, P, slices, mode, breaks, s);
  long long *d_roff = h->rw_off.as<long long>(), *part = d_roff + P + 1;
  k_row_offsets<<<(unsigned)blocks, 1024, 0, s>>>(h->rw_cnt.as<int32_t>(), P, slices, d_roff, part);
  if (blocks > 1) {
    k_row_bases<<<1, 1024, 0, s>>>(blocks, P, d_roff, part);
    k_row_shift<<<(unsigned)blocks, 1024, 0, s>>>(P, part, d_roff);
  }
  count_launches(blocks > 1 ? 4 : 2);
  const unsigned grid = (unsigned)(((int64_t)P * slices + 7) / 8);
  auto write = [&]() {
    k_row_write<<<grid, 256, 0, s>>>(h->rw_mask.as<uint32_t>(), h->rw_cnt.as<int32_t>(), h->W, P,
                                     slices, h->rw_off.as<long long>(),
                                     (long long)(h->rw_rows.bytes / sizeof(int32_t)),
                                     h->rw_rows.as<int32_t>());
    count_launches(1);
  };
  // the indices go out before their number is known here, unless the caller
  // only asks for it; they stay unwritten where the last calls' buffer is
  // too small, and are written again once it has grown
  if (rows && h->rw_rows.ptr) write();
  EBIC_CUDA_TRY(cudaGetLastError());
  EBIC_CUDA_TRY(cudaMemcpyAsync(h->h_stage.ptr, h->rw_off.ptr, off_bytes, cudaMemcpyDeviceToHost, s));
  EBIC_CUDA_TRY(cudaStreamSynchronize(s));
  const long long* roff = h->h_stage.as<long long>();
  const long long need = roff[P];
  if (need > *inout_capacity || (need > 0 && !rows)) {
    const long long cap = *inout_capacity;
    *inout_capacity = need;
    return fail(EBIC_ERR_ARG, "the rows need %lld entries, the buffer holds %lld", need, cap);
  }
  if (need > 0) {
    if ((size_t)need * sizeof(int32_t) > h->rw_rows.bytes) {
      EBIC_TRY(h->rw_rows.reserve((size_t)need * sizeof(int32_t)));
      write();
      EBIC_CUDA_TRY(cudaGetLastError());
    }
    EBIC_CUDA_TRY(cudaMemcpyAsync(rows, h->rw_rows.ptr, (size_t)need * sizeof(int32_t),
                                  cudaMemcpyDeviceToHost, s));
    EBIC_CUDA_TRY(cudaStreamSynchronize(s));
  }
  std::memcpy(row_offsets, roff, off_bytes);
  *inout_capacity = need;
  return EBIC_OK;
}

// Steps 6 / 7 for ebic_extract_rows (breaks < 0: strict trends) and
// ebic_extract_rows_approx (at most `breaks` broken pairs per row).
static ebic_status extract_rows(ebic_handle h, const int32_t* offsets, const int32_t* cols,
                                int32_t P, int32_t mode, int32_t breaks, int64_t* row_offsets,
                                int32_t* rows, int64_t* inout_capacity) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  if (P < 0 || P > (1 << 24)) return fail(EBIC_ERR_ARG, "P = %d outside [0, 2^24]", P);
  if (!offsets || !row_offsets || !inout_capacity || *inout_capacity < 0)
    return fail(EBIC_ERR_ARG, "null pointer");
  if (mode != EBIC_ROWS_RISING && mode != EBIC_ROWS_RISING_OR_FALLING)
    return fail(EBIC_ERR_ARG, "bad rows mode %d", mode);
  if (P == 0) {
    row_offsets[0] = 0;
    *inout_capacity = 0;
    return EBIC_OK;
  }
  if (!cols) return fail(EBIC_ERR_ARG, "null pointer");
  if (offsets[0] != 0) return fail(EBIC_ERR_ARG, "offsets[0] must be 0");
  for (int32_t i = 0; i < P; ++i) {
    const int32_t L = offsets[i + 1] - offsets[i];
    if (L < 1 || L > EBIC_MAX_EVAL_LEN)
      return fail(EBIC_ERR_ARG, "series %d has length %d outside [1, %d]", i, L, EBIC_MAX_EVAL_LEN);
  }
  const int32_t total = offsets[P];
  for (int32_t k = 0; k < total; ++k)
    if (cols[k] < 0 || cols[k] >= h->C)
      return fail(EBIC_ERR_ARG, "column index %d at position %d outside [0, %d)", cols[k], k, h->C);
  Guard g(h->device);
  const cudaStream_t s = h->stream;
  const int32_t slices = (h->W + 31) / 32;
  bool planes = false;
  if ((size_t)P * h->W * sizeof(uint32_t) <= kRowMaskBytes)
    EBIC_TRY(want_planes(h, s, false, 12.0 * P, &planes));  // (a series costs 12 evaluations')
  if (planes && h->rw_mask.reserve((size_t)P * h->W * sizeof(uint32_t)) == EBIC_OK)
    return extract_rows_planes(h, offsets, cols, P, total, slices, mode, breaks, row_offsets, rows,
                               inout_capacity);
  // From the fp32 columns (more than 511 of them, or no room for planes or masks):
  // a counting launch, the offsets here, a writing launch.
  const RowTrim trim{h};
  EBIC_TRY(h->st_off.reserve((size_t)(P + 1) * sizeof(int32_t)));
  EBIC_TRY(h->st_cols.reserve((size_t)total * sizeof(int32_t)));
  EBIC_TRY(h->rw_cnt.reserve((size_t)P * sizeof(int32_t)));
  EBIC_CUDA_TRY(cudaMemcpyAsync(h->st_off.ptr, offsets, (size_t)(P + 1) * sizeof(int32_t),
                                cudaMemcpyHostToDevice, s));
  EBIC_CUDA_TRY(cudaMemcpyAsync(h->st_cols.ptr, cols, (size_t)total * sizeof(int32_t),
                                cudaMemcpyHostToDevice, s));
  auto launch = [&](bool write) -> ebic_status {
    auto kern = write ? (breaks < 0 ? k_rows<true, false> : k_rows<true, true>)
                      : (breaks < 0 ? k_rows<false, false> : k_rows<false, true>);
    kern<<<(unsigned)P, kRowThreads, 0, s>>>(
        h->A_c, h->R, h->R_pad, h->st_off.as<int32_t>(), h->st_cols.as<int32_t>(), mode,
        std::max(breaks, 0), h->rw_cnt.as<int32_t>(), h->rw_off.as<long long>(),
        h->rw_rows.as<int32_t>());
    count_launches(1);
    EBIC_CUDA_TRY(cudaGetLastError());
    return EBIC_OK;
  };
  std::vector<int32_t> cnt((size_t)P);
  EBIC_TRY(launch(false));
  EBIC_CUDA_TRY(cudaMemcpyAsync(cnt.data(), h->rw_cnt.ptr, (size_t)P * sizeof(int32_t),
                                cudaMemcpyDeviceToHost, s));
  EBIC_CUDA_TRY(cudaStreamSynchronize(s));
  std::vector<long long> roff((size_t)P + 1, 0);
  for (int32_t i = 0; i < P; ++i) roff[i + 1] = roff[i] + cnt[i];
  const long long need = roff[P];
  if (need > *inout_capacity || (need > 0 && !rows)) {
    const long long cap = *inout_capacity;
    *inout_capacity = need;
    return fail(EBIC_ERR_ARG, "the rows need %lld entries, the buffer holds %lld", need, cap);
  }
  if (need > 0) {
    EBIC_TRY(h->rw_off.reserve(roff.size() * sizeof(long long)));
    EBIC_TRY(h->rw_rows.reserve((size_t)need * sizeof(int32_t)));
    EBIC_CUDA_TRY(cudaMemcpyAsync(h->rw_off.ptr, roff.data(), roff.size() * sizeof(long long),
                                  cudaMemcpyHostToDevice, s));
    EBIC_TRY(launch(true));
    EBIC_CUDA_TRY(cudaMemcpyAsync(rows, h->rw_rows.ptr, (size_t)need * sizeof(int32_t),
                                  cudaMemcpyDeviceToHost, s));
    EBIC_CUDA_TRY(cudaStreamSynchronize(s));
  }
  for (int32_t i = 0; i <= P; ++i) row_offsets[i] = roff[i];
  *inout_capacity = need;
  return EBIC_OK;
}

ebic_status ebic_extract_rows(ebic_handle h, const int32_t* offsets, const int32_t* cols,
                              int32_t P, int32_t mode, int64_t* row_offsets, int32_t* rows,
                              int64_t* inout_capacity) {
  return extract_rows(h, offsets, cols, P, mode, -1, row_offsets, rows, inout_capacity);
}

ebic_status ebic_extract_rows_approx(ebic_handle h, const int32_t* offsets, const int32_t* cols,
                                     int32_t P, int32_t max_breaks, int32_t mode,
                                     int64_t* row_offsets, int32_t* rows,
                                     int64_t* inout_capacity) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  if (max_breaks < 0 || max_breaks > EBIC_MAX_EVAL_LEN)
    return fail(EBIC_ERR_ARG, "max_breaks = %d outside [0, %d]", max_breaks, EBIC_MAX_EVAL_LEN);
  return extract_rows(h, offsets, cols, P, mode, max_breaks, row_offsets, rows, inout_capacity);
}

ebic_status ebic_recovery_relevance(int32_t E, const int64_t* e_row_off, const int32_t* e_rows,
                                    const int64_t* e_col_off, const int32_t* e_cols, int32_t F,
                                    const int64_t* f_row_off, const int32_t* f_rows,
                                    const int64_t* f_col_off, const int32_t* f_cols,
                                    double* out_recovery, double* out_relevance,
                                    double* out_jaccard) {
  if (E < 0 || F < 0 || (int64_t)E * F > (1ll << 26))
    return fail(EBIC_ERR_ARG, "E = %d, F = %d out of range", E, F);
  if (!out_recovery || !out_relevance) return fail(EBIC_ERR_ARG, "null pointer");
  if (E == 0 || F == 0) {
    *out_recovery = 0.0;
    *out_relevance = 0.0;
    return EBIC_OK;
  }
  if (!e_row_off || !e_rows || !e_col_off || !e_cols || !f_row_off || !f_rows || !f_col_off ||
      !f_cols)
    return fail(EBIC_ERR_ARG, "null pointer");
  const struct {
    const int64_t* off;
    const int32_t* v;
    int32_t n;
  } lists[4] = {{e_row_off, e_rows, E}, {e_col_off, e_cols, E}, {f_row_off, f_rows, F},
                {f_col_off, f_cols, F}};
  for (const auto& li : lists) {
    if (li.off[0] != 0) return fail(EBIC_ERR_ARG, "index lists must start at offset 0");
    for (int32_t i = 0; i < li.n; ++i) {
      if (li.off[i + 1] < li.off[i]) return fail(EBIC_ERR_ARG, "offsets must not decrease");
      if (!strictly_ascending(li.v + li.off[i], li.off[i + 1] - li.off[i], 0x7fffffff))
        return fail(EBIC_ERR_ARG, "bicluster %d: indices must be distinct, ascending, >= 0", i);
    }
  }
  DevBuf d[8], dJ, dout;
  auto release = [&]() {
    for (DevBuf& b : d) b.release();
    dJ.release();
    dout.release();
  };
  ebic_status st = EBIC_OK;
  const cudaStream_t s = nullptr;
  for (int i = 0; i < 4 && st == EBIC_OK; ++i) {
    const size_t no = (size_t)lists[i].n + 1, nv = (size_t)std::max<int64_t>(lists[i].off[lists[i].n], 1);
    if ((st = d[2 * i].reserve(no * sizeof(int64_t))) != EBIC_OK) break;
    if ((st = d[2 * i + 1].reserve(nv * sizeof(int32_t))) != EBIC_OK) break;
    if (cudaMemcpy(d[2 * i].ptr, lists[i].off, no * sizeof(int64_t), cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(d[2 * i + 1].ptr, lists[i].v, (size_t)lists[i].off[lists[i].n] * sizeof(int32_t),
                   cudaMemcpyHostToDevice) != cudaSuccess)
      st = fail(EBIC_ERR_CUDA, "copy of the biclusters failed");
  }
  const size_t pairs = (size_t)E * F;
  if (st == EBIC_OK) st = dJ.reserve(pairs * sizeof(double));
  if (st == EBIC_OK) st = dout.reserve(2 * sizeof(double));
  if (st == EBIC_OK) {
    k_jaccard<<<(unsigned)((pairs * 32 + 255) / 256), 256, 0, s>>>(
        E, F, d[0].as<long long>(), d[1].as<int32_t>(), d[2].as<long long>(), d[3].as<int32_t>(),
        d[4].as<long long>(), d[5].as<int32_t>(), d[6].as<long long>(), d[7].as<int32_t>(),
        dJ.as<double>());
    k_recovery_relevance<<<1, 32, 0, s>>>(E, F, dJ.as<double>(), dout.as<double>());
    count_launches(2);
    double out[2];
    if (cudaMemcpy(out, dout.ptr, sizeof(out), cudaMemcpyDeviceToHost) != cudaSuccess ||
        (out_jaccard &&
         cudaMemcpy(out_jaccard, dJ.ptr, pairs * sizeof(double), cudaMemcpyDeviceToHost) !=
             cudaSuccess)) {
      st = fail(EBIC_ERR_CUDA, "scoring failed: %s", cudaGetErrorString(cudaGetLastError()));
    } else {
      *out_recovery = out[0];
      *out_relevance = out[1];
    }
  }
  release();
  return st;
}

}  // extern "C"

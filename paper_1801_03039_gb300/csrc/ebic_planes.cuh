// Rank planes: every value of the matrix as its rank within its own row, bit
// by bit, and the kernels that compare ranks 32 rows at a time.
//
// a[k][p] < a[k][q] depends only on the order of row k's values, so a value
// can stand as the number of smaller values in its row: B = 6 .. 9 bits for up
// to 511 columns instead of 32.  Plane b of column c holds bit b of 32 rows'
// ranks per word (the row order inside a word is the pair table's), and one
// LOP3 per plane compares 32 rows:
//     lt = (~x & y) | (~(x ^ y) & lt)        from the lowest plane up.
// Equal values (+0 and -0 included) have equal ranks.  NaN -- and the padding
// rows -- have all B bits set, above every rank (at most C - 1 < 2^B - 1): a
// NaN on the left of < fails by itself, a NaN on the right has to be masked.
// Along a rising series every column but the last is also a left side, so
// masking the last column's NaN is enough; along a falling one, the first's.
//
// Layout: PL[c][b][W] words, W as in the pair table.
#pragma once

#include "ebic_support.cuh"

namespace ebic {

constexpr int kPlaneMaxCols = 511;      // above: the ranks cost more to build than a load saves
constexpr int kPlaneMinBits = 6;

// Bits of a rank, with the all-ones pattern left for NaN.
inline int plane_bits(int32_t C) {
  int b = kPlaneMinBits;
  while ((1 << b) <= C) ++b;
  return b;
}

// 1 where x < y, one plane up: lt is the answer of the planes below.
__device__ __forceinline__ uint32_t lt_step(uint32_t x, uint32_t y, uint32_t lt) {
  uint32_t r;                                    // (~x & y) | (~(x ^ y) & lt)
  asm("lop3.b32 %0, %1, %2, %3, 0x8e;" : "=r"(r) : "r"(x), "r"(y), "r"(lt));
  return r;
}

// ---------------------------------------------------------------------------
// K2 from the planes.  A thread keeps the planes of four columns p for 64 rows
// in registers and walks its share of the columns q: B plane loads, then B
// LOP3 per word and entry, four 8-byte stores.  Floor: the table's writes (100
// MB at 20,000 x 200, 15 us); 32 us against 415 us with one ballot per 32 fp32
// comparisons (k_pair_table, kept where there are no planes).
// ---------------------------------------------------------------------------
constexpr int kPairCols = 4;

template <int B>
__global__ void __launch_bounds__(128)
k_pair_planes(const uint32_t* __restrict__ PL, int32_t C, int32_t V2, int32_t q_chunk,
              uint32_t* __restrict__ LT) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int32_t v = (int32_t)(t % V2), p0 = (int32_t)(t / V2) * kPairCols;
  if (p0 >= C) return;
  const uint2* P2 = reinterpret_cast<const uint2*>(PL);
  uint2 x[kPairCols][B];
#pragma unroll
  for (int k = 0; k < kPairCols; ++k)
#pragma unroll
    for (int b = 0; b < B; ++b) x[k][b] = __ldg(P2 + ((size_t)min(p0 + k, C - 1) * B + b) * V2 + v);
  const int32_t q_lo = blockIdx.y * q_chunk, q_hi = min(C, q_lo + q_chunk);
  uint2* out = reinterpret_cast<uint2*>(LT) + (size_t)p0 * C * V2 + v;
  for (int32_t q = q_lo; q < q_hi; ++q) {
    uint2 y[B];
#pragma unroll
    for (int b = 0; b < B; ++b) y[b] = __ldg(P2 + ((size_t)q * B + b) * V2 + v);
    uint2 nan = y[0];
#pragma unroll
    for (int b = 1; b < B; ++b) nan = make_uint2(nan.x & y[b].x, nan.y & y[b].y);
#pragma unroll
    for (int k = 0; k < kPairCols; ++k) {
      uint2 l = make_uint2(0u, 0u);
#pragma unroll
      for (int b = 0; b < B; ++b)
        l = make_uint2(lt_step(x[k][b].x, y[b].x, l.x), lt_step(x[k][b].y, y[b].y, l.y));
      if (p0 + k < C) out[((size_t)k * C + q) * V2] = make_uint2(l.x & ~nan.x, l.y & ~nan.y);
    }
  }
}

// ---------------------------------------------------------------------------
// K3 without a pair table.  A warp walks one series over one slice of
// 32 * WID words (1,024 or 2,048 rows): lane l holds WID words of the running
// AND and of the last column's planes; a step loads the next column's B planes
// (one coalesced load each) and compares.  The warp stops when no lane has a row
// left.
//
// A CTA stays on one slice (blockIdx.x % slices) and takes every k-th series, so
// that up to 200 columns the slice's planes of all of them (128 bytes a plane and
// column) stay in its SM's L1; wider matrices read them from L2.  Bound by the
// LOP3 rate (ALU pipe 54 % busy) and the latency of the loads (L1 hits 83 %).
// 25,000 x 100, 2,000 series, both directions: 36 us against 216 us for the fp32
// columns (k_support_gather).
// ---------------------------------------------------------------------------
template <int WID> struct PlaneWords;
template <> struct PlaneWords<1> {
  typedef uint32_t vec;
  static __device__ __forceinline__ void get(const vec& v, uint32_t (&o)[1]) { o[0] = v; }
};
template <> struct PlaneWords<2> {
  typedef uint2 vec;
  static __device__ __forceinline__ void get(const vec& v, uint32_t (&o)[2]) {
    o[0] = v.x;
    o[1] = v.y;
  }
};

// Planes of column c for the words [first, first + WID).
template <int B, int WID>
__device__ __forceinline__ void load_planes(const uint32_t* __restrict__ PL, int32_t W, uint32_t c,
                                            int32_t first, uint32_t (&o)[B][WID]) {
  typedef PlaneWords<WID> PW;
  const uint32_t* base = PL + (size_t)c * B * W + first;
#pragma unroll
  for (int b = 0; b < B; ++b)
    PW::get(__ldg(reinterpret_cast<const typename PW::vec*>(base + (size_t)b * W)), o[b]);
}

template <int B, int WID>
__device__ __forceinline__ void nan_words(const uint32_t (&o)[B][WID], uint32_t (&n)[WID]) {
#pragma unroll
  for (int i = 0; i < WID; ++i) {
    n[i] = kFull;
#pragma unroll
    for (int b = 0; b < B; ++b) n[i] &= o[b][i];
  }
}

// m &= rows with x < y; with DEC also d &= rows with x > y.
template <bool DEC, int B, int WID>
__device__ __forceinline__ void plane_step(const uint32_t (&x)[B][WID], const uint32_t (&y)[B][WID],
                                           uint32_t (&m)[WID], uint32_t (&d)[WID]) {
#pragma unroll
  for (int i = 0; i < WID; ++i) {
    uint32_t lt = 0u, gt = 0u;
#pragma unroll
    for (int b = 0; b < B; ++b) {
      lt = lt_step(x[b][i], y[b][i], lt);
      if (DEC) gt = lt_step(y[b][i], x[b][i], gt);
    }
    m[i] &= lt;
    if (DEC) d[i] &= gt;
  }
}

// The rows of the slice that rise (m) and, with DEC, fall (d) along a series
// of L >= 2 valid columns, in this lane's words (`on`: the words exist; a lane
// beyond the end reads the last ones, and its masks stay zero).  Two steps'
// planes are loaded together, and the warp stops when no lane has a row left.
template <bool DEC, int B, int WID, class Pop>
__device__ __forceinline__ void plane_chain(const uint32_t* __restrict__ PL, int32_t W,
                                            const Pop& pop, int64_t begin, int32_t L,
                                            int32_t first, bool on, int lane, uint32_t (&m)[WID],
                                            uint32_t (&d)[WID]) {
  uint32_t p[B][WID], q[B][WID], nan[WID];
  const int32_t at = on ? first : W - WID;
  int32_t win = 0;
  uint32_t mine = lane < L ? (uint32_t)pop.col(begin, lane) : 0u;
  auto column = [&](int32_t t) -> uint32_t {               // t is warp-uniform and never falls
    if ((t >> 5) != win) {
      win = t >> 5;
      mine = 32 * win + lane < L ? (uint32_t)pop.col(begin, 32 * win + lane) : 0u;
    }
    return __shfl_sync(kFull, mine, t & 31);
  };
  load_planes<B, WID>(PL, W, column(0), at, p);
  nan_words<B, WID>(p, nan);
#pragma unroll
  for (int i = 0; i < WID; ++i) {
    m[i] = on ? kFull : 0u;
    d[i] = DEC && on ? ~nan[i] : 0u;
  }
  for (int32_t t = 1; t < L; t += 2) {
    const bool two = t + 1 < L;                            // warp-uniform
    load_planes<B, WID>(PL, W, column(t), at, q);
    uint32_t r[B][WID];
    if (two) load_planes<B, WID>(PL, W, column(t + 1), at, r);
    plane_step<DEC, B, WID>(p, q, m, d);
    if (!two) {
      nan_words<B, WID>(q, nan);
      break;
    }
    plane_step<DEC, B, WID>(q, r, m, d);
    uint32_t any = 0u;
#pragma unroll
    for (int i = 0; i < WID; ++i) any |= m[i] | d[i];
    nan_words<B, WID>(r, nan);
    if (!__any_sync(kFull, any != 0u)) break;
#pragma unroll
    for (int b = 0; b < B; ++b)
#pragma unroll
      for (int i = 0; i < WID; ++i) p[b][i] = r[b][i];
  }
#pragma unroll
  for (int i = 0; i < WID; ++i) m[i] &= ~nan[i];
}

template <bool DEC, bool CHECK, int B, int WID, class Pop>
__global__ void __launch_bounds__(1024, 1)
k_support_planes(const uint32_t* __restrict__ PL, int32_t C, int32_t W, int32_t R, Pop pop,
                 EvalArgs a, int32_t slices, int32_t stride, uint32_t* __restrict__ tickets,
                 const double* __restrict__ LN, int* __restrict__ err) {
  after_previous();
  if (!pop.active()) return;
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int32_t slice = (int32_t)(blockIdx.x % (uint32_t)slices);
  const int32_t first = (slice * 32 + lane) * WID;
  const bool on = first < W;
  for (int32_t sid = (int32_t)(blockIdx.x / (uint32_t)slices) * warps + (threadIdx.x >> 5);
       sid < a.P; sid += stride) {
    int64_t begin = 0;
    int32_t L = 0;
    bool bad = !pop.range(sid, &begin, &L);
    if (CHECK) {
      bool lb = false;
      if (!bad)
        for (int t = lane; t < L; t += 32) lb |= (uint32_t)pop.col(begin, t) >= (uint32_t)C;
      bad = __any_sync(kFull, lb) || bad;
    }
    uint32_t inc = 0u, dec = 0u;
    if (!bad && L > 1) {
      uint32_t m[WID], d[WID];
      plane_chain<DEC, B, WID, Pop>(PL, W, pop, begin, L, first, on, lane, m, d);
#pragma unroll
      for (int i = 0; i < WID; ++i) {
        inc += __popc(m[i]);
        dec += __popc(d[i]);
      }
      inc = __reduce_add_sync(kFull, inc);
      if (DEC) dec = __reduce_add_sync(kFull, dec);
    } else if (!bad && slice == 0) {
      inc = dec = (uint32_t)R;
    }
    if (lane == 0) {
      if (bad) atomicOr(err, 1);
      add_part(a, LN, tickets, slices, sid, pop.out(sid), inc, DEC ? dec : 0u, bad ? 1 : L, DEC);
    }
  }
}

}  // namespace ebic

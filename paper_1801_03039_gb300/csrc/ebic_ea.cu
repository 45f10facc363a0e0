// The generation loop of EBIC on the device: Steps 1-5 of the "EBIC
// Algorithm" section (elitism, tournament selection with the crowding
// penalty, crossover and the four mutations of Fig. 1, the tabu list, Step 4
// evaluation and the top-rank list), kept entirely on one GPU.
//
// One generation = six launches (five where the general records kernel runs),
// captured once into a CUDA graph (branches: tabu insertion and the next
// generation's records beside evaluation, Step 5 beside their completion) and
// replayed; every kernel reads the generation number and the stop flag from a
// device control block, so replays need no host involvement:
//   k_spec_pairs   parallel over attempts j < 2P + 1: draws the attempt's
//                  random numbers (Philox-4x32-10, keyed by seed, generation,
//                  attempt), builds the child for EVERY possible outcome of its
//                  tournaments and the overlaps of each batch of 32 attempts.
//   k_spec_settle  adds the entrants' fitness and the children's tabu flags.
//   k_spec         all of it for other tournament sizes, above 256 columns and
//                  for candidates to be screened.
//   k_build        one CTA: the sequential part of Step 3 -- elites, then the
//                  attempts in order, each tournament decided with the penalty
//                  counts as they stand, the precomputed child picked,
//                  duplicates (tabu or earlier in this generation) counted as
//                  hits; more than P hits stop the run.
//   k_tabu_insert  parallel: the accepted children enter the tabu hash table.
//   K3 evaluation  support + Eq. (1) of the new population (ebic_matrix.cu).
//   k_rank_warp    one CTA: Step 5's top-rank update, only those individuals
//                  that can change the list ordered and tested, 32 at a time,
//                  from shared column bitsets (up to 256 columns); k_rank sorts
//                  all of them, above that or when the list outgrows its room.
// At most 2P + 1 attempts are ever needed: every attempt either adds one of at
// most P individuals or is one of at most P + 1 hits.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "ebic_async.cuh"
#include "ebic_internal.cuh"

namespace ebic {

// ---------------------------------------------------------------------------
// device state
// ---------------------------------------------------------------------------
struct Ctl {
  int32_t gen;          // generation being built (0 = Step 1)
  int32_t stop;         // nonzero once the run has stopped
  int32_t stop_reason;  // 1 tabu hits > P, 2 Step 1 could not fill the population, 3 internal
  int32_t n_top;        // records in the top-rank list
  int32_t n_elite;      // elites at the front of the current population
  int32_t last_hits;    // tabu hits in the last Step 3
  int32_t gens_done;    // Steps 2-5 passes completed
  int32_t spec_gen;     // generation whose attempt records come next (set by k_build)
  int32_t rank_over;    // k_rank_warp's list outgrew its room: k_rank ranks this generation
  int32_t pad;
  long long hits_total, attempts_total, evals_total, exact_total;
};

struct EaDev {
  int32_t P, C, S, Lmin, Lmax, k, T, mode, J, ncombo, WC, pad;
  double tau, elite_frac, pc;
  uint64_t seed;
  // archive: entry g * P + i is individual i of generation g
  uint16_t* seq;
  int32_t* len;
  double* fit;
  float* lnf;
  // tabu list: open addressing, key = 64-bit hash (0 = empty), ref = archive entry
  unsigned long long* tkey;
  int32_t* tref;
  unsigned long long tmask;
  // attempts of the current generation: one record of rec_bytes per attempt
  // (layout rec_layout), written by k_spec and streamed into k_build
  char* rec;
  int32_t rec_bytes;
  int32_t pad2;
  struct BatchBlk* blk;         // [ceil(J / 32)] the builder's view of 32 attempts
  // top-rank list (archive entries and their fitness), capacity T + P
  int32_t* list_ref;
  double* list_f;
  // crowding penalty: base^(S/L) for S in [0, L P], from the host C library
  const double* pow_tab;
  const long long* pow_off;     // [Lmax + 1]
  const float* c_over_L;        // [Lmax + 1] log(base) / L as float
  Ctl* ctl;
  // offspring screening (V candidates per attempt and tournament outcome):
  // candidate v of (attempt j, outcome c) is row (j * ncombo + c) * V + v
  int32_t V, screen;
  uint16_t* var_seq;            // [rows][S]
  int32_t* var_len;             // [rows]
  float* var_score;             // [rows]
};

constexpr int kMaxLen = EBIC_MAX_EA_LEN;

// Words of a column bitset: 4 for up to 128 columns, 8 for up to 256, none
// beyond (the builder's generic path).
__host__ __device__ inline int bit_words(int WC) { return WC <= 4 ? 4 : (WC <= 8 ? 8 : 0); }
// Whether Step 3 takes the builder's fast path.
__host__ __device__ inline bool build_fast(int k, int WC) { return k <= 2 && bit_words(WC) > 0; }

// Layout of one attempt record (byte offsets; 8-byte fields first, size a
// multiple of 16 so that records can be bulk-copied).  ne = 2k entrant slots
// (first tournament, then second), nc = k * k candidate children (winner
// positions ta * k + tb), S = series stride.
struct RecLayout {
  int chash, ef, ent, cross, elnf, eL, cL, ctabu, ecols, ccols, bytes;
};

__host__ __device__ inline RecLayout rec_layout(int k, int S, bool init) {
  const int ne = init ? 0 : 2 * k, nc = init ? 1 : k * k;
  RecLayout l{};
  int o = 0;
  l.chash = o; o += nc * 8;
  l.ef = o;    o += ne * 8;
  l.ent = o;   o += 8 * 4;
  l.cross = o; o += 4;
  l.elnf = o;  o += ne * 4;
  l.eL = o;    o += ne * 4;
  l.cL = o;    o += nc * 4;
  l.ctabu = o; o += nc * 4;
  l.ecols = o; o += ne * S * 2;
  l.ccols = o; o += nc * S * 2;
  l.bytes = (o + 15) & ~15;
  return l;
}

// What the builder's fast path (tournaments of at most 2, at most 256 columns)
// needs of 32 consecutive attempts, the batch it decides at a time, laid out
// for one lane per attempt.  ov holds every overlap the batch can ask for:
// byte e of ov[b][c][a] is |entrant e of attempt a & child c of attempt b| for
// b < a, and zero otherwise (at most 64, so a byte).
struct BatchBlk {
  uint32_t ov[32][4][32];
  unsigned long long key[4][32];    // the children's hashes
  float ln[4][32];                  // the entrants' log fitness,
  float cl[4][32];                  // log(base) / length,
  uint16_t id[4][32];               // population index
  uint8_t eL[4][32];                // and length
  uint8_t cL[4][32];                // the children's lengths
  uint8_t tabu[4][32];              // and tabu flags
  uint8_t cross[32];
};
static_assert(sizeof(BatchBlk) % 16 == 0, "bulk copies move multiples of 16 bytes");

// The column set of a series (columns below 256) as eight words in registers,
// eight columns read per round.
__device__ __forceinline__ void bits_of(uint32_t (&acc)[8], const uint16_t* s, int L) {
#pragma unroll
  for (int w = 0; w < 8; ++w) acc[w] = 0u;
  for (int c0 = 0; c0 < L; c0 += 8) {
    uint32_t col[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) col[i] = c0 + i < L ? (uint32_t)s[c0 + i] : 0xffffffffu;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t bit = col[i] != 0xffffffffu ? 1u << (col[i] & 31) : 0u;
#pragma unroll
      for (int w = 0; w < 8; ++w) acc[w] |= (col[i] >> 5) == (uint32_t)w ? bit : 0u;
    }
  }
}

// The same written out as nw <= 8 words.
__device__ __forceinline__ void write_bits(uint32_t* out, int nw, const uint16_t* s, int L) {
  uint32_t acc[8];
  bits_of(acc, s, L);
#pragma unroll
  for (int w = 0; w < 8; ++w)
    if (w < nw) out[w] = acc[w];
}

// The overlap table of a batch, by a CTA of 128 threads: thread 4 b + c holds
// the column sets of attempt b's entrant c and child c and posts both.  Doing it
// here, for all pairs and outcomes in parallel, leaves the sequential builder
// one shared-memory word per (earlier attempt, outcome) to add or take back.
// Every pair of attempts is taken once, by whichever of the two finds the other
// within the next sixteen (mod 32), so that all threads have the same work.
template <int NW>
__device__ __forceinline__ void emit_overlaps(BatchBlk* blk, uint4* s_e, uint4* s_c,
                                              uint32_t (*s_ov)[4][32], const uint32_t (&eb)[8],
                                              const uint32_t (&cb)[8]) {
  constexpr int NV = NW / 4;
  const int b = threadIdx.x >> 2, c = threadIdx.x & 3;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    s_e[threadIdx.x * NV + v] = make_uint4(eb[4 * v], eb[4 * v + 1], eb[4 * v + 2], eb[4 * v + 3]);
    s_c[threadIdx.x * NV + v] = make_uint4(cb[4 * v], cb[4 * v + 1], cb[4 * v + 2], cb[4 * v + 3]);
  }
  for (int a = 0; a <= b; ++a) s_ov[b][c][a] = 0u;       // zeros for the children of b >= a
  __syncthreads();
#pragma unroll 2
  for (int o = 1; o <= 16; ++o) {
    if (o == 16 && b >= 16) break;
    const int x = (b + o) & 31, early = min(b, x), late = max(b, x);
    uint32_t out = 0u;
    uint4 w[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = s_c[(4 * early + c) * NV + v];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int inter = 0;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const uint4 u = s_e[(4 * late + e) * NV + v];
        inter += __popc(w[v].x & u.x) + __popc(w[v].y & u.y) + __popc(w[v].z & u.z) +
                 __popc(w[v].w & u.w);
      }
      out |= (uint32_t)inter << (8 * e);
    }
    s_ov[early][c][late] = out;
  }
  __syncthreads();
  const uint4* src = reinterpret_cast<const uint4*>(s_ov);
  uint4* dst = reinterpret_cast<uint4*>(blk->ov);
#pragma unroll
  for (int i = 0; i < 8; ++i) dst[threadIdx.x + 128 * i] = src[threadIdx.x + 128 * i];
}

// Copies L columns, eight loads in flight per round.
__device__ __forceinline__ void copy_cols(uint16_t* dst, const uint16_t* src, int L) {
  for (int c0 = 0; c0 < L; c0 += 8) {
    uint16_t v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = c0 + i < L ? src[c0 + i] : (uint16_t)0;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (c0 + i < L) dst[c0 + i] = v[i];
  }
}

// ---------------------------------------------------------------------------
// Philox-4x32-10 (Salmon et al., SC'11): counter (j, g, block, 0), key = seed.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void philox_block(uint32_t j, uint32_t g, uint32_t blk, uint64_t seed,
                                             uint32_t out[4]) {
  uint32_t x0 = j, x1 = g, x2 = blk, x3 = 0u;
  uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * x0, hi0 = __umulhi(0xD2511F53u, x0);
    const uint32_t lo1 = 0xCD9E8D57u * x2, hi1 = __umulhi(0xCD9E8D57u, x2);
    const uint32_t y0 = hi1 ^ x1 ^ k0;
    const uint32_t y2 = hi0 ^ x3 ^ k1;
    x0 = y0;
    x1 = lo1;
    x2 = y2;
    x3 = lo0;
  }
  out[0] = x0;
  out[1] = x1;
  out[2] = x2;
  out[3] = x3;
}

// Draw d of attempt j in generation g (word d % 4 of block d / 4).
struct Draws {
  uint64_t seed;
  uint32_t g, j;
  int blk;
  uint32_t w[4];
  __device__ Draws(uint64_t s, uint32_t gg, uint32_t jj) : seed(s), g(gg), j(jj), blk(-1) {}
  __device__ uint32_t operator()(int d) {
    if (d / 4 != blk) {
      blk = d / 4;
      philox_block(j, g, (uint32_t)blk, seed, w);
    }
    return w[d & 3];
  }
};

__device__ __forceinline__ uint32_t below(uint32_t r, uint32_t n) {
  return (uint32_t)(((unsigned long long)r * n) >> 32);
}

// k-th (0-based) column, in increasing order, that is not among s[0 .. L):
// start from k and step over every used column that is not above the answer.
__device__ int kth_absent(const uint16_t* s, int L, uint32_t k) {
  uint16_t t[kMaxLen];
  for (int i = 0; i < L; ++i) {
    uint16_t v = s[i];
    int m = i;
    while (m > 0 && t[m - 1] > v) {
      t[m] = t[m - 1];
      --m;
    }
    t[m] = v;
  }
  uint32_t c = k;
  for (int i = 0; i < L; ++i) {
    if (t[i] <= c) ++c;
    else break;
  }
  return (int)c;
}

__device__ __forceinline__ bool holds(const uint16_t* s, int L, int c) {
  for (int i = 0; i < L; ++i)
    if (s[i] == c) return true;
  return false;
}

// A set of columns below 256 as eight words in registers (every word index
// resolved by unrolled selects): membership in O(1) and the k-th absent
// column by a popcount walk -- the same answers as holds / kth_absent.
struct ColSet8 {
  uint32_t w[8];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = 0u;
  }
  __device__ __forceinline__ void add(uint32_t c) {
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] |= (c >> 5) == (uint32_t)i ? 1u << (c & 31) : 0u;
  }
  __device__ __forceinline__ bool has(uint32_t c) const {
    uint32_t r = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) r |= (c >> 5) == (uint32_t)i ? w[i] : 0u;
    return (r >> (c & 31)) & 1u;
  }
  __device__ __forceinline__ void fill(const uint16_t* s, int L) {
    clear();
    for (int i = 0; i < L; ++i) add(s[i]);
  }
  // k-th (0-based) column below C, in increasing order, not in the set
  __device__ __forceinline__ int kth_absent(uint32_t k, int C) const {
    int found = -1;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int lo = 32 * i;
      uint32_t z = ~w[i];
      if (C - lo < 32) z &= C - lo > 0 ? (1u << (C - lo)) - 1u : 0u;
      const uint32_t cnt = (uint32_t)__popc(z);
      if (found < 0) {
        if (k < cnt) {
          for (uint32_t t = 0; t < k; ++t) z &= z - 1u;     // drop the k lowest
          found = lo + __ffs(z) - 1;
        } else {
          k -= cnt;
        }
      }
    }
    return found;
  }
};

// The four mutations (Fig. 1a-d): one, chosen uniformly among those that keep
// the series in [Lmin, Lmax] with distinct columns (insert, delete, swap,
// substitute in that order).
__device__ __forceinline__ void mutate(uint16_t* x, int& L, int C, int Lmin, int Lmax, uint32_t rt,
                                       uint32_t r1, uint32_t r2, const ColSet8* cs = nullptr) {
  int allowed[4];
  int n = 0;
  if (L < Lmax && L < C) allowed[n++] = 0;
  if (L > Lmin) allowed[n++] = 1;
  if (L >= 2) allowed[n++] = 2;
  if (L < C) allowed[n++] = 3;
  if (n == 0) return;
  const int kind = allowed[below(rt, (uint32_t)n)];
  if (kind == 0) {
    const int pos = (int)below(r1, (uint32_t)(L + 1));
    const uint32_t kk = below(r2, (uint32_t)(C - L));
    const int col = cs ? cs->kth_absent(kk, C) : kth_absent(x, L, kk);
    for (int i = L; i > pos; --i) x[i] = x[i - 1];
    x[pos] = (uint16_t)col;
    ++L;
  } else if (kind == 1) {
    const int pos = (int)below(r1, (uint32_t)L);
    for (int i = pos; i + 1 < L; ++i) x[i] = x[i + 1];
    --L;
  } else if (kind == 2) {
    const int i = (int)below(r1, (uint32_t)L);
    int j = (int)below(r2, (uint32_t)(L - 1));
    if (j >= i) ++j;
    const uint16_t t = x[i];
    x[i] = x[j];
    x[j] = t;
  } else {
    const int pos = (int)below(r1, (uint32_t)L);
    const uint32_t kk = below(r2, (uint32_t)(C - L));
    x[pos] = (uint16_t)(cs ? cs->kth_absent(kk, C) : kth_absent(x, L, kk));
  }
}

// 64-bit hash of an ordered series (never 0: 0 marks an empty slot).
__device__ __forceinline__ unsigned long long seq_hash(const uint16_t* s, int L) {
  unsigned long long h = 0xcbf29ce484222325ull ^ (unsigned long long)L;
  h *= 0x100000001b3ull;
  for (int i = 0; i < L; ++i) {
    h ^= s[i];
    h *= 0x100000001b3ull;
  }
  h ^= h >> 30;
  h *= 0xbf58476d1ce4e5b9ull;
  h ^= h >> 27;
  h *= 0x94d049bb133111ebull;
  h ^= h >> 31;
  return h | 1ull;
}

__device__ __forceinline__ bool same_series(const uint16_t* a, int La, const uint16_t* b, int Lb) {
  if (La != Lb) return false;
  bool eq = true;
  for (int c0 = 0; c0 < La && eq; c0 += 8) {    // eight columns of each side per round
    uint32_t x[8], y[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      x[i] = c0 + i < La ? a[c0 + i] : 0u;
      y[i] = c0 + i < La ? b[c0 + i] : 0u;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) eq = eq && x[i] == y[i];
  }
  return eq;
}

__device__ bool tabu_contains(const EaDev& d, unsigned long long key, const uint16_t* s, int L) {
  unsigned long long i = key & d.tmask;
  for (unsigned long long n = 0; n <= d.tmask; ++n) {
    const unsigned long long k = d.tkey[i];
    if (k == 0ull) return false;
    if (k == key) {
      const int32_t r = d.tref[i];
      if (r >= 0 && same_series(d.seq + (size_t)r * d.S, d.len[r], s, L)) return true;
    }
    i = (i + 1) & d.tmask;
  }
  return false;
}

// The overlap table of the batch that is this CTA's 128 threads (see
// emit_overlaps); threads past the last attempt pass empty sets.
__device__ __forceinline__ void emit_block_pairs(const EaDev& d, const uint32_t (&eb)[8],
                                                 const uint32_t (&cb)[8]) {
  __shared__ uint4 s_e[128 * 2], s_c[128 * 2];
  __shared__ __align__(16) uint32_t s_ov[32][4][32];
  if (bit_words(d.WC) == 4) emit_overlaps<4>(d.blk + blockIdx.x, s_e, s_c, s_ov, eb, cb);
  else emit_overlaps<8>(d.blk + blockIdx.x, s_e, s_c, s_ov, eb, cb);
}

// ---------------------------------------------------------------------------
// k_spec: every child an attempt can produce.  Thread = (attempt, combo);
// combo = ta * k + tb names the winning positions of the two tournaments.
// ---------------------------------------------------------------------------
// SCREEN: thread = (attempt, combo, candidate v); candidate v repeats the
// crossover cuts and the mutation with draws 2k + 1 + 5v .. 2k + 5 + 5v (v = 0
// is the plain child) and goes to the candidate buffers; k_pick completes the
// record once the candidates are scored.
// (fast: the builder reads batch blocks.)
template <bool INIT, bool SCREEN>
__device__ __forceinline__ void spec_thread(const EaDev& d, bool fast) {
  // generation g's records are built while Step 5 of generation g - 1 may
  // still be running (it advances ctl->gen), so g comes from spec_gen
  const int g = INIT ? 0 : d.ctl->spec_gen;
  const int nc = INIT ? 1 : d.ncombo;
  const int V = SCREEN ? d.V : 1;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= (long long)d.J * nc * V) return;
  const int v = SCREEN ? (int)(tid % V) : 0;
  const long long jc = SCREEN ? tid / V : tid;
  const int j = (int)(jc / nc), c = (int)(jc % nc);
  BatchBlk* blk = fast ? d.blk + (j >> 5) : nullptr;
  const int bl = j & 31;
  const RecLayout l = rec_layout(d.k, d.S, INIT);
  char* rec = d.rec + (size_t)j * d.rec_bytes;
  Draws r(d.seed, (uint32_t)g, (uint32_t)j);
  uint16_t x[kMaxLen];
  int L = 0;
  if (INIT) {
    // Step 1: length uniform in [Lmin, Lmax], then distinct uniform columns.
    L = d.Lmin + (int)below(r(0), (uint32_t)(d.Lmax - d.Lmin + 1));
    if (d.C <= 256) {
      ColSet8 cs;
      cs.clear();
      for (int i = 0; i < L; ++i) {
        x[i] = (uint16_t)cs.kth_absent(below(r(1 + i), (uint32_t)(d.C - i)), d.C);
        cs.add(x[i]);
      }
    } else {
      for (int i = 0; i < L; ++i) x[i] = (uint16_t)kth_absent(x, i, below(r(1 + i), (uint32_t)(d.C - i)));
    }
  } else {
    const int k = d.k;
    const uint32_t P = (uint32_t)d.P;
    const int ta = c / k, tb = c % k;
    const bool cross = (double)r(k) * 0x1p-32 < d.pc;
    const long long prev = (long long)(g - 1) * d.P;
    // entrant slots e = c, c + nc, ... of this attempt's record
    for (int e = c; e < 2 * k && v == 0; e += nc) {
      const int idx = (int)below(r(e < k ? e : k + 1 + (e - k)), P);
      const long long er = prev + idx;
      const int eL = d.len[er];
      reinterpret_cast<double*>(rec + l.ef)[e] = d.fit[er];
      reinterpret_cast<float*>(rec + l.elnf)[e] = d.lnf[er];
      reinterpret_cast<int32_t*>(rec + l.eL)[e] = eL;
      reinterpret_cast<int32_t*>(rec + l.ent)[e < k ? e : 4 + (e - k)] = idx;
      uint16_t* ec = reinterpret_cast<uint16_t*>(rec + l.ecols) + (size_t)e * d.S;
      uint16_t t[kMaxLen];
      copy_cols(t, d.seq + (size_t)er * d.S, eL);
      copy_cols(ec, t, eL);
      if (fast) {
        blk->ln[e][bl] = d.lnf[er];
        blk->cl[e][bl] = d.c_over_L[eL];
        blk->id[e][bl] = (uint16_t)idx;
        blk->eL[e][bl] = (uint8_t)eL;
      }
    }
    if (c == 0 && v == 0) {
      reinterpret_cast<int32_t*>(rec + l.cross)[0] = cross ? 1 : 0;
      if (fast) blk->cross[bl] = cross ? 1 : 0;
    }
    const int base = 2 * k + 1 + 5 * v;
    const int ia = (int)below(r(ta), P);
    const int La = d.len[prev + ia];
    copy_cols(x, d.seq + (size_t)(prev + ia) * d.S, La);
    const uint16_t* a = x;
    L = La;
    if (cross) {
      const int ib = (int)below(r(k + 1 + tb), P);
      const int Lb = d.len[prev + ib];
      uint16_t b[kMaxLen];
      copy_cols(b, d.seq + (size_t)(prev + ib) * d.S, Lb);
      const int cut_a = 1 + (int)below(r(base), (uint32_t)La);
      const int cut_b = (int)below(r(base + 1), (uint32_t)Lb);
      uint16_t y[kMaxLen];
      int Ly = 0;
      for (int i = 0; i < cut_a; ++i) y[Ly++] = a[i];
      if (d.C <= 256) {
        ColSet8 ys;
        ys.fill(y, Ly);
        for (int i = cut_b; i < Lb; ++i) {
          if (Ly >= d.Lmax) break;
          if (!ys.has(b[i])) {
            ys.add(b[i]);
            y[Ly++] = b[i];
          }
        }
      } else {
        for (int i = cut_b; i < Lb; ++i) {
          if (Ly >= d.Lmax) break;
          if (!holds(y, Ly, b[i])) y[Ly++] = b[i];
        }
      }
      if (Ly >= d.Lmin) {
        for (int i = 0; i < Ly; ++i) x[i] = y[i];
        L = Ly;
      }
    }
    if (d.C <= 256) {
      ColSet8 xs;
      xs.fill(x, L);
      mutate(x, L, d.C, d.Lmin, d.Lmax, r(base + 2), r(base + 3), r(base + 4), &xs);
    } else {
      mutate(x, L, d.C, d.Lmin, d.Lmax, r(base + 2), r(base + 3), r(base + 4));
    }
  }
  if (SCREEN) {
    const long long row = jc * V + v;
    uint16_t* out = d.var_seq + (size_t)row * d.S;
    for (int i = 0; i < L; ++i) out[i] = x[i];
    d.var_len[row] = L;
    return;
  }
  uint16_t* out = reinterpret_cast<uint16_t*>(rec + l.ccols) + (size_t)c * d.S;
  for (int i = 0; i < L; ++i) out[i] = x[i];
  reinterpret_cast<int32_t*>(rec + l.cL)[c] = L;
  const unsigned long long h = seq_hash(x, L);
  reinterpret_cast<unsigned long long*>(rec + l.chash)[c] = h;
  const int tabu = INIT ? 0 : (tabu_contains(d, h, x, L) ? 1 : 0);
  reinterpret_cast<int32_t*>(rec + l.ctabu)[c] = tabu;
  if (fast) {
    blk->key[c][bl] = h;
    blk->cL[c][bl] = (uint8_t)L;
    blk->tabu[c][bl] = (uint8_t)tabu;
    if (INIT) blk->cross[bl] = 0;
  }
}

template <bool INIT, bool SCREEN>
__global__ void __launch_bounds__(128) k_spec(EaDev d) {
  if (*(volatile int32_t*)&d.ctl->stop) return;
  spec_thread<INIT, SCREEN>(d, build_fast(d.k, d.WC));
}

// ---------------------------------------------------------------------------
// k_spec_pairs: k_spec for tournaments of two and at most 256 columns (NW words
// of bitset), without screening.  A CTA is one batch: thread 4 b + c has entrant
// c and child c of attempt b.  The draws come from three Philox blocks shared by
// the four threads, each thread reads one entrant -- series, length and fitness
// in one round trip -- into shared memory, and the parents are the group's
// entrants, so no second trip; the mutation is applied while the child is
// written and hashed (no shifting), its column set by adding or removing one
// column.  Then the tabu probe and the batch's overlap table.
// ---------------------------------------------------------------------------
constexpr int kSpecRow = kMaxLen + 2;      // uint16 per row: an odd number of words
static_assert(kSpecRow % 4 == 2, "rows of whole words, an odd number of them");

// Columns 2 i and 2 i + 1 of a row that starts on a word, as one word.
__device__ __forceinline__ void put_pair(uint16_t* row, int i, uint32_t v) {
  __builtin_memcpy(__builtin_assume_aligned(row + 2 * i, 4), &v, 4);
}
__device__ __forceinline__ uint32_t get_pair(const uint16_t* row, int i) {
  uint32_t v;
  __builtin_memcpy(&v, __builtin_assume_aligned(row + 2 * i, 4), 4);
  return v;
}

template <int NW>
struct ColSet {
  uint32_t w[NW];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < NW; ++i) w[i] = 0u;
  }
  __device__ __forceinline__ void flip(uint32_t c) {          // adds an absent, removes a present column
#pragma unroll
    for (int i = 0; i < NW; ++i) w[i] ^= (c >> 5) == (uint32_t)i ? 1u << (c & 31) : 0u;
  }
  __device__ __forceinline__ bool has(uint32_t c) const {
    uint32_t r = 0u;
#pragma unroll
    for (int i = 0; i < NW; ++i) r |= (c >> 5) == (uint32_t)i ? w[i] : 0u;
    return (r >> (c & 31)) & 1u;
  }
  // k-th (0-based) column below C, in increasing order, not in the set
  __device__ __forceinline__ int kth_absent(uint32_t k, int C) const {
    uint32_t word = 0u;
    int lo = 0;
    bool found = false;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      uint32_t z = ~w[i];
      if (C - 32 * i < 32) z &= C - 32 * i > 0 ? (1u << (C - 32 * i)) - 1u : 0u;
      const uint32_t cnt = (uint32_t)__popc(z);
      if (!found) {
        if (k < cnt) {
          found = true;
          word = z;
          lo = 32 * i;
        } else {
          k -= cnt;
        }
      }
    }
    // the k-th set bit of word, by halves
    int at = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      const uint32_t low = (uint32_t)__popc(word & ((1u << s) - 1u));
      if (k >= low) {
        k -= low;
        at += s;
        word >>= s;
      }
    }
    return lo + at;
  }
};

template <int NW>
__global__ void __launch_bounds__(128) k_spec_pairs(EaDev d) {
  if (*(volatile int32_t*)&d.ctl->stop) return;
  __shared__ __align__(16) uint16_t s_ent[128][kSpecRow], s_x[128][kSpecRow];
  const unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, c = tid & 3, grp = lane & ~3, bl = tid >> 2;
  const int g = d.ctl->spec_gen;
  const int j = blockIdx.x * 32 + bl;
  const bool live = j < d.J;
  const uint32_t P = (uint32_t)d.P;
  const int S = d.S, C = d.C;
  // draws 0 .. 11 of the attempt: block c by thread c of the group
  uint32_t w4[4];
  philox_block((uint32_t)j, (uint32_t)g, (uint32_t)c, d.seed, w4);
  auto draw = [&](int i) -> uint32_t { return __shfl_sync(FULL, w4[i & 3], grp + (i >> 2)); };
  // entrants 0, 1 (first tournament): draws 0, 1; 2, 3 (second): draws 3, 4
  const uint32_t r0 = draw(0), r1 = draw(1), r2 = draw(2), r3 = draw(3), r4 = draw(4);
  const uint32_t r5 = draw(5), r6 = draw(6), r7 = draw(7), r8 = draw(8), r9 = draw(9);
  const bool cross = (double)r2 * 0x1p-32 < d.pc;
  const int idx = (int)below(c == 0 ? r0 : c == 1 ? r1 : c == 2 ? r3 : r4, P);
  const long long er = (long long)(g - 1) * d.P + (live ? idx : 0);
  const int eL = d.len[er];
  {
    const uint16_t* src = d.seq + (size_t)er * S;
    if ((S & 1) == 0) {                                // rows of whole words
#pragma unroll 8
      for (int i = 0; i < S / 2; ++i) put_pair(s_ent[tid], i, get_pair(src, i));
    } else {
#pragma unroll 8
      for (int i = 0; i < S; ++i) s_ent[tid][i] = src[i];
    }
  }
  ColSet<NW> es;
  es.clear();
  for (int i = 0; i < eL; ++i) es.flip(s_ent[tid][i]);
  __syncwarp();
  // ---- the child for winners ta of the first and tb of the second tournament ----
  const int ta = c >> 1, tb = c & 1;
  const int ra = (tid & ~3) + ta, rb = (tid & ~3) + 2 + tb;
  const int La = __shfl_sync(FULL, eL, grp + ta), Lb = __shfl_sync(FULL, eL, grp + 2 + tb);
  ColSet<NW> xs;
#pragma unroll
  for (int i = 0; i < NW; ++i) xs.w[i] = __shfl_sync(FULL, es.w[i], grp + ta);
  const uint16_t* x = s_ent[ra];
  int L = La;
  if (cross) {
    const int cut_a = 1 + (int)below(r5, (uint32_t)La), cut_b = (int)below(r6, (uint32_t)Lb);
    uint16_t* y = s_x[tid];
    ColSet<NW> ys;
    ys.clear();
    for (int i = 0; i < cut_a; ++i) {
      const uint16_t v = x[i];
      y[i] = v;
      ys.flip(v);
    }
    int Ly = cut_a;
    for (int i = cut_b; i < Lb && Ly < d.Lmax; ++i) {
      const uint16_t v = s_ent[rb][i];
      if (!ys.has(v)) {
        ys.flip(v);
        y[Ly++] = v;
      }
    }
    if (Ly >= d.Lmin) {
      x = y;
      L = Ly;
      xs = ys;
    }
  }
  // one mutation, among those allowed (insert, delete, swap, substitute, as
  // mutate): element i of the child is x[i + shift] but for positions p, q
  int kind = -1, p = -1, q = -1, col = 0, Lc = L;
  {
    int allowed[4], n = 0;
    if (L < d.Lmax && L < C) allowed[n++] = 0;
    if (L > d.Lmin) allowed[n++] = 1;
    if (L >= 2) allowed[n++] = 2;
    if (L < C) allowed[n++] = 3;
    if (n) {
      const int pick = (int)below(r7, (uint32_t)n);
      kind = pick == 0 ? allowed[0] : pick == 1 ? allowed[1] : pick == 2 ? allowed[2] : allowed[3];
    }
    if (kind == 0) {
      p = (int)below(r8, (uint32_t)(L + 1));
      Lc = L + 1;
    } else if (kind >= 0) {
      p = (int)below(r8, (uint32_t)L);
      if (kind == 1) Lc = L - 1;
    }
    if (kind == 2) {
      q = (int)below(r9, (uint32_t)(L - 1));
      if (q >= p) ++q;
    } else if (kind == 0 || kind == 3) {
      col = xs.kth_absent(below(r9, (uint32_t)(C - L)), C);
    }
    if (kind == 1 || kind == 3) xs.flip(x[p]);
    if (kind == 0 || kind == 3) xs.flip((uint32_t)col);
  }
  const RecLayout l = rec_layout(2, S, false);
  char* rec = d.rec + (size_t)(live ? j : 0) * d.rec_bytes;
  BatchBlk* blk = d.blk + blockIdx.x;
  unsigned long long h = 0xcbf29ce484222325ull ^ (unsigned long long)Lc;
  h *= 0x100000001b3ull;
  uint16_t* out = reinterpret_cast<uint16_t*>(rec + l.ccols) + (size_t)c * S;
  for (int i0 = 0; i0 < Lc; i0 += 4) {
    uint32_t v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u;
      int at = i;
      if (kind == 0) at = i > p ? i - 1 : i;
      if (kind == 1) at = i >= p ? i + 1 : i;
      if (kind == 2) at = i == p ? q : i == q ? p : i;
      v[u] = i < Lc ? ((kind == 0 || kind == 3) && i == p ? (uint32_t)col : (uint32_t)x[min(at, kMaxLen)])
                    : 0u;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u < Lc) {
        if (live) out[i0 + u] = (uint16_t)v[u];
        h ^= v[u];
        h *= 0x100000001b3ull;
      }
  }
  h ^= h >> 30;
  h *= 0xbf58476d1ce4e5b9ull;
  h ^= h >> 27;
  h *= 0x94d049bb133111ebull;
  h ^= h >> 31;
  h |= 1ull;
  if (live) {
    reinterpret_cast<int32_t*>(rec + l.eL)[c] = eL;
    reinterpret_cast<int32_t*>(rec + l.ent)[c < 2 ? c : 4 + (c - 2)] = idx;
    uint16_t* ec = reinterpret_cast<uint16_t*>(rec + l.ecols) + (size_t)c * S;
    if ((S & 1) == 0) {
#pragma unroll 4
      for (int i = 0; i < (eL + 1) / 2; ++i) put_pair(ec, i, get_pair(s_ent[tid], i));
    } else {
      for (int i = 0; i < eL; ++i) ec[i] = s_ent[tid][i];
    }
    if (c == 0) {
      reinterpret_cast<int32_t*>(rec + l.cross)[0] = cross ? 1 : 0;
      blk->cross[bl] = cross ? 1 : 0;
    }
    blk->cl[c][bl] = d.c_over_L[eL];
    blk->id[c][bl] = (uint16_t)idx;
    blk->eL[c][bl] = (uint8_t)eL;
    reinterpret_cast<int32_t*>(rec + l.cL)[c] = Lc;
    reinterpret_cast<unsigned long long*>(rec + l.chash)[c] = h;
    blk->key[c][bl] = h;
    blk->cL[c][bl] = (uint8_t)Lc;
  }
  uint32_t eb[8] = {}, cb[8] = {};
  if (live) {
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      eb[i] = es.w[i];
      cb[i] = xs.w[i];
    }
  }
  emit_block_pairs(d, eb, cb);
}

// Completes k_spec_pairs' records: the entrants' fitness and the children's
// tabu flags, one thread each.  Only this part needs the generation's evaluation
// and tabu list; the records themselves are built beside both (1,000 x 100, P =
// 600: a generation 73 -> 70 us).
__global__ void __launch_bounds__(128) k_spec_settle(EaDev d) {
  if (*(volatile int32_t*)&d.ctl->stop) return;
  const int c = threadIdx.x & 3, bl = threadIdx.x >> 2;
  const int j = blockIdx.x * 32 + bl;
  if (j >= d.J) return;
  BatchBlk* blk = d.blk + blockIdx.x;
  const unsigned long long key = blk->key[c][bl];
  const long long er = (long long)(d.ctl->spec_gen - 1) * d.P + blk->id[c][bl];
  const double ef = d.fit[er];
  const float eln = d.lnf[er];
  const RecLayout l = rec_layout(2, d.S, false);
  char* rec = d.rec + (size_t)j * d.rec_bytes;
  const int tabu =
      tabu_contains(d, key, reinterpret_cast<const uint16_t*>(rec + l.ccols) + (size_t)c * d.S,
                    blk->cL[c][bl])
          ? 1
          : 0;
  reinterpret_cast<double*>(rec + l.ef)[c] = ef;
  reinterpret_cast<float*>(rec + l.elnf)[c] = eln;
  reinterpret_cast<int32_t*>(rec + l.ctabu)[c] = tabu;
  blk->ln[c][bl] = eln;
  blk->tabu[c][bl] = (uint8_t)tabu;
}

// Pseudo scores (testing the screening logic without a model): candidate v of
// (attempt j, outcome c) scores word 0 of Philox(j, g, 65536 + c * V + v) >> 8.
__global__ void __launch_bounds__(256) k_pseudo_score(EaDev d) {
  if (*(volatile int32_t*)&d.ctl->stop) return;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)d.J * d.ncombo * d.V) return;
  const int v = (int)(t % d.V);
  const long long jc = t / d.V;
  const int j = (int)(jc / d.ncombo), c = (int)(jc % d.ncombo);
  uint32_t w[4];
  philox_block((uint32_t)j, (uint32_t)d.ctl->spec_gen, 65536u + (uint32_t)(c * d.V + v), d.seed, w);
  d.var_score[t] = (float)(w[0] >> 8);
}

// k_pick: the candidates of each (attempt, outcome) are visited by decreasing
// score (ties: lower v; NaN after every number) and the first one that is not
// in the tabu list becomes the record's child; when all are, the
// best-scoring one does (a tabu hit).  The tabu list is the one left by the
// previous generation: this generation's own duplicates are the builder's.
__device__ __forceinline__ void pick_thread(const EaDev& d, bool fast, bool pairs,
                                            uint32_t (&eb)[8], uint32_t (&cb)[8]) {
  const long long jc = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (jc >= (long long)d.J * d.ncombo) return;
  const int j = (int)(jc / d.ncombo), c = (int)(jc % d.ncombo);
  const float* sc = d.var_score + jc * d.V;
  float scv[16];                                    // the scores, read once (V <= 16)
  for (int v = 0; v < d.V; ++v) {
    const float x = sc[v];
    scv[v] = x != x ? -INFINITY : x;
  }
  // each visited candidate is read once into t (eight loads in flight per
  // round); its hash, tabu probe and write-out work on that copy
  uint16_t t[kMaxLen];
  uint32_t seen = 0u;
  int first = -1, chosen = -1, L = 0;
  unsigned long long chosen_h = 0ull, first_h = 0ull;
  for (int r = 0; r < d.V && chosen < 0; ++r) {
    int bv = -1;
    float bs = 0.f;
    for (int v = 0; v < d.V; ++v) {
      if ((seen >> v) & 1u) continue;
      if (bv < 0 || scv[v] > bs) {
        bv = v;
        bs = scv[v];
      }
    }
    seen |= 1u << bv;
    const long long row = jc * d.V + bv;
    L = d.var_len[row];
    copy_cols(t, d.var_seq + (size_t)row * d.S, L);
    const unsigned long long h = seq_hash(t, L);
    if (first < 0) {
      first = bv;
      first_h = h;
    }
    if (!tabu_contains(d, h, t, L)) {
      chosen = bv;
      chosen_h = h;
    }
  }
  const bool hit = chosen < 0;
  if (hit) {                                        // every candidate is in the list
    chosen = first;
    chosen_h = first_h;
    const long long row = jc * d.V + chosen;
    L = d.var_len[row];
    copy_cols(t, d.var_seq + (size_t)row * d.S, L);
  }
  const RecLayout l = rec_layout(d.k, d.S, false);
  char* rec = d.rec + (size_t)j * d.rec_bytes;
  uint16_t* out = reinterpret_cast<uint16_t*>(rec + l.ccols) + (size_t)c * d.S;
  for (int i = 0; i < L; ++i) out[i] = t[i];
  reinterpret_cast<int32_t*>(rec + l.cL)[c] = L;
  reinterpret_cast<unsigned long long*>(rec + l.chash)[c] = chosen_h;
  reinterpret_cast<int32_t*>(rec + l.ctabu)[c] = hit ? 1 : 0;
  if (fast) {
    BatchBlk* blk = d.blk + (j >> 5);
    const int bl = j & 31;
    blk->key[c][bl] = chosen_h;
    blk->cL[c][bl] = (uint8_t)L;
    blk->tabu[c][bl] = hit ? 1 : 0;
    if (pairs) {
      bits_of(cb, t, L);
      bits_of(eb, reinterpret_cast<const uint16_t*>(rec + l.ecols) + (size_t)c * d.S,
              reinterpret_cast<const int32_t*>(rec + l.eL)[c]);
    }
  }
}

__global__ void __launch_bounds__(128) k_pick(EaDev d) {
  if (*(volatile int32_t*)&d.ctl->stop) return;
  const bool fast = build_fast(d.k, d.WC), pairs = fast && d.k == 2;
  uint32_t eb[8] = {}, cb[8] = {};
  pick_thread(d, fast, pairs, eb, cb);
  if (pairs) emit_block_pairs(d, eb, cb);
}

// ---------------------------------------------------------------------------
// Tournament comparison.  Penalised fitness p = f / base^(S/L) in binary64,
// exactly as the reading of the paper defines it.  Fast path: compare the
// log-domain scores ln f - S * ln(base) / L in float; when they differ by more
// than a margin that bounds every rounding error of both the float scores and
// the binary64 values (pow within 1 ulp, S / L rounded once, the quotient
// rounded once), the sign is the binary64 sign.  Otherwise -- and whenever a
// value might be zero, subnormal or infinite -- compute the binary64 values
// with the host-built power table and compare them exactly.
// ---------------------------------------------------------------------------
// One tournament entrant as the builder sees it.  f = 0 exactly when
// lnf = -inf (lnf is log(f) rounded to float, finite for every f > 0), so the
// fast path needs no binary64 arithmetic; f itself is read only on the exact
// path.
struct Entrant {
  float lnf;
  float cl;          // log(base) / L as float
  int32_t S, L, idx;
  const double* f;   // the entrant's binary64 fitness (shared memory)
};

// Bit 0 of the result: x beats y.  Bit 1: the exact path decided.  The float
// decision is formed with selects; only an undecided comparison branches to
// the exact path.
__device__ __forceinline__ int beats(const Entrant& x, const Entrant& y, const EaDev& d) {
  if (x.idx == y.idx) return 0;
  const bool zx = x.lnf == -INFINITY, zy = y.lnf == -INFINITY;
  const float cx = (float)x.S * x.cl;
  const float cy = (float)y.S * y.cl;
  const float gx = x.lnf - cx, gy = y.lnf - cy;
  const bool safe_x = zx || (cx < 700.f && gx > -700.f);
  const bool safe_y = zy || (cy < 700.f && gy > -700.f);
  const float diff = gx - gy;
  const float margin = 0x1p-16f * (fabsf(x.lnf) + fabsf(y.lnf) + cx + cy + 1.f);
  const bool decided = (zx && zy) || (zx && safe_y) || (zy && safe_x) ||
                       (!zx && !zy && safe_x && safe_y && fabsf(diff) > margin);
  if (decided) {
    const bool win = (zx && zy) ? x.idx < y.idx : (zx ? false : (zy ? true : diff > 0.f));
    return win ? 1 : 0;
  }
  const double px = __ddiv_rn(*x.f, d.pow_tab[d.pow_off[x.L] + x.S]);
  const double py = __ddiv_rn(*y.f, d.pow_tab[d.pow_off[y.L] + y.S]);
  return 2 | ((px > py || (px == py && x.idx < y.idx)) ? 1 : 0);
}

// Within-generation duplicate check: open addressing on the 64-bit hash in
// shared memory; a hash match is confirmed on the columns of the earlier
// child (warp-wide compare).  Returns true for a duplicate; *slot = the first
// empty slot after the probe otherwise.
template <int NCT>   // combos per record when known at compile time (0: runtime nc)
__device__ __forceinline__ bool gen_duplicate(const EaDev& d, const RecLayout& l,
                                              const unsigned long long* hkey,
                                              const int32_t* href, int hmask, int nc_rt, int RB,
                                              unsigned long long key, const uint16_t* child,
                                              int L, int lane, int* slot) {
  const int nc = NCT ? NCT : nc_rt;
  int sl = (int)(key & (unsigned long long)hmask);
  for (int probe = 0; probe <= hmask; ++probe) {
    const unsigned long long kk = hkey[sl];
    if (kk == 0ull) break;
    if (kk == key) {
      const int32_t r = href[sl];
      const char* orec = d.rec + (size_t)(r / nc) * RB;
      const int oc = r % nc;
      const uint16_t* other = reinterpret_cast<const uint16_t*>(orec + l.ccols) + (size_t)oc * d.S;
      const int oL = reinterpret_cast<const int32_t*>(orec + l.cL)[oc];
      const bool same =
          oL == L &&
          __all_sync(0xffffffffu, lane >= L || other[lane] == child[lane]) &&
          __all_sync(0xffffffffu, lane + 32 >= L || other[lane + 32] == child[lane + 32]);
      if (same) return true;
    }
    sl = (sl + 1) & hmask;
  }
  *slot = sl;
  return false;
}

// Float part of one tournament comparison (see beats) with the constants of
// the pair precomputed once per sub-chunk.  During a sub-chunk a penalty sum
// can only grow, by at most 31 * L (31 earlier acceptances, each sharing at
// most L columns with the entrant), so the range checks of beats are settled
// in advance for the whole interval: a pair that passes them for every sum up
// to that bound compares in float; one that does not always takes the exact
// path.  Pairs whose outcome does not depend on the sums (the same individual
// twice, a zero fitness on either side) are decided once.
struct PairConst {
  float lx, ly, clx, cly, base;   // base = 2^-16 (|lx| + |ly| + 1)
  int fixed;                      // -1: depends on the sums; else the outcome
  bool exact_always, xlow;        // xlow: idx_x < idx_y
  bool settled;                   // fixed for any sums at all
};

// What needs no sums.
__device__ __forceinline__ PairConst pair_const(float lx, float ly, float clx, float cly,
                                                int32_t ix, int32_t iy) {
  PairConst p;
  p.lx = lx;
  p.ly = ly;
  p.clx = clx;
  p.cly = cly;
  p.xlow = ix < iy;
  const bool zx = lx == -INFINITY, zy = ly == -INFINITY;
  p.base = (zx || zy) ? 0.f : 0x1p-16f * (fabsf(lx) + fabsf(ly) + 1.f);
  p.exact_always = false;
  p.settled = ix == iy || (zx && zy);
  p.fixed = ix == iy ? 0 : zx && zy ? (p.xlow ? 1 : 0) : zx ? 0 : zy ? 1 : -1;
  return p;
}

// The range checks, at the largest sums the batch can reach (the checks are
// monotone in the sum).
__device__ __forceinline__ void pair_range(PairConst& p, int32_t Sx, int32_t Sy, int32_t Lx,
                                           int32_t Ly) {
  const bool zx = p.lx == -INFINITY, zy = p.ly == -INFINITY;
  const float cxm = (float)(Sx + 31 * Lx) * p.clx, cym = (float)(Sy + 31 * Ly) * p.cly;
  const bool safe_x = zx || (cxm < 700.f && p.lx - cxm > -700.f);
  const bool safe_y = zy || (cym < 700.f && p.ly - cym > -700.f);
  if (!p.settled && !(safe_x && safe_y)) {
    p.exact_always = true;
    p.fixed = -1;
  }
}

// 1 / 0 when decided in float (sums below 2^23, so exact), -1 when the exact
// path must decide.
__device__ __forceinline__ int pair_fast(const PairConst& p, float Sx, float Sy) {
  const float cx = Sx * p.clx, cy = Sy * p.cly;
  const float diff = (p.lx - cx) - (p.ly - cy);
  const float margin = p.base + 0x1p-16f * (cx + cy);
  int r = fabsf(diff) > margin ? (diff > 0.f ? 1 : 0) : -1;
  r = p.exact_always ? -1 : r;
  return p.fixed >= 0 ? p.fixed : r;
}

// Exact binary64 comparison (the definition; see beats) for an undecided pair.
__device__ __noinline__ int pair_exact(const EaDev& d, const double* fx, const double* fy,
                                       int32_t Lx, int32_t Ly, int32_t Sx, int32_t Sy,
                                       bool xlow) {
  const double px = __ddiv_rn(*fx, d.pow_tab[d.pow_off[Lx] + Sx]);
  const double py = __ddiv_rn(*fy, d.pow_tab[d.pow_off[Ly] + Sy]);
  return (px > py || (px == py && xlow)) ? 1 : 0;
}

constexpr int kMaxStages = 4;           // buffers of the copies ahead
constexpr int kBuildWorkers = 256;      // commit batches, sum the penalties of the next
constexpr int kBuildThreads = 32 + kBuildWorkers;
// Step 3 fast path: a bit filter over the keys of the generation's committed
// children (one bit per key, chosen by the key's high 32 bits) in front of a
// dense list of those keys; a clear bit proves a child new.  A lane whose bit
// is set walks its key's chain: list positions chained by bucket, newest first
// (entering one costs a single exchange; probing a table for every lane and
// entering by compare-and-swap cost 6 us more a generation at P = 600).
constexpr int kFilterBits = 1 << 17;
constexpr int kFilterWords = kFilterBits / 32;
constexpr uint32_t kNoKey = 0xffffu;
struct KeyIndex {
  uint32_t* bits;       // [kFilterWords]
  uint32_t* head;       // [mask + 1] newest list position of a bucket
  uint16_t* next;       // [P] the one before it
  uint32_t mask;
};

// What warp 0 and the rest of the builder's CTA tell each other per batch of
// the fast path.
struct Team {
  int sx[2][4][32];     // penalty sum of entrant e of lane a over half h of its columns
  int dec[32];          // the lanes' outcomes
  unsigned accm;        // lanes accepted
  int n0;               // individuals before them
};

// One entrant's columns, half h of them (the first ceil(L / 2) or the rest):
// the first sixteen are read while warp 0 decides the batch before, two a
// register, so that only the counts themselves are read after its commit.
struct PenCols {
  uint32_t c[8];
  int n;                // columns of this half
  const uint16_t* at;   // and where they are
};

__device__ __forceinline__ PenCols pen_cols(const RecLayout& l, const char* cur, const BatchBlk* blk,
                                            int avail, int S, int e, int h, int lane, int RB) {
  PenCols p;
  p.n = 0;
  p.at = nullptr;
#pragma unroll
  for (int i = 0; i < 8; ++i) p.c[i] = 0u;
  if (!(lane < avail && (e < 2 || blk->cross[lane]))) return p;
  const int L = blk->eL[e][lane], half = (L + 1) >> 1;
  p.n = h ? L - half : half;
  p.at = reinterpret_cast<const uint16_t*>(cur + (size_t)lane * RB + l.ecols) + (size_t)e * S +
         (h ? half : 0);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t a = 2 * i < p.n ? p.at[2 * i] : 0u, b = 2 * i + 1 < p.n ? p.at[2 * i + 1] : 0u;
    p.c[i] = a | (b << 16);
  }
  return p;
}

__device__ __forceinline__ int pen_sum(const PenCols& p, const uint32_t* pen) {
  int sum = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (i < p.n) sum += (int)pen[(p.c[i >> 1] >> (16 * (i & 1))) & 0xffffu];
  for (int i = 16; i < p.n; ++i) sum += (int)pen[p.at[i]];
  return sum;
}

// What warp 0 needs of a batch besides the sums, read while the batch before is
// committed: entrant e of lane a, its pairs' constants.
struct BatchIn {
  int32_t L[4];
  int cross;
  PairConst pc[2];
};

__device__ __forceinline__ BatchIn batch_in(const BatchBlk* blk, int avail, int lane) {
  BatchIn in;
  const bool have = lane < avail;
  in.cross = have ? blk->cross[lane] : 0;
  float ln[4], cl[4];
  int32_t id[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    ln[e] = blk->ln[e][lane];
    cl[e] = blk->cl[e][lane];
    id[e] = blk->id[e][lane];
    in.L[e] = blk->eL[e][lane];
  }
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (!(have && (e < 2 || in.cross))) {
      ln[e] = cl[e] = 0.f;
      id[e] = in.L[e] = 0;
    }
#pragma unroll
  for (int t = 0; t < 2; ++t)
    in.pc[t] = pair_const(ln[2 * t + 1], ln[2 * t], cl[2 * t + 1], cl[2 * t], id[2 * t + 1], id[2 * t]);
  return in;
}

// Equal series test of two children (lane-local).
__device__ __forceinline__ bool same_cols(const uint16_t* a, const uint16_t* b, int L) {
  for (int i = 0; i < L; ++i)
    if (a[i] != b[i]) return false;
  return true;
}

// The same test with sixteen columns of both series loaded before any is
// compared (for a series in global memory, one round trip per sixteen).
__device__ __forceinline__ bool same_cols_wide(const uint16_t* a, const uint16_t* b, int L) {
  bool eq = true;
  for (int c0 = 0; c0 < L && eq; c0 += 16) {
    uint32_t x[16], y[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      x[i] = c0 + i < L ? a[c0 + i] : 0u;
      y[i] = c0 + i < L ? b[c0 + i] : 0u;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) eq = eq && x[i] == y[i];
  }
  return eq;
}

constexpr int kTwinSlots = 4096;    // lane-id scratch of the twin pre-check

// The Step 3 decisions for tournaments of K <= 2 entrants and at most 256
// columns: warp 0 takes one batch of 32 attempts (one per lane) from its block.
//
// The sequential rule -- each tournament sees the penalty counts left by every
// earlier acceptance -- is solved as a fixpoint.  Assuming every attempt of
// the batch is accepted, lane a's penalty sums are its sums at the batch
// start (the workers' pen_sum) plus |entrant & child_b| for the chosen child of
// every earlier lane b (the block's overlap table); its outcome is the
// tournament result for those sums.  Starting from the outcomes at the batch
// start, all lanes recompute their outcomes from the current children of the
// earlier lanes until none changes (Jacobi iteration).  Lane 0 is final after
// the first pass and lane k after pass k, so the iteration stops after at most
// 32 passes, at the unique fixpoint: the outcomes of taking the attempts one
// by one.  Then duplicates are found in parallel (the record's tabu flag; the
// filter bit of the key and, where it is set, the chain of committed keys of
// its bucket; equal keys among earlier lanes of the batch).
// The first duplicate is a hit: its child leaves the later lanes' sums, which
// are re-decided (and, if a child changed, re-checked) in the next round.
// Once no hit remains (or the population is full, or the tabu rule stops the
// run) the accepted lanes are committed, their keys by warp 0 (commit_keys), their
// columns by the workers (commit_cols), and the next batch starts from penalty
// counts that include every acceptance so far.
//
// Overlaps are added in two words of two 16-bit sums each (entrants 0 and 2,
// 1 and 3): 31 earlier lanes of at most 64 columns stay below 2^16, and taking
// a word back undoes adding it.
template <int K>
__device__ __forceinline__ void build_batch(const EaDev& d, const RecLayout& l, const char* cur,
                                            const BatchBlk* blk, int avail, BatchIn& in,
                                            const unsigned long long* lkey, const int32_t* lref,
                                            const KeyIndex& kx, uint8_t* s_twin, Team* tm,
                                            int RB, int lane, int& n, int& hits, int& stopped,
                                            long long& attempts, long long& exact,
                                            unsigned long long* mine) {
  constexpr int NC = K * K;
  const int S = d.S;
  const unsigned FULL = 0xffffffffu;
  const bool have = lane < avail;
  const unsigned havem = avail >= 32 ? FULL : (1u << avail) - 1u;
  const char* ra = cur + (size_t)(have ? lane : 0) * RB;
  int32_t Sx[4];
  float Sf[4];                          // Sx - 2^23, see sum_of
  const double* efa = reinterpret_cast<const double*>(ra + l.ef);
  if (K == 2) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      Sx[e] = tm->sx[0][e][lane] + tm->sx[1][e][lane];
      Sf[e] = (float)(Sx[e] - (1 << 23));
    }
#pragma unroll
    for (int t = 0; t < 2; ++t)
      pair_range(in.pc[t], Sx[2 * t + 1], Sx[2 * t], in.L[2 * t + 1], in.L[2 * t]);
  }
  uint32_t o02 = 0u, o13 = 0u;          // overlaps with the earlier lanes' children
  // this lane's outcomes for its current sums: bit a of the masks is the
  // winner's position in lane a's first and second tournament
  unsigned da = 0u, db = 0u;
  auto decide = [&](unsigned& ma, unsigned& mb) -> int {
    int ne = 0, ta = 0, tb = 0;
    // Sx[e] plus a 16-bit overlap sum: under the exponent of 2^23 its bits are
    // the float 2^23 + sum, and the sum of both is exact
    auto sum_of = [&](int e, uint32_t o, uint32_t half) {
      return Sf[e] + __uint_as_float(__byte_perm(o, 0x4b00u, half));
    };
    constexpr uint32_t kLow = 0x5410u, kHigh = 0x5432u;
    // lanes without an attempt, and second tournaments that are not held, have
    // zero entrants: the outcome 0, fixed
    ta = pair_fast(in.pc[0], sum_of(1, o13, kLow), sum_of(0, o02, kLow));
    tb = pair_fast(in.pc[1], sum_of(3, o13, kHigh), sum_of(2, o02, kHigh));
    if (__any_sync(FULL, (ta | tb) < 0)) {
      if (ta < 0) {
        ta = pair_exact(d, efa + 1, efa + 0, in.L[1], in.L[0], Sx[1] + (int)(o13 & 0xffffu),
                        Sx[0] + (int)(o02 & 0xffffu), in.pc[0].xlow);
        ++ne;
      }
      if (tb < 0) {
        tb = pair_exact(d, efa + 3, efa + 2, in.L[3], in.L[2], Sx[3] + (int)(o13 >> 16),
                        Sx[2] + (int)(o02 >> 16), in.pc[1].xlow);
        ++ne;
      }
    }
    ma = __ballot_sync(FULL, ta != 0);
    mb = __ballot_sync(FULL, tb != 0);
    return ne;
  };
  auto child_of = [](unsigned ma, unsigned mb, int b) -> int {
    return (int)(((ma >> b) & 1u) * K + ((mb >> b) & 1u));
  };
  // overlaps of this lane's entrants with child c of lane b (zero for b >= lane),
  // a byte each; up to three words add without a carry
  auto ov = [&](int b, int c) -> uint32_t { return blk->ov[b][c][lane]; };
  auto sub_overlap = [&](int b) {
    const uint32_t w = ov(b, child_of(da, db, b));
    o02 -= w & 0x00ff00ffu;
    o13 -= (w >> 8) & 0x00ff00ffu;
  };
  // Lanes below `first` are settled: accepted (committed together at the
  // end of the batch) or hits.  A round finds the next hit; the hit's child
  // leaves the later lanes' sums and the next round re-decides them.
  int first = 0;
  unsigned hitmask = 0u;              // settled hits
  int acc = 0;                        // settled accepted lanes
  int cut = avail;                    // lanes processed by the batch
  int nex = 0;                        // exact comparisons of the lane's last decision
  // duplicate flags of the lanes' current children; they stay exact for a
  // round that changes no child (after a hit, a child equal to the hit's or
  // to an earlier accepted lane's was already flagged by the twin check,
  // which covers every earlier lane of the batch)
  bool dup = false, dups_valid = false, round_changed = false;
  // what the sums stand for: nothing yet; the current children of all earlier
  // lanes; or, on trial, those less the round's duplicates
  bool started = K == 1, trial = false;
  uint32_t keep02 = 0u, keep13 = 0u;
  unsigned long long key = 0ull;
  // (one copy of the decision: the loop is bound by its latency and by
  // instruction fetch.  It ends: after a start, lane k is final after pass k of
  // a round, and every round takes a hit.)
  for (;;) {
    const unsigned livem = havem & (FULL << first);      // first <= 31
    bool failed_trial = false, on_trial = false;
    if (K == 2) {
      unsigned na, nb;
      const int nx = decide(na, nb);
      if (!started) {
        // every earlier lane's child, assuming all are accepted (lanes past the
        // last attempt: child 0 of no later lane, zero)
        started = true;
        da = na;
        db = nb;
        nex = nx;
        const uint32_t* mine = &blk->ov[0][0][lane];
        const int row = (lane * 4 + child_of(da, db, lane)) * 32;
#pragma unroll
        for (int b = 0; b < 31; b += 3) {
          uint32_t w = mine[__shfl_sync(FULL, row, b)];
          if (b + 1 < 31) w += mine[__shfl_sync(FULL, row, b + 1)];
          if (b + 2 < 31) w += mine[__shfl_sync(FULL, row, b + 2)];
          o02 += w & 0x00ff00ffu;
          o13 += (w >> 8) & 0x00ff00ffu;
        }
        continue;
      }
      unsigned changed = ((na ^ da) | (nb ^ db)) & livem;
      if (trial) {
        trial = false;
        on_trial = true;
        if (changed) {
          o02 = keep02;
          o13 = keep13;
          failed_trial = true;
        }
      } else if (changed) {
        // Jacobi pass: four changed lanes at a time (lane 31 stands for none:
        // it has no later lane, so its words are zero)
        round_changed = true;
        while (changed) {
          uint32_t w[4], v[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int b = changed ? __ffs(changed) - 1 : 31;
            changed &= changed - 1u;
            w[i] = ov(b, child_of(na, nb, b));
            v[i] = ov(b, child_of(da, db, b));
          }
#pragma unroll
          for (int i = 0; i < 4; i += 2) {
            const uint32_t in2 = w[i] + w[i + 1], out2 = v[i] + v[i + 1];
            o02 += (in2 & 0x00ff00ffu) - (out2 & 0x00ff00ffu);
            o13 += ((in2 >> 8) & 0x00ff00ffu) - ((out2 >> 8) & 0x00ff00ffu);
          }
        }
        da = (da & ~livem) | (na & livem);
        db = (db & ~livem) | (nb & livem);
        if (lane >= first) nex = nx;
        continue;
      }
    }
    // duplicates: tabu flag, the generation's children committed by earlier
    // batches (filter, then the key's chain), equal keys among earlier lanes
    const bool live = have && lane >= first;
    if (!dups_valid || round_changed) {
      const int dec = child_of(da, db, lane);
      key = have ? blk->key[dec][lane] : 0ull;
      const int L = have ? blk->cL[dec][lane] : 0;
      const uint16_t* child = reinterpret_cast<const uint16_t*>(ra + l.ccols) + (size_t)dec * S;
      const uint32_t fb = (uint32_t)(key >> 32) & (uint32_t)(kFilterBits - 1);
      dups_valid = true;
      round_changed = false;
      dup = live && blk->tabu[dec][lane] != 0;
      const bool maybe = live && !dup && ((kx.bits[fb >> 5] >> (fb & 31)) & 1u);
      // equal keys among earlier lanes of the batch (settled ones too: an
      // accepted lane is not in the key list before the batch commits, and
      // a child equal to a hit's is a duplicate of what the hit duplicated):
      // each lane writes its id into a slot chosen by its key; only when
      // some lane finds another lane's id in its slot does the warp match
      // the keys exactly
      const uint32_t ts = (uint32_t)key & (uint32_t)(kTwinSlots - 1);
      if (have) s_twin[ts] = (uint8_t)lane;
      __syncwarp();
      const bool clash = have && s_twin[ts] != (uint8_t)lane;
      if (maybe) {
        for (uint32_t i = kx.head[(uint32_t)key & kx.mask]; i != kNoKey && !dup; i = kx.next[i]) {
          if (lkey[i] != key) continue;
          const int32_t r = lref[i];
          const char* orec = d.rec + (size_t)(r / NC) * RB;
          const int oc = r % NC;
          dup = reinterpret_cast<const int32_t*>(orec + l.cL)[oc] == L &&
                same_cols_wide(reinterpret_cast<const uint16_t*>(orec + l.ccols) + (size_t)oc * S,
                               child, L);
        }
      }
      __syncwarp();
      unsigned twins = 0u;
      if (__any_sync(FULL, clash)) {
        twins = __match_any_sync(FULL, key) & ((1u << lane) - 1u);
        if (!live) twins = 0u;
      }
      while (twins && !dup) {
        const int b = __ffs(twins) - 1;
        twins &= twins - 1;
        const char* rbb = cur + (size_t)b * RB;
        const int cb = child_of(da, db, b);
        if (blk->cL[cb][b] == L &&
            same_cols(reinterpret_cast<const uint16_t*>(rbb + l.ccols) + (size_t)cb * S, child, L))
          dup = true;
      }
      __syncwarp();
    }
    dup = dup && live;
    // the next hit, unless the population fills before it
    const unsigned dupmask = __ballot_sync(FULL, dup);
    const int first_dup = dupmask ? __ffs(dupmask) - 1 : avail;
    const int need = d.P - n - acc;
    // Several hits at once: when every duplicate of the round is a hit
    // (the population fills after the last one and the tabu rule does not
    // stop the run), take all their children out of the later lanes' sums
    // and decide once more, on trial.  If no lane -- hits included -- changes,
    // these are exactly the sequential outcome's hits and the batch is settled;
    // otherwise the sums go back and the hits are taken one per round.
    const int m = __popc(dupmask);
    if (m >= 2 && !failed_trial && (31 - __clz(dupmask) - first) - (m - 1) < need &&
        hits + m <= d.P) {
      if (K == 2 && !on_trial) {
        keep02 = o02;
        keep13 = o13;
        unsigned rest = dupmask;
        while (rest) {
          const int b = __ffs(rest) - 1;
          rest &= rest - 1;
          sub_overlap(b);
        }
        trial = true;
        continue;
      }
      hitmask |= dupmask;
      hits += m;
      const int free_lanes = (avail - first) - m;
      if (free_lanes >= need) {
        // the need-th accepted lane fills the population and ends the batch
        unsigned am = __ballot_sync(FULL, have && lane >= first && !dup);
        for (int t = 1; t < need; ++t) am &= am - 1;
        cut = __ffs(am);
        acc += need;
      } else {
        acc += free_lanes;
      }
      break;
    }
    if (first_dup - first >= need) {
      acc += need;
      cut = first + need;
      break;
    }
    acc += first_dup - first;
    if (first_dup >= avail) break;
    hitmask |= 1u << first_dup;
    if (++hits > d.P) {
      stopped = 1;
      cut = first_dup + 1;
      break;
    }
    if (first_dup + 1 >= avail) break;
    // the hit's child is not accepted: take it out of the later lanes' sums
    // and go on with the rest of the batch
    if (K == 2) sub_overlap(first_dup);
    first = first_dup + 1;
  }
  const unsigned accm = __ballot_sync(FULL, have && lane < cut && !((hitmask >> lane) & 1u));
  tm->dec[lane] = child_of(da, db, lane);
  if (lane == 0) {
    tm->accm = accm;
    tm->n0 = n;
  }
  *mine = key;
  const int ex = have && lane < cut ? nex : 0;
  if (__any_sync(FULL, ex != 0)) exact += (int)__reduce_add_sync(FULL, (unsigned)ex);
  attempts += cut;
  n += acc;
}

// Commits a batch's accepted lanes in lane order: warp 0 enters a lane's key
// (list, filter bit, chain) ...
__device__ __forceinline__ void commit_keys(const BatchBlk* blk, int j0, const EaDev& d,
                                            const KeyIndex& kx, unsigned long long* lkey,
                                            int32_t* lref, int E, const Team* tm, int nc,
                                            long long base, unsigned long long key, int lane) {
  const unsigned accm = tm->accm;
  if ((accm >> lane) & 1u) {
    const int at = tm->n0 + __popc(accm & ((1u << lane) - 1u)), dec = tm->dec[lane];
    const uint32_t fb = (uint32_t)(key >> 32) & (uint32_t)(kFilterBits - 1);
    kx.next[at - E] = (uint16_t)atomicExch(&kx.head[(uint32_t)key & kx.mask], (uint32_t)(at - E));
    atomicOr(&kx.bits[fb >> 5], 1u << (fb & 31));
    lkey[at - E] = key;
    lref[at - E] = (int32_t)((j0 + lane) * nc + dec);
    d.len[base + at] = blk->cL[dec][lane];
  }
  __syncwarp();
}

// ... and eight worker threads a lane its columns: archive row, penalty counts.
__device__ __forceinline__ void commit_cols(const EaDev& d, const RecLayout& l, const char* cur,
                                            const BatchBlk* blk, uint32_t* pen, const Team* tm,
                                            long long base, int RB, int wt) {
  const int a = wt >> 3, sub = wt & 7;
  const unsigned accm = tm->accm;
  if (!((accm >> a) & 1u)) return;
  const int at = tm->n0 + __popc(accm & ((1u << a) - 1u)), dec = tm->dec[a];
  const int L = blk->cL[dec][a];
  const uint16_t* child =
      reinterpret_cast<const uint16_t*>(cur + (size_t)a * RB + l.ccols) + (size_t)dec * d.S;
  uint16_t* dst = d.seq + (size_t)(base + at) * d.S;
  for (int c = sub; c < L; c += 8) {
    const uint16_t v = child[c];
    atomicAdd(&pen[v], 1u);
    dst[c] = v;
  }
}

// ---------------------------------------------------------------------------
// k_build: Steps 2-3 (or the acceptance part of Step 1).  The decisions are
// sequential (each tournament sees the penalty counts left by every earlier
// acceptance), so warp 0 makes them from shared memory only.  The attempt
// records and, in the fast path, the batch blocks (both written by the records'
// kernels) are streamed with TMA bulk copies into a ring of buffers completed
// through mbarriers: two chunks of kB records, or up to four batches of 32.
// Every wait is bounded: on expiry the kernel records stop reason 4, drains its
// own copies in flight and returns.  Accepted children go to the archive
// straight from the shared-memory records.
//
// Fast path (tournaments of at most 2, at most 256 columns; Step 1, without
// tournaments, alike), per batch of 32 attempts: warp 0 decides, meanwhile the
// eight worker warps wait for the next batch's copies and read its entrants'
// columns, one (entrant, half of its columns) a warp; then the workers count the
// accepted children's columns and sum the next batch's penalties, while warp 0
// enters the keys and prepares the next pairs.  Bound by the latency of that
// chain (2.2 us a batch: about half the decisions, a third the commit and the
// sums, the rest duplicates and barriers), so it is kept short: one copy of the
// decision, outcomes in two ballots, overlaps added three words at a time.  All
// warps taking part in every phase, and two buffers: 59 us instead of 50 a
// generation at 1,000 x 100, P = 600 (83 us with the overlaps counted here), 363
// instead of 283 us at 20,000 x 200, P = 4,096 (649 us with the committed keys
// scanned instead of chained, 891 us with both).
//
// Shared memory, general path: hkey[H] (u64) | href[H] | pen[C] | cLf[Lmax + 1]
// | 2 record buffers (128-byte aligned); hkey / href are the generation's hash
// set of committed children.  Fast path: lkey[P] (u64) | lref[P] | pen[C] |
// filter [kFilterWords] | chain heads [H / 4] | chain links [P] (u16) | record
// buffers (128-byte aligned) | block buffers; lkey / lref list the committed
// children in commit order, filter and chains find them by key.
// ---------------------------------------------------------------------------
template <bool INIT>
__global__ void __launch_bounds__(kBuildThreads, 1) k_build(EaDev d, int hmask, int kB, int depth) {
  extern __shared__ __align__(128) unsigned long long smem_u64[];
  if (*(volatile int32_t*)&d.ctl->stop) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = d.ctl->gen, n_top = d.ctl->n_top;
  if (tid == 0) d.ctl->spec_gen = g + 1;    // read by the next k_spec only
  const int H = hmask + 1, k = d.k, nc = INIT ? 1 : k * k, S = d.S;
  const RecLayout l = rec_layout(k, S, INIT);
  const int RB = d.rec_bytes;
  const bool fast = build_fast(d.k, d.WC);
  const int HL = fast ? d.P : H;         // entries of the key set or list
  unsigned long long* hkey = smem_u64;
  int32_t* href = reinterpret_cast<int32_t*>(hkey + HL);
  uint32_t* pen = reinterpret_cast<uint32_t*>(href + HL);
  float* cLf = reinterpret_cast<float*>(pen + d.C);
  // aligned by offsets from the shared base (integer round trips through
  // uintptr_t would lose the shared address space)
  char* const sbase = reinterpret_cast<char*>(smem_u64);
  KeyIndex kx;
  kx.bits = pen + d.C;
  kx.head = kx.bits + kFilterWords;
  kx.mask = (uint32_t)H / 4u - 1u;
  kx.next = reinterpret_cast<uint16_t*>(kx.head + H / 4);
  char* const fixed_end = fast ? reinterpret_cast<char*>(kx.next + d.P)
                               : reinterpret_cast<char*>(cLf + d.Lmax + 1);
  char* buf0 = sbase + ((fixed_end - sbase + 127) & ~(ptrdiff_t)127);
  // record buffer i at buf0 + i * kB * RB (computed, not looked up, so that the
  // compiler keeps the shared-memory address space of every record access);
  // the block buffers behind them
  const size_t buf_bytes = (size_t)kB * RB;
  BatchBlk* blk0 = reinterpret_cast<BatchBlk*>(buf0 + depth * buf_bytes);
  __shared__ __align__(8) unsigned long long bars[kMaxStages];
  __shared__ int s_n, s_done, s_E, s_fail;
  __shared__ uint8_t s_twin[kTwinSlots];  // lane ids by key (fast path twin pre-check)
  __shared__ Team s_team;                 // the fast path's batch protocol

  const int nchunks = (d.J + kB - 1) / kB;
  if (tid == 0) {
    for (int i = 0; i < depth; ++i) mbar_init(&bars[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  __syncthreads();
  // the chunks' copies are issued by one thread: in the fast path not one of
  // warp 0, which decides meanwhile
  const int issuer = fast ? 32 : 0;
  const bool tours = !INIT && k == 2;   // the fast path's batches hold tournaments
  int issued = 0, istage = 0;           // chunks whose copies it has issued, next buffer
  auto issue = [&]() {
    const int j0 = issued * kB, cnt = min(kB, d.J - j0);
    unsigned long long* bar = &bars[istage];
    if (fast) {
      // without tournaments nothing asks for overlaps
      const uint32_t skip = tours ? 0u : (uint32_t)sizeof(blk0->ov);
      mbar_expect(bar, (uint32_t)cnt * RB + (uint32_t)sizeof(BatchBlk) - skip);
      bulk_copy_to(buf0 + istage * buf_bytes, d.rec + (size_t)j0 * RB, (uint32_t)cnt * RB, bar);
      bulk_copy_to(reinterpret_cast<char*>(blk0 + istage) + skip,
                   reinterpret_cast<const char*>(d.blk + issued) + skip,
                   (uint32_t)sizeof(BatchBlk) - skip, bar);
    } else {
      bulk_load(buf0 + istage * buf_bytes, d.rec + (size_t)j0 * RB, (uint32_t)cnt * RB, bar);
    }
    ++issued;
    if (++istage == depth) istage = 0;
  };
  if (tid == issuer)
    while (issued < depth && issued < nchunks) issue();
  if (!fast)
    for (int i = tid; i < H; i += kBuildThreads) hkey[i] = 0ull;
  if (fast) {
#pragma unroll 8
    for (int i = tid; i < kFilterWords; i += kBuildThreads) kx.bits[i] = 0u;
    for (int i = tid; i < H / 4; i += kBuildThreads) kx.head[i] = kNoKey;
  }
  for (int i = tid; i < d.C; i += kBuildThreads) pen[i] = 0u;
  if (!fast)
    for (int i = tid; i <= d.Lmax; i += kBuildThreads) cLf[i] = d.c_over_L[i];
  const long long base = (long long)g * d.P;
  if (tid == 0) {
    int E = 0;
    if (!INIT) {
      E = (int)ceil(d.elite_frac * (double)n_top);
      if (E > d.P) E = d.P;
    }
    s_E = E;
    s_done = 0;
  }
  __syncthreads();
  const int E = s_E;
  // Step 2: elites copied in order, each column use counted; a thread a column,
  // so that the copies take two round trips however many elites there are.
  for (int i0 = tid; i0 < E * S; i0 += 4 * kBuildThreads) {
    int32_t src[4], L[4];
    uint16_t v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int at = i0 + i * kBuildThreads;
      src[i] = at < E * S ? d.list_ref[at / S] : -1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      L[i] = src[i] >= 0 ? d.len[src[i]] : 0;
      v[i] = src[i] >= 0 ? d.seq[(size_t)src[i] * S + (i0 + i * kBuildThreads) % S] : (uint16_t)0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = (i0 + i * kBuildThreads) / S, c = (i0 + i * kBuildThreads) % S;
      if (c >= L[i]) continue;
      d.seq[(size_t)(base + e) * S + c] = v[i];
      atomicAdd(&pen[v[i]], 1u);
      if (c == 0) d.len[base + e] = L[i];
    }
  }
  if (!fast) __syncthreads();           // (the fast path has its own)

  int n = E, hits = 0, stopped = 0;
  long long attempts = 0, exact = 0;
  int chunk = 0;
  if (fast) {
    const bool decider = warp == 0;
    const int wt = tid - 32;            // worker threads
    int stage = 0;
    uint32_t phase = 0u;
    unsigned long long key = 0ull;      // of the decider's lane
    BatchIn in;
    PenCols pc;
    // batch c, in the given buffer, once it has landed: the workers wait before
    // the barrier at which warp 0's wait is sure to end, and only they report
    auto ahead = [&](int c, int st, uint32_t ph) {
      if (!mbar_wait(&bars[st], ph)) {
        s_fail = 1;
        return;
      }
      if (!tours) return;
      const int avail = min(32, d.J - c * 32);
      if (decider) in = batch_in(blk0 + st, avail, lane);
      else
        pc = pen_cols(l, buf0 + st * buf_bytes, blk0 + st, avail, S, (warp - 1) & 3,
                      (warp - 1) >> 2, lane, RB);
    };
    if (nchunks > 0) ahead(0, 0, 0u);
    __syncthreads();
    while (chunk < nchunks && !s_fail) {
      const char* cur = buf0 + stage * buf_bytes;
      const BatchBlk* blk = blk0 + stage;
      const int j0 = chunk * 32, avail = min(32, d.J - j0);
      const bool wrap = stage + 1 == depth;
      const int nstage = wrap ? 0 : stage + 1;
      const uint32_t nphase = wrap ? phase ^ 1u : phase;
      if (tours && !decider) s_team.sx[(warp - 1) >> 2][(warp - 1) & 3][lane] = pen_sum(pc, pen);
      __syncthreads();
      if (decider) {
        if (tours)
          build_batch<2>(d, l, cur, blk, avail, in, hkey, href, kx, s_twin, &s_team, RB, lane,
                         n, hits, stopped, attempts, exact, &key);
        else
          build_batch<1>(d, l, cur, blk, avail, in, hkey, href, kx, s_twin, &s_team, RB, lane,
                         n, hits, stopped, attempts, exact, &key);
        if (INIT && stopped) stopped = 2;
        if (lane == 0) {
          s_n = n;
          s_done = (n >= d.P || stopped) ? 1 : 0;
        }
      } else {
        // the buffer of the batch before is free: refill it
        if (tid == issuer && chunk > 0 && issued < nchunks) issue();
        if (chunk + 1 < nchunks) ahead(chunk + 1, nstage, nphase);
      }
      __syncthreads();
      const bool over = s_done || s_fail;     // (a lost batch: the drain waits for it once more)
      if (decider) {
        commit_keys(blk, j0, d, kx, hkey, href, E, &s_team, nc, base, key, lane);
        if (!over && chunk + 1 < nchunks) ahead(chunk + 1, nstage, nphase);
      } else {
        commit_cols(d, l, cur, blk, pen, &s_team, base, RB, wt);
        asm volatile("bar.sync 1, %0;" ::"n"(kBuildWorkers) : "memory");
      }
      ++chunk;
      if (over) break;
      stage = nstage;
      phase = nphase;
    }
  }
  for (; !fast && chunk < nchunks; ++chunk) {
    char* cur = buf0 + (chunk & 1) * buf_bytes;
    if (warp == 0) {
      const bool ok = mbar_wait(&bars[chunk & 1], (uint32_t)((chunk >> 1) & 1));
      if (!ok) {
        stopped = 4;
      } else {
        for (int a = 0; a < kB && n < d.P; ++a) {
          const int j = chunk * kB + a;
          if (j >= d.J) {
            stopped = 3;
            break;
          }
          const char* rc = cur + (size_t)a * RB;
          ++attempts;
          int combo = 0;
          if (!INIT) {
            const int32_t* ent = reinterpret_cast<const int32_t*>(rc + l.ent);
            const int cr = *reinterpret_cast<const int32_t*>(rc + l.cross);
            const double* ef = reinterpret_cast<const double*>(rc + l.ef);
            const float* elnf = reinterpret_cast<const float*>(rc + l.elnf);
            const int32_t* eL = reinterpret_cast<const int32_t*>(rc + l.eL);
            const uint16_t* ecols = reinterpret_cast<const uint16_t*>(rc + l.ecols);
            const int nE = cr ? 2 * k : k;
            // penalty sums: lanes 8q .. 8q + 7 sum entrant 4 * pass + q
            uint32_t part0 = 0u, part1 = 0u;
#pragma unroll
            for (int pass = 0; pass < 2; ++pass) {
              if (pass * 4 < nE) {
                const int e = pass * 4 + (lane >> 3);
                uint32_t v = 0;
                if (e < nE) {
                  const int L = eL[e];
                  const uint16_t* cs = ecols + (size_t)e * S;
                  for (int c = lane & 7; c < L; c += 8) v += pen[cs[c]];
                }
                v += __shfl_xor_sync(0xffffffffu, v, 4);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                if (pass == 0) part0 = v;
                else part1 = v;
              }
            }
            // tournaments, computed alike on every lane from registers
            int pos0 = 0, pos1 = 0, nex = 0;
            for (int tour = 0; tour < (cr ? 2 : 1); ++tour) {
              Entrant best, x;
              int best_t = 0;
              for (int t = 0; t < k; ++t) {
                const int e = tour * k + t;
                x.lnf = elnf[e];
                x.S = (int32_t)__shfl_sync(0xffffffffu, e < 4 ? part0 : part1, (e & 3) * 8);
                x.L = eL[e];
                x.cl = cLf[x.L];
                x.idx = ent[(tour ? 4 : 0) + t];
                x.f = ef + e;
                if (t == 0) {
                  best = x;
                } else {
                  const int r = beats(x, best, d);
                  nex += r >> 1;
                  if (r & 1) {
                    best = x;
                    best_t = t;
                  }
                }
              }
              for (int t = 0; t < best_t; ++t)
                if (ent[(tour ? 4 : 0) + t] == best.idx) {
                  best_t = t;
                  break;
                }
              if (tour == 0) pos0 = best_t;
              else pos1 = best_t;
            }
            exact += nex;
            combo = pos0 * k + pos1;
          }
          const int L = reinterpret_cast<const int32_t*>(rc + l.cL)[combo];
          const unsigned long long key = reinterpret_cast<const unsigned long long*>(rc + l.chash)[combo];
          const uint16_t* child = reinterpret_cast<const uint16_t*>(rc + l.ccols) + (size_t)combo * S;
          int slot = 0;
          const bool dup = reinterpret_cast<const int32_t*>(rc + l.ctabu)[combo] != 0 ||
                           gen_duplicate<0>(d, l, hkey, href, hmask, nc, RB, key, child, L, lane, &slot);
          if (dup) {
            if (++hits > d.P) {
              stopped = INIT ? 2 : 1;
              break;
            }
            continue;
          }
          const int32_t rec_id = (int32_t)(j * nc + combo);
          uint16_t* dst = d.seq + (size_t)(base + n) * S;
          if (lane < L) {
            pen[child[lane]] += 1u;
            dst[lane] = child[lane];
          }
          if (lane + 32 < L) {
            pen[child[lane + 32]] += 1u;
            dst[lane + 32] = child[lane + 32];
          }
          if (lane == 0) {
            hkey[slot] = key;
            href[slot] = rec_id;
            d.len[base + n] = L;
          }
          __syncwarp();
          ++n;
        }
      }
      if (lane == 0) {
        s_n = n;
        s_done = (n >= d.P || stopped) ? 1 : 0;
        if (stopped == 4) s_fail = 1;
      }
    }
    __syncthreads();            // the consumed buffer may now be refilled
    if (s_done) {
      ++chunk;
      break;
    }
    if (tid == issuer && issued < nchunks) issue();
  }
  // every attempt consumed without filling the population: cannot happen
  // (2P + 1 attempts always suffice), reported as an internal error
  if (tid == 0 && s_n < d.P && !s_done && !s_fail) s_fail = 2;
  // drain: copies issued but not consumed must land before the CTA exits
  if (tid == issuer) {
    for (int c = chunk; c < issued; ++c)
      if (!mbar_wait(&bars[c % depth], (uint32_t)((c / depth) & 1))) s_fail = 1;
  }
  __syncthreads();
  if (tid == 0) {
    Ctl* ctl = d.ctl;
    ctl->last_hits = hits;
    // (atomics without a result: no round trip)
    atomicAdd(reinterpret_cast<unsigned long long*>(&ctl->hits_total), (unsigned long long)hits);
    atomicAdd(reinterpret_cast<unsigned long long*>(&ctl->attempts_total), (unsigned long long)attempts);
    atomicAdd(reinterpret_cast<unsigned long long*>(&ctl->exact_total), (unsigned long long)exact);
    ctl->n_elite = E;
    if (s_fail) stopped = s_fail == 2 ? 3 : 4;
    if (stopped) {
      ctl->stop_reason = stopped;
      __threadfence();
      ctl->stop = 1;
    }
  }
}

// ---------------------------------------------------------------------------
// k_tabu_insert: the generation's new (non-elite) individuals enter the tabu
// list.  Lookups happen in later launches only.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_tabu_insert(EaDev d) {
  if (*(volatile int32_t*)&d.ctl->stop) return;
  // the generation k_build just built: Step 5 of that generation may run
  // beside this kernel and advance ctl->gen, so it comes from spec_gen
  const int g = d.ctl->spec_gen - 1;
  const int slot = d.ctl->n_elite + (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (slot >= d.P) return;
  const long long e = (long long)g * d.P + slot;
  uint16_t x[kMaxLen];                              // the series, eight loads in flight
  const int L = d.len[e];
  copy_cols(x, d.seq + (size_t)e * d.S, L);
  const unsigned long long key = seq_hash(x, L);
  unsigned long long i = key & d.tmask;
  for (unsigned long long n = 0; n <= d.tmask; ++n) {
    if (atomicCAS(&d.tkey[i], 0ull, key) == 0ull) {
      d.tref[i] = (int32_t)e;
      return;
    }
    i = (i + 1) & d.tmask;
  }
  atomicExch(&d.ctl->stop_reason, 3);   // table full: cannot happen at load <= 1/2
  atomicExch(&d.ctl->stop, 1);
}

// ---------------------------------------------------------------------------
// k_rank: Step 5 (and the list part of Step 1).  One CTA of 1,024 threads.
// The population is sorted by decreasing fitness (ties: lower slot first),
// then visited in that order: an individual joins unless a listed record of
// higher or equal fitness overlaps it (|a & b| / min(|a|, |b|) > tau); when it
// joins it evicts the overlapping records of lower fitness and goes after all
// records of higher or equal fitness.  Finally the list keeps its T best.
//
// The visit stops early once T listed records have a fitness strictly above
// the current individual: records above it can only be evicted by fitter
// individuals (already visited), and everything visited from here on ranks
// below those T records, so it would be cut by the final trim -- and what it
// could still evict also ranks below them.  The result is the same list.
// ---------------------------------------------------------------------------
constexpr int kRankThreads = 1024;

// only_over: run only if k_rank_warp gave this generation up.
__global__ void __launch_bounds__(kRankThreads) k_rank(EaDev d, int Pp, int only_over) {
  extern __shared__ unsigned long long smem_u64[];
  if (*(volatile int32_t*)&d.ctl->stop) return;
  if (only_over && *(volatile int32_t*)&d.ctl->rank_over == 0) return;
  const int tid = threadIdx.x;
  const int g = d.ctl->gen;
  const long long base = (long long)g * d.P;
  const int cap = d.T + d.P;
  unsigned long long* skey = smem_u64;                             // [Pp]
  int32_t* sidx = reinterpret_cast<int32_t*>(skey + Pp);           // [Pp]
  double* lf = reinterpret_cast<double*>(sidx + Pp);               // [cap]
  double* lf2 = lf + cap;                                          // [cap]
  int32_t* lr = reinterpret_cast<int32_t*>(lf2 + cap);             // [cap]
  int32_t* lr2 = lr + cap;                                         // [cap]
  uint8_t* ov = reinterpret_cast<uint8_t*>(lr2 + cap);             // [cap]
  uint32_t* xbits = reinterpret_cast<uint32_t*>(ov + ((cap + 15) & ~15));   // [WC]
  __shared__ int s_warp[32];

  // sort keys: ascending (~bits(f), slot) == descending fitness, then slot
  for (int i = tid; i < Pp; i += kRankThreads) {
    if (i < d.P) {
      skey[i] = ~(unsigned long long)__double_as_longlong(d.fit[base + i]);
      sidx[i] = i;
    } else {
      skey[i] = ~0ull;
      sidx[i] = 0x7fffffff;
    }
  }
  __syncthreads();
  for (int size = 2; size <= Pp; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = tid; i < Pp; i += kRankThreads) {
        const int jx = i ^ stride;
        if (jx > i) {
          const bool up = (i & size) == 0;
          const unsigned long long ka = skey[i], kb = skey[jx];
          const int ia = sidx[i], ib = sidx[jx];
          const bool a_gt_b = ka > kb || (ka == kb && ia > ib);
          if (a_gt_b == up) {
            skey[i] = kb;
            skey[jx] = ka;
            sidx[i] = ib;
            sidx[jx] = ia;
          }
        }
      }
      __syncthreads();
    }
  }

  int n = d.ctl->n_top;
  for (int i = tid; i < n; i += kRankThreads) {
    lr[i] = d.list_ref[i];
    lf[i] = d.list_f[i];
  }
  __syncthreads();

  for (int oi = 0; oi < d.P; ++oi) {
    const int xi = sidx[oi];
    const long long xe = base + xi;
    const double xf = d.fit[xe];
    const int xL = d.len[xe];
    const uint16_t* xs = d.seq + (size_t)xe * d.S;
    int above = 0;
    for (int t0 = 0; t0 < n; t0 += kRankThreads) {
      const int t = t0 + tid;
      above += __syncthreads_count(t < n && lf[t] > xf);
    }
    if (above >= d.T) break;                                   // see the note above
    for (int w = tid; w < d.WC; w += kRankThreads) xbits[w] = 0u;
    __syncthreads();
    if (tid < xL) atomicOr(&xbits[xs[tid] >> 5], 1u << (xs[tid] & 31));
    __syncthreads();
    int blocked = 0;
    for (int t0 = 0; t0 < n; t0 += kRankThreads) {
      const int t = t0 + tid;
      bool hit = false;
      if (t < n) {
        const int32_t r = lr[t];
        const int L = d.len[r];
        const uint16_t* s = d.seq + (size_t)r * d.S;
        int inter = 0;
        for (int c = 0; c < L; ++c) inter += (xbits[s[c] >> 5] >> (s[c] & 31)) & 1u;
        const int mn = L < xL ? L : xL;
        const bool o = (double)inter > d.tau * (double)mn;
        ov[t] = o ? 1 : 0;
        hit = o && lf[t] >= xf;
      }
      blocked += __syncthreads_or(hit);
    }
    if (blocked) continue;
    // evict overlapping records of lower fitness (stable compaction into lr2/lf2)
    int m = 0;
    for (int t0 = 0; t0 < n; t0 += kRankThreads) {
      const int t = t0 + tid;
      const bool keep = t < n && !(ov[t] && lf[t] < xf);
      const unsigned bal = __ballot_sync(0xffffffffu, keep);
      const int lane = tid & 31, warp = tid >> 5;
      if (lane == 0) s_warp[warp] = __popc(bal);
      __syncthreads();
      if (warp == 0) {
        int v = s_warp[lane];
        for (int o = 1; o < 32; o <<= 1) {
          const int u = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += u;
        }
        s_warp[lane] = v;          // inclusive prefix over warps
      }
      __syncthreads();
      const int before = (warp ? s_warp[warp - 1] : 0) + __popc(bal & ((1u << lane) - 1u));
      if (keep) {
        lr2[m + before] = lr[t];
        lf2[m + before] = lf[t];
      }
      const int chunk_total = s_warp[31];
      __syncthreads();
      m += chunk_total;
    }
    // insert after every kept record of higher or equal fitness
    int pos = 0;
    for (int t0 = 0; t0 < m; t0 += kRankThreads) {
      const int t = t0 + tid;
      pos += __syncthreads_count(t < m && lf2[t] >= xf);
    }
    for (int t = tid; t < m; t += kRankThreads) {
      const int dst = t < pos ? t : t + 1;
      lr[dst] = lr2[t];
      lf[dst] = lf2[t];
    }
    if (tid == 0) {
      lr[pos] = (int32_t)xe;
      lf[pos] = xf;
    }
    n = m + 1;
    __syncthreads();
  }
  if (n > d.T) n = d.T;
  for (int i = tid; i < n; i += kRankThreads) {
    d.list_ref[i] = lr[i];
    d.list_f[i] = lf[i];
  }
  if (tid == 0) {
    Ctl* ctl = d.ctl;
    ctl->rank_over = 0;
    ctl->n_top = n;
    ctl->evals_total += d.P;
    if (g > 0) ctl->gens_done = g;
    ctl->gen = g + 1;
  }
}

// ---------------------------------------------------------------------------
// k_rank_warp: the same Step 5 for column sets of at most NW * 32 columns,
// arranged so that only what can change the list is ordered and looked at.
//
// Once the list is full, an individual less fit than its last record would end
// the visit (T listed records are fitter), so only those at least as fit -- some
// 30 of 600 in a running search -- are collected and put in order by counting
// (rank = how many come first).  If evictions then leave fewer than T records,
// or the list was not full, the rest is sorted whole (a bitonic network in
// registers) and the visit goes on.
//
// Whether an individual is blocked, or ends the visit, depends on the list
// alone, which changes only when one joins (1.4 times a generation).  So the
// sixteen warps test the next 32 individuals in visiting order against the list
// at once, and one warp takes them in: the first that is neither blocked nor the
// end joins, the later ones are tested against it, and only when it evicted
// records is the whole test repeated from there.  Overlaps are popcounts of bitset intersections, and
// |a & b| > tau * min(|a|, |b|) is an integer test against floor(tau * m) (the
// binary64 product, as in k_rank).  The list is kept sorted by decreasing
// fitness, so the records of fitness >= f(x) form a prefix of length ge; nothing
// in that prefix can move (evictions need lower fitness, and x goes after every
// record of higher or equal fitness), so an accepted x only rewrites the
// suffix: a stable compaction of the kept records, then a shift by one, then x
// at position ge.
//
// A list that outgrows `cap` records (only where T + P of them do not fit the
// shared memory) sets ctl->rank_over and leaves everything to k_rank.
// Latency-bound: 10 us a generation at P = 600 (28 us sorting everybody and
// visiting one by one), 101 us for the first generations of P = 4,096 (184 us in
// k_rank, whose list had no room in shared memory here).
//
// Shared memory: skey[Ns] (u64) | sidx[Ns] | lm[cap] (RankRec, 16 B) |
//                lbits[cap][NW] | thr[Lmax + 1]
// ---------------------------------------------------------------------------
struct RankRec {
  double f;
  int32_t r, L;
};

constexpr int kRankWarpThreads = 512;
constexpr int kRankWindow = 32;         // individuals tested at once (two a warp)

template <int NW>
__device__ __forceinline__ int overlap_bits(const uint32_t* a, const uint32_t (&xb)[NW]) {
  int inter = 0;
#pragma unroll
  for (int v = 0; v < NW / 4; ++v) {
    const uint4 w = reinterpret_cast<const uint4*>(a)[v];
    inter += __popc(w.x & xb[4 * v]) + __popc(w.y & xb[4 * v + 1]) +
             __popc(w.z & xb[4 * v + 2]) + __popc(w.w & xb[4 * v + 3]);
  }
  return inter;
}

// Bitonic sort of N = EPT * kRankWarpThreads (key, index) pairs into
// ascending order (key, then index), thread t holding elements EPT t .. EPT t
// + EPT - 1 in registers: compare-exchanges within a thread, with a partner
// thread of the warp by shuffles, and through shared memory (skey / sidx, N
// entries) only for partners in other warps.
template <int EPT>
__device__ __forceinline__ void sort_pairs(unsigned long long* skey, int32_t* sidx, int tid) {
  constexpr int N = EPT * kRankWarpThreads;
  unsigned long long k[EPT];
  int32_t x[EPT];
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    k[q] = skey[EPT * tid + q];
    x[q] = sidx[EPT * tid + q];
  }
  // element e of the block-direction `up` keeps the smaller of the pair when
  // it is the lower position of an ascending block (or the upper of a
  // descending one), the larger otherwise
  auto keep = [](unsigned long long& ka, int32_t& xa, unsigned long long kb, int32_t xb,
                 bool want_min) {
    const bool a_gt_b = ka > kb || (ka == kb && xa > xb);
    if (a_gt_b == want_min) {
      ka = kb;
      xa = xb;
    }
  };
  for (int size = 2; size <= N; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= 32 * EPT) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
          skey[EPT * tid + q] = k[q];
          sidx[EPT * tid + q] = x[q];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
          const int e = EPT * tid + q, p = e ^ stride;
          keep(k[q], x[q], skey[p], sidx[p], (e < p) == ((e & size) == 0));
        }
      } else if (stride >= EPT) {
        const int lane_x = stride / EPT;
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
          const int e = EPT * tid + q, p = e ^ stride;
          const unsigned long long kp = __shfl_xor_sync(0xffffffffu, k[q], lane_x);
          const int32_t xp = __shfl_xor_sync(0xffffffffu, x[q], lane_x);
          keep(k[q], x[q], kp, xp, (e < p) == ((e & size) == 0));
        }
      } else {
        // (the in-thread stride as a compile-time constant keeps k and x in
        // registers)
#pragma unroll
        for (int ls = EPT / 2; ls > 0; ls >>= 1) {
          if (ls != stride) continue;
#pragma unroll
          for (int q = 0; q < EPT; ++q) {
            if (q & ls) continue;
            const int e = EPT * tid + q;
            const bool up = (e & size) == 0;
            const unsigned long long ka = k[q], kb = k[q ^ ls];
            const int32_t xa = x[q], xb = x[q ^ ls];
            const bool a_gt_b = ka > kb || (ka == kb && xa > xb);
            if (a_gt_b == up) {
              k[q] = kb;
              x[q] = xb;
              k[q ^ ls] = ka;
              x[q ^ ls] = xa;
            }
          }
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    skey[EPT * tid + q] = k[q];
    sidx[EPT * tid + q] = x[q];
  }
  __syncthreads();
}

// One slot of the window: an individual in visiting order.
template <int NW>
struct RankSlot {
  __align__(16) uint32_t bits[NW];
  double f;
  int32_t pos, x, L;      // position in the visiting order, population index, length
  int32_t above, ge;      // listed records strictly fitter, and at least as fit
  int32_t block;          // one of the latter overlaps x
};

// By one warp: x joins the list of n records at place ge; returns the new n.
template <int NW>
__device__ __forceinline__ int rank_insert(RankRec* lm, uint32_t* lbits, const int32_t* thr, int n,
                                           const RankSlot<NW>& x, int ge, int32_t entry, int lane) {
  const unsigned FULL = 0xffffffffu;
  const int xL = x.L;
  uint32_t xb[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) xb[w] = x.bits[w];
  // suffix [ge, n): stable compaction of the kept records (not: overlapping
  // and less fit) ...
  int m = ge;
  for (int t0 = ge; t0 < n; t0 += 32) {
    const int t = t0 + lane;
    bool keep = false;
    RankRec rec{0.0, 0, 0};
    uint4 b[NW / 4];
    if (t < n) {
      rec = lm[t];
#pragma unroll
      for (int v = 0; v < NW / 4; ++v) b[v] = reinterpret_cast<const uint4*>(lbits + (size_t)t * NW)[v];
      keep = !(overlap_bits<NW>(lbits + (size_t)t * NW, xb) > thr[min(rec.L, xL)]);
    }
    const unsigned bal = __ballot_sync(FULL, keep);
    __syncwarp();
    if (keep) {
      const int dst = m + __popc(bal & ((1u << lane) - 1u));
      lm[dst] = rec;
#pragma unroll
      for (int v = 0; v < NW / 4; ++v) reinterpret_cast<uint4*>(lbits + (size_t)dst * NW)[v] = b[v];
    }
    __syncwarp();
    m += __popc(bal);
  }
  // ... shifted up by one (from the end), and x at ge
  for (int t0 = ((m - 1) & ~31); t0 >= ge - 31 && t0 >= 0; t0 -= 32) {
    const int t = t0 + lane;
    const bool mv = t >= ge && t < m;
    RankRec rec{0.0, 0, 0};
    uint4 b[NW / 4];
    if (mv) {
      rec = lm[t];
#pragma unroll
      for (int v = 0; v < NW / 4; ++v) b[v] = reinterpret_cast<const uint4*>(lbits + (size_t)t * NW)[v];
    }
    __syncwarp();
    if (mv) {
      lm[t + 1] = rec;
#pragma unroll
      for (int v = 0; v < NW / 4; ++v) reinterpret_cast<uint4*>(lbits + (size_t)(t + 1) * NW)[v] = b[v];
    }
    __syncwarp();
  }
  if (lane == 0) lm[ge] = RankRec{x.f, entry, xL};
#pragma unroll
  for (int w = 0; w < NW; ++w)
    if (lane == w) lbits[(size_t)ge * NW + w] = xb[w];
  __syncwarp();
  return m + 1;
}

template <int NW>
__global__ void __launch_bounds__(kRankWarpThreads) k_rank_warp(EaDev d, int Pp, int cap) {
  extern __shared__ __align__(128) unsigned long long smem_u64[];
  if (*(volatile int32_t*)&d.ctl->stop) return;
  const unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = d.ctl->gen;
  const long long base = (long long)g * d.P;
  const int P = d.P, T = d.T;
  const int Ns = Pp > kRankWarpThreads ? Pp : kRankWarpThreads;   // sorted entries
  unsigned long long* skey = smem_u64;
  int32_t* sidx = reinterpret_cast<int32_t*>(skey + Ns);
  RankRec* lm = reinterpret_cast<RankRec*>(sidx + Ns);            // (Ns * 12: 16-byte aligned)
  uint32_t* lbits = reinterpret_cast<uint32_t*>(lm + cap);
  int32_t* thr = reinterpret_cast<int32_t*>(lbits + (size_t)cap * NW);
  __shared__ RankSlot<NW> slots[kRankWindow];
  __shared__ int s_k, s_n, s_took, s_flag;
  __shared__ uint16_t s_cand[kRankWarpThreads], s_ord[kRankWarpThreads];

  if (tid == 0) s_k = 0;
  if (tid < kRankWindow) slots[tid].pos = -1;
  int n = d.ctl->n_top;
  const bool full = n >= T;
  // f >= the last record's <=> key <= theta (keys ascend as fitness descends)
  const unsigned long long theta =
      full ? ~(unsigned long long)__double_as_longlong(d.list_f[T - 1]) : 0ull;
  for (int t = tid; t < n; t += kRankWarpThreads) {
    const int32_t r = d.list_ref[t];
    const int L = d.len[r];
    lm[t] = RankRec{d.list_f[t], r, L};
    write_bits(lbits + (size_t)t * NW, NW, d.seq + (size_t)r * d.S, L);
  }
  for (int m = tid; m <= d.Lmax; m += kRankWarpThreads) thr[m] = (int32_t)floor(d.tau * (double)m);
  __syncthreads();
  for (int i = tid; i < Ns; i += kRankWarpThreads) {
    const unsigned long long key =
        i < P ? ~(unsigned long long)__double_as_longlong(d.fit[base + i]) : ~0ull;
    skey[i] = key;
    sidx[i] = i < P ? i : 0x7fffffff;
    if (full && i < P && key <= theta) {
      const int k = atomicAdd(&s_k, 1);
      if (k < kRankWarpThreads) s_cand[k] = (uint16_t)i;
    }
  }
  __syncthreads();
  auto sort_all = [&]() {
    switch (Ns / kRankWarpThreads) {     // Ns is a power of two >= 512
      case 1: sort_pairs<1>(skey, sidx, tid); break;
      case 2: sort_pairs<2>(skey, sidx, tid); break;
      case 4: sort_pairs<4>(skey, sidx, tid); break;
      default: sort_pairs<8>(skey, sidx, tid); break;
    }
  };
  int K = s_k;                            // individuals of this round of the visit
  bool part = full && K <= kRankWarpThreads;
  if (part) {
    if (tid < K) {
      const int i = s_cand[tid];
      const unsigned long long key = skey[i];
      int rank = 0;
      for (int j = 0; j < K; ++j) {
        const int o = s_cand[j];
        const unsigned long long ko = skey[o];
        rank += ko < key || (ko == key && o < i) ? 1 : 0;
      }
      s_ord[rank] = (uint16_t)i;
    }
    __syncthreads();
  } else {
    sort_all();
    K = P;
  }
  bool over = false;
  for (;;) {
    int pos = 0;
    bool ended = false;
    while (pos < K) {
      const int wn = min(kRankWindow, K - pos);
      for (int j = warp; j < wn; j += kRankWarpThreads / 32) {
        const int p = pos + j;
        RankSlot<NW>& s = slots[p & (kRankWindow - 1)];
        if (s.pos != p) {                 // warp-uniform: not tested before
          __syncwarp();
          const int xi = part ? s_ord[p] : sidx[p];
          const unsigned long long key = part ? skey[xi] : skey[p];
          const uint16_t* cs = d.seq + (size_t)(base + xi) * d.S;
          const uint32_t c0 = lane < d.S ? cs[lane] : 0u, c1 = lane + 32 < d.S ? cs[lane + 32] : 0u;
          const int L = d.len[base + xi];
          const uint32_t b0 = lane < L ? 1u << (c0 & 31) : 0u, b1 = lane + 32 < L ? 1u << (c1 & 31) : 0u;
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            const uint32_t word = __reduce_or_sync(FULL, ((c0 >> 5) == (uint32_t)w ? b0 : 0u) |
                                                             ((c1 >> 5) == (uint32_t)w ? b1 : 0u));
            if (lane == w) s.bits[w] = word;
          }
          if (lane == 0) {
            s.f = __longlong_as_double((long long)~key);
            s.pos = p;
            s.x = xi;
            s.L = L;
          }
          __syncwarp();
        }
        const double xf = s.f;
        const int xL = s.L;
        uint32_t xb[NW];
#pragma unroll
        for (int w = 0; w < NW; ++w) xb[w] = s.bits[w];
        // records strictly fitter (above), of higher or equal fitness (ge, a
        // prefix), and whether one of the latter overlaps x (blocks it)
        int above = 0, ge = 0;
        bool block = false;
        for (int t0 = 0; t0 < n; t0 += 32) {
          const int t = t0 + lane;
          bool is_ge = false, is_above = false;
          if (t < n) {
            const RankRec rec = lm[t];
            is_above = rec.f > xf;
            is_ge = rec.f >= xf;
            if (is_ge)
              block = block || overlap_bits<NW>(lbits + (size_t)t * NW, xb) > thr[min(rec.L, xL)];
          }
          above += __popc(__ballot_sync(FULL, is_above));
          const unsigned gb = __ballot_sync(FULL, is_ge);
          ge += __popc(gb);
          if (gb != FULL) break;                  // the prefix ends in this chunk
        }
        const bool any = __any_sync(FULL, block);
        if (lane == 0) {
          s.above = above;
          s.ge = ge;
          s.block = any ? 1 : 0;
        }
      }
      __syncthreads();
      if (warp == 0) {
        // lane i has the i-th of the window; the first that is not blocked joins
        // (or ends the visit: see k_rank).  A joining x that evicts nobody adds
        // one record, at least as fit as everyone after it: what that changes
        // for the others is settled here.  Evictions can unblock: test again.
        const RankSlot<NW>& s = slots[(pos + lane) & (kRankWindow - 1)];
        const bool in = lane < wn;
        const double xf = in ? s.f : 0.0;
        const int xL = in ? s.L : 0;
        int above = in ? s.above : 0, ge = in ? s.ge : 0, took = wn, flag = 0, from = 0;
        bool block = in && s.block != 0;
        for (;;) {
          const bool end = above >= T;
          const unsigned hit = __ballot_sync(FULL, in && lane >= from && (end || !block));
          if (!hit) break;
          const int j = __ffs(hit) - 1;
          if (__shfl_sync(FULL, end ? 1 : 0, j)) flag = 1;
          else if (n >= cap) flag = 2;
          if (flag) break;
          const RankSlot<NW>& y = slots[(pos + j) & (kRankWindow - 1)];
          const int m = rank_insert<NW>(lm, lbits, thr, n, y, __shfl_sync(FULL, ge, j),
                                        (int32_t)(base + y.x), lane);
          const bool evicted = m != n + 1;
          n = m;
          if (evicted) {
            took = j + 1;
            break;
          }
          from = j + 1;
          if (in && lane > j) {
            uint32_t yb[NW];
#pragma unroll
            for (int w = 0; w < NW; ++w) yb[w] = y.bits[w];
            above += y.f > xf ? 1 : 0;
            ge += 1;
            block = block || overlap_bits<NW>(s.bits, yb) > thr[min(y.L, xL)];
          }
        }
        if (lane == 0) {
          s_n = n;
          s_took = took;
          s_flag = flag;
        }
      }
      __syncthreads();
      n = s_n;
      pos += s_took;
      ended = s_flag == 1;
      over = s_flag == 2;
      if (ended || over) break;                   // block-uniform
    }
    if (ended || over || !part || n >= T) break;
    // fewer than T records are left: the rest of the population, sorted
    part = false;
    __syncthreads();
    for (int i = tid; i < P; i += kRankWarpThreads)
      if (skey[i] <= theta) {
        skey[i] = ~0ull;
        sidx[i] = 0x7fffffff;
      }
    if (tid < kRankWindow) slots[tid].pos = -1;
    K = P - K;
    __syncthreads();
    sort_all();
  }
  if (over) {                                     // k_rank starts over from the stored list
    if (tid == 0) d.ctl->rank_over = 1;
    return;
  }
  if (n > T) n = T;
  for (int i = tid; i < n; i += kRankWarpThreads) {
    const RankRec rec = lm[i];
    d.list_ref[i] = rec.r;
    d.list_f[i] = rec.f;
  }
  if (tid == 0) {
    Ctl* ctl = d.ctl;
    ctl->n_top = n;
    ctl->evals_total += d.P;
    if (g > 0) ctl->gens_done = g;
    ctl->gen = g + 1;
  }
}

// Shared bytes of k_rank_warp<NW> for `cap` list records besides those per record.
static size_t rank_warp_fixed(int Pp, int Lmax) {
  return (size_t)std::max(Pp, kRankWarpThreads) * 12 + (size_t)(Lmax + 1) * 4 + 16;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct EaState {
  ebic_params_t p{};
  int32_t S = 0, J = 0, ncombo = 0, WC = 0, Pp = 0, hmask = 0, kB = 64, depth = 2;
  long long entries = 0;
  DevBuf seq, len, inc, dec, fit, lnf;
  DevBuf counters;               // of split series, for the run's evaluations alone
  DevBuf tkey, tref;
  DevBuf rec, blk;
  int32_t rec_bytes = 0;
  DevBuf list_ref, list_f;
  DevBuf pow_tab, pow_off, c_over_L;
  DevBuf ctl, gather;
  HostBuf h_ctl, h_gather;
  size_t smem_build = 0, smem_rank = 0;
  size_t smem_rank_all = 0;      // k_rank
  int32_t rank_nw = 0;           // k_rank_warp<rank_nw> (0: k_rank)
  int32_t rank_cap = 0;          // its list records
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  EaDev dev{};
  ArchivePop apop{};
  EvalArgs eargs{};
  ebic_eval_tuning_t tuning{};   // evaluation shape chosen at Step 1
  bool initialised = false;
  // offspring screening
  ebic_surrogate_ctx* sur = nullptr;   // attached surrogate (EBIC_SCREEN_SURROGATE)
  std::shared_ptr<const bool> sur_alive;
  bool lost_scores = false;            // as of the last read_ctl
  long long var_rows = 0;
  DevBuf var_seq, var_len, var_score, act;
  int32_t launches_per_gen = 5;
  cudaGraph_t multi_graph = nullptr;   // kGraphGens generations
  cudaGraphExec_t multi = nullptr;
  bool multi_tried = false;
  long long stepped = 0;               // generations ebic_run_step has replayed
  cudaStream_t side = nullptr, side2 = nullptr;   // other branches of the generation graph
  cudaEvent_t fork_ev[4] = {nullptr, nullptr, nullptr, nullptr};
  // In-graph timing of k_build: two event-record nodes bracket it in the
  // graph; each replay points them at the next pair of a ring of events.
  int32_t tslots = 0;
  std::vector<cudaEvent_t> tev;        // [2 * tslots]: begin, end per slot
  cudaGraphNode_t tnode[2] = {nullptr, nullptr};
  long long tlaunched = 0, tharvested = 0, tcount = 0;
  double tsum_ms = 0.0;

  void release() {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (multi) cudaGraphExecDestroy(multi);
    if (multi_graph) cudaGraphDestroy(multi_graph);
    exec = multi = nullptr;
    graph = multi_graph = nullptr;
    for (cudaEvent_t& e : fork_ev) {
      if (e) cudaEventDestroy(e);
      e = nullptr;
    }
    for (cudaEvent_t& e : tev)
      if (e) cudaEventDestroy(e);
    tev.clear();
    tslots = 0;
    if (side) cudaStreamDestroy(side);
    if (side2) cudaStreamDestroy(side2);
    side = side2 = nullptr;
    for (DevBuf* b : {&seq, &len, &inc, &dec, &fit, &lnf, &counters, &tkey, &tref, &rec, &blk,
                      &list_ref, &list_f, &pow_tab, &pow_off, &c_over_L, &ctl, &gather, &var_seq,
                      &var_len, &var_score, &act})
      b->release();
    sur = nullptr;
    h_ctl.release();
    h_gather.release();
    initialised = false;
  }
};

void ea_release(ebic_ctx* h) {
  if (h->ea) {
    h->ea->release();
    delete h->ea;
    h->ea = nullptr;
  }
}

static ebic_status validate(const ebic_ctx* h, const ebic_params_t* p) {
  if (!p) return fail(EBIC_ERR_ARG, "null params");
  if (h->C > 8192) return fail(EBIC_ERR_ARG, "the EA supports at most 8192 columns");
  if (p->pop_size < 2 || p->pop_size > 4096)
    return fail(EBIC_ERR_ARG, "pop_size %d outside [2, 4096]", p->pop_size);
  if (p->len_min < 1 || p->len_max < p->len_min || p->len_max > h->C ||
      p->len_max > EBIC_MAX_EA_LEN)
    return fail(EBIC_ERR_ARG, "lengths [%d, %d] invalid for %d columns (max %d)", p->len_min,
                p->len_max, h->C, EBIC_MAX_EA_LEN);
  if (p->iterations < 0) return fail(EBIC_ERR_ARG, "negative iterations");
  if (p->toprank_size < 1 || p->toprank_size > 4096)
    return fail(EBIC_ERR_ARG, "toprank_size %d outside [1, 4096]", p->toprank_size);
  if (p->tournament_k < 1 || p->tournament_k > EBIC_MAX_TOURNAMENT)
    return fail(EBIC_ERR_ARG, "tournament_k %d outside [1, %d]", p->tournament_k,
                EBIC_MAX_TOURNAMENT);
  if (p->support_mode != EBIC_SUPPORT_INC && p->support_mode != EBIC_SUPPORT_INC_PLUS_DEC)
    return fail(EBIC_ERR_ARG, "bad support mode");
  if (!(p->overlap_tau >= 0.0 && p->overlap_tau <= 1.0)) return fail(EBIC_ERR_ARG, "tau");
  if (!(p->elite_frac >= 0.0 && p->elite_frac <= 1.0)) return fail(EBIC_ERR_ARG, "elite_frac");
  if (!(p->penalty_base >= 1.0 && p->penalty_base < 1e6)) return fail(EBIC_ERR_ARG, "base");
  if (!(p->p_crossover >= 0.0 && p->p_crossover <= 1.0)) return fail(EBIC_ERR_ARG, "p_crossover");
  return EBIC_OK;
}

// Whether k_spec_pairs builds the records, in the two launches below.
static bool pairs_form(const EaDev& d) { return d.V <= 1 && d.k == 2 && bit_words(d.WC) != 0; }

static unsigned pairs_grid(const EaState* st) {
  return (unsigned)(((long long)st->J * st->ncombo + 127) / 128);
}

static void launch_pairs(const EaState* st, cudaStream_t s) {
  if (bit_words(st->dev.WC) == 4) k_spec_pairs<4><<<pairs_grid(st), 128, 0, s>>>(st->dev);
  else k_spec_pairs<8><<<pairs_grid(st), 128, 0, s>>>(st->dev);
}

static void launch_settle(const EaState* st, cudaStream_t s) {
  k_spec_settle<<<pairs_grid(st), 128, 0, s>>>(st->dev);
}

// Attempt records of one Steps 2-5 generation: k_spec, or (screening) the
// candidates, their scores and the pick.  Returns the launch count in *n.
// With `mid` (profiling, screening only), events mid[0] and mid[1] are
// recorded after the candidates and after their scores.
static ebic_status launch_records(EaState* st, cudaStream_t s, int* n,
                                  cudaEvent_t* mid = nullptr) {
  const EaDev& d = st->dev;
  const long long jc = (long long)st->J * st->ncombo;
  if (d.V <= 1) {
    const unsigned grid = (unsigned)((jc + 127) / 128);
    if (pairs_form(d)) {
      launch_pairs(st, s);
      launch_settle(st, s);
      *n = 2;
    } else {
      k_spec<false, false><<<grid, 128, 0, s>>>(d);
      *n = 1;
    }
    return EBIC_OK;
  }
  const long long rows = jc * d.V;
  k_spec<false, true><<<(unsigned)((rows + 127) / 128), 128, 0, s>>>(d);
  if (mid) cudaEventRecord(mid[0], s);
  int ns = 1;
  if (d.screen == EBIC_SCREEN_SURROGATE) {
    EBIC_TRY(sur_forward_scores(st->sur, d.var_seq, d.var_len, d.S, (int32_t)rows, st->act.ptr,
                                d.var_score, s, &ns));
  } else {
    k_pseudo_score<<<(unsigned)((rows + 255) / 256), 256, 0, s>>>(d);
  }
  if (mid) cudaEventRecord(mid[1], s);
  k_pick<<<(unsigned)((jc + 127) / 128), 128, 0, s>>>(d);
  *n = 2 + ns;
  EBIC_CUDA_TRY(cudaGetLastError());
  return EBIC_OK;
}

// One launch, or two where k_rank stands by for a list that outgrows
// k_rank_warp's room.
static int launch_rank(const EaState* st, cudaStream_t s) {
  if (st->rank_nw == 4)
    k_rank_warp<4><<<1, kRankWarpThreads, st->smem_rank, s>>>(st->dev, st->Pp, st->rank_cap);
  else if (st->rank_nw == 8)
    k_rank_warp<8><<<1, kRankWarpThreads, st->smem_rank, s>>>(st->dev, st->Pp, st->rank_cap);
  const bool all = st->rank_nw == 0, stand_by = !all && st->rank_cap < st->p.toprank_size + st->p.pop_size;
  if (all || stand_by)
    k_rank<<<1, kRankThreads, st->smem_rank_all, s>>>(st->dev, st->Pp, stand_by ? 1 : 0);
  return stand_by ? 2 : 1;
}

// One generation g as captured for replay.  Step 3 first; then tabu
// insertion beside the evaluation; Step 5 of g as soon as the evaluation is
// done, beside the attempt records of g + 1 (which need g's fitness and tabu
// list, not its top-rank list, which only the next Step 2 reads; tabu
// insertion and the records take the generation from spec_gen, not from
// the counter Step 5 advances):
//
//   k_build(g) -+- eval(g) -+- k_rank(g) ---------------+- (next replay)
//               |           +---------+                 |
//               +- k_tabu_insert(g) --+- records(g + 1) -+
//               +- k_spec_pairs(g + 1) -+
//
// Where k_spec_pairs builds the records, it needs neither (a third branch), and
// only k_spec_settle comes after the fitness and the tabu list.
//
// The records of generation 1 are built at the end of ebic_run_init.
static ebic_status launch_generation(ebic_ctx* h, EaState* st, cudaStream_t s) {
  const EaDev& d = st->dev;
  cudaStream_t s2 = st->side;
  if (st->tslots) EBIC_CUDA_TRY(cudaEventRecordWithFlags(st->tev[0], s, cudaEventRecordExternal));
  k_build<false><<<1, kBuildThreads, st->smem_build, s>>>(d, st->hmask, st->kB, st->depth);
  if (st->tslots) EBIC_CUDA_TRY(cudaEventRecordWithFlags(st->tev[1], s, cudaEventRecordExternal));
  EBIC_CUDA_TRY(cudaEventRecord(st->fork_ev[0], s));
  EBIC_CUDA_TRY(cudaStreamWaitEvent(s2, st->fork_ev[0], 0));
  k_tabu_insert<<<(unsigned)((st->p.pop_size + 255) / 256), 256, 0, s2>>>(d);
  EBIC_CUDA_TRY(cudaGetLastError());
  const bool pairs = pairs_form(d);
  if (pairs) {
    EBIC_CUDA_TRY(cudaStreamWaitEvent(st->side2, st->fork_ev[0], 0));
    launch_pairs(st, st->side2);
    EBIC_CUDA_TRY(cudaGetLastError());
    EBIC_CUDA_TRY(cudaEventRecord(st->fork_ev[2], st->side2));
    EBIC_CUDA_TRY(cudaStreamWaitEvent(s2, st->fork_ev[2], 0));
  }
  EBIC_TRY(eval_archive(h, st->apop, st->eargs, s));
  // Step 5 right after the evaluation (it needs the fitness, not the tabu
  // list); the next attempt records after both
  EBIC_CUDA_TRY(cudaEventRecord(st->fork_ev[1], s));
  EBIC_CUDA_TRY(cudaStreamWaitEvent(s2, st->fork_ev[1], 0));
  const int nrank = launch_rank(st, s);
  EBIC_CUDA_TRY(cudaGetLastError());
  int nrec = 2;
  if (pairs) launch_settle(st, s2);
  else EBIC_TRY(launch_records(st, s2, &nrec));
  EBIC_CUDA_TRY(cudaGetLastError());
  st->launches_per_gen = nrec + nrank + 3;
  EBIC_CUDA_TRY(cudaEventRecord(st->fork_ev[3], s2));
  EBIC_CUDA_TRY(cudaStreamWaitEvent(s, st->fork_ev[3], 0));
  return EBIC_OK;
}

static ebic_status read_ctl(EaState* st, cudaStream_t s, Ctl* out) {
  EBIC_CUDA_TRY(cudaMemcpyAsync(st->h_ctl.ptr, st->ctl.ptr, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
  const bool scored = st->sur && *st->sur_alive;
  int* lost = reinterpret_cast<int*>(st->h_ctl.as<char>() + sizeof(Ctl));
  if (scored)
    EBIC_CUDA_TRY(cudaMemcpyAsync(lost, sur_lost_scores(st->sur), sizeof(int), cudaMemcpyDeviceToHost, s));
  EBIC_CUDA_TRY(cudaStreamSynchronize(s));
  std::memcpy(out, st->h_ctl.ptr, sizeof(Ctl));
  st->lost_scores = scored && *lost != 0;
  return EBIC_OK;
}

static void fill_stats(const Ctl& c, ebic_stats_t* stats) {
  if (!stats) return;
  stats->generations_done = c.gens_done;
  stats->stop_reason = c.stop_reason;
  stats->tabu_hits_total = c.hits_total;
  stats->attempts_total = c.attempts_total;
  stats->evaluations_total = c.evals_total;
  stats->last_gen_hits = c.last_hits;
  stats->toprank_n = c.n_top;
  stats->exact_tournaments = c.exact_total;
}

// Opts a kernel in to all the dynamic shared memory the device allows it.  The
// setting belongs to the function, not to a run: were it the run's own size, a
// smaller run started later on another handle would take it away again.
template <class K>
static ebic_status allow_smem(const ebic_ctx* h, K* kern) {
  int most = 0;
  cudaFuncAttributes fa{};
  EBIC_CUDA_TRY(cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device));
  EBIC_CUDA_TRY(cudaFuncGetAttributes(&fa, kern));
  EBIC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     most - (int)fa.sharedSizeBytes));
  return EBIC_OK;
}

static ebic_status run_init(ebic_ctx* h, const ebic_params_t* p) {
  EBIC_TRY(validate(h, p));
  ea_release(h);
  EaState* st = new EaState();
  h->ea = st;
  st->p = *p;
  const int32_t P = p->pop_size, k = p->tournament_k, T = p->toprank_size;
  st->S = p->len_max;
  st->J = 2 * P + 1;
  st->ncombo = k * k;
  st->WC = (h->C + 31) / 32;
  st->Pp = 1;
  while (st->Pp < P) st->Pp <<= 1;
  int H = 1;
  while (H < 2 * P) H <<= 1;
  st->hmask = H - 1;
  st->entries = (long long)(p->iterations + 1) * P;
  const cudaStream_t s = h->stream;
  const size_t E = (size_t)st->entries;
  EBIC_TRY(st->seq.reserve(E * st->S * sizeof(uint16_t)));
  EBIC_TRY(st->len.reserve(E * sizeof(int32_t)));
  EBIC_TRY(st->inc.reserve(E * sizeof(uint32_t)));
  EBIC_TRY(st->dec.reserve(E * sizeof(uint32_t)));
  EBIC_TRY(st->fit.reserve(E * sizeof(double)));
  EBIC_TRY(st->lnf.reserve(E * sizeof(float)));
  EBIC_TRY(st->counters.reserve_zeroed((size_t)P * 2 * sizeof(unsigned long long), s));
  unsigned long long tcap = 1;
  while (tcap < 2ull * E) tcap <<= 1;
  EBIC_TRY(st->tkey.reserve(tcap * sizeof(unsigned long long)));
  EBIC_TRY(st->tref.reserve(tcap * sizeof(int32_t)));
  EBIC_CUDA_TRY(cudaMemsetAsync(st->tkey.ptr, 0, tcap * sizeof(unsigned long long), s));
  EBIC_CUDA_TRY(cudaMemsetAsync(st->dec.ptr, 0, E * sizeof(uint32_t), s));
  // attempt records: sized for the larger (Steps 2-5) layout
  st->rec_bytes = rec_layout(k, st->S, false).bytes;
  EBIC_TRY(st->rec.reserve((size_t)st->J * st->rec_bytes));
  const bool fast = build_fast(k, st->WC);
  if (fast) EBIC_TRY(st->blk.reserve((size_t)((st->J + 31) / 32) * sizeof(BatchBlk)));
  EBIC_TRY(st->list_ref.reserve((size_t)(T + P) * sizeof(int32_t)));
  EBIC_TRY(st->list_f.reserve((size_t)(T + P) * sizeof(double)));
  EBIC_TRY(st->ctl.reserve(sizeof(Ctl)));
  EBIC_TRY(st->h_ctl.reserve(sizeof(Ctl) + sizeof(int)));
  EBIC_CUDA_TRY(cudaMemsetAsync(st->ctl.ptr, 0, sizeof(Ctl), s));

  // Crowding-penalty table base^(S / L) (host C library pow), L in
  // [len_min, len_max], S in [0, L * P]; and log(base) / L as float.
  std::vector<long long> off((size_t)p->len_max + 1, 0);
  long long total = 0;
  for (int L = p->len_min; L <= p->len_max; ++L) {
    off[L] = total;
    total += (long long)L * P + 1;
  }
  std::vector<double> tab((size_t)total);
  fill_table(total, 4096, [&](long long lo, long long hi) {
    int L = p->len_min;
    while (L < p->len_max && off[L + 1] <= lo) ++L;
    for (long long i = lo; i < hi; ++i) {
      if (L < p->len_max && off[L + 1] <= i) ++L;
      tab[(size_t)i] = std::pow(p->penalty_base, (double)(i - off[L]) / (double)L);
    }
  });
  std::vector<float> cl((size_t)p->len_max + 1, 0.f);
  for (int L = 1; L <= p->len_max; ++L) cl[L] = (float)(std::log(p->penalty_base) / (double)L);
  EBIC_TRY(st->pow_tab.reserve(tab.size() * sizeof(double)));
  EBIC_TRY(st->pow_off.reserve(off.size() * sizeof(long long)));
  EBIC_TRY(st->c_over_L.reserve(cl.size() * sizeof(float)));
  EBIC_CUDA_TRY(cudaMemcpyAsync(st->pow_tab.ptr, tab.data(), tab.size() * sizeof(double),
                                cudaMemcpyHostToDevice, s));
  EBIC_CUDA_TRY(cudaMemcpyAsync(st->pow_off.ptr, off.data(), off.size() * sizeof(long long),
                                cudaMemcpyHostToDevice, s));
  EBIC_CUDA_TRY(cudaMemcpyAsync(st->c_over_L.ptr, cl.data(), cl.size() * sizeof(float),
                                cudaMemcpyHostToDevice, s));

  EaDev& d = st->dev;
  d.P = P;
  d.C = h->C;
  d.S = st->S;
  d.Lmin = p->len_min;
  d.Lmax = p->len_max;
  d.k = k;
  d.T = T;
  d.mode = p->support_mode;
  d.J = st->J;
  d.ncombo = st->ncombo;
  d.WC = st->WC;
  d.tau = p->overlap_tau;
  d.elite_frac = p->elite_frac;
  d.pc = p->p_crossover;
  d.seed = p->seed;
  d.seq = st->seq.as<uint16_t>();
  d.len = st->len.as<int32_t>();
  d.fit = st->fit.as<double>();
  d.lnf = st->lnf.as<float>();
  d.tkey = st->tkey.as<unsigned long long>();
  d.tref = st->tref.as<int32_t>();
  d.tmask = tcap - 1;
  d.rec = st->rec.as<char>();
  d.rec_bytes = st->rec_bytes;
  d.blk = st->blk.as<BatchBlk>();
  d.list_ref = st->list_ref.as<int32_t>();
  d.list_f = st->list_f.as<double>();
  d.pow_tab = st->pow_tab.as<double>();
  d.pow_off = st->pow_off.as<long long>();
  d.c_over_L = st->c_over_L.as<float>();
  d.ctl = st->ctl.as<Ctl>();

  // Offspring screening: candidate buffers (zeroed, so that a pass over rows
  // no k_spec has written yet reads empty series), scores, activations.
  d.V = 1;
  d.screen = EBIC_SCREEN_OFF;
  if (h->screen_mode != EBIC_SCREEN_OFF && h->screen_v > 1) {
    const int32_t V = h->screen_v;
    if (h->screen_mode == EBIC_SCREEN_SURROGATE && !h->screen_sur)
      return fail(EBIC_ERR_STATE, "surrogate screening without a surrogate");
    const long long rows = (long long)st->J * st->ncombo * V;
    if (rows > (1ll << 22))
      return fail(EBIC_ERR_ARG, "screening needs %lld candidate rows per generation (max %lld)",
                  rows, 1ll << 22);
    EBIC_TRY(st->var_seq.reserve_zeroed((size_t)rows * st->S * sizeof(uint16_t), s));
    EBIC_TRY(st->var_len.reserve_zeroed((size_t)rows * sizeof(int32_t), s));
    EBIC_TRY(st->var_score.reserve((size_t)rows * sizeof(float)));
    if (h->screen_mode == EBIC_SCREEN_SURROGATE) {
      st->sur = h->screen_sur;
      st->sur_alive = sur_alive(st->sur);
    }
    st->var_rows = rows;
    d.V = V;
    d.screen = h->screen_mode;
    d.var_seq = st->var_seq.as<uint16_t>();
    d.var_len = st->var_len.as<int32_t>();
    d.var_score = st->var_score.as<float>();
  }

  st->apop.seq = d.seq;
  st->apop.len = d.len;
  st->apop.stride = st->S;
  st->apop.P = P;
  st->apop.gen = &d.ctl->gen;
  st->apop.stop = &d.ctl->stop;
  EvalArgs& a = st->eargs;
  a.P = P;
  a.sigma = p->sigma;
  a.mode = p->support_mode;
  a.want_dec = p->support_mode == EBIC_SUPPORT_INC_PLUS_DEC;
  a.inc = st->inc.as<uint32_t>();
  a.dec = a.want_dec ? st->dec.as<uint32_t>() : nullptr;
  a.fit = d.fit;
  a.lnf = d.lnf;
  // the captured generations keep this pointer: never the handle's counters,
  // which other evaluations outgrow
  a.counters = st->counters.as<uint32_t>();

  // build: the fixed parts of k_build's two layouts, then the buffers: two of
  // kB records, or (fast path) as many of a batch's 32 records and its block as
  // fit, two at least (they fit at the largest sizes: 4,096 individuals, 256
  // columns, length 64: 194 KB).
  const size_t set_bytes = sizeof(unsigned long long) + sizeof(int32_t);
  const size_t fixed_gen = (size_t)H * set_bytes + (size_t)h->C * sizeof(uint32_t) +
                           (size_t)(p->len_max + 2) * sizeof(float) + 128;
  const size_t fixed_fast = (size_t)P * set_bytes + (size_t)h->C * sizeof(uint32_t) +
                            (size_t)kFilterWords * sizeof(uint32_t) +
                            (size_t)H / 4 * sizeof(uint32_t) + (size_t)P * sizeof(uint16_t) + 128;
  if (fast) {
    const size_t stage = sizeof(BatchBlk) + 32 * (size_t)st->rec_bytes;
    st->kB = 32;
    st->depth = (int)std::clamp<size_t>((216 * 1024 - fixed_fast) / stage, 2, kMaxStages);
    st->smem_build = fixed_fast + st->depth * stage;
  } else {
    st->kB = 64;
    st->depth = 2;
    while (st->kB > 2 && fixed_gen + 2 * (size_t)st->kB * st->rec_bytes > 200 * 1024) st->kB >>= 1;
    st->smem_build = fixed_gen + 2 * (size_t)st->kB * st->rec_bytes;
  }
  const size_t cap = (size_t)T + P;
  st->smem_rank_all = (size_t)st->Pp * (sizeof(unsigned long long) + sizeof(int32_t)) +
                      cap * (2 * sizeof(double) + 2 * sizeof(int32_t)) + ((cap + 15) & ~(size_t)15) +
                      (size_t)st->WC * sizeof(uint32_t);
  // Step 5 from shared bitsets when the columns and sizes allow: room for
  // every record the list can hold, or for at least T and 256 joining ones
  st->rank_nw = 0;
  const int rnw = bit_words(st->WC);
  if (rnw && st->Pp <= 8 * kRankWarpThreads) {    // the register sort holds 8 per thread
    const size_t fixed_rank = rank_warp_fixed(st->Pp, p->len_max), rec = sizeof(RankRec) + 4 * rnw;
    const size_t room = (200 * 1024 - fixed_rank) / rec;
    if (std::min(room, cap) >= std::min(cap, (size_t)T + 256)) {
      st->rank_nw = rnw;
      st->rank_cap = (int32_t)std::min(room, cap);
      st->smem_rank = fixed_rank + st->rank_cap * rec;
    }
  }
  const bool need_all = st->rank_nw == 0 || (size_t)st->rank_cap < cap;
  if (st->smem_build > 220 * 1024 ||
      (need_all && st->smem_rank_all > 220 * 1024))
    return fail(EBIC_ERR_ARG, "population / top-rank sizes need more shared memory than a CTA has "
                              "(build %zu B, rank %zu B)",
                st->smem_build, st->smem_rank_all);
  EBIC_TRY(allow_smem(h, k_build<true>));
  EBIC_TRY(allow_smem(h, k_build<false>));
  if (st->rank_nw == 4) EBIC_TRY(allow_smem(h, k_rank_warp<4>));
  else if (st->rank_nw == 8) EBIC_TRY(allow_smem(h, k_rank_warp<8>));
  if (need_all) EBIC_TRY(allow_smem(h, k_rank));

  // The pair table pays for itself over a run; build it when it fits.
  if (h->path != EBIC_PATH_GATHER && !h->LT) {
    size_t free_b = 0, total_b = 0;
    cudaMemGetInfo(&free_b, &total_b);
    const size_t need = (size_t)h->C * h->C * h->W * sizeof(uint32_t);
    if (need < free_b / 2) EBIC_TRY(build_pair_table(h, s));
  }

  // A run without a table evaluates from the rank planes, all its generations.
  if (resolve_path(h) == EBIC_PATH_GATHER) {
    bool planes = false;
    EBIC_TRY(want_planes(h, s, false, kPlanesNow, &planes));
  }

  // Step 1: initial population, evaluation (autotuned once), top-rank list.
  const EaDev& dd = st->dev;
  const unsigned sblocks = (unsigned)((st->J + 127) / 128);
  k_spec<true, false><<<sblocks, 128, 0, s>>>(dd);
  k_build<true><<<1, kBuildThreads, st->smem_build, s>>>(dd, st->hmask, st->kB, st->depth);
  k_tabu_insert<<<(unsigned)((P + 255) / 256), 256, 0, s>>>(dd);
  count_launches(3);
  EBIC_CUDA_TRY(cudaGetLastError());
  Ctl c{};
  EBIC_TRY(read_ctl(st, s, &c));
  // The evaluation of the initial population, with the launch shape set by
  // hand (a nonzero kernel), else with the one the autotuner picks on it
  // (its candidates are evaluations of that population).  Either way any
  // scratch the shape needs is allocated here, before the capture below.
  const ebic_eval_tuning_t user_tuning = h->tuning;
  if (!c.stop) {
    if (user_tuning.kernel != 0) {
      EBIC_TRY(eval_archive(h, st->apop, a, s));
    } else {
      float us = 0.f;
      EBIC_TRY(autotune_archive(h, st->apop, a, s, &us));
    }
  }
  count_launches((uint64_t)launch_rank(st, s));
  EBIC_CUDA_TRY(cudaGetLastError());
  // attempt records of generation 1
  int nrec = 0;
  EBIC_TRY(launch_records(st, s, &nrec));
  count_launches((uint64_t)nrec);

  // One generation (Steps 2-5) captured as a graph for replay.
  st->tuning = h->tuning;
  EBIC_CUDA_TRY(cudaStreamCreateWithFlags(&st->side, cudaStreamNonBlocking));
  EBIC_CUDA_TRY(cudaStreamCreateWithFlags(&st->side2, cudaStreamNonBlocking));
  for (cudaEvent_t& e : st->fork_ev) EBIC_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  if (h->ktime_slots > 0) {
    st->tev.assign(2 * (size_t)h->ktime_slots, nullptr);
    st->tslots = h->ktime_slots;
    for (cudaEvent_t& e : st->tev) EBIC_CUDA_TRY(cudaEventCreate(&e));
  }
  EBIC_CUDA_TRY(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  ebic_status cap_st = launch_generation(h, st, s);
  cudaGraph_t graph = nullptr;
  cudaError_t ce = cudaStreamEndCapture(s, &graph);
  h->tuning = user_tuning;
  if (cap_st != EBIC_OK) {
    if (graph) cudaGraphDestroy(graph);
    return cap_st;
  }
  EBIC_CUDA_TRY(ce);
  st->graph = graph;
  if (st->tslots) {
    size_t n = 0;
    EBIC_CUDA_TRY(cudaGraphGetNodes(graph, nullptr, &n));
    std::vector<cudaGraphNode_t> nodes(n);
    EBIC_CUDA_TRY(cudaGraphGetNodes(graph, nodes.data(), &n));
    for (cudaGraphNode_t nd : nodes) {
      cudaGraphNodeType t;
      EBIC_CUDA_TRY(cudaGraphNodeGetType(nd, &t));
      if (t != cudaGraphNodeTypeEventRecord) continue;
      cudaEvent_t e = nullptr;
      EBIC_CUDA_TRY(cudaGraphEventRecordNodeGetEvent(nd, &e));
      for (int j = 0; j < 2; ++j)
        if (e == st->tev[j]) st->tnode[j] = nd;
    }
    if (!st->tnode[0] || !st->tnode[1])
      return fail(EBIC_ERR_DEVICE, "the captured generation has no timing nodes");
  }
  EBIC_CUDA_TRY(cudaGraphInstantiate(&st->exec, graph, 0));
  EBIC_CUDA_TRY(cudaStreamSynchronize(s));
  st->initialised = true;
  return EBIC_OK;
}

// Adds the k_build time of timing slot `slot` to the running sum (waits for
// that replay to finish).
static ebic_status harvest_timing(EaState* st, long long slot) {
  cudaEvent_t a = st->tev[2 * (size_t)(slot % st->tslots)];
  cudaEvent_t b = st->tev[2 * (size_t)(slot % st->tslots) + 1];
  EBIC_CUDA_TRY(cudaEventSynchronize(b));
  float ms = 0.f;
  EBIC_CUDA_TRY(cudaEventElapsedTime(&ms, a, b));
  st->tsum_ms += ms;
  st->tcount += 1;
  return EBIC_OK;
}

// One replay of the generation graph; with in-graph timing on, its two event
// nodes first move to the next slot of the ring (harvesting the replay that
// used the slot before).
static ebic_status graph_launch(EaState* st, cudaStream_t s) {
  if (st->tslots) {
    if (st->tlaunched - st->tharvested >= st->tslots) EBIC_TRY(harvest_timing(st, st->tharvested++));
    const size_t k = 2 * (size_t)(st->tlaunched % st->tslots);
    EBIC_CUDA_TRY(cudaGraphExecEventRecordNodeSetEvent(st->exec, st->tnode[0], st->tev[k]));
    EBIC_CUDA_TRY(cudaGraphExecEventRecordNodeSetEvent(st->exec, st->tnode[1], st->tev[k + 1]));
  }
  EBIC_CUDA_TRY(cudaGraphLaunch(st->exec, s));
  if (st->tslots) st->tlaunched += 1;    // a slot counts once its replay is queued
  return EBIC_OK;
}

// Longer runs replay their generations kGraphGens to a graph: consecutive replays
// of the one-generation graph leave 4 us between its last kernel and the next
// k_build, two generations inside a graph leave 0.5 us (1,000 x 100, P = 600: 76.8
// -> 73.0 ms for 1,000 generations).  Making and releasing the larger graph takes
// 350 us, so it is made by the call with which a run reaches kMultiFrom generations
// (a run of 16 generations of 200 x 20, P = 100: 1,174 us without it, 1,521 with;
// of 64: 3,268 and 3,456; of 128: 6,180 and 6,170; of 256: 11,998 and 11,584).
// Shorter calls and runs with in-graph timing, whose event nodes move from replay to
// replay, keep the one-generation graph, and so does a run whose larger graph cannot
// be made.
constexpr int32_t kGraphGens = 16, kMultiFrom = 128;

static void make_multi(EaState* st) {
  st->multi_tried = true;
  cudaGraph_t many = nullptr;
  cudaError_t e = cudaGraphCreate(&many, 0);
  cudaGraphNode_t prev = nullptr;
  for (int32_t i = 0; i < kGraphGens && e == cudaSuccess; ++i) {
    cudaGraphNode_t node = nullptr;
    e = cudaGraphAddChildGraphNode(&node, many, prev ? &prev : nullptr, prev ? 1 : 0, st->graph);
    prev = node;
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&st->multi, many, 0);
  if (e == cudaSuccess) {
    st->multi_graph = many;
    return;
  }
  cudaGetLastError();
  st->multi = nullptr;
  if (many) cudaGraphDestroy(many);
}

// A run's graph reads the weights of the surrogate it screens with.
static ebic_status scorer_left(const EaState* st) {
  if (st->sur && !*st->sur_alive)
    return fail(EBIC_ERR_STATE, "the surrogate this run screens with has been released");
  return EBIC_OK;
}

static ebic_status run_step(ebic_ctx* h, int32_t generations, ebic_stats_t* stats) {
  EaState* st = h->ea;
  if (!st || !st->initialised) return fail(EBIC_ERR_STATE, "ebic_run_init has not run");
  if (generations > 0) EBIC_TRY(scorer_left(st));
  if (generations < 0) return fail(EBIC_ERR_ARG, "negative generation count");
  const cudaStream_t s = h->stream;
  Ctl c{};
  EBIC_TRY(read_ctl(st, s, &c));
  if (!c.stop && c.gens_done + generations > st->p.iterations)
    return fail(EBIC_ERR_STATE, "the run was sized for %d generations (%d done, %d asked)",
                st->p.iterations, c.gens_done, generations);
  int32_t left = c.stop ? 0 : generations;
  st->stepped += left;
  if (left >= kGraphGens && st->stepped >= kMultiFrom && !st->tslots && !st->multi_tried)
    make_multi(st);
  while (left > 0) {
    const int32_t chunk = std::min<int32_t>(left, 64);
    int32_t i = 0;
    for (; st->multi && i + kGraphGens <= chunk; i += kGraphGens)
      EBIC_CUDA_TRY(cudaGraphLaunch(st->multi, s));
    for (; i < chunk; ++i) EBIC_TRY(graph_launch(st, s));
    count_launches((uint64_t)chunk * st->launches_per_gen);
    left -= chunk;
    EBIC_TRY(read_ctl(st, s, &c));
    if (c.stop) break;
  }
  EBIC_TRY(read_ctl(st, s, &c));
  fill_stats(c, stats);
  if (c.stop_reason == 3) return fail(EBIC_ERR_DEVICE, "internal EA error (code 3)");
  if (c.stop_reason == 4)
    return fail(EBIC_ERR_TIMEOUT, "a bounded wait for streamed attempt records expired");
  if (st->lost_scores) {
    EBIC_CUDA_TRY(cudaMemsetAsync(sur_lost_scores(st->sur), 0, sizeof(int), s));
    EBIC_CUDA_TRY(cudaStreamSynchronize(s));
    return fail(EBIC_ERR_TIMEOUT, "a bounded device wait expired while candidates were scored: some "
                                  "were picked without their scores");
  }
  return EBIC_OK;
}

ebic_status ea_archive(ebic_ctx* h, const uint16_t** seq, const int32_t** len, const double** fit,
                       long long* n, int32_t* stride) {
  EaState* st = h->ea;
  if (!st || !st->initialised) return fail(EBIC_ERR_STATE, "the handle has no run");
  Ctl c{};
  EBIC_TRY(read_ctl(st, h->stream, &c));
  *seq = st->seq.as<uint16_t>();
  *len = st->len.as<int32_t>();
  *fit = st->fit.as<double>();
  *stride = st->S;
  // generations 0 .. c.gen - 1 are evaluated (c.gen counts Step 1 as one)
  *n = std::min<long long>((long long)c.gen * st->p.pop_size, st->entries);
  return EBIC_OK;
}

// Gathers n records (archive entries refs[i], or g * P + i when refs is
// null) into packed rows: seq [n][S], then len, inc, dec (int32) and fitness.
__global__ void __launch_bounds__(256) k_gather(EaDev d, const int32_t* refs, long long first,
                                                int n, const uint32_t* inc, const uint32_t* dec,
                                                uint16_t* o_seq, int32_t* o_len, uint32_t* o_inc,
                                                uint32_t* o_dec, double* o_fit) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const long long r = refs ? (long long)refs[i] : first + i;
  const int L = d.len[r];
  for (int c = 0; c < d.S; ++c) o_seq[(size_t)i * d.S + c] = c < L ? d.seq[(size_t)r * d.S + c] : 0;
  o_len[i] = L;
  o_inc[i] = inc[r];
  o_dec[i] = dec[r];
  o_fit[i] = d.fit[r];
}

// Steps 2-5 replayed on the caller's stream without waiting or reading back.
static ebic_status run_step_async(ebic_ctx* h, int32_t generations, cudaStream_t s) {
  EaState* st = h->ea;
  if (!st || !st->initialised) return fail(EBIC_ERR_STATE, "ebic_run_init has not run");
  if (generations > 0) EBIC_TRY(scorer_left(st));
  if (generations < 0) return fail(EBIC_ERR_ARG, "negative generation count");
  for (int32_t i = 0; i < generations; ++i) EBIC_TRY(graph_launch(st, s));
  count_launches((uint64_t)generations * st->launches_per_gen);
  return EBIC_OK;
}

// One generation as separate launches with events between them, in the
// order of the graph's dependencies: Step 3, tabu insertion, evaluation,
// Step 5, then the next generation's attempt records (reported first).
static ebic_status run_step_profiled(ebic_ctx* h, float* us, cudaStream_t s) {
  EaState* st = h->ea;
  if (!st || !st->initialised) return fail(EBIC_ERR_STATE, "ebic_run_init has not run");
  EBIC_TRY(scorer_left(st));
  cudaEvent_t ev[8];
  for (int i = 0; i < 8; ++i) EBIC_CUDA_TRY(cudaEventCreate(&ev[i]));
  const EaDev& d = st->dev;
  cudaEventRecord(ev[0], s);
  k_build<false><<<1, kBuildThreads, st->smem_build, s>>>(d, st->hmask, st->kB, st->depth);
  cudaEventRecord(ev[1], s);
  k_tabu_insert<<<(unsigned)((st->p.pop_size + 255) / 256), 256, 0, s>>>(d);
  cudaEventRecord(ev[2], s);
  const ebic_eval_tuning_t user = h->tuning;
  h->tuning = st->tuning;
  ebic_status es = eval_archive(h, st->apop, st->eargs, s);
  h->tuning = user;
  cudaEventRecord(ev[3], s);
  const int nrank = launch_rank(st, s);
  cudaEventRecord(ev[4], s);
  int nrec = 0;
  const bool screened = d.V > 1;
  ebic_status rs = launch_records(st, s, &nrec, screened ? ev + 6 : nullptr);
  cudaEventRecord(ev[5], s);
  count_launches((uint64_t)(2 + nrank + nrec));
  cudaError_t e = cudaGetLastError();                   // of the launches
  const cudaError_t waited = cudaEventSynchronize(ev[5]);
  if (e == cudaSuccess) e = waited;
  // kernel_us order: records, build, tabu insertion, evaluation, rank; then,
  // when screening, the records stage split into candidates, scores, pick
  const int from[5] = {4, 0, 1, 2, 3};
  for (int i = 0; i < 5 && us; ++i) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ev[from[i]], ev[from[i] + 1]);
    us[i] = ms * 1000.f;
  }
  if (us) {
    us[5] = us[6] = us[7] = 0.f;
    if (screened && rs == EBIC_OK) {
      const cudaEvent_t* seg[4] = {&ev[4], &ev[6], &ev[7], &ev[5]};
      for (int i = 0; i < 3; ++i) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, *seg[i], *seg[i + 1]);
        us[5 + i] = ms * 1000.f;
      }
    }
  }
  for (int i = 0; i < 8; ++i) cudaEventDestroy(ev[i]);
  EBIC_TRY(rs);
  EBIC_TRY(es);
  EBIC_CUDA_TRY(e);
  return EBIC_OK;
}

static ebic_status get_records(ebic_ctx* h, bool toprank, int32_t* offsets, int32_t* cols,
                               double* fitness, uint32_t* inc, uint32_t* dec, int32_t* inout_n) {
  EaState* st = h->ea;
  if (!st || !st->initialised) return fail(EBIC_ERR_STATE, "ebic_run_init has not run");
  if (!offsets || !cols || !inout_n || *inout_n < 0) return fail(EBIC_ERR_ARG, "null pointer");
  const cudaStream_t s = h->stream;
  Ctl c{};
  EBIC_TRY(read_ctl(st, s, &c));
  const int32_t P = st->p.pop_size, S = st->S;
  // the list, or the last evaluated generation (c.gen - 1)
  const int32_t avail = toprank ? c.n_top : (c.gen > 0 ? P : 0);
  const int32_t n = std::min<int32_t>(*inout_n, avail);
  offsets[0] = 0;
  *inout_n = n;
  if (n == 0) return EBIC_OK;
  const size_t row = (size_t)S * sizeof(uint16_t);
  const size_t bytes = (size_t)n * (row + 3 * sizeof(int32_t) + sizeof(double));
  EBIC_TRY(st->gather.reserve(bytes));
  EBIC_TRY(st->h_gather.reserve(bytes));
  // regions by decreasing element size, so every one is aligned:
  // fitness [n] (8 B) | len, inc, dec [n] (4 B) | seq [n][S] (2 B)
  char* dbase = static_cast<char*>(st->gather.ptr);
  double* o_fit = reinterpret_cast<double*>(dbase);
  int32_t* o_len = reinterpret_cast<int32_t*>(o_fit + n);
  uint32_t* o_inc = reinterpret_cast<uint32_t*>(o_len + n);
  uint32_t* o_dec = o_inc + n;
  uint16_t* o_seq = reinterpret_cast<uint16_t*>(o_dec + n);
  k_gather<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
      st->dev, toprank ? st->list_ref.as<int32_t>() : nullptr, (long long)(c.gen - 1) * P, n,
      st->inc.as<uint32_t>(), st->dec.as<uint32_t>(), o_seq, o_len, o_inc, o_dec, o_fit);
  count_launches(1);
  EBIC_CUDA_TRY(cudaGetLastError());
  EBIC_CUDA_TRY(cudaMemcpyAsync(st->h_gather.ptr, st->gather.ptr, bytes, cudaMemcpyDeviceToHost, s));
  EBIC_CUDA_TRY(cudaStreamSynchronize(s));
  const double* h_fit = static_cast<const double*>(st->h_gather.ptr);
  const int32_t* h_len = reinterpret_cast<const int32_t*>(h_fit + n);
  const uint32_t* h_inc = reinterpret_cast<const uint32_t*>(h_len + n);
  const uint32_t* h_dec = h_inc + n;
  const uint16_t* h_seq = reinterpret_cast<const uint16_t*>(h_dec + n);
  for (int32_t i = 0; i < n; ++i) {
    const int32_t L = h_len[i];
    for (int32_t t = 0; t < L; ++t) cols[offsets[i] + t] = h_seq[(size_t)i * S + t];
    offsets[i + 1] = offsets[i] + L;
    if (fitness) fitness[i] = h_fit[i];
    if (inc) inc[i] = h_inc[i];
    if (dec) dec[i] = h_dec[i];
  }
  return EBIC_OK;
}

}  // namespace ebic

using namespace ebic;

extern "C" {

void ebic_default_params(ebic_params_t* p) {
  if (!p) return;
  p->pop_size = 100;
  p->len_min = 2;
  p->len_max = 6;
  p->iterations = 10;
  p->sigma = 10;
  p->toprank_size = 100;
  p->tournament_k = 2;
  p->support_mode = EBIC_SUPPORT_INC;
  p->overlap_tau = 0.5;
  p->elite_frac = 0.25;
  p->penalty_base = 1.2;
  p->p_crossover = 0.5;
  p->seed = 0;
}

ebic_status ebic_run_init(ebic_handle h, const ebic_params_t* p) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != h->device) cudaSetDevice(h->device);
  ebic_status st = run_init(h, p);
  if (st != EBIC_OK) ea_release(h);
  if (prev >= 0 && prev != h->device) cudaSetDevice(prev);
  return st;
}

ebic_status ebic_run_step(ebic_handle h, int32_t generations, ebic_stats_t* stats) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  return run_step(h, generations, stats);
}

ebic_status ebic_run_step_async(ebic_handle h, int32_t generations, void* stream) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  return run_step_async(h, generations, static_cast<cudaStream_t>(stream));
}

ebic_status ebic_run_step_profiled(ebic_handle h, float* kernel_us) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  return run_step_profiled(h, kernel_us, h->stream);
}

ebic_status ebic_set_kernel_timing(ebic_handle h, int32_t slots) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  if (slots < 0 || slots > (1 << 20)) return fail(EBIC_ERR_ARG, "timing slots %d outside [0, 2^20]", slots);
  h->ktime_slots = slots;
  return EBIC_OK;
}

ebic_status ebic_read_kernel_timing(ebic_handle h, int32_t reset, double* mean_us, long long* count) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  EaState* st = h->ea;
  if (!st || !st->initialised) return fail(EBIC_ERR_STATE, "ebic_run_init has not run");
  if (!st->tslots) return fail(EBIC_ERR_STATE, "the run was started without kernel timing");
  while (st->tharvested < st->tlaunched) EBIC_TRY(harvest_timing(st, st->tharvested++));
  if (mean_us) *mean_us = st->tcount ? 1e3 * st->tsum_ms / (double)st->tcount : 0.0;
  if (count) *count = st->tcount;
  if (reset) {
    st->tsum_ms = 0.0;
    st->tcount = 0;
  }
  return EBIC_OK;
}

ebic_status ebic_run_screen(ebic_handle h, ebic_surrogate s, int32_t oversample, int32_t mode) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  if (oversample < 1 || oversample > 16)
    return fail(EBIC_ERR_ARG, "oversample %d outside [1, 16]", oversample);
  if (mode != EBIC_SCREEN_OFF && mode != EBIC_SCREEN_SURROGATE && mode != EBIC_SCREEN_PSEUDO)
    return fail(EBIC_ERR_ARG, "bad screening mode %d", mode);
  if (mode == EBIC_SCREEN_SURROGATE && !s) return fail(EBIC_ERR_ARG, "surrogate mode needs a surrogate");
  if (mode == EBIC_SCREEN_SURROGATE && sur_columns(s) != h->C)
    return fail(EBIC_ERR_ARG, "the surrogate has %d columns, the matrix %d", sur_columns(s), h->C);
  // the handle holds one reference to its screening surrogate
  if (h->screen_sur) sur_attach(h->screen_sur, -1);
  h->screen_sur = mode == EBIC_SCREEN_SURROGATE ? s : nullptr;
  if (h->screen_sur) sur_attach(h->screen_sur, +1);
  h->screen_v = oversample;
  h->screen_mode = mode;
  return EBIC_OK;
}

ebic_status ebic_get_toprank(ebic_handle h, int32_t* offsets, int32_t* cols, double* fitness,
                             uint32_t* inc, int32_t* inout_n) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  return get_records(h, true, offsets, cols, fitness, inc, nullptr, inout_n);
}

ebic_status ebic_get_population(ebic_handle h, int32_t* offsets, int32_t* cols, uint32_t* inc,
                                uint32_t* dec, double* fitness, int32_t* inout_n) {
  if (!h) return fail(EBIC_ERR_ARG, "null handle");
  return get_records(h, false, offsets, cols, fitness, inc, dec, inout_n);
}

ebic_status ebic_run_generations(ebic_handle h, const ebic_params_t* p, int32_t* out_offsets,
                                 int32_t* out_cols, double* out_fitness, int32_t* inout_n,
                                 ebic_stats_t* stats) {
  if (!h || !p) return fail(EBIC_ERR_ARG, "null pointer");
  EBIC_TRY(ebic_run_init(h, p));
  EBIC_TRY(ebic_run_step(h, p->iterations, stats));
  return ebic_get_toprank(h, out_offsets, out_cols, out_fitness, nullptr, inout_n);
}

}  // extern "C"

// One training step of the surrogate on the fifth-generation tensor cores
// (tcgen05.mma, bf16 operands, fp32 accumulators in tensor memory), in four
// launches:
//   k_train_tc    forward and reverse pass of a tile of 128 series in one CTA:
//                 minibatch draw, features, x W1, h1 W2, the output layer and
//                 the loss, dh2 W2^T, dh1 W1^T, the segment's column sums.  The accumulators never leave
//                 tensor memory except through an epilogue, each epilogue feeds
//                 the next product a quarter of K at a time through 16 KB of
//                 shared memory, and W1^T and W2^T serve both directions from
//                 one copy;
//   k_wgrad_tc    the weight gradients h1^T dh2 and x^T dh1 (K = the batch,
//                 split-K), both operands MN-major as they lie in memory;
//   k_emb_part    the embedding gradient;
//   k_finish      partial sums in split order, Adam, every copy of the weights.
// Products, rounding points and summation orders are those of separate kernels
// per step (GEMM by GEMM): results do not depend on the fusion.
//
// The tile kernel is latency-bound (32 tiles at a batch of 4,096 on 152 SMs, a
// chain of thirteen MMA groups each); per step 172 us as 31 launches of one
// operation each.
//
// Operand layouts, no swizzle, core matrices of 8 rows x 16 bytes: element
// (r, c) of a matrix whose core matrices are ordered row-group by row-group is
// at cm(r, c, C) (ebic_tcmlp.cuh).  Read with rows = M or N and 16-byte runs
// along K it is K-major: lbo 128 (next 8 k), sbo C * 16 (next 8 rows).  Read the
// other way -- rows = K, runs along M or N -- the same bytes are an MN-major
// operand: sbo 128 (next 8 of M or N), lbo C * 16 (next 8 k).  That is how W^T
// serves the reverse pass, and how the activations enter the weight gradients
// without a transpose.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "ebic_async.cuh"
#include "ebic_tcmlp.cuh"

namespace ebic {

namespace tct {

using namespace tc;
typedef __nv_bfloat16 bf;

// instruction-descriptor bits: A / B are MN-major
constexpr uint32_t kAmn = 1u << 15, kBmn = 1u << 16;

// Word 0 | word 1 of Philox-4x32-10 at counter (b, step, 0x5EED, 0), key seed,
// modulo n: the minibatch draw.
__device__ __forceinline__ int32_t draw_row(uint64_t seed, uint32_t step, uint32_t b, long long n) {
  uint32_t x0 = b, x1 = step, x2 = 0x5EEDu, x3 = 0u;
  uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * x0, hi0 = __umulhi(0xD2511F53u, x0);
    const uint32_t lo1 = 0xCD9E8D57u * x2, hi1 = __umulhi(0xCD9E8D57u, x2);
    const uint32_t y0 = hi1 ^ x1 ^ k0, y2 = hi0 ^ x3 ^ k1;
    x0 = y0;
    x1 = lo1;
    x2 = y2;
    x3 = lo0;
  }
  return (int32_t)((((unsigned long long)x0 << 32 | x1) % (unsigned long long)n));
}

// Two runs of 8 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void ld8x2(uint32_t ta, uint32_t tb, float (&v)[8], float (&u)[8]) {
  uint32_t r[8], t[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(ta));
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(t[0]), "=r"(t[1]), "=r"(t[2]), "=r"(t[3]), "=r"(t[4]), "=r"(t[5]),
                 "=r"(t[6]), "=r"(t[7])
               : "r"(tb));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    v[i] = __uint_as_float(r[i]);
    u[i] = __uint_as_float(t[i]);
  }
}

// Eight fp32 values rounded to bf16 into 16 bytes.
__device__ __forceinline__ uint4 pack8(const float* v) {
  __align__(16) bf o[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) o[i] = __float2bfloat16_rn(v[i]);
  return *reinterpret_cast<const uint4*>(o);
}

// The order in which a warp per row would sum y: lane l adds columns l, l + 32,
// ..., then a butterfly.  p[l] is at ps[l * 128].
__device__ __forceinline__ float tree32(const float* ps) {
  float q[16];
#pragma unroll
  for (int l = 0; l < 16; ++l) q[l] = ps[l * kTT] + ps[(l + 16) * kTT];
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int l = 0; l < 8; ++l)
      if (l < o) q[l] = q[l] + q[l + o];
  return q[0];
}

}  // namespace tct

// What a training call reads back.  `lost` is set by a kernel whose bounded wait
// expired; from then on k_finish leaves the parameters as they are and counts no
// step, until the host has reported it and cleared the word.
struct TrainWords {
  float loss;
  int32_t lost;
  int32_t done, drawn;                      // replays: steps finished, steps drawn
};

// The buffers of one step (device pointers; B rows).
struct TrainBufs {
  __nv_bfloat16 *x, *h1, *h2, *dh1, *dh2;   // [B][80], [B][256] x 4
  float *dx;                                // [B][64]
  float *y, *dy, *sq;                       // [B]
  int32_t* idx;                             // [B] rows of the minibatch
  TrainWords* words;
};

// Where the minibatch comes from: rows idx (nullptr: 0 .. B - 1), or, with
// draw, drawn from n rows for step `step` + words->done and left in
// their idx.
struct TrainRows {
  const int32_t* idx;
  bool draw;
  uint64_t seed;
  uint32_t step;
  long long n;
};

__global__ void __launch_bounds__(tc::kThreads, 1)
k_train_tc(const uint16_t* __restrict__ seq, const int32_t* __restrict__ len, int32_t stride,
           TrainRows rows, int32_t B, int32_t C, const float* __restrict__ emb,
           const float* __restrict__ cmean, const float* __restrict__ csd, float len_scale,
           const __nv_bfloat16* __restrict__ wpack, const float* __restrict__ b1,
           const float* __restrict__ b2, const float* __restrict__ w3,
           const float* __restrict__ b3, const float* __restrict__ target, TrainBufs o,
           float* __restrict__ cpart) {
  using namespace tct;
  extern __shared__ __align__(128) unsigned char tsm[];
  bf* sW1 = reinterpret_cast<bf*>(tsm);                        // W1^T, 256 x 80
  bf* sW2 = sW1 + kH * kF;                                     // W2^T, 256 x 256
  bf* sX = sW2 + kH * kH;                                      // x, 128 x 80
  bf* sH = sX;                                                 // a quarter, 128 x 64
  float* b1s = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(sX) + kXH);
  float* b2s = b1s + kH;
  float* w3s = b2s + kH;
  float* dys = w3s + kH;                                       // [128]
  float* sqs = dys + kTT;                                      // [128]
  __shared__ __align__(8) unsigned long long wbar, mbar;
  __shared__ uint32_t tslot;
  __shared__ int32_t s_row[kTT];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ntiles = (B + kTT - 1) / kTT;
  if (tid == 0) {
    mbar_init(&wbar, 1);
    mbar_init(&mbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (tid == 0) bulk_load(sW1, wpack, (uint32_t)(kW1 + kW2), &wbar);
  warm_rows(emb, C, tid, kThreads);
  for (int i = tid; i < kH; i += kThreads) {
    b1s[i] = b1[i];
    b2s[i] = b2[i];
    w3s[i] = w3[i];
  }
  const float bias3 = b3[0];
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&tslot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tslot;
  const uint32_t aX = smem_addr(sX), aW1 = smem_addr(sW1), aW2 = smem_addr(sW2);
  const int q = warp & 3, cg = warp >> 2, row = 32 * q + lane;
  const uint32_t tlane = tmem + ((uint32_t)(32 * q) << 16);
  uint32_t ph = 0;
  bool ok = true, weights = false;
  auto wait_mma = [&]() -> bool {
    const bool w = mbar_wait(&mbar, ph);
    ph ^= 1u;
    fence_after();
    return __syncthreads_and(w) != 0;
  };
  // shared-memory writes of every thread visible to the tensor cores
  auto publish = [&]() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    fence_before();
    __syncthreads();
    fence_after();
  };
  // this thread's 16 values of column group cg into the operand quarter
  auto put = [&](const float (&v)[16]) {
#pragma unroll
    for (int g8 = 0; g8 < 2; ++g8)
      *reinterpret_cast<uint4*>(sH + cm(row, 16 * cg + 8 * g8, kQ)) = pack8(v + 8 * g8);
  };
  // the operand quarter to columns [64 h, 64 h + 64) of dst by warps 8 .. 15, 64
  // bytes of eight rows per warp and store (a thread's own row would touch 32
  // lines a store)
  auto copy_out = [&](int r0, int h, bf* dst) {
    if (warp < 8) return;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = tid - 256 + 256 * i, g = (t >> 3) & 7, r = (t >> 6) * 8 + (t & 7);
      const uint4 u = *reinterpret_cast<const uint4*>(sH + cm(r, 8 * g, kQ));
      if (r0 + r < B)
        *reinterpret_cast<uint4*>(dst + (size_t)(r0 + r) * kH + kQ * h + 8 * g) = u;
    }
  };
  // by warps 0 .. 7, the column sums of the operand quarter (scaled by dys with `scale`) in the
  // order of k_colsum_all -- a tile is one of its segments: row class lane / 4
  // adds its sixteen rows in order, then the classes are added in order
  auto col_sums = [&](int tile, int h, int which, bool scale) {
    if (warp >= 8) return;
    const int c = 8 * warp + 2 * (lane & 3);
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int r = 8 * j + (lane >> 2);
      const __nv_bfloat162 u = *reinterpret_cast<const __nv_bfloat162*>(sH + cm(r, c, kQ));
      if (scale) {
        s0 = __fmaf_rn(dys[r], __low2float(u), s0);
        s1 = __fmaf_rn(dys[r], __high2float(u), s1);
      } else {
        s0 = __fadd_rn(s0, __low2float(u));
        s1 = __fadd_rn(s1, __high2float(u));
      }
    }
    float t0 = 0.f, t1 = 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      t0 += __shfl_sync(0xffffffffu, s0, 4 * r + (lane & 3));
      t1 += __shfl_sync(0xffffffffu, s1, 4 * r + (lane & 3));
    }
    if (lane < 4)
      *reinterpret_cast<float2*>(cpart + ((size_t)which * ntiles + tile) * kH + kQ * h + c) =
          make_float2(t0, t1);
  };
  for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
    const int r0 = tile * kTT, grow = r0 + row;
    // ---- the minibatch rows ----
    if (tid < kTT) {
      const int b = r0 + tid;
      int32_t r = b < B ? b : 0;
      if (rows.draw) {
        r = b < B ? draw_row(rows.seed, rows.step + (uint32_t)o.words->done, (uint32_t)b, rows.n) : 0;
        if (b < B) o.idx[b] = r;
      } else if (rows.idx && b < B) {
        r = rows.idx[b];
      }
      s_row[tid] = r;
    }
    __syncthreads();
    // ---- features: warp w builds rows [8 w, 8 w + 8) ----
    {
      const int rb = warp * 8;
      const bool in = lane < 8 && r0 + rb + lane < B;
      const long long sr = in ? s_row[rb + lane] : 0;
      const int L = in ? min(max(len[sr], 0), stride) : 0;
      float4 acc[4];
      float m, dsum;
      gather_rows(seq + (size_t)sr * stride, L, lane, C, emb, cmean, csd, acc, m, dsum);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = rb + 2 * j + (lane >> 4), c = 4 * (lane & 15);
        const uint2 u = pack4(acc[j].x, acc[j].y, acc[j].z, acc[j].w);
        *reinterpret_cast<uint2*>(sX + cm(r, c, kF)) = u;
        if (r0 + r < B) *reinterpret_cast<uint2*>(o.x + (size_t)(r0 + r) * kF + c) = u;
      }
      if (lane < 8) {
        const uint2 st = pack4(L ? m / (float)L : 0.f, L ? dsum / (float)L : 0.f,
                               (float)L / len_scale, 0.f);
        const uint4 u = make_uint4(st.x, st.y, 0u, 0u), z = make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(sX + cm(rb + lane, 64, kF)) = u;
        *reinterpret_cast<uint4*>(sX + cm(rb + lane, 72, kF)) = z;
        if (in) {
          uint4* dst = reinterpret_cast<uint4*>(o.x + (size_t)(r0 + rb + lane) * kF + 64);
          dst[0] = u;
          dst[1] = z;
        }
      }
    }
    publish();
    if (!weights) {                      // the weights have had the features' time to land
      const bool w = mbar_wait(&wbar, 0);
      if (!(ok = __syncthreads_and(w) != 0)) break;
      weights = true;
    }
    // ---- x W1 into TMEM columns [0, 256) ----
    if (tid == 0) {
      for (int k0 = 0; k0 < kF; k0 += 16)
        mma(tmem, sdesc(aX + (k0 / 8) * 128, 128, (kF / 8) * 128),
            sdesc(aW1 + (k0 / 8) * 128, 128, (kF / 8) * 128), idesc(kTT, kH), k0 > 0);
      commit(&mbar);
    }
    if (!(ok = wait_mma())) break;
    // ---- h1 by quarters of 64 columns, each followed by its share of h1 W2
    // into columns [256, 512); bit i of on1[h]: column 64 h + 16 cg + i > 0 ----
    uint32_t on1[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      float v[16];
      ld16(tlane + (uint32_t)(kQ * h + 16 * cg), v);
      on1[h] = 0u;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        v[i] = fmaxf(v[i] + b1s[kQ * h + 16 * cg + i], 0.f);
        on1[h] |= __bfloat162float(__float2bfloat16_rn(v[i])) > 0.f ? 1u << i : 0u;
      }
      put(v);
      publish();
      if (tid == 0) {
        for (int k0 = 0; k0 < kQ; k0 += 16)
          mma(tmem + (uint32_t)kH, sdesc(aX + (k0 / 8) * 128, 128, (kQ / 8) * 128),
              sdesc(aW2 + ((kQ * h + k0) / 8) * 128, 128, (kH / 8) * 128), idesc(kTT, kH),
              h > 0 || k0 > 0);
        commit(&mbar);
      }
      copy_out(r0, h, o.h1);
      if (!(ok = wait_mma())) break;         // nothing more issued behind a lost phase
    }
    if (!ok) break;
    // ---- y, the loss and dy: thread cg of a row takes columns 8 cg .. 8 cg + 7 of
    // every 32 ----
    {
      float p[8];
#pragma unroll
      for (int l = 0; l < 8; ++l) p[l] = 0.f;
#pragma unroll 2
      for (int i = 8 * cg; i < kH; i += 64) {
        float v[8], u[8];
        ld8x2(tlane + (uint32_t)(kH + i), tlane + (uint32_t)(kH + i + 32), v, u);
#pragma unroll
        for (int l = 0; l < 8; ++l)
          p[l] = __fmaf_rn(__bfloat162float(__float2bfloat16_rn(fmaxf(v[l] + b2s[i + l], 0.f))),
                           w3s[i + l], p[l]);
#pragma unroll
        for (int l = 0; l < 8; ++l)
          p[l] = __fmaf_rn(__bfloat162float(__float2bfloat16_rn(fmaxf(u[l] + b2s[i + 32 + l], 0.f))),
                           w3s[i + 32 + l], p[l]);
      }
      float* ps = reinterpret_cast<float*>(sH);                // [32][128]
#pragma unroll
      for (int l = 0; l < 8; ++l) ps[(8 * cg + l) * kTT + row] = p[l];
      __syncthreads();
      if (cg == 0) {
        float s = tree32(ps + row);
        s += bias3;
        float dyv = 0.f, sqv = 0.f;
        if (grow < B) {
          const float r = s - target[s_row[row]];
          dyv = 2.f * r / (float)B;
          sqv = r * r / (float)B;
        }
        dys[row] = dyv;
        sqs[row] = sqv;
      }
    }
    __syncthreads();
    const float dyr = dys[row];
    if (warp == 7 && lane < 16) {            // this segment's loss (lanes 0-7) and b3 sums
      const float* X = lane < 8 ? sqs : dys;
      float s = 0.f;
#pragma unroll
      for (int j = 0; j < 16; ++j) s += X[8 * j + (lane & 7)];
      float t = 0.f;
#pragma unroll
      for (int r = 0; r < 8; ++r) t += __shfl_sync(0xffffu, s, (lane & 8) + r);
      if ((lane & 7) == 0)
        cpart[(size_t)3 * ntiles * kH + (size_t)(lane >> 3) * ntiles + tile] = t;
    }
    // ---- dh2 by quarters, each followed by its share of dh2 W2^T into columns
    // [0, 256) ----
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      float v[16];
      ld16(tlane + (uint32_t)(kH + kQ * h + 16 * cg), v);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = fmaxf(v[i] + b2s[kQ * h + 16 * cg + i], 0.f);
      put(v);                                // h2, for the gradient of w3
      __syncthreads();
      col_sums(tile, h, 0, true);
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 16; ++i)
        v[i] = __bfloat162float(__float2bfloat16_rn(v[i])) > 0.f
                   ? dyr * w3s[kQ * h + 16 * cg + i]
                   : 0.f;
      put(v);
      publish();
      if (tid == 0) {
        for (int k0 = 0; k0 < kQ; k0 += 16)
          mma(tmem, sdesc(aX + (k0 / 8) * 128, 128, (kQ / 8) * 128),
              sdesc(aW2 + ((kQ * h + k0) / 8) * (kH / 8) * 128, (kH / 8) * 128, 128),
              idesc(kTT, kH) | kBmn, h > 0 || k0 > 0);
        commit(&mbar);
      }
      copy_out(r0, h, o.dh2);
      col_sums(tile, h, 1, false);
      if (!(ok = wait_mma())) break;         // nothing more issued behind a lost phase
    }
    if (!ok) break;
    // ---- dh1 by quarters, each followed by its share of dh1 W1^T (the 64
    // embedding dimensions) into columns [256, 320) ----
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      float v[16];
      ld16(tlane + (uint32_t)(kQ * h + 16 * cg), v);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = (on1[h] >> i) & 1u ? v[i] : 0.f;
      put(v);
      publish();
      if (tid == 0) {
        for (int k0 = 0; k0 < kQ; k0 += 16)
          mma(tmem + (uint32_t)kH, sdesc(aX + (k0 / 8) * 128, 128, (kQ / 8) * 128),
              sdesc(aW1 + ((kQ * h + k0) / 8) * (kF / 8) * 128, (kF / 8) * 128, 128),
              idesc(kTT, kEmb) | kBmn, h > 0 || k0 > 0);
        commit(&mbar);
      }
      copy_out(r0, h, o.dh1);
      col_sums(tile, h, 2, false);
      if (!(ok = wait_mma())) break;         // nothing more issued behind a lost phase
    }
    if (!ok) break;
    {
      float v[16];
      ld16(tlane + (uint32_t)(kH + 16 * cg), v);
      if (grow < B) {
        float4* dst = reinterpret_cast<float4*>(o.dx + (size_t)grow * kEmb + 16 * cg);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          dst[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      }
    }
    fence_before();
    __syncthreads();
    fence_after();
  }
  if (!ok) {
    if (tid == 0) atomicExch(&o.words->lost, 1);
    if (weights) mbar_wait(&mbar, ph ^ 1u);               // let the MMAs finish before freeing
  }
  if (!weights) mbar_wait(&wbar, 0);                      // let the copy land before leaving
  // (k_finish advances `done` and reads `drawn`)
  if (rows.draw && blockIdx.x == 0 && tid == 0) o.words->drawn += 1;
  fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
}

// ---------------------------------------------------------------------------
// Weight gradients, split-K over the batch: D[m][n] = sum over rows b of
// A[b][m] B[b][n].  grid = (256 / 64 column tiles, 3 row tiles, splits): row
// tiles 0 and 1 are h1^T dh2, tile 2 is x^T dh1.  A CTA brings 256 rows of its
// 128 and 64 columns into shared memory with 16-byte asynchronous copies -- the
// rows are K and the columns contiguous, so both operands are MN-major as they
// come -- and one thread issues the MMAs, K = 16 each; split z takes rows
// [z kchunk, (z + 1) kchunk) and writes slice z, summed later in split order.
// ---------------------------------------------------------------------------
namespace tct {
constexpr int kSlab = 256;                  // rows in shared memory at a time
constexpr int kWN = 64;                     // columns of D per CTA
constexpr uint32_t kWCols = 64;             // TMEM columns
constexpr size_t kWgSmem = (size_t)kSlab * (kTT + kWN) * 2;

__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(on ? 16 : 0)
               : "memory");
}
}  // namespace tct

__global__ void __launch_bounds__(256)
k_wgrad_tc(TrainBufs o, int32_t B, int32_t kchunk, float* __restrict__ w2part,
           float* __restrict__ w1part) {
  using namespace tct;
  extern __shared__ __align__(128) unsigned char wsm[];
  __shared__ __align__(8) unsigned long long mbar;
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool first = blockIdx.y == 2;                     // x^T dh1
  const bf* A = first ? o.x : o.h1 + blockIdx.y * kTT;
  const bf* Bm = (first ? o.dh1 : o.dh2) + blockIdx.x * kWN;
  const int lda = first ? kF : kH, mcols = first ? kF : kTT;
  const uint32_t aA = smem_addr(wsm), aB = aA + kSlab * kTT * 2;
  const int kbeg = blockIdx.z * kchunk, kend = min(B, kbeg + kchunk);
  if (tid == 0) {
    mbar_init(&mbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&tslot)),
                 "r"(kWCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tslot;
  uint32_t ph = 0;
  bool ok = true;
  for (int k0 = kbeg; k0 < kend && ok; k0 += kSlab) {
    const int nk = min(kSlab, (kend - k0 + 15) / 16 * 16);      // rows the MMAs read
    // core matrix (k / 8, column / 8): 8 rows of 16 bytes; rows past the end
    // and columns past A's arrive as zeros
    // (a warp's copies: 8 rows of 64 bytes in memory, 512 bytes in a row here)
    for (int i = tid; i < nk * (kTT / 8); i += 256) {
      const int g = (i >> 3) % (kTT / 8), k = (i >> 3) / (kTT / 8) * 8 + (i & 7);
      const bool on = k0 + k < kend && 8 * g < mcols;
      cp16(aA + (uint32_t)(((k >> 3) * (kTT / 8) + g) * 128 + (k & 7) * 16),
           on ? A + (size_t)(k0 + k) * lda + 8 * g : A, on);
    }
    for (int i = tid; i < nk * (kWN / 8); i += 256) {
      const int g = (i >> 3) % (kWN / 8), k = (i >> 3) / (kWN / 8) * 8 + (i & 7);
      const bool on = k0 + k < kend;
      cp16(aB + (uint32_t)(((k >> 3) * (kWN / 8) + g) * 128 + (k & 7) * 16),
           on ? Bm + (size_t)(k0 + k) * kH + 8 * g : Bm, on);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    fence_before();
    __syncthreads();
    fence_after();
    if (tid == 0) {
      for (int kk = 0; kk < nk; kk += 16)
        mma(tmem, sdesc(aA + (uint32_t)(kk / 8) * (kTT / 8) * 128, (kTT / 8) * 128, 128),
            sdesc(aB + (uint32_t)(kk / 8) * (kWN / 8) * 128, (kWN / 8) * 128, 128),
            idesc(kTT, kWN) | kAmn | kBmn, k0 > kbeg || kk > 0);
      commit(&mbar);
    }
    const bool w = mbar_wait(&mbar, ph);
    ph ^= 1u;
    ok = __syncthreads_and(w) != 0;
    fence_after();
  }
  if (ok) {
    const int q = warp & 3, cg = warp >> 2, m = 32 * q + lane;
    float v[32];
    if (kbeg < kend) {
      ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(32 * cg), v);
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = 0.f;
    }
    if (m < mcols) {
      float* dst = first ? w1part + ((size_t)blockIdx.z * kF + m) * kH
                         : w2part + ((size_t)blockIdx.z * kH + blockIdx.y * kTT + m) * kH;
      float4* d4 = reinterpret_cast<float4*>(dst + blockIdx.x * kWN + 32 * cg);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        d4[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
  } else {
    mbar_wait(&mbar, ph ^ 1u);                      // let the MMAs finish before freeing
    if (tid == 0) atomicExch(&o.words->lost, 1);
  }
  fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kWCols)
                 : "memory");
}

// ---------------------------------------------------------------------------
// The five column sums of a step, sum_b scale[b] X[b][j], for the mma.sync
// kernels (k_train_tc forms them from its tile), in two fixed-order levels: CTA (32-column tile of one of them, segment of kColSeg rows) has its
// eight warps take every eighth row, each in row order, adds the warps in order
// and writes the segment's sums; k_finish adds the segments in order.  Column
// tiles 0-7: h2 scaled by dy (w3), 8-15: dh2 (b2), 16-23: dh1 (b1), 24: the
// squared errors (loss), 25: dy (b3).  part: [3][segments][256], then loss
// and b3 [segments] each.
// ---------------------------------------------------------------------------
constexpr int kColSeg = 128;
static_assert(kColSeg == tc::kTT, "a tile of k_train_tc is one segment");
__global__ void __launch_bounds__(256) k_colsum_all(TrainBufs o, int32_t B, float* __restrict__ part) {
  constexpr int kH = tc::kH;
  const int what = blockIdx.x >> 3, lane = threadIdx.x & 31, r0 = threadIdx.x >> 5;
  const int nseg = gridDim.y, seg = blockIdx.y;
  const int b_lo = seg * kColSeg, b_hi = min(B, b_lo + kColSeg);
  float s = 0.f;
  if (what < 3) {
    const int c = (blockIdx.x & 7) * 32 + lane;
    const __nv_bfloat16* X = what == 0 ? o.h2 : what == 1 ? o.dh2 : o.dh1;
#pragma unroll 8
    for (int b = b_lo + r0; b < b_hi; b += 8) {
      const float v = __bfloat162float(X[(size_t)b * kH + c]);
      s = what == 0 ? __fmaf_rn(o.dy[b], v, s) : __fadd_rn(s, v);
    }
  } else if (lane == 0) {
    const float* X = blockIdx.x == 24 ? o.sq : o.dy;
#pragma unroll 8
    for (int b = b_lo + r0; b < b_hi; b += 8) s += X[b];
  }
  __shared__ float red[8][33];
  red[r0][lane] = s;
  __syncthreads();
  if (r0 != 0) return;
  float t = 0.f;
  for (int q = 0; q < 8; ++q) t += red[q][lane];
  if (what < 3)
    part[((size_t)what * nseg + seg) * kH + (blockIdx.x & 7) * 32 + lane] = t;
  else if (lane == 0)
    part[(size_t)3 * nseg * kH + (size_t)(blockIdx.x - 24) * nseg + seg] = t;
}

// ---------------------------------------------------------------------------
// Embedding gradient without atomics on sums: dEmb[c] = sum over the batch's
// series b of (occurrences of c in series b) * dx[b].  CTA (32 columns, segment
// of series) accumulates its segment in series order into part[segment][c][64];
// k_finish adds the segments in order.  The occurrences of 128 series are
// counted in shared memory by all threads at once and turned into floats; then
// warp w takes columns 4 w .. 4 w + 3 with two dimensions a lane, every multiply
// predicated on the count (branches, or conversions in the loop, cost more than
// the multiplies they save: 17-25 us).  Latency-bound.
// ---------------------------------------------------------------------------
constexpr int kEmbCols = 32, kEmbRows = 128;
constexpr size_t kEmbSmem = (size_t)kEmbRows * 64 * 4 + (size_t)kEmbCols * kEmbRows * 4;
__global__ void __launch_bounds__(256)
k_emb_part(const uint16_t* __restrict__ seq, const int32_t* __restrict__ len, int32_t stride,
           const int32_t* __restrict__ idx, int32_t B, int32_t C, int32_t seg_len,
           const float* __restrict__ dx, float* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char esm[];
  float* dxs = reinterpret_cast<float*>(esm);                       // [kEmbRows][64]
  uint32_t* cnt = reinterpret_cast<uint32_t*>(dxs + kEmbRows * 64); // [kEmbCols][kEmbRows]
  float* cf = reinterpret_cast<float*>(cnt);                        // the same, as floats
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c0 = blockIdx.x * kEmbCols, seg = blockIdx.y;
  float acc[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = 0.f;
  const int b_lo = seg * seg_len, b_hi = min(B, b_lo + seg_len);
  for (int b0 = b_lo; b0 < b_hi; b0 += kEmbRows) {
    const int nb = min(kEmbRows, b_hi - b0);
    for (int i = tid; i < nb * 16; i += 256)
      tct::cp16(smem_addr(dxs) + 16u * i, dx + (size_t)b0 * 64 + 4 * i, true);
    const int bb = tid >> 1;                               // two threads a series
    int L = 0;
    const uint16_t* sp = seq;
    if (bb < nb) {
      const long long r = idx ? (long long)idx[b0 + bb] : b0 + bb;
      L = min(max(len[r], 0), stride);
      sp += (size_t)r * stride;
    }
    for (int i = tid; i < kEmbCols * kEmbRows; i += 256) cnt[i] = 0u;
    for (int i = nb * 64 + tid; i < ((nb + 7) & ~7) * 64; i += 256) dxs[i] = 0.f;
    __syncthreads();
    for (int i0 = tid & 1; i0 < L; i0 += 16) {             // eight columns in flight
      int c[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) c[u] = i0 + 2 * u < L ? (int)__ldg(sp + i0 + 2 * u) : C;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = c[u] - c0;
        if (c[u] < C && t >= 0 && t < kEmbCols) atomicAdd(cnt + t * kEmbRows + bb, 1u);
      }
    }
    __syncthreads();
    for (int i = tid; i < kEmbCols * kEmbRows; i += 256) cf[i] = (float)cnt[i];
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (int g = 0; g < nb; g += 4) {
      float4 w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        w[k] = *reinterpret_cast<const float4*>(cf + (4 * warp + k) * kEmbRows + g);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 u = reinterpret_cast<const float2*>(dxs + (g + j) * 64)[lane];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float f = j == 0 ? w[k].x : j == 1 ? w[k].y : j == 2 ? w[k].z : w[k].w;
          const float a0 = __fmaf_rn(f, u.x, acc[k][0]), a1 = __fmaf_rn(f, u.y, acc[k][1]);
          acc[k][0] = f != 0.f ? a0 : acc[k][0];
          acc[k][1] = f != 0.f ? a1 : acc[k][1];
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (c0 + 4 * warp + k < C)
      reinterpret_cast<float2*>(part + ((size_t)seg * C + c0 + 4 * warp + k) * 64)[lane] =
          make_float2(acc[k][0], acc[k][1]);
}

// ---------------------------------------------------------------------------
// The end of a step, one thread per parameter: the gradient from its partial
// sums in order, and with `update` Adam and every bf16 copy of the weights.
// ---------------------------------------------------------------------------
struct FinishArgs {
  long long o_w1, o_b1, o_w2, o_b2, o_w3, o_b3, n_par;   // Emb | W1 | b1 | W2 | b2 | w3 | b3
  const float *epart, *w1part, *w2part, *cpart;
  int nemb, ks, nseg;
  float *par, *grad, *mom, *vel;
  TrainWords* words;
  __nv_bfloat16 *w1b, *w2b, *pack_sync, *pack_tc;
  int update;
  float lr, c1, c2;                                      // Adam's bias corrections,
  const float2* ctab;                                    // or those of step drawn - 1
};

__device__ __forceinline__ float sum_in_order(const float* __restrict__ p, int n, long long step) {
  float s = 0.f;
  int z = 0;
  for (; z + 8 <= n; z += 8) {
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = p[(z + i) * step];
#pragma unroll
    for (int i = 0; i < 8; ++i) s += v[i];
  }
  for (; z < n; ++z) s += p[z * step];
  return s;
}

__global__ void __launch_bounds__(256) k_finish(FinishArgs a) {
  constexpr int kF = tc::kF, kH = tc::kH;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const float* cs = a.cpart;
  const size_t cw = (size_t)a.nseg * kH;
  if (i > a.n_par) return;
  const int32_t lost = a.words->lost;                    // then the step changes nothing
  if (i == a.n_par) {
    const float loss = sum_in_order(cs + 3 * cw, a.nseg, 1);
    if (lost) return;
    a.words->loss = loss;
    if (a.ctab) a.words->done += 1;                         // (k_train_tc reads it next)
    return;
  }
  float g;
  if (i < a.o_w1) g = sum_in_order(a.epart + i, a.nemb, a.o_w1);
  else if (i < a.o_b1) g = sum_in_order(a.w1part + (i - a.o_w1), a.ks, (long long)kF * kH);
  else if (i < a.o_w2) g = sum_in_order(cs + 2 * cw + (i - a.o_b1), a.nseg, kH);
  else if (i < a.o_b2) g = sum_in_order(a.w2part + (i - a.o_w2), a.ks, (long long)kH * kH);
  else if (i < a.o_w3) g = sum_in_order(cs + cw + (i - a.o_b2), a.nseg, kH);
  else if (i < a.o_b3) g = sum_in_order(cs + (i - a.o_w3), a.nseg, kH);
  else g = sum_in_order(cs + 3 * cw + a.nseg, a.nseg, 1);
  if (lost) return;
  a.grad[i] = g;
  if (!a.update) return;
  float c1 = a.c1, c2 = a.c2;
  if (a.ctab) {
    const float2 c = a.ctab[a.words->drawn - 1];
    c1 = c.x;
    c2 = c.y;
  }
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float mi = b1 * a.mom[i] + (1.f - b1) * g;
  const float vi = b2 * a.vel[i] + (1.f - b2) * g * g;
  a.mom[i] = mi;
  a.vel[i] = vi;
  const float pi = a.par[i] - a.lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  a.par[i] = pi;
  const __nv_bfloat16 p16 = __float2bfloat16_rn(pi);
  if (i >= a.o_w1 && i < a.o_b1) {
    const int j = (int)(i - a.o_w1), k = j / kH, n = j % kH;
    a.w1b[j] = p16;
    a.pack_sync[n * (kF + 8) + k] = p16;
    a.pack_tc[tc::cm(n, k, kF)] = p16;
  } else if (i >= a.o_w2 && i < a.o_b2) {
    const int j = (int)(i - a.o_w2), k = j / kH, n = j % kH;
    a.w2b[j] = p16;
    a.pack_sync[kH * (kF + 8) + n * (kH + 8) + k] = p16;
    a.pack_tc[kH * kF + tc::cm(n, k, kH)] = p16;
  }
}

}  // namespace ebic

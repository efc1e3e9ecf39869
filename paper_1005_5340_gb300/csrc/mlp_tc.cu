// Tensor-core kernels of the guess network (sm_103a, tcgen05 + TMA + mbarrier,
// inline PTX) for networks of up to 12 inputs, 256 units per hidden layer and
// 4 outputs; learn.cu keeps CUDA-core kernels for the others.
//
// Float32 accuracy on the bf16 tensor cores: a float32 value is the sum of
// three bf16 planes x = x0 + x1 + x2 (8 significant bits each) and the
// products of planes are exact in float32.  Activations times bf16 weights take
// three products (x0 w, x1 w, x2 w, all 24 bits of x); float32 times float32
// takes the six of weight 2^-16 or more.  The tensor core truncates when it
// accumulates, so the leading product x0 w0 has an accumulator of its own and
// the small ones share another: 16 truncations at full scale over K = 256
// instead of 96.  (Relative error against float64, 40000 rows: forward 2.1e-7,
// gradient 3.2e-7; one accumulator for all products gave 1.6e-6 and 1.8e-6,
// the CUDA-core kernels give 4e-7 and 9e-7.)
//
//   mlp_forward_kernel   one pass over the rows: features -> layer 1 (CUDA
//                        cores, up to 12 FMAs per unit) -> tanh -> layer 2 ->
//                        tanh -> output; the hidden layers never leave the SM
//                        unless a backward pass follows (H1 and H2 stored)
//   mlp_dh1_kernel       dH1 = (dH2 W2) (1 - H1^2), dH2 = (dY W3) (1 - H2^2)
//                        formed on the way into shared memory
//   mlp_dw2_kernel       dW2 = dH2^T H1 (reduction over the rows, per-CTA
//                        partial sums), with db2, dW3 and db3
//   mlp_dw1_kernel       dW1 = dH1^T F and db1 (CUDA cores, one unit per thread)
//   mlp_reduce_kernel    the partial sums of all CTAs, in order
// The forward pass is bound by the 512 tanhf per row (ALU); the backward
// kernels by the traffic of H1, H2 and dH1.
// 1.74 M rows, bf16 weights: 15.8 -> 1.34 ms; a gradient of 218 k rows in
// float32: 6.17 -> 1.21 ms (against the CUDA-core kernels).
//
// Every mbarrier wait is bounded; on expiry the kernel records an error code,
// stops issuing work, lets its copies and MMAs in flight finish and frees its
// tensor memory; a forward CTA then sets every output of its rows to NaN.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.h"
#include "mlp_tc.h"
#include "tc_ptx.h"

namespace tddft {
namespace {
using namespace ptx;

constexpr int MW = kMlpMaxWidth;        // 256: padded units of a hidden layer
constexpr int MT = 128;                 // rows per tile
constexpr int kEpiWarps = 16;           // four per TMEM lane quadrant
constexpr int kThreads = 64 + 32 * kEpiWarps;   // producer, MMA, epilogue
constexpr int kRing = 3;                // ring of 64-deep weight tiles
constexpr uint32_t kTileB = MW * 64 * 2;        // 32 KB: MW rows x 64 bf16
constexpr uint32_t kTileA = MT * 64 * 2;        // 16 KB: one plane of a 64-unit chunk
constexpr uint32_t kBufA = 3 * kTileA;          // a chunk's planes; two buffers
constexpr uint32_t kTHi = 0, kTLo = 256;        // tensor memory: leading and small products

__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// x = p[0] + p[1] + p[2], bf16 planes
__device__ __forceinline__ void split3(float x, __nv_bfloat16 (&p)[3]) {
  p[0] = __float2bfloat16_rn(x);
  const float r = x - __bfloat162float(p[0]);
  p[1] = __float2bfloat16_rn(r);
  p[2] = __float2bfloat16_rn(r - __bfloat162float(p[1]));
}
// planes of (x, y) packed, x in the low half
__device__ __forceinline__ void split3_pair(float x, float y, uint32_t (&w)[3]) {
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
    w[p] = *(const uint32_t *)&v;
    if (p < 2) {
      x -= __bfloat162float(v.x);
      y -= __bfloat162float(v.y);
    }
  }
}

// Range.  Planes below 2^-126 lose bits and a value above the largest bf16 has
// no plane, so the gradient of the second layer's input is held times 2^48
// (exact: what float32 holds at all keeps its 24 bits) and values beyond
// kDh2Max (2^52 unscaled) and infinities stay out of the tensor cores: their
// planes are zero, and the kernel adds them, or computes its rows again, in
// float32 on the CUDA cores when its pipeline has ended.  So for weights
// beyond kW2Max (256 products with one below it do not overflow).  NaN has
// planes.  Activations are at most 1; only below 2^-110 do they have fewer
// bits, an absolute error of 2^-134 per product.  (Gradient of 218 k rows:
// 1.19 -> 1.21 ms.)
constexpr float kDh2Scale = 0x1p48f, kDh2Unscale = 0x1p-48f, kDh2Max = 0x1p100f, kW2Max = 0x1p18f;
// the entry t (1 - h^2) of dH2 times 2^48, t = sum dY W3 as float32 has it (the
// scale comes in with 1 - h^2, so that no term of t overflows for it): one
// rounding wherever it is formed (both passes take the same decision on it)
__device__ __forceinline__ float dh2_scaled(float t, float h) {
  return __fmul_rn(t, fmaf(-kDh2Scale * h, h, kDh2Scale));
}
__device__ __forceinline__ float dh2_of(float t, float h) {
  return __fmul_rn(t, fmaf(-h, h, 1.f));
}
// Values without planes set to zero; whether there are any
template <int N>
__device__ __forceinline__ bool drop_odd(float (&x)[N]) {
  float m = 0.f;
#pragma unroll
  for (int j = 0; j < N; ++j) m = fmaxf(m, fabsf(x[j]));   // (skips NaN)
  if (m <= kDh2Max) return false;
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (fabsf(x[j]) > kDh2Max) x[j] = 0.f;
  return true;
}

// Weights as the kernels read them, once per call (they change every Adam
// step): padded W1, output weights (each float32, and rounded to bf16) and
// biases, the planes of W2 and of its transpose.
__global__ void mlp_prepare_kernel(MlpTc tc) {
  const float *prm = tc.params;
  const int W = tc.width, ni = tc.n_in, no = tc.n_out;
  const float *w1 = prm, *b1 = w1 + (int64_t)W * ni, *w2 = b1 + W, *b2 = w2 + (int64_t)W * W,
              *w3 = b2 + W, *b3 = w3 + (int64_t)no * W;
  const int n = blockIdx.x, k = threadIdx.x;   // MW x MW threads
  __nv_bfloat16 p[3];
  const float v2 = n < W && k < W ? w2[(int64_t)n * W + k] : 0.f;
  const bool plain = !(fabsf(v2) > kW2Max);
  const int odd = __syncthreads_or(!plain);
  split3(plain ? v2 : 0.f, p);
  for (int q = 0; q < 3; ++q) {
    tc.w2[((int64_t)q * MW + n) * MW + k] = p[q];
    tc.w2t[((int64_t)q * MW + k) * MW + n] = p[q];
  }
  if (k < kMlpMaxIn) {
    const float v = n < W && k < ni ? w1[(int64_t)n * ni + k] : 0.f;
    tc.w1[n * kMlpMaxIn + k] = v;
    tc.w1[(MW + n) * kMlpMaxIn + k] = __bfloat162float(__float2bfloat16_rn(v));
  }
  if (k == 0) {
    tc.vec[n] = n < W ? b1[n] : 0.f;
    tc.vec[MW + n] = n < W ? b2[n] : 0.f;
    bool inf3 = false;
    for (int o = 0; o < kMlpMaxOut; ++o) {
      const float v = n < W && o < no ? w3[(int64_t)o * W + n] : 0.f;
      tc.vec[(2 + o) * MW + n] = v;
      tc.vec[(2 + kMlpMaxOut + o) * MW + n] = __bfloat162float(__float2bfloat16_rn(v));
      inf3 |= isinf(v) != 0;
    }
    // dW2's copy: a unit with an infinite weight (0 x inf in rows past the end)
    // is zero there and left to the CUDA cores
    for (int o = 0; o < kMlpMaxOut; ++o)
      tc.w3_dw2[o * MW + n] = inf3 ? 0.f : tc.vec[(2 + o) * MW + n];
    tc.odd_w[n] = (odd ? 1 : 0) | (inf3 ? 2 : 0);
    if (n < kMlpMaxOut) tc.vec[(2 + 2 * kMlpMaxOut) * MW + n] = n < no ? b3[n] : 0.f;
  }
}

constexpr int kRingMax = 4;
struct Ctl {
  uint64_t lim;   // limit of the roles' waits (ns)
  uint64_t full[kRingMax], empty[kRingMax], afull[2], aempty[2], d2full, d2empty, yfull[2], drain;
  uint32_t tslot;
  int abort_flag;
  int odd;   // some value has no planes: the CUDA cores finish the rows
};

// Shared by the roles: a bounded wait of a whole warp that records its code.
__device__ __forceinline__ bool role_wait(uint64_t *bar, uint32_t parity, Ctl *ct, int *err,
                                          int code) {
  // (the limit is read only where the first try fails)
  const bool ok = mbar_try_wait(bar, parity) ||
                  mbar_wait(bar, parity, *(volatile uint64_t *)&ct->lim);
  if (__all_sync(0xffffffffu, ok && !*(volatile int *)&ct->abort_flag)) return true;
  if ((threadIdx.x & 31) == 0) atomicExch(err, code);
  *(volatile int *)&ct->abort_flag = 1;
  return false;
}
__device__ __forceinline__ void warp_arrive(uint64_t *bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}

__device__ __forceinline__ void ctl_init(Ctl *ct, int full_arrivals) {
  for (int i = 0; i < kRingMax; ++i) {
    mbar_init(&ct->full[i], full_arrivals);
    mbar_init(&ct->empty[i], 1);
  }
  for (int i = 0; i < 2; ++i) {
    mbar_init(&ct->afull[i], kEpiWarps);
    mbar_init(&ct->aempty[i], 1);
    mbar_init(&ct->yfull[i], kEpiWarps);
  }
  mbar_init(&ct->d2full, 1);
  mbar_init(&ct->d2empty, kEpiWarps);
  mbar_init(&ct->drain, 1);
  ct->abort_flag = 0;
  ct->odd = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// tensor memory of the whole SM, by warp 1 (before and after a block barrier),
// and the roles' wait limit
__device__ __forceinline__ uint32_t tmem_open(Ctl *ct, int warp, uint64_t lim) {
  if (threadIdx.x == 0) ct->lim = lim;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
        smem_u32(&ct->tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  return ct->tslot;
}
__device__ __forceinline__ void tmem_close(uint32_t tmem, int warp) {
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

// Weight tiles of one row tile, in order: per 64-deep chunk its planes.
__device__ __forceinline__ void ring_producer(Ctl *ct, uint8_t *ring, const CUtensorMap *map,
                                              int n_tiles, int nc, int planes, int *err) {
  if ((threadIdx.x & 31) != 0) return;
  int g = 0;
  bool ok = true;
  for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x)
    for (int c = 0; c < nc && ok; ++c)
      for (int p = 0; p < planes; ++p, ++g) {
        const int s = g % kRing;
        if (!mbar_wait(&ct->empty[s], ((uint32_t)(g / kRing) & 1u) ^ 1u, ct->lim) ||
            *(volatile int *)&ct->abort_flag) {
          atomicExch(err, 41);
          *(volatile int *)&ct->abort_flag = 1;
          ok = false;
          break;
        }
        mbar_expect_tx(&ct->full[s], kTileB);
        tma_load_2d(ring + s * kTileB, map, &ct->full[s], c * 64, p * MW);
      }
  // copies in flight land before the CTA may exit
  for (int h = max(0, g - kRing); h < g; ++h)
    mbar_wait(&ct->full[h % kRing], (uint32_t)(h / kRing) & 1u);
}

// The chunk product D2 += A x weight planes: with one weight plane x0 w, x1 w,
// x2 w; with three the six leading products; x0 w0 into the leading accumulator.
struct RingState {
  int slot = 0;
  uint32_t phase = 0;
};
template <int PLANES>
__device__ __forceinline__ bool chunk_mma(Ctl *ct, uint32_t leader, uint32_t ring_lo,
                                          uint32_t a_lo, uint32_t tmem, bool first, RingState &rs,
                                          int *err) {
  constexpr uint32_t idesc = idesc_bf16(MT, MW);
#pragma unroll
  for (int w = 0; w < PLANES; ++w) {
    if (!role_wait(&ct->full[rs.slot], rs.phase, ct, err, 42)) return false;
    fence_after();
    const uint32_t b = ring_lo + (uint32_t)rs.slot * (kTileB >> 4);
#pragma unroll
    for (int a = 0; a < (PLANES == 1 ? 3 : 3 - w); ++a) {
      const bool hi = w == 0 && a == 0;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        mma_bf16_if(leader, tmem + (hi ? kTHi : kTLo), desc_of(a_lo + a * (kTileA >> 4) + 2 * k),
                    desc_of(b + 2 * k), idesc,
                    (first && k == 0 && w == 0 && a <= 1) ? 0u : 1u);
    }
    mma_commit_if(leader, &ct->empty[rs.slot]);
    if (++rs.slot == kRing) {
      rs.slot = 0;
      rs.phase ^= 1u;
    }
  }
  return true;
}

// 16 values (units 16 g .. of a chunk) of tile row lr into the chunk's A
// planes: two 16-byte pieces of each plane's 128-byte swizzled row
__device__ __forceinline__ void put_planes(uint8_t *buf, int lr, int g, const float (&h)[16]) {
  uint32_t w[3][8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    uint32_t q[3];
    split3_pair(h[2 * j], h[2 * j + 1], q);
#pragma unroll
    for (int p = 0; p < 3; ++p) w[p][j] = q[p];
  }
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    uint8_t *row = buf + p * kTileA + lr * 128;
    *(uint4 *)(row + (((2 * g) ^ (lr & 7)) << 4)) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
    *(uint4 *)(row + (((2 * g + 1) ^ (lr & 7)) << 4)) =
        make_uint4(w[p][4], w[p][5], w[p][6], w[p][7]);
  }
  fence_async_smem();
}
// 16 columns of both accumulators, added
__device__ __forceinline__ void get_sum(uint32_t trow, int c0, float (&v)[16]) {
  float lo[16];
  tmem_ld16(trow + kTHi + (uint32_t)c0, v);
  tmem_ld16(trow + kTLo + (uint32_t)c0, lo);
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] += lo[j];
}

// 16 consecutive columns of a row to or from global memory (W columns live)
__device__ __forceinline__ void put16(float *dst, int c0, int W, const float (&v)[16]) {
  if ((W & 3) == 0 && c0 + 16 <= W) {
#pragma unroll
    for (int j = 0; j < 16; j += 4)
      *(float4 *)(dst + c0 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (c0 + j < W) dst[c0 + j] = v[j];
  }
}
__device__ __forceinline__ void get16(const float *src, int c0, int W, bool live, float (&v)[16]) {
  if (live && (W & 3) == 0 && c0 + 16 <= W) {
#pragma unroll
    for (int j = 0; j < 16; j += 4) {
      const float4 q = *(const float4 *)(src + c0 + j);
      v[j] = q.x;
      v[j + 1] = q.y;
      v[j + 2] = q.z;
      v[j + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = live && c0 + j < W ? src[c0 + j] : 0.f;
  }
}

// This thread's share of whether some unit has bit `what` of odd_w
__device__ __forceinline__ int odd_weight(const MlpTc &tc, int what) {
  return threadIdx.x < MW ? tc.odd_w[threadIdx.x] & what : 0;
}

// A forward CTA's rows on the CUDA cores, one row at a time (buf: 2 MW floats)
template <int PLANES, bool STORE>
__device__ __noinline__ void forward_rows(const MlpTc &tc, int64_t rows, int n_tiles,
                                          const float *F, float *H2, float *Y, const float *sw1,
                                          const float *sb1, const float *sb2, const float *sw3,
                                          float *buf) {
  const int n = threadIdx.x, W = tc.width, ni = tc.n_in;
  const float *w2 = tc.params + (int64_t)W * ni + W + (int64_t)n * W;
  for (int64_t t = blockIdx.x; t < n_tiles; t += gridDim.x)
    for (int64_t r = t * MT; r < min(rows, (t + 1) * MT); ++r) {
      if (n < W) {
        float s = 0.f;
        for (int i = 0; i < ni; ++i) s = fmaf(F[r * ni + i], sw1[n * kMlpMaxIn + i], s);
        buf[n] = tanhf(s + sb1[n]);
      }
      __syncthreads();
      if (n < W) {
        float s = 0.f;
        for (int k = 0; k < W; ++k)
          s = fmaf(buf[k], PLANES == 1 ? __bfloat162float(__float2bfloat16_rn(w2[k])) : w2[k], s);
        s = tanhf(s + sb2[n]);
        buf[MW + n] = s;
        if (STORE) H2[r * W + n] = s;
      }
      __syncthreads();
      if (n < tc.n_out) {
        float s = 0.f;
        for (int k = 0; k < W; ++k) s = fmaf(buf[MW + k], sw3[n * MW + k], s);
        Y[r * tc.n_out + n] = s + tc.vec[(2 + 2 * kMlpMaxOut) * MW + n];
      }
    }
}

constexpr size_t kFwdSmem = 1024 + 2 * kBufA + kRing * kTileB + MW * kMlpMaxIn * 4 + 2 * MW * 4 +
                            kMlpMaxOut * MW * 4 + 2 * 3 * MT * kMlpMaxOut * 4 + sizeof(Ctl) + 64;

// One CTA per SM walks 128-row tiles.  Over the sequence u of 64-unit chunks
// the epilogue warps form layer 1 and its planes while the MMA warp multiplies
// the chunk before, and they take the output of tile t after the first chunk
// of tile t + 1: the tanhf never wait for the tensor cores.
template <int PLANES, bool STORE>
__global__ void __launch_bounds__(kThreads, 1)
    mlp_forward_kernel(const __grid_constant__ CUtensorMap map2, MlpTc tc, int64_t rows,
                       const float *__restrict__ F, float *__restrict__ H1,
                       float *__restrict__ H2, float *__restrict__ Y, int *err) {
  extern __shared__ uint8_t smem_raw[];
  const uint64_t lim = wait_limit(err);   // (loaded ahead of their use)
  const int odd_w = odd_weight(tc, 1);
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *sA = smem, *ring = sA + 2 * kBufA;
  float *sw1 = (float *)(ring + kRing * kTileB), *sb1 = sw1 + MW * kMlpMaxIn, *sb2 = sb1 + MW,
        *sw3 = sb2 + MW, *sy = sw3 + kMlpMaxOut * MW;   // sy: [2][groups 1..3][MT][kMlpMaxOut]
  Ctl *ct = (Ctl *)(sy + 2 * 3 * MT * kMlpMaxOut);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int W = tc.width, nc = (W + 63) / 64;
  const int n_tiles = (int)((rows + MT - 1) / MT);
  if (threadIdx.x == 0) ctl_init(ct, 1);
  for (int i = threadIdx.x; i < MW; i += kThreads) {
    sb1[i] = tc.vec[i];
    sb2[i] = tc.vec[MW + i];
  }
  for (int i = threadIdx.x; i < MW * kMlpMaxIn; i += kThreads)
    sw1[i] = tc.w1[(PLANES == 1 ? MW * kMlpMaxIn : 0) + i];
  for (int i = threadIdx.x; i < kMlpMaxOut * MW; i += kThreads)
    sw3[i] = tc.vec[(2 + (PLANES == 1 ? kMlpMaxOut : 0)) * MW + i];
  const bool odd = __syncthreads_or(odd_w) != 0;
  const uint32_t tmem = tmem_open(ct, warp, lim);

  if (warp == 0) {
    ring_producer(ct, ring, &map2, n_tiles, nc, PLANES, err);
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t leader = elect_one();
    const uint32_t a_lo = desc_lo(smem_u32(sA)), ring_lo = desc_lo(smem_u32(ring));
    const int mine = (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    RingState rs;
    bool ok = true;
    for (int u = 0; u < mine * nc && ok; ++u) {
      const int lt = u / nc, c = u - lt * nc;
      ok = role_wait(&ct->afull[u & 1], (uint32_t)(u >> 1) & 1u, ct, err, 46) &&
           (c > 0 || lt == 0 || role_wait(&ct->d2empty, (uint32_t)(lt - 1) & 1u, ct, err, 47));
      if (!ok) break;
      fence_after();
      ok = chunk_mma<PLANES>(ct, leader, ring_lo, a_lo + (uint32_t)(u & 1) * (kBufA >> 4), tmem,
                             c == 0, rs, err);
      if (!ok) break;
      mma_commit_if(leader, &ct->aempty[u & 1]);
      if (c == nc - 1) mma_commit_if(leader, &ct->d2full);
    }
    mma_commit_if(leader, &ct->drain);
    mbar_wait(&ct->drain, 0u);
    __syncwarp();
  } else {
    // epilogue warp: lane quadrant q (rows 32 q + lane), unit group g
    const int q = warp & 3, g = (warp - 2) >> 2, lr = 32 * q + lane;
    const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16);
    float fx[kMlpMaxIn], fn[kMlpMaxIn];   // this tile's and the next tile's features
    auto load_f = [&](int64_t t) {
      const int64_t r = t * MT + lr;
#pragma unroll
      for (int i = 0; i < kMlpMaxIn; ++i)
        fn[i] = (r < rows && i < tc.n_in) ? F[r * tc.n_in + i] : 0.f;
    };
    // output of local tile lt (global tile t): layer 2's tanh, then the output layer
    auto output = [&](int lt, int64_t t) -> bool {
      if (!role_wait(&ct->d2full, (uint32_t)lt & 1u, ct, err, 48)) return false;
      fence_after();
      const int64_t r = t * MT + lr;
      float y[kMlpMaxOut] = {};
#pragma unroll 1
      for (int s = 0; s < 4; ++s) {
        const int c0 = 64 * g + 16 * s;
        if (c0 >= W) break;
        float v[16];
        get_sum(trow, c0, v);
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = tanhf(v[j] + sb2[c0 + j]);
        if (STORE && r < rows) put16(H2 + r * W, c0, W, v);
#pragma unroll
        for (int o = 0; o < kMlpMaxOut; ++o)
          if (o < tc.n_out) {
#pragma unroll
            for (int j = 0; j < 16; ++j) y[o] = fmaf(v[j], sw3[o * MW + c0 + j], y[o]);
          }
      }
      fence_before();
      warp_arrive(&ct->d2empty);
      float *yb = sy + ((lt & 1) * 3) * MT * kMlpMaxOut + lr * kMlpMaxOut;
      if (g > 0) {
#pragma unroll
        for (int o = 0; o < kMlpMaxOut; ++o) yb[(g - 1) * MT * kMlpMaxOut + o] = y[o];
      }
      warp_arrive(&ct->yfull[lt & 1]);
      if (g == 0) {
        if (!role_wait(&ct->yfull[lt & 1], (uint32_t)(lt >> 1) & 1u, ct, err, 49)) return false;
#pragma unroll
        for (int o = 0; o < kMlpMaxOut; ++o)
          if (o < tc.n_out && r < rows) {
            float s = y[o];
            for (int k = 0; k < 3; ++k) s += yb[k * MT * kMlpMaxOut + o];
            Y[r * tc.n_out + o] = s + tc.vec[(2 + 2 * kMlpMaxOut) * MW + o];
          }
      }
      return true;
    };
    int lt = 0;
    bool ok = true;
    load_f(blockIdx.x);
    for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++lt) {
#pragma unroll
      for (int i = 0; i < kMlpMaxIn; ++i) fx[i] = fn[i];
      load_f(t + gridDim.x);
      for (int c = 0; c < nc; ++c) {
        const int u = lt * nc + c, c0 = 64 * c + 16 * g;
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float4 *w = (const float4 *)(sw1 + (c0 + j) * kMlpMaxIn);
          float s = 0.f;
#pragma unroll
          for (int i = 0; i < kMlpMaxIn; i += 4) {
            const float4 x = w[i / 4];
            s = fmaf(fx[i], x.x, s);
            s = fmaf(fx[i + 1], x.y, s);
            s = fmaf(fx[i + 2], x.z, s);
            s = fmaf(fx[i + 3], x.w, s);
          }
          v[j] = tanhf(s + sb1[c0 + j]);
        }
        if (c0 + 16 > W) {   // padded units are zero also for infinite features
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c0 + j >= W) v[j] = 0.f;
        }
        const int64_t r = t * MT + lr;
        if (STORE && r < rows) put16(H1 + r * W, c0, W, v);
        // the buffer's previous planes (chunk u - 2) have been read
        if (u > 1 && !(ok = role_wait(&ct->aempty[u & 1], (uint32_t)((u >> 1) - 1) & 1u, ct, err, 52)))
          break;
        put_planes(sA + (u & 1) * kBufA, lr, g, v);
        warp_arrive(&ct->afull[u & 1]);
        if (c == 0 && lt > 0 && !(ok = output(lt - 1, t - gridDim.x))) break;
      }
    }
    if (ok && lt > 0) output(lt - 1, (int64_t)blockIdx.x + (int64_t)(lt - 1) * gridDim.x);
  }
  tmem_close(tmem, warp);
  if (*(volatile int *)&ct->abort_flag) {
    // (all roles have ended) nothing of this CTA passes for an output
    for (int64_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
      const int64_t y0 = t * MT * tc.n_out, y1 = min(rows, (t + 1) * MT) * tc.n_out;
      for (int64_t i = y0 + threadIdx.x; i < y1; i += kThreads) Y[i] = __int_as_float(0x7FC00000);
    }
  } else if (odd) {
    forward_rows<PLANES, STORE>(tc, rows, n_tiles, F, H2, Y, sw1, sb1, sb2, sw3, (float *)sA);
  }
}

// A dH1 CTA's rows on the CUDA cores, one row at a time (buf: MW floats)
__device__ __noinline__ void dh1_rows(const MlpTc &tc, int64_t rows, int n_tiles, const float *dY,
                                      const float *H1, const float *H2, float *dH1, float *buf) {
  const int n = threadIdx.x, W = tc.width, no = tc.n_out;
  const float *w2 = tc.params + (int64_t)W * tc.n_in + W, *w3 = tc.vec + 2 * MW;
  for (int64_t t = blockIdx.x; t < n_tiles; t += gridDim.x)
    for (int64_t r = t * MT; r < min(rows, (t + 1) * MT); ++r) {
      if (n < W) {
        float s = 0.f;
        for (int o = 0; o < no; ++o) s = fmaf(dY[r * no + o], w3[o * MW + n], s);
        buf[n] = dh2_of(s, H2[r * W + n]);
      }
      __syncthreads();
      if (n < W) {
        const float h = H1[r * W + n];
        float s = 0.f;
        for (int i = 0; i < W; ++i) s = fmaf(buf[i], w2[(int64_t)i * W + n], s);
        dH1[r * W + n] = s * fmaf(-h, h, 1.f);
      }
      __syncthreads();
    }
}

constexpr size_t kDh1Smem =
    1024 + 2 * kBufA + kRing * kTileB + kMlpMaxOut * MW * 4 + sizeof(Ctl) + 64;

// dH1 of 128-row tiles, scheduled as the forward pass: each chunk's dH2 goes
// from registers into the A planes; the next chunk's H2 is loaded ahead.
__global__ void __launch_bounds__(kThreads, 1)
    mlp_dh1_kernel(const __grid_constant__ CUtensorMap map2t, MlpTc tc, int64_t rows,
                   const float *__restrict__ dY, const float *__restrict__ H1,
                   const float *__restrict__ H2, float *__restrict__ dH1, int *err) {
  extern __shared__ uint8_t smem_raw[];
  const uint64_t lim = wait_limit(err);
  const int odd_w = odd_weight(tc, 1);
  uint8_t *sA = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *ring = sA + 2 * kBufA;
  float *sw3 = (float *)(ring + kRing * kTileB);
  Ctl *ct = (Ctl *)(sw3 + kMlpMaxOut * MW);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int W = tc.width, nc = (W + 63) / 64, no = tc.n_out;
  const int n_tiles = (int)((rows + MT - 1) / MT);
  if (threadIdx.x == 0) ctl_init(ct, 1);
  for (int i = threadIdx.x; i < kMlpMaxOut * MW; i += kThreads)
    sw3[i] = tc.vec[2 * MW + i];
  const bool odd_w2 = __syncthreads_or(odd_w) != 0;
  const uint32_t tmem = tmem_open(ct, warp, lim);
  if (warp == 0) {
    ring_producer(ct, ring, &map2t, n_tiles, nc, 3, err);
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t leader = elect_one();
    const uint32_t a_lo = desc_lo(smem_u32(sA)), ring_lo = desc_lo(smem_u32(ring));
    const int mine = (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    RingState rs;
    bool ok = true;
    for (int u = 0; u < mine * nc && ok; ++u) {
      const int lt = u / nc, c = u - lt * nc;
      ok = role_wait(&ct->afull[u & 1], (uint32_t)(u >> 1) & 1u, ct, err, 61) &&
           (c > 0 || lt == 0 || role_wait(&ct->d2empty, (uint32_t)(lt - 1) & 1u, ct, err, 62));
      if (!ok) break;
      fence_after();
      ok = chunk_mma<3>(ct, leader, ring_lo, a_lo + (uint32_t)(u & 1) * (kBufA >> 4), tmem, c == 0,
                        rs, err);
      if (!ok) break;
      mma_commit_if(leader, &ct->aempty[u & 1]);
      if (c == nc - 1) mma_commit_if(leader, &ct->d2full);
    }
    mma_commit_if(leader, &ct->drain);
    mbar_wait(&ct->drain, 0u);
    __syncwarp();
  } else {
    const int q = warp & 3, g = (warp - 2) >> 2, lr = 32 * q + lane;
    const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16);
    auto output = [&](int lt, int64_t t) -> bool {
      const int64_t r = t * MT + lr;
      float hn[16];
      get16(H1 + r * W, 64 * g, W, r < rows, hn);
      if (!role_wait(&ct->d2full, (uint32_t)lt & 1u, ct, err, 63)) return false;
      fence_after();
#pragma unroll 1
      for (int s = 0; s < 4; ++s) {
        const int c0 = 64 * g + 16 * s;
        if (c0 >= W) break;
        float h[16], v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) h[j] = hn[j];
        if (s < 3) get16(H1 + r * W, c0 + 16, W, r < rows, hn);
        get_sum(trow, c0, v);
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = v[j] * kDh2Unscale * fmaf(-h[j], h[j], 1.f);
        if (r < rows) put16(dH1 + r * W, c0, W, v);
      }
      fence_before();
      warp_arrive(&ct->d2empty);
      return true;
    };
    int lt = 0;
    bool ok = true;
    float hn[16];
    get16(H2 + ((int64_t)blockIdx.x * MT + lr) * W, 16 * g, W,
          (int64_t)blockIdx.x * MT + lr < rows, hn);
    for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++lt) {
      const int64_t r = t * MT + lr;
      float dy[kMlpMaxOut];
#pragma unroll
      for (int o = 0; o < kMlpMaxOut; ++o) dy[o] = r < rows && o < no ? dY[r * no + o] : 0.f;
      for (int c = 0; c < nc; ++c) {
        const int u = lt * nc + c, c0 = 64 * c + 16 * g;
        float h[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) h[j] = hn[j];
        {
          const int64_t rn = c + 1 < nc ? r : r + (int64_t)gridDim.x * MT;
          get16(H2 + rn * W, c + 1 < nc ? c0 + 64 : 16 * g, W, rn < rows, hn);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          float s = 0.f;
#pragma unroll
          for (int o = 0; o < kMlpMaxOut; ++o)
            if (o < no) s = fmaf(dy[o], sw3[o * MW + c0 + j], s);
          h[j] = dh2_scaled(s, h[j]);
        }
        if (drop_odd(h)) *(volatile int *)&ct->odd = 1;
        if (u > 1 && !(ok = role_wait(&ct->aempty[u & 1], (uint32_t)((u >> 1) - 1) & 1u, ct, err, 64)))
          break;
        put_planes(sA + (u & 1) * kBufA, lr, g, h);
        warp_arrive(&ct->afull[u & 1]);
        if (c == 0 && lt > 0 && !(ok = output(lt - 1, t - gridDim.x))) break;
      }
    }
    if (ok && lt > 0) output(lt - 1, (int64_t)blockIdx.x + (int64_t)(lt - 1) * gridDim.x);
  }
  tmem_close(tmem, warp);
  if ((odd_w2 || *(volatile int *)&ct->odd) && !*(volatile int *)&ct->abort_flag)
    dh1_rows(tc, rows, n_tiles, dY, H1, H2, dH1, (float *)sA);
}

// dW2 over a CTA's rows: D[i][j] += sum_r dH2[r][i] H1[r][j] for the 256 units
// i and half of the units j (CTA pairs share the rows, so that the leading
// and the small products each have an accumulator).  Both operands are
// transposed on the way into shared memory: a thread owns one unit (lane =
// column, coalesced reads) and eight (dH2) or four (H1) rows, a 16- or 8-byte
// piece of its unit's K-major, 128-byte swizzled row.  The four 16-row K steps
// of the 64-deep tile are the ring's slots.  Every kDwDrain K steps the
// accumulators are added to the CTA's float32 partial sums in global memory,
// which bounds the truncations.  The same threads sum db2 and dW3 of their
// unit (and db3).
// (Products and sums without planes follow at the end, row by row.)
constexpr int kDwRows = 16, kDwDrain = 24;
constexpr uint32_t kDwA = MW * 128, kDwB = (MW / 2) * 128;   // planes of 256 and 128 units
constexpr size_t kDw2Smem = 1024 + 3 * (kDwA + kDwB) + sizeof(Ctl) + 64;

// The entries of dH2 that the planes left out, into dW2 and db2: thread i adds
// unit i's, which no other thread touches.
__device__ __noinline__ void dw2_odd(const MlpTc &tc, int64_t rows, int64_t b0, int64_t step,
                                     int n_mine, int half, const float *dY, const float *H1,
                                     const float *H2, float *pw) {
  const int i = threadIdx.x, W = tc.width, no = tc.n_out;
  if (i >= W) return;
  const float *w3 = tc.vec + 2 * MW + i;
  const bool all = (tc.odd_w[i] & 2) != 0;
  const int j0 = half * (MW / 2), j1 = min(W, j0 + MW / 2);
  for (int g = 0; g < n_mine; ++g) {
    const int64_t ra = (b0 + g * step) * kDwRows;
    for (int64_t r = ra; r < min(rows, ra + kDwRows); ++r) {
      float t = 0.f;
      for (int o = 0; o < no; ++o) t = fmaf(dY[r * no + o], w3[o * MW], t);
      const float h = H2[r * W + i], d = dh2_of(t, h);
      if (!all && !(fabsf(dh2_scaled(t, h)) > kDh2Max)) continue;
      for (int j = j0; j < j1; ++j) pw[i * MW + j] = fmaf(d, H1[r * W + j], pw[i * MW + j]);
      if (half == 0) pw[MW * MW + i] += d;   // db2, of the first row group
    }
  }
}

__global__ void __launch_bounds__(kThreads, 1)
    mlp_dw2_kernel(MlpTc tc, int64_t rows, const float *__restrict__ dY,
                   const float *__restrict__ H1, const float *__restrict__ H2,
                   float *__restrict__ part, int *err) {
  extern __shared__ uint8_t smem_raw[];
  const uint64_t lim = wait_limit(err);
  const int odd_w3 = odd_weight(tc, 2);
  uint8_t *sa = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *sb = sa + 3 * kDwA;
  Ctl *ct = (Ctl *)(sb + 3 * kDwB);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int W = tc.width, no = tc.n_out;
  const int half = blockIdx.x & 1;
  const int64_t n_blk = (rows + kDwRows - 1) / kDwRows, step = gridDim.x >> 1,
                b0 = blockIdx.x >> 1;
  const int n_mine = (int)((n_blk - b0 + step - 1) / step);   // >= 1
  if (threadIdx.x == 0) ctl_init(ct, kEpiWarps);
  const uint32_t tmem = tmem_open(ct, warp, lim);
  if (odd_w3) *(volatile int *)&ct->odd = 1;
  float *pw = part + b0 * tc.part_stride;
  if (warp == 1) {
    constexpr uint32_t idesc = idesc_bf16(MT, MW / 2);
    const uint32_t leader = elect_one(), a_lo = desc_lo(smem_u32(sa)), b_lo = desc_lo(smem_u32(sb));
    bool ok = true;
    for (int g = 0; g < n_mine && ok; ++g) {
      const int s = g % kRingMax, in_group = g % kDwDrain;
      if (!(ok = role_wait(&ct->full[s], (uint32_t)(g / kRingMax) & 1u, ct, err, 71))) break;
      if (in_group == 0 && g > 0 &&
          !(ok = role_wait(&ct->d2empty, (uint32_t)(g / kDwDrain - 1) & 1u, ct, err, 74)))
        break;
      fence_after();
#pragma unroll
      for (int w = 0; w < 3; ++w)
#pragma unroll
        for (int a = 0; a < 3 - w; ++a)
#pragma unroll
          for (int m = 0; m < 2; ++m)
            mma_bf16_if(leader, tmem + (w + a == 0 ? kTHi : kTLo) + (uint32_t)(m * (MW / 2)),
                        desc_of(a_lo + (uint32_t)((a * kDwA + m * MT * 128) >> 4) + 2 * s),
                        desc_of(b_lo + (uint32_t)((w * kDwB) >> 4) + 2 * s), idesc,
                        (in_group == 0 && w == 0 && a <= 1) ? 0u : 1u);
      mma_commit_if(leader, &ct->empty[s]);
      if (in_group == kDwDrain - 1 || g == n_mine - 1) mma_commit_if(leader, &ct->d2full);
    }
    mma_commit_if(leader, &ct->drain);
    mbar_wait(&ct->drain, 0u);
    __syncwarp();
  } else if (warp >= 2) {
    const int et = (int)threadIdx.x - 64;
    const int i = et & (MW - 1), grp = et >> 8;                    // dH2: unit i, rows 8 grp ..
    const int jl = et & (MW / 2 - 1), quad = et >> 7;              // H1: unit j, rows 4 quad ..
    const int j = half * (MW / 2) + jl;
    float w3[kMlpMaxOut], g3[kMlpMaxOut] = {}, gb2 = 0.f, gb3 = 0.f;
#pragma unroll
    for (int o = 0; o < kMlpMaxOut; ++o) w3[o] = tc.w3_dw2[o * MW + i];
    float n2[8], n1[4], ndy;   // the next block's values; lane l: dY entry l of the 8 rows
    auto load = [&](int g) {
      const int64_t ra = (b0 + g * step) * kDwRows;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int64_t r = ra + 8 * grp + e;
        n2[e] = i < W && r < rows ? H2[r * W + i] : 0.f;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int64_t r = ra + 4 * quad + e;
        n1[e] = j < W && r < rows ? H1[r * W + j] : 0.f;
      }
      const int64_t at = (ra + 8 * grp) * no + lane;
      ndy = lane < 8 * no && at < rows * no ? dY[at] : 0.f;
    };
    // adds the accumulators of drain group k to this CTA's partial sums
    auto drain = [&](int k) -> bool {
      if (!role_wait(&ct->d2full, (uint32_t)k & 1u, ct, err, 73)) return false;
      fence_after();
      const int q = warp & 3, cg = (warp - 2) >> 2;
#pragma unroll 1
      for (int ms = 0; ms < 4; ++ms) {   // M half, 16-column piece
        const int m = ms >> 1, c0 = 32 * cg + 16 * (ms & 1);
        float v[16], old[16];
        float *dst = pw + (int64_t)(m * MT + 32 * q + lane) * MW + half * (MW / 2);
        get16(dst, c0, MW, k > 0, old);
        get_sum(tmem + ((uint32_t)(32 * q) << 16), m * (MW / 2) + c0, v);
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = fmaf(v[e], kDh2Unscale, old[e]);
        put16(dst, c0, MW, v);
      }
      fence_before();
      warp_arrive(&ct->d2empty);
      return true;
    };
    bool ok = true;
    load(0);
    for (int g = 0; g < n_mine && ok; ++g) {
      const int s = g % kRingMax;
      float h1[4], h2[8], d2[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) h2[e] = n2[e];
#pragma unroll
      for (int e = 0; e < 4; ++e) h1[e] = n1[e];
      const float dyl = ndy;
      if (g + 1 < n_mine) load(g + 1);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float t = 0.f;
#pragma unroll
        for (int o = 0; o < kMlpMaxOut; ++o)
          if (o < no) {
            const float dy = __shfl_sync(0xffffffffu, dyl, e * no + o);
            t = fmaf(dy, w3[o], t);
            g3[o] = fmaf(dy, h2[e], g3[o]);
            if (i == o) gb3 += dy;
          }
        d2[e] = dh2_scaled(t, h2[e]);
      }
      if (drop_odd(d2)) *(volatile int *)&ct->odd = 1;
#pragma unroll
      for (int e = 0; e < 8; ++e) gb2 = fmaf(d2[e], kDh2Unscale, gb2);
      if (g >= kRingMax &&
          !(ok = role_wait(&ct->empty[s], (uint32_t)(g / kRingMax - 1) & 1u, ct, err, 72)))
        break;
      uint32_t wa[3][4], wb[3][2];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        uint32_t x[3];
        split3_pair(d2[2 * e], d2[2 * e + 1], x);
#pragma unroll
        for (int p = 0; p < 3; ++p) wa[p][e] = x[p];
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        uint32_t x[3];
        split3_pair(h1[2 * e], h1[2 * e + 1], x);
#pragma unroll
        for (int p = 0; p < 3; ++p) wb[p][e] = x[p];
      }
      uint8_t *at = sa + i * 128 + (((2 * s + grp) ^ (i & 7)) << 4);
      uint8_t *bt = sb + jl * 128 + (((2 * s + (quad >> 1)) ^ (jl & 7)) << 4) + (quad & 1) * 8;
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        *(uint4 *)(at + p * kDwA) = make_uint4(wa[p][0], wa[p][1], wa[p][2], wa[p][3]);
        *(uint2 *)(bt + p * kDwB) = make_uint2(wb[p][0], wb[p][1]);
      }
      fence_async_smem();
      warp_arrive(&ct->full[s]);
      if ((g % kDwDrain == kDwDrain - 1 || g == n_mine - 1) && !(ok = drain(g / kDwDrain))) break;
    }
    if (half == 0) {
      // [grp] rows of db2, dW3 and db3 per unit
      float *ps = pw + (int64_t)MW * MW + grp * (1 + 2 * kMlpMaxOut) * MW;
      ps[i] = gb2;
#pragma unroll
      for (int o = 0; o < kMlpMaxOut; ++o) ps[(1 + o) * MW + i] = g3[o];
      if (i < kMlpMaxOut) ps[(1 + kMlpMaxOut) * MW + i] = gb3;
    }
  }
  tmem_close(tmem, warp);
  if (*(volatile int *)&ct->odd && !*(volatile int *)&ct->abort_flag)
    dw2_odd(tc, rows, b0, step, n_mine, half, dY, H1, H2, pw);
}

// dW1[j][f] = sum_r dH1[r][j] F[r][f] and db1[j]: thread j, rows in blocks of
// 64 whose features are staged in shared memory.
constexpr int kDw1Rows = 64;
__global__ void __launch_bounds__(MW) mlp_dw1_kernel(MlpTc tc, int64_t rows,
                                                     const float *__restrict__ F,
                                                     const float *__restrict__ dH1,
                                                     float *__restrict__ part) {
  __shared__ __align__(16) float sf[kDw1Rows][kMlpMaxIn];
  const int j = threadIdx.x, W = tc.width, ni = tc.n_in;
  float acc[kMlpMaxIn] = {}, b1 = 0.f;
  for (int64_t r0 = (int64_t)blockIdx.x * kDw1Rows; r0 < rows;
       r0 += (int64_t)gridDim.x * kDw1Rows) {
    __syncthreads();
    for (int i = j; i < kDw1Rows * kMlpMaxIn; i += MW) {
      const int r = i / kMlpMaxIn, f = i % kMlpMaxIn;
      sf[r][f] = (r0 + r < rows && f < ni) ? F[(r0 + r) * ni + f] : 0.f;
    }
    __syncthreads();
    if (j >= W) continue;
    const int n = (int)min((int64_t)kDw1Rows, rows - r0);
#pragma unroll 8
    for (int r = 0; r < n; ++r) {
      const float d = dH1[(r0 + r) * W + j];
      b1 += d;
#pragma unroll
      for (int f = 0; f < kMlpMaxIn; f += 4) {
        if (f >= ni) break;
        const float4 x = *(const float4 *)&sf[r][f];
        acc[f] = fmaf(d, x.x, acc[f]);
        acc[f + 1] = fmaf(d, x.y, acc[f + 1]);
        acc[f + 2] = fmaf(d, x.z, acc[f + 2]);
        acc[f + 3] = fmaf(d, x.w, acc[f + 3]);
      }
    }
  }
  float *p = part + (int64_t)blockIdx.x * (kMlpMaxIn + 1) * MW;
#pragma unroll
  for (int f = 0; f < kMlpMaxIn; ++f) p[f * MW + j] = acc[f];
  p[kMlpMaxIn * MW + j] = b1;
}

// grad = the CTAs' partial sums (deterministic): 32 parameters per block, each
// by 8 threads that take every 8th partial, added in order.
__global__ void __launch_bounds__(256) mlp_reduce_kernel(MlpTc tc, int n2,
                                                         const float *__restrict__ part2, int n1,
                                                         const float *__restrict__ part1,
                                                         float *__restrict__ grad) {
  __shared__ float red[8][32];
  const int W = tc.width, ni = tc.n_in, no = tc.n_out;
  const int64_t oB1 = (int64_t)W * ni, oW2 = oB1 + W, oB2 = oW2 + (int64_t)W * W, oW3 = oB2 + W,
                oB3 = oW3 + (int64_t)no * W, n = oB3 + no;
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * 32 + lane;
  float s = 0.f;
  if (i < n) {
    const float *src;
    int64_t stride = tc.part_stride, second = 0;   // second: the other row group's sums
    int cnt = n2;
    const int64_t side = (int64_t)MW * MW, grp = (1 + 2 * kMlpMaxOut) * MW;
    if (i < oW2) {
      stride = (kMlpMaxIn + 1) * MW;
      cnt = n1;
      src = i < oB1 ? part1 + (i % ni) * MW + i / ni : part1 + kMlpMaxIn * MW + (i - oB1);
    } else if (i < oB2) {
      const int64_t e = i - oW2;
      src = part2 + (e / W) * MW + e % W;
    } else {
      second = grp;
      if (i < oW3) {
        src = part2 + side + (i - oB2);
      } else if (i < oB3) {
        const int64_t e = i - oW3;
        src = part2 + side + (1 + e / W) * MW + e % W;
      } else {
        src = part2 + side + (1 + kMlpMaxOut) * MW + (i - oB3);
      }
    }
#pragma unroll 8
    for (int c = slice; c < cnt; c += 8) {
      s += src[c * stride];
      if (second) s += src[c * stride + second];
    }
  }
  red[slice][lane] = s;
  __syncthreads();
  if (slice == 0 && i < n) {
    for (int k = 1; k < 8; ++k) s += red[k][lane];
    grad[i] = s;
  }
}

template <class K>
cudaError_t allow_smem(K k, size_t bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int PLANES, bool STORE>
cudaError_t launch_forward(cudaStream_t st, const MlpTc &tc, int64_t rows, const float *F,
                           float *H1, float *H2, float *Y) {
  const cudaError_t e = allow_smem(mlp_forward_kernel<PLANES, STORE>, kFwdSmem);
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<int64_t>((rows + MT - 1) / MT, sm_count());
  mlp_forward_kernel<PLANES, STORE><<<grid, kThreads, kFwdSmem, st>>>(tc.map2, tc, rows, F, H1, H2,
                                                                      Y, tc.err);
  return cudaGetLastError();
}

// row groups of the dW2 kernel (two CTAs each) and CTAs of the dW1 kernel
int dw2_groups(int64_t rows) {
  return (int)std::min<int64_t>((rows + kDwRows - 1) / kDwRows, std::max(1, sm_count() / 2));
}
int dw1_ctas(int64_t rows) {
  return (int)std::min<int64_t>((rows + kDw1Rows - 1) / kDw1Rows, 4 * (int64_t)sm_count());
}
constexpr int64_t kPartStride = (int64_t)MW * MW + 2 * (1 + 2 * kMlpMaxOut) * MW;
}  // namespace

bool mlp_tc_fits(int n_in, int width, int n_out) {
  return n_in <= kMlpMaxIn && width <= kMlpMaxWidth && n_out <= kMlpMaxOut;
}

size_t mlp_tc_bytes(int64_t max_rows) {
  return (size_t)6 * MW * MW * sizeof(__nv_bfloat16) +
         (size_t)(2 * kMlpMaxIn + 4 + 3 * kMlpMaxOut) * MW * sizeof(float) + 256 +
         (size_t)(dw2_groups(max_rows) * kPartStride +
                  (int64_t)dw1_ctas(max_rows) * (kMlpMaxIn + 1) * MW) * sizeof(float);
}

cudaError_t mlp_tc_init(MlpTc &tc, int n_in, int width, int n_out, int64_t max_rows,
                        const float *params, void *mem, cudaStream_t st) {
  tc.params = params;
  tc.n_in = n_in;
  tc.width = width;
  tc.n_out = n_out;
  tc.part_stride = kPartStride;
  tc.w2 = (__nv_bfloat16 *)mem;
  tc.w2t = tc.w2 + 3 * MW * MW;
  tc.w1 = (float *)(tc.w2t + 3 * MW * MW);
  tc.vec = tc.w1 + 2 * MW * kMlpMaxIn;
  tc.w3_dw2 = tc.vec + (3 + 2 * kMlpMaxOut) * MW;
  tc.odd_w = (int *)(tc.w3_dw2 + kMlpMaxOut * MW);
  tc.err = tc.odd_w + MW;
  tc.part2 = (float *)((char *)tc.err + 256);
  tc.part1 = tc.part2 + dw2_groups(max_rows) * kPartStride;
  cudaError_t e = encode_bf16_map(&tc.map2, tc.w2, 3 * MW, MW, MW);
  if (e == cudaSuccess) e = encode_bf16_map(&tc.map2t, tc.w2t, 3 * MW, MW, MW);
  if (e == cudaSuccess) e = cudaMemsetAsync(tc.err, 0, 256, st);
  return e;
}

cudaError_t mlp_tc_forward(cudaStream_t st, const MlpTc &tc, int64_t rows, const float *F,
                           float *H1, float *H2, float *Y, bool bf16) {
  mlp_prepare_kernel<<<MW, MW, 0, st>>>(tc);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (bf16) return launch_forward<1, false>(st, tc, rows, F, nullptr, nullptr, Y);
  return H1 ? launch_forward<3, true>(st, tc, rows, F, H1, H2, Y)
            : launch_forward<3, false>(st, tc, rows, F, nullptr, nullptr, Y);
}

cudaError_t mlp_tc_backward(cudaStream_t st, const MlpTc &tc, int64_t rows, const float *F,
                            const float *dY, const float *H1, const float *H2, float *dH1,
                            float *grad) {
  cudaError_t e = allow_smem(mlp_dh1_kernel, kDh1Smem);
  if (e == cudaSuccess) e = allow_smem(mlp_dw2_kernel, kDw2Smem);
  if (e != cudaSuccess) return e;
  const int g1 = (int)std::min<int64_t>((rows + MT - 1) / MT, sm_count());
  const int n2 = dw2_groups(rows), n1 = dw1_ctas(rows);
  mlp_dh1_kernel<<<g1, kThreads, kDh1Smem, st>>>(tc.map2t, tc, rows, dY, H1, H2, dH1, tc.err);
  mlp_dw2_kernel<<<2 * n2, kThreads, kDw2Smem, st>>>(tc, rows, dY, H1, H2, tc.part2, tc.err);
  mlp_dw1_kernel<<<n1, MW, 0, st>>>(tc, rows, F, dH1, tc.part1);
  const int64_t n = (int64_t)tc.width * tc.n_in + tc.width + (int64_t)tc.width * tc.width +
                    tc.width + (int64_t)tc.n_out * tc.width + tc.n_out;
  mlp_reduce_kernel<<<(unsigned)((n + 31) / 32), 256, 0, st>>>(tc, n2, tc.part2, n1, tc.part1,
                                                               grad);
  return cudaGetLastError();
}

}  // namespace tddft

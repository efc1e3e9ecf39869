// Float64 matrix products emulated on the bf16 tensor cores (sm_103a,
// tcgen05 + TMA + mbarrier, inline PTX) by error-free splitting of both
// operands into integer slices (the Ozaki scheme).
//
// Every row of an operand is scaled by a power of two 2^e (|x| < 2^e over the
// row) and cut into s integer slices,
//     x = 2^e sum_{i=1..s} q_i 2^(-7 i),   q_1 in [-128, 128], q_i in [-64, 64],
// each q_i an exact bf16.  The product of two rows is then
//     2^(eA+eB) sum_t 2^(-7 t) G_t,        G_t = sum_{i+j=t} sum_k qA_i qB_j ,
// kept for t <= s+1 (pairs below the last slice's weight are dropped).  The
// t-1 pairs of a group contribute at most 2^12 (s+2) per k, so over a K chunk
// of L <= 2^12 / (s+2) entries every partial sum of G_t is an integer of at
// most 2^24 and the float32 accumulation in tensor memory is exact.  The
// epilogue warps read each G_t of a chunk, convert it to an integer and add
// it, shifted to its weight, into one 64-bit integer accumulator per output;
// u = max(0, 7s - 35) low bits are dropped so that the accumulator stays below
// 2^63 over up to 1024 chunks.  The float64 result is 2^(eA+eB+u-7(s+1)) acc,
// with an error of about (1 + (s+1)/4) 2^(-7s) 2^(eA+eB) K at most (2^-42
// relative for s = 6).
//
// One CTA computes a 128 x BN output tile (BN 64, 80 or 96):
//   warp 0     TMA producer: per 64-deep K block, the s slices of the A tile
//              (16 KB each, a ring of 6 to 9) and of the B tile (8 to 12 KB
//              each, side by side, two K blocks); 128-byte swizzle
//   warp 1     tcgen05.mma issuer (M = 128, K = 16).  The pairs of slice A_i
//              with neighbouring B slices are one MMA of up to 256 columns:
//              the B slices are rows of one operand, their groups i + j
//              neighbouring columns of tensor memory (s groups x BN columns).
//              Pair by pair (N = BN) every MMA read its A tile for 64 to 96
//              columns and took 55 to 66 clocks against 32 to 48 at the
//              tensor core's rate; 64-atom operator, products 1447 -> 1150 us.
//   warps 2-9  epilogue (two warps per TMEM lane quadrant, half of the columns
//              each): per chunk, TMEM -> registers -> int64 accumulators, a
//              phase's groups while the issuer is at the next one's; at the end
//              the float64 tile is stored (C or C^T)
// The issuer's waits and commits cost as much as its MMAs: one barrier per phase
// of B slices and one release per K block (12 + 12 a block -> 8 + 7: 1.98 ->
// 1.78 us per block of 6 slices, N = 64).
// Every mbarrier wait is bounded; on expiry the CTA records an error code,
// stops issuing work, waits (bounded) for its TMA copies in flight and still
// frees its TMEM.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "tc_ptx.h"

namespace cg = cooperative_groups;

namespace tddft {
namespace {
using namespace ptx;

constexpr int OZ_BM = 128, OZ_BN = 64, OZ_BK = 64;
constexpr int OZ_EPI_WARPS = 8;                        // 2 per TMEM lane quadrant
constexpr int OZ_THREADS = 64 + 32 * OZ_EPI_WARPS;      // producer, MMA, epilogue
constexpr uint32_t OZ_A_BYTES = OZ_BM * OZ_BK * 2;   // 16 KB
// The N tile is 64 columns or the widest of 96 and 80 whose s groups fit in
// tensor memory (s x BN <= 512), chosen per launch (tile_plan): a wide tile
// reads fewer operand bytes per column, a narrow one pads less.  Shared memory
// holds the B slices of two K blocks and as many A slices as fit.
template <int S, int BN> struct OzShape {
  static constexpr int EPI_COLS = BN / 2;                      // columns per epilogue thread
  static constexpr uint32_t B_BYTES = BN * OZ_BK * 2;
  static constexpr uint32_t A_OFF = 2 * S * B_BYTES;           // after two K blocks of B
  static constexpr int AS_FIT = (int)((227 * 1024 - 1024 - 1024 - A_OFF) / OZ_A_BYTES);
  static constexpr int AS = AS_FIT < 9 ? AS_FIT : 9;           // A slices
  static constexpr size_t SMEM = A_OFF + (size_t)AS * OZ_A_BYTES + 1024 + 512;
  // groups that one MMA takes, and the phases of a K block (see the issuer)
  static constexpr int W = 256 / BN < S ? 256 / BN : S, NP = (S + W - 1) / W;
  __host__ __device__ static constexpr int gh(int p) { return S - 1 - (NP - 1 - p) * W; }   // last group of phase p
  __host__ __device__ static constexpr int gl(int p) { return p == 0 ? 0 : gh(p - 1) + 1; }
  // A slices held while a phase before the last runs; the last one frees them
  static_assert(NP < 2 || AS > S - 1 - W, "A ring too short");
};
__host__ __device__ constexpr int oz_wide_bn(int S) {
  return S * 96 <= 512 ? 96 : (S * 80 <= 512 ? 80 : 64);
}

struct OzArgs {
  int M, N;
  int KpA, KpB; // slice-plane widths of the two operands
  int ns;       // slices (the kernel's template argument)
  int cb;       // K blocks per exact chunk
  const int *eA, *eB;
  OzEpilogue ep;
  int vec;      // kOzC with 16-byte aligned rows: double2 stores
  const GTile *tiles;   // grouped product: one entry per M tile (NULL: plain row tiles)
  int mgroup;           // M tiles per group of the L2-aware tile order
  int Mt, Nt;           // M tiles (rows / 128, or table entries) and N tiles
  int drop;             // low bits dropped from the integer accumulators (drop_bits)
  int ksplit;           // > 1: a cluster of ksplit CTAs per tile, each a share of its K chunks
  int *err;
  const int *dcnt;
  int mul_n;
};

// Low bits dropped from the integer accumulator for S slices: with u(S) the
// largest value, 2^(24 + 7(S-1) - u) summed over up to 1024 chunks (and the
// lower groups, < 1% more) stays below 2^63.  With 8 slices the drop's own
// rounding would exceed the slices' error, so there it follows the product's
// chunk count (2^10 chunks at most: every halving needs one bit less).
int drop_bits(int S, int chunks) {
  int u = std::max(0, 7 * S - 35);
  if (S == 8)
    for (int c = 1024; u > 0 && c / 2 >= chunks; c /= 2) --u;
  return u;
}
constexpr int kOzMaxChunks = 1024;

// Columns j0 .. j0 + N - 1 of acc (N = 16, 32 or 40) from a group's values v, at
// weight 2^sh; a negative sh is a rounded right shift of the (exact, < 2^25)
// group sum.
template <int N, int EC>
__device__ __forceinline__ void add_group(long long (&acc)[EC], const float *v, int j0, int sh) {
  // (one 32 x 32 + 64-bit multiply-add each; a weight above 2^30 occurs with 8
  // slices only)
  if (sh >= 0 && sh <= 30) {
    const int w = 1 << sh;
#pragma unroll
    for (int j = 0; j < N; ++j)
      acc[j0 + j] += (long long)__float2int_rn(v[j]) * (long long)w;
  } else if (sh >= 0) {
#pragma unroll
    for (int j = 0; j < N; ++j) acc[j0 + j] += (long long)__float2int_rn(v[j]) << sh;
  } else {
    const int r = -sh, half = 1 << (r - 1);
#pragma unroll
    for (int j = 0; j < N; ++j) acc[j0 + j] += (long long)((__float2int_rn(v[j]) + half) >> r);
  }
}

// acc += G_t of every group (t = grp + 2) read from tensor memory, at weight
// 2^(7 (S - 1 - grp) - drop).  One group's values are live at a time (the loop is
// not unrolled: ns == S, passed at run time).
// tcol: this thread's lane and its first column (h EPI_COLS) in group 0.
// With 96-wide groups, half h = 0 reads 32 + 16 columns, h = 1 reads 16 +
// 32, so that every 32-column load starts on a multiple of 32 columns; the
// 40 columns of an 80-wide group's half are five 8-column loads.
template <int S, int BN>
__device__ __forceinline__ bool read_groups(uint32_t tcol, int h,
                                            long long (&acc)[OzShape<S, BN>::EPI_COLS], int ns,
                                            int drop, uint64_t *tempty, uint64_t *tfull,
                                            uint32_t ph, uint64_t lim, int *abort_flag) {
  using Shape = OzShape<S, BN>;
#pragma unroll 1
  for (int grp = 0; grp < ns; ++grp) {
    const int past = grp - Shape::gl(Shape::NP > 1 ? 1 : 0);   // groups past the first phase
    if (grp == 0 || (past >= 0 && past % Shape::W == 0)) {
      // the next phase's groups complete; tcgen05.ld is warp-collective: one
      // decision per warp
      const int p = grp == 0 ? 0 : 1 + past / Shape::W;
      bool have = mbar_wait(&tfull[p], ph, lim);
      have = __all_sync(0xffffffffu, have && !*(volatile int *)abort_flag);
      if (!have) return false;
      fence_after();
    }
    const int sh = 7 * (S - 1 - grp) - drop;
    const uint32_t g0 = tcol + (uint32_t)(grp * BN);
    float v[BN == 80 ? 40 : 32], u[16];
    if constexpr (BN == 64) {
      tmem_ld32(g0, v);
    } else if constexpr (BN == 80) {
      tmem_ld8x5(g0, v);
    } else if (h == 0) {
      tmem_ld32(g0, v);
      tmem_ld16(g0 + 32, u);
    } else {
      tmem_ld16(g0, u);
      tmem_ld32(g0 + 16, v);
    }
    // this group's accumulator may be overwritten by the next chunk
    fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&tempty[grp]);
    if constexpr (BN == 64 || BN == 80) {
      add_group<OzShape<S, BN>::EPI_COLS>(acc, v, 0, sh);
    } else if (h == 0) {
      add_group<32>(acc, v, 0, sh);
      add_group<16>(acc, u, 32, sh);
    } else {
      add_group<16>(acc, u, 0, sh);
      add_group<32>(acc, v, 16, sh);
    }
  }
  return true;
}

// 2^e for a normal-range exponent (clamped to [-1022, 1023])
__device__ __forceinline__ double pow2(int e) {
  e = max(-1022, min(1023, e));
  return __longlong_as_double((long long)(e + 1023) << 52);
}

// One output of the split form, C = x 2^(eB[n]) for row m and column n.
__device__ __forceinline__ void store_one(const OzEpilogue &ep, int atom, int m, int n, double x) {
  if (ep.mode == kOzC) {
    ep.C[(int64_t)m * ep.ldc + n] = x;
  } else if (ep.mode == kOzCT) {
    ep.C[(int64_t)n * ep.ldc + m] = x;
  } else if (ep.mode == kOzBetaT) {
    const int aoA = ep.aoff[atom], nA = ep.aoff[atom + 1] - aoA;
    const int r = m - aoA * ep.n_occ, E = r / nA, c = r - E * nA;
    ep.C[((int64_t)n * ep.n_occ + E) * ep.ldc + aoA + c] = x;
  } else {
    const int B = ep.orb_atom[m], b = m - ep.aoff[B], jj = n / ep.n_occ, E = n - jj * ep.n_occ;
    ep.C[(int64_t)jj * ep.ldc + ep.xoff5[B] + (int64_t)b * ep.n_occ + E] = x;
  }
}

// SPLIT: the CTAs of a cluster (ksplit of them) share one tile.
template <int S, int BN, bool SPLIT>
__global__ void __launch_bounds__(OZ_THREADS, 1)
    ozaki_gemm_kernel(const __grid_constant__ CUtensorMap mapA,
                      const __grid_constant__ CUtensorMap mapB, OzArgs a) {
  int N = a.N;
  if (a.dcnt) N = (int)min((int64_t)N, (int64_t)a.mul_n * (*a.dcnt));
  using Shape = OzShape<S, BN>;
  constexpr int AS = Shape::AS, NP = Shape::NP;
  constexpr int OZ_EPI_COLS = Shape::EPI_COLS;
  // Persistent: CTA b walks tiles t = b, b + gridDim.x, ...  Tile t -> (mt,
  // nt) in an L2-aware order: the M tiles (rows of A, or entries of the tile
  // table) in groups of a.mgroup (A panels that fit in L2 together), every N
  // tile of a group before the next group, the M tile fastest within it, so
  // that each A panel is read from DRAM about once.  Tiles past the live
  // columns are skipped by every role alike.
  const int Mt = a.Mt, Nt = a.Nt, n_tiles = Mt * Nt;
  // split form: the CTAs of a cluster share one tile (the launch has a
  // cluster per tile), CTA `rank` the K chunks [rank c / ks, (rank + 1) c / ks)
  const int ks = SPLIT ? a.ksplit : 1;
  const int rank = SPLIT ? (int)(blockIdx.x % ks) : 0;
  const int tile0 = SPLIT ? (int)(blockIdx.x / ks) : (int)blockIdx.x;
  const int tstep = SPLIT ? n_tiles : (int)gridDim.x;
  struct Tile {
    int m0, xoff, kb0, nkb, rows_valid, atom, n0;   // K blocks kb0 .. kb0 + nkb - 1
  };
  auto tile_of = [&](int t, Tile &T) -> bool {
    const int G = a.mgroup;
    const int g = t / (G * Nt), r = t - g * (G * Nt);
    const int Gg = min(G, Mt - g * G);
    const int mt = g * G + r % Gg, nt = r / Gg;
    T.n0 = nt * BN;
    if (T.n0 >= N) return false;
    if (a.tiles) {
      const GTile gt = a.tiles[mt];
      T.m0 = gt.row0;
      T.xoff = gt.xoff;
      T.nkb = gt.nkb;
      T.rows_valid = gt.rows;
      T.atom = gt.atom;
    } else {
      T.m0 = mt * OZ_BM;
      T.xoff = 0;
      T.nkb = a.KpA / OZ_BK;
      T.rows_valid = min(OZ_BM, a.M - T.m0);
      T.atom = -1;
    }
    T.kb0 = 0;
    if constexpr (SPLIT) {
      const int nch = (T.nkb + a.cb - 1) / a.cb;
      T.kb0 = rank * nch / ks * a.cb;
      T.nkb = min(T.nkb, (rank + 1) * nch / ks * a.cb) - T.kb0;
    }
    return true;
  };
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t *full_a = (uint64_t *)(smem + Shape::A_OFF + AS * OZ_A_BYTES);
  uint64_t *empty_a = full_a + AS;
  uint64_t *full_b = empty_a + AS;
  uint64_t *empty_b = full_b + 2 * NP;    // full_b: [2][NP], a K block's B slices phase by phase
  uint64_t *tfull = empty_b + 2;          // [NP] a chunk's groups, phase by phase
  uint64_t *tempty = tfull + Shape::NP;   // [kOzMaxSlices] one per TMEM group
  uint64_t *drain = tempty + kOzMaxSlices;   // completion of every MMA this CTA issued
  uint32_t *tslot = (uint32_t *)(drain + 1);
  __shared__ int abort_flag;
  const uint64_t lim = wait_limit(a.err);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int s = S;
  const int cb = a.cb;
  constexpr uint32_t tcols = S * BN <= 256 ? 256u : 512u;

  if (threadIdx.x == 0) {
    for (int i = 0; i < AS; ++i) {
      mbar_init(&full_a[i], 1);
      mbar_init(&empty_a[i], 1);
    }
    for (int i = 0; i < 2 * NP; ++i) mbar_init(&full_b[i], 1);
    for (int i = 0; i < 2; ++i) mbar_init(&empty_b[i], 1);
    for (int p = 0; p < NP; ++p) mbar_init(&tfull[p], 1);
    for (int q = 0; q < kOzMaxSlices; ++q)
      mbar_init(&tempty[q], OZ_EPI_WARPS);   // one arrival per epilogue warp
    mbar_init(drain, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(tcols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {
      // producer: the A slices go round a ring of AS tiles, the B slices
      // round two K blocks.  Of a K block: the first phase's B and A slices,
      // the other phases' B slices, then the other A slices (the last phase
      // frees A slices from its first step on, which needs every B).
      int ga = 0, gb = 0;   // A slices and phases of B slices issued
      bool ok = true;
      auto freed = [&](uint64_t *empty, uint32_t ph) {
        if (!mbar_wait(empty, ph ^ 1u, lim)) {
          atomicExch(a.err, 21);
          abort_flag = 1;
          return false;
        }
        return !*(volatile int *)&abort_flag;
      };
      for (int t = tile0; t < n_tiles && ok; t += tstep) {
        Tile T;
        if (!tile_of(t, T)) continue;
        for (int kb = 0; kb < T.nkb && ok; ++kb) {
          const int kx = (T.kb0 + kb) * OZ_BK;
          auto load_a = [&](int i) {
            const int slot = ga % AS;
            ok = ok && freed(&empty_a[slot], (uint32_t)(ga / AS) & 1u);
            if (!ok) return;
            mbar_expect_tx(&full_a[slot], OZ_A_BYTES);
            tma_load_2d(smem + Shape::A_OFF + slot * OZ_A_BYTES, &mapA, &full_a[slot],
                        i * a.KpA + kx, T.m0);
            ++ga;
          };
          auto load_b = [&](int p) {
            const int half = gb / NP & 1, lo = Shape::gl(p), hi = Shape::gh(p);
            if (p == 0) ok = ok && freed(&empty_b[half], (uint32_t)(gb / NP >> 1) & 1u);
            if (!ok) return;
            uint64_t *bar = &full_b[gb % (2 * NP)];
            mbar_expect_tx(bar, (hi - lo + 1) * Shape::B_BYTES);
            for (int j = lo; j <= hi; ++j)
              tma_load_2d(smem + (half * S + j) * Shape::B_BYTES, &mapB, bar,
                          j * a.KpB + T.xoff + kx, T.n0);
            ++gb;
          };
          load_b(0);
          for (int i = 0; i <= Shape::gh(0); ++i) load_a(i);
          for (int p = 1; p < NP; ++p) load_b(p);
          for (int i = Shape::gh(0) + 1; i < S; ++i) load_a(i);
        }
      }
      // copies in flight: the latest use of every barrier must have completed
      // before the CTA may exit
      for (int h = max(0, ga - AS); h < ga; ++h) mbar_wait(&full_a[h % AS], (uint32_t)(h / AS) & 1u);
      for (int h = max(0, gb - 2 * NP); h < gb; ++h)
        mbar_wait(&full_b[h % (2 * NP)], (uint32_t)(h / (2 * NP)) & 1u);
    }
    __syncwarp();
  } else if (warp == 1) {
    // The whole warp runs the schedule; the elected lane issues.  Slice A_i
    // against neighbouring B slices is one MMA: the B tiles of a K block lie
    // one after the other (rows of one operand), and the groups i + j of
    // neighbouring j are neighbouring TMEM columns.  Up to W groups (256
    // columns) at a time, in phases of groups gl .. gh: A_i x B_j, j from
    // gl - i (or 0) to gh - i, for i = 0 .. gh; i = 0 touches every group of the phase
    // first.  Exact integer sums: any order gives the same bits.
    const uint32_t leader = elect_one();
    const uint32_t lo0 = desc_lo(smem_u32(smem));
    int a0 = 0;            // A ring slot and phase of the K block's slice 0
    uint32_t pa0 = 0;
    int bc = 0;            // K blocks issued (the B half is bc & 1)
    int gc = 0;            // chunks issued by this CTA (over its tiles)
    bool ok = true;
    auto wait_for = [&](uint64_t *bar, uint32_t ph, int code) {
      if (ok && !warp_wait(bar, ph, lim)) {
        if (lane == 0) atomicExch(a.err, code);
        abort_flag = 1;
        ok = false;
      }
    };
    for (int t = tile0; t < n_tiles && ok; t += tstep) {
      Tile T;
      if (!tile_of(t, T)) continue;
      const int nchunks = (T.nkb + cb - 1) / cb;
      for (int c = 0; c < nchunks && ok; ++c, ++gc) {
        const int kb1 = min(T.nkb, (c + 1) * cb);
        for (int kb = c * cb; kb < kb1 && ok; ++kb, ++bc) {
          const bool first_kb = kb == c * cb;
          const uint32_t pb = (uint32_t)(bc >> 1) & 1u;
          const uint32_t lob = lo0 + (uint32_t)((bc & 1) * S) * (Shape::B_BYTES >> 4);
          auto slot_of = [&](int i) { return (a0 + i) % AS; };
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            const int gl = Shape::gl(p), gh = Shape::gh(p);
            wait_for(&full_b[(bc & 1) * NP + p], pb, 23);
            // the phase's groups of the previous chunk (of this tile or the
            // one before) drained by the epilogue, which drains them in
            // order: the first phase overlaps the drain of the later groups
            if (first_kb && gc > 0) {
#pragma unroll
              for (int g = gl; g <= gh; ++g) wait_for(&tempty[g], (uint32_t)(gc - 1) & 1u, 22);
            }
            if (!ok) break;
#pragma unroll
            for (int i = 0; i <= gh; ++i) {
              if (i >= gl) wait_for(&full_a[slot_of(i)], pa0 ^ ((uint32_t)((a0 + i) / AS) & 1u), 23);
              if (!ok) break;
              fence_after();
              const int jl = gl > i ? gl - i : 0, n = gh - i - jl + 1;
              const uint32_t la =
                  lo0 + ((Shape::A_OFF + (uint32_t)slot_of(i) * OZ_A_BYTES) >> 4);
              const uint32_t lb = lob + (uint32_t)jl * (Shape::B_BYTES >> 4);
              const uint32_t d = tmem + (uint32_t)((i + jl) * BN);
#pragma unroll
              for (int k = 0; k < OZ_BK / 16; ++k)   // 32 bytes per K step
                mma_bf16_if(leader, d, desc_of(la + 2 * k), desc_of(lb + 2 * k),
                            idesc_bf16(OZ_BM, n * BN), (first_kb && i == 0 && k == 0) ? 0u : 1u);
              // A_i has no later use (free once these MMAs complete)
              if (p == NP - 1) mma_commit_if(leader, &empty_a[slot_of(i)]);
            }
            if (!ok) break;
            // (the epilogue reads them while the later phases still run)
            if (kb == kb1 - 1) mma_commit_if(leader, &tfull[p]);
          }
          if (!ok) break;
          mma_commit_if(leader, &empty_b[bc & 1]);
          pa0 ^= (uint32_t)((a0 + S) / AS) & 1u;
          a0 = (a0 + S) % AS;
        }
      }
    }
    // every MMA issued here (also after an abort) completes before the
    // tensor memory is freed
    mma_commit_if(leader, drain);
    mbar_wait(drain, 0u);
    __syncwarp();
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31 (rows of the tile)
    // and half h = (w - 2) / 4 of every group's columns (EPI_COLS of them)
    const int q = warp & 3, h = (warp - 2) >> 2;
    const int lr = q * 32 + lane;
    const uint32_t tcol = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * OZ_EPI_COLS);
    int gc = 0;   // chunks drained (over this CTA's tiles)
    for (int t = tile0; t < n_tiles; t += tstep) {
      Tile T;
      if (!tile_of(t, T)) continue;
      const int m = T.m0 + lr;
      const int nc = T.n0 + h * OZ_EPI_COLS;
      const int nchunks = (T.nkb + cb - 1) / cb;
      long long acc[OZ_EPI_COLS];
#pragma unroll
      for (int j = 0; j < OZ_EPI_COLS; ++j) acc[j] = 0;
      bool ok = true;
      for (int c = 0; c < nchunks; ++c, ++gc) {
        if (!read_groups<S, BN>(tcol, h, acc, a.ns, a.drop, tempty, tfull, (uint32_t)gc & 1u, lim,
                                &abort_flag)) {
          if (lane == 0) atomicExch(a.err, 24);
          abort_flag = 1;
          ok = false;
          break;
        }
      }
      if (!ok) break;
      if constexpr (SPLIT) {
        // this CTA's partial sums to its shared memory (the ring is idle: the
        // last chunk's MMAs, and with them every copy, have completed)
        long long *part = (long long *)smem;   // [BN][OZ_BM]
#pragma unroll
        for (int j = 0; j < OZ_EPI_COLS; ++j) part[(h * OZ_EPI_COLS + j) * OZ_BM + lr] = acc[j];
      } else
      if (lr < T.rows_valid && nc < N) {
        // C = acc 2^(eA + eB + u - 7(S+1)), as two exact power-of-two factors
        const double fa = pow2(a.eA[m] + a.drop - 7 * (S + 1));
        const OzEpilogue &ep = a.ep;
        if (ep.mode == kOzC) {
          double *crow = ep.C + (int64_t)m * ep.ldc + nc;
          if (a.vec && nc + OZ_EPI_COLS <= N) {
#pragma unroll
            for (int j = 0; j < OZ_EPI_COLS; j += 2) {
              double2 w;
              w.x = (double)acc[j] * fa * pow2(__ldg(a.eB + nc + j));
              w.y = (double)acc[j + 1] * fa * pow2(__ldg(a.eB + nc + j + 1));
              *(double2 *)(crow + j) = w;
            }
          } else {
#pragma unroll
            for (int j = 0; j < OZ_EPI_COLS; ++j)
              if (nc + j < N) crow[j] = (double)acc[j] * fa * pow2(__ldg(a.eB + nc + j));
          }
        } else if (ep.mode == kOzCT) {
#pragma unroll
          for (int j = 0; j < OZ_EPI_COLS; ++j)
            if (nc + j < N)
              ep.C[(int64_t)(nc + j) * ep.ldc + m] =
                  (double)acc[j] * fa * pow2(__ldg(a.eB + nc + j));
        } else if (ep.mode == kOzBetaT) {
          // row m = (atom A, E, c): beta^T[(j n_occ + E)][ao_A + c] for column j
          const int aoA = ep.aoff[T.atom], nA = ep.aoff[T.atom + 1] - aoA;
          const int r = m - aoA * ep.n_occ, E = r / nA, c = r - E * nA;
          double *dst = ep.C + (int64_t)E * ep.ldc + aoA + c;
          const int64_t step = (int64_t)ep.n_occ * ep.ldc;
#pragma unroll
          for (int j = 0; j < OZ_EPI_COLS; ++j)
            if (nc + j < N)
              dst[(int64_t)(nc + j) * step] = (double)acc[j] * fa * pow2(__ldg(a.eB + nc + j));
        } else {
          // kOzGammaCat: row m = orbital (atom B, b), column n = j n_occ + E ->
          // Gcat[j][xoff_B + b n_occ + E]
          const int B = ep.orb_atom[m], b = m - ep.aoff[B];
          const int64_t xo = ep.xoff5[B] + (int64_t)b * ep.n_occ;
          int jj = nc / ep.n_occ, E = nc - jj * ep.n_occ;
#pragma unroll
          for (int j = 0; j < OZ_EPI_COLS; ++j) {
            if (nc + j < N)
              ep.C[(int64_t)jj * ep.ldc + xo + E] =
                  (double)acc[j] * fa * pow2(__ldg(a.eB + nc + j));
            if (++E == ep.n_occ) {
              E = 0;
              ++jj;
            }
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols));
  }
  if constexpr (SPLIT) {
    // the cluster's integer partial sums added (exact in any order) and
    // stored, the columns shared out over its CTAs.  Every thread of every
    // CTA gets here: the roles above end by themselves, after an abort too.
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    Tile T;
    if (tile0 < n_tiles && tile_of(tile0, T) && !*(volatile int *)&abort_flag) {
      const int row = threadIdx.x & (OZ_BM - 1);
      for (int j = rank + ks * (int)(threadIdx.x / OZ_BM); j < BN;
           j += ks * (OZ_THREADS / OZ_BM)) {
        const int m = T.m0 + row, n = T.n0 + j;
        if (threadIdx.x >= OZ_THREADS / OZ_BM * OZ_BM || row >= T.rows_valid || n >= N) continue;
        long long sum = 0;
        for (int q = 0; q < ks; ++q)
          sum += cl.map_shared_rank((const long long *)smem, q)[j * OZ_BM + row];
        store_one(a.ep, T.atom, m, n,
                  (double)sum * pow2(a.eA[m] + a.drop - 7 * (S + 1)) * pow2(a.eB[n]));
      }
    }
    cl.sync();   // partial sums stay until every CTA has read them
  }
}

// ---------------------------------------------------------------------------
// Slicing, in integer arithmetic on the float64 bit patterns (float64 ops run
// at 1/64 of the float32 rate on this part).  The row exponent is e = f - 1022
// for the largest biased exponent field f of the row (so |x| < 2^e); each x
// becomes the fixed-point integer F = round(x 2^(7s - e)), |F| <= 2^(7s),
// and F is written as balanced base-128 digits, most significant first:
//   F = sum_i q_i 128^(s-i),   q_1 in [-128, 128],  q_i in [-64, 63] (i > 1),
// so x = 2^e sum_i q_i 2^(-7i) up to the rounding of F.  Zero and subnormal
// values (below 2^-1022, far under any row's scale) count as zero.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int exp_field(double x) {
  return (int)((__double_as_longlong(x) >> 52) & 0x7FF);
}
__device__ __forceinline__ int row_exponent_of_field(int fmax) {
  return fmax > 0 ? fmax - 1022 : 0;
}
__device__ __forceinline__ long long fixed_point(double x, int e, int s) {
  const long long b = __double_as_longlong(x);
  const int f = (int)((b >> 52) & 0x7FF);
  if (f == 0) return 0;
  const long long M = (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);   // x = +-M 2^(f - 1075)
  const int sh = f - 1075 + 7 * s - e;
  long long F;
  if (sh >= 0) F = M << sh;                       // only for s = 8 (sh <= 3)
  else if (sh < -62) F = 0;
  else F = (M + (1ll << (-sh - 1))) >> (-sh);     // round half up in magnitude
  return b < 0 ? -F : F;
}
// The high half of float32(q) is bf16(q) for |q| <= 128 (8 significant bits at
// most); q + 1.5 * 2^23 is formed in the integer pipe, the float subtraction
// is exact.
__device__ __forceinline__ unsigned int float_bits(int q) {
  return __float_as_uint(__int_as_float(0x4B400000 + q) - 12582912.0f);
}
// Slices of four neighbouring entries of a row with exponent e, stored as
// four bf16 at dst + i*Kp for slice i (k a multiple of 4: 8-byte stores).
// With the offset sum_{t < S-1} 64 128^t added to F, the balanced digit t is
// the plain base-128 digit minus 64, so the digits are independent 7-bit
// fields: four of them in the low 28 bits, the others above.
template <int S>
__device__ __forceinline__ void store_slices(const double (&x)[4], int e, int Kp,
                                             __nv_bfloat16 *dst) {
  constexpr long long kOff = [] {
    long long o = 0;
    for (int t = 0; t < S - 1; ++t) o = o * 128 + 64;
    return o;
  }();
  int lo[4], hi[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const long long F = fixed_point(x[j], e, S) + kOff;
    lo[j] = S <= 4 ? (int)F : (int)(F & 0xFFFFFFF);
    hi[j] = S <= 4 ? 0 : (int)(F >> 28);
  }
#pragma unroll
  for (int i = 0; i < S; ++i) {
    const int t = S - 1 - i;   // digit of weight 128^t
    unsigned int f[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int v = t < 4 ? lo[j] >> (7 * (t & 3)) : hi[j] >> (7 * (t & 3));
      f[j] = float_bits(i == 0 ? v : (v & 127) - 64);
    }
    uint2 w;
    w.x = __byte_perm(f[0], f[1], 0x7632);
    w.y = __byte_perm(f[2], f[3], 0x7632);
    *(uint2 *)(dst + (int64_t)i * Kp) = w;
  }
}

// Entry k of row x of the operand: x[k] for k < Kdim, or, with a column map,
// x[cols[k]] (zero where cols[k] < 0).
__device__ __forceinline__ double gathered(const double *x, const int *cols, int k, int Kdim) {
  if (k >= Kdim) return 0.0;
  if (!cols) return x[k];
  const int c = cols[k];
  return c >= 0 ? x[c] : 0.0;
}
template <int S>
__device__ __forceinline__ void slice_at(const double *x, const int *cols, int k, int Kdim, int e,
                                         int Kp, __nv_bfloat16 *qr) {
  double v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = gathered(x, cols, k + j, Kdim);
  store_slices<S>(v, e, Kp, qr + k);
}

// Rows, WPR warps per row (8 rows per CTA, or 1): the exponent of the row's
// largest entry, then its slices (the second read comes from L1 or L2).
template <int S, int WPR>
__global__ void __launch_bounds__(256) oz_slice_rows_kernel(int rows, int Kdim,
                                                            const double *__restrict__ X,
                                                            int64_t ldx,
                                                            const int *__restrict__ cols, int Kp,
                                                            __nv_bfloat16 *__restrict__ Q,
                                                            int *__restrict__ E, const int *dcnt,
                                                            int mul) {
  __shared__ int red[8];
  const int live = dcnt ? min(rows, mul * (*dcnt)) : rows;
  const int warp = threadIdx.x >> 5;
  const int r = blockIdx.x * (8 / WPR) + warp / WPR;
  const int t = (warp % WPR) * 32 + (threadIdx.x & 31);
  const bool on = r < live;
  const double *x = X + (int64_t)r * ldx;
  int fm = 0;
  if (on) {
#pragma unroll 4
    for (int k = t; k < Kdim; k += 32 * WPR) fm = max(fm, exp_field(gathered(x, cols, k, Kdim)));
  }
  for (int o = 16; o > 0; o >>= 1) fm = max(fm, __shfl_xor_sync(0xffffffffu, fm, o));
  if (WPR > 1) {
    if ((threadIdx.x & 31) == 0) red[warp] = fm;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < WPR; ++w) fm = max(fm, red[w]);
  }
  if (!on) return;
  const int e = row_exponent_of_field(fm);
  if (t == 0) E[r] = e;
  __nv_bfloat16 *qr = Q + (int64_t)r * S * Kp;
  for (int k = 4 * t; k < Kp; k += 128 * WPR) slice_at<S>(x, cols, k, Kdim, e, Kp, qr);
}

// Long rows: grid (chunks, rows).  Pass 1 raises E[r] (preset to a large
// negative value) to the exponent of each chunk's largest entry; pass 2
// slices every chunk with the row's exponent (a row of zeros keeps the preset
// value and gives zero slices).
constexpr int OZ_CHUNK = 2048;

__global__ void __launch_bounds__(256) oz_rowmax_kernel(int rows, int Kdim,
                                                        const double *__restrict__ X, int64_t ldx,
                                                        const int *__restrict__ cols,
                                                        int *__restrict__ E, const int *dcnt,
                                                        int mul) {
  int live = rows;
  if (dcnt) live = min(rows, mul * (*dcnt));
  const int r = blockIdx.y;
  if (r >= live) return;
  const double *x = X + (int64_t)r * ldx;
  const int k0 = blockIdx.x * OZ_CHUNK, k1 = min(Kdim, k0 + OZ_CHUNK);
  int fm = 0;
#pragma unroll 4
  for (int k = k0 + threadIdx.x; k < k1; k += 256) fm = max(fm, exp_field(gathered(x, cols, k, Kdim)));
  for (int o = 16; o > 0; o >>= 1) fm = max(fm, __shfl_xor_sync(0xffffffffu, fm, o));
  if ((threadIdx.x & 31) == 0 && fm > 0) atomicMax(E + r, row_exponent_of_field(fm));
}

template <int S>
__global__ void __launch_bounds__(256) oz_slice_chunks_kernel(int rows, int Kdim,
                                                              const double *__restrict__ X,
                                                              int64_t ldx,
                                                              const int *__restrict__ cols, int Kp,
                                                              __nv_bfloat16 *__restrict__ Q,
                                                              const int *__restrict__ E,
                                                              const int *dcnt, int mul) {
  int live = rows;
  if (dcnt) live = min(rows, mul * (*dcnt));
  const int r = blockIdx.y;
  if (r >= live) return;
  const int e = E[r];   // a row of zeros: every entry gives F = 0 whatever e is
  const int k0 = blockIdx.x * OZ_CHUNK, k1 = min(Kp, k0 + OZ_CHUNK);
  for (int k = k0 + 4 * threadIdx.x; k < k1; k += 1024)
    slice_at<S>(X + (int64_t)r * ldx, cols, k, Kdim, e, Kp, Q + (int64_t)r * S * Kp);
}

// Columns of a row-major matrix, 32 per CTA: one 64-row tile staged through
// shared memory and written as rows of the transposed operand.
template <int S>
__device__ __forceinline__ void slice_col_tile(int Kdim, int live, const double *X, int64_t ldx,
                                               int Kp, __nv_bfloat16 *Q, int n0, int k0,
                                               const int *ecol, double (*tile)[66]) {
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, n = n0 + tx;
#pragma unroll
  for (int rr = ty; rr < 64; rr += 8) {
    const int k = k0 + rr;
    tile[tx][rr] = (k < Kdim && n < live) ? X[(int64_t)k * ldx + n] : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int col = 16 * h + (threadIdx.x >> 4), k4 = 4 * (threadIdx.x & 15);
    if (n0 + col < live) {
      const double2 a = *(const double2 *)&tile[col][k4], b = *(const double2 *)&tile[col][k4 + 2];
      const double v[4] = {a.x, a.y, b.x, b.y};
      store_slices<S>(v, ecol[col], Kp, Q + (int64_t)(n0 + col) * S * Kp + k0 + k4);
    }
  }
  __syncthreads();
}

// Short columns: exponents and slices in one launch (grid: column groups).
template <int S>
__global__ void __launch_bounds__(256) oz_slice_cols_kernel(int Kdim, int N,
                                                            const double *__restrict__ X,
                                                            int64_t ldx, int Kp,
                                                            __nv_bfloat16 *__restrict__ Q,
                                                            int *__restrict__ E, const int *dcnt,
                                                            int mul) {
  __shared__ __align__(16) double tile[32][66];
  __shared__ int red[8][32];
  __shared__ int ecol[32];
  int live = N;
  if (dcnt) live = (int)min((int64_t)N, (int64_t)mul * (*dcnt));
  const int n0 = blockIdx.x * 32;
  if (n0 >= live) return;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int n = n0 + tx;
  int fm = 0;
  if (n < live) {
#pragma unroll 8
    for (int k = ty; k < Kdim; k += 8) fm = max(fm, exp_field(X[(int64_t)k * ldx + n]));
  }
  red[ty][tx] = fm;
  __syncthreads();
  if (ty == 0) {
    int v = 0;
    for (int i = 0; i < 8; ++i) v = max(v, red[i][tx]);
    const int e = row_exponent_of_field(v);
    if (n < live) E[n] = e;
    ecol[tx] = e;
  }
  __syncthreads();
  for (int k0 = 0; k0 < Kp; k0 += 64)
    slice_col_tile<S>(Kdim, live, X, ldx, Kp, Q, n0, k0, ecol, tile);
}

// Long columns: the same in two passes over a grid (column groups, K chunks),
// the exponents by atomic maximum into a preset E as for long rows.
constexpr int OZ_CCHUNK = 256;

__global__ void __launch_bounds__(256) oz_colmax_kernel(int Kdim, int N,
                                                        const double *__restrict__ X, int64_t ldx,
                                                        int *__restrict__ E, const int *dcnt,
                                                        int mul) {
  __shared__ int red[8][32];
  int live = N;
  if (dcnt) live = (int)min((int64_t)N, (int64_t)mul * (*dcnt));
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, n = blockIdx.x * 32 + tx;
  if (blockIdx.x * 32 >= live) return;
  const int k0 = blockIdx.y * OZ_CCHUNK, k1 = min(Kdim, k0 + OZ_CCHUNK);
  int fm = 0;
  if (n < live) {
#pragma unroll 8
    for (int k = k0 + ty; k < k1; k += 8) fm = max(fm, exp_field(X[(int64_t)k * ldx + n]));
  }
  red[ty][tx] = fm;
  __syncthreads();
  if (ty == 0 && n < live) {
    int v = 0;
    for (int i = 0; i < 8; ++i) v = max(v, red[i][tx]);
    if (v > 0) atomicMax(E + n, row_exponent_of_field(v));
  }
}

template <int S>
__global__ void __launch_bounds__(256) oz_slice_col_chunks_kernel(
    int Kdim, int N, const double *__restrict__ X, int64_t ldx, int Kp,
    __nv_bfloat16 *__restrict__ Q, const int *__restrict__ E, const int *dcnt, int mul) {
  __shared__ __align__(16) double tile[32][66];
  __shared__ int ecol[32];
  int live = N;
  if (dcnt) live = (int)min((int64_t)N, (int64_t)mul * (*dcnt));
  const int n0 = blockIdx.x * 32;
  if (n0 >= live) return;
  if (threadIdx.x < 32) ecol[threadIdx.x] = n0 + threadIdx.x < live ? E[n0 + threadIdx.x] : 0;
  const int k1 = min(Kp, (int)(blockIdx.y + 1) * OZ_CCHUNK);
  for (int k0 = blockIdx.y * OZ_CCHUNK; k0 < k1; k0 += 64)   // (the tile's barrier covers ecol)
    slice_col_tile<S>(Kdim, live, X, ldx, Kp, Q, n0, k0, ecol, tile);
}

// f(integral_constant<S>) for the slice count s of an operand
template <class F>
cudaError_t with_slices(int s, F &&f) {
  switch (s) {
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 5: return f(std::integral_constant<int, 5>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
    case 8: return f(std::integral_constant<int, 8>{});
    default: return cudaErrorInvalidValue;
  }
}

int chunk_blocks(int s) { return std::max(1, 4096 / (s + 2) / OZ_BK); }

template <int S, int BN>
cudaError_t launch_oz_kernel(cudaStream_t st, int ctas, const CUtensorMap &mA,
                             const CUtensorMap &mB, const OzArgs &a) {
  if (a.ksplit <= 1) {
    ozaki_gemm_kernel<S, BN, false><<<ctas, OZ_THREADS, OzShape<S, BN>::SMEM, st>>>(mA, mB, a);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(OZ_THREADS);
  cfg.dynamicSmemBytes = OzShape<S, BN>::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = a.ksplit;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ozaki_gemm_kernel<S, BN, true>, mA, mB, a);
}

template <int S, int BN>
cudaError_t set_smem_attr() {
  constexpr int bytes = (int)OzShape<S, BN>::SMEM;
  const cudaError_t e = cudaFuncSetAttribute(ozaki_gemm_kernel<S, BN, false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(ozaki_gemm_kernel<S, BN, true>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// Clusters of c CTAs (one CTA per SM) that run at once.  GPCs hold 16 to 20
// SMs, so 152 SMs take 76 clusters of 2, 36 of 4, 23 of 6, but 15 of 7 or 8.
// (0 for a size that cannot be asked; single CTAs always run.)
int active_clusters(int c) {
  static PerDevice fits[9];
  const int fit = fits[c].get([c] {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c * 256);
    cfg.blockDim = dim3(OZ_THREADS);
    cfg.dynamicSmemBytes = OzShape<6, 64>::SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = c;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, ozaki_gemm_kernel<6, 64, true>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    return n;
  });
  return c == 1 && fit < 1 ? sm_count() : fit;
}

// Clocks per K block of a tile: an MMA of N columns takes N / 2 at the tensor
// core's rate and at least 40 + N / 4 (operand reads and issue), the slices
// come from L2 at 54 bytes a clock at most.  Measured per block, 15% of it at
// the chunks' ends: 5 slices 2670 clocks at N = 64 and 3530 at 96, 6 slices
// 3400 at 64 and 4010 at 80 (pair by pair: 4600 at 64, 5460 at 80).
double block_clocks(int S, int bn) {
  const int W = std::min(S, 256 / bn), np = (S + W - 1) / W;
  double mma = 0;
  for (int p = 0, gl = 0; p < np; ++p) {
    const int gh = S - 1 - (np - 1 - p) * W;
    for (int i = 0; i <= gh; ++i) {
      const int n = (gh - std::max(i, gl) + 1) * bn;
      mma += std::max(0.5 * n, 40 + 0.25 * n);
    }
    gl = gh + 1;
  }
  return std::max(OZ_BK / 16 * mma, S * (OZ_BM + bn) * OZ_BK * 2 / 54.0);
}

// N tile and K split of a product of Mt row tiles, N columns and nch K chunks:
// the least of waves x chunks per CTA x clocks per block, with half a chunk
// for the sum over a cluster and a third for a tile's start.  Exact integer
// sums: every plan gives the same bits.
// (1000 x 129 x 9080, 6 slices: 24 CTAs of 64 columns 455 us -> 16
// clusters of 6, 80 columns each, 65 us.)
struct TilePlan {
  int bn, ks;
};
TilePlan tile_plan(int S, int Mt, int N, int nch) {
  TilePlan best{64, 1};
  double least = 1e300;
  for (int bn : {64, oz_wide_bn(S)}) {
    const double tiles = (double)Mt * ((N + bn - 1) / bn);
    for (int ks = 1; ks <= std::min(8, nch); ++ks) {
      const int fit = active_clusters(ks);
      if (fit < 1) continue;
      const double cost = std::ceil(tiles / fit) * ((nch + ks - 1) / ks + (ks > 1 ? 0.83 : 0.33)) *
                          block_clocks(S, bn);
      if (cost < least) {
        least = cost;
        best = TilePlan{bn, ks};
      }
    }
  }
  return best;
}
}  // namespace

// Dynamic shared memory limits of every slice count (once; outside any
// stream capture).
cudaError_t oz_init_attributes() {
  static PerDevice done;
  cudaError_t e = cudaSuccess;
  done.get([&e] {
    for (int n = kOzMinSlices; n <= kOzMaxSlices && e == cudaSuccess; ++n)
      e = with_slices(n, [](auto sc) {
        constexpr int S = decltype(sc)::value, W = oz_wide_bn(S);
        const cudaError_t r = set_smem_attr<S, 64>();
        return W == 64 || r != cudaSuccess ? r : set_smem_attr<S, W>();
      });
    return e == cudaSuccess ? 1 : 0;
  });
  return e;
}

cudaError_t oz_operand(OzOperand &op, __nv_bfloat16 *q, int *e, int64_t rows, int Kdim, int s,
                       int box_rows) {
  if (s < kOzMinSlices || s > kOzMaxSlices || rows < 1 || Kdim < 1) return cudaErrorInvalidValue;
  op.q = q;
  op.e = e;
  op.rows = rows;
  op.Kp = round_up(Kdim, OZ_BK);
  op.s = s;
  const cudaError_t r = encode_bf16_map(&op.map, q, rows, (int64_t)s * op.Kp, box_rows);
  // the B role (box_rows OZ_BN) also takes boxes of the wide N tile
  if (r != cudaSuccess || box_rows != OZ_BN) return r;
  return encode_bf16_map(&op.map_wide, q, rows, (int64_t)s * op.Kp, oz_wide_bn(s));
}

// Rows up to this length take one warp each, then one CTA; from OZ_LONG_ROW on
// (and for columns from OZ_LONG_COL on) chunks go to separate CTAs, with the
// exponent by atomic maximum in a pass of its own.
constexpr int OZ_WARP_ROW = 2048, OZ_LONG_ROW = 8192, OZ_LONG_COL = 512;

cudaError_t launch_oz_slice_rows(cudaStream_t st, const double *X, int64_t ldx, int rows, int Kdim,
                                 OzOperand &op, const int *dcnt, int mul, const int *cols) {
  if (rows <= 0) return cudaSuccess;
  if (rows > op.rows || Kdim > op.Kp) return cudaErrorInvalidValue;
  return with_slices(op.s, [&](auto sc) {
    constexpr int S = decltype(sc)::value;
    if (op.Kp >= OZ_LONG_ROW && rows <= 65535) {
      cudaError_t e = cudaMemsetAsync(op.e, 0x80, (size_t)rows * sizeof(int), st);
      if (e != cudaSuccess) return e;
      dim3 g1((Kdim + OZ_CHUNK - 1) / OZ_CHUNK, rows), g2((op.Kp + OZ_CHUNK - 1) / OZ_CHUNK, rows);
      oz_rowmax_kernel<<<g1, 256, 0, st>>>(rows, Kdim, X, ldx, cols, op.e, dcnt, mul);
      oz_slice_chunks_kernel<S><<<g2, 256, 0, st>>>(rows, Kdim, X, ldx, cols, op.Kp, op.q, op.e,
                                                    dcnt, mul);
    } else if (op.Kp <= OZ_WARP_ROW) {
      oz_slice_rows_kernel<S, 1><<<(rows + 7) / 8, 256, 0, st>>>(rows, Kdim, X, ldx, cols, op.Kp,
                                                                 op.q, op.e, dcnt, mul);
    } else {
      oz_slice_rows_kernel<S, 8><<<rows, 256, 0, st>>>(rows, Kdim, X, ldx, cols, op.Kp, op.q, op.e,
                                                       dcnt, mul);
    }
    return cudaGetLastError();
  });
}

cudaError_t launch_oz_slice_cols(cudaStream_t st, const double *X, int64_t ldx, int Kdim, int N,
                                 OzOperand &op, const int *dcnt, int mul) {
  if (N <= 0) return cudaSuccess;
  if (N > op.rows || Kdim > op.Kp) return cudaErrorInvalidValue;
  return with_slices(op.s, [&](auto sc) {
    constexpr int S = decltype(sc)::value;
    const int chunks = (op.Kp + OZ_CCHUNK - 1) / OZ_CCHUNK;
    if (op.Kp >= OZ_LONG_COL && chunks <= 65535) {
      cudaError_t e = cudaMemsetAsync(op.e, 0x80, (size_t)N * sizeof(int), st);
      if (e != cudaSuccess) return e;
      const dim3 grid((N + 31) / 32, chunks);
      oz_colmax_kernel<<<grid, 256, 0, st>>>(Kdim, N, X, ldx, op.e, dcnt, mul);
      oz_slice_col_chunks_kernel<S><<<grid, 256, 0, st>>>(Kdim, N, X, ldx, op.Kp, op.q, op.e, dcnt,
                                                          mul);
    } else {
      oz_slice_cols_kernel<S><<<(N + 31) / 32, 256, 0, st>>>(Kdim, N, X, ldx, op.Kp, op.q, op.e,
                                                             dcnt, mul);
    }
    return cudaGetLastError();
  });
}

cudaError_t launch_gemm_oz_ex(cudaStream_t st, const OzOperand &A, const OzOperand &B, int M,
                              int N, const OzEpilogue &ep, const GTile *tiles, int n_tiles,
                              int max_nkb, int *err, const int *dcnt, int mul_n) {
  if (N <= 0 || (tiles ? n_tiles <= 0 : M <= 0)) return cudaSuccess;
  if (A.s != B.s || N > B.rows || (!tiles && (A.Kp != B.Kp || M > A.rows)))
    return cudaErrorInvalidValue;
  cudaError_t e = oz_init_attributes();
  if (e != cudaSuccess) return e;
  OzArgs a;
  a.M = M;
  a.N = N;
  a.KpA = A.Kp;
  a.KpB = B.Kp;
  a.ns = A.s;
  a.cb = chunk_blocks(A.s);
  const int nkb = tiles ? max_nkb : A.Kp / OZ_BK;
  if ((nkb + a.cb - 1) / a.cb > kOzMaxChunks) return cudaErrorInvalidValue;
  a.eA = A.e;
  a.eB = B.e;
  a.ep = ep;
  a.vec = (ep.mode == kOzC && (ep.ldc % 2) == 0 && ((uintptr_t)ep.C & 15) == 0) ? 1 : 0;
  a.tiles = tiles;
  {
    // M tiles whose A panels (s slices of the whole K) fill about 40 MB of L2
    const double panel = (double)OZ_BM * A.s * A.Kp * sizeof(__nv_bfloat16);
    const int Mt = tiles ? n_tiles : (M + OZ_BM - 1) / OZ_BM;
    a.mgroup = std::max(1, std::min(Mt, (int)(40.0e6 / panel)));
  }
  a.err = err;
  a.dcnt = dcnt;
  a.mul_n = mul_n;
  a.Mt = tiles ? n_tiles : (M + OZ_BM - 1) / OZ_BM;
  const int nch = (nkb + a.cb - 1) / a.cb;
  a.drop = drop_bits(A.s, nch);
  const TilePlan plan = tile_plan(A.s, a.Mt, N, nch);
  a.Nt = (N + plan.bn - 1) / plan.bn;
  a.ksplit = plan.ks;
  const int64_t all = (int64_t)a.Mt * a.Nt;
  if (all * plan.ks > INT32_MAX) return cudaErrorInvalidConfiguration;
  // unsplit: a persistent grid, one CTA per SM at most, each walking its share
  // of the tiles; split: one cluster per tile
  const int ctas = (int)(plan.ks > 1 ? all * plan.ks : std::min<int64_t>(all, active_clusters(1)));
  return with_slices(A.s, [&](auto sc) {
    constexpr int S = decltype(sc)::value, W = oz_wide_bn(S);
    if (plan.bn == 64) return launch_oz_kernel<S, 64>(st, ctas, A.map, B.map, a);
    return launch_oz_kernel<S, W>(st, ctas, A.map, B.map_wide, a);
  });
}

cudaError_t launch_gemm_oz(cudaStream_t st, const OzOperand &A, const OzOperand &B, int M, int N,
                           double *C, int64_t ldc, int trans, int *err, const int *dcnt,
                           int mul_n) {
  OzEpilogue ep;
  ep.mode = trans ? kOzCT : kOzC;
  ep.C = C;
  ep.ldc = ldc;
  return launch_gemm_oz_ex(st, A, B, M, N, ep, nullptr, 0, 0, err, dcnt, mul_n);
}

// Constants sliced once; dynamic operands sized for `slots` right-hand sides.
cudaError_t oz_setup(cudaStream_t st, const DevSystem &sys, OzWork &oz, int slots,
                     std::vector<void *> &allocs) {
  const int s = oz.s, np = sys.n_prod, no = sys.n_orb, nv = sys.n_virt;
  const int64_t rowsB = 2 * (int64_t)slots * sys.n_occ;
  const int64_t rows6 = 6 * (int64_t)sys.n_occ;   // the three dipole columns
  const int64_t rowsT = std::max(rowsB, rows6);
  const int KpK = round_up(np, OZ_BK), Kp1 = round_up(no, OZ_BK), Kp2 = round_up(nv, OZ_BK);
  auto alloc = [&](size_t bytes, void **p) -> cudaError_t {
    cudaError_t e = cudaMalloc(p, bytes + 16);
    if (e == cudaSuccess) allocs.push_back(*p);
    return e;
  };
  void *qK, *qXvT, *qXv, *qZ, *qT, *e;
  const size_t bf = sizeof(__nv_bfloat16);
  const int64_t rowsZ = 2 * (int64_t)slots;
  cudaError_t r = alloc((size_t)np * s * KpK * bf, &qK);
  if (r == cudaSuccess) r = alloc((size_t)nv * s * Kp1 * bf, &qXvT);
  if (r == cudaSuccess) r = alloc((size_t)no * s * Kp2 * bf, &qXv);
  if (r == cudaSuccess) r = alloc((size_t)rowsZ * s * KpK * bf, &qZ);
  if (r == cudaSuccess) r = alloc((size_t)rowsT * s * std::max(Kp1, Kp2) * bf, &qT);
  const int64_t ne = (int64_t)np + nv + no + rowsZ + 2 * rowsT;
  if (r == cudaSuccess) r = alloc((size_t)ne * sizeof(int), &e);
  if (r == cudaSuccess) r = alloc(ptx::kErrInts * sizeof(int), (void **)&oz.err);
  if (r != cudaSuccess) return r;
  int *ep = (int *)e;
  auto bq = [](void *p) { return (__nv_bfloat16 *)p; };
  r = oz_operand(oz.K, bq(qK), ep, np, np, s, OZ_BM);
  ep += np;
  if (r == cudaSuccess) r = oz_operand(oz.XvT, bq(qXvT), ep, nv, no, s, OZ_BM);
  ep += nv;
  if (r == cudaSuccess) r = oz_operand(oz.Xv, bq(qXv), ep, no, nv, s, OZ_BM);
  ep += no;
  if (r == cudaSuccess) r = oz_operand(oz.Z, bq(qZ), ep, rowsZ, np, s, OZ_BN);
  ep += rowsZ;
  if (r == cudaSuccess) r = oz_operand(oz.Bt1, bq(qT), ep, rowsT, no, s, OZ_BN);
  ep += rowsT;
  if (r == cudaSuccess) r = oz_operand(oz.Bt2, bq(qT), ep, rowsT, nv, s, OZ_BN);
  if (r == cudaSuccess) r = oz_init_attributes();
  if (r == cudaSuccess) r = cudaMemsetAsync(oz.err, 0, ptx::kErrInts * sizeof(int), st);
  if (r == cudaSuccess) r = launch_oz_slice_rows(st, sys.K, np, np, np, oz.K);
  if (r == cudaSuccess) r = launch_oz_slice_rows(st, sys.XvT, no, nv, no, oz.XvT);
  if (r == cudaSuccess) r = launch_oz_slice_rows(st, sys.Xv, nv, no, nv, oz.Xv);
  return r;
}

}  // namespace tddft

// ---------------------------------------------------------------------------
// C boundary: one emulated float64 product on device buffers
// ---------------------------------------------------------------------------
extern "C" tddft_status tddft_gemm_f64_emulated(int32_t M, int32_t N, int32_t K, const double *A,
                                                int64_t lda, const double *B, int64_t ldb,
                                                double *C, int64_t ldc, int32_t slices,
                                                void *stream) {
  using namespace tddft;
  if (M < 1 || N < 1 || K < 1 || !A || !B || !C) return TDDFT_ERR_INVALID_ARG;
  if (slices < kOzMinSlices || slices > kOzMaxSlices) return TDDFT_ERR_INVALID_ARG;
  if (lda < K || ldb < N || ldc < N) return TDDFT_ERR_SHAPE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int Kp = round_up(K, OZ_BK);
  // one scratch block: error ints, exponents, the two sliced operands
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t n_err = up(ptx::kErrInts * sizeof(int)), n_e = up(((size_t)M + N) * sizeof(int)),
               n_qa = up((size_t)M * slices * Kp * sizeof(__nv_bfloat16)),
               n_qb = up((size_t)N * slices * Kp * sizeof(__nv_bfloat16));
  char *ws = nullptr;
  cudaError_t e = scratch_alloc((void **)&ws, n_err + n_e + n_qa + n_qb, st);
  if (e != cudaSuccess) {
    cudaGetLastError();   // not left for a later check
    return e == cudaErrorMemoryAllocation ? TDDFT_ERR_NOMEM : TDDFT_ERR_CUDA;
  }
  int *err = (int *)ws, *ea = (int *)(ws + n_err), *eb = ea + M;
  __nv_bfloat16 *qa = (__nv_bfloat16 *)(ws + n_err + n_e),
                *qb = (__nv_bfloat16 *)(ws + n_err + n_e + n_qa);
  OzOperand oa, ob;
  e = oz_operand(oa, qa, ea, M, K, slices, OZ_BM);
  if (e == cudaSuccess) e = oz_operand(ob, qb, eb, N, K, slices, OZ_BN);
  if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, ptx::kErrInts * sizeof(int), st);
  if (e == cudaSuccess) e = launch_oz_slice_rows(st, A, lda, M, K, oa);
  if (e == cudaSuccess) e = launch_oz_slice_cols(st, B, ldb, K, N, ob);
  if (e == cudaSuccess) e = launch_gemm_oz(st, oa, ob, M, N, C, ldc, 0, err);
  int herr = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st);
  const cudaError_t ef = cudaFreeAsync(ws, st);
  if (e == cudaSuccess) e = ef;
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaErrorMemoryAllocation) return TDDFT_ERR_NOMEM;
  if (e != cudaSuccess) return TDDFT_ERR_CUDA;
  return herr ? TDDFT_ERR_TIMEOUT : TDDFT_OK;
}

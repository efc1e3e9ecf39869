// Float64 kernels of the matrix-free operator A(omega) z = z - chi0(omega) (K z)
// (Sec. 4.1) with chi0 . y applied by the steps of Sec. 4.2 (Fig. f:flops,
// Table t:flops), re-associated so that the vertex is read instead of the
// stored alpha object:
//   W_k(y)  = sum_{nu in block k} y^nu V_nu              (steps 1+2, per block)
//   beta    = W(y) X_occ                                 (steps 1+2)
//   a       = X_virt^T beta,  a^{FE} *= D_EF(omega)      (step 3 + denominator)
//   gamma   = X_virt a                                   (step 4)
//   n_mu    = sum_ab V_mu^{ab} (X_occ gamma^T)^{ab}      (step 5, blockdot.cu)
// Complex vectors are kept as two real planes; X, V and K are real, so only
// the D(omega) scaling mixes the planes.
#include <algorithm>
#include <type_traits>

#include "internal.h"

namespace tddft {

// ---------------------------------------------------------------------------
// The float64 kernels are bound by the FP64 pipe (about 2 FMA per clock and
// SM, so one warp-wide DFMA every 15 clocks per SM): loads, address
// arithmetic and L2 traffic are nearly free next to it.  What counts is that
// no DFMA is spent on padding and that every SM gets the same share, so the
// tiles are small, one output per lane where that fills the lanes, and all
// of them keep one summation order per output whatever the tile or the
// number of right-hand sides (host-driven, graph and batch launches of the
// same right-hand side give the same bits).  chi0 z of 3 vectors on 4 atoms:
// 406 -> 52 us; A z of 48 vectors on 24 atoms: 7.31 -> 3.95 ms (1.03 TFLOP/s
// of the measured 1.10); of 96 vectors on 64 atoms 89.5 -> 87.6 ms.
// ---------------------------------------------------------------------------
namespace {

// ---------------------------------------------------------------------------
// C[M x N] = A[M x K] . B[K x N], all row-major float64 (DFMA).
// A BM x BN tile per CTA; the four warps take one K quarter each
// (ceil(K/4) entries, staged per warp through registers into a double
// buffer in shared memory, no block barrier in the loop), and the quarters
// are added in order at the end: p0 + p1 + p2 + p3 (add: to C).  The K quarters depend on
// K alone, so every tile shape sums an output in the same order.
// A lane holds TM x TN outputs.  Every edge is bounds-checked.
// ---------------------------------------------------------------------------
constexpr int GF_WARPS = 4;

template <int BM, int BN, int TM, int TN, int KD>
__global__ void __launch_bounds__(32 * GF_WARPS)
    gemm_f64_kernel(int M, int N, int K, const double *__restrict__ A, int64_t lda,
                    const double *__restrict__ B, int64_t ldb, double *__restrict__ C, int64_t ldc,
                    const int *__restrict__ dcnt, int mul_m, int mul_n, int m_tiles, int add) {
  constexpr int LN = BN / TN;                               // lanes along N
  static_assert((BM / TM) * LN == 32, "one warp covers the tile");
  constexpr int LA = (BM * KD + 31) / 32, LB = (BN * KD + 31) / 32;   // loads per lane
  constexpr int AS = BM + 2, STAGE = KD * (AS + BN);
  constexpr int SM1 = GF_WARPS * 2 * STAGE, SM2 = GF_WARPS * BM * BN;
  __shared__ double smem[SM1 > SM2 ? SM1 : SM2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the M tile fastest: concurrent CTAs share their B columns in L2
  const int64_t m0 = (int64_t)(blockIdx.x % m_tiles) * BM;
  const int64_t n0 = (int64_t)(blockIdx.x / m_tiles) * BN;
  if (dcnt) {
    // graph replays: the live extent is read on the device
    const int c = *dcnt;
    if (mul_m) M = min(M, mul_m * c);
    if (mul_n) N = (int)min((int64_t)N, (int64_t)mul_n * c);
  }
  if (m0 >= M || n0 >= N) return;
  const int kq = (K + GF_WARPS - 1) / GF_WARPS;
  const int kb = min(K, warp * kq), len = min(K, kb + kq) - kb;
  A += kb;
  B += (int64_t)kb * ldb;
  double *st = smem + warp * 2 * STAGE;
  const int lm = (lane / LN) * TM, ln = (lane % LN) * TN;
  double acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;

  double ra[LA], rb[LB];
  auto load_regs = [&](int k0) {
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      const int idx = lane + 32 * l, i = idx / KD, kk = idx % KD;      // BM rows x KD
      ra[l] = (i < BM && m0 + i < M && k0 + kk < len) ? A[(m0 + i) * lda + k0 + kk] : 0.0;
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int idx = lane + 32 * l, kk = idx / BN, j = idx % BN;      // KD x BN columns
      rb[l] = (kk < KD && n0 + j < N && k0 + kk < len) ? B[(int64_t)(k0 + kk) * ldb + n0 + j] : 0.0;
    }
  };
  auto store_smem = [&](double *s) {
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      const int idx = lane + 32 * l;
      if (idx < BM * KD) s[(idx % KD) * AS + idx / KD] = ra[l];
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int idx = lane + 32 * l;
      if (idx < BN * KD) s[KD * AS + idx] = rb[l];
    }
  };
  if (len > 0) {
    load_regs(0);
    store_smem(st);
  }
  __syncwarp();
  for (int k0 = 0, buf = 0; k0 < len; k0 += KD, buf ^= 1) {
    const double *as = st + buf * STAGE + lm, *bs = st + buf * STAGE + KD * AS + ln;
    const bool more = k0 + KD < len;
    if (more) load_regs(k0 + KD);
    const int kn = min(KD, len - k0);
#pragma unroll 4
    for (int kk = 0; kk < kn; ++kk) {
      double a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = as[kk * AS + i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = bs[kk * BN + j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (more) store_smem(st + (buf ^ 1) * STAGE);
    __syncwarp();
  }
  __syncthreads();   // every warp is done with its stages: smem holds the quarters now
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) smem[(warp * BM + lm + i) * BN + ln + j] = acc[i][j];
  __syncthreads();
  for (int o = threadIdx.x; o < BM * BN; o += 32 * GF_WARPS) {
    const int i = o / BN, j = o % BN;
    if (m0 + i >= M || n0 + j >= N) continue;
    double s = smem[o];
#pragma unroll
    for (int w = 1; w < GF_WARPS; ++w) s += smem[w * BM * BN + o];
    double *c = C + (m0 + i) * ldc + n0 + j;
    *c = add ? *c + s : s;
  }
}

// ---------------------------------------------------------------------------
// W[c][k][ab] = sum_{nu in block k} Y[c][nu] * V_nu[ab]  (per block k, column c)
// One CTA per (block, group of VC columns); a thread owns one entry ab of the
// block's n_A x n_B (the pads of W are neither written nor read).
// ---------------------------------------------------------------------------
template <int VC>
__global__ void __launch_bounds__(256) vertex_contract(int nb, int ncols, int n_prod,
                                                       const int *__restrict__ aoff,
                                                       const int2 *__restrict__ blk_atoms,
                                                       const int *__restrict__ blk_ptr,
                                                       const int *__restrict__ blk_prod,
                                                       const double *__restrict__ Vpad,
                                                       const double *__restrict__ Y,
                                                       double *__restrict__ W,
                                                       const int *__restrict__ dcnt) {
  __shared__ double ys[32][VC];
  const int k = blockIdx.x;
  const int c0 = blockIdx.y * VC;
  if (dcnt) ncols = min(ncols, 2 * *dcnt);
  if (c0 >= ncols) return;
  const int t = threadIdx.x;
  const int2 AB = blk_atoms[k];
  const int nB = aoff[AB.y + 1] - aoff[AB.y], nAB = (aoff[AB.x + 1] - aoff[AB.x]) * nB;
  const int at = t < nAB ? (t / nB) * kMaxOrb + t % nB : 0;
  const int p0 = blk_ptr[k], p1 = blk_ptr[k + 1];
  double acc[VC];
#pragma unroll
  for (int c = 0; c < VC; ++c) acc[c] = 0.0;
  for (int q0 = p0; q0 < p1; q0 += 32) {
    __syncthreads();
    if (t < 32 * VC) {
      const int pp = t / VC, c = t % VC, q = q0 + pp;
      ys[pp][c] = (q < p1 && c0 + c < ncols) ? Y[(int64_t)(c0 + c) * n_prod + blk_prod[q]] : 0.0;
    }
    __syncthreads();
    if (t >= nAB) continue;
    const int qn = min(32, p1 - q0);
#pragma unroll 4
    for (int pp = 0; pp < qn; ++pp) {
      const double v = Vpad[(int64_t)(q0 + pp) * kBlk + at];
#pragma unroll
      for (int c = 0; c < VC; ++c) acc[c] = fma(ys[pp][c], v, acc[c]);
    }
  }
  if (t >= nAB) return;
#pragma unroll
  for (int c = 0; c < VC; ++c)
    if (c0 + c < ncols) W[((int64_t)(c0 + c) * nb + k) * kBlk + at] = acc[c];
}

// ---------------------------------------------------------------------------
// beta[aoff[A]+a][c][E] = sum over blocks touching atom A of
//   (W_k or W_k^T)[a][b] * Xo[aoff[B]+b][E]
// One thread per output (E fastest, then the column, then a): every lane is
// live whatever n_occ and n_A are, and the operands (W: one or two addresses
// per warp, X_occ: coalesced) come from L1 well inside the DFMA's 15 clocks.
// An entry's operands are loaded together, ahead of its chain.  (96 columns
// on 24 atoms: 1412 -> 415 us against 128 threads over E and 16 padded rows.)
// ---------------------------------------------------------------------------
constexpr int BT_THREADS = 256;

__global__ void __launch_bounds__(BT_THREADS) beta_kernel(
    int n_atoms, int ncols, int nb, int n_occ, const int *__restrict__ aoff,
    const int *__restrict__ adj_ptr, const int4 *__restrict__ adj, const double *__restrict__ W,
    const double *__restrict__ Xo, double *__restrict__ beta, const int *__restrict__ dcnt) {
  const int A = blockIdx.x % n_atoms;
  // ncols is the column stride of beta; nact the live columns
  const int nact = dcnt ? min(ncols, 2 * *dcnt) : ncols;
  const int aoA = aoff[A], nA = aoff[A + 1] - aoA;
  const int64_t i = (int64_t)(blockIdx.x / n_atoms) * BT_THREADS + threadIdx.x;
  if (nact <= 0 || i >= (int64_t)nA * nact * n_occ) return;
  const int64_t row = i / n_occ;
  const int E = (int)(i - row * n_occ);
  const int a = (int)(row / nact), c = (int)(row - (int64_t)a * nact);
  const double *Wc = W + (int64_t)c * nb * kBlk;
  double acc = 0.0;
  for (int e = adj_ptr[A]; e < adj_ptr[A + 1]; ++e) {
    const int4 ent = adj[e];   // (block, other atom, transposed)
    const int bo = aoff[ent.y], nB = aoff[ent.y + 1] - bo;
    const double *w = Wc + (int64_t)ent.x * kBlk + (ent.z ? a : a * kMaxOrb);
    const int ws = ent.z ? kMaxOrb : 1;
    const double *x = Xo + (int64_t)bo * n_occ + E;
    double wr[kMaxOrb], xr[kMaxOrb];
#pragma unroll
    for (int b = 0; b < kMaxOrb; ++b)
      if (b < nB) {
        wr[b] = w[b * ws];
        xr[b] = x[(int64_t)b * n_occ];
      }
#pragma unroll
    for (int b = 0; b < kMaxOrb; ++b)
      if (b < nB) acc = fma(wr[b], xr[b], acc);
  }
  beta[((int64_t)(aoA + a) * ncols + c) * n_occ + E] = acc;
}

// ---------------------------------------------------------------------------
// a[F][(2s, 2s+1)][E] *= D_EF(omega_s),
// D = n_E [1/(omega - Delta + i eps) - 1/(omega + Delta + i eps)],
// Delta = e_F - e_E  (eq. response-mat, both orderings of the pair merged).
// ---------------------------------------------------------------------------
// 1 / x for x > 0 of normal range (here x is a product of two sums of
// squares, between ~1e-10 and ~1e4): a float32 seed refined by two
// Newton-Raphson steps y <- y + y (1 - x y), each squaring the relative
// error (2^-23 -> 2^-46 -> below the float64 rounding).
__device__ __forceinline__ double recip_nr(double x) {
  float yf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"((float)x));
  double y = (double)yf;
  double e = fma(-x, y, 1.0);
  y = fma(y, e, y);
  e = fma(-x, y, 1.0);
  return fma(y, e, y);
}

// D(omega) of one (occupied E, virtual F) pair, Delta = e_F - e_E:
// occ [1/(omega - Delta + i eps) - 1/(omega + Delta + i eps)] from
// xm = omega - Delta and xp = omega + Delta; the two denominators share one
// reciprocal: 1/Am = Ap / (Am Ap), 1/Ap = Am / (Am Ap).
// (A refinement cycle of the emulated forms amplifies the last bit of D:
// 2 occ Delta / (z^2 - Delta^2) saves five FP64 operations and moves a
// converged spectrum by 3e-9, so the form is kept.)
__device__ __forceinline__ double2 d_factor(double w, double delta, double eps, double e2,
                                            double occ) {
  const double xm = w - delta, xp = w + delta;
  const double Am = fma(xm, xm, e2), Ap = fma(xp, xp, e2);
  const double q = occ * recip_nr(Am * Ap);
  const double im2 = Ap * q, ip2 = Am * q;   // occ / Am, occ / Ap
  return make_double2(xm * im2 - xp * ip2, eps * (ip2 - im2));
}

// D of consecutive columns: computed anew where the frequency changes (the
// three field directions of a frequency follow one another).
struct DOfColumn {
  double w;
  double2 d;
  __device__ __forceinline__ void at(bool first, double w_new, double delta, double eps, double e2,
                                     double occ) {
    if (!first && w_new == w) return;
    w = w_new;
    d = d_factor(w, delta, eps, e2, occ);
  }
};

// a[F][(2s, 2s+1)][E] *= D_EF(omega_s): one thread per (F, G columns s, E).
// Bound by its FP64 operations, about 21 for a D and 4 for a product with it
// (64 right-hand sides on 64 atoms: a D per column 247 us, per frequency 123).
template <int G>
__global__ void __launch_bounds__(128) dscale_kernel(
    int n_virt, int S, int n_occ, double occ_value, const double *__restrict__ energy,
    const double *__restrict__ omega, double eps, double e2, double *__restrict__ a,
    const int *__restrict__ dcnt) {
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  const int64_t row = i / n_occ;   // F * chunks + chunk
  const int chunks = (S + G - 1) / G;
  const int F = (int)(row / chunks), s0 = (int)(row - (int64_t)F * chunks) * G,
            E = (int)(i - row * n_occ);
  const int live = dcnt ? min(S, *dcnt) : S;
  if (F >= n_virt || s0 >= live) return;
  const double delta = energy[n_occ + F] - energy[E];
  double *at = a + ((int64_t)F * 2 * S + 2 * s0) * n_occ + E;
  double re[G], im[G];
#pragma unroll
  for (int q = 0; q < G; ++q)
    if (s0 + q < live) {
      re[q] = at[(int64_t)(2 * q) * n_occ];
      im[q] = at[(int64_t)(2 * q + 1) * n_occ];
    }
  DOfColumn D;
#pragma unroll
  for (int q = 0; q < G; ++q)
    if (s0 + q < live) {
      D.at(q == 0, omega[s0 + q], delta, eps, e2, occ_value);
      at[(int64_t)(2 * q) * n_occ] = D.d.x * re[q] - D.d.y * im[q];
      at[(int64_t)(2 * q + 1) * n_occ] = D.d.x * im[q] + D.d.y * re[q];
    }
}

__global__ void i2p_kernel(int n_rhs, int n, const double *__restrict__ in, double *__restrict__ out) {
  const int64_t total = (int64_t)n_rhs * n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / n, mu = i % n;
    out[(2 * r) * n + mu] = in[2 * i];
    out[(2 * r + 1) * n + mu] = in[2 * i + 1];
  }
}

__global__ void p2i_kernel(int n_rhs, int n, const double *__restrict__ in, double *__restrict__ out) {
  const int64_t total = (int64_t)n_rhs * n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / n, mu = i % n;
    out[2 * i] = in[(2 * r) * n + mu];
    out[2 * i + 1] = in[(2 * r + 1) * n + mu];
  }
}

// a[F][(2s, 2s+1)][E] = D_EF(omega_{(g0+s)/3}) * a3[F][(2k, 2k+1)][E], k = (g0+s) % 3:
// one thread per (F, frequency, E), its three columns or those of them in 0 .. S - 1
__global__ void __launch_bounds__(128) rhs_expand_kernel(
    int n_virt, int S, int n_occ, int g0, double occ_value, const double *__restrict__ energy,
    const double *__restrict__ omega_all, double eps, double e2, const double *__restrict__ a3,
    double *__restrict__ a) {
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  const int64_t row = i / n_occ;   // F * frequencies + frequency
  const int f0 = g0 / 3, nf = (g0 + S - 1) / 3 - f0 + 1;
  const int F = (int)(row / nf), f = f0 + (int)(row - (int64_t)F * nf), E = (int)(i - row * n_occ);
  if (F >= n_virt) return;
  const double2 d = d_factor(omega_all[f], energy[n_occ + F] - energy[E], eps, e2, occ_value);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int s = 3 * f + k - g0;
    if (s < 0 || s >= S) continue;
    const double *src = a3 + ((int64_t)F * 6 + 2 * k) * n_occ + E;
    double *dst = a + ((int64_t)F * 2 * S + 2 * s) * n_occ + E;
    const double re = src[0], im = src[n_occ];
    dst[0] = d.x * re - d.y * im;
    dst[n_occ] = d.x * im + d.y * re;
  }
}

// Z3 rows (d_0, 0, d_1, 0, d_2, 0)
__global__ void dipole_rows_kernel(int n_prod, const double *__restrict__ dip, double *__restrict__ Z3) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 3 * n_prod; i += gridDim.x * blockDim.x) {
    const int k = i / n_prod, mu = i % n_prod;
    Z3[(2 * k) * n_prod + mu] = dip[(int64_t)k * n_prod + mu];
    Z3[(2 * k + 1) * n_prod + mu] = 0.0;
  }
}

int grid_for(int64_t total, int threads) {
  int64_t g = (total + threads - 1) / threads;
  if (g > 152 * 32) g = 152 * 32;
  return (int)(g < 1 ? 1 : g);
}
}  // namespace

// The tile of a float64 GEMM: the one whose busiest SM has the fewest padded
// outputs, the pipe's only cost (smaller tiles read their operands more often,
// hence the few per cent against them).  6 x 280 x 280 takes 4 x 8 tiles on 70
// SMs (32 x 128 tiles ran on 3); 96 x 2960 x 2960 went from 3.08 ms in 72 CTAs
// of 32 x 128 to 1.51 ms in 279 of 32 x 32.
template <int BM, int BN, int TM, int TN, int KD>
struct GemmTile {
  static double cost(int M, int N, double penalty) {
    const double n = (double)((M + BM - 1) / BM) * ((N + BN - 1) / BN);
    const double sm = sm_count();
    return (n <= sm ? 1.0 : (double)(int64_t)((n + sm - 1) / sm)) * BM * BN * penalty;
  }
  static cudaError_t launch(cudaStream_t st, int M, int N, int K, const double *A, int64_t lda,
                            const double *B, int64_t ldb, double *C, int64_t ldc, const int *dcnt,
                            int mul_m, int mul_n, int add) {
    const int mt = (M + BM - 1) / BM;
    const int64_t n = (int64_t)mt * ((N + BN - 1) / BN);
    if (n > INT32_MAX) return cudaErrorInvalidConfiguration;
    gemm_f64_kernel<BM, BN, TM, TN, KD><<<(unsigned)n, 32 * GF_WARPS, 0, st>>>(
        M, N, K, A, lda, B, ldb, C, ldc, dcnt, mul_m, mul_n, mt, add);
    return cudaGetLastError();
  }
};

cudaError_t launch_gemm_f64(cudaStream_t st, int M, int N, int K, const double *A, int64_t lda,
                            const double *B, int64_t ldb, double *C, int64_t ldc,
                            const int *dcnt, int mul_m, int mul_n) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  using T32 = GemmTile<32, 32, 4, 8, 8>;
  using T16 = GemmTile<16, 16, 2, 4, 16>;
  using T8 = GemmTile<8, 8, 1, 2, 16>;
  using T4 = GemmTile<4, 8, 1, 1, 16>;
  const double c32 = T32::cost(M, N, 1.0), c16 = T16::cost(M, N, 1.03),
               c8 = T8::cost(M, N, 1.08), c4 = T4::cost(M, N, 1.15);
  // Above 8192 entries K goes in equal sections, one launch each, the later
  // ones added to C: no chain of the kernel's K quarters is longer than 2048,
  // whatever the tile or the live right-hand sides (K z of 9080 products, 1
  // vector 602 -> 608 us, 64 vectors 17.07 -> 17.08 ms).
  constexpr int kSection = 8192;
  const int sections = std::max(1, (K + kSection - 1) / kSection), ks = (K + sections - 1) / sections;
  auto go = [&](auto t) {
    for (int k0 = 0, sec = 0; sec < sections; ++sec, k0 += ks) {
      const cudaError_t e = decltype(t)::launch(st, M, N, std::min(ks, K - k0), A + k0, lda,
                                                B + (int64_t)k0 * ldb, ldb, C, ldc, dcnt, mul_m,
                                                mul_n, sec > 0);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  };
  if (c32 <= c16 && c32 <= c8 && c32 <= c4) return go(T32{});
  if (c16 <= c8 && c16 <= c4) return go(T16{});
  return c8 <= c4 ? go(T8{}) : go(T4{});
}

namespace {
// Columns per CTA of the vertex contraction: as many as leave about four
// CTAs per SM (a vertex block is then read once for all of them).
cudaError_t launch_vertex(cudaStream_t st, const DevSystem &sys, int ncols, const double *Y,
                          double *W, const int *dcnt) {
  auto go = [&](auto vc) {
    constexpr int VC = decltype(vc)::value;
    const dim3 grid(sys.n_blocks, (ncols + VC - 1) / VC);
    if (grid.y > 65535) return cudaErrorInvalidConfiguration;
    vertex_contract<VC><<<grid, 256, 0, st>>>(sys.n_blocks, ncols, sys.n_prod, sys.aoff,
                                              sys.blk_atoms, sys.blk_ptr, sys.blk_prod, sys.Vpad, Y,
                                              W, dcnt);
    return cudaGetLastError();
  };
  const int64_t want = 4 * (int64_t)sm_count();
  auto ctas = [&](int vc) { return (int64_t)sys.n_blocks * ((ncols + vc - 1) / vc); };
  if (ctas(8) >= want) return go(std::integral_constant<int, 8>{});
  if (ctas(4) >= want) return go(std::integral_constant<int, 4>{});
  if (ctas(2) >= want) return go(std::integral_constant<int, 2>{});
  return go(std::integral_constant<int, 1>{});
}

cudaError_t launch_beta(cudaStream_t st, const DevSystem &sys, int ncols, const double *W,
                        double *beta, const int *dcnt) {
  const int64_t per_atom =
      ((int64_t)kMaxOrb * ncols * sys.n_occ + BT_THREADS - 1) / BT_THREADS;
  if (per_atom * sys.n_atoms > INT32_MAX) return cudaErrorInvalidConfiguration;
  beta_kernel<<<(unsigned)(per_atom * sys.n_atoms), BT_THREADS, 0, st>>>(
      sys.n_atoms, ncols, sys.n_blocks, sys.n_occ, sys.aoff, sys.adj_ptr, sys.adj, W, sys.Xo, beta,
      dcnt);
  return cudaGetLastError();
}

cudaError_t launch_dscale(cudaStream_t st, const DevSystem &sys, int S, const double *omega,
                          double eps, double *a, const int *dcnt) {
  // six columns per thread (two D where the frequencies come in threes, three
  // where a group starts elsewhere), or three where that would leave SMs idle
  const int64_t per = (int64_t)sys.n_virt * sys.n_occ;
  const bool six = per * ((S + 5) / 6) >= (int64_t)sm_count() * 1024;
  const int64_t n = (per * (six ? (S + 5) / 6 : (S + 2) / 3) + 127) / 128;
  if (n > INT32_MAX) return cudaErrorInvalidConfiguration;
  auto *kernel = six ? dscale_kernel<6> : dscale_kernel<3>;
  kernel<<<(unsigned)n, 128, 0, st>>>(sys.n_virt, S, sys.n_occ, sys.occ_value, sys.energy, omega,
                                      eps, eps * eps, a, dcnt);
  return cudaGetLastError();
}

cudaError_t launch_rhs_expand(cudaStream_t st, const DevSystem &sys, int S, int g0,
                              const double *omega_all, double eps, const double *a3, double *a) {
  const int nf = (g0 + S - 1) / 3 - g0 / 3 + 1;
  const int64_t n = ((int64_t)sys.n_virt * nf * sys.n_occ + 127) / 128;
  if (n > INT32_MAX) return cudaErrorInvalidConfiguration;
  rhs_expand_kernel<<<(unsigned)n, 128, 0, st>>>(sys.n_virt, S, sys.n_occ, g0,
                                                 sys.occ_value, sys.energy, omega_all, eps,
                                                 eps * eps, a3, a);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_interleaved_to_planar(cudaStream_t st, int n_rhs, int n, const double *in,
                                         double *out) {
  i2p_kernel<<<grid_for((int64_t)n_rhs * n, 256), 256, 0, st>>>(n_rhs, n, in, out);
  return cudaGetLastError();
}

cudaError_t launch_planar_to_interleaved(cudaStream_t st, int n_rhs, int n, const double *in,
                                         double *out) {
  p2i_kernel<<<grid_for((int64_t)n_rhs * n, 256), 256, 0, st>>>(n_rhs, n, in, out);
  return cudaGetLastError();
}

namespace {
struct Scope {
  Timer *t;
  cudaStream_t st;
  int cls;
  double flops;
  cudaEvent_t a = nullptr;
  Scope(Timer *t_, cudaStream_t st_, int cls_, double fl) : t(t_), st(st_), cls(cls_), flops(fl) {
    if (t && t->on) t->begin(st, cls, &a);
  }
  ~Scope() {
    if (t && t->on) t->end(st, cls, a, flops);
  }
};
}  // namespace

namespace {
// Step 2 on the stored transition vertex, emulated float64: rows of Ysrc
// (n_rows columns y, row stride n_prod) gathered per atom and sliced, then
// beta^T[(c n_occ + E)][a] (into wk.beta) per atom on the tensor cores.
cudaError_t alpha_beta_emulated(cudaStream_t st, const DevSystem &sys, OpWork &wk, int n_rows,
                                const double *Ysrc, const int *dcnt) {
  AlphaRoute &ar = *wk.ar;
  cudaError_t err;
  {
    Scope sc(wk.timer, st, kcOzSlice, 0.0);
    err = launch_oz_slice_rows(st, Ysrc, sys.n_prod, n_rows, ar.kcat2, ar.oycat, dcnt, 2, ar.lcat);
    if (err != cudaSuccess) return err;
  }
  Scope sc(wk.timer, st, kcOzStep2, n_rows * ar.flops2);
  OzEpilogue eb;
  eb.mode = kOzBetaT;
  eb.C = wk.beta;
  eb.ldc = sys.n_orb;
  eb.aoff = sys.aoff;
  eb.n_occ = sys.n_occ;
  return launch_gemm_oz_ex(st, ar.oa2, ar.oycat, 0, n_rows, eb, ar.tiles2, ar.n_tiles2,
                           ar.max_nkb2, wk.oz->err, dcnt, 2);
}

// Transform 2 (X_virt a, a = wk.abuf [n_virt][ncols n_occ]) written per atom
// into Gcat, step 5 per atom, and Out = Zin - n (subtract) or n.
cudaError_t alpha_dot_emulated(cudaStream_t st, const DevSystem &sys, OpWork &wk, int ncols,
                               const double *Zin, int subtract, double *Out, const int *dcnt,
                               int timer_class) {
  AlphaRoute &ar = *wk.ar;
  OzWork &oz = *wk.oz;
  const int64_t ncolE = (int64_t)ncols * sys.n_occ;
  cudaError_t err;
  {
    Scope sc(wk.timer, st, kcOzSlice, 0.0);
    err = launch_oz_slice_cols(st, wk.abuf, ncolE, sys.n_virt, (int)ncolE, oz.Bt2, dcnt,
                               2 * sys.n_occ);
    if (err != cudaSuccess) return err;
  }
  {
    Scope sc(wk.timer, st, timer_class,
             timer_class == kcOzT2 ? 2.0 * sys.n_virt * (double)sys.n_orb * ncolE : 0.0);
    OzEpilogue eg;
    eg.mode = kOzGammaCat;
    eg.C = ar.gcat64;
    eg.ldc = ar.kcat5;
    eg.aoff = sys.aoff;
    eg.orb_atom = ar.orb_atom;
    eg.xoff5 = ar.xoff5;
    eg.n_occ = sys.n_occ;
    err = launch_gemm_oz_ex(st, oz.Xv, oz.Bt2, sys.n_orb, (int)ncolE, eg, nullptr, 0, 0, oz.err,
                            dcnt, 2 * sys.n_occ);
    if (err != cudaSuccess) return err;
  }
  {
    Scope sc(wk.timer, st, kcOzSlice, 0.0);
    err = launch_oz_slice_rows(st, ar.gcat64, ar.kcat5, ncols, ar.kcat5, ar.ogcat, dcnt, 2);
    if (err != cudaSuccess) return err;
  }
  {
    Scope sc(wk.timer, st, kcOzStep5, ncols * ar.flops5);
    OzEpilogue ep;
    ep.mode = kOzC;
    ep.C = ar.P2d;
    ep.ldc = ar.ldp;
    err = launch_gemm_oz_ex(st, ar.oa5, ar.ogcat, 0, ncols, ep, ar.tiles5, ar.n_tiles5,
                            ar.max_nkb5, oz.err, dcnt, 2);
    if (err != cudaSuccess) return err;
  }
  Scope sc(wk.timer, st, kcCombine, 0.0);
  return launch_alpha_combine(st, ar, ncols, sys.n_prod, true, Zin, subtract, Out, dcnt);
}

// chi0 (or A) with every dense product emulated in float64 and steps 2 and
// 5 on the stored transition vertex; Y = K z (kA) or z (kChi0).
cudaError_t apply_alpha_emulated(cudaStream_t st, const DevSystem &sys, OpWork &wk, int S,
                                 OpMode mode, double eps, const double *Y, const double *Zin,
                                 double *Out) {
  const int ncols = 2 * S;
  const int64_t ncolE = (int64_t)ncols * sys.n_occ;
  OzWork &oz = *wk.oz;
  cudaError_t err = alpha_beta_emulated(st, sys, wk, ncols, Y, wk.dcnt);
  if (err != cudaSuccess) return err;
  {
    Scope sc(wk.timer, st, kcOzSlice, 0.0);
    err = launch_oz_slice_rows(st, wk.beta, sys.n_orb, (int)ncolE, sys.n_orb, oz.Bt1, wk.dcnt,
                               2 * sys.n_occ);
    if (err != cudaSuccess) return err;
  }
  {
    Scope sc(wk.timer, st, kcOzT1, 2.0 * sys.n_virt * (double)sys.n_orb * ncolE);
    err = launch_gemm_oz(st, oz.XvT, oz.Bt1, sys.n_virt, (int)ncolE, wk.abuf, ncolE, 0, oz.err,
                         wk.dcnt, 2 * sys.n_occ);
    if (err != cudaSuccess) return err;
  }
  {
    Scope sc(wk.timer, st, kcDscale, 0.0);
    if ((err = launch_dscale(st, sys, S, wk.omega, eps, wk.abuf, wk.dcnt)) != cudaSuccess)
      return err;
  }
  return alpha_dot_emulated(st, sys, wk, ncols, Zin, mode == kA ? 1 : 0, Out, wk.dcnt, kcOzT2);
}
}  // namespace

cudaError_t launch_rhs_formation(cudaStream_t st, const DevSystem &sys, OpWork &wk, int S, int g0,
                                 const double *omega_all, double eps, double *Z3, double *a3,
                                 double *Out) {
  if (S <= 0) return cudaSuccess;
  if (S > wk.slots) return cudaErrorInvalidValue;
  const int np = sys.n_prod;
  cudaError_t err;
  Scope sc(wk.timer, st, kcRhs, 0.0);
  dipole_rows_kernel<<<grid_for(3 * (int64_t)np, 256), 256, 0, st>>>(np, sys.dip, Z3);
  if (wk.oz && wk.ar) {
    // emulated float64 on the stored transition vertex: beta(d_k) and
    // X_virt^T beta once, then per right-hand side D(omega), X_virt a, step 5
    Timer *saved = wk.timer;
    wk.timer = nullptr;
    const int n6 = 6 * sys.n_occ;
    err = alpha_beta_emulated(st, sys, wk, 6, Z3, nullptr);
    if (err == cudaSuccess)
      err = launch_oz_slice_rows(st, wk.beta, sys.n_orb, n6, sys.n_orb, wk.oz->Bt1);
    if (err == cudaSuccess)
      err = launch_gemm_oz(st, wk.oz->XvT, wk.oz->Bt1, sys.n_virt, n6, a3, n6, 0, wk.oz->err);
    if (err == cudaSuccess) err = launch_rhs_expand(st, sys, S, g0, omega_all, eps, a3, wk.abuf);
    if (err == cudaSuccess)
      err = alpha_dot_emulated(st, sys, wk, 2 * S, nullptr, 0, Out, nullptr, kcRhs);
    wk.timer = saved;
    return err;
  }
  // omega-independent part for the three directions (6 real columns)
  if ((err = launch_vertex(st, sys, 6, Z3, wk.W, nullptr)) != cudaSuccess) return err;
  if ((err = launch_beta(st, sys, 6, wk.W, wk.beta, nullptr)) != cudaSuccess) return err;
  const int n6 = 6 * sys.n_occ;
  if (wk.oz) {
    err = launch_oz_slice_cols(st, wk.beta, n6, sys.n_orb, n6, wk.oz->Bt1);
    if (err == cudaSuccess)
      err = launch_gemm_oz(st, wk.oz->XvT, wk.oz->Bt1, sys.n_virt, n6, a3, n6, 0, wk.oz->err);
  } else {
    err = launch_gemm_f64(st, sys.n_virt, n6, sys.n_orb, sys.XvT, sys.n_orb, wk.beta, n6, a3, n6);
  }
  if (err != cudaSuccess) return err;
  // per right-hand side: D(omega) a_k, X_virt a, block dot
  const int64_t ncolE = (int64_t)2 * S * sys.n_occ;
  if ((err = launch_rhs_expand(st, sys, S, g0, omega_all, eps, a3, wk.abuf)) != cudaSuccess)
    return err;
  if (wk.oz) {
    err = launch_oz_slice_cols(st, wk.abuf, ncolE, sys.n_virt, (int)ncolE, wk.oz->Bt2);
    if (err == cudaSuccess)
      err = launch_gemm_oz(st, wk.oz->Xv, wk.oz->Bt2, sys.n_orb, (int)ncolE, wk.gamma, ncolE, 0,
                           wk.oz->err);
  } else {
    err = launch_gemm_f64(st, sys.n_orb, (int)ncolE, sys.n_virt, sys.Xv, sys.n_virt, wk.abuf,
                          ncolE, wk.gamma, ncolE);
  }
  if (err != cudaSuccess) return err;
  return launch_block_dot(st, 2 * S, sys, sys.Vpad, sys.Xo, wk.gamma, nullptr, 0, Out,
                          nullptr);
}

cudaError_t launch_apply_operator(cudaStream_t st, const DevSystem &sys, OpWork &wk, int S,
                                  OpMode mode, double eps, const double *Zin, double *Out) {
  if (S <= 0) return cudaSuccess;
  if (S > wk.slots) return cudaErrorInvalidValue;
  const int ncols = 2 * S;
  const int np = sys.n_prod;
  cudaError_t err;
  const double *Y = Zin;
  if (mode == kKernel || mode == kA) {
    // Y = Z K  (K symmetric, so row c of Y is K z_c)
    double *Yout = (mode == kKernel) ? Out : wk.Y;
    if (wk.oz) {
      // emulated: (K z_c)_mu = sum_nu K[mu][nu] z_c[nu], stored transposed
      {
        Scope sc(wk.timer, st, kcOzSlice, 0.0);
        err = launch_oz_slice_rows(st, Zin, np, ncols, np, wk.oz->Z, wk.dcnt, 2);
      }
      Scope sc(wk.timer, st, kcOzK, 2.0 * ncols * (double)np * np);
      if (err == cudaSuccess)
        err = launch_gemm_oz(st, wk.oz->K, wk.oz->Z, np, ncols, Yout, np, 1, wk.oz->err, wk.dcnt,
                             2);
    } else {
      Scope sc(wk.timer, st, kcGemmK, 2.0 * ncols * (double)np * np);
      err = launch_gemm_f64(st, ncols, np, np, Zin, np, sys.K, np, Yout, np, wk.dcnt, 2, 0);
    }
    if (err != cudaSuccess || mode == kKernel) return err;
    Y = wk.Y;
  }
  if (wk.oz && wk.ar) return apply_alpha_emulated(st, sys, wk, S, mode, eps, Y, Zin, Out);
  {
    Scope sc(wk.timer, st, kcVertex, 2.0 * ncols * (double)kBlk * np);
    if ((err = launch_vertex(st, sys, ncols, Y, wk.W, wk.dcnt)) != cudaSuccess) return err;
  }
  {
    Scope sc(wk.timer, st, kcBeta, ncols * sys.sf.beta);
    if ((err = launch_beta(st, sys, ncols, wk.W, wk.beta, wk.dcnt)) != cudaSuccess) return err;
  }
  const int64_t ncolE = (int64_t)ncols * sys.n_occ;
  if (ncolE > INT32_MAX) return cudaErrorInvalidValue;
  const double tflops = 2.0 * sys.n_virt * (double)sys.n_orb * (double)ncolE;
  if (wk.oz) {
    // emulated: slices of the columns of beta (rows of beta^T), then X_virt^T beta
    {
      Scope sc(wk.timer, st, kcOzSlice, 0.0);
      err = launch_oz_slice_cols(st, wk.beta, ncolE, sys.n_orb, (int)ncolE, wk.oz->Bt1, wk.dcnt,
                                 2 * sys.n_occ);
    }
    Scope sc(wk.timer, st, kcOzT1, tflops);
    if (err == cudaSuccess)
      err = launch_gemm_oz(st, wk.oz->XvT, wk.oz->Bt1, sys.n_virt, (int)ncolE, wk.abuf, ncolE, 0,
                           wk.oz->err, wk.dcnt, 2 * sys.n_occ);
    if (err != cudaSuccess) return err;
  } else {
    Scope sc(wk.timer, st, kcGemmT1, tflops);
    err = launch_gemm_f64(st, sys.n_virt, (int)ncolE, sys.n_orb, sys.XvT, sys.n_orb, wk.beta,
                          ncolE, wk.abuf, ncolE, wk.dcnt, 0, 2 * sys.n_occ);
    if (err != cudaSuccess) return err;
  }
  {
    Scope sc(wk.timer, st, kcDscale, 0.0);
    if ((err = launch_dscale(st, sys, S, wk.omega, eps, wk.abuf, wk.dcnt)) != cudaSuccess)
      return err;
  }
  if (wk.oz) {
    {
      Scope sc(wk.timer, st, kcOzSlice, 0.0);
      err = launch_oz_slice_cols(st, wk.abuf, ncolE, sys.n_virt, (int)ncolE, wk.oz->Bt2, wk.dcnt,
                                 2 * sys.n_occ);
    }
    Scope sc(wk.timer, st, kcOzT2, tflops);
    if (err == cudaSuccess)
      err = launch_gemm_oz(st, wk.oz->Xv, wk.oz->Bt2, sys.n_orb, (int)ncolE, wk.gamma, ncolE, 0,
                           wk.oz->err, wk.dcnt, 2 * sys.n_occ);
    if (err != cudaSuccess) return err;
  } else {
    Scope sc(wk.timer, st, kcGemmT2, tflops);
    err = launch_gemm_f64(st, sys.n_orb, (int)ncolE, sys.n_virt, sys.Xv, sys.n_virt, wk.abuf,
                          ncolE, wk.gamma, ncolE, wk.dcnt, 0, 2 * sys.n_occ);
    if (err != cudaSuccess) return err;
  }
  {
    Scope sc(wk.timer, st, kcSddmm, ncols * sys.sf.dot);
    err = launch_block_dot(st, ncols, sys, sys.Vpad, sys.Xo, wk.gamma, Zin,
                           mode == kA ? 1 : 0, Out, wk.dcnt);
    if (err != cudaSuccess) return err;
  }
  return cudaSuccess;
}

}  // namespace tddft

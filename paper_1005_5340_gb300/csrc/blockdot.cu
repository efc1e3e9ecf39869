// Step 5 of the chi0 product (Table t:flops): on every orbital block
// k = (A, B) and for every real column c,
//   G[a][b] = sum_E Xo[A+a][E] gamma_c[B+b][E]   (+ gamma_c[A+a][E] Xo[B+b][E] if A != B)
//   n_c[mu] = sum_ab V_mu[a][b] G[a][b]            for the products mu of block k
//   Out[c][mu] = Zin[c][mu] - n_c[mu]  (A operator)  or  n_c[mu]  (chi0 only).
// One CTA handles one block and BC columns.  The kernel is bound by the FP64
// pipe, so both phases spend no DFMA on padding: lanes run over the compact
// n_A x n_B entries of G (8 / BC warps per column), and the dots give each
// (product, column) to four lanes, a quarter of the entries each, so that
// only two additions per lane reduce them.  Shared-memory operands feed one
// DFMA each, which the pipe's 15 clocks per warp and SM hide.  (96 columns on 24
// atoms: 838 -> 562 us; 384 columns on 4 atoms: 151 -> 65 us per launch.)
// float64 throughout; gamma is laid out [n_orb][ncols][n_occ].
#include <type_traits>

#include "internal.h"

namespace tddft {
namespace {

constexpr int BD_E = 16;             // occupied states staged per step
constexpr int BD_GS = kBlk + 4;      // row stride of G (bank-conflict free over 8 columns)

template <int BC>
__global__ void __launch_bounds__(256) block_dot_kernel(
    int ncols, int n_occ, int n_prod, const int *__restrict__ aoff,
    const int2 *__restrict__ blk_atoms, const int *__restrict__ blk_ptr,
    const int *__restrict__ blk_prod, const double *__restrict__ Vpad,
    const double *__restrict__ Xo, const double *__restrict__ gamma,
    const double *__restrict__ Zin, int subtract, double *__restrict__ Out,
    const int *__restrict__ dcnt) {
  constexpr int WPC = 8 / BC;        // warps per column
  constexpr int GE = 2 * BC * BD_E * (kMaxOrb + 1);
  __shared__ double XA[BD_E][kMaxOrb + 1], XB[BD_E][kMaxOrb + 1];
  // gamma slices of the A and B rows, [2][BC][BD_E][kMaxOrb + 1], reused for G
  __shared__ double gbuf[GE > BC * BD_GS ? GE : BC * BD_GS];
  __shared__ int vat[kBlk];          // entry ab of the compact block in a padded vertex block
  auto gA = [&](int c, int e, int r) -> double & {
    return gbuf[(c * BD_E + e) * (kMaxOrb + 1) + r];
  };
  auto gB = [&](int c, int e, int r) -> double & {
    return gbuf[((BC + c) * BD_E + e) * (kMaxOrb + 1) + r];
  };
  const int k = blockIdx.x;
  const int c0 = blockIdx.y * BC;
  const int nact = dcnt ? min(ncols, 2 * *dcnt) : ncols;   // ncols: stride; nact: live
  if (c0 >= nact) return;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int2 AB = blk_atoms[k];
  const int aoA = aoff[AB.x], nA = aoff[AB.x + 1] - aoA;
  const int aoB = aoff[AB.y], nB = aoff[AB.y + 1] - aoB;
  const int nAB = nA * nB;
  const bool bilocal = AB.x != AB.y;
  if (t < nAB) vat[t] = (t / nB) * kMaxOrb + t % nB;
  // this thread's column and entries w0 + 32 WPC r of G
  const int cl = warp / WPC, w0 = (warp % WPC) * 32;
  const bool col = c0 + cl < nact;
  int ra[BC], rb[BC];
  double G[BC];
#pragma unroll
  for (int r = 0; r < BC; ++r) {
    const int ab = min(w0 + 32 * WPC * r + lane, nAB - 1);
    ra[r] = ab / nB;
    rb[r] = ab % nB;
    G[r] = 0.0;
  }
  for (int E0 = 0; E0 < n_occ; E0 += BD_E) {
    __syncthreads();
    {
      const int e = t / kMaxOrb, r = t % kMaxOrb, E = E0 + e;   // BD_E x kMaxOrb = 256 threads
      XA[e][r] = (r < nA && E < n_occ) ? Xo[(int64_t)(aoA + r) * n_occ + E] : 0.0;
      XB[e][r] = (r < nB && E < n_occ) ? Xo[(int64_t)(aoB + r) * n_occ + E] : 0.0;
    }
#pragma unroll
    for (int i = t; i < BC * BD_E * kMaxOrb; i += 256) {
      // e fastest: contiguous in gamma
      const int c = i / (BD_E * kMaxOrb), rem = i % (BD_E * kMaxOrb);
      const int r = rem / BD_E, e = rem % BD_E, E = E0 + e, cc = c0 + c;
      const bool live = cc < nact && E < n_occ;
      gA(c, e, r) = live && r < nA ? gamma[((int64_t)(aoA + r) * ncols + cc) * n_occ + E] : 0.0;
      gB(c, e, r) = live && r < nB ? gamma[((int64_t)(aoB + r) * ncols + cc) * n_occ + E] : 0.0;
    }
    __syncthreads();
    if (!col) continue;
    const int en = min(BD_E, n_occ - E0);
#pragma unroll 2
    for (int e = 0; e < en; ++e)
#pragma unroll
      for (int r = 0; r < BC; ++r)
        if (w0 + 32 * WPC * r < nAB) {   // the same for the whole warp
          G[r] = fma(XA[e][ra[r]], gB(cl, e, rb[r]), G[r]);
          if (bilocal) G[r] = fma(gA(cl, e, ra[r]), XB[e][rb[r]], G[r]);
        }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < BC; ++r) {
    const int ab = w0 + 32 * WPC * r + lane;
    if (ab < nAB) gbuf[cl * BD_GS + ab] = G[r];
  }
  __syncthreads();
  // dots: lanes 4 o .. 4 o + 3 take output o = (product, column), column fastest
  const int p0 = blk_ptr[k], total = (blk_ptr[k + 1] - p0) * BC;
  const int sub = t & 3;
  for (int base = 0; base < total; base += 64) {
    const int o = base + (t >> 2), c = o % BC, q = p0 + o / BC;
    const bool live = o < total && c0 + c < nact;
    double s = 0.0;
    if (live) {
      const double *v = Vpad + (int64_t)q * kBlk, *g = gbuf + c * BD_GS;
#pragma unroll 8
      for (int ab = sub; ab < nAB; ab += 4) s = fma(v[vat[ab]], g[ab], s);
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (live && sub == 0) {
      const int64_t at = (int64_t)(c0 + c) * n_prod + blk_prod[q];
      Out[at] = subtract ? Zin[at] - s : s;
    }
  }
}

}  // namespace

cudaError_t launch_block_dot(cudaStream_t st, int ncols, const DevSystem &sys,
                             const double *Vpad, const double *Xo, const double *gamma,
                             const double *Zin, int subtract, double *Out, const int *dcnt) {
  auto go = [&](auto bc) {
    constexpr int BC = decltype(bc)::value;
    const dim3 grid(sys.n_blocks, (ncols + BC - 1) / BC);
    if (grid.y > 65535) return cudaErrorInvalidConfiguration;
    block_dot_kernel<BC><<<grid, 256, 0, st>>>(ncols, sys.n_occ, sys.n_prod, sys.aoff,
                                               sys.blk_atoms, sys.blk_ptr, sys.blk_prod, Vpad, Xo,
                                               gamma, Zin, subtract, Out, dcnt);
    return cudaGetLastError();
  };
  // as many columns per CTA as leave about four CTAs per SM
  auto ctas = [&](int bc) { return (int64_t)sys.n_blocks * ((ncols + bc - 1) / bc); };
  const int64_t want = 4 * (int64_t)sm_count();
  if (ctas(8) >= want) return go(std::integral_constant<int, 8>{});
  if (ctas(4) >= want) return go(std::integral_constant<int, 4>{});
  if (ctas(2) >= want) return go(std::integral_constant<int, 2>{});
  return go(std::integral_constant<int, 1>{});
}

}  // namespace tddft

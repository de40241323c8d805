// One 4 x 8 tile of a small FP64 complex product, by one CTA of eight warps.
//
// An FP64 instruction occupies a partition's pipe for 64 clocks here, so a 16 x 16 tile of one
// CTA takes K x 512 clocks (13 us at K = 50) while the other SMs of a small product stand idle.
// A 4 x 8 tile is one output a lane, its K range shared by the eight warps and added up in a fixed
// order: K x 64 clocks, and eight times as many CTAs. Each operand element is used by one warp only,
// so the operands come straight from L1 / L2, eight steps of K in flight. On average
// over a sequence's calls at n = 50, m = 18: products 4.2 us, 16.3 with 16 x 16 tiles, Gram matrices
// 3.9 and 11.8; products of m <= 140: 28.8 and 46; eight of m = 68 to 160 in one launch: 140 us, 176
// with 32 x 32 tiles (98 at the pipe's rate).
#pragma once
#include "gevp_internal.cuh"

namespace gevp {
namespace {

constexpr int ZS_M = 4, ZS_N = 8, ZS_WARPS = 8, ZS_THREADS = 32 * ZS_WARPS;
// cost of a tile besides its K steps (first loads, the sum over the warps, the store), in the unit
// of the tile rules (an output's K step: 2 clocks)
constexpr double kZsOverhead = 750.0;

// sum over k in [kb, ke) of op(A)(gm, k) op(B)(k, gn) for lane (gm = m0 + lane / 8, gn = n0 + lane % 8);
// threads t < 64 return component t / 32 of lane t % 32's sum. part: [ZS_WARPS][64] of the CTA.
template <int OPA, int OPB>
__device__ __forceinline__ double zsmall_tile(int M, int N, const double2* A, int64_t lda, const double2* B,
                                              int64_t ldb, int maskB, int m0, int n0, int kb, int ke,
                                              double (*part)[64]) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int gm = min(m0 + lane / ZS_N, M - 1), gn = min(n0 + lane % ZS_N, N - 1);
  const int per = (max(ke - kb, 0) + ZS_WARPS - 1) / ZS_WARPS;
  const int k1 = min(ke, kb + (warp + 1) * per);
  double2 acc = make_double2(0.0, 0.0);
  for (int k = kb + warp * per; k < k1; k += 8) {
    double2 a[8], b[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int kk = min(k + u, k1 - 1);
      a[u] = OPA == 0 ? A[(int64_t)gm * lda + kk] : A[(int64_t)kk * lda + gm];
      b[u] = OPB == 0 ? B[(int64_t)kk * ldb + gn] : B[(int64_t)gn * ldb + kk];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (k + u < k1) {
        double2 x = OPA == 0 ? a[u] : zconj(a[u]), y = OPB == 0 ? b[u] : zconj(b[u]);
        if (maskB) {
          if (k + u < gn) y = make_double2(0.0, 0.0);
          else if (k + u == gn) y = zscale(y, 0.5);
        }
        zfma(acc, x, y);
      }
    }
  }
  part[warp][lane] = acc.x;
  part[warp][32 + lane] = acc.y;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 64) {
    s = part[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < ZS_WARPS; ++w) s += part[w][threadIdx.x];
  }
  return s;
}
__device__ __forceinline__ double zsmall_tile(int opA, int opB, int M, int N, const double2* A, int64_t lda,
                                              const double2* B, int64_t ldb, int maskB, int m0, int n0, int kb,
                                              int ke, double (*part)[64]) {
  if (opA == 0)
    return opB == 0 ? zsmall_tile<0, 0>(M, N, A, lda, B, ldb, maskB, m0, n0, kb, ke, part)
                    : zsmall_tile<0, 1>(M, N, A, lda, B, ldb, 0, m0, n0, kb, ke, part);
  return opB == 0 ? zsmall_tile<1, 0>(M, N, A, lda, B, ldb, maskB, m0, n0, kb, ke, part)
                  : zsmall_tile<1, 1>(M, N, A, lda, B, ldb, 0, m0, n0, kb, ke, part);
}

}  // namespace
}  // namespace gevp

// Chebyshev filter steps on the tcgen05 tensor cores.
//
// Complex product by the three-real-product (Gauss) formula with FP32 accumulation in TMEM:
//   T1 = Cr Yr,  T2 = Ci Yi,  T3 = (Cr + Ci)(Yr + Yi),   Re = T1 - T2,  Im = T3 - T1 - T2,
// followed by the scaled three-term recurrence Y_{j+1} = alpha C Y_j + beta Y_j + gamma Y_{j-1}
// with the recurrence state kept in FP32.
//
// Precision. Each real operand x is stored as nsplit BF16 pieces x = x0 + x1 + x2 + ...
// (x0 = bf16(x), x1 = bf16(x - x0), ...). nsplit = 1 is the BF16 filter. nsplit = 3 keeps
// the six products x_a y_b with a + b <= 2 (about 24 significant bits, FP32 class), accumulated in
// the same TMEM accumulators. A pipeline stage then holds the three pieces of one part (re, im or
// re + im) of C and of Y for one K block, which serve all six products of that part: half the
// bytes through L2 and shared memory of a stage per product pair (n = 2048, m = 140, six
// products: 27.8 us a step; 31.5 with the operands of one piece pair a stage). With the pairs and the
// unrolled issue by three threads: 26.7 us, n = 4096, m = 250: 118 to 95.5 us (67 clocks an MMA at the
// tensor cores' rate, 78 here, 96 before).
//
// Layout (all K-major, as the MMA wants both operands): the planes of C are n_pad x n_pad
// row-major BF16 (row i = output row, contiguous k); the block Y is stored transposed,
// Y^T planes ncols x n_pad (row c = column c of Y, contiguous k), and so is the FP32 state.
// Padding rows/columns are zero, so the padded K contributes nothing.
//
// A pair of CTAs (cta_group::2): 256 rows of C (UMMA M = 256) x one chunk of up to 160 columns of Y
// (N), over a slice of K (split-K across grid.z, so that n = 2048 still fills the 152 SMs). Each CTA
// holds its 128 rows of C and half of the columns, so Y is loaded once a pair: n = 4100, m = 211 in
// BF16, bound by the loads of 90 KB for 12 MMAs, 43.3 to 32.1 us a step. Warp 0 lane 0 of each CTA
// issues its TMA loads (128B-swizzled boxes, a pipeline of two or three stages), one lane of warps 1
// to 3 of the leader the MMAs of both CTAs, a warp for each of the three TMEM accumulators of N
// columns; then all four warps read TMEM back (warp w owns lanes 32w..32w+31) and write the FP32
// partial product transposed (coalesced along rows). A second kernel sums the split-K partials in a
// fixed order (deterministic) and applies the recurrence.
//
// Every mbarrier wait is bounded; on expiry the kernel records an error code, skips the
// rest of its work, frees its TMEM and returns.
#include "gevp_internal.cuh"
#include "tc_ptx.cuh"
#include <cuda.h>
#include <algorithm>
#include <cstring>
#include <vector>

namespace gevp {

namespace {

constexpr int TM = 128;
constexpr int TK = 64;
constexpr int STAGES = 3;          // at most; two for the widest tiles
constexpr int NFULL = 6;           // barriers of arrived stages: a multiple of 3 and of the stages
constexpr size_t TC_SMEM = 231424;  // dynamic shared memory: one CTA an SM
constexpr int NMAX = 160;
constexpr int MAXSPLIT = 3;
constexpr int MAXSEG = 6;

struct TcMaps {
  CUtensorMap a[MAXSPLIT * 3];   // C planes: [piece][re, im, re+im]
  CUtensorMap b[MAXSPLIT * 3];   // Y^T planes
};

struct TcParams {
  int n_pad;
  int nchunk;
  int kb_per_split;
  int ncols_pad;      // rows of the Y^T planes (multiple of nchunk)
  int nsplit;         // pieces per operand
  uint32_t tmem_cols; // power of two >= 3 * nchunk
  int nst;            // pipeline stages (tc_stages)
  float2* ws;         // [ksplit][ncols_pad][n_pad]
  int* err;
};

// One output tile of a pair of CTAs: rows m0..m0+255 of C times columns c0..c0+nchunk-1 of the block
// over K slice z, this CTA's (rank of the pair) the 128 rows from m0 + 128 rank. amaps/bmaps: the
// tensor maps of the pieces of C and of the block (kernel parameter space or global memory).
__device__ __forceinline__ void tc_tile(const CUtensorMap* amaps, const CUtensorMap* bmaps, const TcParams& p,
                                        int m0, int c0, int z, int rank) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[NFULL], empty[STAGES], done;
  __shared__ uint32_t tmem_sh;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int nkb_total = p.n_pad / TK;
  const int kb0 = z * p.kb_per_split;
  const int kb1 = min(kb0 + p.kb_per_split, nkb_total);
  const int nkb = max(0, kb1 - kb0);
  // a stage: one K block, either the three parts of a single piece, or the pieces of one part
  const bool by_part = p.nsplit > 1;
  const int group = by_part ? 3 : 1, boxes = by_part ? p.nsplit : 3;
  const int niter = nkb * group;
  const uint32_t a_bytes = TM * TK * 2;
  const uint32_t b_bytes = (uint32_t)(p.nchunk / 2) * TK * 2;   // half of the columns in each CTA
  const uint32_t stage_bytes = 3 * a_bytes + 3 * b_bytes;
  auto tile = [&](int s, int which) -> uint8_t* {
    uint8_t* base = smem + (size_t)s * stage_bytes;
    return which < 3 ? base + which * a_bytes : base + 3 * a_bytes + (which - 3) * b_bytes;
  };
  if (threadIdx.x == 0) {
    for (int s = 0; s < NFULL; ++s) mbar_init(&full[s], 1);
    for (int s = 0; s < STAGES; ++s) mbar_init(&empty[s], by_part ? 1 : 3);   // a commit of each issuing warp
    mbar_init(&done, 3);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  pair_sync();   // both CTAs run (the allocation takes both), their barriers are initialised
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_sh)),
                 "r"(p.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_sh;
  const int row0 = m0 + TM * rank;

  if (warp == 0 && lane == 0) {
    int issued = 0;
    for (int i = 0; i < niter; ++i, issued = i) {
      const int s = i % p.nst;
      if (i >= p.nst && !pair_wait(&empty[s], ((uint32_t)(i / p.nst) & 1u) ^ 1u, p.err, 1)) break;
      if (rank == 0) mbar_expect_tx(&full[i % NFULL], 2u * (uint32_t)boxes * (a_bytes + b_bytes));
      const uint32_t bar = pair_mapa(su32(&full[i % NFULL]), 0);
      const int part = i % group;
      const int kx = (kb0 + i / group) * TK;
      for (int w = 0; w < boxes; ++w) {
        const int map = by_part ? 3 * w + part : w;
        pair_tma_2d(tile(s, w), amaps + map, kx, row0, bar);
        pair_tma_2d(tile(s, 3 + w), bmaps + map, kx, c0 + rank * (p.nchunk / 2), bar);
      }
    }
    // every copy issued has landed before the CTAs leave (bounded; immediate unless a wait
    // elsewhere gave up)
    if (rank == 0)
      for (int i = max(0, issued - p.nst); i < issued; ++i)
        mbar_wait(&full[i % NFULL], (uint32_t)(i / NFULL) & 1u, p.err, 4);
    // and so has every release of a stage (an arrival after this CTA has left would count on a barrier of
    // the next one)
    for (int i = max(0, issued - p.nst); i < issued; ++i)
      if (!pair_wait(&empty[i % p.nst], (uint32_t)(i / p.nst) & 1u, p.err, 5)) break;
  } else if (warp > 0 && lane == 0 && rank == 0) {
    // Warp 1 + part issues that part's MMAs, so that three threads share the issue: one alone takes
    // 80 clocks an MMA, more than the 72 of a 144-wide tile. The order within an accumulator is one
    // thread's. Iteration i signals full[i % 6]: by parts, that barrier is always the same warp's (6 is
    // a multiple of 3), so the warp sees each of its phases, and none is waited for a phase early.
    const uint32_t idesc = idesc_bf16(2 * TM, p.nchunk);
    const int part = warp - 1;
    const uint32_t dt = tmem + (uint32_t)(part * p.nchunk);
    for (int i = by_part ? part : 0; i < niter; i += group) {
      const int s = i % p.nst;
      if (!mbar_wait(&full[i % NFULL], (uint32_t)(i / NFULL) & 1u, p.err, 2)) break;
      fence_after();
      const uint32_t acc0 = i >= group ? 1u : 0u;
      if (!by_part) {
        const uint64_t a = sdesc(su32(tile(s, part))), b = sdesc(su32(tile(s, 3 + part)));
#pragma unroll
        for (int kk = 0; kk < TK / 16; ++kk) {
          const uint64_t off = (uint64_t)(kk * 32) >> 4;   // 16 bf16 = 32 B along K inside the swizzle row
          pair_umma(dt, a + off, b + off, idesc, kk > 0 ? 1u : acc0);
        }
      } else {
        const uint64_t d[3] = {sdesc(su32(tile(s, 0))), sdesc(su32(tile(s, 1))), sdesc(su32(tile(s, 2)))};
        const uint64_t e[3] = {sdesc(su32(tile(s, 3))), sdesc(su32(tile(s, 4))), sdesc(su32(tile(s, 5)))};
#pragma unroll
        for (int seg = 0; seg < MAXSEG; ++seg) {
          // (a piece, b piece) with a + b <= nsplit - 1
          constexpr int kA[MAXSEG] = {0, 0, 1, 0, 1, 2}, kB[MAXSEG] = {0, 1, 0, 2, 1, 0};
          if (seg >= 3 && p.nsplit < 3) break;
#pragma unroll
          for (int kk = 0; kk < TK / 16; ++kk) {
            const uint64_t off = (uint64_t)(kk * 32) >> 4;
            pair_umma(dt, d[kA[seg]] + off, e[kB[seg]] + off, idesc, (seg > 0 || kk > 0) ? 1u : acc0);
          }
        }
      }
      pair_commit(&empty[s]);
    }
    pair_commit(&done);
  }
  __syncwarp();
  const bool have = __all_sync(0xffffffffu, pair_wait(&done, 0, p.err, 3) ? 1 : 0) != 0;
  fence_after();
  const int row = row0 + warp * 32 + lane;
  float2* out = p.ws + (size_t)z * p.ncols_pad * p.n_pad;
  const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
  for (int cc = 0; cc < p.nchunk; cc += 16) {
    uint32_t t1[16], t2[16], t3[16];
    if (have && niter > 0) {
      tmem_ld16(tmem + lane_base + (uint32_t)cc, t1);
      tmem_ld16(tmem + lane_base + (uint32_t)(p.nchunk + cc), t2);
      tmem_ld16(tmem + lane_base + (uint32_t)(2 * p.nchunk + cc), t3);
      tmem_wait_ld();
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j) t1[j] = t2[j] = t3[j] = 0u;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      float a = __uint_as_float(t1[j]), b = __uint_as_float(t2[j]), c = __uint_as_float(t3[j]);
      int col = c0 + cc + j;
      if (row < p.n_pad && col < p.ncols_pad) out[(size_t)col * p.n_pad + row] = make_float2(a - b, c - a - b);
    }
  }
  fence_before();
  __syncthreads();
  pair_sync();   // neither CTA leaves while the other's MMAs or copies may touch it
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
  pair_sync();
}

__global__ void __launch_bounds__(128, 1) __cluster_dims__(2, 1, 1)
    cheb_tc_kernel(const __grid_constant__ TcMaps maps, const __grid_constant__ TcParams p) {
  tc_tile(maps.a, maps.b, p, (int)(blockIdx.x >> 1) * 2 * TM, blockIdx.y * p.nchunk, blockIdx.z, blockIdx.x & 1);
}

// v = hi + lo to about 2^-48, hi the leading 24 bits of v (truncated), from the IEEE-754 fields: an
// FP64 conversion or addition takes 64 times an FP32 one here, and the pieces of a matrix need
// ten of them per value.
struct FPair {
  float hi, lo;
};
__device__ __forceinline__ FPair fsplit(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int ef = (int)((b >> 52) & 0x7FF) - 896;   // the FP32 exponent field
  FPair r;
  if (ef <= 52 || ef >= 255) {   // 0, tiny (the low part would be subnormal), too large, Inf or NaN
    r.hi = (float)v;
    r.lo = 0.f;
    return r;
  }
  const uint32_t sign = (uint32_t)(b >> 32) & 0x80000000u;
  r.hi = __uint_as_float(sign | (uint32_t)ef << 23 | ((uint32_t)(b >> 29) & 0x7FFFFFu));
  const uint32_t m = (uint32_t)b & 0x1FFFFFFFu;   // 29 bits, unit 2^(ef - 179)
  r.lo = (float)(int)m * __uint_as_float(sign | (uint32_t)(ef - 52) << 23);
  return r;
}
// the sum of two such values (exact first sum, rounded low part)
__device__ __forceinline__ FPair fsum(FPair a, FPair b) {
  FPair r;
  const float s = a.hi + b.hi, t = s - a.hi;
  const float lo = ((a.hi - (s - t)) + (b.hi - t)) + (a.lo + b.lo);
  r.hi = s + lo;   // (after a cancellation the low part is not below half a unit of s)
  r.lo = lo - (r.hi - s);
  return r;
}

// nsplit BF16 pieces of two neighbouring values, one 4-byte store per piece (piece p at base + p ps):
// each piece is the nearest BF16 of the remainder, and the remainder minus it is exact in FP32
// (Sterbenz); the low part, below half a unit of hi, decides where hi alone is a tie and joins
// after the first piece
__device__ __forceinline__ void store_pieces(const FPair& a, const FPair& b, int nsplit, __nv_bfloat16* at, size_t ps) {
  auto first = [](const FPair& v) {
    uint32_t b = __float_as_uint(v.hi);
    if ((b & 0xFFFFu) == 0x8000u && v.lo != 0.f) b += (__float_as_uint(v.lo) ^ b) >> 31 ? ~0u : 1u;
    return __float2bfloat16_rn(__uint_as_float(b));
  };
  __nv_bfloat16 ha = first(a), hb = first(b);
  float ra = (a.hi - __bfloat162float(ha)) + a.lo, rb = (b.hi - __bfloat162float(hb)) + b.lo;
  for (int p = 0;; ++p) {
    __nv_bfloat162 v;
    v.x = ha;
    v.y = hb;
    *(__nv_bfloat162*)(at + (size_t)p * ps) = v;
    if (p + 1 >= nsplit) break;
    ha = __float2bfloat16_rn(ra);
    hb = __float2bfloat16_rn(rb);
    ra -= __bfloat162float(ha);
    rb -= __bfloat162float(hb);
  }
}

struct YPlanes {
  __nv_bfloat16* base;   // [piece][part re, im, re+im][ncols_pad][n_pad]
  size_t plane;          // ncols_pad * n_pad
  int nsplit;
  // entries e and e + 1 (e even)
  __device__ __forceinline__ void store2(int64_t e, float2 y0, float2 y1) const {
    const FPair x0{y0.x, 0.f}, x1{y1.x, 0.f}, z0{y0.y, 0.f}, z1{y1.y, 0.f};
    store_pieces(x0, x1, nsplit, base + e, 3 * plane);
    store_pieces(z0, z1, nsplit, base + plane + e, 3 * plane);
    store_pieces(fsum(x0, z0), fsum(x1, z1), nsplit, base + 2 * plane + e, 3 * plane);
  }
};

// Sum split-K partials (fixed order) and apply the recurrence; write the FP32 state and
// the BF16 pieces of the new block. All arrays are transposed (column-major in Y).
// ksplit = 0 means the product term is zero (first step of the corrected filter).
// With R non-null the forcing term pc[col] * R[col][row] is added (residual-corrected
// filter: the recurrence runs on the defect D_j = p_j(C) Q - Q p_j(Theta)).
__device__ __forceinline__ void tc_epilogue_body(int n, int ncols, int n_pad, int ncols_pad, int ksplit,
                                                 const float2* ws, const float2* cur, const float2* prev, float2* outp,
                                                 const YPlanes& yp, float alpha, float beta, float gamma,
                                                 const float2* R, const float* pc) {
  // two neighbouring rows (n_pad is even) of a column a thread
  const int64_t plane = (int64_t)ncols_pad * n_pad;
  const uint32_t half = (uint32_t)n_pad / 2, total = (uint32_t)ncols_pad * half;
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < total; q += gridDim.x * blockDim.x) {
    const int col = (int)(q / half), row = 2 * (int)(q % half);
    const int64_t e = (int64_t)col * n_pad + row;
    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
    if (col < ncols && row < n) {
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
      for (int z = 0; z < ksplit; ++z) {
        const float4 v = *(const float4*)(ws + (int64_t)z * plane + e);
        acc.x += v.x;
        acc.y += v.y;
        acc.z += v.z;
        acc.w += v.w;
      }
      y = make_float4(alpha * acc.x, alpha * acc.y, alpha * acc.z, alpha * acc.w);
      auto axpy = [&](float f, const float2* p) {
        const float4 v = *(const float4*)(p + e);
        y.x += f * v.x;
        y.y += f * v.y;
        y.z += f * v.z;
        y.w += f * v.w;
      };
      if (cur) axpy(beta, cur);
      if (prev) axpy(gamma, prev);
      if (R) axpy(pc[col], R);
      if (row + 1 >= n) y.z = y.w = 0.f;
    }
    *(float4*)(outp + e) = y;
    yp.store2(e, make_float2(y.x, y.y), make_float2(y.z, y.w));
  }
}

__global__ void cheb_tc_epilogue(int n, int ncols, int n_pad, int ncols_pad, int ksplit, const float2* ws,
                                 const float2* cur, const float2* prev, float2* outp, YPlanes yp, float alpha,
                                 float beta, float gamma, const float2* R, const float* pc) {
  tc_epilogue_body(n, ncols, n_pad, ncols_pad, ksplit, ws, cur, prev, outp, yp, alpha, beta, gamma, R, pc);
}

// R^T = (W - Q diag(theta))^T in FP32 (residual of the Rayleigh-Ritz pairs), transposed.
__device__ __forceinline__ void resid_to_state_body(int n, int m, int n_pad, int ncols_pad, const double2* Q,
                                                    int64_t ldq, const double2* W, int64_t ldw, const double* theta,
                                                    float2* Rt, int r0, int c0) {
  __shared__ float2 t[32][33];
  int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  for (int k = ty; k < 32; k += 8) {
    int r = r0 + k, c = c0 + tx;
    float2 v = make_float2(0.f, 0.f);
    if (r < n && c < m) {
      double2 q = Q[(int64_t)r * ldq + c], w = W[(int64_t)r * ldw + c];
      double th = theta[c];
      v = make_float2((float)(w.x - th * q.x), (float)(w.y - th * q.y));
    }
    t[k][tx] = v;
  }
  __syncthreads();
  for (int k = ty; k < 32; k += 8) {
    int c = c0 + k, r = r0 + tx;
    if (c < ncols_pad && r < n_pad) Rt[(int64_t)c * n_pad + r] = t[tx][k];
  }
}

__global__ void resid_to_state(int n, int m, int n_pad, int ncols_pad, const double2* Q, int64_t ldq,
                               const double2* W, int64_t ldw, const double* theta, float2* Rt) {
  resid_to_state_body(n, m, n_pad, ncols_pad, Q, ldq, W, ldw, theta, Rt, blockIdx.x * 32, blockIdx.y * 32);
}

// Y = Q diag(pd) + D (FP64 out, row-major): the filtered block from the defect D^T.
__device__ __forceinline__ void defect_to_y_body(int n, int m, int n_pad, const float2* Dt, const double2* Q,
                                                 int64_t ldq, const double* pd, double2* Y, int64_t ldy, int r0,
                                                 int c0) {
  __shared__ float2 t[32][33];
  int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  for (int k = ty; k < 32; k += 8) {
    int c = c0 + k, r = r0 + tx;
    t[k][tx] = (c < m && r < n) ? Dt[(int64_t)c * n_pad + r] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  for (int k = ty; k < 32; k += 8) {
    int r = r0 + k, c = c0 + tx;
    if (r < n && c < m) {
      float2 d = t[tx][k];
      double2 q = Q[(int64_t)r * ldq + c];
      double p = pd[c];
      Y[(int64_t)r * ldy + c] = make_double2(fma(q.x, p, (double)d.x), fma(q.y, p, (double)d.y));
    }
  }
}

__global__ void defect_to_y(int n, int m, int n_pad, const float2* Dt, const double2* Q, int64_t ldq,
                            const double* pd, double2* Y, int64_t ldy) {
  defect_to_y_body(n, m, n_pad, Dt, Q, ldq, pd, Y, ldy, blockIdx.x * 32, blockIdx.y * 32);
}

// C (FP64, n x n) -> BF16 pieces [piece][re, im, re+im][n_pad][n_pad] (zero padding), two
// neighbouring entries a thread. Bound by its integer and FP32 instructions and the planes' bytes
// (n = 2048, three pieces: 28 us; 205 with FP64 conversions).
__device__ __forceinline__ void c_to_planes_body(int64_t n, int n_pad, const double2* C, int64_t ldc,
                                                 __nv_bfloat16* planes, int nsplit) {
  const size_t total = (size_t)n_pad * n_pad;
  const uint32_t half = (uint32_t)n_pad / 2;
  for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < total / 2;
       q += (uint64_t)gridDim.x * blockDim.x) {
    const int64_t i = (int64_t)(q / half), j = 2 * (int64_t)(q % half);
    const double2 zero = make_double2(0.0, 0.0);
    const double2 u = (i < n && j < n) ? C[i * ldc + j] : zero, v = (i < n && j + 1 < n) ? C[i * ldc + j + 1] : zero;
    const FPair ux = fsplit(u.x), uy = fsplit(u.y), vx = fsplit(v.x), vy = fsplit(v.y);
    __nv_bfloat16* at = planes + (size_t)i * n_pad + j;
    store_pieces(ux, vx, nsplit, at, 3 * total);
    store_pieces(uy, vy, nsplit, at + total, 3 * total);
    store_pieces(fsum(ux, uy), fsum(vx, vy), nsplit, at + 2 * total, 3 * total);
  }
}

__global__ void __launch_bounds__(256) c_to_planes(int64_t n, int n_pad, const double2* C, int64_t ldc,
                                                   __nv_bfloat16* planes, int nsplit) {
  c_to_planes_body(n, n_pad, C, ldc, planes, nsplit);
}

// Y (FP64 row-major n x m, ld) -> transposed FP32 state + BF16 pieces (ncols_pad x n_pad),
// through a 32 x 32 shared-memory tile for coalescing on both sides.
__global__ void y_to_state(int n, int m, int n_pad, int ncols_pad, const double2* Y, int64_t ldy, float2* st,
                           YPlanes yp) {
  __shared__ float2 t[32][33];
  int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  int tx = threadIdx.x % 32, ty = threadIdx.x / 32;   // 256 threads: ty 0..7
  for (int k = ty; k < 32; k += 8) {
    int r = r0 + k, c = c0 + tx;
    double2 v = (r < n && c < m) ? Y[(int64_t)r * ldy + c] : make_double2(0.0, 0.0);
    t[k][tx] = make_float2((float)v.x, (float)v.y);
  }
  __syncthreads();
  for (int k = threadIdx.x / 16; k < 32; k += 16) {
    const int c = c0 + k, r = r0 + 2 * (threadIdx.x % 16);
    if (c < ncols_pad && r < n_pad) {
      const float2 u = t[r - r0][k], v = t[r - r0 + 1][k];
      const int64_t e = (int64_t)c * n_pad + r;
      *(float4*)(st + e) = make_float4(u.x, u.y, v.x, v.y);
      yp.store2(e, u, v);
    }
  }
}

__global__ void state_to_y(int n, int m, int n_pad, const float2* st, double2* Y, int64_t ldy) {
  __shared__ float2 t[32][33];
  int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  for (int k = ty; k < 32; k += 8) {
    int c = c0 + k, r = r0 + tx;
    t[k][tx] = (c < m && r < n) ? st[(int64_t)c * n_pad + r] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  for (int k = ty; k < 32; k += 8) {
    int r = r0 + k, c = c0 + tx;
    if (r < n && c < m) {
      float2 v = t[tx][k];
      Y[(int64_t)r * ldy + c] = make_double2(v.x, v.y);
    }
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

bool encode_2d(CUtensorMap* map, void* base, uint64_t inner, uint64_t outer, uint32_t box_inner, uint32_t box_outer) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {inner * 2};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t es[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

constexpr int kKsplitMax = 16;
constexpr int kDegMax = 64;

int tc_stages(int nchunk) {
  return (int)std::min<size_t>(STAGES, (TC_SMEM - 1024) / (3 * TM * TK * 2 + 3 * (size_t)(nchunk / 2) * TK * 2));
}
int pad_to(int x, int a) { return (x + a - 1) / a * a; }

void chunking(int m, int* nchunks, int* nchunk) {
  int k = (m + NMAX - 1) / NMAX;
  int c = pad_to((m + k - 1) / k, 16);
  *nchunks = k;
  *nchunk = c;
}

}  // namespace

struct FilterTC {
  int n_pad = 0;                    // of the problem it was last reserved for
  int cap_n = 0, cap_cols = 0;      // what the arena holds
  int c_nsplit = 0;                 // pieces of C currently stored
  __nv_bfloat16* Cp = nullptr;      // [MAXSPLIT][3][n_pad][n_pad]
  __nv_bfloat16* Yp = nullptr;      // [MAXSPLIT][3][ncols_pad][n_pad]
  float2 *S0 = nullptr, *S1 = nullptr, *S2 = nullptr, *S3 = nullptr, *ws = nullptr;
  float* pcoef = nullptr;           // device: [kDegMax][ncols_pad]
  double* pfinal = nullptr;         // device: [ncols_pad]
  float* h_pcoef = nullptr;         // pinned host staging
  double* h_pfinal = nullptr;
  int* err = nullptr;
  size_t bytes = 0;
  void* arena = nullptr;
};

bool tc_filter_supported() {
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  return major == 10 && minor == 3 && get_encode() != nullptr;
}

// Zero fill on stream s: a plain cudaMemset runs on the legacy default stream, which is
// not ordered with the library's non-blocking streams, and could land after the planes
// that s writes next.
cudaError_t filter_tc_reserve(FilterTC** pf, int64_t n, int m, cudaStream_t s) {
  if (!*pf) *pf = new FilterTC();
  FilterTC* f = *pf;
  int n_pad = pad_to((int)n, TM);
  int nchunks, nchunk;
  chunking(m, &nchunks, &nchunk);
  int ncols_pad = nchunks * pad_to(nchunk, 32);   // also as twice as many tiles of half the width
  // the padding and the launch follow the problem, not the largest one so far
  f->n_pad = n_pad;
  if (n_pad <= f->cap_n && ncols_pad <= f->cap_cols && f->arena) return cudaSuccess;
  n_pad = std::max(n_pad, f->cap_n);
  ncols_pad = std::max(ncols_pad, f->cap_cols);
  if (f->arena) cudaFree(f->arena);
  f->arena = nullptr;
  f->c_nsplit = 0;
  size_t np2 = (size_t)n_pad * n_pad, nc = (size_t)ncols_pad * n_pad;
  auto al = [](size_t b) { return (b + 1023) & ~(size_t)1023; };
  size_t bytes = al((size_t)MAXSPLIT * 3 * np2 * 2) + al((size_t)MAXSPLIT * 3 * nc * 2) + 4 * al(nc * 8) +
                 al((size_t)kKsplitMax * nc * 8) + al((size_t)kDegMax * ncols_pad * 4) + al((size_t)ncols_pad * 8) +
                 1024;
  cudaError_t e = cudaMalloc(&f->arena, bytes);
  if (e != cudaSuccess) { f->arena = nullptr; f->cap_n = f->cap_cols = 0; return e; }
  e = cudaMemsetAsync(f->arena, 0, bytes, s);
  if (e != cudaSuccess) return e;
  char* p = (char*)f->arena;
  f->Cp = (__nv_bfloat16*)p; p += al((size_t)MAXSPLIT * 3 * np2 * 2);
  f->Yp = (__nv_bfloat16*)p; p += al((size_t)MAXSPLIT * 3 * nc * 2);
  f->S0 = (float2*)p; p += al(nc * 8);
  f->S1 = (float2*)p; p += al(nc * 8);
  f->S2 = (float2*)p; p += al(nc * 8);
  f->S3 = (float2*)p; p += al(nc * 8);
  f->ws = (float2*)p; p += al((size_t)kKsplitMax * nc * 8);
  f->pcoef = (float*)p; p += al((size_t)kDegMax * ncols_pad * 4);
  f->pfinal = (double*)p; p += al((size_t)ncols_pad * 8);
  if (f->h_pcoef) cudaFreeHost(f->h_pcoef);
  if (f->h_pfinal) cudaFreeHost(f->h_pfinal);
  f->h_pcoef = nullptr;
  f->h_pfinal = nullptr;
  cudaMallocHost(&f->h_pcoef, (size_t)kDegMax * ncols_pad * 4);
  cudaMallocHost(&f->h_pfinal, (size_t)ncols_pad * 8);
  f->err = (int*)p;
  f->cap_n = n_pad;
  f->cap_cols = ncols_pad;
  f->bytes = bytes;
  return cudaSuccess;
}

const int* filter_tc_error(const FilterTC* f) { return f->err; }

void filter_tc_release(FilterTC* f) {
  if (!f) return;
  if (f->h_pcoef) cudaFreeHost(f->h_pcoef);
  if (f->h_pfinal) cudaFreeHost(f->h_pfinal);
  if (f->arena) cudaFree(f->arena);
  delete f;
}

// Convert C (FP64) into its BF16 pieces; once per problem.
cudaError_t filter_tc_set_matrix(FilterTC* f, int64_t n, const double2* C, int64_t ldc, int nsplit, cudaStream_t s) {
  int64_t total = (int64_t)f->n_pad * f->n_pad / 2;
  int blocks = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
  c_to_planes<<<blocks, 256, 0, s>>>(n, f->n_pad, C, ldc, f->Cp, nsplit);
  LAUNCH_NOTE(1);
  f->c_nsplit = nsplit;
  return cudaGetLastError();
}

namespace {

// Shared driver of the plain and the residual-corrected filter.
cudaError_t run_filter(FilterTC* f, int64_t n, int m, const double2* Y, int64_t ldy, const double2* W, int64_t ldw,
                       const double* theta_dev, const double* theta_host, double2* Yout, int64_t ldo, int deg,
                       double lo, double hi, double sc, int nsplit, int* err_host, cudaStream_t s) {
  if (deg < 1 || deg > kDegMax || nsplit < 1 || nsplit > MAXSPLIT || f->c_nsplit < nsplit) return cudaErrorInvalidValue;
  const bool corrected = (W != nullptr);
  int nchunks, nchunk;
  chunking(m, &nchunks, &nchunk);
  const int n_pad = f->n_pad;
  const int mtiles = n_pad / TM;
  const int nkb = n_pad / TK;
  // K slices: those of the arena's order (the largest served so far), which keeps the
  // order of the FP32 sums, and with it the result, what it is with the block padded to that order
  const int cap_kb = f->cap_n / TK;
  const int want = std::max(1, std::min(std::min(kKsplitMax, cap_kb / 2), 152 / std::max(f->cap_n / TM * nchunks, 1)));
  const int kbps = (cap_kb + want - 1) / want;
  const int ks = (nkb + kbps - 1) / kbps;
  // where that leaves SMs idle, narrower column tiles: they share no sums, so they change nothing else
  // (n = 2048, m = 140 in an arena of order 4096: 41.6 us a step, 52.8 with 144-wide tiles)
  if (nchunk > 64 && 2 * mtiles * nchunks * ks <= 152) {
    nchunk = pad_to((m + 2 * nchunks - 1) / (2 * nchunks), 16);
    nchunks = (m + nchunk - 1) / nchunk;
  }
  const int ncols_pad = nchunks * nchunk;   // of the active columns, at most what was reserved
  const size_t cplane = (size_t)n_pad * n_pad, yplane = (size_t)ncols_pad * n_pad;
  TcMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  for (int pc = 0; pc < nsplit; ++pc)
    for (int part = 0; part < 3; ++part) {
      if (!encode_2d(&maps.a[3 * pc + part], f->Cp + (3 * pc + part) * cplane, n_pad, n_pad, TK, TM) ||
          !encode_2d(&maps.b[3 * pc + part], f->Yp + (3 * pc + part) * yplane, n_pad, ncols_pad, TK, nchunk / 2))
        return cudaErrorNotSupported;
    }
  YPlanes yp{f->Yp, yplane, nsplit};
  TcParams p;
  p.n_pad = n_pad;
  p.nchunk = nchunk;
  p.kb_per_split = kbps;
  p.ncols_pad = ncols_pad;
  p.nsplit = nsplit;
  p.ws = f->ws;
  p.err = f->err;
  p.tmem_cols = 32;
  while (p.tmem_cols < 3u * (uint32_t)nchunk) p.tmem_cols *= 2;
  p.nst = tc_stages(nchunk);
  cudaFuncSetAttribute(cheb_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM);
  cudaMemsetAsync(f->err, 0, sizeof(int), s);
  // recurrence coefficients (the same for the block and for the scalars p_j(theta))
  double e = 0.5 * (hi - lo), c = 0.5 * (hi + lo);
  double sigma = e / (sc - c), sigma1 = sigma;
  std::vector<double> al(deg), be(deg), ga(deg);
  for (int j = 0; j < deg; ++j) {
    if (j == 0) {
      al[0] = sigma1 / e;
      be[0] = -c * sigma1 / e;
      ga[0] = 0.0;
    } else {
      double sn = 1.0 / (2.0 / sigma1 - sigma);
      al[j] = 2.0 * sn / e;
      be[j] = -al[j] * c;
      ga[j] = -sigma * sn;
      sigma = sn;
    }
  }
  dim3 tg((n_pad + 31) / 32, (ncols_pad + 31) / 32);
  int64_t total = (int64_t)ncols_pad * n_pad / 2;
  int eblocks = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
  dim3 grid((mtiles + 1) / 2 * 2, nchunks, ks);
  float2* prev = nullptr;
  float2* cur = f->S0;
  float2* nxt = f->S1;
  float2* spare = f->S2;
  int j0 = 0;
  if (corrected) {
    // scalar recurrence p_j(theta_c) on the host: pcoef[j][c] = alpha_j p_j(theta_c), pfinal = p_deg
    for (int col = 0; col < m; ++col) {
      double th = theta_host[col];
      double pm1 = 0.0, p0 = 1.0;
      for (int j = 0; j < deg; ++j) {
        f->h_pcoef[(size_t)j * ncols_pad + col] = (float)(al[j] * p0);
        double p1 = al[j] * th * p0 + be[j] * p0 + ga[j] * pm1;
        pm1 = p0;
        p0 = p1;
      }
      f->h_pfinal[col] = p0;
    }
    cudaMemcpyAsync(f->pcoef, f->h_pcoef, (size_t)deg * ncols_pad * 4, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(f->pfinal, f->h_pfinal, (size_t)ncols_pad * 8, cudaMemcpyHostToDevice, s);
    resid_to_state<<<tg, 256, 0, s>>>((int)n, m, n_pad, ncols_pad, Y, ldy, W, ldw, theta_dev, f->S3);
    LAUNCH_NOTE(1);
    // D_1 = alpha_0 R (no product: D_0 = 0)
    cheb_tc_epilogue<<<eblocks, 256, 0, s>>>((int)n, m, n_pad, ncols_pad, 0, f->ws, nullptr, nullptr, cur, yp, 0.f, 0.f,
                                             0.f, f->S3, f->pcoef);
    LAUNCH_NOTE(1);
    j0 = 1;
  } else {
    y_to_state<<<tg, 256, 0, s>>>((int)n, m, n_pad, ncols_pad, Y, ldy, f->S0, yp);
    LAUNCH_NOTE(1);
  }
  for (int j = j0; j < deg; ++j) {
    cheb_tc_kernel<<<grid, 128, TC_SMEM, s>>>(maps, p);
    LAUNCH_NOTE(1);
    const float2* Rj = corrected ? f->S3 : nullptr;
    const float* pcj = corrected ? f->pcoef + (size_t)j * ncols_pad : nullptr;
    cheb_tc_epilogue<<<eblocks, 256, 0, s>>>((int)n, m, n_pad, ncols_pad, ks, f->ws, cur, prev, nxt, yp, (float)al[j],
                                             (float)be[j], (float)ga[j], Rj, pcj);
    LAUNCH_NOTE(1);
    float2* old_prev = prev ? prev : spare;
    prev = cur;
    cur = nxt;
    nxt = old_prev;
  }
  if (corrected) defect_to_y<<<tg, 256, 0, s>>>((int)n, m, n_pad, cur, Y, ldy, f->pfinal, Yout, ldo);
  else state_to_y<<<tg, 256, 0, s>>>((int)n, m, n_pad, cur, Yout, ldo);
  LAUNCH_NOTE(1);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  if (err_host) cudaMemcpyAsync(err_host, f->err, sizeof(int), cudaMemcpyDeviceToHost, s);
  return cudaSuccess;
}

}  // namespace

// Y (FP64 n x m, ld ldy) -> p(C) Y written to Yout (FP64, ld ldo); the same polynomial as
// the FP64 filter: degree deg, damped interval [lo, hi], scaling point sc.
cudaError_t filter_tc_apply(FilterTC* f, int64_t n, int m, const double2* Y, int64_t ldy, double2* Yout,
                            int64_t ldo, int deg, double lo, double hi, double sc, int nsplit, int* err_host,
                            cudaStream_t s) {
  return run_filter(f, n, m, Y, ldy, nullptr, 0, nullptr, nullptr, Yout, ldo, deg, lo, hi, sc, nsplit, err_host, s);
}

// Residual-corrected filter: Y = p(C) Q computed as Q p(Theta) + D, where the defect
//   D_{j+1} = alpha_j C D_j + beta_j D_j + gamma_j D_{j-1} + alpha_j R diag(p_j(Theta)),  D_0 = 0,
// follows from C Q = Q Theta + R (R = W - Q Theta, the FP64 Rayleigh-Ritz residual). The
// products C D_j run on the tensor cores; their rounding is relative to ||D||, which
// shrinks with ||R||, so the filtered block stays accurate to about u ||R|| instead of
// u ||Y||. theta (host) are the Ritz values of the columns of Q.
cudaError_t filter_tc_apply_corrected(FilterTC* f, int64_t n, int m, const double2* Q, int64_t ldq, const double2* W,
                                      int64_t ldw, const double* theta_dev, const double* theta_host, double2* Yout,
                                      int64_t ldo, int deg, double lo, double hi, double sc, int nsplit,
                                      cudaStream_t s) {
  return run_filter(f, n, m, Q, ldq, W, ldw, theta_dev, theta_host, Yout, ldo, deg, lo, hi, sc, nsplit, nullptr, s);
}

// One plain product D = C Y for tests of the tensor-core GEMM: a degree-1 filter with
// e = 1, c = 0 and scaling point 1 gives alpha = 1, beta = 0 exactly.
cudaError_t filter_tc_product(FilterTC* f, int64_t n, int m, const double2* Y, int64_t ldy, double2* D, int64_t ldd,
                              int nsplit, int* err_host, cudaStream_t s) {
  return run_filter(f, n, m, Y, ldy, nullptr, 0, nullptr, nullptr, D, ldd, 1, -1.0, 1.0, 1.0, nsplit, err_host, s);
}

// ===================================================================== grouped form
// The residual-corrected filter for every problem of a k-point batch at once: one launch
// per recurrence step covers the output tiles of all problems (a global tile list with a
// prefix sum per problem, BDesc::unit_start), and one launch per step applies the
// recurrence to all problems. The coefficients, the degree and the activity of each
// problem are read from device memory (BDesc::fco, pcoef, pfinal, flags), so the launch
// sequence is the same in every round and is captured once. The tensor maps live in
// global memory, 18 per problem.
namespace {

__device__ __forceinline__ bool tcg_runs(const BDesc& d, int j) { return d.flags[6] != 0 && j < d.flags[1]; }

__global__ void __launch_bounds__(128, 1) __cluster_dims__(2, 1, 1)
    cheb_tcg_kernel(const BDesc* D, int np, int j, int nst, int* err) {
  const int u = blockIdx.x >> 1;   // a pair of CTAs a unit
  int lo = 0, hi = np - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (D[mid].unit_start <= u) lo = mid; else hi = mid - 1;
  }
  const BDesc& d = D[lo];
  if (!tcg_runs(d, j)) return;
  const int local = u - d.unit_start;
  const int per_z = (d.mtiles + 1) / 2 * d.nchunks;
  const int z = local / per_z, r = local % per_z;
  if (z >= d.ks) return;
  TcParams p;
  p.n_pad = d.n_pad;
  p.nchunk = d.nchunk;
  p.kb_per_split = d.kbps;
  p.ncols_pad = d.ncols_pad;
  p.nsplit = d.nsplit;
  p.tmem_cols = d.tmem_cols;
  p.nst = nst;
  p.ws = d.tws;
  p.err = err;
  const CUtensorMap* maps = (const CUtensorMap*)d.maps;
  tc_tile(maps, maps + MAXSPLIT * 3, p, (r / d.nchunks) * 2 * TM, (r % d.nchunks) * d.nchunk, z, blockIdx.x & 1);
}

// j = 0: D_1 = alpha_0 R; j >= 1: D_{j+1} from the split-K partials of C D_j. D_k is kept
// in S[(k - 1) mod 3].
__global__ void tcg_epilogue(const BDesc* D, int j) {
  const BDesc& d = D[blockIdx.y];
  if (!tcg_runs(d, j)) return;
  float2* S[3] = {d.S0, d.S1, d.S2};
  float2* outp = S[j % 3];
  const float2* cur = j >= 1 ? S[(j - 1) % 3] : nullptr;
  const float2* prev = j >= 2 ? S[(j - 2) % 3] : nullptr;
  const float al = j >= 1 ? (float)d.fco[3 * j] : 0.f;
  const float be = j >= 1 ? (float)d.fco[3 * j + 1] : 0.f;
  const float ga = j >= 1 ? (float)d.fco[3 * j + 2] : 0.f;
  YPlanes yp{d.Yp, (size_t)d.ncols_pad * d.n_pad, d.nsplit};
  tc_epilogue_body(d.n, d.m, d.n_pad, d.ncols_pad, j >= 1 ? d.ks : 0, d.tws, cur, prev, outp, yp, al, be, ga, d.S3,
                   d.pcoef + (size_t)j * d.ncols_pad);
}

__global__ void tcg_resid_to_state(const BDesc* D) {
  const BDesc& d = D[blockIdx.z];
  if (d.flags[6] == 0) return;
  const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  if (r0 >= d.n_pad || c0 >= d.ncols_pad) return;
  resid_to_state_body(d.n, d.m, d.n_pad, d.ncols_pad, d.Q, d.m, d.W, d.m, d.theta, d.S3, r0, c0);
}

// Y1 = Q diag(p_deg(theta)) + D_deg
__global__ void tcg_defect_to_y(const BDesc* D) {
  const BDesc& d = D[blockIdx.z];
  if (d.flags[6] == 0) return;
  const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  if (r0 >= d.n || c0 >= d.m) return;
  float2* S[3] = {d.S0, d.S1, d.S2};
  const int deg = d.flags[1];
  defect_to_y_body(d.n, d.m, d.n_pad, S[(deg - 1) % 3], d.Q, d.m, d.pfinal, d.Y1, d.m, r0, c0);
}

__global__ void tcg_c_to_planes(const BDesc* D) {
  const BDesc& d = D[blockIdx.y];
  if (d.flags[0] == 0) return;
  c_to_planes_body(d.n, d.n_pad, d.C, d.n, d.Cp, d.nsplit);
}

}  // namespace

void tcg_geometry(int64_t n, int m, int* n_pad, int* ncols_pad, int* nchunk, int* nchunks) {
  *n_pad = pad_to((int)n, TM);
  chunking(m, nchunks, nchunk);
  *ncols_pad = *nchunks * *nchunk;
}

size_t tcg_map_bytes() { return sizeof(CUtensorMap) * MAXSPLIT * 3 * 2; }

bool tcg_encode_maps(const BDesc& d, void* maps_host) {
  CUtensorMap* a = (CUtensorMap*)maps_host;
  CUtensorMap* b = a + MAXSPLIT * 3;
  std::memset(maps_host, 0, tcg_map_bytes());
  const size_t cplane = (size_t)d.n_pad * d.n_pad, yplane = (size_t)d.ncols_pad * d.n_pad;
  for (int pc = 0; pc < d.nsplit; ++pc)
    for (int part = 0; part < 3; ++part) {
      if (!encode_2d(&a[3 * pc + part], d.Cp + (3 * pc + part) * cplane, d.n_pad, d.n_pad, TK, TM) ||
          !encode_2d(&b[3 * pc + part], d.Yp + (3 * pc + part) * yplane, d.n_pad, d.ncols_pad, TK, d.nchunk / 2))
        return false;
    }
  return true;
}

void tcg_set_matrix(const BDesc* D, int np, int64_t npad2_max, cudaStream_t s) {
  int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((npad2_max / 2 + 255) / 256, 512));
  tcg_c_to_planes<<<dim3(blocks, np), 256, 0, s>>>(D);
  LAUNCH_NOTE(1);
}

cudaError_t tcg_prepare() {
  return cudaFuncSetAttribute(cheb_tcg_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM);
}

// The launch sequence of one filter application (no host synchronisation, capturable);
// tcg_prepare must have been called first.
cudaError_t tcg_filter(const BDesc* D, const TcgShape& g, int* err, cudaStream_t s) {
  const int nst = tc_stages(g.nchunk_max);
  dim3 tg((g.n_pad_max + 31) / 32, (g.ncols_pad_max + 31) / 32, g.np);
  int eb = (int)std::max<int64_t>(1, std::min<int64_t>((g.nc_max / 2 + 255) / 256, 128));
  tcg_resid_to_state<<<tg, 256, 0, s>>>(D);
  tcg_epilogue<<<dim3(eb, g.np), 256, 0, s>>>(D, 0);
  LAUNCH_NOTE(2);
  for (int j = 1; j < g.steps; ++j) {
    cheb_tcg_kernel<<<2 * g.units, 128, TC_SMEM, s>>>(D, g.np, j, nst, err);
    tcg_epilogue<<<dim3(eb, g.np), 256, 0, s>>>(D, j);
    LAUNCH_NOTE(2);
  }
  tcg_defect_to_y<<<tg, 256, 0, s>>>(D);
  LAUNCH_NOTE(1);
  return cudaGetLastError();
}

}  // namespace gevp

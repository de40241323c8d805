// Tall-skinny kernels of the orthonormalisation (CholQR) and the Rayleigh-Ritz projection.
//
// zgram: G = X^H Y for n x mx and n x my blocks with n >> m (the Gram matrix Y^H Y of
//   CholQR, the projection Q^H W of Rayleigh-Ritz, the overlaps Q_lock^H Y). On this part
//   one SM retires about 1.7 FP64 FMAs per clock, so the product is FP64-pipe bound and
//   the whole job is to keep all 152 SMs busy with little else: the m x m result is cut
//   into 16 x 16 tiles (only the lower ones when the result is Hermitian, half the
//   flops), n into slices so that the CTAs cover the SMs several times over, and the
//   slices of a tile are summed in slice order by whichever CTA of that tile finishes
//   last (a per-tile arrival counter), so there is no second launch and the sum is
//   deterministic. A Hermitian result is written to both triangles.
//
// cholinv: the Cholesky factor L of D W D + shift I (W the Gram matrix, lower triangle
//   read; D = diag(W)^-1/2 the column scaling of CholQR) and its inverse, for m up to a
//   few hundred, in the CTAs of one thread-block cluster per matrix. A one-CTA factorisation
//   would take close to a millisecond at m = 140 (m^3/3 complex multiply-adds at two FP64 FMAs
//   per clock). Here the rows are dealt cyclically to the P CTAs (row i to CTA i mod P) and held
//   in shared memory with the rows of the inverse's accumulator S (initially I). Panels of eight
//   columns J, one cluster barrier per panel:
//     every CTA gathers, through distributed shared memory, the raw panel A[e, J], e >= j0, and
//     the raw rows S[J, :] (all final after the panel before), eliminates the 8 x 8 diagonal block
//     redundantly (T = its unit-pivot inverse accumulator, a_q its pivots), forms for its own
//     rows i below the panel the multipliers M_i = A[i, J] T^H diag(1/a) T = A[i, J] A_JJ^-1, and
//     updates
//       A[i, e] -= M_i A[e, J]^H   (e > J; the trailing Cholesky update)
//       S[i, e] -= M_i S[J, e]     (e <= J; the inverse, L X = I, right-looking)
//     L[i, J] = A[i, J] T^H diag(a)^-1/2 and the rows J of L^-1, diag(a)^-1/2 T S[J, :], are
//     written as they become known. Raw values and multipliers keep the other CTAs' rows out
//     of the dependence: nothing is exchanged but the gather.
//   Within a panel the reads (columns J of A, rows J of S) and the writes (columns > J of A, rows
//   > J of S) never meet, so one barrier per panel suffices. The barrier is split: a CTA first
//   updates what the next panel reads (the next eight columns, its own rows of S among the next
//   block), arrives, updates the rest while the other CTAs catch up, and waits before the next
//   gather. At m = 256 half the time is the FP64 pipe's (4/3 m^3 FMAs on P SMs at two a clock);
//   below, the panel's chain of FP64 operations at 64 clocks each. Measured m = 128 232 us, 140
//   262 us, 256 805 us (320 us and 1.2 ms at m = 140 and 256 with one column a step).
//   A matrix within 1e-9 of the identity after scaling (the second pass of CholQR2) needs no
//   elimination: L^-1 = I - N to FP64 rounding (m = 140: 9 us).
//   The output Li = L^-1 D (columns scaled by D) makes Y Li^H = Y D L^-H, the orthonormal
//   factor of one CholQR pass, a single product; it is also the inverse of D^-1 L, the
//   Cholesky factor of W itself (shift 0), which is written out on request (the leaves
//   of the recursive factorisation of B). A non-positive pivot stops the cluster (every
//   CTA eliminates the same block, so the decision is uniform) and sets *info to its 1-based
//   index plus a caller's offset; rows before that panel have been written then. W may share
//   memory with the factor's output: every CTA reads its rows of W before the first cluster
//   barrier and writes the factor after it.
#include "gevp_internal.cuh"
#include "zsmall.cuh"
#include <cooperative_groups.h>
#include <algorithm>

namespace gevp {

namespace {

constexpr int GT = 16;   // zgram output tile edge
constexpr int GK = 16;   // rows staged per step

__global__ void __launch_bounds__(256) zgram_kernel(int64_t n, int mx, int my, const double2* __restrict__ X,
                                                    int64_t ldx, const double2* __restrict__ Y, int64_t ldy,
                                                    double2* G, int64_t ldg, int herm, int ntj, int slices,
                                                    int64_t per, double2* part, unsigned* cnt) {
  __shared__ double2 Xs[GK][GT];
  __shared__ double2 Ys[GK][GT];
  __shared__ int last;
  const int tile = blockIdx.x;
  const int ti = tile / ntj, tj = tile % ntj;
  if (herm && tj > ti) return;
  const int slice = blockIdx.y;
  const int tid = threadIdx.x;
  const int ty = tid / GT, tx = tid % GT;
  const int64_t k0 = (int64_t)slice * per;
  const int64_t k1 = min(n, k0 + per);
  const int lr = tid / GT, lc = tid % GT;   // staging: row lr, column lc of the tile
  const int xc = ti * GT + lc, yc = tj * GT + lc;
  double2 acc = make_double2(0.0, 0.0);
  for (int64_t k = k0; k < k1; k += GK) {
    const int64_t kr = k + lr;
    Xs[lr][lc] = (kr < k1 && xc < mx) ? X[kr * ldx + xc] : make_double2(0.0, 0.0);
    Ys[lr][lc] = (kr < k1 && yc < my) ? Y[kr * ldy + yc] : make_double2(0.0, 0.0);
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) zfma(acc, zconj(Xs[kk][ty]), Ys[kk][tx]);
    __syncthreads();
  }
  const int i = ti * GT + ty, j = tj * GT + tx;
  if (slices > 1) {
    part[((int64_t)tile * slices + slice) * (GT * GT) + tid] = acc;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = (atomicAdd(&cnt[tile], 1u) == (unsigned)(slices - 1));
    __syncthreads();
    if (!last) return;
    __threadfence();
    acc = make_double2(0.0, 0.0);
    const double2* p = part + (int64_t)tile * slices * (GT * GT) + tid;
    for (int s = 0; s < slices; ++s) acc = zadd(acc, __ldcg(p + (int64_t)s * (GT * GT)));
    if (tid == 0) cnt[tile] = 0u;   // ready for the next launch (stream order)
  }
  if (i >= mx || j >= my) return;
  if (!herm) {
    G[(int64_t)i * ldg + j] = acc;
    return;
  }
  if (j > i) return;   // the diagonal tile's upper half comes from the lower one
  if (j == i) {
    G[(int64_t)i * ldg + i] = make_double2(acc.x, 0.0);
  } else {
    G[(int64_t)i * ldg + j] = acc;
    G[(int64_t)j * ldg + i] = zconj(acc);
  }
}

// the same for short columns, on 4 x 8 tiles (zsmall.cuh)
__global__ void __launch_bounds__(ZS_THREADS) zgram_small_kernel(int n, int mx, int my, const double2* __restrict__ X,
                                                                 int64_t ldx, const double2* __restrict__ Y,
                                                                 int64_t ldy, double2* G, int64_t ldg, int herm) {
  __shared__ double part[ZS_WARPS][64];
  const int m0 = blockIdx.y * ZS_M, n0 = blockIdx.x * ZS_N;
  if (herm && n0 > m0 + ZS_M - 1) return;
  const double v = zsmall_tile<1, 0>(mx, my, X, ldx, Y, ldy, 0, m0, n0, 0, n, part);
  const int lane = threadIdx.x % 32, comp = threadIdx.x / 32;
  const int i = m0 + lane / ZS_N, j = n0 + lane % ZS_N;
  if (comp > 1 || i >= mx || j >= my || (herm && j > i)) return;
  ((double*)(G + (int64_t)i * ldg + j))[comp] = herm && i == j && comp ? 0.0 : v;
  if (herm && j < i) ((double*)(G + (int64_t)j * ldg + i))[comp] = comp ? -v : v;
}

constexpr int CT = 256;          // threads per cholinv CTA
constexpr int kCholInvMax = 288; // largest order (shared-memory bound at 16 CTAs)

// split cluster barrier: arrive (release) and, later, wait (acquire) for the phase
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

struct CholProb {
  int m;
  const double2* W;
  int64_t ldw;
  double shift;
  double2* Li;
  int64_t ldi;
  double2* Lf;
  int64_t ldl;
  int* info;
  int info_base;
};
struct CholOne {
  CholProb p;
  __device__ bool get(int, CholProb& o) const {
    o = p;
    return true;
  }
};
// the Gram matrices of a batch: Gw -> Gwi, the pivot in flags[2]
struct CholBatch {
  const BDesc* D;
  double shift_factor;
  __device__ bool get(int b, CholProb& o) const {
    const BDesc& d = D[b];
    if (d.flags[0] == 0) return false;
    const double m = d.m;
    o.m = d.m;
    o.W = d.Gw;
    o.ldw = d.m;
    o.shift = shift_factor * 11.0 * (d.n * m + m * (m + 1.0)) * 1.1102230246251565e-16 * m;
    o.Li = d.Gwi;
    o.ldi = d.m;
    o.Lf = nullptr;
    o.ldl = 0;
    o.info = d.flags + 2;
    o.info_base = 0;
    return true;
  }
};

constexpr int NB = 8;   // columns of a panel

// 1 / v for a pivot v > 0: the PTX instruction rcp.approx.ftz.f64 (about 20 bits) and one step of
// Chebyshev's cubically convergent iteration for f(r) = 1 / r - v (Traub, Iterative Methods for the
// Solution of Equations, 1964): with e = 1 - v r, r (1 + e + e^2) has the relative error e^3, below
// 2^-59, and the last rounding. Three dependent FP64 operations where the division has more (n = 777:
// 3.00 and 3.06 ms a reduction, m = 140: 788 and 809 us a CholQR2); its error, below 2^-52, acts like a
// rounding of A_JJ^-1.
__device__ __forceinline__ double pivot_recip(double v) {
  const int ex = __double2hiint(v) >> 20;   // (an FP64 comparison would cost as much as an FMA)
  if (ex < 64 || ex > 1982) return 1.0 / v;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(v));
  const double e = fma(-v, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// An SM retires two FP64 lanes per clock, a warp's instruction every 64 clocks in each of its four
// partitions whether the next one depends on it or not. So the kernel counts FP64 instructions
// per partition: sums are cut into (entry, real or imaginary part) items of at most sixteen
// FMAs, packed densely into the eight warps.
//
// The pair of a with which dot2(pair(part, a), b) is Re(a b) (part 0) or Im(a b) (part 1); the sign
// is flipped by an integer instruction
__device__ __forceinline__ double2 part_pair(int part, double2 a) {
  const double ny = __hiloint2double(__double2hiint(a.y) ^ (int)0x80000000, __double2loint(a.y));
  return part == 0 ? make_double2(a.x, ny) : make_double2(a.y, a.x);
}
__device__ __forceinline__ double dot2(double2 p, double2 b, double acc) { return fma(p.y, b.y, fma(p.x, b.x, acc)); }

template <int P, class Src>
__global__ void __launch_bounds__(CT, 1) cholinv_cluster_kernel(Src src) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  CholProb pr;
  if (!src.get(blockIdx.x / P, pr)) return;   // uniform over the cluster
  extern __shared__ double2 csm[];
  constexpr int RMAX = (kCholInvMax + P - 1) / P;
  constexpr int XMAX = (kCholInvMax + 31) / 32;
  __shared__ double2 F[NB][NB], T[NB][NB];   // the diagonal block, its inverse's accumulator
  __shared__ double2 M[2][RMAX][NB];         // part_pair(part, M)
  __shared__ double2 L[RMAX][NB], Ls[RMAX][NB];   // Ls = -L diag(1/a)
  __shared__ double rp[NB], rs[NB];          // 1 / a_q, a_q^-1/2
  __shared__ double dsc[kCholInvMax];        // D
  __shared__ double2* rA[P];
  __shared__ double2* rS[P];
  __shared__ int bad;
  __shared__ float devw[CT / 32], devs;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int m = pr.m;
  const int rank = (int)cl.block_rank();
  const int R = (m + P - 1) / P;
  double2* Arow = csm;              // [R][m]: own rows i = rank + P t of the matrix being factored
  double2* Srow = csm + R * m;      // [R][m]: own rows of the inverse's accumulator
  double2* G = csm + 2 * R * m;     // [NB][m]: S[j0 + q][x] for x < j0, I in J, conj(A[x][j0 + q]) after
  if (tid < P) {
    rA[tid] = cl.map_shared_rank(Arow, tid);
    rS[tid] = cl.map_shared_rank(Srow, tid);
  }
  if (tid == 0) bad = 0;
  for (int i = tid; i < m; i += CT) {
    const double v = pr.W[(int64_t)i * pr.ldw + i].x;
    dsc[i] = v > 0.0 ? 1.0 / sqrt(v) : 1.0;
  }
  __syncthreads();
  for (int e = tid; e < R * m; e += CT) {
    const int t = e / m, c = e % m, i = rank + P * t;
    double2 a = make_double2(0.0, 0.0), s = make_double2(0.0, 0.0);
    if (i < m && c <= i) {
      a = zscale(pr.W[(int64_t)i * pr.ldw + c], dsc[i] * dsc[c]);
      if (c == i) a = make_double2(a.x + pr.shift, 0.0);
      if (c == i) s = make_double2(1.0, 0.0);
    }
    Arow[e] = a;
    Srow[e] = s;
  }
  // D W D + shift I = I + E with ||E||_F below 1e-9 (the second pass of CholQR2): L = I + N, L^-1 =
  // I - N up to O(||E||^2) < 1e-18, N the lower triangle of E with its diagonal halved. (Squares in
  // FP32: only their size matters.)
  float dev = 0.f;
  for (int e = tid; e < R * m; e += CT) {
    const int c = e % m, i = rank + P * (e / m);
    if (i >= m || c > i) continue;
    const float x = c == i ? (float)(Arow[e].x - 1.0) : (float)Arow[e].x, y = (float)Arow[e].y;
    dev += (x * x + y * y) * (c == i ? 1.f : 2.f);
  }
  for (int o = 16; o > 0; o >>= 1) dev += __shfl_xor_sync(0xffffffffu, dev, o);
  if (lane == 0) devw[warp] = dev;
  __syncthreads();
  if (tid == 0) {
    float t = 0.f;
    for (int w = 0; w < CT / 32; ++w) t += devw[w];
    devs = t;
  }
  cl.sync();
  dev = 0.f;
  for (int q = 0; q < P; ++q) dev += *cl.map_shared_rank(&devs, q);   // in rank order: the same in every CTA
  if (dev < 1e-18f) {
    for (int e = tid; e < R * m; e += CT) {
      const int c = e % m, i = rank + P * (e / m);
      if (i >= m) continue;
      double2 a = c <= i ? Arow[e] : make_double2(0.0, 0.0), l = a;
      if (c == i) {
        a = make_double2(1.5 - 0.5 * a.x, 0.0);
        l = make_double2(2.0 - a.x, 0.0);
      } else {
        a = make_double2(-a.x, -a.y);
      }
      pr.Li[(int64_t)i * pr.ldi + c] = zscale(a, dsc[c]);
      if (pr.Lf) pr.Lf[(int64_t)i * pr.ldl + c] = zscale(l, 1.0 / dsc[i]);
    }
    cl.sync();
    return;
  }
  for (int j0 = 0; j0 < m; j0 += NB) {
    const int nb = min(NB, m - j0), j1 = j0 + nb, j2 = min(m, j1 + NB);
    // own rows below the panel: i = rank + P t >= j1, nr of them from t0, the first nn in the next block
    const int t0 = j1 > rank ? (j1 - rank + P - 1) / P : 0;
    const int nr = max(0, (rank < m ? (m - 1 - rank) / P + 1 : 0) - t0);
    int nn = 0;
    while (nn < nr && rank + P * (t0 + nn) < j2) ++nn;
    if (j0 > 0) {
      __syncthreads();   // the last panel's G and M have been read
      cluster_wait();
    }
    // gather, a column q of the panel to a warp: row j0 + q of S (x < j0), the diagonal block,
    // column j0 + q of A; every load in flight before the first is stored
    if (warp < nb) {
      const int q = warp;
      const double2* sr = rS[(j0 + q) % P] + ((j0 + q) / P) * m;
      double2 v[XMAX];
#pragma unroll
      for (int k = 0; k < XMAX; ++k) {
        const int x = lane + 32 * k;
        if (x < m) v[k] = *(x < j0 ? sr + x : rA[x % P] + (x / P) * m + j0 + q);
      }
#pragma unroll
      for (int k = 0; k < XMAX; ++k) {
        const int x = lane + 32 * k;
        if (x >= m) continue;
        double2 g = v[k];
        if (x >= j1) {
          g.y = -g.y;
        } else if (x >= j0) {
          F[x - j0][q] = g;
          g = make_double2(x - j0 == q ? 1.0 : 0.0, 0.0);
          T[x - j0][q] = g;
        }
        G[q * m + x] = g;
      }
    }
    __syncthreads();
    // eliminate the diagonal block (four warps, one per partition): F[i][q], q <= i, keeps the raw
    // columns. The products F[i][c] conj(F[e][c]) do not wait for the pivot's reciprocal.
    if (tid < 2 * NB * NB) {
      const int part = tid / (NB * NB), i = tid / NB % NB, e = tid % NB;
      for (int c = 0; c < nb; ++c) {
        const double a = F[c][c].x;
        const int hi = __double2hiint(a);
        if (hi <= 0 || hi >= 0x7ff00000) {   // not positive (below 2^-1042 counted as zero), or not finite
          if (tid == 0) bad = c + 1;
          break;
        }
        const double r = pivot_recip(a);
        if (tid == 0) rp[c] = r;
        if (i > c && i < nb && e <= i) {
          double* at = (double*)(e > c ? &F[i][e] : &T[i][e]) + part;
          const double2 w = e > c ? zconj(F[e][c]) : T[c][e];
          *at = fma(-r, dot2(part_pair(part, F[i][c]), w, 0.0), *at);
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
    }
    __syncthreads();
    if (bad) {   // the same in every CTA
      if (rank == 0 && tid == 0) atomicCAS(pr.info, 0, pr.info_base + j0 + bad);
      break;
    }
    // L = A[i, J] T^H, then M = -L diag(1/a) T
    for (int x = tid; x < 2 * nr * NB; x += CT) {
      const int part = x >= nr * NB, y = x - part * nr * NB, tt = y / NB, c = y % NB;
      double v = 0.0;
      if (c < nb)
        for (int r = 0; r <= c; ++r) v = dot2(part_pair(part, zconj(T[c][r])), Arow[(t0 + tt) * m + j0 + r], v);
      ((double*)&L[tt][c])[part] = v;
      ((double*)&Ls[tt][c])[part] = c < nb ? -rp[c] * v : 0.0;
    }
    __syncthreads();
    for (int x = tid; x < 2 * nr * NB; x += CT) {
      const int part = x >= nr * NB, y = x - part * nr * NB, tt = y / NB, r = y % NB;
      double v = 0.0;
      for (int c = r; c < nb; ++c) v = dot2(part_pair(part, Ls[tt][c]), T[c][r], v);
      if (part == 0) {
        M[0][tt][r].x = v;
        M[1][tt][r].y = v;
      } else {
        M[0][tt][r].y = __hiloint2double(__double2hiint(v) ^ (int)0x80000000, __double2loint(v));
        M[1][tt][r].x = v;
      }
    }
    __syncthreads();
    // entry (own row tt below, column x): S where x < j1, A from there on
    auto update = [&](int part, int tt, int x) {
      double* at = (double*)((x < j1 ? Srow : Arow) + (t0 + tt) * m + x) + part;
      double v = *at;
      const double2* mr = M[part][tt];
      if (nb == NB) {
#pragma unroll
        for (int q = 0; q < NB; ++q) v = dot2(mr[q], G[q * m + x], v);
      } else {
        for (int q = 0; q < nb; ++q) v = dot2(mr[q], G[q * m + x], v);
      }
      *at = v;
    };
    // first part: the next panel's columns of all own rows, and the own rows of S in the next block
    const int n1 = nr * NB, n2 = n1 + nn * j1;
    for (int x = tid; x < 2 * n2; x += CT) {
      const int part = x >= n2, y = x - part * n2;
      if (y < n1) {
        const int tt = y / NB, c = j1 + y % NB;
        if (c <= rank + P * (t0 + tt)) update(part, tt, c);
      } else {
        update(part, (y - n1) / j1, (y - n1) % j1);
      }
    }
    if (j1 < m) cluster_arrive();
    // the rest, while the other CTAs finish their first parts: (row, part) in pieces of 32 columns,
    // dealt to the warps
    int piece = 0;
    for (int tt = nn; tt < nr; ++tt) {
      const int i = rank + P * (t0 + tt), n = j1 + max(0, i + 1 - j2);
      for (int part = 0; part < 2; ++part)
        for (int x0 = 0; x0 < n; x0 += 32, ++piece) {
          if (piece % (CT / 32) != warp) continue;
          const int x = x0 + lane;
          if (x < n) update(part, tt, x < j1 ? x : x - j1 + j2);
        }
    }
    // results: L[i, J] of the own rows below, the own rows of the block
    if (tid >= CT - NB && tid - (CT - NB) < nb) rs[tid - (CT - NB)] = rsqrt(F[tid - (CT - NB)][tid - (CT - NB)].x);
    __syncthreads();
    if (pr.Lf)
      for (int x = tid; x < nr * NB; x += CT) {
        const int tt = x / NB, q = x % NB, i = rank + P * (t0 + tt);
        // the factor of W + shift D^-2: D^-1 times the factor of D W D + shift I
        if (q < nb) pr.Lf[(int64_t)i * pr.ldl + j0 + q] = zscale(L[tt][q], rs[q] / dsc[i]);
      }
    for (int q = 0; q < nb; ++q) {
      const int i = j0 + q;
      if (i % P != rank) continue;
      const double ri = rs[q];
      for (int x = tid; x < 2 * m; x += CT) {
        const int part = x >= m, c = x - part * m;
        double v = 0.0;
        if (c <= i) {
          for (int r = 0; r <= q; ++r) v = dot2(part_pair(part, T[q][r]), G[r * m + c], v);
          v *= ri * dsc[c];
        }
        ((double*)(pr.Li + (int64_t)i * pr.ldi + c))[part] = v;
      }
      if (pr.Lf)
        for (int c = j0 + tid; c < m; c += CT) {
          double2 l = make_double2(0.0, 0.0);
          if (c < i) l = zscale(F[q][c - j0], rs[c - j0] / dsc[i]);
          else if (c == i) l = make_double2(F[q][q].x * ri / dsc[i], 0.0);
          pr.Lf[(int64_t)i * pr.ldl + c] = l;
        }
    }
  }
  cl.sync();   // no CTA leaves while another may still read its shared memory
}

template <int P>
size_t cholinv_smem(int m) {
  return ((size_t)2 * ((m + P - 1) / P) + NB) * m * sizeof(double2);
}

// np matrices of order up to m, one cluster of P CTAs each
template <int P, class Src>
bool cholinv_launch(const Src& src, int np, int m, cudaStream_t s) {
  constexpr int kMaxSmem = 203 * 1024;   // with the static arrays below the SM's 227 KB
  const size_t smem = cholinv_smem<P>(m);
  if (smem > kMaxSmem) return false;
  auto* kern = cholinv_cluster_kernel<P, Src>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P * np, 1, 1);
  cfg.blockDim = dim3(CT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = P;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  // whether the device can run it, asked once (other threads wait for the answer)
  static const bool usable = [&] {
    cudaLaunchConfig_t probe = cfg;
    probe.gridDim = dim3(P, 1, 1);
    probe.dynamicSmemBytes = kMaxSmem;
    int nclusters = 0;
    const bool ok =
        (P <= 8 || cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&nclusters, kern, &probe) == cudaSuccess && nclusters > 0;
    if (!ok) cudaGetLastError();
    return ok;
  }();
  if (!usable) return false;
  if (cudaLaunchKernelEx(&cfg, kern, src) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  LAUNCH_NOTE(1);
  return true;
}

// sixteen CTAs a matrix, or eight where the device cannot schedule sixteen
template <class Src>
bool cholinv_any(const Src& src, int np, int m, cudaStream_t s) {
  return cholinv_launch<16>(src, np, m, s) || cholinv_launch<8>(src, np, m, s);
}

constexpr int kSMs = 152;

__global__ void pivot_recip_kernel(int64_t n, const double* v, double* r) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) r[i] = pivot_recip(v[i]);
}

}  // namespace

void pivot_recips(int64_t n, const double* v, double* r, cudaStream_t s) {
  if (n <= 0) return;
  pivot_recip_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, v, r);
  LAUNCH_NOTE(1);
}

int cholinv_max_order() { return kCholInvMax; }

bool cholinv_small(int m, const double2* W, int64_t ldw, double shift, double2* Li, int64_t ldi, double2* Lf,
                   int64_t ldl, int* info, cudaStream_t s, int info_base) {
  if (m < 1 || m > kCholInvMax) return false;
  CholOne src;
  src.p = CholProb{m, W, ldw, shift, Li, ldi, Lf, ldl, info, info_base};
  return cholinv_any(src, 1, m, s);
}

bool cholinv_batched(const BDesc* D, int np, int mmax, double shift_factor, cudaStream_t s) {
  if (mmax < 1 || mmax > kCholInvMax) return false;
  CholBatch src{D, shift_factor};
  return cholinv_any(src, np, mmax, s);
}

namespace {

// The recursion of chol_recursive: a block of order n splits as n1 + n2 (n1 a multiple of
// 128 near n / 2):
//   [A11 .  ]   [L11  .  ] [L11^H L21^H]
//   [A21 A22] = [L21 L22 ] [  .   L22^H],   L21 = A21 L11^-H,  A22 - L21 L21^H = L22 L22^H,
//   (L^-1)21 = -L22^-1 L21 L11^-1,
// the four off-diagonal products emulated, leaves of order <= kCholLeaf factored and
// inverted in one cluster launch each.
struct CholRec {
  const CholRes& r;
  cudaError_t err = cudaSuccess;

  bool product(OzOperand& a, OzOperand& b, int triA, int triB, double2* D, int64_t ldd) {
    err = oz_gemm(a, b, triA, triB, D, ldd, r.flags, r.s, nullptr, r.ws, r.ws_bytes);
    return err == cudaSuccess;
  }
  bool split(OzOperand& op, bool roleA, int rows, int K, const double2* X, int64_t ldx, int conj, int mask,
             bool cols) {
    err = oz_split(op, roleA ? r.memA : r.memB, rows, K, X, ldx, conj, mask, r.S, r.flags + 1, r.s, cols, nullptr,
                   r.group);
    return err == cudaSuccess;
  }
  // false with err == cudaSuccess: a leaf could not be launched (nothing enqueued if k0 == 0)
  bool run(int64_t n, double2* A, int64_t lda, double2* Li, int64_t ldi, int64_t k0) {
    if (n <= kCholLeaf) return cholinv_small((int)n, A, lda, 0.0, Li, ldi, A, lda, r.info, r.s, (int)k0);
    const int64_t n1 = std::max<int64_t>(128, (n / 2) / 128 * 128), n2 = n - n1;
    double2 *A21 = A + n1 * lda, *A22 = A21 + n1, *Li21 = Li + n1 * ldi, *Li22 = Li21 + n1;
    OzOperand a, b;
    const int i1 = (int)n1, i2 = (int)n2;
    if (!run(n1, A, lda, Li, ldi, k0)) return false;
    // L21 = A21 L11^-H: the columns of L11^-H are the conjugated rows of L11^-1 (k <= j)
    if (!split(a, true, i2, i1, A21, lda, 0, 0, false) || !split(b, false, i1, i1, Li, ldi, 1, 2, false) ||
        !product(a, b, 0, 2, A21, lda))
      return false;
    // A22 -= L21 L21^H (lower triangle), the product through the scratch T
    if (!split(a, true, i2, i1, A21, lda, 0, 0, false) || !split(b, false, i2, i1, A21, lda, 1, 0, false) ||
        !product(a, b, 0, 0, r.T, r.ldt))
      return false;
    zsub_lower(n2, A22, lda, r.T, r.ldt, r.s);
    if (!run(n2, A22, lda, Li22, ldi, k0 + n1)) {
      if (err == cudaSuccess) err = cudaErrorLaunchFailure;   // the first leaf launched: this one should too
      return false;
    }
    // T = L21 L11^-1 (the columns of the lower L11^-1 from their diagonal down), then
    // (L^-1)21 = -L22^-1 T
    if (!split(a, true, i2, i1, A21, lda, 0, 0, false) || !split(b, false, i1, i1, Li, ldi, 0, 3, true) ||
        !product(a, b, 0, 1, r.T, r.ldt))
      return false;
    if (!split(a, true, i2, i2, Li22, ldi, 0, 2, false) || !split(b, false, i1, i2, r.T, r.ldt, 0, 0, true) ||
        !product(a, b, 1, 0, Li21, ldi))
      return false;
    zneg(n2, n1, Li21, ldi, r.s);
    return true;
  }
};

}  // namespace

cudaError_t chol_recursive(int64_t n, double2* A, int64_t lda, double2* Li, int64_t ldi, const CholRes& r) {
  if (n < 1 || cholinv_max_order() < kCholLeaf) return cudaErrorNotSupported;
  if (n > kCholLeaf) zero_upper(n, Li, ldi, r.s);   // the leaves and products fill the lower part
  CholRec rec{r};
  if (!rec.run(n, A, lda, Li, ldi, 0)) return rec.err == cudaSuccess ? cudaErrorNotSupported : rec.err;
  if (n > kCholLeaf) zero_upper(n, A, lda, r.s);
  return cudaSuccess;
}

size_t zgram_counters() { return 4096; }

void zgram(int64_t n, int mx, int my, const double2* X, int64_t ldx, const double2* Y, int64_t ldy, double2* G,
           int64_t ldg, int herm, double2* part, size_t part_elems, unsigned* cnt, cudaStream_t s) {
  if (mx <= 0 || my <= 0) return;
  const int nti = (mx + GT - 1) / GT, ntj = (my + GT - 1) / GT;
  const int64_t tiles = (int64_t)nti * ntj;
  const int64_t active = herm ? (int64_t)nti * (nti + 1) / 2 : tiles;
  // slices: about eight CTAs per SM over the active tiles (the FP64 pipe is the limit, so
  // the point is an even spread), at least 2 GK rows each, within the partials' room and
  // the counters
  int64_t slices = (8 * kSMs + active - 1) / active;
  slices = std::min<int64_t>(slices, std::max<int64_t>(1, n / (2 * GK)));
  if (tiles > (int64_t)zgram_counters() || !part) slices = 1;
  while (slices > 1 && (size_t)(tiles * slices * GT * GT) > part_elems) slices /= 2;
  if (n == 0) slices = 1;
  int64_t per = (n + slices - 1) / slices;
  per = (per + GK - 1) / GK * GK;
  slices = n > 0 ? (n + per - 1) / per : 1;
  dim3 grid((unsigned)tiles, (unsigned)slices);
  void* kt0 = kt_enabled() ? kt_begin(s) : nullptr;
  // 4 x 8 tiles where the busiest SM's share of them is the smaller (slices: a second pass over the
  // partials)
  const int64_t tm = (mx + ZS_M - 1) / ZS_M, tn = (my + ZS_N - 1) / ZS_N;
  const double small = std::ceil((double)(herm ? tm * tn / 2 + std::min(tm, tn) : tm * tn) / kSMs) *
                       (ZS_M * ZS_N * (double)n + kZsOverhead);
  const double large = std::ceil((double)(active * slices) / kSMs) * (GT * GT * (double)per) +
                       (slices > 1 ? 2.0 * kZsOverhead : 0.0);
  // (a long column needs several CTAs an SM to hide its loads: n = 2048, m = 88 took 135 us)
  if (n > 0 && n <= 512 && small < large && tm <= 65535)
    zgram_small_kernel<<<dim3((unsigned)tn, (unsigned)tm), ZS_THREADS, 0, s>>>((int)n, mx, my, X, ldx, Y, ldy, G, ldg, herm);
  else zgram_kernel<<<grid, GT * GT, 0, s>>>(n, mx, my, X, ldx, Y, ldy, G, ldg, herm, ntj, (int)slices, per, part, cnt);
  LAUNCH_NOTE(1);
  if (kt0) {
    // work: 8 flop per complex multiply-add of the tiles formed (16 x 16 granularity)
    const double f = 8.0 * (double)active * (GT * GT) * (double)n;
    kt_end(kt0, 2, f, f, s);
  }
}

}  // namespace gevp

// FP32 eigenvectors of a small dense Hermitian matrix, the starting point of the FP64
// refinement in heev.cu: Householder tridiagonalisation, the implicit QL iteration on the real
// tridiagonal matrix, back-transformation.
//
// heev32_tri_kernel, one thread-block cluster of P CTAs per matrix:
//   1. G is scaled by a power of two and held in the CTAs' shared memory, row i in CTA i mod P.
//      (may_skip: when G is nearly diagonal already nothing else is done, see below.)
//   2. Tridiagonalisation, G <- H_k^H G H_k for k = 0 .. m-2, H_k = I - tau v v^H. Column k is
//      known to every CTA, and every warp forms v and tau itself (a warp reduction, no block
//      barrier). Each warp multiplies its own rows, p_i = tau (G v)_i, and sends p_i and, from
//      the owner of row k + 1, that row to all CTAs; one cluster barrier; then every CTA has
//      p, forms w = p - tau/2 (p^H v) v, updates its rows G -= v w^H + w v^H and computes
//      column k + 1 from the row it was sent. A thread owns the same entries in every step, so
//      one block barrier (for column k + 1) and one cluster barrier per step suffice.
//   3. QL: warp 0 of CTA 0 runs the scalar recurrence (all lanes alike) and leaves each
//      sweep's rotations in a shared-memory ring; warp 1 copies them to global memory and
//      publishes the number of finished sweeps; the remaining warps of all CTAs hold the rows of
//      the tridiagonal's eigenvector matrix, 32 to a warp, in shared memory and apply the
//      sweeps as they come. The recurrence is the critical path (about 100 clocks a rotation).
// heev32_back_kernel: one warp per eigenvector applies the reflectors, H_0 .. H_{m-2}, and writes
// the column to its place in ascending order in FP64.
//
// Why not Jacobi: a parallel Jacobi sweep is m - 1 rounds, each a cluster barrier and a rotation
// of all of G and Z, and a dense matrix takes eight or nine sweeps (m = 140: 1250 rounds of 3.9
// us; measured 5 ms, and 1.1 ms for the two sweeps of a warm start). The reduction here is m
// steps and the QL recurrence about m^2 rotations of 50 ns: m = 48 0.22 ms (Jacobi 0.90), m = 140
// 1.07 (4.5), m = 256 2.9 (18.9), m = 600 16 (36).
//
// Nearly diagonal matrices (may_skip; the projection of a block that has almost converged): every
// coupling at most 1e-3 of its diagonal gap (gaps below eta0 = 1e-6 ||G||_F counted as eta0:
// clusters, which FP32 cannot resolve either), and at most 1e-5 of it for gaps between eta0 and
// delta = 2 ||offdiag(G)||_F. The FP64 refinement started from Z = I has the clustering threshold
// delta in its first step: it corrects the pairs farther apart than delta there (to about
// 1e-6), those between eta0 and delta in its second step (to about 1e-10), and, converging
// quadratically, reaches FP64 accuracy in its last step as it would from computed vectors; the
// clusters go to the exact rotations after it.
//
// Every wait on another warp's or CTA's progress is bounded, and so are QL's sweeps and their memory;
// if one runs out the eigenvectors are written as NaN (the solver then reports that it did not
// converge, the per-step entry points the error).
#include "gevp_internal.cuh"
#include <cooperative_groups.h>
#include <algorithm>

namespace gevp {

namespace {

constexpr int HT = 512;            // threads of a CTA
constexpr int HW = HT / 32;
constexpr int kRing = 2048;        // rotations in flight between the recurrence and the copier
constexpr int kSweepRing = 128;    // sweeps in flight
constexpr uint32_t kSpin = 1u << 24;
constexpr int kHeevMax = 600;      // largest order: 38 rows of 600 FP32 complex in each of 16 CTAs

// one matrix: G is read; V, tau, rot, sweeps, ZT, w are scratch; ctl: 4 words
struct Heev32 {
  int m;
  const float2* G;
  float2* V;        // m x m: reflector k in row k
  float2* tau;      // m
  float2* rot;      // (c, s), 2 m^2
  int4* sweeps;     // (first column, rotations, offset), m^2
  float* ZT;        // m x m: row j = the tridiagonal's eigenvector j
  float* w;         // eigenvalues (scaled), unsorted
  int* ctl;         // [0] published sweeps, [1] 1 + all sweeps when done, [2] skipped, [3] failed (1 a wait, 2 QL)
  double2* Z;       // result, ld ldz
  int64_t ldz;
};

struct SrcOne {
  Heev32 p;
  __device__ bool get(int, Heev32& o) const {
    o = p;
    return true;
  }
};
// problems of a batch: the refinement's FP64 scratch holds this kernel's (it is written later)
struct SrcBatch {
  const BDesc* D;
  __device__ bool get(int b, Heev32& o) const {
    const BDesc& d = D[b];
    if (d.active && *d.active == 0) return false;
    o.m = d.m;
    o.G = d.G32;
    o.V = (float2*)d.hT;
    o.tau = d.Z32;
    o.rot = (float2*)d.hR;
    o.sweeps = (int4*)d.hS;
    o.ZT = (float*)d.hE;
    o.w = d.w32;
    o.ctl = d.perm;
    o.Z = d.hZ;
    o.ldz = d.m;
    return true;
  }
};

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a += conj(b) c
__device__ __forceinline__ void cfmac(float2& a, float2 b, float2 c) {
  a.x = fmaf(b.x, c.x, fmaf(b.y, c.y, a.x));
  a.y = fmaf(b.x, c.y, fmaf(-b.y, c.x, a.y));
}
__device__ __forceinline__ float wsum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float2 wsum2(float2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  return v;
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <int P>
__device__ __forceinline__ void group_sync() {
  if constexpr (P == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
}

// shared memory: the G rows, later the Z rows, the ring and the staging (CTA-wide), then the
// vectors of the reduction
__host__ __device__ inline int h_rows(int m, int P) { return (m + P - 1) / P; }
__host__ __device__ inline int h_groups(int m, int P) { return ((m + 31) / 32 + P - 1) / P; }   // Z row groups a CTA
__host__ __device__ inline size_t h_big(int m, int P) {
  const size_t g = (size_t)h_rows(m, P) * m * 8;
  const size_t z = (size_t)h_groups(m, P) * (32 * (m | 1) * 4 + 32 * 8) + kRing * 8 + kSweepRing * 8 + 16;
  return ((g > z ? g : z) + 15) / 16 * 16;
}
__host__ __device__ inline size_t h_smem(int m, int P) { return h_big(m, P) + (size_t)6 * m * 8 + (size_t)2 * m * 4; }

// Implicit QL iteration (Wilkinson shifts, chased from the bottom up; the procedure imtql2 of Martin
// and Wilkinson, Handbook for Automatic Computation II, published in EISPACK) on the symmetric
// tridiagonal matrix d[0..m-1], e[0..m-2] (shared memory, entries about 1 or less; d receives the
// eigenvalues), by one warp with all lanes alike. Rotation i mixes columns i and i + 1 of the
// eigenvector matrix: z_{i+1} <- s z_i + c z_{i+1}, z_i <- c z_i - s z_{i+1}; a sweep's come in
// descending i, without gaps. A coupling is negligible at FP32 rounding of its diagonal
// neighbours. Bound by the latency of one rotation's chain (a reciprocal square root and nine
// dependent multiply-adds).
template <class Sink>
__device__ __forceinline__ void ql_warp(int m, float* d, float* e, int lane, Sink& sink) {
  int sweeps = 0;
  for (int l = 0; l < m; ++l) {
    for (;;) {
      // the first negligible coupling at or after l
      int mm = m - 1;
      for (int b = l; b < m - 1; b += 32) {
        const int i = b + lane;
        const bool z = i < m - 1 && !(fabsf(e[i]) > 6e-8f * (fabsf(d[i]) + fabsf(d[i + 1])) + 1e-15f);
        const unsigned bal = __ballot_sync(0xffffffffu, z);
        if (bal) {
          mm = b + __ffs(bal) - 1;
          break;
        }
      }
      if (mm == l) break;
      // Two sweeps an eigenvalue are usual, thirty the limit: of all of them together, as the sweeps from
      // one l also split what lies above (three values of 416: 124 at one l, 760 in all)
      if (sweeps++ == 30 * m) {
        sink.gave_up(fabsf(e[l]));
        return;
      }
      if (!sink.room(mm - l)) return;
      const float el = e[l];
      float g = (d[l + 1] - d[l]) / (2.f * el);
      float r = sqrtf(g * g + 1.f);
      g = d[mm] - d[l] + el / (g + copysignf(r, g));
      float s = 1.f, c = 1.f, pp = 0.f;
      float ei = e[mm - 1], di = d[mm - 1], d1 = d[mm];
      sink.start(mm);
      __syncwarp();
      // (all lanes store the same values: a predicate on one lane would cost a branch a rotation)
      for (int i = mm - 1; i >= l; --i) {
        const int in = max(i - 1, 0);
        const float en = e[in], dn = d[in];   // for the next rotation (not written before it)
        const float f = s * ei, b = c * ei;
        const float h = fmaf(f, f, g * g);
        const bool ok = h > 1e-36f;           // else nothing is left to rotate: the identity
        float ri;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ri) : "f"(h));
        ri = ok ? ri : 0.f;
        e[i + 1] = h * ri;
        s = f * ri;
        c = ok ? g * ri : 1.f;
        g = d1 - pp;
        r = fmaf(di - g, s, 2.f * c * b);
        pp = s * r;
        d[i + 1] = g + pp;
        sink.rotation(i, c, s);
        g = fmaf(c, r, -b);
        d1 = di;
        ei = en;
        di = dn;
      }
      d[l] = d1 - pp;
      e[l] = g;
      e[mm] = 0.f;
      sink.end(mm - 1, l);
      __syncwarp();
    }
  }
}

template <int P, int NT, class Src>
__global__ void __launch_bounds__(HT, 1) heev32_tri_kernel(Src src, int may_skip) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char hsm[];
  __shared__ float red[HW][2];
  __shared__ float part[4];
  __shared__ volatile int ring_pub[4];   // [0] rotations, [1] sweeps published by the recurrence, [2] done; [3] rotations copied
  __shared__ volatile int ring_sc;       // sweeps copied
  Heev32 p;
  const int rank = P == 1 ? 0 : (int)(blockIdx.x % P);
  if (!src.get(blockIdx.x / P, p)) return;   // uniform over the cluster
  const int m = p.m;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int R = h_rows(m, P);
  float2* A = (float2*)hsm;   // own rows i = rank + P t
  float2* vec = (float2*)(hsm + h_big(m, P));
  float2* xb[2] = {vec, vec + m};
  float2* pb[2] = {vec + 2 * m, vec + 3 * m};
  float2* rb[2] = {vec + 4 * m, vec + 5 * m};
  float* d = (float*)(vec + 6 * m);
  float* e = d + m;
  cg::cluster_group cl = cg::this_cluster();
  auto remote = [&](auto* q, int r) {
    if constexpr (P == 1) return q;
    else return cl.map_shared_rank(q, r);
  };
  // sums (or maxima) over the cluster, in rank order
  auto all_sum = [&](float v, int slot, bool is_max) {
    v = is_max ? v : wsum(v);
    if (is_max)
      for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) red[warp][0] = v;
    __syncthreads();
    if (tid == 0) {
      float t = 0.f;
      for (int q = 0; q < HW; ++q) t = is_max ? fmaxf(t, red[q][0]) : t + red[q][0];
      part[slot] = t;
    }
    group_sync<P>();
    float t = 0.f;
    for (int q = 0; q < P; ++q) {
      const float o = *remote(&part[slot], q);
      t = is_max ? fmaxf(t, o) : t + o;
    }
    return t;
  };

  // ---- load and scale
  float mx = 0.f;
  for (int t = warp; t < R; t += HW) {
    const int i = rank + P * t;
    for (int j = lane; j < m; j += 32) {
      const float2 g = i < m ? p.G[(int64_t)i * m + j] : make_float2(0.f, 0.f);
      A[t * m + j] = g;
      mx = fmaxf(mx, fmaxf(fabsf(g.x), fabsf(g.y)));
    }
  }
  if (rank == 0 && tid < 4) {
    p.ctl[tid] = 0;
    ring_pub[tid] = 0;
    ring_sc = 0;
  }
  mx = all_sum(mx, 0, true);
  int ex = 0;
  if (mx > 0.f && mx < 3e38f) ex = ilogbf(mx);
  const float sc = ldexpf(1.f, max(-126, min(126, -ex)));
  float fro = 0.f, off = 0.f;
  for (int t = warp; t < R; t += HW) {
    const int i = rank + P * t;
    for (int j = lane; j < m; j += 32) {
      const float2 g = make_float2(A[t * m + j].x * sc, A[t * m + j].y * sc);
      A[t * m + j] = g;
      const float s = g.x * g.x + g.y * g.y;
      fro += s;
      if (i != j) off += s;
    }
  }
  fro = all_sum(fro, 1, false);
  off = all_sum(off, 2, false);
  bool skip = !(off > 1e-16f * fro);
  if (!skip && may_skip) {
    const float eta0 = 1e-6f * sqrtf(fro), delta = 2.f * sqrtf(off);
    bool c = false;
    for (int t = warp; t < R; t += HW) {
      const int i = rank + P * t;
      if (i >= m) break;
      const float di = A[t * m + i].x;
      for (int j = lane; j < m; j += 32) {
        if (i == j) continue;
        const float2 g = A[t * m + j];
        const float gap = fabsf(di - p.G[(int64_t)j * m + j].x * sc);
        const float a = hypotf(g.x, g.y);
        c |= a > 1e-3f * fmaxf(gap, eta0) || (gap > eta0 && gap <= delta && a > 1e-5f * gap);
      }
    }
    skip = !(all_sum(c ? 1.f : 0.f, 3, true) > 0.f);
  }
  if (skip) {
    if (rank == 0) {
      for (int i = tid; i < m; i += HT) p.w[i] = p.G[(int64_t)i * m + i].x;
      if (tid == 0) p.ctl[2] = 1;
    }
    group_sync<P>();   // no CTA leaves while another may still read its shared memory
    return;
  }

  // ---- tridiagonalisation
  for (int j = tid; j < m; j += HT) {
    const float2 g = p.G[j];   // row 0
    xb[0][j] = make_float2(g.x * sc, -g.y * sc);
    if (j == 0) d[0] = g.x * sc;
  }
  group_sync<P>();
  for (int k = 0; k + 1 < m; ++k) {
    const int cur = k & 1;
    const float2* x = xb[cur];
    // v, tau, beta from column k (every warp)
    float2 v[NT];
    float xn = 0.f;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int j = 32 * t + lane;
      v[t] = (j > k + 1 && j < m) ? x[j] : make_float2(0.f, 0.f);
      xn += v[t].x * v[t].x + v[t].y * v[t].y;
    }
    const float2 al = x[k + 1];
    xn = wsum(xn);
    float beta = al.x;
    float2 tau = make_float2(0.f, 0.f), inv = make_float2(0.f, 0.f);
    // A column below 1e-15 of the matrix's largest entry (which is about 1 here) counts as reduced: QL
    // drops such couplings, FP32 rounding is 1e-7, and its squares would leave the FP32 range (1 / |x|^2
    // infinite, the reflector NaN). Matrices of low rank and graded ones come here: their rounding
    // residue shrinks by 1e-8 a step.
    if ((xn > 0.f || al.y != 0.f) && al.x * al.x + al.y * al.y + xn > 1e-30f) {
      beta = -copysignf(sqrtf(al.x * al.x + al.y * al.y + xn), al.x);
      const float ib = 1.f / beta;
      tau = make_float2((beta - al.x) * ib, -al.y * ib);
      const float2 df = make_float2(al.x - beta, al.y);
      const float n2 = 1.f / (df.x * df.x + df.y * df.y);
      inv = make_float2(df.x * n2, -df.y * n2);
    }
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int j = 32 * t + lane;
      v[t] = j == k + 1 ? make_float2(1.f, 0.f) : cmul(v[t], inv);
    }
    if (rank == k % P && warp == HW - 1) {
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const int j = 32 * t + lane;
        if (j > k && j < m) p.V[(int64_t)k * m + j] = v[t];
      }
      if (lane == 0) p.tau[k] = tau;
    }
    if (tid == 0) e[k] = beta;
    // row k + 1 (before this step's update) to every CTA
    if (rank == (k + 1) % P) {
      const float2* row = A + (k + 1) / P * m;
      for (int q = tid; q < P * (m - k - 1); q += HT) {
        const int j = k + 1 + q / P;
        remote(rb[cur], q % P)[j] = row[j];
      }
    }
    // p = tau G v on the own rows
    for (int t = warp; t < R; t += HW) {
      const int i = rank + P * t;
      if (i <= k || i >= m) continue;
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int s = 0; s < NT; ++s) {
        const int j = 32 * s + lane;
        if (j > k && j < m) cfma(acc, A[t * m + j], v[s]);
      }
      acc = cmul(tau, wsum2(acc));
      if (lane < P) remote(pb[cur], lane)[i] = acc;
    }
    group_sync<P>();
    // w = p - tau / 2 (p^H v) v; column k + 1; the own rows
    float2 w[NT];
    float2 dot = make_float2(0.f, 0.f);
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int j = 32 * t + lane;
      w[t] = (j > k && j < m) ? pb[cur][j] : make_float2(0.f, 0.f);
      cfmac(dot, w[t], v[t]);
    }
    dot = cmul(make_float2(-0.5f * tau.x, -0.5f * tau.y), wsum2(dot));
#pragma unroll
    for (int t = 0; t < NT; ++t) cfma(w[t], dot, v[t]);
    if (warp == 0) {
      float2 w1 = pb[cur][k + 1];   // w at k + 1, where v = 1
      w1 = make_float2(w1.x + dot.x, w1.y + dot.y);
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const int j = 32 * t + lane;
        if (j <= k || j >= m) continue;
        const float2 r = rb[cur][j];
        // conj(G[k+1][j]) - v_j conj(w_{k+1}) - w_j
        const float2 c = cmul(v[t], make_float2(w1.x, -w1.y));
        const float2 y = make_float2(r.x - c.x - w[t].x, -r.y - c.y - w[t].y);
        if (j == k + 1) d[j] = y.x;
        else xb[cur ^ 1][j] = y;
      }
    }
    for (int t = warp; t < R; t += HW) {
      const int i = rank + P * t;
      if (i <= k + 1 || i >= m) continue;
      const float2 vi = cmul(x[i], inv);
      float2 wi = pb[cur][i];
      cfma(wi, dot, vi);
#pragma unroll
      for (int s = 0; s < NT; ++s) {
        const int j = 32 * s + lane;
        if (j > k + 1 && j < m) {
          float2 a = A[t * m + j];
          const float2 b = cmul(vi, make_float2(w[s].x, -w[s].y)), c = cmul(wi, make_float2(v[s].x, -v[s].y));
          A[t * m + j] = make_float2(a.x - b.x - c.x, a.y - b.y - c.y);
        }
      }
    }
    __syncthreads();
  }
  if (tid == 0) e[m - 1] = 0.f;
  group_sync<P>();   // the G rows are free from here on

  // ---- QL
  const int ldz = m | 1;
  const int ng = h_groups(m, P);
  float* zrows = (float*)hsm;                               // [ng][32][ldz]
  float2* stage = (float2*)(zrows + (size_t)ng * 32 * ldz + ((ng * 32 * ldz) & 1));   // [ng][32]
  float2* ring = stage + 32 * ng;
  int2* sring = (int2*)(ring + kRing);
  const int64_t cap = (int64_t)2 * m * m - m;
  if (rank == 0 && warp == 0) {
    struct ToRing {
      float2* ring;
      int2* sring;
      volatile int* pub;
      volatile int* sc;
      int* failed;
      int m, lane, pos, ns, pos0;
      int64_t cap;
      __device__ void gave_up(float) {
        if (lane == 0) *failed = 2;
      }
      __device__ bool room(int) {
        if (pos + m > cap || ns + 1 >= m * m) {
          gave_up(0.f);
          return false;
        }
        int ok = 0;   // lane 0's decision holds for the warp
        if (lane == 0) {
          uint32_t spin = 0;
          while ((pos + m - pub[3] > kRing || ns + 1 - *sc > kSweepRing) && ++spin < kSpin) __nanosleep(64);
          ok = spin < kSpin;
          if (!ok) *failed = 1;
        }
        pos0 = pos;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();
        return ok != 0;
      }
      __device__ void start(int) {}
      __device__ void rotation(int, float c, float s) {
        ring[pos % kRing] = make_float2(c, s);
        ++pos;
      }
      __device__ void end(int first, int) {
        if (pos == pos0) return;
        if (lane == 0) sring[ns % kSweepRing] = make_int2(first, pos - pos0);
        __syncwarp();
        __threadfence_block();
        ++ns;
        if (lane == 0) pub[1] = ns;
      }
    } sink{ring, sring, ring_pub, &ring_sc, p.ctl + 3, m, lane, 0, 0, 0, cap};
    ql_warp(m, d, e, lane, sink);
    __threadfence_block();
    if (lane == 0) ring_pub[2] = 1;
    for (int i = lane; i < m; i += 32) p.w[i] = d[i];
  } else if (rank == 0 && warp == 1) {
    int done = 0, sc_ = 0, off_ = 0;
    uint32_t spin = 0;
    while (spin < kSpin) {
      // one reading for the whole warp: lanes that saw different counts would publish a sweep that
      // others have not copied
      int fin = 0, ns = 0;
      if (lane == 0) {
        fin = ring_pub[2];
        __threadfence_block();
        ns = ring_pub[1];
        __threadfence_block();
      }
      fin = __shfl_sync(0xffffffffu, fin, 0);
      ns = __shfl_sync(0xffffffffu, ns, 0);
      __syncwarp();   // the other lanes' reads of the ring come after lane 0's of the count
      if (ns > sc_) {
        spin = 0;
        for (int q = sc_ + lane; q < ns; q += 32) {
          // offsets: the sweeps' counts add up in order
          int o = off_;
          for (int u = sc_; u < q; ++u) o += sring[u % kSweepRing].y;
          const int2 s = sring[q % kSweepRing];
          p.sweeps[q] = make_int4(s.x, s.y, o, 0);
        }
        int o = off_;
        for (int u = sc_; u < ns; ++u) o += sring[u % kSweepRing].y;
        for (int q = done + lane; q < o; q += 32) p.rot[q] = ring[q % kRing];
        off_ = o;
        done = o;
        sc_ = ns;
        __threadfence();
        __syncwarp();
        if (lane == 0) {
          ring_pub[3] = done;
          ring_sc = sc_;
          st_release(&p.ctl[0], sc_);
        }
      } else if (fin) {
        break;
      } else {
        __nanosleep(64);
        ++spin;
      }
    }
    if (lane == 0) {
      if (spin >= kSpin) p.ctl[3] = 1;
      st_release(&p.ctl[1], sc_ + 1);
    }
  } else {
    // Z row groups: group grp (rows 32 grp ..) lives in CTA grp mod P, warps from 2 on
    for (int t = warp - 2; t >= 0 && t < ng; t += HW - 2) {
      const int grp = rank + P * t;
      if (32 * grp >= m) break;
      float* zr = zrows + (size_t)(t * 32 + lane) * ldz;
      const int row = 32 * grp + lane;
      for (int j = 0; j < m; ++j) zr[j] = j == row ? 1.f : 0.f;
      float2* st = stage + 32 * t;
      int mine = 0;
      uint32_t spin = 0;
      for (;;) {
        int n = 0, fin = 0;
        if (lane == 0) {
          fin = ld_acquire(&p.ctl[1]);
          n = fin ? fin - 1 : ld_acquire(&p.ctl[0]);
        }
        n = __shfl_sync(0xffffffffu, n, 0);
        fin = __shfl_sync(0xffffffffu, fin, 0);
        __syncwarp();   // (a shuffle alone orders no memory: the sweeps are read behind lane 0's acquire)
        if (mine >= n) {
          if (fin) break;
          __nanosleep(128);
          if (++spin >= kSpin) {
            if (lane == 0) p.ctl[3] = 1;
            break;
          }
          continue;
        }
        spin = 0;
        for (; mine < n; ++mine) {
          const int4 s = __ldcg(p.sweeps + mine);
          const float2* q = p.rot + s.z;
          float f = zr[s.x + 1];
          float2 nx = lane < s.y ? __ldcg(q + lane) : make_float2(1.f, 0.f);
          for (int b = 0; b < s.y; b += 32) {
            __syncwarp();
            st[lane] = nx;
            __syncwarp();
            if (b + 32 + lane < s.y) nx = __ldcg(q + b + 32 + lane);
            const int cnt = min(32, s.y - b);
            float* zi = zr + s.x - b;
            for (int u = 0; u < cnt; ++u) {
              const float2 cs = st[u];
              const float z = zi[-u];
              zi[1 - u] = fmaf(cs.y, z, cs.x * f);
              f = fmaf(cs.x, z, -cs.y * f);
            }
          }
          zr[s.x + 1 - s.y] = f;
        }
      }
      __syncwarp();
      if (row < m)
        for (int j = 0; j < m; ++j) p.ZT[(int64_t)j * m + row] = zr[j];
    }
  }
  group_sync<P>();
}

// one warp per eigenvector: y = H_0 (H_1 (... H_{m-2} z)), written to the column of its rank
constexpr int HB_CH = 8;   // reflectors staged at a time
template <int NT, class Src>
__global__ void __launch_bounds__(256) heev32_back_kernel(Src src) {
  extern __shared__ float2 vsm[];   // [HB_CH][m]
  Heev32 p;
  if (!src.get(blockIdx.y, p)) return;
  const int m = p.m;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int j0 = blockIdx.x * 8;
  if (j0 >= m) return;
  const int j = min(m - 1, j0 + warp);
  const bool skip = p.ctl[2] != 0, bad = p.ctl[3] != 0;
  const int kj = rank_key(p.w[j]);
  int rk = 0;
  for (int i = lane; i < m; i += 32) rk += rank_before(rank_key(p.w[i]), i, kj, j) ? 1 : 0;
  for (int o = 16; o > 0; o >>= 1) rk += __shfl_xor_sync(0xffffffffu, rk, o);
  float2 y[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    const int r = 32 * t + lane;
    y[t] = make_float2(skip ? (r == j ? 1.f : 0.f) : (r < m ? p.ZT[(int64_t)j * m + r] : 0.f), 0.f);
  }
  if (!skip) {
    for (int k1 = m - 2; k1 >= 0; k1 -= HB_CH) {
      const int cnt = min(HB_CH, k1 + 1);
      __syncthreads();
      for (int q = threadIdx.x; q < cnt * m; q += 256) {
        const int k = k1 - q / m, r = q % m;
        vsm[q] = r > k ? p.V[(int64_t)k * m + r] : make_float2(0.f, 0.f);
      }
      __syncthreads();
      for (int u = 0; u < cnt; ++u) {
        const float2* v = vsm + u * m;
        float2 dot = make_float2(0.f, 0.f);
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const int r = 32 * t + lane;
          if (r < m) cfmac(dot, v[r], y[t]);
        }
        const float2 tau = p.tau[k1 - u];
        dot = cmul(tau, wsum2(dot));
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const int r = 32 * t + lane;
          if (r < m) {
            const float2 c = cmul(dot, v[r]);
            y[t] = make_float2(y[t].x - c.x, y[t].y - c.y);
          }
        }
      }
    }
  }
  if (j0 + warp >= m) return;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    const int r = 32 * t + lane;
    if (r < m) p.Z[(int64_t)r * p.ldz + rk] = bad ? make_double2(nan, nan) : make_double2(y[t].x, y[t].y);
  }
}

// Lanczos: the eigenvalues of the tridiagonal matrix of alpha, beta and the squared first entries
// of its eigenvectors (the Ritz weights of the start vector), then the bounds; one warp a problem.
// ab: alpha_j, beta_j interleaved, ab[2 k_max] (an int) the steps made, negative after a
// breakdown. out[0..4] as lanczos_bounds (gevp_internal.cuh) says.
__device__ void lanczos_tail(int k, int64_t n, int count, const float* ab, int ke, double* out) {
  __shared__ float d[64], e[64], z[64], ws[64], zs[64];
  const int lane = threadIdx.x;
  int kk = ke < 0 ? -ke : min(ke, k);
  kk = max(kk, 1);
  float mx = 0.f;
  for (int i = lane; i < kk; i += 32) {
    d[i] = ab[2 * i];
    e[i] = i + 1 < kk ? ab[2 * i + 1] : 0.f;
    z[i] = i == 0 ? 1.f : 0.f;
    mx = fmaxf(mx, fmaxf(fabsf(d[i]), fabsf(e[i])));
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  int ex = 0;
  if (mx > 0.f && mx < 3e38f) ex = max(-126, min(126, ilogbf(mx)));
  const float sc = ldexpf(1.f, -ex);
  for (int i = lane; i < kk; i += 32) {
    d[i] *= sc;
    e[i] *= sc;
  }
  __syncwarp();
  struct FirstRow {
    float* z;
    int lane;
    float f;
    __device__ void gave_up(float el) { left = fmaxf(left, el); }
    __device__ bool room(int) { return true; }
    __device__ void start(int mm) { f = z[mm]; }
    __device__ void rotation(int i, float c, float s) {
      const float zi = z[i];
      z[i + 1] = fmaf(s, zi, c * f);
      f = fmaf(c, zi, -s * f);
      last = i;
    }
    __device__ void end(int, int) {
      if (last >= 0) z[last] = f;
      last = -1;
    }
    int last;
    float left;   // the largest coupling that an eigenvalue was left with
  } sink{z, lane, 0.f, -1, 0.f};
  ql_warp(kk, d, e, lane, sink);
  __syncwarp();
  for (int i = lane; i < kk; i += 32) {
    int r = 0;
    for (int j = 0; j < kk; ++j) r += rank_before(rank_key(d[j]), j, rank_key(d[i]), i) ? 1 : 0;
    ws[r] = d[i];
    zs[r] = z[i];
  }
  __syncwarp();
  if (lane != 0) return;
  const double up = ldexp(1.0, ex);
  const double tmin = ws[0] * up, tmax = ws[kk - 1] * up;
  const double beta = ke < 0 ? 0.0 : fabs((double)ab[2 * (kk - 1) + 1]);
  out[0] = tmin;
  out[1] = tmax;
  out[2] = tmax + beta + 1e-5 * fmax(fabs(tmin), fabs(tmax)) + sink.left * up;
  out[4] = beta;
  double aest = tmax, cum = 0.0;
  if (count > 0)
    for (int r = 0; r < kk; ++r) {
      cum += (double)zs[r] * zs[r] * (double)n;
      if (cum >= (double)count) {
        aest = ws[r] * up;
        break;
      }
    }
  out[3] = aest;
}
__global__ void __launch_bounds__(32) lanczos_tail_kernel(int k, int64_t n, int count, const float* ab, int k_max,
                                                          double* out) {
  lanczos_tail(k, n, count, ab, ((const int*)ab)[2 * k_max], out);
}
__global__ void __launch_bounds__(32) lanczos_tail_batched_kernel(const BDesc* D, int k, int use_count, int k_max,
                                                                  int out_off) {
  const BDesc& b = D[blockIdx.x];
  if (b.active && *b.active == 0) return;
  lanczos_tail(k, b.n, use_count ? b.m : 0, b.ab, ((const int*)b.ab)[2 * k_max], b.bounds + out_off);
}

template <int P, int NT, class Src>
bool tri_launch(const Src& src, int np, int mmax, int may_skip, cudaStream_t s) {
  auto* kern = heev32_tri_kernel<P, NT, Src>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P * np, 1, 1);
  cfg.blockDim = dim3(HT, 1, 1);
  cfg.dynamicSmemBytes = h_smem(mmax, P);
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
    constexpr int kSmem = 220 * 1024;
    cudaLaunchConfig_t probe = cfg;
    probe.gridDim = dim3(P, 1, 1);
    probe.dynamicSmemBytes = kSmem;
    int n = 0;
    const bool ok =
        (P <= 8 || cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, kern, &probe) == cudaSuccess && n > 0;
    if (!ok) cudaGetLastError();
    return ok;
  }();
  if (!usable) return false;
  if (cfg.dynamicSmemBytes > 220 * 1024) return false;
  if (cudaLaunchKernelEx(&cfg, kern, src, may_skip) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  constexpr int NB = NT;
  heev32_back_kernel<NB, Src><<<dim3((mmax + 7) / 8, np), 256, (size_t)HB_CH * mmax * sizeof(float2), s>>>(src);
  LAUNCH_NOTE(2);
  return true;
}

// CTAs per matrix: one holds G and has no cluster barriers up to 72 rows; above that a step is
// bound by the instructions of one SM (m = 72: 1.5 us a step), so eight share them; sixteen where eight
// cannot hold G
template <class Src>
bool tri_dispatch(const Src& src, int np, int mmax, int may_skip, cudaStream_t s) {
  if (mmax < 1 || mmax > kHeevMax) return false;
  if (mmax <= 32) return tri_launch<1, 1>(src, np, mmax, may_skip, s);
  if (mmax <= 72) return tri_launch<1, 3>(src, np, mmax, may_skip, s);
  if (mmax <= 160) return tri_launch<8, 5>(src, np, mmax, may_skip, s);
  if (mmax <= 256) return tri_launch<8, 8>(src, np, mmax, may_skip, s);
  if (mmax <= 416) return tri_launch<8, 13>(src, np, mmax, may_skip, s);
  return tri_launch<16, 19>(src, np, mmax, may_skip, s);
}

}  // namespace

bool heev32(int m, const float2* G, double2* Z, int64_t ldz, float* w, int* ctl, float2* tau, double2* sV, double2* sR,
            double2* sS, double2* sZ, int may_skip, cudaStream_t s) {
  SrcOne src;
  src.p.m = m;
  src.p.G = G;
  src.p.V = (float2*)sV;
  src.p.tau = tau;
  src.p.rot = (float2*)sR;
  src.p.sweeps = (int4*)sS;
  src.p.ZT = (float*)sZ;
  src.p.w = w;
  src.p.ctl = ctl;
  src.p.Z = Z;
  src.p.ldz = ldz;
  return tri_dispatch(src, 1, m, may_skip, s);
}

void lanczos_tail(int k, int64_t n, int count, const float* ab, int k_max, double* out, cudaStream_t s) {
  lanczos_tail_kernel<<<1, 32, 0, s>>>(k, n, count, ab, k_max, out);
  LAUNCH_NOTE(1);
}
void lanczos_tail_batched(const BDesc* D, int np, int k, int use_count, int k_max, int out_off, cudaStream_t s) {
  lanczos_tail_batched_kernel<<<np, 32, 0, s>>>(D, k, use_count, k_max, out_off);
  LAUNCH_NOTE(1);
}

bool heev32_batched(const BDesc* D, int np, int mmax, cudaStream_t s) {
  SrcBatch src{D};
  return tri_dispatch(src, np, mmax, 0, s);
}

}  // namespace gevp

// k-step Lanczos with full re-orthogonalisation on an FP32 copy of a Hermitian matrix, for
// the Chebyshev filter's interval: an upper bound of the spectrum (largest Ritz value plus
// the last residual norm |beta_k|, as in Zhou, Saad, Tiago & Chelikowsky 2006) and an
// estimate of the count-th eigenvalue from the Ritz values weighted by the squared first
// components of the tridiagonal's eigenvectors (a Lanczos quadrature of the spectral
// density). Bounds need a few digits only, so FP32 suffices; the matrix-vector product is
// HBM/L2 bound (one warp per row, coalesced row reads).
#include "gevp_internal.cuh"
#include <algorithm>
#include <atomic>
#include <cooperative_groups.h>

namespace gevp {

namespace {

constexpr int KMAX = 64;
constexpr int kLanczosSmem = 180 * 1024;   // dynamic, of a Lanczos CTA

__device__ __forceinline__ uint64_t mix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

__global__ void matvec32_kernel(int64_t n, const float2* M, int64_t ldm, const float2* v, float2* w) {
  int64_t row = blockIdx.x * (int64_t)(blockDim.x / 32) + threadIdx.x / 32;
  int lane = threadIdx.x % 32;
  if (row >= n) return;
  const float2* r = M + row * ldm;
  float2 acc = make_float2(0.f, 0.f);
  for (int64_t j = lane; j < n; j += 32) cfma(acc, r[j], v[j]);
  for (int o = 16; o > 0; o >>= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
  }
  if (lane == 0) w[row] = acc;
}

__device__ float2 warp_sum2(float2 v) {
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  return v;
}

// V: (k+1) vectors of length n, vector-major. ab[2j] = alpha_j, ab[2j+1] = beta_j.
// ab[2*KMAX] (as int) = effective number of steps.
__global__ void __launch_bounds__(1024) lanczos_init_kernel(int64_t n, float2* V, uint64_t seed, float* ab) {
  __shared__ float red[32];
  float s = 0.f;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    uint64_t h1 = mix64(seed ^ mix64(2 * (uint64_t)i)), h2 = mix64(seed ^ mix64(2 * (uint64_t)i + 1));
    float u1 = ((float)(h1 >> 40) + 0.5f) * (1.0f / 16777216.0f);
    float u2 = ((float)(h2 >> 40) + 0.5f) * (1.0f / 16777216.0f);
    float2 z = make_float2(u1 - 0.5f, u2 - 0.5f);
    V[i] = z;
    s += z.x * z.x + z.y * z.y;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int i = 0; i < (int)(blockDim.x / 32); ++i) t += red[i];
    red[0] = rsqrtf(t);
    ((int*)ab)[2 * KMAX] = 0;
  }
  __syncthreads();
  float inv = red[0];
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) { float2 z = V[i]; V[i] = make_float2(z.x * inv, z.y * inv); }
}

// Lanczos steps j0 .. k-1 of one problem by a cluster of CTAs, each owning a slice of the rows: the
// product with its rows of M (full; otherwise w holds it), two passes of classical Gram-Schmidt
// against V[0..j], the norm, its slice of V[j+1]. The coefficients are added up over the cluster
// by every CTA in rank order, so all take the same decisions. One CTA with all rows is bound by its own
// loads of V (14.7 us a step at n = 50, 34.5 at n = 2048, where the vectors are 16 KB each); here a
// slice and its vectors stay in L1 and a step is three or four cluster barriers: 5.4 and 9.7 us, 4.8
// and 26 with the product (1.7 and 9.9 us as a launch over the whole GPU).
struct LanczosOne {
  int64_t n;
  const float2* M;
  int64_t ldm;
  float2 *V, *w;
  float* ab;
};
struct LanczosSrcOne {
  LanczosOne p;
  __device__ bool get(int, LanczosOne& o) const {
    o = p;
    return true;
  }
};
struct LanczosSrcBatch {
  const BDesc* D;
  __device__ bool get(int i, LanczosOne& o) const {
    const BDesc& d = D[i];
    if (d.active && *d.active == 0) return false;
    o = LanczosOne{d.n, d.M32, d.n, d.V, d.lvec, d.ab};
    return true;
  }
};

constexpr int LT = 1024;         // threads of a Lanczos CTA
constexpr int kLanczosCta = 16;  // CTAs of a cluster at most

template <class Src>
__global__ void __launch_bounds__(LT, 1) lanczos_cluster_kernel(Src src, int j0, int k, int full) {
  extern __shared__ float2 lsm[];
  __shared__ float2 slot[2][kLanczosCta][KMAX + 1];
  __shared__ float2 hp[KMAX + 1], h[KMAX + 1];
  __shared__ float red[LT / 32];
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  LanczosOne p;
  if (!src.get((int)blockIdx.x / C, p)) return;   // (the whole cluster)
  const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
  int* keff = (int*)(p.ab + 2 * KMAX);
  if (*keff < j0) return;   // broke down earlier (rank 0 writes it after the barriers below)
  const int64_t n = p.n, per = (n + C - 1) / C, r0 = min(n, rank * per);
  const int rows = (int)(min(n, r0 + per) - r0);
  float2* ws = lsm;
  float2* vs = lsm + per;
  int turn = 0;
  // h[c] = sum over the CTAs of their hp[c], c < cnt; each writes its part to every CTA (two buffers in
  // turn: a part is read before its CTA arrives at the next barrier)
  auto add_up = [&](int cnt) {
    __syncthreads();
    if (C == 1) {
      for (int c = tid; c < cnt; c += LT) h[c] = hp[c];
    } else {
      for (int t = tid; t < cnt * C; t += LT) {
        float2* to = cl.map_shared_rank(&slot[turn][rank][t / C], t % C);
        *to = hp[t / C];
      }
      cl.sync();
      for (int c = tid; c < cnt; c += LT) {
        float2 t = slot[turn][0][c];
        for (int r = 1; r < C; ++r) {
          const float2 v = slot[turn][r][c];
          t.x += v.x;
          t.y += v.y;
        }
        h[c] = t;
      }
      turn ^= 1;
    }
    __syncthreads();
  };
  float bprev = j0 > 0 ? p.ab[2 * j0 - 1] : 0.f;
  int made = 0;
  if (C > 1) cl.sync();   // every CTA has started before another writes to its slots
  for (int j = j0; j < k; ++j) {
    if (full) {
      const float2* vj = p.V + (int64_t)j * n;
      for (int64_t i = tid; i < n; i += LT) vs[i] = __ldcg(vj + i);
      __syncthreads();
      for (int i = warp; i < rows; i += LT / 32) {
        const float2* m = p.M + (r0 + i) * p.ldm;
        float2 a0 = make_float2(0.f, 0.f), a1 = a0;
        int64_t c = lane;
        for (; c + 224 < n; c += 256) {   // eight loads in flight a lane
          float2 x[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) x[u] = m[c + 32 * u];
#pragma unroll
          for (int u = 0; u < 8; ++u) cfma(u % 2 ? a1 : a0, x[u], vs[c + 32 * u]);
        }
        for (; c < n; c += 32) cfma(a0, m[c], vs[c]);
        a0.x += a1.x;
        a0.y += a1.y;
        a0 = warp_sum2(a0);
        if (lane == 0) ws[i] = a0;
      }
    } else {
      for (int i = tid; i < rows; i += LT) ws[i] = p.w[r0 + i];
    }
    __syncthreads();
    float alpha = 0.f;
    for (int pass = 0; pass < 2; ++pass) {
      for (int c = warp; c <= j; c += LT / 32) {
        const float2* vc = p.V + (int64_t)c * n + r0;
        float2 d = make_float2(0.f, 0.f);
        for (int i = lane; i < rows; i += 32) {
          const float2 a = vc[i], b = ws[i];
          d.x += a.x * b.x + a.y * b.y;   // conj(a) * b
          d.y += a.x * b.y - a.y * b.x;
        }
        d = warp_sum2(d);
        if (lane == 0) hp[c] = d;
      }
      add_up(j + 1);
      if (pass == 0) alpha = h[j].x;
      for (int i0 = 0; i0 < rows; i0 += LT / 8) {   // eight lanes a row
        const int i = i0 + tid / 8;
        float2 d = make_float2(0.f, 0.f);
        if (i < rows)
          for (int c = tid % 8; c <= j; c += 8) cfma(d, p.V[(int64_t)c * n + r0 + i], h[c]);
        for (int o = 4; o > 0; o >>= 1) {
          d.x += __shfl_xor_sync(0xffffffffu, d.x, o);
          d.y += __shfl_xor_sync(0xffffffffu, d.y, o);
        }
        if (i < rows && tid % 8 == 0) ws[i] = make_float2(ws[i].x - d.x, ws[i].y - d.y);
      }
      __syncthreads();
    }
    float s = 0.f;
    for (int i = tid; i < rows; i += LT) s += ws[i].x * ws[i].x + ws[i].y * ws[i].y;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (warp == 0) {
      s = red[lane];
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) hp[0] = make_float2(s, 0.f);
    }
    add_up(1);
    const float nrm = sqrtf(h[0].x);
    const bool go = nrm > 1e-6f * (fabsf(alpha) + bprev) && nrm > 0.f;
    if (rank == 0 && tid == 0) {
      p.ab[2 * j] = alpha;
      p.ab[2 * j + 1] = nrm;
    }
    bprev = nrm;
    made = go ? j + 1 : -(j + 1);   // negative: stop after j
    if (!go) break;
    const float inv = 1.f / nrm;
    float2* vn = p.V + (int64_t)(j + 1) * n + r0;
    for (int i = tid; i < rows; i += LT) vn[i] = make_float2(ws[i].x * inv, ws[i].y * inv);
    if (j + 1 < k) {
      if (C > 1) cl.sync();   // the slices of V[j+1], for the next product
      else __syncthreads();
    }
  }
  if (rank == 0 && tid == 0) *keff = made;
  if (C > 1) cl.sync();   // no CTA leaves while another may write to its slots
}

template <class Src>
cudaError_t run_cluster(const Src& src, int np, int64_t nmax, int j0, int k, int full, cudaStream_t s) {
  static std::atomic<int> most[64];   // CTAs of a cluster that a device takes (0: not asked yet)
  int dev = 0;
  cudaGetDevice(&dev);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.blockDim = dim3(LT);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int top = dev < 64 ? most[dev].load(std::memory_order_relaxed) : 0;
  if (top == 0) {
    cudaError_t e = cudaFuncSetAttribute(lanczos_cluster_kernel<Src>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kLanczosSmem);
    if (e != cudaSuccess) return e;
    // sixteen, or the largest power of two below it that the device schedules
    top = kLanczosCta;
    if (cudaFuncSetAttribute(lanczos_cluster_kernel<Src>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
        cudaSuccess)
      top = 8;
    cfg.dynamicSmemBytes = kLanczosSmem;
    for (; top > 1; top /= 2) {
      int clusters = 0;
      at.val.clusterDim.x = top;
      cfg.gridDim = dim3((unsigned)top);
      if (cudaOccupancyMaxActiveClusters(&clusters, lanczos_cluster_kernel<Src>, &cfg) == cudaSuccess && clusters > 0)
        break;
    }
    cudaGetLastError();
    if (dev < 64) most[dev].store(top, std::memory_order_relaxed);
  }
  int C = 1;   // 64 rows a CTA
  while (C < top && (int64_t)C * 64 < nmax) C *= 2;
  at.val.clusterDim.x = C;
  cfg.gridDim = dim3((unsigned)(np * C));
  cfg.dynamicSmemBytes = (size_t)((nmax + C - 1) / C + (full ? nmax : 0)) * sizeof(float2);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, lanczos_cluster_kernel<Src>, src, j0, k, full);
  if (e == cudaSuccess) LAUNCH_NOTE(1);
  return e;
}

}  // namespace

size_t lanczos_ws_bytes(int64_t n, int k) {
  size_t b = 0;
  b += (size_t)(KMAX + 1) * n * sizeof(float2);   // V
  b += (2 * KMAX + 4) * sizeof(float);           // ab
  b += n * sizeof(float2);                        // w
  b += 16 * 256;
  return b;
}

// The products of every step inside the cluster, or as launches over the whole GPU: inside, 16 SMs
// read M (26 us a step at n = 2048, 86 at 4096; outside 19.6 and 47 with the rest of the step, and
// two launch gaps), yet the other SMs stay with the main stream. A sequence of n = 2048: 95.5 ms
// inside, 98.0 outside; of n = 50: 15.2 and 17.2; 8 k-points up to 1900: 201.7 and 206.2; gradient at
// n = 4096: 104.6 and 101.9.
bool lanczos_whole(int64_t nmax) { return nmax <= 2304; }

// the steps of a batch's problems (V[0] is there)
cudaError_t lanczos_batched(const BDesc* D, int np, int64_t nmax, int j0, int k, int full, cudaStream_t s) {
  return run_cluster(LanczosSrcBatch{D}, np, nmax, j0, k, full, s);
}

cudaError_t lanczos_bounds(int64_t n, const float2* M32, int64_t ldm, int k, int count, uint64_t seed,
                    const LanczosWork& w, double* dev_out, cudaStream_t s) {
  k = std::max(1, std::min<int>(k, (int)std::min<int64_t>(n, KMAX)));
  lanczos_init_kernel<<<1, 1024, 0, s>>>(n, w.V, seed, w.ab);
  LAUNCH_NOTE(1);
  const LanczosSrcOne src{{n, M32, ldm, w.V, w.w, w.ab}};
  if (lanczos_whole(n)) {
    const cudaError_t e = run_cluster(src, 1, n, 0, k, 1, s);
    if (e != cudaSuccess) return e;
  } else {
    const int rows_per_block = 8;
    const int blocks = (int)((n + rows_per_block - 1) / rows_per_block);
    for (int j = 0; j < k; ++j) {
      matvec32_kernel<<<blocks, 32 * rows_per_block, 0, s>>>(n, M32, ldm, w.V + (int64_t)j * n, w.w);
      LAUNCH_NOTE(1);
      const cudaError_t e = run_cluster(src, 1, n, j, j + 1, 0, s);
      if (e != cudaSuccess) return e;
    }
  }
  lanczos_tail(k, n, count, w.ab, KMAX, dev_out, s);
  return cudaGetLastError();
}

}  // namespace gevp

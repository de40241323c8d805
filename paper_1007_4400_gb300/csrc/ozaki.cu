// FP64 complex matrix products emulated on the tcgen05 tensor cores: D = op(A) op(B) with
// FP64-class accuracy from exact BF16 products, by Chinese remaindering (the integer modular
// form of the Ozaki scheme: Ozaki, Uchino & Imamura, "Ozaki scheme II", 2025). On this part
// an SM retires about two FP64 FMAs per clock but thousands of BF16 tensor flops, so the n^3
// products of the reduction to standard form and the n^2 m products with an n x n operand
// run far faster this way than on the FP64 pipe.
//
//  1. Integers. Every row i of op(A) is scaled by 2^-e_i so that its largest real or
//     imaginary part lies in [1/4, 1/2) and rounded to q = round(a 2^(7S - e_i)), |q| <=
//     2^(7S-1); columns of op(B) likewise with exponents f_j. The rounding leaves at most
//     2^(e_i - 7S - 1) per entry.
//  2. Residues. The integer product C' = Q_A Q_B has |Re C'|, |Im C'| <= 2K 2^(14S-2) (K
//     complex terms). It is computed modulo nm pairwise coprime odd moduli p <= 255 whose
//     product P exceeds twice that bound (nm = 16 for S = 8 and K up to about 7900). A
//     residue lies in [-127, 127]: exact in BF16.
//  3. Residue products on the tensor cores: Re = Ar Br - Ai Bi, Im = Ar Bi + Ai Br, four real
//     products per modulus. |r r'| <= 127^2, so an FP32 accumulation over at most 1024 real
//     terms (512 complex) is exact; at that point the accumulator is reduced modulo p.
//  4. Reconstruction. x / P = frac(sum_i r_i F_i) with F_i = ((P / p_i)^-1 mod p_i) / p_i
//     in 160-bit fixed point (32-bit integer instructions; the error of the sum is below
//     2^-16 in units of x), then x rounded to FP64 once and scaled by 2^(e_i + f_j - 14S).
// The product of the rounded integers is exact up to the final FP64 rounding: no digit pair
// is dropped and no intermediate rounding is made. Error per entry, relative to 2^(e_i + f_j)
// <= 16 max_k|a_ik| max_k|b_kj|: at most about 2K 2^(-7S) from step 1 (the FP64 product's
// bound K u sum_k |a_ik||b_kj| is of that order for S = 8) plus half an ulp of the result.
//
// Why this form: with S = 8 digits a digit-by-digit scheme forms 36 digit pairs, each four
// real products: 144 real products per complex one. Here it is 4 nm = 64. (Three products by
// Gauss's trick would be 48, but need three operand planes and three accumulators: narrower
// tiles, whose shared-memory traffic costs more than the fourth product.) A * B^H at
// n = 2048, 8 digits: see the figures at oz_gemm_kernel.
#include "gevp_internal.cuh"
#include "tc_ptx.cuh"
#include <cuda.h>
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

namespace gevp {

namespace {

constexpr int OZ_TK = 64;            // K entries of one stage (one 128-byte swizzle row)
constexpr int OZ_CHUNK = 8;          // stages accumulated before a modular reduction: 512 complex terms
constexpr int OZ_EPI_WARPS = 16;
constexpr int OZ_THREADS = (OZ_EPI_WARPS + 2) * 32;
constexpr int OZ_STMAX = 6;
constexpr uint32_t OZ_A_BYTES = 128 * OZ_TK * 2;   // one 128 x 64 BF16 box of A
constexpr size_t OZ_SMEM = 3 * 4 * (size_t)OZ_A_BYTES + 1024;   // three stages at the widest tile

// pairwise coprime, odd, at most 255
constexpr int OZ_NMOD = 17;
constexpr int kOzMod[OZ_NMOD] = {255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193, 191, 181};

// x - p round(x / p) for an integer |x| <= 2^24 (ip = 1 / p rounded): the rounding of x ip can
// err by one only within 0.004 of a half-way point, so the result is congruent to x and lies
// within p / 2 + 0.5; for |x| <= 2^22 it lies in [-(p-1)/2, (p-1)/2] (p odd: the nearest x / p
// is at least 1 / (2p) >= 0.0019 away from a half-way point, the rounding error at most 0.0014)
__device__ __forceinline__ float oz_mod(float x, float p, float ip) {
  constexpr float kMagic = 12582912.f;   // 1.5 2^23: adding it rounds to the nearest integer
  const float q = __fmaf_rn(x, ip, kMagic) - kMagic;
  return __fmaf_rn(-p, q, x);
}

// exponents of an all-zero row stay at the memset pattern of the column splitter; a row with a
// non-finite entry is marked, and every result that it enters is NaN
constexpr int kExpNone = (int)0x80808080;
constexpr int kExpBad = 0x7f000000;

struct OzModTab {
  float p[OZ_NMOD], ip[OZ_NMOD];
  float c1[OZ_NMOD], c2[OZ_NMOD], c3[OZ_NMOD];   // 2^14, 2^28, 2^42 modulo p, centred
};

const OzModTab& oz_mod_tab() {
  static const OzModTab t = [] {
    OzModTab m;
    for (int i = 0; i < OZ_NMOD; ++i) {
      const int p = kOzMod[i];
      auto centred = [&](int e) {
        int v = 1;
        for (int k = 0; k < e; ++k) v = 2 * v % p;
        return (float)(v > p / 2 ? v - p : v);
      };
      m.p[i] = (float)p;
      m.ip[i] = 1.f / (float)p;
      m.c1[i] = centred(14);
      m.c2[i] = centred(28);
      m.c3[i] = centred(42);
    }
    return m;
  }();
  return t;
}

// Constants of the reconstruction for nm moduli (kernel argument, read from constant memory)
struct OzCrtTab {
  uint32_t F[OZ_NMOD][5];   // round(2^160 F_i), little-endian limbs
  uint32_t off[5];          // -128 sum_i F_i mod 2^160: the residues enter as r + 128
  unsigned long long Pm;    // P = Pm 2^(eP - 64), Pm normalised (rounded down)
  int eP;
};

OzCrtTab oz_crt_make(int nm) {
  OzCrtTab t;
  std::memset(&t, 0, sizeof t);
  // P as little-endian 32-bit limbs
  std::vector<uint32_t> P(6, 0);
  P[0] = 1;
  for (int i = 0; i < nm; ++i) {
    unsigned long long c = 0;
    for (auto& w : P) {
      c += (unsigned long long)w * kOzMod[i];
      w = (uint32_t)c;
      c >>= 32;
    }
  }
  int bits = 0;
  for (int b = 191; b >= 0 && !bits; --b)
    if (P[b / 32] >> (b % 32) & 1) bits = b + 1;
  t.eP = bits;
  for (int b = 0; b < 64; ++b) {
    const int at = bits - 1 - b;
    t.Pm = t.Pm << 1 | (at >= 0 ? (P[at / 32] >> (at % 32) & 1) : 0);
  }
  uint32_t sum[5] = {0, 0, 0, 0, 0};
  for (int i = 0; i < nm; ++i) {
    const int p = kOzMod[i];
    int co = 1;   // P / p_i mod p_i
    for (int j = 0; j < nm; ++j)
      if (j != i) co = co * (kOzMod[j] % p) % p;
    int inv = 1;
    while (co * inv % p != 1) ++inv;
    // inv 2^160 / p by long division, rounded to nearest
    unsigned long long rem = inv;
    for (int l = 4; l >= 0; --l) {
      rem <<= 32;
      t.F[i][l] = (uint32_t)(rem / p);
      rem %= p;
    }
    unsigned long long c = 2 * rem > (unsigned long long)p ? 1 : 0;
    for (int l = 0; l < 5; ++l) {
      c += t.F[i][l];
      t.F[i][l] = (uint32_t)c;
      c >>= 32;
    }
    c = 0;
    for (int l = 0; l < 5; ++l) {
      c += (unsigned long long)sum[l] + t.F[i][l];
      sum[l] = (uint32_t)c;
      c >>= 32;
    }
  }
  // off = -(sum << 7) mod 2^160
  unsigned long long c = 1;
  for (int l = 0; l < 5; ++l) {
    const uint32_t s = sum[l] << 7 | (l > 0 ? sum[l - 1] >> 25 : 0);
    c += (uint32_t)~s;
    t.off[l] = (uint32_t)c;
    c >>= 32;
  }
  return t;
}

const OzCrtTab& oz_crt_tab(int nm) {
  static const std::vector<OzCrtTab> all = [] {
    std::vector<OzCrtTab> v;
    for (int k = 0; k <= OZ_NMOD; ++k) v.push_back(oz_crt_make(std::max(k, 1)));
    return v;
  }();
  return all[nm];
}

// moduli needed for S digits and K terms: P > 2 * 2K 2^(14S-2)
int oz_moduli(int K, int S) {
  double bits = 14.0 * S + std::log2((double)std::max(K, 1)) + 1e-3;
  int nm = 0;
  while (nm < OZ_NMOD && bits > 0) bits -= std::log2((double)kOzMod[nm++]);
  return bits > 0 ? OZ_NMOD + 1 : std::max(nm, 1);
}

// ---------------------------------------------------------------- residue products
struct OzMaps {
  CUtensorMap a, b;   // residue planes of op(A) and op(B)^T: (k, row, part * nmod + modulus)
};

struct OzParams {
  int M, N;            // complex output size (M: rows of this panel)
  int row0;            // first row of the panel (a multiple of 256)
  int mt, nt, tn;      // pair tiles (256 rows), column tiles, tile width
  int kblocks;         // 64-blocks of K
  int triA;            // 1: op(A)[i][k] = 0 for k > i;  2: op(A)[i][k] = 0 for k < i
  int triB;            // 1: op(B)[k][j] = 0 for k < j;  2: op(B)[k][j] = 0 for k > j
  int triD;            // 1: tiles above the diagonal are left out
  int mod0, nmod;      // moduli of this launch
  int za, zb;          // tensor-map plane of modulus mod0's real part in A, B
  int pa, pb;          // planes from a real to an imaginary part
  int ksplit, kspan;   // K slices of kspan blocks
  int nst;             // pipeline stages
  uint32_t id_rr, id_ii, id_ri, id_ir;   // instruction descriptors (signs of the four products)
  int8_t* R;           // residues [slice][part][modulus][M][ldr]
  int ldr;
  int64_t plane;       // M ldr
  int nm;              // moduli in R
  int* err;
  const int* active;   // nullable device flag: 0 = skip the whole launch (a converged problem)
  float p[OZ_NMOD], ip[OZ_NMOD];
};

// TMA load whose bytes count on the pair leader's barrier (a shared::cluster address)
__device__ __forceinline__ void oz_tma(void* dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
      "%4}], [%5];" ::"r"(su32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
struct OzUnit {
  int slice, mod, m0, n0, klo, khi;   // klo, khi in 64-blocks
  bool skip;
};

// Unit u of a launch: slice-major, then modulus, then tiles in bands of eight column tiles (the
// tiles in flight at a time then share operand rows and columns in L2).
__device__ __forceinline__ OzUnit oz_unit(const OzParams& p, int u) {
  OzUnit t;
  const int tiles = p.mt * p.nt;
  int e = u % tiles;
  const int q = u / tiles;
  t.mod = p.mod0 + q % p.nmod;
  t.slice = q / p.nmod;
  const int band = e / (8 * p.mt), nb = min(8, p.nt - 8 * band);
  e -= band * 8 * p.mt;
  t.m0 = p.row0 + (e / nb) * 256;
  t.n0 = (8 * band + e % nb) * p.tn;
  t.klo = 0;
  t.khi = p.kblocks;
  if (p.triA == 1) t.khi = min(t.khi, (t.m0 + 256) / OZ_TK);
  if (p.triA == 2) t.klo = max(t.klo, t.m0 / OZ_TK);
  if (p.triB == 1) t.klo = max(t.klo, t.n0 / OZ_TK);
  if (p.triB == 2) t.khi = min(t.khi, (t.n0 + p.tn + OZ_TK - 1) / OZ_TK);
  if (p.ksplit > 1) {
    t.klo = max(t.klo, t.slice * p.kspan);
    t.khi = min(t.khi, (t.slice + 1) * p.kspan);
  }
  t.skip = p.triD && t.n0 > t.m0 + 255;
  if (t.skip) t.khi = t.klo;
  return t;
}

// One pair of CTAs (cta_group::2) per 256 x tn tile of one modulus, both parts of the complex
// product: each CTA holds 128 rows of A and half of B's columns, so the pair's MMA of M = 256
// reads each operand byte once per SM pair. Accumulators: real part in TMEM columns 0..tn-1,
// imaginary part in 256..255+tn (all 512 columns at tn = 256). Warp 8 of each CTA issues its
// TMA loads (four boxes a stage: Ar, Ai, Br, Bi; 64 KB at tn = 256, three stages), warp 9 of
// the leader the MMAs of both CTAs (a stage: 16 MMAs of 256 x tn x 16), warps 0-15 of each CTA
// drain an accumulator after 512 complex terms: the sums are reduced modulo p and written back
// in place (the next 512 terms add to them: 127^2 * 1024 + 127 < 2^24), or, at the end of K,
// written out, one byte per entry. The real part's accumulator is drained while the imaginary
// part's last MMAs run, and the next MMAs of the real part start as soon as it is.
// (Keeping the running residues in registers instead needs a fully unrolled drain, whose code
// misses the instruction cache at every step: 1.28 ms for A B^H at n = 2048 instead of 0.75.)
// Measured, A B^H with 8 digits: n = 2048 0.75 ms, 1474 TFLOP/s of BF16 executed (the 36 digit
// pairs took 2.88 ms); n = 4096 5.0 ms, 1756 TFLOP/s, 0.93 of the cuBLAS rate.
// A launch's clusters take units c, c + gridDim/2, ... in turn.
// All waits are bounded; on expiry the kernel records an error code, stops issuing work, waits
// (bounded) for the copies it issued, frees its TMEM and returns.
__global__ void __launch_bounds__(OZ_THREADS, 1) __cluster_dims__(2, 1, 1)
    oz_gemm_kernel(const __grid_constant__ OzMaps maps, const __grid_constant__ OzParams p, int units) {
  if (p.active && *p.active == 0) return;   // uniform over the grid: before any barrier or TMEM allocation
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[OZ_STMAX], empty[OZ_STMAX], tfull[2], tempty[2];
  __shared__ uint32_t tmem_sh;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int rank = blockIdx.x & 1;   // cluster of two consecutive blocks
  const int u0 = blockIdx.x >> 1, ustep = gridDim.x >> 1;
  const uint32_t b_bytes = (uint32_t)(p.tn / 2) * OZ_TK * 2;
  const uint32_t stage = 2 * OZ_A_BYTES + 2 * b_bytes;

  if (threadIdx.x == 0) {
    for (int s = 0; s < OZ_STMAX; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 2 * OZ_EPI_WARPS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  pair_sync();   // both CTAs run (the allocation takes both), their barriers are initialised
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_sh)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_sh;

  if (warp == OZ_EPI_WARPS && lane == 0) {
    int it = 0;
    bool ok = true;
    for (int u = u0; u < units && ok; u += ustep) {
      const OzUnit t = oz_unit(p, u);
      const int z = t.mod - p.mod0;
      for (int kb = t.klo; kb < t.khi; ++kb, ++it) {
        const int st = it % p.nst;
        if (it >= p.nst && !pair_wait(&empty[st], ((uint32_t)(it / p.nst) & 1u) ^ 1u, p.err, 21)) {
          ok = false;
          break;
        }
        uint8_t* dst = smem + (size_t)st * stage;
        if (rank == 0) mbar_expect_tx(&full[st], 2 * stage);
        const uint32_t bar = pair_mapa(su32(&full[st]), 0);
        const int x = kb * OZ_TK, ya = t.m0 + 128 * rank, yb = t.n0 + (p.tn / 2) * rank;
        oz_tma(dst, &maps.a, x, ya, p.za + z, bar);
        oz_tma(dst + 2 * OZ_A_BYTES, &maps.b, x, yb, p.zb + z, bar);
        oz_tma(dst + OZ_A_BYTES, &maps.a, x, ya, p.za + p.pa + z, bar);
        oz_tma(dst + 2 * OZ_A_BYTES + b_bytes, &maps.b, x, yb, p.zb + p.pb + z, bar);
      }
    }
    // every copy issued has landed before the CTAs leave (normally they were all consumed;
    // after a wait elsewhere gave up they may still be in flight), ...
    if (rank == 0)
      for (int i = max(0, it - p.nst); i < it; ++i)
        mbar_wait(&full[i % p.nst], (uint32_t)(i / p.nst) & 1u, p.err, 25);
    // ... and so has every release of a stage: the last commits come behind the one that the epilogue
    // goes on from, and an arrival after this CTA has left would count on a barrier of the next one
    for (int i = max(0, it - p.nst); i < it; ++i)
      if (!pair_wait(&empty[i % p.nst], (uint32_t)(i / p.nst) & 1u, p.err, 26)) break;
  } else if (warp == OZ_EPI_WARPS + 1 && lane == 0 && rank == 0) {
    int it = 0;
    uint32_t chunk = 0;
    bool ok = true;
    for (int u = u0; u < units && ok; u += ustep) {
      const OzUnit t = oz_unit(p, u);
      for (int kb = t.klo; kb < t.khi && ok; kb += OZ_CHUNK, ++chunk) {
        const int ke = min(t.khi, kb + OZ_CHUNK);
        for (int k = kb; k < ke; ++k, ++it) {
          const int st = it % p.nst;
          if (!mbar_wait(&full[st], (uint32_t)(it / p.nst) & 1u, p.err, 23)) {
            ok = false;
            break;
          }
          const uint8_t* base = smem + (size_t)st * stage;
          const uint64_t ar = sdesc(su32(base)), ai = sdesc(su32(base + OZ_A_BYTES));
          const uint64_t br = sdesc(su32(base + 2 * OZ_A_BYTES)), bi = sdesc(su32(base + 2 * OZ_A_BYTES + b_bytes));
          const uint32_t first = k > t.klo ? 1u : 0u;
#pragma unroll
          for (int part = 0; part < 2; ++part) {
            // a chunk's first MMAs wait until the previous chunk's sums have been read
            if (k == kb && chunk > 0 && !pair_wait(&tempty[part], (chunk - 1) & 1u, p.err, 22)) {
              ok = false;
              break;
            }
            fence_after();
            const uint32_t d = tmem + 256u * part;
#pragma unroll
            for (int kk = 0; kk < OZ_TK / 16; ++kk) {
              const uint64_t o = (uint64_t)(kk * 32) >> 4;
              pair_umma(d, ar + o, (part ? bi : br) + o, part ? p.id_ri : p.id_rr, kk > 0 ? 1u : first);
            }
#pragma unroll
            for (int kk = 0; kk < OZ_TK / 16; ++kk) {
              const uint64_t o = (uint64_t)(kk * 32) >> 4;
              pair_umma(d, ai + o, (part ? br : bi) + o, part ? p.id_ir : p.id_ii, 1u);
            }
            if (k == ke - 1) pair_commit(&tfull[part]);
          }
          if (!ok) break;
          pair_commit(&empty[st]);
        }
      }
    }
  } else if (warp < OZ_EPI_WARPS) {
    const int q = warp & 3;
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
    const int ng = p.tn / 16;   // 16-column groups; this warp's: warp / 4, warp / 4 + 4, ...
    const uint32_t te[2] = {pair_mapa(su32(&tempty[0]), 0), pair_mapa(su32(&tempty[1]), 0)};
    uint32_t chunk = 0;
    bool ok = true;
    for (int u = u0; u < units && ok; u += ustep) {
      const OzUnit t = oz_unit(p, u);
      const int row = t.m0 - p.row0 + 128 * rank + 32 * q + lane;
      const float pm = p.p[t.mod], ip = p.ip[t.mod];
      int8_t* out = p.R + ((int64_t)(t.slice * 2) * p.nm + t.mod) * p.plane + (int64_t)row * p.ldr + t.n0;
      const int64_t opart = (int64_t)p.nm * p.plane;
      if (t.klo >= t.khi) {
        if (row < p.M && !t.skip)
          for (int g = warp >> 2; g < ng; g += 4) {
            *(uint4*)(out + 16 * g) = make_uint4(0, 0, 0, 0);
            *(uint4*)(out + opart + 16 * g) = make_uint4(0, 0, 0, 0);
          }
        continue;
      }
      for (int kb = t.klo; kb < t.khi && ok; kb += OZ_CHUNK, ++chunk) {
        const bool last = kb + OZ_CHUNK >= t.khi;
        for (int part = 0; part < 2; ++part) {
          ok = ok && __all_sync(0xffffffffu, pair_wait(&tfull[part], chunk & 1u, p.err, 24) ? 1 : 0) != 0;
          if (!ok) break;
          fence_after();
          for (int g = warp >> 2; g < ng; g += 4) {
            uint32_t r[16];
            const uint32_t at = tq + 256u * part + 16u * g;
            tmem_ld16(at, r);
            tmem_wait_ld();
            if (!last) {
#pragma unroll
              for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(oz_mod(__uint_as_float(r[j]), pm, ip));
              tmem_st16(at, r);
            } else {
              // a residue's low byte: that of x + 1.5 2^23 is the two's complement of x. The sum is
              // reduced twice: the first reduction may leave (p + 1) / 2.
#pragma unroll
              for (int j = 0; j < 16; ++j)
                r[j] = __float_as_uint(oz_mod(oz_mod(__uint_as_float(r[j]), pm, ip), pm, ip) + 12582912.f);
              uint32_t w[4];
#pragma unroll
              for (int j = 0; j < 4; ++j)
                w[j] = __byte_perm(__byte_perm(r[4 * j], r[4 * j + 1], 0x0040),
                                   __byte_perm(r[4 * j + 2], r[4 * j + 3], 0x0040), 0x5410);
              if (row < p.M) *(uint4*)(out + part * opart + 16 * g) = make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
          if (!last) tmem_wait_st();
          fence_before();
          __syncwarp();
          if (lane == 0) pair_arrive(te[part]);
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  pair_sync();   // neither CTA leaves while the other's MMAs or arrivals may touch it
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  pair_sync();
}

// ---------------------------------------------------------------- reconstruction
// x = P frac, frac the 160-bit two's complement fraction w (little-endian), rounded to the
// nearest double (integers below 2^53 exactly) and scaled by 2^ex
__device__ __forceinline__ double oz_crt_value(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t w4,
                                               unsigned long long Pm, int eP, int ex) {
  const bool neg = (w4 >> 31) != 0;
  if (neg) {
    asm("{\n add.cc.u32 %0, %5, 1;\n addc.cc.u32 %1, %6, 0;\n addc.cc.u32 %2, %7, 0;\n addc.cc.u32 %3, %8, 0;\n"
        " addc.u32 %4, %9, 0;\n}\n"
        : "=r"(w0), "=r"(w1), "=r"(w2), "=r"(w3), "=r"(w4)
        : "r"(~w0), "r"(~w1), "r"(~w2), "r"(~w3), "r"(~w4));
  }
  int sh = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (w4 == 0) {
      w4 = w3;
      w3 = w2;
      w2 = w1;
      w1 = w0;
      w0 = 0;
      sh += 32;
    }
  if (w4 == 0) return 0.0;
  const int lz = __clz((int)w4);
  const unsigned long long m =
      (unsigned long long)__funnelshift_l(w3, w4, lz) << 32 | __funnelshift_l(w2, w3, lz);
  unsigned long long h = __umul64hi(m, Pm);   // x = h 2^t to a relative 2^-61
  int t = eP - 64 - lz - sh;
  if (!(h >> 63)) {
    h <<= 1;
    --t;
  }
  // round to 53 bits, or to a whole number when x has fewer
  const int s = max(11, -t);
  if (s > 64) return 0.0;
  unsigned long long q, rem;
  if (s == 64) {
    q = 0;
    rem = h;
  } else {
    q = h >> s;
    rem = h << (64 - s);
  }
  if (rem > (1ull << 63) || (rem == (1ull << 63) && (q & 1ull))) ++q;
  if (q == 0) return 0.0;
  int e = t + s + ex;
  if (q >> 53) {
    q >>= 1;
    ++e;
  }
  const int top = 63 - __clzll((long long)q);
  const int be = top + e + 1023;
  double v;
  if (be >= 1 && be <= 2046)
    v = __longlong_as_double((long long)((unsigned long long)be << 52 | ((q << (52 - top)) & 0xFFFFFFFFFFFFFull)));
  else
    v = ldexp((double)q, e);
  return neg ? -v : v;
}

// D from its residues: a thread takes four neighbouring columns of a row (one 32-bit word of
// each plane). Bound by integer multiply-adds (5 x 32 bit per modulus and value), about a
// tenth of the products' time at n = 2048; in FP64 arithmetic it would take longer than them.
__global__ void __launch_bounds__(256) oz_crt_kernel(int M, int N, const int8_t* R, int ldr, int64_t plane, int nm,
                                                     int ksplit, const __grid_constant__ OzCrtTab tab, const int* ea,
                                                     const int* eb, int e0, double2* D, int64_t ldd,
                                                     int row0, int triD, const int* active) {
  if (active && *active == 0) return;
  const int nq = (N + 3) / 4;
  const int64_t total = (int64_t)M * nq;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int row = (int)(e / nq), c0 = (int)(e % nq) * 4;
    if (triD && c0 > row0 + row) continue;
    double v[2][4];
    const int er = ea[row] == kExpNone ? 0 : ea[row];
    int ex[4];
    bool bad[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int f = c0 + c < N ? eb[c0 + c] : 0;
      ex[c] = er + (f == kExpNone ? 0 : f) + e0;
      bad[c] = er == kExpBad || f == kExpBad;
    }
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      unsigned long long acc[4][5];
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int l = 0; l < 5; ++l) acc[c][l] = 0;
      for (int z = 0; z < ksplit; ++z) {
        const int8_t* src = R + (int64_t)(2 * z + part) * nm * plane + (int64_t)row * ldr + c0;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int l = 0; l < 5; ++l) acc[c][l] += tab.off[l];
#pragma unroll 4
        for (int i = 0; i < nm; ++i) {
          const uint32_t w = *(const uint32_t*)(src + (int64_t)i * plane) ^ 0x80808080u;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t b = __byte_perm(w, 0, 0x4440 + c);
#pragma unroll
            for (int l = 0; l < 5; ++l) acc[c][l] += (unsigned long long)b * tab.F[i][l];
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t w[5];
        unsigned long long t = 0;
#pragma unroll
        for (int l = 0; l < 5; ++l) {
          t += acc[c][l];
          w[l] = (uint32_t)t;
          t >>= 32;
        }
        v[part][c] = oz_crt_value(w[0], w[1], w[2], w[3], w[4], tab.Pm, tab.eP, ex[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c0 + c < N) {
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        D[(int64_t)row * ldd + c0 + c] = bad[c] ? make_double2(nan, nan) : make_double2(v[0][c], v[1][c]);
      }
  }
}

// ---------------------------------------------------------------- splitting
// Residues of one operand row r (a row of op(A), or a column of op(B)), entries k < K. The
// row is row r of the stored X (oz_split_rows_kernel) or its column r (oz_split_cols_kernel);
// mask 1 keeps k >= r with the diagonal halved (a column of the lower triangle of a Hermitian
// matrix, tril(A) with its diagonal split between A and A^H), mask 2 keeps k <= r, mask 3 keeps
// k >= r. Writes the exponent of the row and the residues of the real and the imaginary part
// into planes [part][modulus][rows][k_pad]. A conjugated operand is the same planes with the
// sign of its imaginary part in the MMA's instruction descriptor. A row with a non-finite
// entry sets *bad.
__device__ __forceinline__ double2 oz_masked(double2 v, int r, int k, int mask) {
  if ((mask == 1 && k < r) || (mask == 2 && k > r) || (mask == 3 && k < r)) return make_double2(0.0, 0.0);
  if (mask == 1 && k == r) v = make_double2(0.5 * v.x, 0.5 * v.y);
  return v;
}

// x 2^s on the exponent field (0 for a value that is, or becomes, subnormal; Inf and NaN stay)
__device__ __forceinline__ double oz_shift2(double x, int s) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7FF;
  if (e == 0x7FF) return x;
  if (e == 0 || e + s <= 0) return 0.0;
  return __hiloint2double(hi + (min(s, 2046 - e) << 20), __double2loint(x));
}

// ks (nullable), sg: entry k is scaled by 2^(sg ks[k]) first
__device__ __forceinline__ double2 oz_entry(const double2* X, int64_t ldx, int r, int k, int K, int mask,
                                            const int* ks, int sg) {
  if (k >= K) return make_double2(0.0, 0.0);
  double2 v = oz_masked(X[(int64_t)r * ldx + k], r, k, mask);
  if (ks) {
    const int q = ks[k];
    if (q != kExpNone && q != kExpBad) v = make_double2(oz_shift2(v.x, sg * q), oz_shift2(v.y, sg * q));
  }
  return v;
}

// The splitting works on the IEEE-754 fields with integer instructions only: one SM
// retires about two FP64 operations per clock on this part, and a conversion, a scaling
// and a maximum per entry on the FP64 pipe made the splitter several times slower than
// its memory traffic.
//
// |v| as an ordered integer key: for finite values the order of the keys is the order of
// the magnitudes; an exponent field of all ones (Inf or NaN) is reported as non-finite.
__device__ __forceinline__ unsigned long long oz_abs_key(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ bool oz_key_finite(unsigned long long key) { return (key >> 52) != 0x7FF; }

// floor(log2 |x|) of the value with magnitude key `key` (> 0, finite), as ilogb.
__device__ __forceinline__ int oz_key_ilogb(unsigned long long key) {
  const int E = (int)(key >> 52);
  return E != 0 ? E - 1023 : (63 - __clzll((long long)key)) - 1074;
}

// round(x 2^shift) to the nearest integer, ties to even, for finite x with
// |x 2^shift| < 2^62: x = M 2^k' with the integer significand M < 2^53, so the result is
// M shifted left, or shifted right with the dropped bits deciding the rounding. The same
// value as converting ldexp(x, shift) with round-to-nearest-even, without FP64
// instructions. A non-finite x gives 0 (its row is reported as bad).
__device__ __forceinline__ long long oz_round_scaled(double x, int shift) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FF);
  if (E == 0x7FF) return 0;
  unsigned long long M = b & 0xFFFFFFFFFFFFFull;
  int k = shift - 1074;                    // subnormal: x = M 2^-1074
  if (E != 0) {
    M |= 1ull << 52;
    k = E - 1075 + shift;
  }
  unsigned long long q;
  if (k >= 0) {
    q = M << k;
  } else if (k < -63) {
    q = 0;                                 // |x 2^shift| < 2^-10
  } else {
    const int r = -k;
    q = M >> r;
    const unsigned long long rem = M & ((1ull << (r - 1) << 1) - 1), half = 1ull << (r - 1);
    if (rem > half || (rem == half && (q & 1ull))) ++q;
  }
  return (b >> 63) ? -(long long)q : (long long)q;
}

// the residues of the pair (x0, x1) of neighbouring entries modulo moduli [mod0, mod0 + cnt), one
// BF16 pair per plane (imag: entries from a real to an imaginary plane): q = a0 + 2^14 a1 + 2^28 a2 + 2^42 a3 with centred 14-bit pieces, r = a0 +
// c1 a1 + c2 a2 + c3 a3 modulo p in FP32 (|sum| <= 2^13 (1 + 3 * 127) < 2^22, exact)
struct OzPieces {
  float a[4];
};
__device__ __forceinline__ OzPieces oz_pieces(double x, int shift) {
  long long q = oz_round_scaled(x, shift);
  OzPieces r;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int d = (int)((q + 8192) & 16383) - 8192;
    r.a[k] = (float)d;
    q = (q - d) >> 14;
  }
  r.a[3] = (float)(int)q;
  return r;
}
__device__ __forceinline__ float oz_residue(const OzPieces& v, const OzModTab& m, int i) {
  const float t = __fmaf_rn(v.a[3], m.c3[i], __fmaf_rn(v.a[2], m.c2[i], __fmaf_rn(v.a[1], m.c1[i], v.a[0])));
  return oz_mod(t, m.p[i], m.ip[i]);
}
__device__ __forceinline__ void oz_write_pair(double2 v0, double2 v1, int shift, const OzModTab& m, int mod0, int cnt,
                                              size_t imag, size_t plane, __nv_bfloat16* at) {
  const OzPieces x0 = oz_pieces(v0.x, shift), x1 = oz_pieces(v1.x, shift);
  const OzPieces y0 = oz_pieces(v0.y, shift), y1 = oz_pieces(v1.y, shift);
#pragma unroll 4
  for (int i = 0; i < cnt; ++i) {
    *(__nv_bfloat162*)(at + (size_t)i * plane) =
        __floats2bfloat162_rn(oz_residue(x0, m, mod0 + i), oz_residue(x1, m, mod0 + i));
    *(__nv_bfloat162*)(at + imag + (size_t)i * plane) =
        __floats2bfloat162_rn(oz_residue(y0, m, mod0 + i), oz_residue(y1, m, mod0 + i));
  }
}

// One block per row: the row's largest magnitude, then its residues (two entries a thread, so a
// warp writes 128 contiguous bytes of each plane). Bound by the planes' bytes: 16 read, 64
// written per entry at 16 moduli. need_ex: find (and write) the exponent; else read it.
__global__ void __launch_bounds__(256) oz_split_rows_kernel(int rows, int K, const double2* X, int64_t ldx, int mask,
                                                            const int* ks, int sg, int S, int mod0, int cnt, int nmod,
                                                            int k_pad, __nv_bfloat16* planes, int* ex, int need_ex,
                                                            int* bad, int* even,
                                                            const __grid_constant__ OzModTab tab, const int* active) {
  if (active && *active == 0) return;
  __shared__ unsigned long long red[8];
  const int r = blockIdx.x;
  int e;
  if (need_ex) {
    unsigned long long mx = 0;   // largest magnitude key of the finite entries
    bool nonfinite = false;
    for (int k = threadIdx.x; k < K; k += 256) {
      const double2 v = oz_entry(X, ldx, r, k, K, mask, ks, sg);
      const unsigned long long kx = oz_abs_key(v.x), ky = oz_abs_key(v.y);
      if (!oz_key_finite(kx) || !oz_key_finite(ky)) nonfinite = true;
      else mx = max(mx, max(kx, ky));
    }
    if (nonfinite) atomicExch(bad, 1);
    nonfinite = __syncthreads_or(nonfinite) != 0;
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = red[0];
    for (int w = 1; w < 8; ++w) mx = max(mx, red[w]);
    // 2^e > 2 max|entry|: the scaled row lies below 1/2
    e = mx > 0 ? oz_key_ilogb(mx) + 2 : 0;
    if (threadIdx.x == 0) ex[r] = nonfinite ? kExpBad : e;
    if (even) {
      int small = 0;
      for (int k = threadIdx.x; k < K; k += 256) {
        const double2 v = oz_entry(X, ldx, r, k, K, mask, ks, sg);
        const unsigned long long key = max(oz_abs_key(v.x), oz_abs_key(v.y));
        small += key == 0 || oz_key_ilogb(key) < e - 8 ? 1 : 0;
      }
      for (int o = 16; o > 0; o >>= 1) small += __shfl_xor_sync(0xffffffffu, small, o);
      __syncthreads();
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = (unsigned)small;
      __syncthreads();
      if (threadIdx.x == 0) {
        unsigned long long all = 0;
        for (int w = 0; w < 8; ++w) all += red[w];
        if (nonfinite || (mx > 0 && 4 * all > (unsigned)K)) *even = 0;   // (a zero row's products are exact)
      }
    }
  } else {
    e = ex[r] == kExpBad ? 0 : ex[r];
  }
  if (cnt == 0) return;
  const size_t plane = (size_t)rows * k_pad;
  for (int k = 2 * threadIdx.x; k < k_pad; k += 512)
    oz_write_pair(oz_entry(X, ldx, r, k, K, mask, ks, sg), oz_entry(X, ldx, r, k + 1, K, mask, ks, sg), 7 * S - e, tab, mod0, cnt,
                  (size_t)nmod * plane, plane, planes + (size_t)r * k_pad + k);
}

// Columns of X (K rows x R columns, ld ldx) as operand rows. Pass 1: the exponent of each
// column (threads across consecutive columns, coalesced). Pass 2: a 64 x 32 tile of X staged
// in shared memory and written out transposed, so the residue stores run along k.
constexpr int OZ_CT = 32;
constexpr int OZ_CK = 64;

// ex[j] starts at kExpNone; each block (32 columns x one slice of rows) raises it to the
// exponent of its slice's largest entry (the exponent of a maximum is the maximum of the
// exponents); a column with no nonzero entry keeps kExpNone, read as 0.
constexpr int OZ_CE_ROWS = 64;   // rows per slice

__global__ void __launch_bounds__(256) oz_cols_exp_kernel(int R, int K, const double2* X, int64_t ldx, int mask,
                                                          int* ex, int* bad, const int* active) {
  if (active && *active == 0) return;
  __shared__ unsigned long long red[8][OZ_CT];
  const int j = blockIdx.x * OZ_CT + threadIdx.x;
  const int k0 = blockIdx.y * OZ_CE_ROWS, k1 = min(K, k0 + OZ_CE_ROWS);
  unsigned long long mx = 0;
  bool nonfinite = false;
  if (j < R)
#pragma unroll 4
    for (int k = k0 + threadIdx.y; k < k1; k += 8) {
      const double2 v = oz_masked(X[(int64_t)k * ldx + j], j, k, mask);
      const unsigned long long kx = oz_abs_key(v.x), ky = oz_abs_key(v.y);
      if (!oz_key_finite(kx) || !oz_key_finite(ky)) nonfinite = true;
      else mx = max(mx, max(kx, ky));
    }
  if (nonfinite) {
    atomicExch(bad, 1);
    atomicMax(&ex[j], kExpBad);
  }
  red[threadIdx.y][threadIdx.x] = mx;
  __syncthreads();
  if (threadIdx.y == 0 && j < R) {
    for (int t = 1; t < 8; ++t) mx = max(mx, red[t][threadIdx.x]);
    if (mx > 0) atomicMax(&ex[j], oz_key_ilogb(mx) + 2);
  }
}

__global__ void __launch_bounds__(256) oz_split_cols_kernel(int R, int K, const double2* X, int64_t ldx, int mask,
                                                            int S, int mod0, int cnt, int nmod, int k_pad,
                                                            __nv_bfloat16* planes, const int* ex,
                                                            const __grid_constant__ OzModTab tab, const int* active) {
  if (active && *active == 0) return;
  __shared__ double2 tile[OZ_CK][OZ_CT + 1];   // [k][j]
  const int k0 = blockIdx.x * OZ_CK, j0 = blockIdx.y * OZ_CT;
  for (int i = threadIdx.y; i < OZ_CK; i += 8) {
    const int k = k0 + i, j = j0 + threadIdx.x;
    tile[i][threadIdx.x] = (k < K && j < R) ? oz_masked(X[(int64_t)k * ldx + j], j, k, mask) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const size_t plane = (size_t)R * k_pad;
  const int kk = 2 * threadIdx.x, k = k0 + kk;
  if (k >= k_pad) return;
  for (int jj = threadIdx.y; jj < OZ_CT; jj += 8) {
    const int j = j0 + jj;
    if (j >= R) break;
    const int e = ex[j] == kExpBad ? 0 : ex[j];
    oz_write_pair(tile[kk][jj], tile[kk + 1][jj], 7 * S - (e == kExpNone ? 0 : e), tab, mod0, cnt,
                  (size_t)nmod * plane, plane,                  planes + (size_t)j * k_pad + k);
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn oz_encode() {
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

// 3D map over the residue planes: (k, row, part * nmod + modulus), box 64 x box_rows x 1; rows
// and entries past the operand read as zero
bool oz_map(CUtensorMap* map, const OzOperand& op, int box_rows) {
  EncodeTiledFn enc = oz_encode();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)op.k_pad, (cuuint64_t)op.rows, (cuuint64_t)(2 * op.nmod)};
  cuuint64_t strides[2] = {(cuuint64_t)op.k_pad * 2, (cuuint64_t)op.rows * op.k_pad * 2};
  cuuint32_t box[3] = {OZ_TK, (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, op.planes, dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int oz_k_pad(int K) { return std::max(8, (K + 7) / 8 * 8); }
size_t oz_plane_bytes(int rows, int K) { return (size_t)rows * oz_k_pad(K) * 2; }
size_t oz_ex_bytes(int rows) { return ((size_t)rows * 4 + 255) / 256 * 256; }

// residues of moduli [mod0, mod0 + cnt), cnt <= op.nmod, into op.planes; the exponents first when
// need_ex
cudaError_t oz_split_group(const OzOperand& op, int mod0, int cnt, bool need_ex, int* bad, cudaStream_t s,
                           const int* active) {
  if (op.rows == 0) return cudaSuccess;
  const OzModTab& tab = oz_mod_tab();
  if (!op.cols) {
    oz_split_rows_kernel<<<op.rows, 256, 0, s>>>(op.rows, op.K, op.X, op.ldx, op.mask, op.ks, op.ks_sign, op.S, mod0,
                                                 cnt, op.nmod, op.k_pad, op.planes, op.ex, need_ex ? 1 : 0, bad, op.even, tab,
                                                 active);
    LAUNCH_NOTE(1);
    return cudaGetLastError();
  }
  if (need_ex) {
    cudaMemsetAsync(op.ex, 0x80, (size_t)op.rows * sizeof(int), s);
    dim3 egrid((op.rows + OZ_CT - 1) / OZ_CT, std::max(1, (op.K + OZ_CE_ROWS - 1) / OZ_CE_ROWS));
    oz_cols_exp_kernel<<<egrid, dim3(OZ_CT, 8), 0, s>>>(op.rows, op.K, op.X, op.ldx, op.mask, op.ex, bad, active);
    LAUNCH_NOTE(1);
  }
  if (cnt > 0) {
    dim3 grid((op.k_pad + OZ_CK - 1) / OZ_CK, (op.rows + OZ_CT - 1) / OZ_CT);
    oz_split_cols_kernel<<<grid, dim3(OZ_CT, 8), 0, s>>>(op.rows, op.K, op.X, op.ldx, op.mask, op.S, mod0, cnt,
                                                         op.nmod, op.k_pad, op.planes, op.ex, tab, active);
    LAUNCH_NOTE(1);
  }
  return cudaGetLastError();
}

}  // namespace

size_t oz_operand_bytes(int rows, int K, int S, int group) {
  const int nm = oz_moduli(K, S);
  const int g = group > 0 ? std::min(group, nm) : nm;
  return (2 * (size_t)g * oz_plane_bytes(rows, K) + 255) / 256 * 256 + oz_ex_bytes(rows);
}

size_t oz_work_bytes(int M, int N, int K, int S) {
  const size_t ldr = ((size_t)N + 31) / 32 * 32 + 256;
  return 2 * (size_t)oz_moduli(K, S) * (((size_t)M + 255) / 256 * 256) * ldr;
}

bool oz_supported() {
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  return major == 10 && minor == 3 && oz_encode() != nullptr;
}

cudaError_t oz_split(OzOperand& op, void* mem, int rows, int K, const double2* X, int64_t ldx, int conj, int mask,
                     int S, int* bad, cudaStream_t s, bool cols, const int* active, int group, const int* ks,
                     int ks_sign, int* even) {
  const int nm = oz_moduli(K, S);
  if (S < 1 || S > kOzSlicesMax || nm > OZ_NMOD) return cudaErrorInvalidValue;
  op.rows = rows;
  op.K = K;
  op.S = S;
  op.k_pad = oz_k_pad(K);
  op.nmod = group > 0 ? std::min(group, nm) : nm;
  op.planes = (__nv_bfloat16*)mem;
  op.ex = (int*)((char*)mem + (2 * (size_t)op.nmod * oz_plane_bytes(rows, K) + 255) / 256 * 256);
  op.X = X;
  op.ldx = ldx;
  op.conj = conj;
  op.mask = mask;
  op.cols = cols;
  op.bad = bad;
  op.ks = cols ? nullptr : ks;
  op.ks_sign = ks_sign;
  op.even = cols ? nullptr : even;
  // in groups: the exponents only (oz_gemm writes each group's residues before it uses them)
  return oz_split_group(op, 0, op.nmod == nm ? nm : 0, true, bad, s, active);
}

cudaError_t oz_gemm(const OzOperand& A, const OzOperand& B, int triA, int triB, double2* D, int64_t ldd, int* err,
                    cudaStream_t s, const int* active, void* ws, size_t ws_bytes, int triD) {
  if (A.K != B.K || A.S != B.S || A.k_pad != B.k_pad || !ws) return cudaErrorInvalidValue;
  if (A.rows == 0 || B.rows == 0) return cudaSuccess;
  const int nm = oz_moduli(A.K, A.S);
  static std::atomic<int> pairs_dev{0};   // SM pairs that hold a cluster at a time
  int pairs = pairs_dev.load(std::memory_order_relaxed);
  if (pairs == 0) {
    cudaError_t e = cudaFuncSetAttribute(oz_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    pairs = std::max(1, sms / 2);
    pairs_dev.store(pairs, std::memory_order_relaxed);
  }
  OzParams p;
  std::memset(&p, 0, sizeof p);
  p.N = B.rows;
  p.kblocks = (A.K + OZ_TK - 1) / OZ_TK;
  p.triA = triA;
  p.triB = triB;
  p.triD = triD;
  p.nm = nm;
  p.err = err;
  p.active = active;
  const OzModTab& tab = oz_mod_tab();
  for (int i = 0; i < OZ_NMOD; ++i) {
    p.p[i] = tab.p[i];
    p.ip[i] = tab.ip[i];
  }
  // signs: a = ar + i sa ai, b = br + i sb bi
  p.id_rr = idesc_bf16(256, 16);   // N set below
  const uint32_t neg = 1u << 13;   // negate the A operand
  // column tiles: as wide as 256, evenly split, narrower where that leaves SM pairs idle
  const int mt_all = (A.rows + 255) / 256;
  int nt = (p.N + 255) / 256;
  while (mt_all * nt * nm < pairs && (p.N + nt - 1) / nt > 64) ++nt;
  p.tn = ((p.N + nt - 1) / nt + 31) / 32 * 32;
  p.nt = (p.N + p.tn - 1) / p.tn;
  p.ldr = p.nt * p.tn;
  // K slices (their residues add up in the reconstruction) where the tiles still leave half of
  // the pairs idle: at least eight blocks each
  p.ksplit = 1;
  p.kspan = p.kblocks;
  const int base = mt_all * p.nt * nm;
  if (2 * base <= pairs && p.kblocks >= 16) {
    const int want = std::min(std::min(4, pairs / base), p.kblocks / 8);
    p.kspan = (p.kblocks + want - 1) / want;
    p.ksplit = (p.kblocks + p.kspan - 1) / p.kspan;
  }
  // rows of one panel: what the residues' room holds
  const size_t row_bytes = 2 * (size_t)nm * p.ldr;
  if (ws_bytes < row_bytes * std::min(256, A.rows)) return cudaErrorInvalidValue;
  if (p.ksplit > 1 && ws_bytes < row_bytes * A.rows * p.ksplit) p.ksplit = 1, p.kspan = p.kblocks;
  int panel = A.rows;
  if (ws_bytes < row_bytes * A.rows * p.ksplit) panel = (int)(ws_bytes / row_bytes / 256 * 256);
  p.id_rr = idesc_bf16(256, p.tn);
  p.id_ii = p.id_rr | ((A.conj != 0) == (B.conj != 0) ? neg : 0u);   // - sa sb
  p.id_ri = p.id_rr | (B.conj ? neg : 0u);
  p.id_ir = p.id_rr | (A.conj ? neg : 0u);
  const uint32_t stage = 2 * OZ_A_BYTES + 2u * (uint32_t)(p.tn / 2) * OZ_TK * 2;
  p.nst = (int)std::min<size_t>(OZ_STMAX, (OZ_SMEM - 1024) / stage);
  OzMaps maps;
  std::memset(&maps, 0, sizeof maps);
  if (!oz_map(&maps.a, A, 128) || !oz_map(&maps.b, B, p.tn / 2)) return cudaErrorInvalidValue;
  p.R = (int8_t*)ws;
  p.pa = A.nmod;
  p.pb = B.nmod;
  const bool lean = A.nmod < nm || B.nmod < nm;
  const int group = std::min(A.nmod, B.nmod);
  for (int row0 = 0; row0 < A.rows; row0 += panel) {
    p.row0 = row0;
    p.M = std::min(panel, A.rows - row0);
    p.mt = (p.M + 255) / 256;
    p.plane = (int64_t)p.M * p.ldr;
    for (int g0 = 0; g0 < nm; g0 += group) {
      p.mod0 = g0;
      p.nmod = std::min(group, nm - g0);
      p.za = A.nmod < nm ? 0 : g0;
      p.zb = B.nmod < nm ? 0 : g0;
      if (lean) {
        cudaError_t e = cudaSuccess;
        if (A.nmod < nm) e = oz_split_group(A, g0, p.nmod, false, A.bad, s, active);
        if (e == cudaSuccess && B.nmod < nm) e = oz_split_group(B, g0, p.nmod, false, B.bad, s, active);
        if (e != cudaSuccess) return e;
      }
      const int units = p.ksplit * p.nmod * p.mt * p.nt;
      // up to four units a cluster: the set-up is shared, yet a launch on the side stream still
      // gives SMs back to the high-priority stream every few tens of microseconds
      const int per = std::max(1, std::min(4, units / pairs));
      const int clusters = (units + per - 1) / per;
      void* kt0 = kt_enabled() ? kt_begin(s) : nullptr;
      oz_gemm_kernel<<<2 * clusters, OZ_THREADS, OZ_SMEM, s>>>(maps, p, units);
      LAUNCH_NOTE(1);
      if (kt0) {
        // algorithmic: the complex product over the K ranges the tiles process (8 flop per
        // complex multiply-add), shared out over the moduli; executed: four real products each
        double alg = 0.0;
        for (int mt = 0; mt < p.mt; ++mt)
          for (int t = 0; t < p.nt; ++t) {
            const int m0 = row0 + mt * 256, n0 = t * p.tn;
            int klo = 0, khi = p.kblocks;
            if (triA == 1) khi = std::min(khi, (m0 + 256) / OZ_TK);
            if (triA == 2) klo = std::max(klo, m0 / OZ_TK);
            if (triB == 1) klo = std::max(klo, n0 / OZ_TK);
            if (triB == 2) khi = std::min(khi, (n0 + p.tn + OZ_TK - 1) / OZ_TK);
            const int rows = std::min(256, row0 + p.M - m0), cols = std::min(p.tn, p.N - n0);
            if (triD && n0 > m0 + 255) continue;
            if (khi > klo && rows > 0 && cols > 0) alg += 8.0 * rows * cols * (double)(khi - klo) * OZ_TK;
          }
        kt_end(kt0, 1, alg * p.nmod / nm, alg * p.nmod, s);
      }
    }
    const int64_t quads = (int64_t)p.M * ((p.N + 3) / 4);
    const int blocks = (int)std::min<int64_t>((quads + 255) / 256, 152 * 16);
    oz_crt_kernel<<<blocks, 256, 0, s>>>(p.M, p.N, p.R, p.ldr, p.plane, nm, p.ksplit, oz_crt_tab(nm), A.ex + row0, B.ex,
                                         -14 * A.S, D + (int64_t)row0 * ldd, ldd, row0, triD, active);
    LAUNCH_NOTE(1);
  }
  return cudaGetLastError();
}

}  // namespace gevp

// FP64 matrix products on the 16-bit tensor cores through residues.
//
//   D(m, n) = sum_k A(m, k) B(n, k)   for FP64 A and B, real or complex
//
// The FP64 pipe of this part issues 2 FMAs a clock and SM (1.26 TFLOP/s in all), the 16-bit tensor
// cores about 1500 times that, and 16-bit integers up to 2^7 multiply and add exactly in their FP32
// accumulators. So every row of A and of B is scaled by a power of two to integers of about kBeta
// bits (a 2-norm of at most 2^kBeta, so that no inner product exceeds 2^(2 kBeta)), and the integer
// product is formed exactly by the Chinese remainder theorem (the modular form of the
// error-free matrix products: K. Ozaki, Y. Uchino, T. Imamura, "Ozaki Scheme II", arXiv:2504.08009, 2025): kMods pairwise coprime moduli of at most 8 bits, one
// GEMM of symmetric residues (bf16, |r| <= 128) per modulus, and the product recovered modulo
// P = prod p_i > 2 * 2^(2 kBeta). The only errors are the rounding of the operands to integers, half
// a unit of 2^-kBeta of the row's norm (5 bits below the FP64 rounding of an element of the row's
// size), and one rounding of the result: some 2^-59 |a| |b| of the rows' norms, whatever K.
//
// That is below the rounding of a chain of FP64 FMAs, about 2^-54 S with S = sum_k |A(m, k)| |B(n, k)|, while S is at
// least 2^-5 of the norms' bounds, as it is for operands whose large elements meet (S is 0.6 |a| |b| for random ones).
// Rows that are graded over many decades can have results far below their norms, which FMAs get right and a grid
// relative to the norm does not. So the engine forms S as well, in one more product: the magnitudes as bf16, rounded
// down, go through the GEMM as a plane beside the residues, and the reconstruction replaces every result with too small
// an S by the chain of FMAs over the original operands (fma_results). Where S is zero the result is, exactly.
// Measured against quads, two half transforms of K = 48, worst element and rms in units of 2^-53 S: random operands
// 0.16 and 0.025 (FMAs 0.78 and 0.12), elements spread over two decades 0.9 and 0.09 (3.4 and 0.39), four 3.9 and 0.28
// (7.9 and 0.85), eight 7.5 and 0.82 (9.3 and 1.4). The plane costs 6% of an h-BN-shaped call (17.5 -> 18.6 ms); the
// same with L and C falling by 2 / 4 / 20 decades from their diagonals takes 24 / 140 / 256 ms (some 390 on the FP64
// pipe alone).
//
//   1. rns_convert_kernel: per operand row, the scale from its norm; then residues [plane][batch][row][K], the
//      magnitudes as the last plane, K-major (complex operands as interleaved (re, im) pairs along K; the column
//      operand of a complex product as two rows, (re, -im) for the real and (im, re) for the imaginary part).
//   2. rns_gemm_kernel: tcgen05 (128 x up to 256 tiles, TMA-fed), one job per (plane, batch, tile).
//      After every kSegStages K blocks the FP32 sums, exact below 2^24, are reduced modulo p and the
//      running residue is kept as one byte per element in Y [plane][batch][row][col] (of S: see count16).
//   3. rns_crt_kernel: recovers the signed 117-bit integer as a 64-bit fraction of P, rounds it to FP64, undoes the
//      scales, takes the results with a small S from FMAs and writes the caller's layout.
//
// A row with an infinity or a NaN has no scale. Its magnitudes count as the smallest, so its results come from FMAs,
// except where its elements meet zeros only: NaN, as an infinity or NaN times zero is.

#include <cuda.h>
#include <cuda_bf16.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>

#include "rns.h"
#include "tc_common.cuh"

namespace dmet {

namespace {

using namespace tc;

constexpr int kMods = 15;
constexpr int kPlanes = kMods + 1;  // the residues, then the magnitudes
constexpr int kBeta = 58;
__host__ __device__ constexpr int mod_of(int i) {
  constexpr int p[kMods] = {256, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};
  return p[i];
}

using u128 = unsigned __int128;

__host__ __device__ constexpr u128 mod_product() {
  u128 p = 1;
  for (int i = 0; i < kMods; ++i) p *= (u128)mod_of(i);
  return p;
}
// x / P = sum r_i c_i (mod 1) for the residues r_i of x, with c_i = ((P / p_i)^-1 mod p_i) / p_i, as fixed-point
// fractions of 72 bits in words of 32, 20 and 20 bits: a byte times a 20-bit word, kMods times, fits 32 bits, so
// a residue adds with three 32-bit multiply-adds (the top word wraps: modulo 1).
constexpr int kLimb = 20, kFrac = 32 + 2 * kLimb;
static_assert(255 * kMods + 1 <= 1 << (32 - kLimb), "the 20-bit words' sums");
__host__ __device__ constexpr int crt_inverse(int i) {
  const int p = mod_of(i), a = (int)((mod_product() / (u128)p) % (u128)p);
  int inv = 1;
  while ((a * inv) % p != 1) ++inv;
  return inv;
}
__host__ __device__ constexpr u128 crt_fraction(int i) {
  const u128 p = (u128)mod_of(i);
  return (((u128)crt_inverse(i) << kFrac) + p / 2) / p;
}
// Minus the sum's offset for residues stored with 128 added (mod 1), plus half of the last bit that crt_fold keeps.
__host__ __device__ constexpr u128 crt_offset() {
  u128 t = 0;
  for (int i = 0; i < kMods; ++i) t += 128 * crt_fraction(i);
  t = ((u128)1 << (kFrac + 16)) - t + ((u128)1 << (kFrac - 65));
  return t & (((u128)1 << kFrac) - 1);
}
__host__ __device__ constexpr unsigned frac_word(u128 x, int j) {
  return j == 2 ? (unsigned)(x >> (2 * kLimb)) : (unsigned)(x >> (j * kLimb)) & ((1u << kLimb) - 1);
}

constexpr bool mods_ok() {
  for (int i = 0; i < kMods; ++i)
    for (int j = 0; j < i; ++j) {
      int a = mod_of(i), b = mod_of(j);
      while (b) {
        const int t = a % b;
        a = b;
        b = t;
      }
      if (a != 1) return false;
    }
  return true;
}
static_assert(mods_ok(), "the moduli must be pairwise coprime");
static_assert((mod_product() >> (2 * kBeta + 1)) != 0, "P must exceed 2 * 2^(2 kBeta)");
static_assert((mod_product() >> 117) == 1, "P in [2^117, 2^118)");

// Symmetric residue of 2^(16 j) modulo p.
__host__ __device__ constexpr int chunk_weight(int i, int j) {
  const int p = mod_of(i);
  int r = 1;
  for (int t = 0; t < 16 * j; ++t) r = (r * 2) % p;
  return r > p / 2 ? r - p : r;
}

constexpr int kPoison = -(1 << 28);  // scale of a row that holds an infinity or a NaN

// Two values at a time on the paired FP32 pipe, each rounded as the scalar form (x: the low half). Instructions bound
// the conversion (issue at 79%): 22 880 x 520 in 224 us with the scalar form, 204 with this; the GEMM of
// 5720 x 208 x 52 in 55 batches, bound by its epilogue, 357 and 315.
using f32x2 = unsigned long long;
constexpr f32x2 both(unsigned bits) { return ((f32x2)bits << 32) | bits; }
__device__ __forceinline__ f32x2 pack2(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
constexpr f32x2 both_of(float x) { return both(__builtin_bit_cast(unsigned, x)); }
constexpr f32x2 kMagic2 = both(0x4B400000u), kMinusMagic2 = both(0xCB400000u);  // +- 1.5 * 2^23: rounds to an integer
// v - p * rint(v / p) for integers |v| <= 2^24: a residue with |r| <= (p + 1) / 2 (the rounding of v / p
// can pick the neighbour when v / p lies within 2^-9 of a half-integer), so at most 128 for p = 256 and
// 127 for the others: it fits a byte, modulo 256 for p = 256. (p = 255 would reach 128 and is left out.)
__device__ __forceinline__ f32x2 sym_mod2(f32x2 v, f32x2 minus_p, f32x2 rp) {
  return fma2(add2(fma2(v, rp, kMagic2), kMinusMagic2), minus_p, v);
}

__constant__ float kModF[kMods] = {256, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};

// ---------------- operand conversion ----------------

enum { SRC_COMPLEX = 0, SRC_COMPLEX2 = 1, SRC_REAL = 2 };

struct ConvArgs {
  const double* src;
  const int4* tab;  // batch z reads tab[tab0 + z].x (sel 0) or .y (sel 1) in units of sbatch, K from .w
  int tab0, sel;
  long long sbatch;       // batch stride, in elements (complex or real)
  long long s_row, s_k;   // strides of a row and of a k index, in elements
  int rows, K, Kp;        // Kp: real K, padded to the GEMM's K block
  int conj;
  __nv_bfloat16* R;       // [plane][batch][rows (x 2 for SRC_COMPLEX2)][Kp]
  long long smod;         // elements per plane
  int* exps;              // [batch][rows]
};

struct RowNorm {
  float s;  // sum of squares in units of 2^(2 e)
  int e;    // biased exponent of the reference
  int bad;
};

__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((unsigned)(e + 127) << 23); }

__device__ __forceinline__ void norm_add(RowNorm& n, double x) {
  const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu;
  int e = (int)(hi >> 20);
  if (e == 0x7ff) n.bad = 1;
  if (e == 0) {
    if ((hi | (unsigned)__double2loint(x)) == 0) return;
    e = 1;  // subnormal: counted as the smallest normal
  }
  int d = e - n.e;
  if (d > 0) {
    n.s = d < 60 ? n.s * pow2f(-2 * d) : 0.f;
    n.e = e;
    d = 0;
  }
  if (d > -60) {
    const float f = __uint_as_float(((unsigned)(127 + d) << 23) | ((hi & 0xfffffu) << 3) | 7u);
    n.s = fmaf(f, f, n.s);
  }
}

__device__ __forceinline__ void norm_merge(RowNorm& a, float s, int e, int bad) {
  a.bad |= bad;
  const int d = e - a.e;
  if (d > 0) {
    a.s = (d < 60 ? a.s * pow2f(-2 * d) : 0.f) + s;
    a.e = e;
  } else if (d > -60) {
    a.s += s * pow2f(2 * d);
  }
}

// The power s for which the row times 2^s has a 2-norm of at most 2^kBeta.
__device__ __forceinline__ int norm_scale(const RowNorm& n) {
  if (n.bad) return kPoison;
  if (n.s == 0.f) return 0;
  const unsigned b = __float_as_uint(n.s * 1.001f);
  const int se = (int)(b >> 23) - 127;                    // floor(log2 s)
  return kBeta - (n.e - 1023 + ((se + 2) >> 1));
}

// rint(x 2^s) as a two's-complement integer (round half away from zero), |result| <= 2^kBeta (so the binary point of
// x's 53 bits moves left by at most 6).
__device__ __forceinline__ long long to_int(double x, int s) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const int e = (int)((hi >> 20) & 0x7ff);
  const unsigned mh = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)__double2loint(x)) << 6;
  const int r = min(max(1081 - s - (e ? e : 1), 0), 63);
  const long long t = (long long)((m + ((1ull << r) >> 1)) >> r);
  return (int)hi < 0 ? -t : t;
}

// |x| 2^(s - kBeta), at most 1, as a bf16 rounded down; what is below 2^-62 (or subnormal, whose exponent says less)
// counts as that, so that products of two are normal in FP32 and only a zero gives a zero.
constexpr int kMagMin = -62;
__device__ __forceinline__ unsigned magnitude(double x, int s) {
  const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu;
  const int e = (int)(hi >> 20), E = e ? e - 1023 + s - kBeta : kMagMin - 1;
  const unsigned b = E < kMagMin ? (unsigned)(kMagMin + 127) << 7 : ((unsigned)(E + 127) << 7) | ((hi >> 13) & 0x7fu);
  return (hi | (unsigned)__double2loint(x)) ? b : 0u;
}

// Four signed 16-bit digits of a, as floats: a = sum c_j 2^(16 j).
__device__ __forceinline__ void digits(long long a, float (&c)[4]) {
  const unsigned long long b = (unsigned long long)a + 0x8000800080008000ull;
  const unsigned lo = (unsigned)b, hi = (unsigned)(b >> 32);
  constexpr float bias = 8388608.f + 32768.f;  // 2^23 + 2^15
  c[0] = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7610)) - bias;
  c[1] = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7632)) - bias;
  c[2] = __uint_as_float(__byte_perm(hi, 0x4B000000u, 0x7610)) - bias;
  c[3] = __uint_as_float(__byte_perm(hi, 0x4B000000u, 0x7632)) - bias;
}

// |c_j w_j| <= 2^22 for j = 1, 2, 2^18 for j = 3 (|a| <= 2^59) and 2^15 for j = 0: the sum is exact.
struct ModConst {
  f32x2 w1, w2, w3, rp, minus_p;
};
constexpr ModConst mod_const(int i) {
  return ModConst{both_of((float)chunk_weight(i, 1)), both_of((float)chunk_weight(i, 2)),
                  both_of((float)chunk_weight(i, 3)), both_of(1.0f / (float)mod_of(i)), both_of(-(float)mod_of(i))};
}
struct ModTable {
  ModConst m[kMods];
};
constexpr ModTable mod_table() {
  ModTable t{};
  for (int i = 0; i < kMods; ++i) t.m[i] = mod_const(i);
  return t;
}
__constant__ ModTable kModTable = mod_table();

__device__ __forceinline__ f32x2 residues(const f32x2 (&c)[4], const ModConst& m) {
  return sym_mod2(fma2(c[3], m.w3, fma2(c[2], m.w2, fma2(c[1], m.w1, c[0]))), m.minus_p, m.rp);
}

// The residues of one (re, im) or (k, k + 1) pair of each of RW rows, modulus by modulus (rows side by side: their
// chains overlap and share the constants and the plane's address; off: byte offset of a row's pair in a plane, 2 KiB
// planes and up to 4 GiB, or ~0 for a row that is not stored).
// TABLE: the moduli's constants from constant memory, for the kernel that holds the next tile in registers beside four
// rows (80 registers; as immediates 104, and 2 CTAs per SM: 22 880 x 520 in 225 us against 202); elsewhere as
// immediates (5720 x 52 in 55 batches: 182 us, 226 from the table).
template <int SRC, int RW, bool TABLE, int I>
__device__ __forceinline__ void store_residues(const f32x2 (&c)[RW][4], const unsigned (&off)[RW], char* plane,
                                               long long smod, unsigned row2) {
  if constexpr (I < kMods) {
    constexpr ModConst imm = mod_const(I);
#pragma unroll
    for (int i = 0; i < RW; ++i) {
      float re, im;
      unpack2(TABLE ? residues(c[i], kModTable.m[I]) : residues(c[i], imm), re, im);
      if (off[i] != ~0u) {
        *reinterpret_cast<__nv_bfloat162*>(plane + off[i]) = __floats2bfloat162_rn(re, SRC == SRC_COMPLEX2 ? -im : im);
        if constexpr (SRC == SRC_COMPLEX2)
          *reinterpret_cast<__nv_bfloat162*>(plane + (off[i] + row2)) = __floats2bfloat162_rn(im, re);
      }
    }
    store_residues<SRC, RW, TABLE, I + 1>(c, off, plane + smod, smod, row2);
  }
}

// One CTA converts RB operand rows (32, or 8 where that would leave SMs idle): first their norms, then the
// residues, 32 (re, im) or (k, k + 1) pairs at a time, a lane per pair, so that every store of a warp is 128
// contiguous bytes. Rows that are contiguous in memory (s_row = 1) pass through a transpose in shared memory.
template <int SRC, int RB, bool rowfast>
__global__ void __launch_bounds__(256) rns_convert_kernel(const ConvArgs a) {
  constexpr int KL = 256 / RB, RW = RB / 8;  // k lanes per row, rows per warp
  __shared__ double2 tile[rowfast ? 32 : 1][RB + 1];
  __shared__ float sh_s[KL][RB];
  __shared__ int sh_e[KL][RB], sh_bad[KL][RB], sh_scale[RB];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int trow = threadIdx.x % RB, tk = threadIdx.x / RB;
  const int z = blockIdx.y, r0 = blockIdx.x * RB;
  long long off = (long long)z * a.sbatch;
  int K = a.K;
  if (a.tab) {
    const int4 t = a.tab[a.tab0 + z];
    off = (a.sel ? (long long)t.y : (long long)t.x) * a.sbatch;
    K = t.w;
  }
  const double2* src2 = reinterpret_cast<const double2*>(a.src) + off;
  const double* src1 = a.src + off;

  // one element (its second component zero for a real one), zero outside
  auto element = [&](int r, int k) {
    double2 v = make_double2(0.0, 0.0);
    if (r < a.rows && k < K) {
      const long long at = (long long)r * a.s_row + (long long)k * a.s_k;
      if constexpr (SRC == SRC_REAL) v.x = src1[at];
      else v = src2[at];
    }
    return v;
  };
  // norms, four loads in flight per thread
  auto norm_of = [&](int r, int k0, int step) {
    RowNorm n{0.f, 0, 0};
    auto add = [&](double2 v) {
      norm_add(n, v.x);
      if constexpr (SRC != SRC_REAL) norm_add(n, v.y);
    };
    if (r >= a.rows) return n;
    int k = k0;
    for (; k + 3 * step < K; k += 4 * step) {
      double2 v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = element(r, k + i * step);
#pragma unroll
      for (int i = 0; i < 4; ++i) add(v[i]);
    }
    for (; k < K; k += step) add(element(r, k));
    return n;
  };
  if constexpr (rowfast) {
    RowNorm n = norm_of(r0 + trow, tk, KL);
    sh_s[tk][trow] = n.s;
    sh_e[tk][trow] = n.e;
    sh_bad[tk][trow] = n.bad;
    __syncthreads();
    if (tk == 0) {
      for (int w = 1; w < KL; ++w) norm_merge(n, sh_s[w][trow], sh_e[w][trow], sh_bad[w][trow]);
      sh_scale[trow] = norm_scale(n);
    }
  } else {
    for (int i = 0; i < RW; ++i) {
      RowNorm n = norm_of(r0 + warp * RW + i, lane, 32);
      const int e = __reduce_max_sync(0xffffffffu, n.e), d = n.e - e;
      n.s = d > -60 ? n.s * pow2f(2 * d) : 0.f;
      n.e = e;
      n.bad = __any_sync(0xffffffffu, n.bad);
#pragma unroll
      for (int o = 16; o; o >>= 1) n.s += __shfl_xor_sync(0xffffffffu, n.s, o);
      if (lane == 0) sh_scale[warp * RW + i] = norm_scale(n);
    }
  }
  __syncthreads();
  if (threadIdx.x < RB && r0 + trow < a.rows) a.exps[(long long)z * a.rows + r0 + trow] = sh_scale[trow];

  constexpr int RR = SRC == SRC_COMPLEX2 ? 2 : 1;
  const int upad = a.Kp / 2;
  // pair u of row r: (re, im), or (k, k + 1) of a real operand
  auto pair = [&](int r, int u) {
    if constexpr (SRC == SRC_REAL) return make_double2(element(r, 2 * u).x, element(r, 2 * u + 1).x);
    else return element(r, u);
  };
  // a thread's share of the transpose of the tile of 32 pairs from u on: the next tile's is loaded before the current
  // one is converted (22 880 x 520: 286 us without, 224 with, both before the paired arithmetic)
  static_assert(RW * KL == 32, "a thread's share of a tile");
  double2 next[RW];
  auto fetch = [&](int u) {
#pragma unroll
    for (int i = 0; i < RW; ++i) next[i] = pair(r0 + trow, u + tk + i * KL);
  };
  if constexpr (rowfast) fetch(0);
  for (int u0 = 0; u0 < upad; u0 += 32) {
    if constexpr (rowfast) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < RW; ++i) tile[tk + i * KL][trow] = next[i];
      __syncthreads();
      if (u0 + 32 < upad) fetch(u0 + 32);
    }
    const int u = u0 + lane;
    f32x2 c[RW][4];
    unsigned off[RW];
#pragma unroll
    for (int i = 0; i < RW; ++i) {
      const int rl = warp * RW + i, r = r0 + rl;
      const double2 v = rowfast ? tile[rowfast ? lane : 0][rl] : pair(r, u0 + lane);
      const int s = sh_scale[rl];
      long long ar = 0, ai = 0;
      if (s != kPoison) {
        ar = to_int(v.x, s);
        ai = to_int(v.y, s);
        if (SRC != SRC_REAL && a.conj) ai = -ai;
      }
      float cr[4], ci[4];
      digits(ar, cr);
      digits(ai, ci);
#pragma unroll
      for (int j = 0; j < 4; ++j) c[i][j] = pack2(cr[j], ci[j]);
      off[i] = u < upad && r < a.rows ? (unsigned)((((long long)z * a.rows + r) * RR * a.Kp + 2 * u) * 2) : ~0u;
      if (off[i] != ~0u) {
        const unsigned mx = magnitude(v.x, s), my = magnitude(v.y, s);
        char* at = reinterpret_cast<char*>(a.R) + (long long)kMods * a.smod * 2 + off[i];
        *reinterpret_cast<unsigned*>(at) = mx | (my << 16);
        if constexpr (SRC == SRC_COMPLEX2) *reinterpret_cast<unsigned*>(at + (unsigned)a.Kp * 2u) = my | (mx << 16);
      }
    }
    store_residues<SRC, RW, rowfast && RW == 4, 0>(c, off, reinterpret_cast<char*>(a.R), a.smod * 2,
                                                   (unsigned)a.Kp * 2u);
  }
}

// ---------------- GEMM of residues ----------------

constexpr int kTileM = 128;
constexpr int kBK = 64;             // K elements per stage (128-byte rows)
constexpr int kSegStages = 15;      // 960 K per segment: 960 * 128^2 + 128 < 2^24
constexpr int kStages = 4;
constexpr int kEpi = 8;             // epilogue warps
constexpr int kGemmThreads = 32 * (4 + kEpi);
constexpr int kABytes = kTileM * 128;
constexpr int kBBytes = 256 * 128;
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kGemmSmem = 1024 + kStages * kStageBytes + 256;

struct GemmArgs {
  int nbatch, rows, cols;   // per batch entry
  int rt, ct, bn;           // row tiles, column tiles, tile width (a multiple of 16, <= 256)
  int tri, h0;              // tri: only tiles with a column <= the last row (square product, bn = 256); row 0 of
                            // this launch is row 256 h0 of the product
  int row0;                 // first row of the launch in the row operand
  int jobs;                 // tiles per (plane, batch)
  int nkb, seg;             // K blocks, and how many of them between reductions (at most kSegStages)
  signed char* Y;           // [plane][batch] in tiles (y_tile)
  long long ymod;
  int ldy;
};

// Y, the products' residues, lies in tiles of 32 rows x 16 columns, a row's 16 bytes after the other's: a warp of the
// GEMM's epilogue stores, and one of the reconstruction loads, 512 contiguous bytes with a lane per row. (Row by row
// the same accesses touched 32 lines each: 5720 x 208 x 52 in 55 batches took 523 us for the GEMM and 509 for the
// reconstruction, 357 and 324 so.) Offset of the tile with row group rg and column c (a multiple of 16) of a batch
// entry of `rows` rows.
__host__ __device__ inline long long y_tile(int z, int rows, int ldy, int rg, int c) {
  return (((long long)z * ((rows + 31) >> 5) + rg) * (ldy >> 4) + (c >> 4)) * 512;
}

struct Tile {
  int mod, z, m0, n0;
};

// Lower triangle: the row tiles 2 h and 2 h + 1 have h0 + h + 1 column tiles each; pairs of jobs take them side by side.
__host__ __device__ inline int tri_jobs_before(int h, int h0) { return h * h0 + h * (h + 1) / 2; }

// Job `job` of a launch.
__device__ __forceinline__ Tile tile_of(const GemmArgs& g, int job) {
  Tile t;
  const int per = g.nbatch * g.jobs;
  t.mod = job / per;
  int r = job - t.mod * per;
  t.z = r / g.jobs;
  r -= t.z * g.jobs;
  int mt, nt;
  if (g.tri) {
    const int u = r >> 1;
    const float c = (float)(2 * g.h0 + 1);
    int h = (int)((sqrtf(c * c + 8.f * (float)u) - c) * 0.5f);
    while (h > 0 && tri_jobs_before(h, g.h0) > u) --h;
    while (tri_jobs_before(h + 1, g.h0) <= u) ++h;
    mt = 2 * h + (r & 1);
    nt = u - tri_jobs_before(h, g.h0);
  } else {
    mt = r / g.ct;
    nt = r - mt * g.ct;
  }
  t.m0 = mt * kTileM;
  t.n0 = nt * g.bn;
  return t;
}

// 16 accumulator columns to bytes: v (+ the running residue) modulo p.
__device__ __forceinline__ uint4 reduce16(const uint32_t (&v)[16], bool add, uint4 prev, f32x2 minus_p, f32x2 rp) {
  uint32_t w[4];
  const uint32_t pv[4] = {prev.x, prev.y, prev.z, prev.w};
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    float b[4];
#pragma unroll
    for (int c = 0; c < 4; c += 2) {
      f32x2 x = pack2(__uint_as_float(v[4 * g + c]), __uint_as_float(v[4 * g + c + 1]));
      if (add)
        x = add2(x, pack2((float)(int)(signed char)(pv[g] >> (8 * c)), (float)(int)(signed char)(pv[g] >> (8 * c + 8))));
      unpack2(add2(sym_mod2(x, minus_p, rp), kMagic2), b[c], b[c + 1]);  // the low byte is the residue's
    }
    w[g] = __byte_perm(__byte_perm(__float_as_uint(b[0]), __float_as_uint(b[1]), 0x0040),
                       __byte_perm(__float_as_uint(b[2]), __float_as_uint(b[3]), 0x0040), 0x5410);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// 16 sums of magnitudes to bytes: 2 n + (S != 0), n = 127 S rounded down (within one), a segment added to the next: S is
// at most 1 over all of K, so n stays below 128. An S other than zero is at least 2^-124, so its upper byte is not zero.
// (With conversions to integers instead of the rounding constant the GEMM of 2465 x 61 x 17 in 76 batches took 189 us, 184
// so, and an h-BN-shaped call 18.60 ms, 18.57.)
__device__ __forceinline__ uint4 count16(const uint32_t (&v)[16], bool add, uint4 prev) {
  constexpr f32x2 scale = both_of(127.f), minus_half = both_of(-0.5f);
  uint32_t w[4];
  const uint32_t pv[4] = {prev.x, prev.y, prev.z, prev.w};
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    float b[4];
#pragma unroll
    for (int c = 0; c < 4; c += 2) {
      const f32x2 x = pack2(__uint_as_float(v[4 * g + c]), __uint_as_float(v[4 * g + c + 1]));
      unpack2(add2(fma2(x, scale, minus_half), kMagic2), b[c], b[c + 1]);  // the low byte is n
    }
    const uint32_t n = __byte_perm(__byte_perm(__float_as_uint(b[0]), __float_as_uint(b[1]), 0x0040),
                                   __byte_perm(__float_as_uint(b[2]), __float_as_uint(b[3]), 0x0040), 0x5410);
    const uint32_t t = __byte_perm(__byte_perm(v[4 * g], v[4 * g + 1], 0x0073),
                                   __byte_perm(v[4 * g + 2], v[4 * g + 3], 0x0073), 0x5410);
    w[g] = (n << 1) | (((t + 0x7f7f7f7fu) >> 7) & 0x01010101u);
    if (add) w[g] = (w[g] + (pv[g] & 0xfefefefeu)) | (pv[g] & 0x01010101u);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Bound by the L2 reads of the operands: a 128 x 256 tile reads 48 KB per 512 clocks of MMA, and the L2 gives some
// 10 TB/s in all. Every CTA loads its own tiles, without TMA multicast: the same code runs where several GPUs take part
// (pairs of CTAs that shared the column tile by multicast: 17.39 ms for an h-BN-shaped call, 17.50 so).
__global__ void __launch_bounds__(kGemmThreads, 1)
    rns_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmArgs g,
                    int njobs, unsigned int* err, unsigned long long lim, int withhold) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + kStages * kStageBytes);
  // bars: full[S], empty[S], accf[2], acce[2], done; then the TMEM address and a counter
  volatile uint32_t* tmem_slot = (volatile uint32_t*)(bars + 2 * kStages + 5);
  volatile int* consumed = (volatile int*)(bars + 2 * kStages + 5) + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto full = [&](int s) { return smem_u32(bars + s); };
  auto empty = [&](int s) { return smem_u32(bars + kStages + s); };
  auto accf = [&](int b) { return smem_u32(bars + 2 * kStages + b); };
  auto acce = [&](int b) { return smem_u32(bars + 2 * kStages + 2 + b); };
  const uint32_t done_bar = smem_u32(bars + 2 * kStages + 4);
  auto a_tile = [&](int s) { return smem_u32(smem + s * kStageBytes); };
  auto b_tile = [&](int s) { return smem_u32(smem + s * kStageBytes + kABytes); };
  const int job0 = (int)blockIdx.x, njob = (int)gridDim.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf(b), 1);
      mbar_init(acce(b), kEpi);
    }
    mbar_init(done_bar, 1);
    *consumed = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(bars + 2 * kStages + 5), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  int issued = 0;
  if (warp == 0) {
    if (lane == 0) {
      prefetch_tmap(&tmA);
      prefetch_tmap(&tmB);
      const uint32_t bytes = kABytes + (uint32_t)g.bn * 128u;
      bool ok = !withhold;
      for (int jb = job0; jb < njobs && ok; jb += njob) {
        const Tile t = tile_of(g, jb);
        const int ra = t.z * g.rows + g.row0 + t.m0, rb = t.z * g.cols + t.n0;
        for (int kb = 0; kb < g.nkb; ++kb) {
          const int s = issued % kStages, ph = (issued / kStages) & 1;
          if (!mbar_wait(empty(s), ph ^ 1, err, 1u, lim)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(full(s), bytes);
          tma_load_3d(a_tile(s), &tmA, full(s), kb * kBK, ra, t.mod);
          tma_load_3d(b_tile(s), &tmB, full(s), kb * kBK, rb, t.mod);
          ++issued;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_f32acc(1, kTileM, g.bn);
      int it = 0, gs = 0;
      bool ok = true;
      for (int jb = job0; jb < njobs && ok; jb += njob) {
        for (int k0 = 0; k0 < g.nkb && ok; k0 += g.seg, ++gs) {
          const int b = gs & 1, u = gs >> 1;
          if (!mbar_wait(acce(b), (u & 1) ^ 1, err, 2u, lim)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const int k1 = min(g.nkb, k0 + g.seg);
          for (int kb = k0; kb < k1; ++kb) {
            const int s = it % kStages, ph = (it / kStages) & 1;
            if (!mbar_wait(full(s), ph, err, 4u, lim)) {
              ok = false;
              break;
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              umma<0>(tmem + b * 256, smem_desc<128>(a_tile(s) + kk * 32), smem_desc<128>(b_tile(s) + kk * 32), idesc,
                      (kb > k0 || kk) ? 1u : 0u);
            umma_commit(empty(s));
            ++it;
            *consumed = it;
          }
          if (ok) umma_commit(accf(b));
        }
      }
      umma_commit(done_bar);
      mbar_wait(done_bar, 0, err, 16u, lim);
    }
  } else if (warp >= 4) {
    const int quad = warp & 3, half = (warp - 4) >> 2;
    bool ok = true;
    int gs = 0;
    for (int jb = job0; jb < njobs && ok; jb += njob) {
      const Tile t = tile_of(g, jb);
      const bool mags = t.mod == kMods;
      const float p = kModF[mags ? 0 : t.mod];
      const f32x2 minus_p = pack2(-p, -p), rp = pack2(1.0f / p, 1.0f / p);
      const int row = t.m0 + quad * 32 + lane;
      signed char* y =
          g.Y + (long long)t.mod * g.ymod + y_tile(t.z, g.rows, g.ldy, t.m0 / 32 + quad, t.n0) + lane * 16;
      const bool rok = row < g.rows;
      const int cols = min(g.bn, g.ldy - t.n0);
      for (int k0 = 0; k0 < g.nkb; k0 += g.seg, ++gs) {
        const int b = gs & 1, u = gs >> 1;
        // the running residues, on their way while the MMAs finish (one at a time behind each accumulator
        // read, their latency was most of the epilogue)
        uint4 prev[8];
        if (k0 && rok) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (half * 16 + 32 * i < cols) prev[i] = *reinterpret_cast<const uint4*>(y + (half + 2 * i) * 512);
        }
        if (!__all_sync(0xffffffffu, mbar_wait(accf(b), u & 1, err, 8u, lim))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t tm = tmem + b * 256 + ((uint32_t)(quad * 32) << 16);
        auto drain = [&](auto to_bytes) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int c = half * 16 + 32 * i;
            if (c >= cols) break;  // (uniform)
            uint32_t v[16];
            tmem_ld_32x32b_x16(tm + c, v);
            tmem_ld_wait();
            const uint4 w = to_bytes(v, prev[i]);
            if (rok) *reinterpret_cast<uint4*>(y + (half + 2 * i) * 512) = w;
          }
        };
        // (two loops: with the choice within one an h-BN-shaped call took 18.83 ms, so 18.60)
        if (mags) drain([&](const uint32_t (&v)[16], uint4 o) { return count16(v, k0 != 0, o); });
        else drain([&](const uint32_t (&v)[16], uint4 o) { return reduce16(v, k0 != 0, o, minus_p, rp); });
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce(b));
      }
    }
  }
  __syncthreads();
  if (warp == 0 && lane == 0) {
    // copies issued but never consumed (only after an expired wait) must land before exit
    for (int i = *consumed; i < issued; ++i) mbar_wait(full(i % kStages), (i / kStages) & 1, err, 32u, lim);
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ---------------- reconstruction ----------------

// An operand of the product, for the results that are taken from FMAs.
struct FmaSide {
  const double* src;           // the launch's first row
  long long sbatch, s_row, s_k;
  int sel, conj;               // as in ConvArgs
};

struct CrtArgs {
  const signed char* Y;
  long long ymod;
  int ldy, rows, cols;      // cols: real columns (2 per complex column)
  int row0;                 // first row of the launch in the product
  const int* ea;            // [batch][ea_rows] scales, from row row0
  const int* eb;            // [batch][columns (complex or real)]
  int ea_rows, eb_rows;
  // complex: D[z.. + row map + column map]
  double2* D;
  const int4* tab;
  int tab0;
  long long sD;
  int r_div, c_div;
  long long r_hi, r_lo, c_hi, c_lo;
  // real
  double* out;
  long long ldo;
  int tri;
  double alpha;
  int scaled;               // alpha != 1 (tested as an integer: the FP64 pipe is slow)
  int beta;
  FmaSide rside, cside;
  int rows_are_m, K;
};

struct Frac {
  unsigned w[3];  // low, middle, top word
};
__device__ __forceinline__ Frac frac_start() {
  constexpr u128 off = crt_offset();
  return Frac{{frac_word(off, 0), frac_word(off, 1), frac_word(off, 2)}};
}
// u = residue + 128
__device__ __forceinline__ void frac_add(Frac& f, unsigned u, unsigned c0, unsigned c1, unsigned c2) {
  f.w[0] += u * c0;
  f.w[1] += u * c1;
  f.w[2] += u * c2;
}
__device__ __forceinline__ unsigned long long frac_fold(const Frac& f) {
  constexpr unsigned mask = (1u << kLimb) - 1;
  const unsigned m = f.w[1] + (f.w[0] >> kLimb), t = f.w[2] + (m >> kLimb);
  return ((unsigned long long)t << 32) | ((m & mask) << (32 - kLimb)) | ((f.w[0] & mask) >> (2 * kLimb - 32));
}

template <int I>
__device__ __forceinline__ void crt_add(const uint2 (&y)[kMods], int w, int c, Frac& f) {
  if constexpr (I < kMods) {
    constexpr u128 C = crt_fraction(I);
    frac_add(f, __byte_perm(w ? y[I].y : y[I].x, 0, 0x4440 + c), frac_word(C, 0), frac_word(C, 1), frac_word(C, 2));
    crt_add<I + 1>(y, w, c, f);
  }
}

// Results outside FP64's normal range, and those of poisoned rows.
__device__ __noinline__ double scaled_value(unsigned long long r, int e, bool poison, bool neg) {
  if (poison) return __longlong_as_double(0x7ff8000000000000ll);
  const double d = scalbn((double)r, e - 52);
  return neg ? -d : d;
}

// x 2^-s from the signed fraction f = 2^64 x / P: |f| P in integers (the FP64 pipe would take a conversion and a
// multiplication per value, each 1/64 of the rate), rounded to FP64. The fraction is good to 2^-62.7 of P, that is
// to 2^-61.3 of the product of the two rows' norm bounds, below the rounding of the operands.
__device__ __forceinline__ double crt_value(unsigned long long f, int s) {
  constexpr unsigned long long P64 = (unsigned long long)(mod_product() >> 54);
  const unsigned sign = (unsigned)(f >> 32) & 0x80000000u;
  const unsigned long long a = sign ? 0ull - f : f;
  const int lz = __clzll((long long)(a | 1));
  unsigned long long h = __umul64hi(a << lz, P64);
  int e = 63 + 54 - lz - s;
  if (!(h >> 63)) {
    h <<= 1;
    --e;
  }
  const unsigned long long r = (h >> 11) + ((h >> 10) & 1);
  if ((unsigned)(e + 1021) > 2043u) return scaled_value(r, e, s < kPoison / 2, sign != 0);
  const unsigned hi = (unsigned)(r >> 32) + ((unsigned)(e + 1022) << 20);
  return a ? __hiloint2double((int)(hi | sign), (int)(unsigned)r) : 0.0;
}

__device__ __forceinline__ long long map_index(int x, int div, long long hi, long long lo) {
  if (div == INT_MAX) return x * lo;
  const int q = x / div;
  return q * hi + (x - q * div) * lo;
}

// Output of a warp's 32 rows x 16 columns (8 complex) from its stage[32][17], a lane per row. Complex results whose
// rows are contiguous in the output leave as 512 contiguous bytes per store, the others as 128-byte segments
// of a row (radrs: the rows' offsets).
__device__ __forceinline__ void put_complex(const CrtArgs& a, double2* d, double re, double im) {
  double2 v = make_double2(re, im);
  if (a.scaled) {
    v.x *= a.alpha;
    v.y *= a.alpha;
  }
  if (a.beta) {
    const double2 o = *d;
    v.x += o.x;
    v.y += o.y;
  }
  *d = v;
}

__device__ __forceinline__ void store_complex(const CrtArgs& a, double2* D, const double* st, long long* radrs, int c0,
                                              int rbase, int lane) {
  const int row = rbase + lane;
  const long long radr = map_index(a.row0 + row, a.r_div, a.r_hi, a.r_lo);
  if (a.r_lo == 1) {
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int cc = (c0 >> 1) + c;
      if (2 * cc >= a.cols) break;
      if (row < a.rows)
        put_complex(a, D + radr + map_index(cc, a.c_div, a.c_hi, a.c_lo), st[lane * 17 + 2 * c], st[lane * 17 + 2 * c + 1]);
    }
    return;
  }
  radrs[lane] = radr;
  __syncwarp();
  // 4 rows x 8 complex columns per pass
  const int cc = (c0 >> 1) + (lane & 7);
  const long long cadr = map_index(cc, a.c_div, a.c_hi, a.c_lo);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int rl = i * 4 + (lane >> 3);
    if (rbase + rl < a.rows && 2 * cc < a.cols)
      put_complex(a, D + radrs[rl] + cadr, st[rl * 17 + 2 * (lane & 7)], st[rl * 17 + 2 * (lane & 7) + 1]);
  }
  __syncwarp();
}

// Results whose S is below kMinCount / 127 of the norms' bounds come from FMAs: the residues' error, about 2^-59 of
// those bounds, is then above the 2^-54 S of a chain.
constexpr unsigned kMinCount = 4;

// Bit 4 h + i (real: element i of the word) or 2 h + i (complex: pair i, by the larger modulus bound S_re + S_im) of
// the result for results with a small S. w: four bytes of count16.
template <bool CPLX>
__device__ __forceinline__ unsigned small_sums(unsigned w) {
  const unsigned n = (w >> 1) & 0x7f7f7f7fu;
  if constexpr (CPLX) {
    constexpr unsigned add = 0x8000u - 2 * kMinCount;
    const unsigned sum = (n & 0x00ff00ffu) + ((n >> 8) & 0x00ff00ffu), any = (w | w >> 8) & 0x00010001u;
    const unsigned ok = (sum + (add << 16 | add)) | ((any ^ 0x00010001u) << 15);
    return ((~ok >> 15) & 1u) | ((~ok >> 30) & 2u);
  } else {
    const unsigned ok = (n + 0x01010101u * (0x80u - kMinCount)) | ((~w & 0x01010101u) << 7), bad = ~ok & 0x80808080u;
    return ((bad >> 7) & 1u) | ((bad >> 14) & 2u) | ((bad >> 21) & 4u) | ((bad >> 28) & 8u);
  }
}

// The results of a warp's 32 x 16 (8 complex) that `flags` marks, a bit per column and lane (row), as FMAs: listed in
// order of columns, a lane per result while there are 32, 32 / n lanes for each of the last n (one lane each: 400 us
// more for an FFTDF call of 2.1 ms with a few results of K = 432, and the h-BN-shaped call of 2 decades 30 ms, now 24).
template <bool CPLX>
__device__ __noinline__ void fma_results(const CrtArgs& a, double* st, unsigned short* list, unsigned flags, int c0,
                                         int rbase, int z) {
  const int lane = threadIdx.x & 31, cbase = CPLX ? c0 >> 1 : c0;
  int n = 0;
#pragma unroll 1
  for (int c = 0; c < (CPLX ? 8 : 16); ++c) {
    const bool f = (flags >> c & 1u) && rbase + lane < a.rows && (cbase + c) * (CPLX ? 2 : 1) < a.cols &&
                   !(a.tri && cbase + c > a.row0 + rbase + lane);
    const unsigned b = __ballot_sync(0xffffffffu, f);
    if (f) list[n + __popc(b & ((1u << lane) - 1u))] = (unsigned short)(c << 5 | lane);
    n += __popc(b);
  }
  __syncwarp();
  long long zr = z, zc = z;
  int K = a.K;
  if (CPLX && a.tab) {
    const int4 t = a.tab[a.tab0 + z];
    zr = a.rside.sel ? t.y : t.x;
    zc = a.cside.sel ? t.y : t.x;
    K = t.w;
  }
#pragma unroll 1
  for (int t0 = 0; t0 < n; t0 += 32) {
    int g = 1;  // lanes per result
    while ((n - t0) * g <= 16) g *= 2;
    const int t = t0 + lane / g, k0 = lane & (g - 1);
    const int item = t < n ? list[t] : 0, r = item & 31, c = item >> 5;
    const long long ro = zr * a.rside.sbatch + (rbase + r) * a.rside.s_row;
    const long long co = zc * a.cside.sbatch + (cbase + c) * a.cside.s_row;
    const int Kt = t < n ? K : 0;
    double re = 0.0, im = 0.0;
    if constexpr (CPLX) {
      const double2* p = reinterpret_cast<const double2*>(a.rside.src) + ro;
      const double2* q = reinterpret_cast<const double2*>(a.cside.src) + co;
      long long ps = a.rside.s_k, qs = a.cside.s_k;
      if (!a.rows_are_m) {
        const double2* x = p;
        p = q;
        q = x;
        ps = a.cside.s_k;
        qs = a.rside.s_k;
      }
      const bool cj = a.rside.conj | a.cside.conj;  // (of the m operand)
#pragma unroll 4
      for (int k = k0; k < Kt; k += g) {
        double2 u = p[k * ps];
        const double2 v = q[k * qs];
        if (cj) u.y = -u.y;
        re = fma(u.x, v.x, re);
        im = fma(u.x, v.y, im);
        re = fma(-u.y, v.y, re);
        im = fma(u.y, v.x, im);
      }
    } else {
      const double* p = a.rside.src + ro;
      const double* q = a.cside.src + co;
#pragma unroll 4
      for (int k = k0; k < Kt; k += g) re = fma(p[k * a.rside.s_k], q[k * a.cside.s_k], re);
    }
    for (int o = g >> 1; o; o >>= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      if constexpr (CPLX) im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (t < n && k0 == 0) {
      st[r * 17 + (CPLX ? 2 * c : c)] = re;
      if constexpr (CPLX) st[r * 17 + 2 * c + 1] = im;
    }
  }
  __syncwarp();
}

// A warp takes 32 rows x 16 columns, a lane per row, 8 columns at a time (15 planes of 8 bytes in registers, so
// that four CTAs fit an SM). Bound by issue (157 instructions per value, 45 of them the multiply-adds of the
// fractions): 65.4 M values in 324 us. The same with the whole integer in 64-bit multiply-adds on
// 30-bit limbs and 16 columns a time took 238 instructions at half the occupancy, twice the time.
template <bool CPLX>
__global__ void __launch_bounds__(256, 4) rns_crt_kernel(const __grid_constant__ CrtArgs a) {
  __shared__ double stage[8][32 * 17];
  __shared__ long long radrs[CPLX ? 8 : 1][32];
  __shared__ unsigned short list[8][CPLX ? 256 : 512];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int z = blockIdx.y;
  const long long item = (long long)blockIdx.x * 8 + warp;
  const int nc = (a.cols + 15) / 16;
  const int rg = (int)(item / nc);
  const int c0 = (int)(item - (long long)rg * nc) * 16, rbase = rg * 32, row = rbase + lane;
  if (rbase >= a.rows) return;                                     // (whole warps leave)
  if (!CPLX && a.tri && c0 > a.row0 + rbase + 31) return;
  const bool rok = row < a.rows;
  const signed char* yp = a.Y + y_tile(z, a.rows, a.ldy, rg, c0) + lane * 16;  // (rows past the end: padding)
  const int sa = rok ? a.ea[(long long)z * a.ea_rows + row] : 0;
  const int* ebp = a.eb + (long long)z * a.eb_rows;
  double* st = stage[warp];
  unsigned flags = 0;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    if (c0 + 8 * h >= a.cols) break;
    uint2 y[kMods];
#pragma unroll
    for (int i = 0; i < kMods; ++i) {
      y[i] = *reinterpret_cast<const uint2*>(yp + (long long)i * a.ymod + 8 * h);
      y[i].x ^= 0x80808080u;
      y[i].y ^= 0x80808080u;
    }
    const uint2 m = *reinterpret_cast<const uint2*>(yp + (long long)kMods * a.ymod + 8 * h);
    flags |= CPLX ? (small_sums<CPLX>(m.x) | small_sums<CPLX>(m.y) << 2) << (4 * h)
                  : (small_sums<CPLX>(m.x) | small_sums<CPLX>(m.y) << 4) << (8 * h);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      Frac f = frac_start();
      crt_add<0>(y, c >> 2, c & 3, f);
      const int sb = ebp[min(c0 + 8 * h + c, a.cols - 1) >> (CPLX ? 1 : 0)];
      st[lane * 17 + 8 * h + c] = crt_value(frac_fold(f), sa + sb);
    }
  }
  __syncwarp();
  if (__any_sync(0xffffffffu, flags != 0)) fma_results<CPLX>(a, st, list[warp], flags, c0, rbase, z);
  if constexpr (CPLX) {
    double2* D = a.D + (a.tab ? (long long)a.tab[a.tab0 + z].z : (long long)z) * a.sD;
    store_complex(a, D, st, radrs[warp], c0, rbase, lane);
  } else {
    // 2 rows x 16 columns per pass
    const int col = c0 + (lane & 15);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int rl = i * 2 + (lane >> 4);
      const long long m = (long long)a.row0 + rbase + rl;
      if (rbase + rl >= a.rows || col >= a.cols || (a.tri && col > m)) continue;
      double* d = a.out + (a.tri ? m * (m + 1) / 2 + col : m * a.ldo + col);
      *d += a.alpha * st[rl * 17 + (lane & 15)];
    }
  }
}

unsigned crt_blocks(int rows, int cols) {
  return (unsigned)(((long long)((rows + 31) / 32) * ((cols + 15) / 16) + 7) / 8);
}

// ---------------- host side ----------------

inline long long pad_to(long long x, long long m) { return (x + m - 1) / m * m; }

// One operand in the engine's terms.
struct Side {
  int src;              // SRC_*
  const double* base;
  int sel;
  long long sbatch, s_row, s_k;
  int rows, conj;
};

// `o` from row r0 on, for the chunk of batch entries from batch0 on.
FmaSide fma_side(const Side& o, int r0, const int4* tab, long long batch0) {
  const int w = o.src == SRC_REAL ? 1 : 2;
  return {o.base + (long long)w * (r0 * o.s_row + (tab ? 0 : batch0 * o.sbatch)), o.sbatch, o.s_row, o.s_k, o.sel, o.conj};
}

cudaError_t convert(const Side& o, int r0, int nrows, const int4* tab, int tab0, int K, int Kp, int nb,
                    long long batch0, __nv_bfloat16* R, long long smod, int* exps, int sms, cudaStream_t s) {
  ConvArgs a;
  std::memset(&a, 0, sizeof(a));
  a.src = fma_side(o, r0, tab, batch0).src;
  a.tab = tab;
  a.tab0 = tab0;
  a.sel = o.sel;
  a.sbatch = o.sbatch;
  a.s_row = o.s_row;
  a.s_k = o.s_k;
  a.rows = nrows;
  a.K = K;
  a.Kp = Kp;
  a.conj = o.conj;
  a.R = R;
  a.smod = smod;
  a.exps = exps;
  const bool few = (long long)((nrows + 31) / 32) * nb < 2 * sms;
  const dim3 grid(few ? (nrows + 7) / 8 : (nrows + 31) / 32, nb);
  const bool rf = o.s_row == 1;
  auto go = [&](auto wide_rows, auto wide_k, auto narrow_rows, auto narrow_k) {
    if (few && rf) narrow_rows<<<grid, 256, 0, s>>>(a);
    else if (few) narrow_k<<<grid, 256, 0, s>>>(a);
    else if (rf) wide_rows<<<grid, 256, 0, s>>>(a);
    else wide_k<<<grid, 256, 0, s>>>(a);
  };
#define DMET_RNS_CONVERT(S)                                                              \
  go(rns_convert_kernel<S, 32, true>, rns_convert_kernel<S, 32, false>, rns_convert_kernel<S, 8, true>, \
     rns_convert_kernel<S, 8, false>)
  if (o.src == SRC_COMPLEX) DMET_RNS_CONVERT(SRC_COMPLEX);
  else if (o.src == SRC_COMPLEX2) DMET_RNS_CONVERT(SRC_COMPLEX2);
  else go(rns_convert_kernel<SRC_REAL, 32, true>, rns_convert_kernel<SRC_REAL, 32, true>,
          rns_convert_kernel<SRC_REAL, 8, true>, rns_convert_kernel<SRC_REAL, 8, true>);  // (real rows are contiguous)
#undef DMET_RNS_CONVERT
  return cudaGetLastError();
}

int tile_width(int cols) {
  const int ct = (cols + 255) / 256;
  return (int)pad_to((cols + ct - 1) / ct, 16);
}

cudaError_t gemm(const __nv_bfloat16* RA, long long smodA, const __nv_bfloat16* RB, long long smodB, GemmArgs g, int Kp,
                 int total_rows_a, const RnsCtx& c, cudaStream_t s) {
  CUtensorMap ma, mb;
  cudaError_t e = make_tmap_rows128(&ma, RA, Kp, (unsigned long long)g.nbatch * total_rows_a, kPlanes, smodA, kTileM);
  if (e != cudaSuccess) return e;
  g.jobs = g.tri ? 2 * tri_jobs_before((g.rt + 1) / 2, g.h0) : g.rt * g.ct;
  e = make_tmap_rows128(&mb, RB, Kp, (unsigned long long)g.nbatch * g.cols, kPlanes, smodB, g.bn);
  if (e != cudaSuccess) return e;
  const int segs = (g.nkb + kSegStages - 1) / kSegStages;
  g.seg = (g.nkb + segs - 1) / segs;
  const int njobs = kPlanes * g.nbatch * g.jobs;
  e = cudaFuncSetAttribute(rns_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmSmem);
  if (e != cudaSuccess) return e;
  rns_gemm_kernel<<<std::min(njobs, c.sms), kGemmThreads, kGemmSmem, s>>>(ma, mb, g, njobs, c.err, c.wait_ns,
                                                                         c.withhold_loads);
  return cudaGetLastError();
}

// Splits the context's scratch; every piece starts on a 1024-byte boundary.
struct Carve {
  char* p;
  char* end;
  void* take(size_t n) {
    char* q = (char*)(((uintptr_t)p + 1023) & ~(uintptr_t)1023);
    p = q + n;
    return q;
  }
};

struct ZPlan {
  Side rows, cols;
  int K, Kp, ldy;
  size_t row_bytes, col_bytes, y_bytes, exps;  // per batch entry: row residues, column residues, Y, the rows' scales
  bool rows_are_m;
};

ZPlan zplan(const ZgemmArgs& a, int al, bool cj, int bl) {
  ZPlan p;
  Side A{SRC_COMPLEX, reinterpret_cast<const double*>(a.A), 0, a.sA, al == A_KM ? 1 : a.lda, al == A_KM ? a.lda : 1, a.M,
         cj ? 1 : 0};
  Side B{SRC_COMPLEX, reinterpret_cast<const double*>(a.B), 1, a.sB, bl == B_KN ? 1 : a.ldb, bl == B_KN ? a.ldb : 1, a.N,
         0};
  p.rows_are_m = a.M > a.N;
  p.rows = p.rows_are_m ? A : B;
  p.cols = p.rows_are_m ? B : A;
  p.cols.src = SRC_COMPLEX2;
  p.K = a.K;
  p.Kp = (int)pad_to(2ll * a.K, kBK);
  p.ldy = (int)pad_to(2ll * p.cols.rows, 16);
  p.row_bytes = (size_t)p.rows.rows * p.Kp * 2 * kPlanes;
  p.col_bytes = (size_t)2 * p.cols.rows * p.Kp * 2 * kPlanes;
  p.y_bytes = (size_t)pad_to(p.rows.rows, 32) * p.ldy * kPlanes;
  p.exps = ((size_t)p.rows.rows + p.cols.rows) * 4 + 4096;
  return p;
}

// How a product runs in the scratch there is: chunks of nb whole batch entries, or of nr rows of one entry. False: not
// at all (less than 128 rows fit beside the column operand and the scales).
struct ZChunks {
  int nb, nr;
  long long launches;  // chunks
};
bool zchunks(const ZPlan& p, int batch, size_t bytes, ZChunks* c) {
  if (bytes <= 16384) return false;
  const size_t avail = bytes - 16384, fixed = p.col_bytes + p.exps;
  const int rows = p.rows.rows;
  c->nb = (int)std::min<size_t>((size_t)batch, avail / (p.row_bytes + p.col_bytes + p.y_bytes + p.exps));
  c->nr = rows;
  if (c->nb < 1) {
    c->nb = 1;
    if (fixed >= avail) return false;
    const size_t per_row = ((size_t)p.Kp * 2 + p.ldy) * kPlanes;
    c->nr = (int)std::min<size_t>((size_t)rows, (avail - fixed) / per_row / 128 * 128);
    if (c->nr < 1) return false;
  }
  c->launches = (long long)((batch + c->nb - 1) / c->nb) * ((rows + c->nr - 1) / c->nr);
  return true;
}

}  // namespace

size_t rns_need(const ZgemmArgs& a) {
  const ZPlan p = zplan(a, A_KM, false, B_KN);
  return (p.row_bytes + p.col_bytes + p.y_bytes + p.exps) * a.batch + 16384;
}

size_t rns_need(const DsyrkArgs& a) {
  const size_t kp = (size_t)pad_to(a.K, kBK), rows = (size_t)a.M + (a.mode ? a.N : 0);
  return rows * kp * 2 * kPlanes + (size_t)pad_to(a.M, 32) * pad_to(a.N, 16) * kPlanes + rows * 4 + 65536;
}

// Where the line between the two lies (fitted to shapes from 8 x 256 x 8 to 128 x 22 880 x 1024, single and batched): the
// FP64 kernel takes 0.27 us per k and 16 x 16 complex tile and SM (less where a tile has few rows); the residues
// take 28 us for their four launches, 85 ns per k of a conversion that few CTAs share, 34 ps per complex
// result (reconstruction and epilogue) and 12 ps per converted real element, and the MMAs. A 128 x 4096 product:
// K = 8, 35 against 43 us; K = 16, 64 against 44; K = 64, 238 against 48. (At large sizes a result
// takes 20 ps and a converted element 9 since Y lies in tiles; the line, where the launches count, is where it was.)
// A product that the scratch only lets run in chunks pays the launches for each: where that is many, FMAs are faster.
bool rns_takes_zgemm(const ZgemmArgs& a, const RnsCtx& c) {
  if (!c.scratch || a.lower || a.M <= 0 || a.N <= 0 || a.K <= 0 || a.batch <= 0) return false;
  const ZPlan p = zplan(a, A_KM, false, B_KN);
  ZChunks ch;
  if (!zchunks(p, a.batch, c.bytes, &ch)) return false;
  const double ctas = std::ceil((double)((a.M + 15) / 16) * ((a.N + 15) / 16) * a.batch / c.sms);
  const double fp64 = 5 + 0.27 * a.K * ctas * std::min(16, (a.M + 1) / 2 * 2) / 16.0;
  const double mn = (double)a.M * a.N * a.batch, conv = ((double)p.rows.rows + 2.0 * p.cols.rows) * p.Kp * a.batch;
  return fp64 > 28.0 * ch.launches + 0.085 * a.K + 34e-6 * mn + 12e-6 * conv + 8.0 * kPlanes / 1.2e9 * mn * a.K;
}

cudaError_t rns_zgemm(const ZgemmArgs& a, int al, bool cj, int bl, const RnsCtx& c, cudaStream_t s, int* launches) {
  const ZPlan p = zplan(a, al, cj, bl);
  ZChunks ch;
  if (!zchunks(p, a.batch, c.bytes, &ch)) return cudaErrorInvalidValue;  // (rns_takes_zgemm tells first)
  const int nb = ch.nb, nr = ch.nr;
  for (int b0 = 0; b0 < a.batch; b0 += nb) {
    const int n = std::min(nb, a.batch - b0);
    for (int r0 = 0; r0 < p.rows.rows; r0 += nr) {
      const int m = std::min(nr, p.rows.rows - r0);
      Carve w{(char*)c.scratch, (char*)c.scratch + c.bytes};
      const long long smA = (long long)n * m * p.Kp, smB = (long long)n * 2 * p.cols.rows * p.Kp;
      // (the column operand first: it stays in place over the row chunks of an entry)
      __nv_bfloat16* RB = (__nv_bfloat16*)w.take((size_t)smB * 2 * kPlanes);
      int* eb = (int*)w.take((size_t)n * p.cols.rows * 4);
      __nv_bfloat16* RA = (__nv_bfloat16*)w.take((size_t)smA * 2 * kPlanes);
      signed char* Y = (signed char*)w.take((size_t)n * pad_to(m, 32) * p.ldy * kPlanes);
      int* ea = (int*)w.take((size_t)n * m * 4);
      if (w.p > w.end) return cudaErrorInvalidValue;
      cudaError_t e = cudaSuccess;
      if (r0 == 0) e = convert(p.cols, 0, p.cols.rows, a.tab, a.tab0 + b0, p.K, p.Kp, n, b0, RB, smB, eb, c.sms, s);
      if (e != cudaSuccess) return e;
      e = convert(p.rows, r0, m, a.tab, a.tab0 + b0, p.K, p.Kp, n, b0, RA, smA, ea, c.sms, s);
      if (e != cudaSuccess) return e;
      CrtArgs x;
      std::memset(&x, 0, sizeof(x));
      x.rows = m;
      x.cols = 2 * p.cols.rows;
      x.row0 = r0;
      x.ea = ea;
      x.eb = eb;
      x.ea_rows = m;
      x.eb_rows = p.cols.rows;
      x.D = a.D + (a.tab ? 0 : (long long)b0 * a.sD);
      x.tab = a.tab;
      x.tab0 = a.tab0 + b0;
      x.sD = a.sD;
      x.r_div = p.rows_are_m ? a.dm_div : a.dn_div;
      x.r_hi = p.rows_are_m ? a.dm_hi : a.dn_hi;
      x.r_lo = p.rows_are_m ? a.dm_lo : a.dn_lo;
      x.c_div = p.rows_are_m ? a.dn_div : a.dm_div;
      x.c_hi = p.rows_are_m ? a.dn_hi : a.dm_hi;
      x.c_lo = p.rows_are_m ? a.dn_lo : a.dm_lo;
      x.alpha = a.alpha;
      x.scaled = a.alpha != 1.0;
      x.beta = a.beta;
      x.rside = fma_side(p.rows, r0, a.tab, b0);
      x.cside = fma_side(p.cols, 0, a.tab, b0);
      x.rows_are_m = p.rows_are_m;
      x.K = p.K;
      GemmArgs g;
      std::memset(&g, 0, sizeof(g));
      g.nbatch = n;
      g.rows = m;
      g.cols = x.cols;
      g.rt = (m + kTileM - 1) / kTileM;
      g.bn = tile_width(g.cols);
      g.ct = (g.cols + g.bn - 1) / g.bn;
      g.nkb = p.Kp / kBK;
      g.Y = Y;
      g.ymod = (long long)n * pad_to(m, 32) * p.ldy;
      g.ldy = p.ldy;
      if ((e = gemm(RA, smA, RB, smB, g, p.Kp, m, c, s)) != cudaSuccess) return e;
      x.Y = Y;
      x.ymod = g.ymod;
      x.ldy = p.ldy;
      const dim3 grid(crt_blocks(m, g.cols), n);
      rns_crt_kernel<true><<<grid, 256, 0, s>>>(x);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      *launches += r0 == 0 ? 4 : 3;
    }
  }
  return cudaSuccess;
}

bool rns_takes_dsyrk(const DsyrkArgs& a, const RnsCtx& c) {
  if (!c.scratch || a.M <= 0 || a.N <= 0 || a.K <= 0) return false;
  // 68 ns per k and 16 x 16 tile and SM on the FP64 pipe, against launches, conversions and results as above: a
  // 64 x 64 result, K = 256: 23 against 32 us, K = 1024: 75 against 50
  const double tm = (a.M + 15) / 16, tn = (a.N + 15) / 16, ctas = a.mode == 0 ? tm * (tm + 1) / 2 : tm * tn;
  const double fp64 = 5 + 0.068 * a.K * std::ceil(ctas / c.sms), mn = (a.mode == 0 ? 0.5 : 1.0) * a.M * (double)a.N;
  const double conv = ((double)a.M + (a.mode ? a.N : 0)) * a.K;
  if (fp64 < 26 + (a.mode ? 8 : 0) + 0.024 * a.K + 17e-6 * mn + 12e-6 * conv + 2.0 * kPlanes / 1.2e9 * mn * a.K)
    return false;
  // at least one K block of both operands and 256 rows of Y
  const size_t ops = ((size_t)a.M + (a.mode ? a.N : 0)) * kBK * 2 * kPlanes, y = (size_t)256 * pad_to(a.N, 16) * kPlanes;
  return ops + y + ((size_t)a.M + a.N) * 4 + (1 << 20) <= c.bytes;
}

cudaError_t rns_dsyrk(const DsyrkArgs& a, const RnsCtx& c, cudaStream_t s, int* launches) {
  const bool tri = a.mode == 0;
  const int N = a.N, M = a.M;
  const long long ldy = pad_to(N, 16);
  const size_t opsrow = (size_t)M + (tri ? 0 : N), exps = ((size_t)M + N) * 4 + 16384;
  const size_t avail = c.bytes - exps;
  // K in chunks whose residues take at most half of the scratch (or what the smallest row chunk
  // leaves), rows of the result in chunks of what is left; every chunk adds into the output
  const size_t ymin = (size_t)256 * ldy * kPlanes;
  const size_t opmax = std::max(avail / 2, opsrow * kBK * 2 * kPlanes);
  long long Kc = std::min<long long>(pad_to(a.K, kBK), (long long)(std::min(opmax, avail - ymin) / (opsrow * 2 * kPlanes)) / kBK * kBK);
  const size_t yav = avail - opsrow * Kc * 2 * kPlanes;
  const int nr = (int)std::min<size_t>((size_t)pad_to(M, 256), yav / ((size_t)ldy * kPlanes) / 256 * 256);
  if (Kc < kBK || nr < 256) return cudaErrorInvalidValue;
  const Side X{SRC_REAL, a.X, 0, 0, 1, a.ldx, M, 0}, Yo{SRC_REAL, a.Y, 0, 0, 1, a.ldy, N, 0};
  for (long long k0 = 0; k0 < a.K; k0 += Kc) {
    const int K = (int)std::min<long long>(Kc, a.K - k0), Kp = (int)pad_to(K, kBK);
    Carve w{(char*)c.scratch, (char*)c.scratch + c.bytes};
    const long long smA = (long long)M * Kp, smB = (long long)N * Kp;
    __nv_bfloat16* RA = (__nv_bfloat16*)w.take((size_t)smA * 2 * kPlanes);
    __nv_bfloat16* RB = tri ? RA : (__nv_bfloat16*)w.take((size_t)smB * 2 * kPlanes);
    int* ea = (int*)w.take((size_t)M * 4);
    int* eb = tri ? ea : (int*)w.take((size_t)N * 4);
    signed char* Y = (signed char*)w.take((size_t)std::min<long long>(nr, pad_to(M, 32)) * ldy * kPlanes);
    if (w.p > w.end) return cudaErrorInvalidValue;
    Side xs = X, ys = Yo;
    xs.base += k0 * a.ldx;
    ys.base += k0 * a.ldy;
    cudaError_t e = convert(xs, 0, M, nullptr, 0, K, Kp, 1, 0, RA, smA, ea, c.sms, s);
    if (e != cudaSuccess) return e;
    if (!tri) {
      e = convert(ys, 0, N, nullptr, 0, K, Kp, 1, 0, RB, smB, eb, c.sms, s);
      if (e != cudaSuccess) return e;
    }
    *launches += tri ? 1 : 2;
    for (int r0 = 0; r0 < M; r0 += nr) {
      const int m = std::min(nr, M - r0);
      GemmArgs g;
      std::memset(&g, 0, sizeof(g));
      g.nbatch = 1;
      g.rows = m;
      g.cols = N;
      g.rt = (m + kTileM - 1) / kTileM;
      g.tri = tri;
      g.h0 = r0 / 256;
      g.row0 = r0;
      g.bn = tri ? 256 : tile_width(N);
      g.ct = (N + g.bn - 1) / g.bn;
      g.nkb = Kp / kBK;
      g.Y = Y;
      g.ymod = pad_to(m, 32) * ldy;
      g.ldy = (int)ldy;
      e = gemm(RA, smA, RB, smB, g, Kp, M, c, s);
      if (e != cudaSuccess) return e;
      CrtArgs x;
      std::memset(&x, 0, sizeof(x));
      x.Y = Y;
      x.ymod = g.ymod;
      x.ldy = (int)ldy;
      x.rows = m;
      x.cols = N;
      x.row0 = r0;
      x.ea = ea + r0;
      x.eb = eb;
      x.out = a.out;
      x.ldo = a.ldo;
      x.tri = tri;
      x.alpha = a.alpha;
      x.rside = fma_side(xs, r0, nullptr, 0);
      x.cside = fma_side(tri ? xs : ys, 0, nullptr, 0);
      x.K = K;
      const dim3 grid(crt_blocks(m, N), 1);
      rns_crt_kernel<false><<<grid, 256, 0, s>>>(x);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      *launches += 2;
    }
  }
  return cudaSuccess;
}

}  // namespace dmet

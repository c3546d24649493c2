// FP64 kernels of the embedded-ERI transformation (Algorithm 1, section 2.1).
//
// GB300 executes FP64 fused multiply-adds on the CUDA cores at a small fraction of its
// FP32 rate, so the plain-FP64 path is bound by the DFMA pipe, not by memory: every
// kernel here keeps its operands in shared memory and registers and spends its issue
// slots on DFMAs. (The large products run on the tensor cores instead: rns.cu.)

#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include "internal.h"

namespace dmet {

namespace {

constexpr int TT = 16;  // tile rows and columns
constexpr int TK = 16;  // complex k-step
constexpr int DK = 64;  // real k-step

__device__ __forceinline__ long long map2(int x, int div, long long hi, long long lo) {
  return (long long)(x / div) * hi + (long long)(x % div) * lo;
}

// The FP64 pipe takes 16 clocks of an SM per warp FMA, so a tile's loads and shared-memory reads hide behind it at
// any tile size and the split of the work decides: 16 x 16 tiles, one output per thread, spread a small product
// over all SMs (16 x 640 x 16 in four batches: 39 us with 64 x 64 tiles of 4 x 4 outputs per thread, 13 so; 64 x 256 x
// 1024: 4134 and 283 us; 104 x 5720 x 26 in 20 batches, which fills the GPU either way: 2604 and 2124 us, less waste on
// ragged edges; 104 x 22 880 x 520 in four: 33.1 and 33.8 ms); the next K step's values load while the current one is summed.
template <int AL, bool CJ, int BL>
__global__ void __launch_bounds__(256) zgemm_fp64_kernel(const ZgemmArgs d) {
  __shared__ __align__(16) double2 As[2][TK][TT + 1];
  __shared__ __align__(16) double2 Bs[2][TK][TT + 1];
  const int tid = threadIdx.x, tx = tid & (TT - 1), ty = tid / TT;
  const unsigned nt = (unsigned)(d.N + TT - 1) / TT;
  const int m0 = (int)(blockIdx.x / nt) * TT, n0 = (int)(blockIdx.x % nt) * TT;
  if (d.lower && n0 >= m0 + TT) return;  // the whole CTA leaves together
  const double2* A = d.A;
  const double2* B = d.B;
  double2* D = d.D;
  int K = d.K;
  if (d.tab) {
    const int4 e = d.tab[d.tab0 + blockIdx.z];
    A += e.x * d.sA;
    B += e.y * d.sB;
    D += e.z * d.sD;
    K = e.w;
  } else {
    A += (long long)blockIdx.z * d.sA;
    B += (long long)blockIdx.z * d.sB;
    D += (long long)blockIdx.z * d.sD;
  }
  // thread (ty, tx) loads element (k = ty, m = tx) of a K-major operand, (k = tx, m = ty) of the other kind
  const int ak = AL == A_KM ? ty : tx, am = AL == A_KM ? tx : ty, bk = BL == B_KN ? ty : tx, bn = BL == B_KN ? tx : ty;
  const bool aok = m0 + am < d.M, bok = n0 + bn < d.N;
  const double2* Ap = A + (AL == A_KM ? ak * d.lda + m0 + am : (m0 + am) * d.lda + ak);
  const double2* Bp = B + (BL == B_KN ? bk * d.ldb + n0 + bn : (n0 + bn) * d.ldb + bk);
  const long long as = AL == A_KM ? TK * d.lda : TK, bs = BL == B_KN ? TK * d.ldb : TK;
  const double2 zero = make_double2(0.0, 0.0);
  double2 av = aok && ak < K ? *Ap : zero, bv = bok && bk < K ? *Bp : zero;
  const bool active = m0 + (tid >> 5) * (32 / TT) < d.M;
  double re = 0.0, im = 0.0;
  for (int k0 = 0, buf = 0; k0 < K; k0 += TK, buf ^= 1) {
    if (CJ) av.y = -av.y;
    As[buf][ak][am] = av;
    Bs[buf][bk][bn] = bv;
    __syncthreads();
    Ap += as;
    Bp += bs;
    av = aok && k0 + TK + ak < K ? *Ap : zero;
    bv = bok && k0 + TK + bk < K ? *Bp : zero;
    if (active) {
      const int kn = min(TK, K - k0);
#pragma unroll 8
      for (int kk = 0; kk < kn; ++kk) {
        const double2 a = As[buf][kk][ty], b = Bs[buf][kk][tx];
        re = fma(a.x, b.x, re);
        im = fma(a.x, b.y, im);
        re = fma(-a.y, b.y, re);
        im = fma(a.y, b.x, im);
      }
    }
  }
  const int m = m0 + ty, n = n0 + tx;
  if (m >= d.M || n >= d.N) return;
  const long long addr = map2(m, d.dm_div, d.dm_hi, d.dm_lo) + map2(n, d.dn_div, d.dn_hi, d.dn_lo);
  double2 v = make_double2(d.alpha * re, d.alpha * im);
  if (d.beta) {
    const double2 o = D[addr];
    v.x += o.x;
    v.y += o.y;
  }
  D[addr] = v;
}

__global__ void __launch_bounds__(256) dsyrk_fp64_kernel(const DsyrkArgs d) {
  __shared__ double Xs[2][DK][TT + 1];
  __shared__ double Ys[2][DK][TT + 1];
  const int tid = threadIdx.x, tx = tid & (TT - 1), ty = tid / TT;
  int m0, n0;
  if (d.mode == 0) {
    const long long t = blockIdx.x;
    long long ti = (long long)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);  // (made exact below)
    while (ti * (ti + 1) / 2 > t) --ti;
    while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
    m0 = (int)ti * TT;
    n0 = (int)(t - ti * (ti + 1) / 2) * TT;
  } else {
    const unsigned nt = (unsigned)(d.N + TT - 1) / TT;
    m0 = (int)(blockIdx.x / nt) * TT;
    n0 = (int)(blockIdx.x % nt) * TT;
  }
  const double* Y = d.mode == 0 ? d.X : d.Y;
  const long long ldy = d.mode == 0 ? d.ldx : d.ldy;
  const bool xok = m0 + tx < d.M, yok = n0 + tx < d.N;
  const double* Xp = d.X + ty * d.ldx + m0 + tx;
  const double* Yp = Y + ty * ldy + n0 + tx;
  constexpr int R = DK / TT;
  double xv[R], yv[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int k = ty + r * TT;
    xv[r] = xok && k < d.K ? Xp[r * TT * d.ldx] : 0.0;
    yv[r] = yok && k < d.K ? Yp[r * TT * ldy] : 0.0;
  }
  double acc = 0.0;
  for (int k0 = 0, buf = 0; k0 < d.K; k0 += DK, buf ^= 1) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      Xs[buf][ty + r * TT][tx] = xv[r];
      Ys[buf][ty + r * TT][tx] = yv[r];
    }
    __syncthreads();
    Xp += DK * d.ldx;
    Yp += DK * ldy;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int k = k0 + DK + ty + r * TT;
      xv[r] = xok && k < d.K ? Xp[r * TT * d.ldx] : 0.0;
      yv[r] = yok && k < d.K ? Yp[r * TT * ldy] : 0.0;
    }
    const int kn = min(DK, d.K - k0);
#pragma unroll 16
    for (int kk = 0; kk < kn; ++kk) acc = fma(Xs[buf][kk][ty], Ys[buf][kk][tx], acc);
  }
  const int m = m0 + ty, n = n0 + tx;
  if (m >= d.M || n >= d.N || (d.mode == 0 && n > m)) return;
  d.out[d.mode == 0 ? (long long)m * (m + 1) / 2 + n : (long long)m * d.ldo + n] += d.alpha * acc;
}

__global__ void gather_orbitals_kernel(const double2* __restrict__ C, double2* __restrict__ Crep,
                                       const int4* __restrict__ tab, int tab0, int nao, int n) {
  const int e = blockIdx.y;
  const int4 t = tab[tab0 + e];
  const double w = t.y ? 0.5 : 1.0;
  const long long sz = (long long)nao * n;
  const double2* src = C + t.x * sz;
  double2* dst = Crep + e * sz;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < sz;
       x += (long long)gridDim.x * blockDim.x) {
    const double2 v = src[x];
    dst[x] = make_double2(w * v.x, w * v.y);
  }
}

// Z + Z^T of every (q, P) matrix, one CTA per 32 x 32 tile of its lower triangle: the tile and its mirror are read along
// their rows and met in shared memory (reading the mirror down its columns, and a pair's (i, j) from a square root,
// took 576 us for 1760 matrices of 104 x 104; this 114).
constexpr int kSymTile = 32;
struct SymTile {
  int i0, j0;
};
__device__ __forceinline__ SymTile sym_tile(int t) {
  int r = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while (r * (r + 1) / 2 > t) --r;
  while ((r + 1) * (r + 2) / 2 <= t) ++r;
  return {r * kSymTile, (t - r * (r + 1) / 2) * kSymTile};
}
__device__ __forceinline__ void load_sym_tile(const double2* z, int n, SymTile t, double2 (&m)[kSymTile][kSymTile + 1]) {
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
#pragma unroll
  for (int r = y; r < kSymTile; r += 8)
    if (t.j0 + r < n && t.i0 + x < n) m[r][x] = z[(long long)(t.j0 + r) * n + t.i0 + x];  // rows j of the mirror
  __syncthreads();
}

// X[(q, P, c)][pair ij] = s (Re or Im of Z_ij + Z_ji)
__global__ void __launch_bounds__(256) pack_pairs_kernel(const double2* __restrict__ Z, double* __restrict__ X, int n,
                                                         int nc, double s) {
  __shared__ double2 m[kSymTile][kSymTile + 1];
  const SymTile t = sym_tile(blockIdx.y + blockIdx.z * gridDim.y);
  if (t.i0 >= n) return;
  const double2* z = Z + (long long)blockIdx.x * n * n;
  load_sym_tile(z, n, t, m);
  const long long npair = (long long)n * (n + 1) / 2;
  double* out = X + (long long)blockIdx.x * nc * npair;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5, j = t.j0 + x;
#pragma unroll
  for (int r = y; r < kSymTile; r += 8) {
    const int i = t.i0 + r;
    if (i >= n || j > i) continue;
    const double2 a = z[(long long)i * n + j], b = m[x][r];
    const long long ij = (long long)i * (i + 1) / 2 + j;
    out[ij] = s * (a.x + b.x);
    if (nc == 2) out[npair + ij] = s * (a.y + b.y);
  }
}

// Lq = (s Re, sim Im) of Z + Z^T
__global__ void __launch_bounds__(256) symmetrize_kernel(const double2* __restrict__ Z, double2* __restrict__ Lq, int n,
                                                         double s, double sim) {
  __shared__ double2 m[kSymTile][kSymTile + 1];
  const SymTile t = sym_tile(blockIdx.y + blockIdx.z * gridDim.y);
  if (t.i0 >= n) return;
  const double2* z = Z + (long long)blockIdx.x * n * n;
  double2* out = Lq + (long long)blockIdx.x * n * n;
  load_sym_tile(z, n, t, m);
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5, j = t.j0 + x;
  double2 v[kSymTile / 8];
#pragma unroll
  for (int h = 0; h < kSymTile / 8; ++h) {
    const int r = y + 8 * h, i = t.i0 + r;
    if (i >= n || j >= n) continue;
    const double2 a = z[(long long)i * n + j], b = m[x][r];
    v[h] = make_double2(s * (a.x + b.x), sim * (a.y + b.y));
    out[(long long)i * n + j] = v[h];
  }
  if (t.i0 == t.j0) return;  // (a diagonal tile is its own mirror)
  __syncthreads();
#pragma unroll
  for (int h = 0; h < kSymTile / 8; ++h) m[x][y + 8 * h] = v[h];
  __syncthreads();
#pragma unroll
  for (int r = y; r < kSymTile; r += 8)
    if (t.j0 + r < n && t.i0 + x < n) out[(long long)(t.j0 + r) * n + t.i0 + x] = m[r][x];
}

// Max of non-negative doubles through their bit patterns (NaN compares above +inf).
__device__ __forceinline__ double wmax(double a, double b) { return (isnan(a) || a > b) ? a : b; }

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = wmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ void atomic_max_nonneg(double* p, double v) {
  atomicMax(reinterpret_cast<unsigned long long*>(p), (unsigned long long)__double_as_longlong(v));
}

__device__ __forceinline__ void block_max_commit(double v, double* out) {
  __shared__ double red[32];
  v = warp_max(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (w == 0) {
    v = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0;
    v = warp_max(v);
    if (lane == 0) atomic_max_nonneg(out, v);
  }
  __syncthreads();
}

// S = s * sum_g S_g (ng split-K partial products of C^+ C); stat = max |S_ij - delta_ij| over
// the lower triangle j <= i (S is Hermitian, and only those tiles of S_g are computed). Eight threads share the
// partials of an element.
__global__ void __launch_bounds__(256) orth_reduce_kernel(const double2* __restrict__ Sg, int ng, int n, double s,
                                                          double* stat) {
  __shared__ double2 sh[8][33];
  const int e = threadIdx.x & 31, gl = threadIdx.x >> 5;
  double v = 0.0;
  const long long nn = (long long)n * n;
  for (long long x0 = blockIdx.x * 32ll; x0 < nn; x0 += gridDim.x * 32ll) {
    const long long x = x0 + e;
    const int i = (int)(x / n), j = (int)(x - (long long)i * n);
    const bool ok = x < nn && j <= i;
    double2 a = make_double2(0.0, 0.0);
    if (ok)
      for (int g = gl; g < ng; g += 8) {
        const double2 b = Sg[g * nn + x];
        a.x += b.x;
        a.y += b.y;
      }
    sh[gl][e] = a;
    __syncthreads();
    if (gl == 0 && ok) {
      for (int g = 1; g < 8; ++g) {
        a.x += sh[g][e].x;
        a.y += sh[g][e].y;
      }
      const double re = s * a.x - (i == j ? 1.0 : 0.0), im = s * a.y;
      v = wmax(v, sqrt(re * re + im * im));
    }
    __syncthreads();
  }
  block_max_commit(v, stat);
}

__global__ void c_real_check_kernel(const double2* __restrict__ C, const int* __restrict__ neg, int nk,
                                    int nao, int n, double* stats) {
  double dv = 0.0, mv = 0.0;
  const long long per = (long long)nao * n, total = per * nk;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total;
       x += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(x / per);
    const double2 a = C[x], b = C[neg[k] * per + x % per];
    const double dr = b.x - a.x, di = b.y + a.y;
    dv = wmax(dv, dr * dr + di * di);
    mv = wmax(mv, a.x * a.x + a.y * a.y);
  }
  // (the square root, once: it keeps the order, rounded)
  block_max_commit(sqrt(dv), stats + 1);
  block_max_commit(sqrt(mv), stats + 2);
}

// |x| of a double as its bit pattern with the sign cleared: for non-negative doubles the
// integer order is the numeric order (NaN patterns sort above +inf).
__device__ __forceinline__ unsigned long long abits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

__device__ __forceinline__ unsigned long long warp_umax(unsigned long long v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  return v;
}

// Symmetries of L over a chunk of aux indices of one k pair (k1, k2): Hermiticity against
// L[k2][k1][P][nu][mu] (checked once per unordered pair, k1 <= k2) and time reversal against
// L[-k1][-k2][P][mu][nu] (checked once per pair of pairs). The transposed partner is read
// through the read-only cache, where the block's other warps have brought its lines.
// Records max-norm differences (component-wise) and max |L| (component-wise) as bit patterns.
constexpr int LCHK_P = 8;
__global__ void __launch_bounds__(256) l_check_kernel(const double2* __restrict__ L, const int* __restrict__ neg,
                                                      int nk, int naux, int nao, double* stats) {
  const int pchunks = (naux + LCHK_P - 1) / LCHK_P;
  const long long nwork = (long long)nk * nk * pchunks;
  unsigned long long hv = 0, tv = 0, mv = 0;
  for (long long w = blockIdx.x; w < nwork; w += gridDim.x) {
    const long long kk = w / pchunks;
    const int P0 = (int)(w % pchunks) * LCHK_P;
    const int k1 = (int)(kk / nk), k2 = (int)(kk % nk);
    const long long kt = (long long)neg[k1] * nk + neg[k2];
    const bool do_h = k1 <= k2, do_t = kk <= kt;
    const long long blk = (long long)nao * nao, pair = blk * naux;
    const double2* a_pair = L + kk * pair;
    const double2* h_pair = L + ((long long)k2 * nk + k1) * pair;
    const double2* t_pair = L + kt * pair;
    const int pend = min(naux, P0 + LCHK_P);
    for (int P = P0; P < pend; ++P) {
      const long long base = (long long)P * blk;
      for (long long e = threadIdx.x; e < blk; e += blockDim.x) {
        const double2 a = a_pair[base + e];
        mv = max(mv, max(abits(a.x), abits(a.y)));
        if (do_h) {
          const int mu = (int)(e / nao), nu = (int)(e % nao);
          const double2 h = __ldg(h_pair + base + (long long)nu * nao + mu);
          hv = max(hv, max(abits(h.x - a.x), abits(h.y + a.y)));
        }
        if (do_t) {
          const double2 t = t_pair[base + e];
          tv = max(tv, max(abits(t.x - a.x), abits(t.y + a.y)));
        }
      }
    }
  }
  hv = warp_umax(hv);
  tv = warp_umax(tv);
  mv = warp_umax(mv);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(reinterpret_cast<unsigned long long*>(stats + 3), hv);
    atomicMax(reinterpret_cast<unsigned long long*>(stats + 4), tv);
    atomicMax(reinterpret_cast<unsigned long long*>(stats + 5), mv);
  }
}

inline int grid_for(long long total, int threads, int cap) {
  long long g = (total + threads - 1) / threads;
  if (g < 1) g = 1;
  return (int)(g < cap ? g : cap);
}

// Largest t with t(t+1)/2 <= x (the row of a lower-triangle index), exact for x < 2^50. (An FP32 square root where it
// comes near enough: the FP64 one takes some 40 instructions of the slow pipe.)
__device__ __forceinline__ long long tri_row(long long x) {
  long long t = x < (1 << 28) ? (long long)((sqrtf(8.f * (float)x + 1.f) - 1.f) * 0.5f)
                              : (long long)((sqrt(8.0 * (double)x + 1.0) - 1.0) * 0.5);
  while (t * (t + 1) / 2 > x) --t;
  while ((t + 1) * (t + 2) / 2 <= x) ++t;
  return t;
}

// out[pos] = full[i][j][k][l] for the (i, j, k, l) that packed position pos stands for.
__global__ void pack_s4_kernel(const double2* __restrict__ full, int na, int nb, int rect, double2* __restrict__ out) {
  const long long np = (long long)na * (na + 1) / 2, ns = (long long)na * (na - 1) / 2;
  const long long nA = np * (np + 1) / 2;
  const long long total = rect ? np * nb * nb : nA + ns * (ns + 1) / 2;
  const long long nb2 = (long long)nb * nb;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total;
       x += (long long)gridDim.x * blockDim.x) {
    long long i, j, k, l;
    if (rect) {
      const long long I = x / nb2, kl = x % nb2;
      i = tri_row(I);
      j = I - i * (i + 1) / 2;
      k = kl / nb;
      l = kl % nb;
    } else if (x < nA) {
      const long long I = tri_row(x), K = x - I * (I + 1) / 2;
      i = tri_row(I);
      j = I - i * (i + 1) / 2;
      k = tri_row(K);
      l = K - k * (k + 1) / 2;
    } else {
      // a = i(i-1)/2 + j with i > j, b = l(l-1)/2 + k with l > k
      const long long y = x - nA, a = tri_row(y), b = y - a * (a + 1) / 2;
      i = tri_row(a) + 1;
      j = a - i * (i - 1) / 2;
      l = tri_row(b) + 1;
      k = b - l * (l - 1) / 2;
    }
    out[x] = full[((i * na + j) * nb + k) * nb + l];
  }
}

}  // namespace

cudaError_t launch_zgemm(const ZgemmArgs& a, int a_layout, bool conj_a, int b_layout, cudaStream_t s) {
  if (a.M <= 0 || a.N <= 0 || a.batch <= 0) return cudaSuccess;
  const long long tiles = (long long)((a.N + TT - 1) / TT) * ((a.M + TT - 1) / TT);
  if (tiles > INT_MAX) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)tiles, 1, a.batch);
  if (a_layout == A_KM && conj_a && b_layout == B_KN)
    zgemm_fp64_kernel<A_KM, true, B_KN><<<grid, 256, 0, s>>>(a);
  else if (a_layout == A_KM && !conj_a && b_layout == B_KN)
    zgemm_fp64_kernel<A_KM, false, B_KN><<<grid, 256, 0, s>>>(a);
  else if (a_layout == A_KM && !conj_a && b_layout == B_NK)
    zgemm_fp64_kernel<A_KM, false, B_NK><<<grid, 256, 0, s>>>(a);
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_dsyrk(const DsyrkArgs& a, cudaStream_t s) {
  if (a.M <= 0 || a.N <= 0) return cudaSuccess;
  const long long mt = (a.M + TT - 1) / TT, nt = (a.N + TT - 1) / TT, tiles = a.mode == 0 ? mt * (mt + 1) / 2 : mt * nt;
  if (tiles > INT_MAX) return cudaErrorInvalidValue;
  dsyrk_fp64_kernel<<<(unsigned)tiles, 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_gather_orbitals(const double2* C, double2* Crep, const int4* tab, int tab0, int n_entries,
                                   int nao, int n, cudaStream_t s) {
  if (n_entries <= 0) return cudaSuccess;
  const dim3 grid(grid_for((long long)nao * n, 256, 64), n_entries, 1);
  gather_orbitals_kernel<<<grid, 256, 0, s>>>(C, Crep, tab, tab0, nao, n);
  return cudaGetLastError();
}

namespace {
// one CTA per (matrix, lower-triangle tile), the tiles over y and z
dim3 sym_grid(long long matrices, int n) {
  const long long t = (n + kSymTile - 1) / kSymTile, tiles = t * (t + 1) / 2, y = tiles < 32768 ? tiles : 32768;
  return dim3((unsigned)matrices, (unsigned)y, (unsigned)((tiles + y - 1) / y));
}
}  // namespace

cudaError_t launch_pack_pairs(const double2* Z, double* X, int nq, int naux, int n, int nc, double sc,
                              cudaStream_t s) {
  pack_pairs_kernel<<<sym_grid((long long)nq * naux, n), 256, 0, s>>>(Z, X, n, nc, sc);
  return cudaGetLastError();
}

cudaError_t launch_symmetrize(const double2* Z, double2* Lq, int nq, int naux, int n, double sc, int conj,
                              cudaStream_t s) {
  symmetrize_kernel<<<sym_grid((long long)nq * naux, n), 256, 0, s>>>(Z, Lq, n, sc, conj ? -sc : sc);
  return cudaGetLastError();
}

cudaError_t launch_orth_reduce(const double2* Sg, int ng, int n, double sc, double* stat, cudaStream_t s) {
  orth_reduce_kernel<<<grid_for((long long)n * n, 32, 152 * 8), 256, 0, s>>>(Sg, ng, n, sc, stat);
  return cudaGetLastError();
}

cudaError_t launch_c_real_check(const double2* C, const int* neg, int nk, int nao, int n, double* stats,
                                cudaStream_t s) {
  c_real_check_kernel<<<grid_for((long long)nk * nao * n, 256, 152 * 4), 256, 0, s>>>(C, neg, nk, nao, n,
                                                                                        stats);
  return cudaGetLastError();
}

cudaError_t launch_l_check(const double2* L, const int* neg, int nk, int naux, int nao, double* stats,
                           cudaStream_t s) {
  const long long pchunks = (naux + LCHK_P - 1) / LCHK_P;
  const long long nwork = (long long)nk * nk * pchunks;
  l_check_kernel<<<(unsigned)(nwork < (1LL << 30) ? nwork : (1LL << 30)), 256, 0, s>>>(L, neg, nk, naux, nao, stats);
  return cudaGetLastError();
}

cudaError_t launch_pack_s4(const double2* full, int na, int nb, int rect, double2* out, cudaStream_t st) {
  const long long np = (long long)na * (na + 1) / 2, ns = (long long)na * (na - 1) / 2;
  const long long total = rect ? np * nb * nb : np * (np + 1) / 2 + ns * (ns + 1) / 2;
  pack_s4_kernel<<<grid_for(total, 256, 152 * 16), 256, 0, st>>>(full, na, nb, rect, out);
  return cudaGetLastError();
}

}  // namespace dmet

// The embedding one-particle Hamiltonian (section 2.1): the reduction of the transformed Fock
// matrices over k (Eq. "fock transform") and the Coulomb / exchange double counting evaluated
// with the 8-fold packed embedding ERIs (Eq. "fock double counting"). FP64 throughout.

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "internal.h"

namespace dmet {

namespace {

// F0[i][j] = s * sum_k Re G[k][i][j], G[k] = C^{k+} F^k C^k.
__global__ void fock_reduce_kernel(const double2* __restrict__ G, int nk, int n, double s, double* __restrict__ F0) {
  const int nn = n * n;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < nn; x += gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int k = 0; k < nk; ++k) v += G[(long long)k * nn + x].x;
    F0[x] = s * v;
  }
}

// The FP64 pipe bounds both sums over the packed ERI (an FMA of a warp takes 16 clocks of an SM), so each stored
// element is used along its row together with its electron-exchange mirror: K = K' + K'^T, where K' takes
// the elements (A, B) with B < A and half of A = B, A = {i, k} giving the index of K' and B = {l, j} the other;
// and J_A = sum_{B <= A} V_AB w_B along the rows, plus sum_{A' > A} V_A'A w_A' down the columns, w_B = gamma_B (2 -
// delta_B). n = 104, staging whole rows (their second halves read down the columns): 562 us for both; so 250 for the rows and 71 for the columns.

__global__ void pair_weights_kernel(const double* __restrict__ gamma, int n, double* __restrict__ w) {
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n * n; x += gridDim.x * blockDim.x) {
    const int l = x / n, j = x - l * n;
    if (j <= l) w[l * (l + 1) / 2 + j] = (l == j ? 1.0 : 2.0) * gamma[x];
  }
}

// part[y][B] = sum of V_AB w_A over share y of the rows A > B: a thread per column, rows in order (a warp reads 256
// contiguous bytes of each), four running sums.
constexpr int kColShares = 16;
__global__ void __launch_bounds__(256) coulomb_columns_kernel(const double* __restrict__ eri, const double* __restrict__ w,
                                                              int npair, double* __restrict__ part) {
  const int B = blockIdx.x * 256 + threadIdx.x, first = blockIdx.x * 256 + 1, span = npair - first;
  const int a0 = first + (int)((long long)span * blockIdx.y / kColShares);
  const int a1 = first + (int)((long long)span * (blockIdx.y + 1) / kColShares);
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  const double* p = eri + (long long)a0 * (a0 + 1) / 2 + B;
  int A = a0;
  for (; A + 4 <= a1; A += 4) {
    double v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      v[r] = B < A + r ? *p : 0.0;
      p += A + r + 1;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) s[r] = fma(v[r], w[A + r], s[r]);
  }
  for (; A < a1; ++A) {
    if (B < A) s[0] = fma(*p, w[A], s[0]);
    p += A + 1;
  }
  if (B < npair) part[(long long)blockIdx.y * npair + B] = (s[0] + s[1]) + (s[2] + s[3]);
}

// One CTA per pair row A = {i, k}, i >= k, long rows first: the row's elements B <= A in shared memory (the last one
// halved, the rest of the pairs {i, j} zero), then thread (h, j), j <= i, over its share h of l <= i:
//   K'_ij += sum_l (ik|lj) gamma_kl   and, for i != k,   K'_kj += sum_l (ki|lj) gamma_il,
// and the row's share of J_A. The rows' sums meet in eight copies of K' (a long chain of additions into one
// rounds sqrt(8) times as much).
constexpr int kExchangeCopies = 8;
__global__ void __launch_bounds__(256) exchange_kernel(const double* __restrict__ eri, const double* __restrict__ gamma,
                                                       const double* __restrict__ w, int n, double* __restrict__ J,
                                                       double* __restrict__ K) {
  extern __shared__ double sm[];
  __shared__ double red[8];
  const int npair = n * (n + 1) / 2, A = npair - 1 - (int)blockIdx.x;
  int i = (int)((sqrtf(8.f * (float)A + 1.f) - 1.f) * 0.5f);
  while (i * (i + 1) / 2 > A) --i;
  while ((i + 1) * (i + 2) / 2 <= A) ++i;
  const int k = A - i * (i + 1) / 2, m = i + 1, len = m * (m + 1) / 2;
  double* row = sm;
  double* gi = sm + len;
  double* gk = gi + m;
  const double* src = eri + (long long)A * (A + 1) / 2;
  double js = 0.0;
  for (int B = threadIdx.x; B < len; B += 256) {
    const double v = B <= A ? src[B] : 0.0;
    row[B] = B == A ? 0.5 * v : v;
    if (B <= A) js = fma(v, w[B], js);
  }
  for (int t = threadIdx.x; t < m; t += 256) {
    gi[t] = gamma[i * n + t];
    gk[t] = gamma[k * n + t];
  }
  __syncthreads();
  const int nsplit = m < 256 ? 256 / m : 1;
  double* Kc = K + (long long)(A % kExchangeCopies) * n * n;
  for (int t = threadIdx.x; t < nsplit * m; t += 256) {
    const int h = t / m, j = t - h * m;
    const int l0 = h * m / nsplit, l1 = (h + 1) * m / nsplit, lm = min(max(j, l0), l1);
    double si = 0.0, sk = 0.0;
    const double* p = row + j * (j + 1) / 2;
#pragma unroll 4
    for (int l = l0; l < lm; ++l) {
      si = fma(p[l], gk[l], si);
      sk = fma(p[l], gi[l], sk);
    }
    const double* q = row + lm * (lm + 1) / 2 + j;
#pragma unroll 4
    for (int l = lm; l < l1; ++l) {
      si = fma(*q, gk[l], si);
      sk = fma(*q, gi[l], sk);
      q += l + 1;
    }
    atomicAdd(&Kc[i * n + j], si);
    if (i != k) atomicAdd(&Kc[k * n + j], sk);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) js += __shfl_xor_sync(0xffffffffu, js, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = js;
  __syncthreads();
  if (threadIdx.x == 0)
    J[A] = ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
}

// out = F0 - (J - K / 2), J = the rows' shares plus the columns', K = sum of the copies of K' + K'^T
__global__ void fock_combine_kernel(const double* __restrict__ F0, const double* __restrict__ J,
                                    const double* __restrict__ part, const double* __restrict__ K, int n,
                                    double* __restrict__ out) {
  const int npair = n * (n + 1) / 2;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n * n; x += gridDim.x * blockDim.x) {
    const int a = x / n, b = x - a * n, i = max(a, b), j = min(a, b), B = i * (i + 1) / 2 + j;
    double c[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int y = 0; y < kColShares; ++y) c[y & 3] += part[(long long)y * npair + B];
    double e[kExchangeCopies];
#pragma unroll
    for (int h = 0; h < kExchangeCopies; ++h) e[h] = K[h * n * n + x] + K[h * n * n + b * n + a];
    const double ex = ((e[0] + e[1]) + (e[2] + e[3])) + ((e[4] + e[5]) + (e[6] + e[7]));
    out[x] = F0[x] - ((J[B] + ((c[0] + c[1]) + (c[2] + c[3]))) - 0.5 * ex);
  }
}

inline int blocks_for(long long total, int threads, int cap) {
  long long b = (total + threads - 1) / threads;
  return (int)(b < 1 ? 1 : (b < cap ? b : cap));
}

// v[z] = tr(L^{-q}_P gamma) = sum_{k,l} Lm[z][k][l] gamma[l][k] for the batch entries z = (q, P) of a
// chunk: Lm[z] = Lq[tab[z].y] (the -q factor). One block per z.
__global__ void __launch_bounds__(256) jk_trace_kernel(const double2* __restrict__ Lq, const int4* __restrict__ tab,
                                                       int n, const double2* __restrict__ gamma, double2* __restrict__ v) {
  const long long nn = (long long)n * n;
  const double2* m = Lq + (long long)tab[blockIdx.x].y * nn;
  double re = 0.0, im = 0.0;
  for (long long x = threadIdx.x; x < nn; x += blockDim.x) {
    const int k = (int)(x / n), l = (int)(x % n);
    const double2 a = m[x], g = gamma[(long long)l * n + k];
    re = fma(a.x, g.x, fma(-a.y, g.y, re));
    im = fma(a.x, g.y, fma(a.y, g.x, im));
  }
  __shared__ double sr[8], si[8];
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, o);
    im += __shfl_xor_sync(0xffffffffu, im, o);
  }
  if ((threadIdx.x & 31) == 0) {
    sr[threadIdx.x >> 5] = re;
    si[threadIdx.x >> 5] = im;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += sr[w];
      b += si[w];
    }
    v[blockIdx.x] = make_double2(a, b);
  }
}

// gt[k][l] = gamma[l][k]
__global__ void transpose_kernel(const double2* __restrict__ g, int n, double2* __restrict__ gt) {
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n * n; x += gridDim.x * blockDim.x)
    gt[x] = g[(x % n) * n + x / n];
}

// v[z] = sum_{k,l} Lq[m(z)][k][l] gt[k][l] for z = (q, P) from z0 on, m(z) = (neg[q], P). One CTA per z; bound by
// reading the factors (the transposed density stays in L2).
__global__ void __launch_bounds__(256) jk_trace_all_kernel(const double2* __restrict__ Lq, const int* __restrict__ neg,
                                                           int naux, long long nn, const double2* __restrict__ gt,
                                                           double2* __restrict__ v) {
  const int q = blockIdx.y, P = blockIdx.x;
  const double2* m = Lq + ((long long)neg[q] * naux + P) * nn;
  double re = 0.0, im = 0.0;
#pragma unroll 4
  for (int x = threadIdx.x; x < (int)nn; x += 256) {
    const double2 a = m[x], g = gt[x];
    re = fma(a.x, g.x, fma(-a.y, g.y, re));
    im = fma(a.x, g.y, fma(a.y, g.x, im));
  }
  __shared__ double sr[8], si[8];
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, o);
    im += __shfl_xor_sync(0xffffffffu, im, o);
  }
  if ((threadIdx.x & 31) == 0) {
    sr[threadIdx.x >> 5] = re;
    si[threadIdx.x >> 5] = im;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < 8; ++w) {
      a += sr[w];
      b += si[w];
    }
    v[(long long)q * naux + P] = make_double2(a, b);
  }
}

// part[y][x] = s sum_z v[z] Lq[z][x] over share y of the z.
__global__ void __launch_bounds__(256) jk_weighted_kernel(const double2* __restrict__ Lq, const double2* __restrict__ v,
                                                          long long nz, long long nn, double s,
                                                          double2* __restrict__ part) {
  const long long x = blockIdx.x * 256ll + threadIdx.x;
  if (x >= nn) return;
  const long long z0 = nz * blockIdx.y / gridDim.y, z1 = nz * (blockIdx.y + 1) / gridDim.y;
  double jr = 0.0, ji = 0.0;
#pragma unroll 4
  for (long long z = z0; z < z1; ++z) {
    const double2 a = Lq[z * nn + x], w = v[z];
    jr = fma(a.x, w.x, fma(-a.y, w.y, jr));
    ji = fma(a.x, w.y, fma(a.y, w.x, ji));
  }
  part[blockIdx.y * nn + x] = make_double2(s * jr, s * ji);
}

// J[x] += s sum_z v[z] Lq[tab[z].x][x] and K[x] += s sum_z Kb[z][x] over the nz entries of a chunk.
__global__ void __launch_bounds__(256) jk_accumulate_kernel(const double2* __restrict__ Lq, const int4* __restrict__ tab,
                                                            const double2* __restrict__ v, const double2* __restrict__ Kb,
                                                            int nz, long long nn, double s, double2* __restrict__ J,
                                                            double2* __restrict__ K) {
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < nn; x += (long long)gridDim.x * blockDim.x) {
    double jr = 0.0, ji = 0.0, kr = 0.0, ki = 0.0;
    for (int z = 0; z < nz; ++z) {
      const double2 a = Lq[(long long)tab[z].x * nn + x], w = v[z], b = Kb[(long long)z * nn + x];
      jr = fma(a.x, w.x, fma(-a.y, w.y, jr));
      ji = fma(a.x, w.y, fma(a.y, w.x, ji));
      kr += b.x;
      ki += b.y;
    }
    J[x] = make_double2(J[x].x + s * jr, J[x].y + s * ji);
    K[x] = make_double2(K[x].x + s * kr, K[x].y + s * ki);
  }
}

}  // namespace

cudaError_t launch_fock_reduce(const double2* G, int nk, int n, double s, double* F0, cudaStream_t st) {
  fock_reduce_kernel<<<blocks_for((long long)n * n, 256, 152 * 8), 256, 0, st>>>(G, nk, n, s, F0);
  return cudaGetLastError();
}

int exchange_copies() { return kExchangeCopies; }

size_t coulomb_scratch(int n) { return (size_t)(kColShares + 1) * ((size_t)n * (n + 1) / 2) * sizeof(double); }

cudaError_t launch_coulomb_exchange(const double* eri, const double* gamma, int n, double* J, double* K, double* scratch,
                                    cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if (n > 1024) return cudaErrorInvalidValue;
  const long long npair = (long long)n * (n + 1) / 2;
  const size_t smem = (size_t)(npair + 2 * n) * sizeof(double);
  if (smem > 227 * 1024 - 64) return cudaErrorInvalidValue;  // the caller checks the size first
  if (smem > 48 * 1024 - 64) {
    cudaError_t e = cudaFuncSetAttribute(exchange_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  double* w = scratch + kColShares * npair;
  pair_weights_kernel<<<blocks_for((long long)n * n, 256, 152), 256, 0, st>>>(gamma, n, w);
  coulomb_columns_kernel<<<dim3((unsigned)((npair + 255) / 256), kColShares), 256, 0, st>>>(eri, w, (int)npair, scratch);
  exchange_kernel<<<(unsigned)npair, 256, smem, st>>>(eri, gamma, w, n, J, K);
  return cudaGetLastError();
}

cudaError_t launch_fock_combine(const double* F0, const double* J, const double* scratch, const double* K, int n,
                                double* out, cudaStream_t st) {
  fock_combine_kernel<<<blocks_for((long long)n * n, 256, 152 * 8), 256, 0, st>>>(F0, J, scratch, K, n, out);
  return cudaGetLastError();
}

cudaError_t launch_jk_trace(const double2* Lq, const int4* tab, int nz, int n, const double2* gamma, double2* v,
                            cudaStream_t st) {
  if (nz <= 0) return cudaSuccess;
  jk_trace_kernel<<<nz, 256, 0, st>>>(Lq, tab, n, gamma, v);
  return cudaGetLastError();
}

cudaError_t launch_jk_accumulate(const double2* Lq, const int4* tab, const double2* v, const double2* Kb, int nz, int n,
                                 double s, double2* J, double2* K, cudaStream_t st) {
  const long long nn = (long long)n * n;
  long long blocks = (nn + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  jk_accumulate_kernel<<<(unsigned)(blocks > 0 ? blocks : 1), 256, 0, st>>>(Lq, tab, v, Kb, nz, nn, s, J, K);
  return cudaGetLastError();
}

// J += s sum_{q,P} Lq[q][P] tr(Lq[-q][P] gamma): two passes over the factors (gt, v and part: scratch of n^2, nk naux
// and jk_coulomb_parts() n^2 values).
int jk_coulomb_parts(long long nn) { return (int)std::max(1LL, 8LL * 152 / std::max(1LL, (nn + 255) / 256)); }

cudaError_t launch_jk_coulomb(const double2* Lq, const int* neg, int nk, int naux, int n, const double2* gamma, double s,
                              double2* gt, double2* v, double2* part, double2* J, cudaStream_t st) {
  const long long nn = (long long)n * n;
  transpose_kernel<<<blocks_for(nn, 256, 152), 256, 0, st>>>(gamma, n, gt);
  jk_trace_all_kernel<<<dim3(naux, nk), 256, 0, st>>>(Lq, neg, naux, nn, gt, v);
  const int parts = jk_coulomb_parts(nn);
  jk_weighted_kernel<<<dim3((unsigned)((nn + 255) / 256), parts), 256, 0, st>>>(Lq, v, (long long)nk * naux, nn, s, part);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? launch_sum_parts(part, parts, nn, J, st) : e;
}

}  // namespace dmet

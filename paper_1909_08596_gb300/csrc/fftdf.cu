// The FFTDF variant of the embedded-ERI transformation (Appendix B, Algorithm 2): the pointwise
// steps around the Fourier transforms of the transformed pair densities, and those transforms: FFTs in
// registers along axes of 2, 3, 5 and 7-smooth lengths up to 32, dense DFTs along others (in registers up to
// 32 points, as batched complex GEMMs above); FP64.

#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"

namespace dmet {

namespace {

inline int grid_for(long long total, int threads, int cap) {
  long long g = (total + threads - 1) / threads;
  if (g < 1) g = 1;
  return (int)(g < cap ? g : cap);
}

// dst[r][x] = s exp(sign * i q.r) src[r][x], q.r = 2 pi sum_d (j_d / g_d)(n_d / N_d) for grid point
// r = (j_1, j_2, j_3) (C order) and the mesh triple n of q.
__global__ void fftdf_phase_kernel(const double2* __restrict__ src, double2* __restrict__ dst, int g0, int g1, int g2,
                                   double f0, double f1, double f2, double sign, double s, long long nx) {
  const long long total = (long long)g0 * g1 * g2 * nx;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const long long r = t / nx;
    const int j2 = (int)(r % g2), j1 = (int)((r / g2) % g1), j0 = (int)(r / ((long long)g1 * g2));
    // exp(sign * 2 pi i (j0 f0 + j1 f1 + j2 f2)), f_d = n_d / (N_d g_d)
    double sn, cs;
    sincospi(2.0 * sign * (j0 * f0 + j1 * f1 + j2 * f2), &sn, &cs);
    const double2 a = src[t];
    dst[t] = make_double2(s * (a.x * cs - a.y * sn), s * (a.x * sn + a.y * cs));
  }
}

// The same phase for a run of q values at once: blockIdx.y is the local index i of a q in the run,
// qtab[i] its q (mesh triple from the mesh, C order). Source block: src + qtab[i] * ng * nx if by_table,
// else src + i * ng * nx; destination block dst + i * ng * nx.
__global__ void fftdf_phase_q_kernel(const double2* __restrict__ src, double2* __restrict__ dst,
                                     const int* __restrict__ qtab, int by_table, int g0, int g1, int g2, int m0,
                                     int m1, int m2, double sign, double s, long long nx) {
  const long long ngx = (long long)g0 * g1 * g2 * nx;
  const int i = blockIdx.y, q = qtab[i];
  const int n0 = q / (m1 * m2), n1 = (q / m2) % m1, n2 = q % m2;
  const double f0 = (double)n0 / ((double)m0 * g0), f1 = (double)n1 / ((double)m1 * g1),
               f2 = (double)n2 / ((double)m2 * g2);
  const double2* in = src + (long long)(by_table ? q : i) * ngx;
  double2* out = dst + (long long)i * ngx;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < ngx;
       t += (long long)gridDim.x * blockDim.x) {
    const long long r = t / nx;
    const int j2 = (int)(r % g2), j1 = (int)((r / g2) % g1), j0 = (int)(r / ((long long)g1 * g2));
    double sn, cs;
    sincospi(2.0 * sign * (j0 * f0 + j1 * f1 + j2 * f2), &sn, &cs);
    const double2 a = in[t];
    out[t] = make_double2(s * (a.x * cs - a.y * sn), s * (a.x * sn + a.y * cs));
  }
}

// buf[G][x] *= v[G]
__global__ void fftdf_kernel_mul(double2* __restrict__ buf, const double* __restrict__ v, long long ng, long long nx) {
  const long long total = ng * nx;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const double w = v[t / nx];
    buf[t] = make_double2(buf[t].x * w, buf[t].y * w);
  }
}

// A dense DFT along the middle axis of [outer][g][inner]: out[o][k][i] = sum_j F[k g + j] in[o][j][i],
// for axes of at most kMaxDftAxis points. One thread per (o, i) column keeps the column's g inputs
// in registers and F in shared memory; the reads and writes of a warp are runs of consecutive i.
constexpr int kMaxDftAxis = 32;
__global__ void __launch_bounds__(256) dft_axis_kernel(const double2* __restrict__ F, int g, long long outer,
                                                      long long inner, const double2* __restrict__ in,
                                                      double2* __restrict__ out) {
  __shared__ double2 f[kMaxDftAxis * kMaxDftAxis];
  for (int t = threadIdx.x; t < g * g; t += blockDim.x) f[t] = F[t];
  __syncthreads();
  const long long total = outer * inner;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < total;
       c += (long long)gridDim.x * blockDim.x) {
    const long long o = c / inner, i = c - o * inner;
    const long long base = o * g * inner + i;
    double2 x[kMaxDftAxis];
#pragma unroll
    for (int j = 0; j < kMaxDftAxis; ++j)
      if (j < g) x[j] = in[base + j * inner];
    for (int k = 0; k < g; ++k) {
      double re = 0.0, im = 0.0;
#pragma unroll
      for (int j = 0; j < kMaxDftAxis; ++j)
        if (j < g) {
          const double2 a = f[k * g + j];
          re = fma(a.x, x[j].x, fma(-a.y, x[j].y, re));
          im = fma(a.x, x[j].y, fma(a.y, x[j].x, im));
        }
      out[base + k * inner] = make_double2(re, im);
    }
  }
}

// ---- FFTs along one axis, a thread per column ----
// The FP64 pipe bounds these passes: a dense DFT of 12 points takes 576 FMAs per column, the mixed-radix FFT about
// 130, and the Bloch phases and the Coulomb kernel join the passes as multiplications instead of passes of
// their own (the phases as products of one factor per axis, tabulated, instead of a sincos per value). The
// forward transform of the last axis, the kernel and its inverse are one pass. 12^3 grid, 8 q, 256 orbital
// pairs: 5.7 ms for six dense passes and three pointwise ones; about 0.6 ms for these five.

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// R-point DFT in place; tw[t stride] = w^t, w the primitive R-th root of the transform's direction (SGN).
template <int R, int SGN>
__device__ __forceinline__ void butterfly(double2 (&x)[R], const double2* tw, int stride) {
  if constexpr (R == 2) {
    const double2 a = x[0], b = x[1];
    x[0] = cadd(a, b);
    x[1] = csub(a, b);
  } else if constexpr (R == 4) {
    const double2 s02 = cadd(x[0], x[2]), d02 = csub(x[0], x[2]), s13 = cadd(x[1], x[3]), d13 = csub(x[1], x[3]);
    const double2 j = make_double2(-SGN * d13.y, SGN * d13.x);  // SGN i (x1 - x3)
    x[0] = cadd(s02, s13);
    x[2] = csub(s02, s13);
    x[1] = cadd(d02, j);
    x[3] = csub(d02, j);
  } else {
    // odd R: X_q, X_{R-q} = x_0 + sum_p (x_p + x_{R-p}) cos +- i sum_p (x_p - x_{R-p}) sin, p <= (R - 1) / 2
    constexpr int H = (R - 1) / 2;
    double2 a[H], b[H];
    double2 s0 = x[0];
#pragma unroll
    for (int p = 0; p < H; ++p) {
      a[p] = cadd(x[p + 1], x[R - 1 - p]);
      b[p] = csub(x[p + 1], x[R - 1 - p]);
      s0 = cadd(s0, a[p]);
    }
    const double2 x0 = x[0];
    x[0] = s0;
#pragma unroll
    for (int q = 1; q <= H; ++q) {
      double2 c = x0, d = make_double2(0.0, 0.0);
#pragma unroll
      for (int p = 0; p < H; ++p) {
        const double2 w = tw[((p + 1) * q % R) * stride];
        c.x = fma(a[p].x, w.x, c.x);
        c.y = fma(a[p].y, w.x, c.y);
        d.x = fma(-b[p].y, w.y, d.x);
        d.y = fma(b[p].x, w.y, d.y);
      }
      x[q] = cadd(c, d);
      x[R - q] = csub(c, d);
    }
  }
}

// DFT of N points in place, in natural order (decimation in time); tw[t stride] = w_N^t.
template <int N, int SGN>
__device__ __forceinline__ void fft(double2 (&x)[N], const double2* tw, int stride) {
  constexpr int R = N % 4 == 0 ? 4 : N % 2 == 0 ? 2 : N % 3 == 0 ? 3 : N % 5 == 0 ? 5 : 7, M = N / R;
  static_assert(N == 1 || R * M == N, "lengths with prime factors 2, 3, 5 and 7");
  if constexpr (N == 1) {
  } else if constexpr (M == 1) {
    butterfly<R, SGN>(x, tw, stride);
  } else {
    double2 y[R][M];
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
      for (int m = 0; m < M; ++m) y[r][m] = x[r + R * m];
      fft<M, SGN>(y[r], tw, stride * R);
    }
#pragma unroll
    for (int k = 0; k < M; ++k) {
      double2 t[R];
#pragma unroll
      for (int r = 0; r < R; ++r) t[r] = r * k == 0 ? y[r][k] : cmul(y[r][k], tw[r * k * stride]);
      butterfly<R, SGN>(t, tw, stride * M);
#pragma unroll
      for (int q = 0; q < R; ++q) x[k + M * q] = t[q];
    }
  }
}

struct FftArgs {
  const double2* in;      // forward pass of the first axis: block qtab[i] of the factors; else in place
  double2* buf;           // [q][grid][nx]
  const double2* F;       // forward DFT matrix of the axis (row 1: the powers of the root)
  const double2* phase;   // [q][g]: exp(-i q.r) along this axis
  const int* qtab;        // or null
  const double* v;        // middle pass: Coulomb kernel [q][grid]
  long long outer, inner; // columns (o, i): base o g inner + i
  long long per_q;        // outer indices per q
};

// MODE 0: phases, forward transform. MODE 1 (last axis): phases, forward, kernel, inverse, conjugate phases.
// MODE 2: inverse, conjugate phases. (No normalisation.)
template <int G, int MODE>
__global__ void __launch_bounds__(128) fft_axis_kernel(const FftArgs a) {
  __shared__ double2 tw[2][G];
  for (int t = threadIdx.x; t < G; t += blockDim.x) {
    const double2 w = G > 1 ? a.F[G + t] : make_double2(1.0, 0.0);
    tw[0][t] = w;
    tw[1][t] = make_double2(w.x, -w.y);
  }
  __syncthreads();
  const long long total = a.outer * a.inner;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < total; c += (long long)gridDim.x * blockDim.x) {
    const long long o = c / a.inner, i = c - o * a.inner, q = o / a.per_q;
    double2* p = a.buf + o * G * a.inner + i;
    const double2* src = p;
    if (MODE == 0 && a.qtab) src = a.in + (a.qtab[q] * a.per_q + (o - q * a.per_q)) * G * a.inner + i;
    const double2* ph = a.phase + q * G;
    double2 x[G];
#pragma unroll
    for (int j = 0; j < G; ++j) x[j] = src[j * a.inner];
    if constexpr (MODE != 2) {
#pragma unroll
      for (int j = 1; j < G; ++j) x[j] = cmul(x[j], ph[j]);
      fft<G, -1>(x, tw[0], 1);
    }
    if constexpr (MODE == 1) {
      const double* v = a.v + o * G;
#pragma unroll
      for (int k = 0; k < G; ++k) {
        const double w = v[k];
        x[k].x *= w;
        x[k].y *= w;
      }
    }
    if constexpr (MODE != 0) {
      fft<G, 1>(x, tw[1], 1);
#pragma unroll
      for (int j = 1; j < G; ++j) {
        const double2 w = ph[j];
        x[j] = cmul(x[j], make_double2(w.x, -w.y));
      }
    }
#pragma unroll
    for (int j = 0; j < G; ++j) p[j * a.inner] = x[j];
  }
}

template <int G>
cudaError_t fft_axis(int mode, const FftArgs& a, cudaStream_t st) {
  const int blocks = grid_for(a.outer * a.inner, 128, 152 * 32);
  if (mode == 0) fft_axis_kernel<G, 0><<<blocks, 128, 0, st>>>(a);
  else if (mode == 1) fft_axis_kernel<G, 1><<<blocks, 128, 0, st>>>(a);
  else fft_axis_kernel<G, 2><<<blocks, 128, 0, st>>>(a);
  return cudaGetLastError();
}

// out[i] += sum_p parts[p n + i]
// Eight threads share the parts of each element (32 elements per CTA), so that a small block with many parts (the
// 104^2 exchange matrix from some 300 parts) still has a few hundred CTAs of loads in flight.
__global__ void __launch_bounds__(256) sum_parts_kernel(const double2* __restrict__ parts, int np, long long n,
                                                        double2* __restrict__ out) {
  __shared__ double2 sh[8][33];
  const int x = threadIdx.x & 31, g = threadIdx.x >> 5;
  for (long long i0 = blockIdx.x * 32ll; i0 < n; i0 += gridDim.x * 32ll) {
    double2 a = make_double2(0.0, 0.0);
    if (i0 + x < n) {
#pragma unroll 4
      for (int p = g; p < np; p += 8) {
        const double2 b = parts[(long long)p * n + i0 + x];
        a.x += b.x;
        a.y += b.y;
      }
    }
    sh[g][x] = a;
    __syncthreads();
    if (g == 0 && i0 + x < n) {
      a = out[i0 + x];
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        a.x += sh[h][x].x;
        a.y += sh[h][x].y;
      }
      out[i0 + x] = a;
    }
    __syncthreads();
  }
}

}  // namespace

// Every length up to 32 that the FFTs take is faster than dense; whole calls with one cell or two and a cubic grid, dense
// against FFTs, in us: 2: 225 and 92, 5: 430 and 154, 7: 598 and 193, 9: 789 and 283, 12: 1819 and 482, 16: 2552 and 775,
// 18: 3087 and 1214, 20: 1652 and 563, 24: 2138 and 822, 28: 4031 and 1258, 30: 7138 and 4208, 32: 4813 and 1753.
bool fftdf_fft_axis(int g) {
  if (g < 1 || g > kMaxDftAxis) return false;
  for (int p : {2, 3, 5, 7})
    while (g % p == 0) g /= p;
  return g == 1;
}

cudaError_t launch_fft_axis(int g, int mode, const double2* in, const int* qtab, double2* buf, const double2* F,
                            const double2* phase, const double* v, long long outer, long long inner, long long per_q,
                            cudaStream_t st) {
  const FftArgs a{in, buf, F, phase, qtab, v, outer, inner, per_q};
  switch (g) {
#define DMET_FFT(G) \
  case G: return fft_axis<G>(mode, a, st);
    DMET_FFT(1) DMET_FFT(2) DMET_FFT(3) DMET_FFT(4) DMET_FFT(5) DMET_FFT(6) DMET_FFT(7) DMET_FFT(8) DMET_FFT(9)
    DMET_FFT(10) DMET_FFT(12) DMET_FFT(14) DMET_FFT(15) DMET_FFT(16) DMET_FFT(18) DMET_FFT(20) DMET_FFT(21)
    DMET_FFT(24) DMET_FFT(25) DMET_FFT(27) DMET_FFT(28) DMET_FFT(30) DMET_FFT(32)
#undef DMET_FFT
  }
  return cudaErrorInvalidValue;
}

bool fftdf_small_axis(int g) { return g >= 1 && g <= kMaxDftAxis; }

cudaError_t launch_dft_axis_small(const double2* F, int g, long long outer, long long inner, const double2* in,
                                  double2* out, cudaStream_t st) {
  if (!fftdf_small_axis(g)) return cudaErrorInvalidValue;
  dft_axis_kernel<<<grid_for(outer * inner, 256, 152 * 8), 256, 0, st>>>(F, g, outer, inner, in, out);
  return cudaGetLastError();
}

cudaError_t launch_sum_parts(const double2* parts, int np, long long n, double2* out, cudaStream_t st) {
  sum_parts_kernel<<<grid_for(n, 32, 152 * 32), 256, 0, st>>>(parts, np, n, out);
  return cudaGetLastError();
}

cudaError_t launch_fftdf_phase(const double2* src, double2* dst, const int grid[3], const int nq[3], const int mesh[3],
                               double sign, double s, long long nx, cudaStream_t st) {
  const long long total = (long long)grid[0] * grid[1] * grid[2] * nx;
  fftdf_phase_kernel<<<grid_for(total, 256, 152 * 16), 256, 0, st>>>(
      src, dst, grid[0], grid[1], grid[2], (double)nq[0] / ((double)mesh[0] * grid[0]),
      (double)nq[1] / ((double)mesh[1] * grid[1]), (double)nq[2] / ((double)mesh[2] * grid[2]), sign, s, nx);
  return cudaGetLastError();
}

cudaError_t launch_fftdf_phase_q(const double2* src, double2* dst, const int* qtab, int nq_run, int by_table,
                                 const int grid[3], const int mesh[3], double sign, double s, long long nx,
                                 cudaStream_t st) {
  if (nq_run <= 0) return cudaSuccess;
  if (nq_run > 65535) return cudaErrorInvalidValue;
  const long long per = (long long)grid[0] * grid[1] * grid[2] * nx;
  const int gx = grid_for(per, 256, std::max(1, 152 * 16 / nq_run));
  fftdf_phase_q_kernel<<<dim3(gx, nq_run), 256, 0, st>>>(src, dst, qtab, by_table, grid[0], grid[1], grid[2], mesh[0],
                                                         mesh[1], mesh[2], sign, s, nx);
  return cudaGetLastError();
}

cudaError_t launch_fftdf_kernel_mul(double2* buf, const double* v, long long ng, long long nx, cudaStream_t st) {
  fftdf_kernel_mul<<<grid_for(ng * nx, 256, 152 * 16), 256, 0, st>>>(buf, v, ng, nx);
  return cudaGetLastError();
}

}  // namespace dmet

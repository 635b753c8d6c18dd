// Device vector kernels of the implicit solver (see krylov.h).
#include "krylov.h"

#include <type_traits>

namespace fedbm {
namespace krylov {
namespace {

int grid_of(int64_t n) {
  const int64_t b = (n + kThreads - 1) / kThreads;
  return int(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

__global__ void axpby_kernel(int64_t n, double a, const double* x, double b, const double* y, double* out) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    out[i] = a * x[i] + b * y[i];
}

__global__ void combination_kernel(int64_t n, int m, const double* V, const double* c, double* y) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    double acc = 0.0;
    for (int j = 0; j < m; ++j) acc += c[j] * V[size_t(j) * n + i];
    y[i] += acc;
  }
}

// sum over the block's threads, in thread 0 (red: one double per warp)
__device__ __forceinline__ double block_sum(double acc, double* red) {
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int q = 0; q < kThreads / 32; ++q) t += red[q];
  __syncthreads();
  return t;
}

// sum of p[0 .. nb) over a warp, in every lane
__device__ __forceinline__ double warp_sum(const double* p, int nb) {
  double acc = 0.0;
  for (int q = threadIdx.x & 31; q < nb; q += 32) acc += p[q];
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  return acc;
}

// This block's chunk [lo, hi) of n values (gridDim.x chunks).
__device__ __forceinline__ void chunk_of(int64_t n, int64_t& lo, int64_t& hi) {
  const int64_t len = ((n + gridDim.x - 1) / gridDim.x + kThreads - 1) / kThreads * kThreads;
  lo = min(n, int64_t(blockIdx.x) * len);
  hi = min(n, lo + len);
}

// part[j][block] = sum over the block's chunk of V_j w for j < m, eight j at a time so
// that w is read once for them and one barrier serves them all.  FP64 arithmetic is
// slow here, and a reduction of one value per thread was mostly the reduction (512
// blocks a vector whatever its length: 21 us for 15 vectors of 82k values).
__device__ void chunk_dots(int64_t n, int64_t lo, int64_t hi, int m, const double* V, const double* w, double* part) {
  __shared__ double red[8][kThreads + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int j0 = 0; j0 < m; j0 += 8) {
    double acc[8] = {};
    for (int64_t i = lo + threadIdx.x; i < hi; i += kThreads) {
      const double wi = w[i];
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j0 + j < m) acc[j] = fma(V[size_t(j0 + j) * n + i], wi, acc[j]);
    }
    // through shared memory, warp j adding up vector j: a third of the additions of a
    // shuffle reduction in every warp
#pragma unroll
    for (int j = 0; j < 8; ++j) red[j][threadIdx.x] = acc[j];
    __syncthreads();
    if (j0 + warp < m) {
      double t = 0.0;
#pragma unroll
      for (int q = 0; q < kThreads / 32; ++q) t += red[warp][q * 32 + lane];
      for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
      if (lane == 0) part[size_t(j0 + warp) * gridDim.x + blockIdx.x] = t;
    }
    __syncthreads();
  }
}

__global__ void dot_partial_kernel(int64_t n, int m, const double* V, const double* w, double* partial) {
  int64_t lo, hi;
  chunk_of(n, lo, hi);
  chunk_dots(n, lo, hi, m, V, w, partial);
}

// h[j] = sum of partial[j][0 .. nb), one warp per j
__global__ void dot_final_kernel(int m, int nb, const double* partial, double* h) {
  const int j = (blockIdx.x * kThreads + threadIdx.x) >> 5;
  if (j >= m) return;
  const double t = warp_sum(partial + size_t(j) * nb, nb);
  if ((threadIdx.x & 31) == 0) h[j] = t;
}

__global__ void direction_kernel(int64_t n, int Np, int Qp, const double* minv, const double* src,
                                 const double* norm_part, int nb, double* v, double* z, double* zpart) {
  __shared__ double red[kThreads / 32];
  __shared__ double scale;
  double s = 1.0;
  if (norm_part) {
    if (threadIdx.x < 32) {
      const double t = warp_sum(norm_part, nb);
      if (threadIdx.x == 0) scale = t > 0.0 ? 1.0 / sqrt(t) : 0.0;
    }
    __syncthreads();
    s = scale;
  }
  double acc = 0.0;
  for (int64_t t = blockIdx.x * int64_t(kThreads) + threadIdx.x; t < n; t += int64_t(gridDim.x) * kThreads) {
    if (norm_part) v[t] = src[t] * s;
    if (minv) {
      // (element k, node r, velocity i): row r of the block times the column of v
      const int64_t kn = t / Qp, k = kn / Np;
      const int i = int(t - kn * Qp);
      const double* col = src + k * Np * Qp + i;
      const double* row = minv + kn * Np * Qp + i;
      double a = 0.0;
#pragma unroll 8
      for (int q = 0; q < Np; ++q) a = fma(row[size_t(q) * Qp], col[size_t(q) * Qp] * s, a);
      z[t] = a;
      acc = fma(a, a, acc);
    }
  }
  if (minv && zpart) {
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) zpart[blockIdx.x] = acc;
  }
}

__global__ void perturb_kernel(int64_t n, double eps, const double* zpart, int nb, const double* Y, const double* x,
                               double* step, double* out) {
  __shared__ double step_s;
  double e = eps;
  if (zpart) {
    if (threadIdx.x < 32) {
      const double t = warp_sum(zpart, nb);
      if (threadIdx.x == 0) step_s = t > 0.0 ? eps / sqrt(t) : eps;
    }
    __syncthreads();
    e = step_s;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) step[0] = e;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    out[i] = Y[i] + e * x[i];
}

__global__ void project_first_kernel(int64_t n, int m, const double* x, const double* Rp, const double* RY,
                                     const double* step, double dtg, const double* V, double* w, double* part) {
  int64_t lo, hi;
  chunk_of(n, lo, hi);
  __shared__ double c_s;
  if (threadIdx.x == 0) c_s = -dtg / step[0];  // one quotient per block: FP64 is slow here
  __syncthreads();
  const double c = c_s;
  for (int64_t i = lo + threadIdx.x; i < hi; i += kThreads) w[i] = x[i] + c * (Rp[i] - RY[i]);
  chunk_dots(n, lo, hi, m, V, w, part);  // every thread reads back only what it wrote
}

__global__ void project_next_kernel(int64_t n, int m, const double* V, const double* part_in, double* h_host, double* w,
                                    double* part_out, double* norm_host) {
  extern __shared__ double h[];
  __shared__ double red[kThreads / 32];
  for (int j = threadIdx.x >> 5; j < m; j += kThreads / 32) {
    const double t = warp_sum(part_in + size_t(j) * gridDim.x, gridDim.x);
    if ((threadIdx.x & 31) == 0) {
      h[j] = t;
      if (blockIdx.x == 0) h_host[j] = t;
    }
  }
  __syncthreads();
  int64_t lo, hi;
  chunk_of(n, lo, hi);
  double acc = 0.0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += kThreads) {
    double t = 0.0;
#pragma unroll 8
    for (int j = 0; j < m; ++j) t = fma(h[j], V[size_t(j) * n + i], t);
    const double wi = w[i] - t;
    w[i] = wi;
    acc = fma(wi, wi, acc);
  }
  if (norm_host) {
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) {
      part_out[blockIdx.x] = acc;
      norm_host[blockIdx.x] = acc;
    }
  } else {
    chunk_dots(n, lo, hi, m, V, w, part_out);
  }
}

__global__ void to_f32_kernel(int64_t n, const double* x, float* y) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    y[i] = float(x[i]);
}
__global__ void to_f64_kernel(int64_t n, const float* x, double* y) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    y[i] = double(x[i]);
}

template <typename R>
__global__ void set_geo_dt_kernel(int64_t K, int stride, int slot, double value, R* geo) {
  for (int64_t k = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; k < K; k += int64_t(gridDim.x) * blockDim.x)
    geo[k * stride + slot] = R(value);
}

}  // namespace

int blocks_of(int64_t n) {
  const int64_t b = (n + 511) / 512;
  return int(b < 1 ? 1 : b > kMaxBlocks ? kMaxBlocks : b);
}

int direction_blocks(int64_t n) {
  const int64_t b = (n + kThreads - 1) / kThreads;
  return int(b < 1 ? 1 : b > kMaxBlocks ? kMaxBlocks : b);
}

cudaError_t direction(int64_t K, int Np, int Qp, const double* minv, const double* src, const double* norm_part,
                      double* v, double* z, double* zpart, cudaStream_t st) {
  const int64_t n = K * Np * Qp;
  direction_kernel<<<direction_blocks(n), kThreads, 0, st>>>(n, Np, Qp, minv, src, norm_part, blocks_of(n), v, z,
                                                             zpart);
  return cudaGetLastError();
}

cudaError_t perturb(int64_t n, double eps, const double* zpart, const double* Y, const double* x, double* step,
                    double* out, cudaStream_t st) {
  perturb_kernel<<<direction_blocks(n), kThreads, 0, st>>>(n, eps, zpart, direction_blocks(n), Y, x, step, out);
  return cudaGetLastError();
}

cudaError_t project_first(int64_t n, int m, const double* x, const double* Rp, const double* RY, const double* step,
                          double dtg, const double* V, double* w, double* part, cudaStream_t st) {
  project_first_kernel<<<blocks_of(n), kThreads, 0, st>>>(n, m, x, Rp, RY, step, dtg, V, w, part);
  return cudaGetLastError();
}

cudaError_t project_next(int64_t n, int m, const double* V, const double* part_in, double* h_host, double* w,
                         double* part_out, double* norm_host, cudaStream_t st) {
  project_next_kernel<<<blocks_of(n), kThreads, size_t(m) * sizeof(double), st>>>(n, m, V, part_in, h_host, w, part_out,
                                                                                 norm_host);
  return cudaGetLastError();
}

cudaError_t axpby(int64_t n, double a, const double* x, double b, const double* y, double* out, cudaStream_t st) {
  axpby_kernel<<<grid_of(n), kThreads, 0, st>>>(n, a, x, b, y, out);
  return cudaGetLastError();
}

cudaError_t add_combination(int64_t n, int m, const double* V, const double* c_dev, double* out, cudaStream_t st) {
  if (m < 1) return cudaSuccess;
  combination_kernel<<<grid_of(n), kThreads, 0, st>>>(n, m, V, c_dev, out);
  return cudaGetLastError();
}

cudaError_t multi_dot(int64_t n, int m, const double* V, const double* w, double* partial, double* h, cudaStream_t st) {
  if (m < 1) return cudaSuccess;
  const int nb = blocks_of(n);
  dot_partial_kernel<<<nb, kThreads, 0, st>>>(n, m, V, w, partial);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  dot_final_kernel<<<(m * 32 + kThreads - 1) / kThreads, kThreads, 0, st>>>(m, nb, partial, h);
  return cudaGetLastError();
}

cudaError_t to_f32(int64_t n, const double* x, float* y, cudaStream_t st) {
  to_f32_kernel<<<grid_of(n), kThreads, 0, st>>>(n, x, y);
  return cudaGetLastError();
}

cudaError_t to_f64(int64_t n, const float* x, double* y, cudaStream_t st) {
  to_f64_kernel<<<grid_of(n), kThreads, 0, st>>>(n, x, y);
  return cudaGetLastError();
}

cudaError_t set_geo_dt(int64_t K, int stride, int slot, double value, void* geo, int real_bytes, cudaStream_t st) {
  const int grid = grid_of(K);
  if (real_bytes == 8) set_geo_dt_kernel<double><<<grid, kThreads, 0, st>>>(K, stride, slot, value, static_cast<double*>(geo));
  else set_geo_dt_kernel<float><<<grid, kThreads, 0, st>>>(K, stride, slot, value, static_cast<float*>(geo));
  return cudaGetLastError();
}

}  // namespace krylov
}  // namespace fedbm

// ---- element-and-velocity block-Jacobi preconditioner --------------------------
// For element k and velocity i the block of (I - dtg J) that couples the
// element's own nodes at velocity i is
//   M = (1 + dtg / tau_k) I + dtg (a_r Dr + a_s Ds) - dtg LIFT diag(c) E,
// where a_r = e_x r_x + e_y r_y, a_s = e_x s_x + e_y s_y, E picks the face
// nodes out of the element's nodes, and c = Fscale (e.n - ab |e.n|) / 2 is the
// numerical flux's coefficient of the element's own trace on each face (the
// strong-form residual of eq. byparts).  Neighbour traces, wall reflection and
// the equilibrium's dependence on the other velocities are left out.  M is
// inverted by Gauss-Jordan elimination with partial pivoting, one thread per
// (element, velocity).
namespace fedbm {
namespace krylov {
namespace {

constexpr int kMaxNp = 28;  // degree 6

template <typename R, int NPT>
__global__ void bj_build_kernel(int64_t K, int Np, int Nfp, int Qp, const R* geo, const double* vel64,
                                const double* ops, const int* fmask, double dtg, double ab, double* minv) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= K * Qp) return;
  const int64_t k = t / Qp;
  const int i = int(t % Qp);
  const R* g = geo + k * 16;
  const double ex = vel64[i], ey = vel64[Qp + i];
  const double ar = ex * double(g[0]) + ey * double(g[2]);
  const double as = ex * double(g[1]) + ey * double(g[3]);
  const double itau = double(g[15]);
  const double* Dr = ops;
  const double* Ds = ops + Np * Np;
  const double* LIFT = ops + 2 * Np * Np;
  const int NF = 3 * Nfp;
  double A[NPT * NPT], B[NPT * NPT];  // Np <= NPT
  for (int n = 0; n < Np; ++n)
    for (int m = 0; m < Np; ++m) {
      A[n * Np + m] = (n == m ? 1.0 + dtg * itau : 0.0) + dtg * (ar * Dr[n * Np + m] + as * Ds[n * Np + m]);
      B[n * Np + m] = n == m ? 1.0 : 0.0;
    }
  for (int f = 0; f < 3; ++f) {
    const double en = ex * double(g[4 + 3 * f]) + ey * double(g[5 + 3 * f]);
    const double c = 0.5 * (en - ab * fabs(en)) * double(g[6 + 3 * f]);
    if (c == 0.0) continue;
    for (int a = 0; a < Nfp; ++a) {
      const int j = f * Nfp + a, m = fmask[j];
      for (int n = 0; n < Np; ++n) A[n * Np + m] -= dtg * LIFT[n * NF + j] * c;
    }
  }
  // Gauss-Jordan with partial pivoting: B <- A^-1
  for (int col = 0; col < Np; ++col) {
    int piv = col;
    for (int r = col + 1; r < Np; ++r)
      if (fabs(A[r * Np + col]) > fabs(A[piv * Np + col])) piv = r;
    if (piv != col)
      for (int q = 0; q < Np; ++q) {
        double x = A[col * Np + q]; A[col * Np + q] = A[piv * Np + q]; A[piv * Np + q] = x;
        x = B[col * Np + q]; B[col * Np + q] = B[piv * Np + q]; B[piv * Np + q] = x;
      }
    const double d = 1.0 / A[col * Np + col];
    for (int q = 0; q < Np; ++q) {
      A[col * Np + q] *= d;
      B[col * Np + q] *= d;
    }
    for (int r = 0; r < Np; ++r) {
      if (r == col) continue;
      const double fct = A[r * Np + col];
      if (fct == 0.0) continue;
      for (int q = 0; q < Np; ++q) {
        A[r * Np + q] -= fct * A[col * Np + q];
        B[r * Np + q] -= fct * B[col * Np + q];
      }
    }
  }
  for (int n = 0; n < Np; ++n)
    for (int m = 0; m < Np; ++m) minv[((k * Np + n) * Np + m) * Qp + i] = B[n * Np + m];
}

}  // namespace

cudaError_t block_jacobi_build(int64_t K, int Np, int Nfp, int Qp, const void* geo, int real_bytes,
                               const double* vel64, const double* ops, const int* fmask, double dtg, double ab,
                               double* minv, cudaStream_t st) {
  if (Np > kMaxNp) return cudaErrorInvalidValue;
  const int64_t n = K * Qp;
  const int blocks = int((n + 127) / 128);
  // the block size rounded up to a degree's node count keeps the per-thread
  // work arrays (local memory) small at low degree
  auto run = [&](auto npt) {
    constexpr int NPT = decltype(npt)::value;
    if (real_bytes == 8)
      bj_build_kernel<double, NPT><<<blocks, 128, 0, st>>>(K, Np, Nfp, Qp, static_cast<const double*>(geo), vel64,
                                                           ops, fmask, dtg, ab, minv);
    else
      bj_build_kernel<float, NPT><<<blocks, 128, 0, st>>>(K, Np, Nfp, Qp, static_cast<const float*>(geo), vel64,
                                                          ops, fmask, dtg, ab, minv);
  };
  if (Np <= 6) run(std::integral_constant<int, 6>{});
  else if (Np <= 15) run(std::integral_constant<int, 15>{});
  else run(std::integral_constant<int, kMaxNp>{});
  return cudaGetLastError();
}

cudaError_t block_jacobi_apply(int64_t K, int Np, int Qp, const double* minv, const double* v, double* z,
                               cudaStream_t st) {
  return direction(K, Np, Qp, minv, v, nullptr, nullptr, z, nullptr, st);
}

}  // namespace krylov
}  // namespace fedbm

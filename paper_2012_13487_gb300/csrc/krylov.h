// Device vector kernels of the implicit solver (Newton-GMRES): FP64 vectors
// of the solver's internal layout [K][Np][Qp], reductions in a fixed order
// (the same result on every run).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fedbm {
namespace krylov {

// Most blocks of a partial-sum reduction (one partial sum per block); a vector of
// n values takes blocks_of(n), at least 512 values each.
constexpr int kMaxBlocks = 608;
constexpr int kThreads = 256;
int blocks_of(int64_t n);

// out = a x + b y (out may alias x or y)
cudaError_t axpby(int64_t n, double a, const double* x, double b, const double* y, double* out, cudaStream_t st);
// out += sum_i c[i] V_i for i < m; V holds m vectors of n values each, c in device memory
cudaError_t add_combination(int64_t n, int m, const double* V, const double* c_dev, double* out, cudaStream_t st);
// h[i] = <V_i, w> for i < m, through partial[m][blocks_of(n)] (device); h in device memory
cudaError_t multi_dot(int64_t n, int m, const double* V, const double* w, double* partial, double* h, cudaStream_t st);
// FP64 <-> FP32 copies
cudaError_t to_f32(int64_t n, const double* x, float* y, cudaStream_t st);
cudaError_t to_f64(int64_t n, const float* x, double* y, cudaStream_t st);
// geo[k][dt slot] = value for every element (a copy of the geometry with a unit time step)
cudaError_t set_geo_dt(int64_t K, int stride, int slot, double value, void* geo, int real_bytes, cudaStream_t st);

}  // namespace krylov
}  // namespace fedbm

namespace fedbm {
namespace krylov {

// Element-and-velocity block-Jacobi preconditioner of (I - dtg J) (see
// krylov.cu): the inverse of every (element, velocity) block, stored
// [K][Np][Np][Qp], built from the FP64 reference operators ops = [Dr | Ds |
// LIFT] (row-major, Np*Np, Np*Np, Np*3Nfp), fmask [3][Nfp], the velocity table
// vel64 [3][Qp] and the element geometry (real_bytes 8 or 4).
cudaError_t block_jacobi_build(int64_t K, int Np, int Nfp, int Qp, const void* geo, int real_bytes,
                               const double* vel64, const double* ops, const int* fmask, double dtg, double ab,
                               double* minv, cudaStream_t st);
// z = M^-1 v, blockwise
cudaError_t block_jacobi_apply(int64_t K, int Np, int Qp, const double* minv, const double* v, double* z,
                               cudaStream_t st);

// ---- one GMRES iteration ---------------------------------------------------------
// The scalars between these kernels (norms, Gram-Schmidt coefficients, the step of
// the difference quotient) stay on the device: a kernel leaves one partial sum per
// block and the blocks of the next each add them up, in the same order.

// v = src / sqrt(sum of norm_part) (norm_part == nullptr: v = src, not written) and z =
// M^-1 v (minv == nullptr: no z); zpart[0 .. return value of direction_blocks) = partial
// sums of z^2
int direction_blocks(int64_t n);
cudaError_t direction(int64_t K, int Np, int Qp, const double* minv, const double* src, const double* norm_part,
                      double* v, double* z, double* zpart, cudaStream_t st);
// step[0] = eps / sqrt(sum of zpart) (zpart == nullptr, or a zero sum: eps); out = Y + step x
cudaError_t perturb(int64_t n, double eps, const double* zpart, const double* Y, const double* x, double* step,
                    double* out, cudaStream_t st);
// w = x - dtg / step[0] (Rp - RY); part[j][blocks_of(n)] = partial <V_j, w> for j < m
cudaError_t project_first(int64_t n, int m, const double* x, const double* Rp, const double* RY, const double* step,
                          double dtg, const double* V, double* w, double* part, cudaStream_t st);
// h_host[j] = h_j = sum of part_in[j], w -= sum_j h_j V_j; then part_out[j] = partial
// <V_j, w>, or, where norm_host is given, part_out[0] = norm_host = partial <w, w>.
// h_host and norm_host are pinned host memory, written by the kernel itself: a copy
// behind it would hold up the kernels queued after it.
cudaError_t project_next(int64_t n, int m, const double* V, const double* part_in, double* h_host, double* w,
                         double* part_out, double* norm_host, cudaStream_t st);

}  // namespace krylov
}  // namespace fedbm

// Work space of the implicit solver (Newton-GMRES) of a single-group solver: its
// device buffers, pinned column and event, taken together or not at all.  A space is
// sized (n, m, s set) only once every buffer exists, and a request that fails gives
// back what was taken before it, so that a call after a recoverable out-of-memory
// asks again instead of running kernels on null pointers.  Host code only: the
// allocation functions come from the caller.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace fedbm {

// Where the buffers come from; every request returns 0 on success.
struct SpaceMemory {
  int (*device)(void** p, size_t bytes);
  int (*pinned)(void** p, size_t bytes);
  int (*event)(void** e);
  void (*free_device)(void* p);
  void (*free_pinned)(void* p);
  void (*free_event)(void* e);
};

struct ImplicitSpace {
  int64_t n = 0;        // K * Np * Qp; 0: nothing is allocated
  int m = 0, s = 0;     // GMRES restart length, stages
  double* u0 = nullptr;     // state at the start of the step
  double* Y = nullptr;      // stage value (Newton iterate)
  double* base = nullptr;   // u0 + dt sum_{j<i} a_ij k_j
  double* RY = nullptr;     // R(Y)
  double* G = nullptr;      // Newton residual, then the GMRES right-hand side -G
  double* d = nullptr;      // Newton update
  double* w = nullptr;      // GMRES work vector
  double* Yp = nullptr;     // Y + eps v
  double* Rp = nullptr;     // R(Y + eps v)
  double* V = nullptr;      // GMRES basis [m+1][n]
  double* k = nullptr;      // stage derivatives [s][n]
  double* partial = nullptr;  // two of [m+1][max_blocks]: the two Gram-Schmidt passes
  double* hdev = nullptr;     // [max(m+2, s)] dot results / combination coefficients
  double* zpart = nullptr;    // [max_blocks] partial sums of |M^-1 v|^2
  double* step = nullptr;     // [1] step of the difference quotient
  double* npart = nullptr;    // [max_blocks] partial sums of |w|^2
  double* hcol = nullptr;     // pinned host memory [2 (m+1) + max_blocks]: h of both passes, npart
  void* column = nullptr;     // event: hcol is complete
  void* x32 = nullptr;        // FP32 state: FP32 copy of the input of R
  void* r32 = nullptr;        // FP32 state: FP32 residual register
  void* scratch = nullptr;    // stage-kernel state output (unused values)
  void* geo_unit = nullptr;   // geometry with dt = 1
  // element-and-velocity block-Jacobi preconditioner (right preconditioning)
  double* minv = nullptr;     // [K][Np][Np][Qp] block inverses of (I - dt gamma J)
  double* z = nullptr;        // M^-1 v
  double* ops = nullptr;      // FP64 Dr | Ds | LIFT of the degree
  int* fmask = nullptr;       // [3][Nfp]
  double minv_dtg = 0;        // dt gamma the inverses were built for (0 = none)

  // Sizes for n values, restart length m, s stages; `geo_bytes` of geometry, values of
  // real_bytes in the stage kernel.  *fresh: the buffers are new (geo_unit is not filled).
  int reserve(const SpaceMemory& mem, int64_t n_, int m_, int s_, int max_blocks, size_t real_bytes, size_t geo_bytes,
              bool* fresh) {
    *fresh = false;
    if (n > 0 && n == n_ && m >= m_ && s >= s_) return 0;
    release(mem);
    const size_t vb = size_t(n_) * sizeof(double), bb = size_t(max_blocks) * sizeof(double);
    const size_t h = size_t(m_ + 2 > s_ ? m_ + 2 : s_) * sizeof(double);
    const struct {
      void* at;  // the member that receives the pointer
      size_t bytes;
    } device[] = {{&u0, vb}, {&Y, vb}, {&base, vb}, {&RY, vb}, {&G, vb}, {&d, vb}, {&w, vb}, {&Yp, vb}, {&Rp, vb},
                  {&V, vb * size_t(m_ + 1)}, {&k, vb * size_t(s_)}, {&partial, 2 * size_t(m_ + 1) * bb}, {&hdev, h},
                  {&zpart, bb}, {&step, sizeof(double)}, {&npart, bb}, {&scratch, size_t(n_) * real_bytes},
                  {&x32, real_bytes == 4 ? size_t(n_) * 4 : 0}, {&r32, real_bytes == 4 ? size_t(n_) * 4 : 0},
                  {&geo_unit, geo_bytes}};
    int rc = 0;
    for (const auto& b : device)
      if (rc == 0 && b.bytes > 0) rc = mem.device(static_cast<void**>(b.at), b.bytes);
    if (rc == 0) rc = mem.pinned(reinterpret_cast<void**>(&hcol), 2 * size_t(m_ + 1) * sizeof(double) + bb);
    if (rc == 0) rc = mem.event(&column);
    if (rc != 0) {
      release(mem);
      return rc;
    }
    n = n_;
    m = m_;
    s = s_;
    *fresh = true;
    return 0;
  }

  // The preconditioner's buffers: Np nodes per element, `op_values` operator entries,
  // `mask_values` face nodes.  *fresh: ops and fmask are not filled.
  int reserve_blocks(const SpaceMemory& mem, int Np, size_t op_values, size_t mask_values, bool* fresh) {
    *fresh = false;
    if (fmask) return 0;  // the last of the four
    release_blocks(mem);
    int rc = mem.device(reinterpret_cast<void**>(&minv), size_t(n) * size_t(Np) * sizeof(double));
    if (rc == 0) rc = mem.device(reinterpret_cast<void**>(&z), size_t(n) * sizeof(double));
    if (rc == 0) rc = mem.device(reinterpret_cast<void**>(&ops), op_values * sizeof(double));
    if (rc == 0) rc = mem.device(reinterpret_cast<void**>(&fmask), mask_values * sizeof(int));
    if (rc != 0) release_blocks(mem);
    else *fresh = true;
    return rc;
  }

  void release_blocks(const SpaceMemory& mem) {
    void* bufs[] = {minv, z, ops, fmask};
    for (void* p : bufs)
      if (p) mem.free_device(p);
    minv = z = ops = nullptr;
    fmask = nullptr;
    minv_dtg = 0;
  }

  void release(const SpaceMemory& mem) {
    release_blocks(mem);
    void* bufs[] = {u0, Y, base, RY, G, d, w, Yp, Rp, V, k, partial, hdev, zpart, step, npart, x32, r32, scratch,
                    geo_unit};
    for (void* p : bufs)
      if (p) mem.free_device(p);
    if (hcol) mem.free_pinned(hcol);
    if (column) mem.free_event(column);
    *this = ImplicitSpace();
  }
};

}  // namespace fedbm

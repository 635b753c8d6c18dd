// Kernels between the caller's canonical arrays and the internal state: encode
// (set_state), decode (get_state) and the node moments (get_moments).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fedbm {
namespace transfer {

// A weight in three FP32 pieces wh + wl + wll and its inverse in two, ih + il, in canonical
// order, with the velocity's internal index (see encode in transfer.cu).
struct alignas(16) DevRow {
  float wh, wl, ih, il;
};
struct alignas(8) DevIndex {
  float wll;
  int32_t at;
};
struct Weights {
  const DevRow* row = nullptr;      // [Q], device memory
  const DevIndex* index = nullptr;  // [Q]
  const double* wide = nullptr;     // [Q][2] w, 1/w
};
// The tables of Q canonical velocities from the weights in the internal order (host).
void weight_tables(const double* w, const int32_t* iperm, int Q, DevRow* row, DevIndex* index, double* wide);

// One case's slice of its group.
struct Shape {
  int store = 0;              // StoreKind
  int64_t K = 0;
  int Np = 0, Q = 0, Qp = 0;
  const double* vel64 = nullptr;   // [3][Qp] e_x, e_y, w in the internal order
  const int32_t* iperm = nullptr;  // [Q] internal index of canonical velocity c
  Weights weights;                 // deviation forms
  int nsm = 0;                     // SMs of the device and shared memory of one, bytes
  int smem_sm = 0;
};

// Once per state type and sizes, before the first of the calls below: lets their kernels
// take the shared memory that these sizes need.
cudaError_t prepare(const Shape& sh);

// canonical FP64 or FP32 [K][Np][Q] -> internal storage [K][Np][Qp] (padding
// velocities zero; deviation forms: the per-element scale too)
cudaError_t encode(const Shape& sh, const double* in, void* out, float* scale, cudaStream_t st);
cudaError_t encode(const Shape& sh, const float* in, void* out, float* scale, cudaStream_t st);

// internal state -> canonical FP64 [K][Np][Q]
cudaError_t decode(const Shape& sh, const void* in, const float* scale, double* out, cudaStream_t st);

// node moments rho, u_x, u_y [K][Np]; vel: the [kVelRows][Qp] table in the
// state's compute precision
cudaError_t moments(const Shape& sh, const void* in, const float* scale, const void* vel, double* rho, double* ux,
                    double* uy, cudaStream_t st);

}  // namespace transfer
}  // namespace fedbm

// Per-degree entry points of the fused stage kernel (one translation unit per
// polynomial degree, so the degrees compile in parallel).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

namespace fedbm {

struct StageEntry {
  // lanes: velocities per thread of the FP32-arithmetic kernels, 1 or 2
  cudaError_t (*launch)(int store_kind, const void* args, int lanes, int grid, int block, size_t smem, cudaStream_t st);
  cudaError_t (*set_smem)(int store_kind, int Qp, int lanes, size_t smem);
  cudaError_t (*upload)(const double* Dr, const double* Ds, const double* LIFT);
  int (*occupancy)(int store_kind, int Qp, int lanes, int block, size_t smem);  // resident CTAs per SM
  // tensor-core form (FP32, BF16 or FP16 state; 128, 256 or 1024 velocities;
  // one element per CTA)
  size_t (*tc_smem)(int store_kind, int Qp);  // dynamic shared memory; 0 = no such form
  int (*tc_tmem_cols)(int Qp);                 // tensor-memory columns per CTA
  cudaError_t (*launch_tc)(int store_kind, const void* args, int grid, size_t smem, cudaStream_t st);
  cudaError_t (*set_smem_tc)(int store_kind, int Qp, size_t smem);
  int (*occupancy_tc)(int store_kind, int Qp, size_t smem);
  // velocity-split form (a cluster of ncl CTAs per element tile; FP64, FP32,
  // BF16 state; Qp a multiple of 8 ncl)
  size_t (*cl_smem)(int store_kind, int Qp, int ncl, int epc);  // 0 = no such form
  cudaError_t (*launch_cl)(int store_kind, const void* args, int nclusters, int ncl, size_t smem, cudaStream_t st);
  cudaError_t (*set_smem_cl)(int store_kind, size_t smem);
  int (*occupancy_cl)(int store_kind, int ncl, size_t smem);  // resident clusters on the device
  // warp-specialised form (a producer warp filling a ring of element tiles for
  // groups of consumer warps; FP32 or BF16 state).  groups: 1 and 2 (the form asked
  // for by number) with 256 padded velocities at degree <= 5, 3 with 1,024 at degree
  // <= 3, 0 for the wide form, from 512 up at degree 1..5
  size_t (*ws_smem)(int store_kind, int Qp, int groups);  // 0 = no such form
  int (*ws_threads)(int store_kind, int Qp, int groups);
  cudaError_t (*launch_ws)(int store_kind, const void* args, int groups, int grid, size_t smem, cudaStream_t st);
  cudaError_t (*set_smem_ws)(int store_kind, int Qp, int groups, size_t smem);
  int (*occupancy_ws)(int store_kind, int Qp, int groups, size_t smem);  // resident CTAs per SM
};

StageEntry stage_entry_p0();
StageEntry stage_entry_p1();
StageEntry stage_entry_p2();
StageEntry stage_entry_p3();
StageEntry stage_entry_p4();
StageEntry stage_entry_p5();
StageEntry stage_entry_p6();

}  // namespace fedbm

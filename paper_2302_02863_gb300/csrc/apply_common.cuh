// Declarations shared by the FP64 apply (apply.cu) and its fixed-point form
// (apply_fixed.cu).
#pragma once

#include "device_common.cuh"

namespace vfd {

// apply.cu: node sums of columns [c0, c0 + cols), P64 -> xhat and ye64 -> yhat
void launch_far_sum(const MeshData &m, OpData &op, int c0, int cols, cudaStream_t st, const int *skip);
void launch_far_couple_sum(const MeshData &m, OpData &op, int c0, int cols, cudaStream_t st, const int *skip);
// apply_fixed.cu: Y = A X with the FP64 operator (OpData::fa)
void apply_fixed(const MeshData &m, OpData &op, const double *X, double *Y, int nrhs, int64_t ld, cudaStream_t st,
                 const int *skip, ApplyDot *dot);
// its kernels for groups of 8 columns from c0 on, ng groups, where `when` says so
struct FaWhen;
enum FaStep { FA_PROJ, FA_COUPLE, FA_NEAR, FA_EXPAND };
void apply_fixed_redo(FaStep step, const MeshData &m, OpData &op, const double *X, double *Y, int c0, int ng, int nrhs,
                      int64_t ld, cudaStream_t st, const FaWhen &when);
// apply_tensor.cu: the same for many columns
bool apply_tensor_fits(const MeshData &m, const OpData &op, int nrhs);
void apply_tensor_alloc(const MeshData &m, OpData &op);   // its workspace, on first use
void apply_tensor(const MeshData &m, OpData &op, const double *X, double *Y, int nrhs, int64_t ld, cudaStream_t st);

}  // namespace vfd

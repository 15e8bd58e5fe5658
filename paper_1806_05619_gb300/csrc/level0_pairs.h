// Level 0 of the mixed forms from FP32 pairs (level0_pairs.cu).
#pragma once

#include <cuda_runtime.h>

#include "fmg_device.cuh"

namespace mlqmc_level0 {

// Coarsest sides that the kernels are built for.
inline bool supported(int n0) { return n0 == 4 || n0 == 6 || n0 == 8 || n0 == 10; }

// Whether a call of B samples takes the kernel with four lanes per row.
bool four_lanes(int n0, int B);

// FP32 band factor, exact FP64 solution (u64, its FP32 copy in u) and F_0 of samples 0..B-1.
bool launch(const mlqmc_dev::FmgArgs& A, int n0, int B, cudaStream_t st);

}  // namespace mlqmc_level0

// Refinement residual with its norm for the converged mixed forms, without the
// FP64 pipe's sums (resnorm_words.cu).
#pragma once

#include <cuda_runtime.h>

#include "fmg_device.cuh"

namespace mlqmc_resnorm {

// Level sides the kernel takes: rows of whole 16-byte words in every array.
inline bool supported(int n) { return n % 4 == 0 && n >= 32; }

// Rows of a warp's strip (by the level alone, so that a sample's norm does not depend on its batch).
inline int rows(int n) { return n <= 256 ? 2 : 8; }

// Partial sums per sample (tiles of 128 columns and eight strips).
inline int chunks(int n) { return ((n + 127) / 128) * ((n + 8 * rows(n) - 1) / (8 * rows(n))); }

// bc = 1 - A u64 of level t (n cells per side) for samples 0..B-1 and
// part[i * chunks(n) + q] = the sum of its squares over tile q. active: null,
// or per-sample flags of the pass before; the bc and the partial sums of a
// sample whose flag is 0 are left as they are (its u64 has not changed since).
bool launch(const mlqmc_dev::FmgArgs& A, int t, int n, int B, double* part, const int* active, int sm_count,
            cudaStream_t st);

}  // namespace mlqmc_resnorm

// The small levels of the FMG (up to 64 cells per side) of a whole sample in
// one CTA's shared memory: a V-cycle's part below the large levels in one
// launch, and the FMG stages of the small levels in one launch.
#pragma once

#include <cuda_runtime.h>

#include "fmg_device.cuh"

namespace mlqmc_small {

constexpr int kMaxTop = 4;  // levels 1..4 (n0 = 4: 8, 16, 32, 64 cells per side)

// One level in the CTA's shared memory: offsets in elements of the working type.
struct Level {
    int n, lg;  // cells per side; log2 n where n0 is a power of two
    int oU, oB, oKx, oKy, oD;
    mlqmc_dev::FastDiv by_n, by_nc;
};

struct Plan {
    Level lv[kMaxTop + 1];
    int top;        // levels 1..top
    int oChol;      // band factor of level 0, by rows and by columns
    int oW;         // FMG stages: FP32 interpolant, or the FP64 solution (converged form)
    int stored_d;   // 1/D from the level's array (FP64; sides that the whole-sample smoother does not take)
    size_t bytes;   // dynamic shared memory
    int threads;
};

// What the FMG stages need beyond FmgArgs.
struct Stages {
    int i0;         // first sample of the launch
    int keep;       // every stage's solution is read later (solution output): write it to the pool
    double thresh;  // converged form: residual norm per cell side (rtol); 0: fixed cycles
    int max_iter;
    int* iters;     // converged form: iters[t] = most corrections beyond the first on level t
};

// Coarsest sides that the kernels are built for.
inline bool supported_n0(int n0) { return n0 == 4 || n0 == 6 || n0 == 8 || n0 == 10; }

// Largest level the kernels take (n <= 64 and, FP64, what shared memory holds); 0: none.
int top_level(int n0, int n_levels, bool fp64);

// Shared-memory plan for levels 1..top. stages: the FMG stages (conv: their converged form).
Plan make_plan(int n0, int top, bool fp64, bool stages, bool conv);

// Opt in to the shared memory (once per device).
bool prepare_f32();
bool prepare_f64();

// Levels top..0 of a V-cycle for samples 0..B-1: bc of level top in, u of level top out (from zero).
bool vcycle_f32(const mlqmc_dev::FmgArgs& A, const Plan& P, int B, cudaStream_t st);
bool vcycle_f64(const mlqmc_dev::FmgArgs& A, const Plan& P, int B, cudaStream_t st);

// FMG stages 1..top of samples S.i0..S.i0+count-1 (mixed forms; FP64 form with fixed cycles).
bool stages_f32(const mlqmc_dev::FmgArgs& A, const Plan& P, const Stages& S, int count, cudaStream_t st);
bool stages_f64(const mlqmc_dev::FmgArgs& A, const Plan& P, const Stages& S, int count, cudaStream_t st);

}  // namespace mlqmc_small

// Small-level FMG kernels of the FP64 form (fmg_small.cuh).
#include "fmg_small.cuh"

namespace mlqmc_small {

bool prepare_f64() { return prepare_all<double>(); }

bool vcycle_f64(const mlqmc_dev::FmgArgs& A, const Plan& P, int B, cudaStream_t st)
{
    return vcycle_launch<double>(A, P, B, st);
}

bool stages_f64(const mlqmc_dev::FmgArgs& A, const Plan& P, const Stages& S, int count, cudaStream_t st)
{
    return stages_launch<double, false>(A, P, S, count, st);
}

}  // namespace mlqmc_small

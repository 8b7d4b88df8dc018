// slater_common.cuh -- argument block and helpers shared by the Slater consumer's kernels
// (slater.cu, slater_reg.cu).
#pragma once

#include "eval_common.cuh"

namespace qmcspl {

constexpr int kSlaterMaxBlock = QMCSPL_SLATER_MAX_BLOCK;
constexpr int kSlaterRegMaxBlock = 128;   // spin blocks the register-resident kernel holds

struct SlaterArgs {
    const void* val;
    const void* grad;
    const void* lap;
    long long n_walkers;
    int n_elec, n_up, n_orb;
    double* logdet;
    double* sign;
    double* kinetic;
    double* drift;
    int arith;                // 0: FP64, 1: double-float
};

// The double-float consumer for spin blocks of at most kSlaterRegMaxBlock electrons: real
// orbitals, outputs of type double or float (slater_reg.cu).
int launch_slater_reg_f64(const SlaterArgs& a, int nmax, cudaStream_t st);
int launch_slater_reg_f32(const SlaterArgs& a, int nmax, cudaStream_t st);

namespace {

// 1 / d in double-float: one Newton step on the float reciprocal, e = 1 - d y to ~2^-48.
__device__ __forceinline__ dfloat df_recip(dfloat d)
{
    const float y = 1.0f / d.h;
    const float p = __fmul_rn(d.h, y);
    const float pe = fmaf(d.h, y, -p);                  // d.h y = p + pe exactly
    const float e = __fsub_rn(__fsub_rn(__fsub_rn(1.0f, p), pe), __fmul_rn(d.l, y));
    return df_norm(y, __fmul_rn(y, e));
}

}  // namespace
}  // namespace qmcspl

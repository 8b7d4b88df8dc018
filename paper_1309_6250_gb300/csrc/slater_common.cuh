// slater_common.cuh -- argument block and helpers shared by the Slater consumer's kernels
// (slater.cu, slater_reg.cu, slater_creg.cu).
#pragma once

#include "eval_common.cuh"

namespace qmcspl {

constexpr int kSlaterMaxBlock = QMCSPL_SLATER_MAX_BLOCK;
constexpr int kSlaterRegMaxBlock = 128;   // spin blocks the register-resident kernels hold: real ...
constexpr int kSlaterCregMaxBlock = 96;   // ... and complex orbitals

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
    int stall;                // test hook: column 0 of the first walker's first block is never announced
};

// The double-float consumer for spin blocks of at most kSlaterRegMaxBlock electrons: real
// orbitals, outputs of type double or float (slater_reg.cu).
int launch_slater_reg_f64(const SlaterArgs& a, int nmax, cudaStream_t st);
int launch_slater_reg_f32(const SlaterArgs& a, int nmax, cudaStream_t st);
// The same for complex orbitals and at most kSlaterCregMaxBlock electrons (slater_creg.cu).
int launch_slater_creg_f64(const SlaterArgs& a, int nmax, cudaStream_t st);
int launch_slater_creg_f32(const SlaterArgs& a, int nmax, cudaStream_t st);
// Address of each file's device word, set by a walker whose waits ran out.
cudaError_t slater_reg_timeout_word(void** p);
cudaError_t slater_creg_timeout_word(void** p);

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

// (h, l) <- h + l with |l| <= ulp(h) / 2.  Three operations do what the full two-sum does: h is a
// sum whose terms cancel only to a multiple of their last place, so it is 0 or no smaller than about l.
__device__ __forceinline__ void quick_norm2(f32x2& h, f32x2& l)
{
    const f32x2 s = add2(h, l);
    l = sub2(l, sub2(s, h));
    h = s;
}

// (H, L) -= f r for a row's multiplier f = (fh, fh), (fl, fl) and a column pair of the pivot row as
// (rh0, rh1), its negative and the negative of (rl0, rl1): df_fma2's steps, after which an entry is
// renormalised (entries are updated n times and reused as pivots, multipliers and reciprocals, which
// assume |lo| << |hi|).
__device__ __forceinline__ void submul2(f32x2& H, f32x2& L, f32x2 fh, f32x2 fl, f32x2 rh, f32x2 nrh, f32x2 nrl)
{
    const f32x2 P = mul2(fh, rh);
    f32x2 E = ffma2(fh, nrh, P);
    E = ffma2(fh, nrl, E);
    E = ffma2(fl, nrh, E);
    const f32x2 S = sub2(H, P);
    const f32x2 BB = sub2(S, H);
    const f32x2 T1 = sub2(H, sub2(S, BB));
    const f32x2 T2 = add2(P, BB);
    L = add2(L, add2(sub2(T1, T2), E));
    H = S;
}

// the same with a renormalisation
__device__ __forceinline__ void eliminate2(f32x2& H, f32x2& L, f32x2 fh, f32x2 fl, f32x2 rh, f32x2 nrh, f32x2 nrl)
{
    submul2(H, L, fh, fl, rh, nrh, nrl);
    quick_norm2(H, L);
}

// Sixteen sums over the warp at once: lane l gets the total of s[l >> 1], added up in the order of a
// butterfly over lane distances 16, 8, 4, 2, 1.  Each exchange halves the sums a lane still carries, so
// the sixteen cost 16 FP64 additions instead of 80.
__device__ __forceinline__ double warp_sum16(double (&s)[16])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 8; h > 0; h >>= 1) {
        const bool up = (lane & (2 * h)) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
            const double keep = up ? s[q + h] : s[q], give = up ? s[q] : s[q + h];
            s[q] = keep + __shfl_xor_sync(kFullMask, give, 2 * h);
        }
    }
    return s[0] + __shfl_xor_sync(kFullMask, s[0], 1);
}

__device__ __forceinline__ void split(float v, float& h, float& l)
{
    h = v;
    l = 0.0f;
}
__device__ __forceinline__ void split(double v, float& h, float& l)
{
    const dfloat d = df_from_double(v);
    h = d.h;
    l = d.l;
}

// ---- mbarriers (one arrival each, never reused; the test hook's barrier expects a second one) ----
__device__ __forceinline__ void mbar_init(uint64_t* bar, int arrivals)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(bar)), "r"(arrivals)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"((unsigned)__cvta_generic_to_shared(bar)) : "memory");
}
// Waits for the arrival: false if it did not come within half a second and kWaitTries tries (about 4 us each;
// a column takes a few).  The tries count only while this warp runs: the clock alone would also count time
// in which the device runs something else.  (Tries without the clock cost blocks of up to 32 electrons 5 %.)
constexpr int kWaitTries = 1 << 17;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
    long long t0 = 0;
    for (int i = 0;; ++i) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(a)
                     : "memory");
        if (done) return true;
        if (i == 0) t0 = clock64();
        else if (clock64() - t0 > (1LL << 30) && i >= kWaitTries) return false;
    }
}

}  // namespace
}  // namespace qmcspl

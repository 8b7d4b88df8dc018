// slater_creg.cu -- the double-float Slater consumer with the matrix in registers, for complex (Bloch)
// orbitals and spin blocks of at most 96 electrons.  The quantities are those of slater.cu's header,
// the scheme that of slater_reg.cu: columns dealt out over the warps, no barrier in the elimination,
// the pivot column and 1 / pivot through shared memory with an mbarrier per column.
//
// What bounds it: a complex update is four error-free multiply-adds and two renormalisations, 54
// packed FP32 operations per two entries: 64 x 64 blocks need 2,048 x 54 / 64 = 1,728 SM clocks per
// elimination step.  slater_cdf_kernel, which it replaces here, moves 32 bytes of shared memory per
// entry and step and meets at four barriers.  The final sums are FP64 here as there (two operations per
// SM clock): as double-float sums they had 1.03 to 1.10 times the drift's rms error and not the range of a
// double.  Measured, 4,096 walkers x (64 + 64), complex float orbitals 10.18 -> 5.25 ms (5.56 with double-float
// sums), complex double 9.57 -> 5.39; 4,096 x (32 + 32) 3.49 -> 0.95 ms (0.92), 4,096 x (12 + 11) 1.35 -> 0.41
// (0.40), 1,024 x (96 + 96) 12.1 -> 5.42 (4.52).
//
// A lane keeps RL rows of CP column pairs, each as four packed pairs (re and im, high and low): 64
// registers, 72 for 65 to 96 electrons.  97 to 112 electrons would need 98 of 128 and stay with
// slater_cdf_kernel.
#include <cooperative_groups.h>

#include "slater_common.cuh"

namespace qmcspl {
namespace {

namespace cg = cooperative_groups;

__device__ int timed_out;   // read and cleared by qmcspl_slater_sync

// G: spin blocks of at most 32 G electrons; see RegShape in slater_reg.cu
template <int G> struct CregShape;
template <> struct CregShape<1> { static constexpr int RL = 1, CP = 8, NW = 2, per_sm = 8; };
template <> struct CregShape<2> { static constexpr int RL = 2, CP = 4, NW = 8, per_sm = 2; };
template <> struct CregShape<3> { static constexpr int RL = 3, CP = 3, NW = 16, per_sm = 1; };

struct CplxEntry2 {          // two columns' entries
    f32x2 rh, rl, ih, il;
};
struct CplxResult {
    double logdet, arg, kin_re, kin_im;
    int singular;
    int stuck;               // a wait ran out: every output of the walker is NaN
};

// a scaled row's column pair: (re h, -re h, -re l), (im h, -im h, im l, -im l)
struct __align__(16) CplxRow2 {
    float re[3][2], pad[2], im[4][2];
};

// X -= f r for a row's complex multiplier f, in slater_cdf_kernel's order: re -= f.re r.re,
// re += f.im r.im, im -= f.re r.im, im -= f.im r.re, both parts renormalised
__device__ __forceinline__ void eliminate_cplx(CplxEntry2& X, float4 f, const CplxRow2& row)
{
    const float4* q = reinterpret_cast<const float4*>(&row);
    const float4 q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3];
    const f32x2 rh = pack2(q0.x, q0.y), nrh = pack2(q0.z, q0.w), nrl = pack2(q1.x, q1.y);
    const f32x2 ih = pack2(q2.x, q2.y), nih = pack2(q2.z, q2.w), il = pack2(q3.x, q3.y), nil = pack2(q3.z, q3.w);
    const f32x2 frh = pack2(f.x, f.x), frl = pack2(f.y, f.y), fih = pack2(f.z, f.z), fil = pack2(f.w, f.w);
    submul2(X.rh, X.rl, frh, frl, rh, nrh, nrl);
    submul2(X.rh, X.rl, fih, fil, nih, ih, il);
    submul2(X.ih, X.il, frh, frl, ih, nih, nil);
    submul2(X.ih, X.il, fih, fil, rh, nrh, nrl);
    quick_norm2(X.rh, X.rl);
    quick_norm2(X.ih, X.il);
}

template <typename T, int G>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(32 * CregShape<G>::NW, CregShape<G>::per_sm)
    slater_creg_kernel(const SlaterArgs a, const long long w0)
{
    constexpr int RL = CregShape<G>::RL, CP = CregShape<G>::CP, NW = CregShape<G>::NW;
    constexpr int N = 32 * RL, NT = 32 * NW, CW = 2 * CP;
    static_assert(CW * NW == N && CW <= 32, "the warps cover the columns, a lane scales one of them");
    constexpr int ld = N + 1;                       // row stride of the inverse in shared memory
    // during the elimination column k's multipliers (re h, re l, im h, im l), xt[k * N + row]; then the
    // inverse by electron, xt[i * ld + j]
    extern __shared__ float4 xct[];
    __shared__ __align__(8) uint64_t ready[N];      // column k and its pivot are written
    __shared__ __align__(16) float4 pinv[N];        // 1 / pivot (re h, re l, im h, im l)
    __shared__ __align__(16) float4 xrow[NW][CW];   // per warp: its part of the pivot row ...
    __shared__ CplxRow2 row[NW][CP];                // ... and scaled
    __shared__ int piv[N], step_of[N];              // pivot row of step k (-1: singular)
    __shared__ double2 pivd[N];
    __shared__ int parity;
    __shared__ double red[NW];
    __shared__ CplxResult mine;

    cg::cluster_group cluster = cg::this_cluster();
    const int spin = blockIdx.x & 1;
    const long long w = w0 + (blockIdx.x >> 1);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int e0 = spin == 0 ? 0 : a.n_up;
    const int n = spin == 0 ? a.n_up : a.n_elec - a.n_up;
    const long long base = w * a.n_elec + e0;       // first position of the block
    const long long O = a.n_orb;
    if (tid == 0) parity = 0;
    for (int k = tid; k < N; k += NT) mbar_init(ready + k, a.stall && k == 0 && w == 0 && spin == 0 ? 2 : 1);

    CplxEntry2 X[RL][CP];                           // [row lane + 32 i][column pair]
    {
        const T* v = static_cast<const T*>(a.val);
#pragma unroll
        for (int i = 0; i < RL; ++i)
#pragma unroll
            for (int m = 0; m < CP; ++m) {
                float h[2][2] = {}, l[2][2] = {};   // [column][re, im]
                const int r = lane + 32 * i;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int c = wid + NW * (2 * m + q);
                    if (r < n && c < n) {
                        const T* z = v + 2 * ((base + r) * O + c);
                        split(__ldg(z), h[q][0], l[q][0]);
                        split(__ldg(z + 1), h[q][1], l[q][1]);
                    }
                }
                X[i][m] = {pack2(h[0][0], h[1][0]), pack2(l[0][0], l[1][0]), pack2(h[0][1], h[1][1]), pack2(l[0][1], l[1][1])};
            }
    }
    unsigned used = 0;                              // bit i: row lane + 32 i is a pivot row already (or past n)
#pragma unroll
    for (int i = 0; i < RL; ++i) used |= (lane + 32 * i >= n ? 1u : 0u) << i;

    // column q of the pair
    auto entry = [](const CplxEntry2& x, int q) __attribute__((always_inline)) {
        float r0, r1, s0, s1, i0, i1, j0, j1;
        unpack2(x.rh, r0, r1);
        unpack2(x.rl, s0, s1);
        unpack2(x.ih, i0, i1);
        unpack2(x.il, j0, j1);
        return q ? make_float4(r1, s1, i1, j1) : make_float4(r0, s0, i0, j0);
    };
    // Called by the warp that holds column k: finds the pivot row (the largest |entry|^2 of the high
    // parts, the lowest row among equals, a NaN only where nothing else is left), writes the column and
    // 1 / pivot for step k.
    auto publish = [&](int k, const float4 (&z)[RL]) __attribute__((always_inline)) {
        unsigned key = 0;
        int p = 0;
        float4 d = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            xct[k * N + lane + 32 * i] = z[i];
            const float v = fmaf(z[i].x, z[i].x, z[i].z * z[i].z);
            const unsigned q = ((used >> i) & 1u) ? 0u : v == v ? __float_as_uint(v) + 2u : 1u;
            if (q > key) {
                key = q;
                p = lane + 32 * i;
                d = z[i];
            }
        }
        const unsigned top = __reduce_max_sync(kFullMask, key);
        const int prow = (int)__reduce_min_sync(kFullMask, key == top ? (unsigned)p : 0x7fffffffu);
        if (key == top && p == prow) {
            const dfloat dr = {d.x, d.y}, di = {d.z, d.w};
            const dfloat rm = df_recip(df_add(df_mul(dr, dr), df_mul(di, di)));
            const dfloat ir = df_mul(dr, rm), ii = df_neg(df_mul(di, rm));
            pinv[k] = make_float4(ir.h, ir.l, ii.h, ii.l);
            piv[k] = d.x == 0.0f && d.z == 0.0f ? -1 : prow;
            pivd[k] = make_double2((double)d.x + (double)d.y, (double)d.z + (double)d.w);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(ready + k);
    };
    // column q of the pair becomes 0
    auto clear = [](CplxEntry2& x, bool z0, bool z1) __attribute__((always_inline)) {
        f32x2* e[4] = {&x.rh, &x.rl, &x.ih, &x.il};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            float v0, v1;
            unpack2(*e[t], v0, v1);
            *e[t] = pack2(z0 ? 0.0f : v0, z1 ? 0.0f : v1);
        }
    };
    __syncthreads();                                // the barriers are initialised
    if (n > 0 && wid == 0) {
        float4 z[RL];
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            z[i] = entry(X[i][0], 0);
            clear(X[i][0], true, false);
        }
        publish(0, z);
    }

    int fail = 0;                                   // 1: singular, 2: a wait ran out
#pragma unroll 1
    for (int k = 0; k < n && wid < n; ++k) {
        const bool there = mbar_wait(ready + k);
        __syncwarp();                               // (step k - 1's row is read by all lanes)
        const int p = piv[k];
        if (!there) fail = 2;                       // (nothing is known about piv[k])
        else if (p < 0) fail = 1;                   // exactly singular
        if (__any_sync(kFullMask, fail)) break;
        const bool mine_row = lane == (p & 31);
#pragma unroll
        for (int i = 0; i < RL; ++i)
            if (mine_row && i == (p >> 5)) used |= 1u << i;
        // ---- this warp's part of the pivot row; the holder's copy becomes 0 ----
        // (one branch per row of the lane, each with its own registers)
        auto take = [&](CplxEntry2(&x)[CP]) __attribute__((always_inline)) {
            if (!mine_row) return;
#pragma unroll
            for (int m = 0; m < CP; ++m) {
                xrow[wid][2 * m] = entry(x[m], 0);
                xrow[wid][2 * m + 1] = entry(x[m], 1);
                x[m] = {0ull, 0ull, 0ull, 0ull};
            }
        };
        switch (p >> 5) {
        case 0: take(X[0]); break;
        case 1: take(X[RL > 1 ? 1 : 0]); break;
        default: take(X[RL > 2 ? 2 : 0]); break;
        }
        // the multiplier of this lane's row i; the pivot row's own is -1
        auto multiplier = [&](int i) __attribute__((always_inline)) {
            return mine_row && i == (p >> 5) ? make_float4(-1.0f, 0.0f, 0.0f, 0.0f) : xct[k * N + lane + 32 * i];
        };
        __syncwarp();
        if (lane < CW) {                            // entry k, whose column is 0 now, becomes 1 / pivot
            const float4 x = wid + NW * lane == k ? make_float4(1.0f, 0.0f, 0.0f, 0.0f) : xrow[wid][lane];
            const float4 v = pinv[k];
            const dfloat xr = {x.x, x.y}, xi = {x.z, x.w}, ir = {v.x, v.y}, ii = {v.z, v.w};
            const dfloat zr = df_add(df_mul(xr, ir), df_neg(df_mul(xi, ii)));
            const dfloat zi = df_add(df_mul(xr, ii), df_mul(xi, ir));
            CplxRow2& r = row[wid][lane >> 1];
            const int q = lane & 1;
            r.re[0][q] = zr.h;
            r.re[1][q] = -zr.h;
            r.re[2][q] = -zr.l;
            r.im[0][q] = zi.h;
            r.im[1][q] = -zi.h;
            r.im[2][q] = zi.l;
            r.im[3][q] = -zi.l;
        }
        __syncwarp();
        const int nc = (k + 1) / NW;                // column k + 1 among its warp's columns
        const bool next_here = k + 1 < n && (k + 1) % NW == wid;
        if (next_here) {
            // the pair with column k + 1, updated ahead of the others (and again with them below);
            // bitwise selects: an index would put the matrix in local memory
            float4 z[RL];
#pragma unroll
            for (int i = 0; i < RL; ++i) {
                CplxEntry2 x = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                for (int m = 0; m < CP; ++m) {
                    const f32x2 mask = m == (nc >> 1) ? ~0ull : 0ull;
                    x.rh |= X[i][m].rh & mask;
                    x.rl |= X[i][m].rl & mask;
                    x.ih |= X[i][m].ih & mask;
                    x.il |= X[i][m].il & mask;
                }
                eliminate_cplx(x, multiplier(i), row[wid][nc >> 1]);
                z[i] = entry(x, nc & 1);
            }
            publish(k + 1, z);
        }
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const float4 f = multiplier(i);
#pragma unroll
            for (int m = 0; m < CP; ++m) eliminate_cplx(X[i][m], f, row[wid][m]);
        }
        if (next_here) {
            // column k + 1 becomes 0, so that its step leaves -f_i / pivot there
#pragma unroll
            for (int i = 0; i < RL; ++i)
#pragma unroll
                for (int m = 0; m < CP; ++m) clear(X[i][m], nc == 2 * m, nc == 2 * m + 1);
        }
    }

    double kin_re = 0.0, kin_im = 0.0;
    const bool sing = __syncthreads_or(fail) != 0;
    const bool stuck = __syncthreads_or(fail == 2) != 0;
    if (n > 0 && !sing) {
        for (int k = tid; k < n; k += NT) step_of[piv[k]] = k;
        __syncthreads();
        // the inverse by electron (column p_j) and orbital (row step_of[i])
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const int r = lane + 32 * i;
            if (r >= n) continue;
            const int o = step_of[r];
#pragma unroll
            for (int m = 0; m < CP; ++m) {
                const int c = wid + NW * 2 * m;
                if (c < n) xct[piv[c] * ld + o] = entry(X[i][m], 0);
                if (c + NW < n) xct[piv[c + NW] * ld + o] = entry(X[i][m], 1);
            }
        }
        // the inversions of k -> p_k, modulo two
        int odd = 0;
        for (int t = tid; t < n * G; t += NT) {     // G threads per step, a G-th of the steps each
            const int k = t / G, part = t - k * G, pk = piv[k];
            for (int m = k + 1 + part; m < n; m += G) odd ^= piv[m] < pk;
        }
        odd = __reduce_xor_sync(kFullMask, odd);
        if (lane == 0 && odd) atomicXor(&parity, 1);
        __syncthreads();
        // T = -1/2 sum_ij X_ji lap phi_j(r_i) and the drift, in FP64 (inverse entries h + l): two electrons
        // per warp at a time, lanes 16 e + 4 c + 2 r and the next getting sum c (r = 0 re, 1 im) of electron e
        const bool want_g = a.drift != nullptr, want_l = a.kinetic != nullptr;
        if (want_g || want_l) {
            const T* gp = static_cast<const T*>(a.grad);
            const T* lp = static_cast<const T*>(a.lap);
            for (int i0 = 2 * wid; i0 < n; i0 += 2 * NW) {
                double s[16];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int i = i0 + e;
#pragma unroll
                    for (int c = 0; c < 8; ++c) s[8 * e + c] = 0.0;
#pragma unroll
                    for (int t = 0; t < RL; ++t) {
                        const int j = lane + 32 * t;
                        if (i >= n || j >= n) continue;
                        const float4 x = xct[i * ld + j];
                        const double xr = (double)x.x + (double)x.y, xi = (double)x.z + (double)x.w;
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            if (c < 3 ? !want_g : !want_l) continue;
                            const T* z = c < 3 ? gp + 2 * (((base + i) * 3 + c) * O + j) : lp + 2 * ((base + i) * O + j);
                            const double zr = __ldg(z), zi = __ldg(z + 1);
                            double &sr = s[8 * e + 2 * c], &si = s[8 * e + 2 * c + 1];
                            sr = fma(xr, zr, fma(-xi, zi, sr));
                            si = fma(xr, zi, fma(xi, zr, si));
                        }
                    }
                }
                const double sum = warp_sum16(s);
                const int i = i0 + (lane >> 4), c = (lane >> 2) & 3, r = (lane >> 1) & 1;
                if (lane & 1) continue;
                if (c == 3) (r ? kin_im : kin_re) += sum;
                else if (want_g && i < n) a.drift[2 * ((base + i) * 3 + c) + r] = sum;
            }
        }
    }
    // ---- the block's sums, then the walker's through the cluster ----
    double part_ld = 0.0, part_arg = 0.0;
    if (!sing)
        for (int k = tid; k < n; k += NT) {
            const double2 z = pivd[k];
            part_ld += 0.5 * log(fma(z.x, z.x, z.y * z.y));
            part_arg += atan2(z.y, z.x);
        }
    auto block_sum = [&](double v) {
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFullMask, v, off);
        __syncthreads();
        if (lane == 0) red[wid] = v;
        __syncthreads();
        double t = 0.0;
        if (tid == 0)
            for (int q = 0; q < NW; ++q) t += red[q];
        return t;
    };
    const double logdet = block_sum(part_ld), phase = block_sum(part_arg);
    const double kr = block_sum(kin_re), ki = block_sum(kin_im);
    if (tid == 0) mine = {logdet, phase + (parity ? M_PI : 0.0), -0.5 * kr, -0.5 * ki, sing ? 1 : 0, stuck ? 1 : 0};
    cluster.sync();
    const CplxResult other = *cluster.map_shared_rank(&mine, spin ^ 1);
    const bool singular = sing || other.singular;
    const bool lost = stuck || other.stuck;
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    const double inf = __longlong_as_double(0x7ff0000000000000LL);
    if (spin == 0 && tid == 0) {
        if (lost) timed_out = 1;
        if (a.logdet) a.logdet[w] = lost ? nan : singular ? -inf : mine.logdet + other.logdet;
        if (a.sign) {
            double sn, cs;
            sincos(mine.arg + other.arg, &sn, &cs);
            a.sign[2 * w] = lost ? nan : singular ? 0.0 : cs;
            a.sign[2 * w + 1] = lost ? nan : singular ? 0.0 : sn;
        }
        if (a.kinetic) {
            a.kinetic[2 * w] = singular ? nan : mine.kin_re + other.kin_re;
            a.kinetic[2 * w + 1] = singular ? nan : mine.kin_im + other.kin_im;
        }
    }
    if (singular && a.drift)
        for (int e = tid; e < 6 * n; e += NT) a.drift[base * 6 + e] = nan;
    cluster.sync();   // the other CTA may still be reading `mine`
}

template <typename T, int G>
int launch_shape(const SlaterArgs& a, cudaStream_t st)
{
    using R = CregShape<G>;
    auto k = slater_creg_kernel<T, G>;
    constexpr int smem = sizeof(float4) * 32 * G * (32 * G + 1);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(slater_creg_kernel)");
    constexpr long long kMaxWalkers = 1LL << 29;    // per launch: two CTAs each, within the grid limit
    for (long long w0 = 0; w0 < a.n_walkers; w0 += kMaxWalkers) {
        const long long m = a.n_walkers - w0 < kMaxWalkers ? a.n_walkers - w0 : kMaxWalkers;
        k<<<(unsigned)(2 * m), 32 * R::NW, smem, st>>>(a, w0);
        const int rc = cuda_error(cudaGetLastError(), "slater_creg_kernel launch");
        if (rc != QMCSPL_OK) return rc;
    }
    return QMCSPL_OK;
}

template <typename T>
int launch_typed(const SlaterArgs& a, int nmax, cudaStream_t st)
{
    if (nmax <= 32) return launch_shape<T, 1>(a, st);
    if (nmax <= 64) return launch_shape<T, 2>(a, st);
    return launch_shape<T, 3>(a, st);
}

}  // namespace

cudaError_t slater_creg_timeout_word(void** p) { return cudaGetSymbolAddress(p, timed_out); }

int launch_slater_creg_f64(const SlaterArgs& a, int nmax, cudaStream_t st) { return launch_typed<double>(a, nmax, st); }
int launch_slater_creg_f32(const SlaterArgs& a, int nmax, cudaStream_t st) { return launch_typed<float>(a, nmax, st); }

}  // namespace qmcspl

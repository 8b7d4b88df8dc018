// slater_reg.cu -- the double-float Slater consumer with the matrix in registers (real orbitals,
// spin blocks of at most 128 electrons).  The quantities are those of slater.cu's header.
//
// What bounds it: every one of the n^3 elimination updates is an error-free multiply-add of float
// pairs (15 packed FP32 operations per two entries, two cycles each), so the FP32 pipe is the floor:
// 128 x 128 blocks need 16,384 x 15 / 128 = 1,920 SM clocks per elimination step.  The kernel it
// replaces kept the matrix in shared memory, where each update also read and wrote 16 bytes, and met
// at four barriers per step: 14.29 ms for 2,048 walkers x (128 + 128) electrons.  Here the matrix
// never leaves the registers and the warps meet at no barrier: 6.79 ms.  Of that about 1 ms is the final
// sums, which stay FP64 (two operations per SM clock): as double-float sums on the FP32 pipe they left
// 5.87 ms, but the drift's rms error against 64 bits was 1.03 (128 electrons) to 1.18 times (12) as large,
// a double's last bits were lost and an infinite gradient gave NaN.  64 + 64 electrons: 2.90 -> 0.88 ms,
// 96 + 96: 6.08 -> 2.50 ms (2,048 walkers); 8 + 8: 0.62 -> 0.14 ms, 32 + 32: 2.24 -> 0.43 ms (4,096);
// double orbitals, 128 + 128: 13.73 -> 6.63 ms.
// Also measured, 128 + 128: 32 x 32 tiles per warp, the pivot row and column through shared memory
// and two barriers per step 7.4 ms (each step's search and scaling lay between the updates, and the
// few lanes that do them compete with the other warps' updates); columns owned by warps in blocks,
// one barrier, 7.2 ms (the holder of the next column is late at every step; dealt out in turn, the
// holders change and nobody waits long).
//
// Work mapping.  One CTA per spin block, the two blocks of a walker in a cluster of two CTAs that
// exchange ln|det|, sign and kinetic energy at the end.  Warp w of NW owns the columns w, w + NW, ...,
// a lane the rows lane + 32 i of them, as float pairs packed by column pair: 64 registers (72 for 65
// to 96 electrons, 32 for up to 32).  So column k lies in one warp, which finds the pivot among its
// own lanes, and a row's entries for a warp's columns lie in one of its lanes: only the pivot column
// (the multipliers) and the pivot itself cross between warps, through a place of their own per
// column in shared memory, with an mbarrier each.  128 electrons fill an SM's register file with one
// CTA; the smaller shapes run two, four or twelve CTAs per SM.
//
// A step k of the Gauss-Jordan elimination, in each warp once column k is written:
//   its part of pivot row p (rows are not swapped, p is recorded) goes from the lane that holds it to
//     shared memory, is scaled by 1 / pivot, one column per lane, and read back by all lanes; the
//     holder's copy becomes 0 and the row's own multiplier -1;
//   the warp that holds column k + 1 brings that column up to date first, finds the next pivot (the
//     largest |entry| over rows not yet used) and writes the column and 1 / pivot;
//   every lane updates its entries.
// The updates are slater_df_kernel's error-free multiply-adds on the same operands; the renormalisation takes
// three operations (quick_norm2) instead of a full two-sum, to the same result.
// After n steps entry (i, j) is the inverse's row (step at which i was the pivot), column p_j.
#include <cooperative_groups.h>

#include "slater_common.cuh"

namespace qmcspl {
namespace {

namespace cg = cooperative_groups;

__device__ int timed_out;   // read and cleared by qmcspl_slater_sync

// RL rows per lane, CP column pairs per lane, NW warps; `per_sm` CTAs fit on an SM with at most 85 registers
// per thread for G = 1 (the compiler takes 80) and 128 for the others.  G: spin blocks of at most 32 G electrons.
template <int G> struct RegShape;
template <> struct RegShape<1> { static constexpr int RL = 1, CP = 8, NW = 2, per_sm = 12; };
template <> struct RegShape<2> { static constexpr int RL = 2, CP = 8, NW = 4, per_sm = 4; };
template <> struct RegShape<3> { static constexpr int RL = 3, CP = 6, NW = 8, per_sm = 2; };
template <> struct RegShape<4> { static constexpr int RL = 4, CP = 4, NW = 16, per_sm = 1; };

struct BlockResult {
    double logdet, kin;
    int odd;         // determinant negative
    int singular;
    int stuck;       // a wait ran out: every output of the walker is NaN
};

template <typename T, int G>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(32 * RegShape<G>::NW, RegShape<G>::per_sm)
    slater_reg_kernel(const SlaterArgs a, const long long w0)
{
    constexpr int RL = RegShape<G>::RL, CP = RegShape<G>::CP, NW = RegShape<G>::NW;
    constexpr int N = 32 * RL, NT = 32 * NW, CW = 2 * CP;
    static_assert(CW * NW == N && CW <= 32, "the warps cover the columns, a lane scales one of them");
    constexpr int ld = N + 1;                       // row stride of the inverse in shared memory
    // during the elimination column k's multipliers (h, l), xt[k * N + row]; then the inverse by
    // electron, xt[i * ld + j]
    extern __shared__ float2 xt[];
    __shared__ __align__(8) uint64_t ready[N];      // column k and its pivot are written
    __shared__ __align__(16) float4 ctrl[N];        // pivot row (< 0: singular), 1 / pivot (h, l)
    __shared__ __align__(8) float xrow[NW][2][CW];  // per warp: its part of the pivot row (h, l) ...
    __shared__ __align__(16) float rowh[NW][CP][4]; // ... and scaled: (r_h0, r_h1, -r_h0, -r_h1)
    __shared__ __align__(8) float rowl[NW][CP][2];  // (-r_l0, -r_l1)
    __shared__ int piv[N], step_of[N];
    __shared__ float2 pivd[N];
    __shared__ int parity;
    __shared__ double red[NW];
    __shared__ BlockResult mine;

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

    f32x2 H[RL][CP], L[RL][CP];                     // [row lane + 32 i][column pair]
    {
        const T* v = static_cast<const T*>(a.val);
#pragma unroll
        for (int i = 0; i < RL; ++i)
#pragma unroll
            for (int m = 0; m < CP; ++m) {
                float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
                const int r = lane + 32 * i, c = wid + NW * 2 * m;
                if (r < n) {
                    if (c < n) split(__ldg(v + (base + r) * O + c), h0, l0);
                    if (c + NW < n) split(__ldg(v + (base + r) * O + c + NW), h1, l1);
                }
                H[i][m] = pack2(h0, h1);
                L[i][m] = pack2(l0, l1);
            }
    }
    unsigned used = 0;                              // bit i: row lane + 32 i is a pivot row already (or past n)
#pragma unroll
    for (int i = 0; i < RL; ++i) used |= (lane + 32 * i >= n ? 1u : 0u) << i;

    // Called by the warp that holds column k, its entries in (h, l): finds the pivot row (the lowest row
    // among equals, a NaN only where nothing else is left), writes the column and 1 / pivot for step k.
    // Every column has a place of its own, so nobody has to wait before writing.
    auto publish = [&](int k, const float (&h)[RL], const float (&l)[RL]) __attribute__((always_inline)) {
        unsigned key = 0;
        int p = 0;
        float dh = 0.0f, dl = 0.0f;
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            xt[k * N + lane + 32 * i] = make_float2(h[i], l[i]);
            const float v = fabsf(h[i]);
            const unsigned q = ((used >> i) & 1u) ? 0u : v == v ? __float_as_uint(v) + 2u : 1u;
            if (q > key) {
                key = q;
                p = lane + 32 * i;
                dh = h[i];
                dl = l[i];
            }
        }
        const unsigned top = __reduce_max_sync(kFullMask, key);
        const int row = (int)__reduce_min_sync(kFullMask, key == top ? (unsigned)p : 0x7fffffffu);
        if (key == top && p == row) {
            const dfloat inv = df_recip({dh, dl});
            ctrl[k] = make_float4(__int_as_float(dh == 0.0f ? -1 : row), inv.h, inv.l, 0.0f);
            piv[k] = row;
            pivd[k] = make_float2(dh, dl);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(ready + k);
    };
    __syncthreads();                                // the barriers are initialised
    if (n > 0 && wid == 0) {
        float h[RL], l[RL], other;
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            unpack2(H[i][0], h[i], other);
            H[i][0] = pack2(0.0f, other);
            unpack2(L[i][0], l[i], other);
            L[i][0] = pack2(0.0f, other);
        }
        publish(0, h, l);
    }

    // The warps run freely, each waiting only for the column it needs next: the holder of column k + 1
    // (the next warp: columns are dealt out in turn) writes it while the others are still in step k.
    int fail = 0;                                   // 1: singular, 2: a wait ran out
#pragma unroll 1
    for (int k = 0; k < n && wid < n; ++k) {
        const bool there = mbar_wait(ready + k);
        __syncwarp();                               // (step k - 1's row is read by all lanes)
        const float4 ct = ctrl[k];
        const int p = __float_as_int(ct.x);
        if (!there) fail = 2;                       // (nothing is known about ctrl[k])
        else if (p < 0) fail = 1;                   // exactly singular
        if (__any_sync(kFullMask, fail)) break;
        const bool mine_row = lane == (p & 31);
#pragma unroll
        for (int i = 0; i < RL; ++i)
            if (mine_row && i == (p >> 5)) used |= 1u << i;
        // ---- this warp's part of the pivot row; the holder's copy becomes 0 ----
        // (one branch per row of the lane, each with its own registers: an index by p would put the
        // matrix in local memory)
        auto take = [&](f32x2(&h)[CP], f32x2(&l)[CP]) __attribute__((always_inline)) {
            if (!mine_row) return;
#pragma unroll
            for (int m = 0; m < CP; ++m) {
                *reinterpret_cast<f32x2*>(&xrow[wid][0][2 * m]) = h[m];
                *reinterpret_cast<f32x2*>(&xrow[wid][1][2 * m]) = l[m];
                h[m] = l[m] = 0ull;
            }
        };
        switch (p >> 5) {
        case 0: take(H[0], L[0]); break;
        case 1: take(H[RL > 1 ? 1 : 0], L[RL > 1 ? 1 : 0]); break;
        case 2: take(H[RL > 2 ? 2 : 0], L[RL > 2 ? 2 : 0]); break;
        default: take(H[RL > 3 ? 3 : 0], L[RL > 3 ? 3 : 0]); break;
        }
        f32x2 fh[RL], fl[RL];                       // the multipliers of this lane's rows
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            float2 f = xt[k * N + lane + 32 * i];
            if (mine_row && i == (p >> 5)) f = make_float2(-1.0f, 0.0f);
            fh[i] = pack2(f.x, f.x);
            fl[i] = pack2(f.y, f.y);
        }
        __syncwarp();
        if (lane < CW) {                            // entry k, whose column is 0 now, becomes 1 / pivot
            const dfloat x = wid + NW * lane == k ? dfloat{1.0f, 0.0f} : dfloat{xrow[wid][0][lane], xrow[wid][1][lane]};
            const dfloat r = df_mul(x, {ct.y, ct.z});
            rowh[wid][lane >> 1][lane & 1] = r.h;
            rowh[wid][lane >> 1][2 + (lane & 1)] = -r.h;
            rowl[wid][lane >> 1][lane & 1] = -r.l;
        }
        __syncwarp();
        auto row_pair = [&](int m, f32x2& rh, f32x2& nrh, f32x2& nrl) __attribute__((always_inline)) {
            const float4 q = *reinterpret_cast<const float4*>(rowh[wid][m]);
            const float2 z = *reinterpret_cast<const float2*>(rowl[wid][m]);
            rh = pack2(q.x, q.y);
            nrh = pack2(q.z, q.w);
            nrl = pack2(z.x, z.y);
        };
        const int nc = (k + 1) / NW;                // column k + 1 among its warp's columns
        const bool next_here = k + 1 < n && (k + 1) % NW == wid;
        if (next_here) {
            // the pair with column k + 1, updated ahead of the others (and again with them below)
            f32x2 xh[RL], xl[RL], rh, nrh, nrl;
            // (bitwise selects, for the same reason as above)
#pragma unroll
            for (int i = 0; i < RL; ++i) xh[i] = xl[i] = 0ull;
#pragma unroll
            for (int m = 0; m < CP; ++m) {
                const f32x2 mask = m == (nc >> 1) ? ~0ull : 0ull;
#pragma unroll
                for (int i = 0; i < RL; ++i) {
                    xh[i] |= H[i][m] & mask;
                    xl[i] |= L[i][m] & mask;
                }
            }
            row_pair(nc >> 1, rh, nrh, nrl);
            float h[RL], l[RL];
#pragma unroll
            for (int i = 0; i < RL; ++i) {
                eliminate2(xh[i], xl[i], fh[i], fl[i], rh, nrh, nrl);
                float h0, h1, l0, l1;
                unpack2(xh[i], h0, h1);
                unpack2(xl[i], l0, l1);
                h[i] = (nc & 1) ? h1 : h0;
                l[i] = (nc & 1) ? l1 : l0;
            }
            publish(k + 1, h, l);
        }
#pragma unroll
        for (int m = 0; m < CP; ++m) {
            f32x2 rh, nrh, nrl;
            row_pair(m, rh, nrh, nrl);
#pragma unroll
            for (int i = 0; i < RL; ++i) eliminate2(H[i][m], L[i][m], fh[i], fl[i], rh, nrh, nrl);
        }
        if (next_here) {
            // column k + 1 becomes 0, so that its step leaves -f_i / pivot there
#pragma unroll
            for (int m = 0; m < CP; ++m)
#pragma unroll
                for (int i = 0; i < RL; ++i) {
                    float h0, h1, l0, l1;
                    unpack2(H[i][m], h0, h1);
                    unpack2(L[i][m], l0, l1);
                    const bool z0 = nc == 2 * m, z1 = nc == 2 * m + 1;
                    H[i][m] = pack2(z0 ? 0.0f : h0, z1 ? 0.0f : h1);
                    L[i][m] = pack2(z0 ? 0.0f : l0, z1 ? 0.0f : l1);
                }
        }
    }

    double part_kin = 0.0;
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
                float h0, h1, l0, l1;
                unpack2(H[i][m], h0, h1);
                unpack2(L[i][m], l0, l1);
                const int c = wid + NW * 2 * m;
                if (c < n) xt[(size_t)piv[c] * ld + o] = make_float2(h0, l0);
                if (c + NW < n) xt[(size_t)piv[c + NW] * ld + o] = make_float2(h1, l1);
            }
        }
        // sign: negative pivots and the inversions of k -> p_k, modulo two
        int odd = 0;
        for (int k = tid; k < n; k += NT) odd ^= pivd[k].x < 0.0f;
        for (int t = tid; t < n * G; t += NT) {     // G threads per step, a G-th of the steps each
            const int k = t / G, part = t - k * G, pk = piv[k];
            for (int m = k + 1 + part; m < n; m += G) odd ^= piv[m] < pk;
        }
        odd = __reduce_xor_sync(kFullMask, odd);
        if (lane == 0 && odd) atomicXor(&parity, 1);
        __syncthreads();
        // T = -1/2 sum_ij X_ji lap phi_j(r_i) and the drift, in FP64 (inverse entries h + l): four electrons
        // per warp at a time, lanes 8 e + 2 c and the next getting sum c of electron e
        const bool want_g = a.drift != nullptr, want_l = a.kinetic != nullptr;
        if (want_g || want_l) {
            const T* gp = static_cast<const T*>(a.grad);
            const T* lp = static_cast<const T*>(a.lap);
            for (int i0 = 4 * wid; i0 < n; i0 += 4 * NW) {
                double s[16];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int i = i0 + e;
#pragma unroll
                    for (int c = 0; c < 4; ++c) s[4 * e + c] = 0.0;
                    if (i >= n) continue;
                    float2 z[RL];
                    T g[RL][4];                     // all of an electron's loads first
#pragma unroll
                    for (int t = 0; t < RL; ++t) {
                        const int jj = lane + 32 * t;
                        const bool on = jj < n;
                        z[t] = on ? xt[(size_t)i * ld + jj] : make_float2(0.0f, 0.0f);
#pragma unroll
                        for (int c = 0; c < 3; ++c) g[t][c] = on && want_g ? __ldg(gp + ((base + i) * 3 + c) * O + jj) : T(0);
                        g[t][3] = on && want_l ? __ldg(lp + (base + i) * O + jj) : T(0);
                    }
#pragma unroll
                    for (int t = 0; t < RL; ++t) {
                        if (32 * t >= n) continue;
                        const double x = (double)z[t].x + (double)z[t].y;
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (c < 3 ? want_g : want_l) s[4 * e + c] = fma(x, (double)g[t][c], s[4 * e + c]);
                    }
                }
                const double sum = warp_sum16(s);
                const int i = i0 + (lane >> 3), c = (lane >> 1) & 3;
                if (lane & 1) continue;
                if (c == 3) part_kin += sum;
                else if (want_g && i < n) a.drift[(base + i) * 3 + c] = sum;
            }
        }
    }
    // ---- the block's sums, then the walker's through the cluster ----
    double part_ld = 0.0;
    if (!sing)
        for (int k = tid; k < n; k += NT) part_ld += log(fabs((double)pivd[k].x + (double)pivd[k].y));
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
    const double logdet = block_sum(part_ld), kin = block_sum(part_kin);
    if (tid == 0) mine = {logdet, -0.5 * kin, parity, sing ? 1 : 0, stuck ? 1 : 0};
    cluster.sync();
    const BlockResult other = *cluster.map_shared_rank(&mine, spin ^ 1);
    const bool singular = sing || other.singular;
    const bool lost = stuck || other.stuck;
    if (spin == 0 && tid == 0) {
        if (lost) timed_out = 1;
        const double nan = __longlong_as_double(0x7ff8000000000000LL);
        const double inf = __longlong_as_double(0x7ff0000000000000LL);
        if (a.logdet) a.logdet[w] = lost ? nan : singular ? -inf : logdet + other.logdet;
        if (a.sign) a.sign[w] = lost ? nan : singular ? 0.0 : ((mine.odd ^ other.odd) ? -1.0 : 1.0);
        if (a.kinetic) a.kinetic[w] = singular ? nan : -0.5 * kin + other.kin;
    }
    if (singular && a.drift) {
        const double nan = __longlong_as_double(0x7ff8000000000000LL);
        for (int e = tid; e < 3 * n; e += NT) a.drift[base * 3 + e] = nan;
    }
    cluster.sync();   // the other CTA may still be reading `mine`
}

template <typename T, int G>
int launch_shape(const SlaterArgs& a, cudaStream_t st)
{
    using R = RegShape<G>;
    auto k = slater_reg_kernel<T, G>;
    constexpr int smem = sizeof(float2) * 32 * G * (32 * G + 1);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(slater_reg_kernel)");
    constexpr long long kMaxWalkers = 1LL << 29;    // per launch: two CTAs each, within the grid limit
    for (long long w0 = 0; w0 < a.n_walkers; w0 += kMaxWalkers) {
        const long long m = a.n_walkers - w0 < kMaxWalkers ? a.n_walkers - w0 : kMaxWalkers;
        k<<<(unsigned)(2 * m), 32 * R::NW, smem, st>>>(a, w0);
        const int rc = cuda_error(cudaGetLastError(), "slater_reg_kernel launch");
        if (rc != QMCSPL_OK) return rc;
    }
    return QMCSPL_OK;
}

template <typename T>
int launch_typed(const SlaterArgs& a, int nmax, cudaStream_t st)
{
    switch ((nmax + 31) / 32) {
    case 0:
    case 1: return launch_shape<T, 1>(a, st);
    case 2: return launch_shape<T, 2>(a, st);
    case 3: return launch_shape<T, 3>(a, st);
    default: return launch_shape<T, 4>(a, st);
    }
}

}  // namespace

cudaError_t slater_reg_timeout_word(void** p) { return cudaGetSymbolAddress(p, timed_out); }

int launch_slater_reg_f64(const SlaterArgs& a, int nmax, cudaStream_t st) { return launch_typed<double>(a, nmax, st); }
int launch_slater_reg_f32(const SlaterArgs& a, int nmax, cudaStream_t st) { return launch_typed<float>(a, nmax, st); }

}  // namespace qmcspl

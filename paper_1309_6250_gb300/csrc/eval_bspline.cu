// eval_bspline.cu -- tricubic B-spline value / gradient / Laplacian evaluation.
//
// Computes, for every position r and orbital n (Appendix, Eq. b-splineapproximation):
//   phi(r)   = sum_{l,m,n=-1..2} b_l(tx) b_m(ty) b_n(tz) beta[ix+l][iy+m][iz+n]
//   grad phi = N_i (a^-1)^T grad_t phi               (chain rule, Sec. II Coordinates)
//   lap phi  = sum_ij N_i N_j (a^-1 a^-T)_ij d2phi/dt_i dt_j, or, with the separate
//              Laplacian table of Sec. III C, the same tricubic sum over beta_lap.
// For Bloch orbitals (Sec. II) the stored functions are Re u and Im u of each orbital and
// the epilogue multiplies by exp(i k.r) with the product rule (bloch_apply).
//
// Work mapping.  A group of L = 2^k lanes shares one position; each lane owns one
// 16-byte chunk of every stored row (2, 4 or 8 orbitals for f64, f32, bf16), the
// group covers one orbital tile of L chunks, and tiles x groups cover the orbitals.
// Per position the group computes the reduced coordinate in FP64 (one lane per axis,
// broadcast by shuffles) and the 1-D weights in registers, then walks the 16 (x, y)
// stencil columns.  Each column is four contiguous z rows (ghost planes make them
// contiguous), read with coalesced 16-byte loads: a warp-wide load instruction moves
// 32 x 16 B of one row.  The z sum is done first, then the (x, y) weights; the
// Hessian-derived Laplacian folds the metric N_i N_j (a^-1 a^-T)_ij into the per-column
// weights so only one accumulator per orbital is needed.
//
// Every warp task (32 lanes x one chunk x 64 rows per table) moves the same number of
// bytes whatever the orbital count, which is what lets the batched kernel mix cells
// with different orbital counts and grids in one launch with a static schedule.
//
// The kernel is a gather bounded by memory bandwidth: no tensor cores, since each
// position gathers its own stencil.
#include <type_traits>

#include "eval_common.cuh"

namespace qmcspl {
namespace {

// Evaluate the groups [w0, w0 + groups per warp) of one cell.  Called by all 32 lanes.
template <typename T, bool LAPTAB>
__device__ __forceinline__ void bspline_warp_task(const EvalArgs& p, long long w0, int lane)
{
    using A = typename Traits<T>::A;
    constexpr int E = Traits<T>::E;
    const int L = 1 << p.lanes_log2;
    const int sub = lane & (L - 1);
    const int gbase = lane & ~(L - 1);
    const long long total = p.n_pos * p.tiles;
    const size_t rowb = (size_t)p.row_stride * sizeof(T);
    const size_t colb = (size_t)p.col_stride * sizeof(T);

    const long long gid = w0 + (lane >> p.lanes_log2);
    const bool active = gid < total;
    const long long q = active ? gid / p.tiles : 0;
    const int tile = active ? (int)(gid - q * p.tiles) : 0;
    const long long ip = active ? order_index(p, q) : q;
    int ix, iy, iz;
    double tx, ty, tz;
    bool ok;
    coords_double(p, ip, L, sub, gbase, ix, iy, iz, tx, ty, tz, ok);
    if (!active) return;
    if (!ok && sub == 0 && tile == 0) atomicOr(p.err, 1);

    A bx[4], dbx[4], d2bx[4], by[4], dby[4], d2by[4], bz[4], dbz[4], d2bz[4];
    bspline_weights<A>((A)tx, bx, dbx, LAPTAB ? nullptr : d2bx);
    bspline_weights<A>((A)ty, by, dby, LAPTAB ? nullptr : d2by);
    bspline_weights<A>((A)tz, bz, dbz, LAPTAB ? nullptr : d2bz);

    int xs[4], ys[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        xs[j] = wrap1(ix + j - 1, p.nx);
        ys[j] = wrap1(iy + j - 1, p.ny);
    }
    const int chunk = tile * L + sub;
    const char* t0 = static_cast<const char*>(p.tab[0]) + (size_t)chunk * 16 + (size_t)iz * rowb;
    const char* t1 = LAPTAB ? static_cast<const char*>(p.tab[1]) + (size_t)chunk * 16 + (size_t)iz * rowb
                            : nullptr;

    A v[E], gx[E], gy[E], gz[E], lp[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = gx[e] = gy[e] = gz[e] = lp[e] = A(0);

    A ml0 = 0, ml1 = 0, ml2 = 0, ml3 = 0, ml4 = 0, ml5 = 0;
    if (!LAPTAB) {
        ml0 = (A)p.ml[0]; ml1 = (A)p.ml[1]; ml2 = (A)p.ml[2];
        ml3 = (A)p.ml[3]; ml4 = (A)p.ml[4]; ml5 = (A)p.ml[5];
    }

#pragma unroll
    for (int l = 0; l < 4; ++l) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const size_t col = (size_t)(xs[l] * p.ny + ys[m]) * colb;
            uint4 raw[4], rawl[4];
#pragma unroll
            for (int n = 0; n < 4; ++n) raw[n] = ldg_table(p, t0 + col + n * rowb);
            if (LAPTAB) {
#pragma unroll
                for (int n = 0; n < 4; ++n) rawl[n] = ldg_table(p, t1 + col + n * rowb);
            }
            A a0[E], a1[E], a2[E], al[E];
#pragma unroll
            for (int e = 0; e < E; ++e) a0[e] = a1[e] = a2[e] = al[e] = A(0);
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                A c[E];
                unpack<T>(raw[n], c);
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    a0[e] = fma(bz[n], c[e], a0[e]);
                    a1[e] = fma(dbz[n], c[e], a1[e]);
                    if (!LAPTAB) a2[e] = fma(d2bz[n], c[e], a2[e]);
                }
                if (LAPTAB) {
                    A cl[E];
                    unpack<T>(rawl[n], cl);
#pragma unroll
                    for (int e = 0; e < E; ++e) al[e] = fma(bz[n], cl[e], al[e]);
                }
            }
            const A w00 = bx[l] * by[m];
            const A w10 = dbx[l] * by[m];
            const A w01 = bx[l] * dby[m];
            A c0 = 0, c1 = 0, c2 = 0;
            if (!LAPTAB) {
                c0 = ml0 * (d2bx[l] * by[m]) + ml1 * (bx[l] * d2by[m]) + ml3 * (dbx[l] * dby[m]);
                c1 = ml4 * w10 + ml5 * w01;
                c2 = ml2 * w00;
            }
#pragma unroll
            for (int e = 0; e < E; ++e) {
                v[e] = fma(w00, a0[e], v[e]);
                gx[e] = fma(w10, a0[e], gx[e]);
                gy[e] = fma(w01, a0[e], gy[e]);
                gz[e] = fma(w00, a1[e], gz[e]);
                if (LAPTAB) {
                    lp[e] = fma(w00, al[e], lp[e]);
                } else {
                    lp[e] = fma(c0, a0[e], fma(c1, a1[e], fma(c2, a2[e], lp[e])));
                }
            }
        }
    }

    const int o0 = chunk * E;
    if (o0 >= p.n_orb) return;
    const bool vec = p.vec_out != 0;
    A cg[3][E];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const A m0 = (A)p.mg[3 * a], m1 = (A)p.mg[3 * a + 1], m2 = (A)p.mg[3 * a + 2];
#pragma unroll
        for (int e = 0; e < E; ++e) cg[a][e] = fma(m0, gx[e], fma(m1, gy[e], m2 * gz[e]));
    }
    if (p.phase) bloch_apply<A, E>(p, ip, v, cg, lp, true, !LAPTAB);
    if (p.val) store_run<A, E>(static_cast<A*>(p.val) + ip * p.n_orb + o0, v, o0, p.n_orb, vec);
    if (p.grad) {
        A* g = static_cast<A*>(p.grad) + ip * 3 * p.n_orb + o0;
#pragma unroll
        for (int a = 0; a < 3; ++a) store_run<A, E>(g + (size_t)a * p.n_orb, cg[a], o0, p.n_orb, vec);
    }
    if (p.lap) store_run<A, E>(static_cast<A*>(p.lap) + ip * p.n_orb + o0, lp, o0, p.n_orb, vec);
}

// The same computation for float and bfloat16 tables with packed FP32 arithmetic
// (fma.rn.f32x2: two orbitals per instruction) and the rows of the next AHEAD stencil columns
// loaded before the current column is contracted.
// stage: with RAGGED, the warp's shared memory for the stores of unaligned rows (see RaggedStore).
// NOREC: for launches without records (coords_float_shared).
template <typename T, bool LAPTAB, int AHEAD, bool RAGGED, bool NOREC>
__device__ __forceinline__ void bspline_warp_task_x2(const EvalArgs& p, long long w0, int lane, float* stage)
{
    constexpr int E = Traits<T>::E;          // orbitals per lane (4 float, 8 bfloat16)
    constexpr int NP = Pairs<T>::N;          // packed pairs per lane
    constexpr int R = LAPTAB ? 8 : 4;        // rows loaded per column
    const int L = 1 << p.lanes_log2;
    const int sub = lane & (L - 1);
    const int gbase = lane & ~(L - 1);
    const long long total = p.n_pos * p.tiles;
    const size_t rowb = (size_t)p.row_stride * sizeof(T);
    const size_t colb = (size_t)p.col_stride * sizeof(T);

    const long long gid = w0 + (lane >> p.lanes_log2);
    const bool active = gid < total;
    const long long q = active ? gid / p.tiles : 0;
    const int tile = active ? (int)(gid - q * p.tiles) : 0;
    const long long ip = active ? order_index(p, q) : q;
    int ix, iy, iz;
    float tx, ty, tz;
    bool ok;
    // (the bfloat16 kernel runs fastest with the rolled form of the reduction, the float one with
    // the written-out form; both give the same bits)
    if constexpr (NOREC) coords_float_shared(p, ip, L, sub, gbase, ix, iy, iz, tx, ty, tz, ok);
    else coords_float<std::is_same<T, __nv_bfloat16>::value>(p, ip, L, sub, gbase, ix, iy, iz, tx, ty, tz, ok);
    if (!RAGGED && !active) return;   // (all lanes take part in the staged stores)
    if (active && !ok && sub == 0 && tile == 0) atomicOr(p.err, 1);

    float bx[4], dbx[4], d2bx[4], by[4], dby[4], d2by[4], bz[4], dbz[4], d2bz[4];
    bspline_weights<float>(tx, bx, dbx, LAPTAB ? nullptr : d2bx);
    bspline_weights<float>(ty, by, dby, LAPTAB ? nullptr : d2by);
    bspline_weights<float>(tz, bz, dbz, LAPTAB ? nullptr : d2bz);
    f32x2 bz2[4], dbz2[4], d2bz2[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        bz2[n] = pack2(bz[n], bz[n]);
        dbz2[n] = pack2(dbz[n], dbz[n]);
        if (!LAPTAB) d2bz2[n] = pack2(d2bz[n], d2bz[n]);
    }
    float ml0 = 0.f, ml1 = 0.f, ml2 = 0.f, ml3 = 0.f, ml4 = 0.f, ml5 = 0.f;
    if (!LAPTAB) {
        ml0 = p.mlf[0]; ml1 = p.mlf[1]; ml2 = p.mlf[2];
        ml3 = p.mlf[3]; ml4 = p.mlf[4]; ml5 = p.mlf[5];
    }
    int xs[4], ys[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        xs[j] = wrap1(ix + j - 1, p.nx);
        ys[j] = wrap1(iy + j - 1, p.ny);
    }
    const int chunk = tile * L + sub;
    const char* t0 = static_cast<const char*>(p.tab[0]) + (size_t)chunk * 16 + (size_t)iz * rowb;
    const char* t1 = LAPTAB ? static_cast<const char*>(p.tab[1]) + (size_t)chunk * 16 + (size_t)iz * rowb
                            : nullptr;

    f32x2 V[NP], GX[NP], GY[NP], GZ[NP], LP[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) V[j] = GX[j] = GY[j] = GZ[j] = LP[j] = 0ull;

    uint4 ring[AHEAD + 1][R];   // column c in slot c mod (AHEAD + 1)
    auto load_column = [&](int c) {
        const size_t col = (size_t)(xs[c >> 2] * p.ny + ys[c & 3]) * colb;
#pragma unroll
        for (int n = 0; n < 4; ++n) ring[c % (AHEAD + 1)][n] = ldg_table(p, t0 + col + n * rowb);
        if (LAPTAB) {
#pragma unroll
            for (int n = 0; n < 4; ++n) ring[c % (AHEAD + 1)][4 + n] = ldg_table(p, t1 + col + n * rowb);
        }
    };
#pragma unroll
    for (int c = 0; c < AHEAD; ++c) load_column(c);
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        const int l = c >> 2, m = c & 3;
        if (c + AHEAD < 16) load_column(c + AHEAD);
        const uint4(&cur)[R] = ring[c % (AHEAD + 1)];
        f32x2 A0[NP], A1[NP], A2[NP], AL[NP];
#pragma unroll
        for (int j = 0; j < NP; ++j) A0[j] = A1[j] = A2[j] = AL[j] = 0ull;
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            f32x2 cv[NP];
            Pairs<T>::get(cur[n], cv);
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                A0[j] = ffma2(bz2[n], cv[j], A0[j]);
                A1[j] = ffma2(dbz2[n], cv[j], A1[j]);
                if (!LAPTAB) A2[j] = ffma2(d2bz2[n], cv[j], A2[j]);
            }
            if (LAPTAB) {
                Pairs<T>::get(cur[4 + n], cv);
#pragma unroll
                for (int j = 0; j < NP; ++j) AL[j] = ffma2(bz2[n], cv[j], AL[j]);
            }
        }
        const float w00 = bx[l] * by[m], w10 = dbx[l] * by[m], w01 = bx[l] * dby[m];
        const f32x2 W00 = pack2(w00, w00), W10 = pack2(w10, w10), W01 = pack2(w01, w01);
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            V[j] = ffma2(W00, A0[j], V[j]);
            GX[j] = ffma2(W10, A0[j], GX[j]);
            GY[j] = ffma2(W01, A0[j], GY[j]);
            GZ[j] = ffma2(W00, A1[j], GZ[j]);
        }
        if (LAPTAB) {
#pragma unroll
            for (int j = 0; j < NP; ++j) LP[j] = ffma2(W00, AL[j], LP[j]);
        } else {
            const float c0 = ml0 * (d2bx[l] * by[m]) + ml1 * (bx[l] * d2by[m]) + ml3 * (dbx[l] * dby[m]);
            const float c1 = ml4 * w10 + ml5 * w01;
            const float c2 = ml2 * w00;
            const f32x2 C0 = pack2(c0, c0), C1 = pack2(c1, c1), C2 = pack2(c2, c2);
#pragma unroll
            for (int j = 0; j < NP; ++j) LP[j] = ffma2(C0, A0[j], ffma2(C1, A1[j], ffma2(C2, A2[j], LP[j])));
        }
    }

    const int o0 = chunk * E;
    if (!RAGGED && o0 >= p.n_orb) return;
    const bool vec = p.vec_out != 0;
    float v[E], gx[E], gy[E], gz[E], lp[E];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        unpack2(V[j], v[2 * j], v[2 * j + 1]);
        unpack2(GX[j], gx[2 * j], gx[2 * j + 1]);
        unpack2(GY[j], gy[2 * j], gy[2 * j + 1]);
        unpack2(GZ[j], gz[2 * j], gz[2 * j + 1]);
        unpack2(LP[j], lp[2 * j], lp[2 * j + 1]);
    }
    float cg[3][E];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float m0 = p.mgf[3 * a], m1 = p.mgf[3 * a + 1], m2 = p.mgf[3 * a + 2];
#pragma unroll
        for (int e = 0; e < E; ++e) cg[a][e] = fmaf(m0, gx[e], fmaf(m1, gy[e], m2 * gz[e]));
    }
    if (p.phase) bloch_apply<float, E>(p, ip, v, cg, lp, true, !LAPTAB);
    if constexpr (RAGGED) {
        RaggedStore<E> out(stage, ip, o0, active, p.n_orb);
        if (p.val) out.put(static_cast<float*>(p.val), v, 1, 0);
        if (p.grad)
#pragma unroll
            for (int a = 0; a < 3; ++a) out.put(static_cast<float*>(p.grad), cg[a], 3, a);
        if (p.lap) out.put(static_cast<float*>(p.lap), lp, 1, 0);
        return;
    }
    if (p.val) store_run<float, E>(static_cast<float*>(p.val) + ip * p.n_orb + o0, v, o0, p.n_orb, vec);
    if (p.grad) {
        float* g = static_cast<float*>(p.grad) + ip * 3 * p.n_orb + o0;
#pragma unroll
        for (int a = 0; a < 3; ++a) store_run<float, E>(g + (size_t)a * p.n_orb, cg[a], o0, p.n_orb, vec);
    }
    if (p.lap) store_run<float, E>(static_cast<float*>(p.lap) + ip * p.n_orb + o0, lp, o0, p.n_orb, vec);
}

// Double-float tables (DF64Tag chunks, see eval_common.cuh): the same stencil walk with every
// product and sum carried as a double-float pair on the FP32 pipe (see df_mad2), results
// converted to double at the store.

template <bool LAPTAB, int UNROLL>
__device__ __forceinline__ void bspline_warp_task_df(const EvalArgs& p, long long w0, int lane)
{
    const int L = 1 << p.lanes_log2;
    const int sub = lane & (L - 1);
    const int gbase = lane & ~(L - 1);
    const long long total = p.n_pos * p.tiles;
    const size_t rowb = (size_t)p.row_stride * 8;
    const size_t colb = (size_t)p.col_stride * 8;

    const long long gid = w0 + (lane >> p.lanes_log2);
    const bool active = gid < total;
    const long long q = active ? gid / p.tiles : 0;
    const int tile = active ? (int)(gid - q * p.tiles) : 0;
    const long long ip = active ? order_index(p, q) : q;
    int ix, iy, iz;
    dfloat tx, ty, tz;
    bool ok;
    if (p.rec) {   // kind-3 record: cell and double-float t, no FP64 work here
        const float4* qr = static_cast<const float4*>(p.rec) + 2 * ip;
        const float4 a = __ldg(qr), b = __ldg(qr + 1);
        unpack_cell(__float_as_int(a.x), ix, iy, iz, ok);
        tx = {a.y, a.z};
        ty = {a.w, b.x};
        tz = {b.y, b.z};
    } else {
        const double r[3] = {p.pos[3 * ip], p.pos[3 * ip + 1], p.pos[3 * ip + 2]};
        double dx, dy, dz;
        reduced_coordinates(p, r, L, sub, gbase, ix, iy, iz, dx, dy, dz, ok);
        tx = df_from_double(dx);
        ty = df_from_double(dy);
        tz = df_from_double(dz);
    }
    if (!active) return;
    if (!ok && sub == 0 && tile == 0) atomicOr(p.err, 1);

    dfloat bx[4], dbx[4], d2bx[4], by[4], dby[4], d2by[4], bz[4], dbz[4], d2bz[4];
    bspline_weights_df(tx, bx, dbx, LAPTAB ? nullptr : d2bx);
    bspline_weights_df(ty, by, dby, LAPTAB ? nullptr : d2by);
    bspline_weights_df(tz, bz, dbz, LAPTAB ? nullptr : d2bz);
    dfloat ml[6];
    if (!LAPTAB)
#pragma unroll
        for (int k = 0; k < 6; ++k) ml[k] = {p.mlf[k], p.mll[k]};
    int xs[4], ys[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        xs[j] = wrap1(ix + j - 1, p.nx);
        ys[j] = wrap1(iy + j - 1, p.ny);
    }
    const int chunk = tile * L + sub;
    const char* t0 = static_cast<const char*>(p.tab[0]) + (size_t)chunk * 16 + (size_t)iz * rowb;
    const char* t1 = LAPTAB ? static_cast<const char*>(p.tab[1]) + (size_t)chunk * 16 + (size_t)iz * rowb
                            : nullptr;
    const f32x2 zero = pack2(p.zero, p.zero);   // (see df_mad2)
    // accumulators (h, l) for value, reduced gradient, Laplacian-table value
    f32x2 Vh = 0, Vl = 0, Xh = 0, Xl = 0, Yh = 0, Yl = 0, Zh = 0, Zl = 0, Lh = 0, Ll = 0;
#pragma unroll UNROLL
    for (int c = 0; c < 16; ++c) {
        const int l = c >> 2, m = c & 3;
        const size_t col = (size_t)(xs[l] * p.ny + ys[m]) * colb;
        uint4 raw[4], rawl[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) raw[n] = ldg_table(p, t0 + col + n * rowb);
        if (LAPTAB) {
#pragma unroll
            for (int n = 0; n < 4; ++n) rawl[n] = ldg_table(p, t1 + col + n * rowb);
        }
        f32x2 A0h, A0l, A1h, A1l, A2h, A2l, ALh, ALl;
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            auto add = [&](f32x2& Ah, f32x2& Al, dfloat w, f32x2 Bh, f32x2 Bl) {
                const f32x2 wh = pack2(w.h, w.h), wl = pack2(w.l, w.l);
                if (n == 0) df_mul2(Ah, Al, wh, wl, Bh, Bl, zero);
                else df_mad2(Ah, Al, wh, wl, Bh, Bl, zero);
            };
            const f32x2 Bh = pack2u(raw[n].x, raw[n].y), Bl = pack2u(raw[n].z, raw[n].w);
            add(A0h, A0l, bz[n], Bh, Bl);
            add(A1h, A1l, dbz[n], Bh, Bl);
            if (!LAPTAB) add(A2h, A2l, d2bz[n], Bh, Bl);
            if (LAPTAB) add(ALh, ALl, bz[n], pack2u(rawl[n].x, rawl[n].y), pack2u(rawl[n].z, rawl[n].w));
        }
        const dfloat w00 = df_mul(bx[l], by[m]), w10 = df_mul(dbx[l], by[m]), w01 = df_mul(bx[l], dby[m]);
        const f32x2 h00 = pack2(w00.h, w00.h), l00 = pack2(w00.l, w00.l);
        const f32x2 h10 = pack2(w10.h, w10.h), l10 = pack2(w10.l, w10.l);
        const f32x2 h01 = pack2(w01.h, w01.h), l01 = pack2(w01.l, w01.l);
        df_mad2(Vh, Vl, h00, l00, A0h, A0l, zero);
        df_mad2(Xh, Xl, h10, l10, A0h, A0l, zero);
        df_mad2(Yh, Yl, h01, l01, A0h, A0l, zero);
        df_mad2(Zh, Zl, h00, l00, A1h, A1l, zero);
        if (LAPTAB) {
            df_mad2(Lh, Ll, h00, l00, ALh, ALl, zero);
        } else {
            // metric folded into per-column weights: lap += c0 A0 + c1 A1 + c2 A2
            const dfloat c0 = df_add(df_add(df_mul(ml[0], df_mul(d2bx[l], by[m])), df_mul(ml[1], df_mul(bx[l], d2by[m]))),
                                     df_mul(ml[3], df_mul(dbx[l], dby[m])));
            const dfloat c1 = df_add(df_mul(ml[4], w10), df_mul(ml[5], w01));
            const dfloat c2 = df_mul(ml[2], w00);
            df_mad2(Lh, Ll, pack2(c0.h, c0.h), pack2(c0.l, c0.l), A0h, A0l, zero);
            df_mad2(Lh, Ll, pack2(c1.h, c1.h), pack2(c1.l, c1.l), A1h, A1l, zero);
            df_mad2(Lh, Ll, pack2(c2.h, c2.h), pack2(c2.l, c2.l), A2h, A2l, zero);
        }
        if (m == 3) {
            df_renorm2(Vh, Vl);
            df_renorm2(Xh, Xl);
            df_renorm2(Yh, Yl);
            df_renorm2(Zh, Zl);
            df_renorm2(Lh, Ll);
        }
    }

    constexpr int E = 2;
    const int o0 = chunk * E;
    if (o0 >= p.n_orb) return;
    const bool vec = p.vec_out != 0;
    float a0, a1, b0, b1;
    dfloat dv[E], dl[E], dg[3][E];
    unpack2(Vh, a0, a1); unpack2(Vl, b0, b1);
    dv[0] = {a0, b0}; dv[1] = {a1, b1};
    unpack2(Lh, a0, a1); unpack2(Ll, b0, b1);
    dl[0] = {a0, b0}; dl[1] = {a1, b1};
    if (p.grad || p.phase) {
        // chain rule in double-float: grad_a = sum_i mg[a][i] grad_t[i]
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            f32x2 Gh = 0, Gl = 0;
            const float m0h = p.mgf[3 * a], m1h = p.mgf[3 * a + 1], m2h = p.mgf[3 * a + 2];
            const float m0l = p.mgl[3 * a], m1l = p.mgl[3 * a + 1], m2l = p.mgl[3 * a + 2];
            df_mad2(Gh, Gl, pack2(m0h, m0h), pack2(m0l, m0l), Xh, Xl, zero);
            df_mad2(Gh, Gl, pack2(m1h, m1h), pack2(m1l, m1l), Yh, Yl, zero);
            df_mad2(Gh, Gl, pack2(m2h, m2h), pack2(m2l, m2l), Zh, Zl, zero);
            unpack2(Gh, a0, a1); unpack2(Gl, b0, b1);
            dg[a][0] = {a0, b0};
            dg[a][1] = {a1, b1};
        }
    }
    if (p.phase) {   // one complex orbital per lane, in double-float
        const double2 ph = __ldg(p.phase + ip);
        const dfloat c = df_from_double(ph.x), sn = df_from_double(ph.y);
        const dfloat k[3] = {df_from_double(p.kc[0]), df_from_double(p.kc[1]), df_from_double(p.kc[2])};
        const dfloat kk = df_add(df_add(df_mul(k[0], k[0]), df_mul(k[1], k[1])), df_mul(k[2], k[2]));
        dfloat gr[3] = {dg[0][0], dg[1][0], dg[2][0]}, gi[3] = {dg[0][1], dg[1][1], dg[2][1]};
        bloch_one<dfloat>(dv[0], dv[1], gr, gi, dl[0], dl[1], k, kk, c, sn, true, !LAPTAB);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            dg[a][0] = gr[a];
            dg[a][1] = gi[a];
        }
    }
    double v[E], lp[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        v[e] = df_to_double(dv[e].h, dv[e].l);
        lp[e] = df_to_double(dl[e].h, dl[e].l);
    }
    if (p.val) store_run<double, E>(static_cast<double*>(p.val) + ip * p.n_orb + o0, v, o0, p.n_orb, vec);
    if (p.grad) {
        double* g = static_cast<double*>(p.grad) + ip * 3 * p.n_orb + o0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double cg[E];
#pragma unroll
            for (int e = 0; e < E; ++e) cg[e] = df_to_double(dg[a][e].h, dg[a][e].l);
            store_run<double, E>(g + (size_t)a * p.n_orb, cg, o0, p.n_orb, vec);
        }
    }
    if (p.lap) store_run<double, E>(static_cast<double*>(p.lap) + ip * p.n_orb + o0, lp, o0, p.n_orb, vec);
}

// float and bfloat16 tables take the packed path, double tables the scalar one.  AHEAD: columns of
// rows in flight (packed path; columns unrolled for double-float tables).
template <typename T, bool LAPTAB, int AHEAD = 1, bool RAGGED = false, bool NOREC = false>
__device__ __forceinline__ void warp_task(const EvalArgs& p, long long w0, int lane, float* stage = nullptr)
{
    if constexpr (std::is_same<T, DF64Tag>::value) bspline_warp_task_df<LAPTAB, AHEAD>(p, w0, lane);
    else if constexpr (sizeof(T) == 8) bspline_warp_task<T, LAPTAB>(p, w0, lane);
    else bspline_warp_task_x2<T, LAPTAB, AHEAD, RAGGED, NOREC>(p, w0, lane, stage);
}

#ifndef QMCSPL_EVAL_THREADS
#define QMCSPL_EVAL_THREADS 512
#endif
#ifndef QMCSPL_EVAL_THREADS_F32_LAP
#define QMCSPL_EVAL_THREADS_F32_LAP 640
#endif
// Threads per block of the B-spline evaluation kernels (one block per SM).  With cell-ordered
// positions the warps of one block evaluate consecutive (neighbouring) positions on one SM, so
// their shared stencil rows hit in that SM's L1; two smaller blocks on an SM would work on
// positions far apart in the order.  512 threads x 128 registers fill the register file; the
// single-cell FP32 kernel with the Laplacian table also comes in a 640-thread shape that fits in
// 96 registers (16 bytes spilled) and runs 20 warps, which hides more of the L1/L2 latency on
// large launches (1.205 vs 1.262 ms on the 128-orbital step; 576, 672 and 768 threads were
// slower).  Launches of only a few rounds of warp tasks keep 512 threads: their last, partly
// filled round costs more with the bigger block.  The batched kernel keeps 512.
template <typename T, bool LAPTAB> struct BspBlock {
    static constexpr int large = QMCSPL_EVAL_THREADS;   // threads of the shape for large launches
};
template <> struct BspBlock<float, true> {
    static constexpr int large = QMCSPL_EVAL_THREADS_F32_LAP;
};
constexpr int kLargeLaunchRounds = 4;   // warp-task rounds from which the large shape is used
inline bool large_launch(long long warps, int threads) { return warps >= (long long)kLargeLaunchRounds * sm_count() * (threads / 32); }

template <typename T, bool LAPTAB, int THREADS, bool RAGGED, bool NOREC = false>
__global__ void __launch_bounds__(THREADS, 1) bspline_vgl_kernel(const EvalArgs p)
{
    constexpr int WPB = THREADS / 32;
    __shared__ __align__(16) float stage[RAGGED ? WPB : 1][kStageFloats<T, RAGGED>];
    const int lane = threadIdx.x & 31;
    const int gpw = 32 >> p.lanes_log2;
    const long long total = p.n_pos * p.tiles;
    const long long warp = (long long)blockIdx.x * WPB + (threadIdx.x >> 5);
    const long long wstride = (long long)gridDim.x * WPB;
    for (long long w0 = warp * gpw; w0 < total; w0 += wstride * gpw)
        warp_task<T, LAPTAB, 1, RAGGED, NOREC>(p, w0, lane, stage[RAGGED ? threadIdx.x >> 5 : 0]);
}

// Launches of at most kSmallWarps warp tasks per SM: a block per warp task, so that they spread over
// all SMs, and three columns of rows in flight (the registers of the missing warps are free), since
// nothing but a warp's own loads hides their latency.
constexpr int kSmallAhead = 3;
template <typename T, bool LAPTAB, bool RAGGED, bool NOREC = false>
__global__ void __launch_bounds__(32, kSmallWarps) bspline_vgl_small_kernel(const EvalArgs p)
{
    __shared__ __align__(16) float stage[kStageFloats<T, RAGGED>];
    const long long w0 = (long long)blockIdx.x << (5 - p.lanes_log2);
    warp_task<T, LAPTAB, kSmallAhead, RAGGED, NOREC>(p, w0, threadIdx.x, stage);
}

// ---- small launches of FP64 tables: one orbital per lane, shared column weights ----
// The FP64 pipe takes a warp instruction every 64 cycles per SM sub-partition, so a small launch
// lasts as long as one warp's instructions: 907 per lane above with the Hessian Laplacian and two
// orbitals, a third of them weights that every lane of a position computes alike.  Here a lane takes
// one orbital (twice the lanes per position, on sub-partitions that were idle) and the lanes of a
// position divide the three axes' weights and the 16 columns' among themselves, through shared
// memory: the same products and sums in the same order, about 410 instructions.  1,000 positions x 8
// orbitals with the Hessian Laplacian: 33 -> 16 us (127 us in blocks of 16 warps).
struct F64Shared {
    double axis[8][3][12];    // per group (at most 8: groups of at least 4 lanes): w, dw, d2w of each axis
    double col[8][16][6];     // w00, w10, w01, c0, c1, c2 of each stencil column
};

template <bool LAPTAB>
__device__ __forceinline__ void bspline_warp_task_f64_lanes(const EvalArgs& p, long long w0, int lane, F64Shared& sh)
{
    const int L = 1 << p.lanes_log2;          // at least 4
    const int sub = lane & (L - 1);
    const int gbase = lane & ~(L - 1);
    const int grp = lane >> p.lanes_log2;
    const size_t rowb = (size_t)p.row_stride * 8;
    const size_t colb = (size_t)p.col_stride * 8;
    const long long gid = w0 + grp;
    const bool active = gid < p.n_pos * p.tiles;
    const long long q = active ? gid / p.tiles : 0;
    const int tile = active ? (int)(gid - q * p.tiles) : 0;
    const long long ip = active ? order_index(p, q) : 0;
    int ix, iy, iz;
    double tx, ty, tz;
    bool ok;
    coords_double(p, ip, L, sub, gbase, ix, iy, iz, tx, ty, tz, ok);
    if (active && !ok && sub == 0 && tile == 0) atomicOr(p.err, 1);
    if (sub < 3) {   // one axis per lane
        double w[4], dw[4], d2w[4];
        bspline_weights<double>(sub == 0 ? tx : sub == 1 ? ty : tz, w, dw, LAPTAB ? nullptr : d2w);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            sh.axis[grp][sub][j] = w[j];
            sh.axis[grp][sub][4 + j] = dw[j];
            if (!LAPTAB) sh.axis[grp][sub][8 + j] = d2w[j];
        }
    }
    __syncwarp();
    const double *ax = sh.axis[grp][0], *ay = sh.axis[grp][1], *az = sh.axis[grp][2];
    for (int c = sub; c < 16; c += L) {
        const int l = c >> 2, m = c & 3;
        const double bx = ax[l], dbx = ax[4 + l], by = ay[m], dby = ay[4 + m];
        const double w00 = bx * by, w10 = dbx * by, w01 = bx * dby;
        sh.col[grp][c][0] = w00;
        sh.col[grp][c][1] = w10;
        sh.col[grp][c][2] = w01;
        if (!LAPTAB) {
            const double d2bx = ax[8 + l], d2by = ay[8 + m];
            sh.col[grp][c][3] = p.ml[0] * (d2bx * by) + p.ml[1] * (bx * d2by) + p.ml[3] * (dbx * dby);
            sh.col[grp][c][4] = p.ml[4] * w10 + p.ml[5] * w01;
            sh.col[grp][c][5] = p.ml[2] * w00;
        }
    }
    __syncwarp();
    const int o = tile * L + sub;             // this lane's orbital
    if (!active || o >= p.n_orb) return;
    double bz[4], dbz[4], d2bz[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        bz[n] = az[n];
        dbz[n] = az[4 + n];
        if (!LAPTAB) d2bz[n] = az[8 + n];
    }
    int xs[4], ys[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        xs[j] = wrap1(ix + j - 1, p.nx);
        ys[j] = wrap1(iy + j - 1, p.ny);
    }
    const char* t0 = static_cast<const char*>(p.tab[0]) + (size_t)o * 8 + (size_t)iz * rowb;
    const char* t1 = LAPTAB ? static_cast<const char*>(p.tab[1]) + (size_t)o * 8 + (size_t)iz * rowb : nullptr;
    double v = 0.0, gx = 0.0, gy = 0.0, gz = 0.0, lp = 0.0;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        const size_t col = (size_t)(xs[c >> 2] * p.ny + ys[c & 3]) * colb;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, al = 0.0;
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const double t = ldg_table8(p, t0 + col + n * rowb);
            a0 = fma(bz[n], t, a0);
            a1 = fma(dbz[n], t, a1);
            if (!LAPTAB) a2 = fma(d2bz[n], t, a2);
            else al = fma(bz[n], ldg_table8(p, t1 + col + n * rowb), al);
        }
        const double* w = sh.col[grp][c];
        v = fma(w[0], a0, v);
        gx = fma(w[1], a0, gx);
        gy = fma(w[2], a0, gy);
        gz = fma(w[0], a1, gz);
        if (LAPTAB) lp = fma(w[0], al, lp);
        else lp = fma(w[3], a0, fma(w[4], a1, fma(w[5], a2, lp)));
    }
    const long long row = ip * p.n_orb + o;
    if (p.val) __stcs(static_cast<double*>(p.val) + row, v);
    if (p.grad)
#pragma unroll
        for (int a = 0; a < 3; ++a)
            __stcs(static_cast<double*>(p.grad) + row + (2 * ip + a) * p.n_orb,
                   fma(p.mg[3 * a], gx, fma(p.mg[3 * a + 1], gy, p.mg[3 * a + 2] * gz)));
    if (p.lap) __stcs(static_cast<double*>(p.lap) + row, lp);
}

template <bool LAPTAB>
__global__ void __launch_bounds__(32) bspline_vgl_f64_lanes_kernel(const EvalArgs p)
{
    __shared__ F64Shared sh;
    bspline_warp_task_f64_lanes<LAPTAB>(p, (long long)blockIdx.x << (5 - p.lanes_log2), threadIdx.x, sh);
}

// Several cells in one launch: warp task w belongs to the cell c with
// start[c] <= w < start[c + 1]; tasks are handed out round-robin over all warps.
struct BatchArgs {
    int n_cells;
    long long start[QMCSPL_MAX_BATCH + 1];   // prefix sums of warp tasks per cell
    EvalArgs cell[QMCSPL_MAX_BATCH];
};
static_assert(sizeof(BatchArgs) <= 32764, "batched kernel parameters exceed the limit");

template <typename T, bool LAPTAB, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) bspline_vgl_batched_kernel(const __grid_constant__ BatchArgs b)
{
    constexpr int WPB = THREADS / 32;
    const int lane = threadIdx.x & 31;
    const long long warp = (long long)blockIdx.x * WPB + (threadIdx.x >> 5);
    const long long wstride = (long long)gridDim.x * WPB;
    const long long total = b.start[b.n_cells];
    int c = 0;
    for (long long w = warp; w < total; w += wstride) {
        while (w >= b.start[c + 1]) ++c;          // tasks only move forward
        const EvalArgs& p = b.cell[c];
        const long long local = w - b.start[c];
        warp_task<T, LAPTAB>(p, local * (32 >> p.lanes_log2), lane);
    }
}

template <typename K>
long long grid_for(K kernel, int threads, long long warps)
{
    long long blocks = (warps + threads / 32 - 1) / (threads / 32);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess)
        per_sm = 1;
    if (per_sm < 1) per_sm = 1;
    const long long cap = (long long)sm_count() * per_sm;
    if (blocks > cap) blocks = cap;
    return blocks < 1 ? 1 : blocks;
}

template <typename T, bool LAPTAB, int THREADS>
int launch_shape(const EvalArgs& a, long long warps, cudaStream_t st)
{
    auto k = bspline_vgl_kernel<T, LAPTAB, THREADS, false>;
    if constexpr (Traits<T>::E >= 4) {
        const bool staged = staged_rows<T>(a, warps, LAPTAB ? 10 : 6);
        if (staged) k = bspline_vgl_kernel<T, LAPTAB, THREADS, true>;
        if constexpr (THREADS == QMCSPL_EVAL_THREADS) {   // (the large shape's launches have records)
            if (!a.rec) k = staged ? bspline_vgl_kernel<T, LAPTAB, THREADS, true, true> : bspline_vgl_kernel<T, LAPTAB, THREADS, false, true>;
        }
    }
    k<<<(unsigned)grid_for(k, THREADS, warps), THREADS, 0, st>>>(a);
    return cuda_error(cudaGetLastError(), "bspline_vgl_kernel launch");
}

template <typename T, bool LAPTAB>
int launch_small(const EvalArgs& a, long long warps, cudaStream_t st)
{
    if constexpr (std::is_same<T, double>::value) {
        // one orbital per lane while that leaves at most a warp per sub-partition of every SM: beyond, the
        // FP64 pipes are busy either way and the weights are better shared by two orbitals.  (Groups of
        // four lanes or more, for the shared weights; Bloch orbitals need Re and Im in one lane.)
        EvalArgs b = a;
        if (b.lanes_log2 < 5) ++b.lanes_log2;
        else b.tiles *= 2;
        const long long gpw = 32 >> b.lanes_log2, w = (b.n_pos * b.tiles + gpw - 1) / gpw;
        if (b.lanes_log2 >= 2 && !b.phase && w <= 4LL * sm_count()) {
            bspline_vgl_f64_lanes_kernel<LAPTAB><<<(unsigned)w, 32, 0, st>>>(b);
            return cuda_error(cudaGetLastError(), "bspline_vgl_f64_lanes_kernel launch");
        }
    }
    auto k = bspline_vgl_small_kernel<T, LAPTAB, false>;
    if constexpr (Traits<T>::E >= 4) {
        if (!a.rec) k = bspline_vgl_small_kernel<T, LAPTAB, false, true>;
    }
    if constexpr (Traits<T>::E == 8) {
        if (staged_rows<T>(a, warps, 0))
            k = a.rec ? bspline_vgl_small_kernel<T, LAPTAB, true> : bspline_vgl_small_kernel<T, LAPTAB, true, true>;
    }
    k<<<(unsigned)warps, 32, 0, st>>>(a);
    return cuda_error(cudaGetLastError(), "bspline_vgl_small_kernel launch");
}

// Block shapes a caller may choose (qmcspl_set_block, the batched launch plan): 512 threads for
// every table type, 640 for float and bfloat16 tables (96 registers).
template <typename T> constexpr bool kHas640 = std::is_same<T, float>::value || std::is_same<T, __nv_bfloat16>::value;

// `threads` = 0: the automatic rule (the small kernel up to kSmallWarps warp tasks per SM, the large
// shape from kLargeLaunchRounds rounds of warp tasks on); 512 or 640: that shape.
template <typename T, bool LAPTAB>
int launch_typed(const EvalArgs& a, int threads, cudaStream_t st)
{
    const int gpw = 32 >> a.lanes_log2;
    const long long warps = (a.n_pos * a.tiles + gpw - 1) / gpw;
    if constexpr (kHas640<T>) {
        if (threads == 640) return launch_shape<T, LAPTAB, 640>(a, warps, st);
    }
    if (threads == QMCSPL_EVAL_THREADS) return launch_shape<T, LAPTAB, QMCSPL_EVAL_THREADS>(a, warps, st);
    if (small_launch(warps)) return launch_small<T, LAPTAB>(a, warps, st);
    constexpr int large = BspBlock<T, LAPTAB>::large;
    if constexpr (large != QMCSPL_EVAL_THREADS) {
        if (large_launch(warps, large)) return launch_shape<T, LAPTAB, large>(a, warps, st);
    }
    return launch_shape<T, LAPTAB, QMCSPL_EVAL_THREADS>(a, warps, st);
}

template <typename T, bool LAPTAB, int THREADS>
int launch_batched_shape(const BatchArgs& b, cudaStream_t st)
{
    const long long blocks = grid_for(bspline_vgl_batched_kernel<T, LAPTAB, THREADS>, THREADS, b.start[b.n_cells]);
    bspline_vgl_batched_kernel<T, LAPTAB, THREADS><<<(unsigned)blocks, THREADS, 0, st>>>(b);
    return cuda_error(cudaGetLastError(), "bspline_vgl_batched_kernel launch");
}

template <typename T, bool LAPTAB>
int launch_batched_typed(const BatchArgs& b, int threads, cudaStream_t st)
{
    if constexpr (kHas640<T>) {
        if (threads == 640) return launch_batched_shape<T, LAPTAB, 640>(b, st);
    }
    return launch_batched_shape<T, LAPTAB, QMCSPL_EVAL_THREADS>(b, st);
}

void set_outputs(const Handle* h, EvalArgs& a, void* val, void* grad, void* lap)
{
    a.val = val;
    a.grad = grad;
    a.lap = lap;
    const size_t ob = (h->storage == QMCSPL_F64 || h->storage == QMCSPL_DF64) ? 8 : 4;
    const uintptr_t al = (uintptr_t)val | (uintptr_t)grad | (uintptr_t)lap;
    a.vec_out = ((h->n_orb * ob) % 16 == 0) && (al % 16 == 0);
}

}  // namespace

// Float and bfloat16 cubic tables, launches below the large shape: the kernels without records divide the
// conversions among the lanes (coords_float_shared), which costs a call less than the pass and its launch:
// 32,768 positions x 16 orbitals, 48^3 26.8 -> 24.0 us (Hessian Laplacian 18.4 -> 14.4), 9,000 x 16 12.3 -> 10.2,
// 12,000 x 128 47.2 -> 45.1, 24,000 x 64 47.5 -> 45.1, 24,000 x 128 bfloat16 61.0 -> 59.1.  The large shape has
// no such form, and there the pass is the faster one: 30,000 x 128 102 us against 116, 30,000 x 64 58 against
// 65.  Tables without a large shape take the same line: near it both are alike, and over more rounds the
// pass is the faster one for many lanes (Hessian Laplacian, 64^3 x 64 orbitals, 30,000 positions 46.1 us with the pass,
// 45.0 without, 200,000 222 and 234; bfloat16, Laplacian table, 64^3 x 128, 30,000 116.5 and 119.3, 200,000 668 and
// 708; few lanes the other way, 47.3 against 41.5 at 120,000 x 16).  So it is for several tiles of one or two lanes,
// which would each reduce all three axes: 12,000 x 109 bfloat16 37.1 us against 39.7, 40,000 x 40 62.7 against 62.6.
bool eval_shares_coordinates(const Handle* h, long long n_pos)
{
    if (h->storage != QMCSPL_F32 && h->storage != QMCSPL_BF16) return false;
    if (h->method == QMCSPL_LAGRANGE || h->method == QMCSPL_PPSPLINE || h->separate_grad || is_general(h)) return false;
    if (h->bloch || h->block_threads == 640 || (h->lanes_log2 < 2 && h->tiles > 1)) return false;
    const int gpw = 32 >> h->lanes_log2;
    const long long warps = (n_pos * h->tiles + gpw - 1) / gpw;
    return !large_launch(warps, BspBlock<float, true>::large);
}

int launch_bspline_vgl(const Handle* h, const double* pos, const Prepared& pr, long long n_pos, void* val,
                       void* grad, void* lap, cudaStream_t st)
{
    EvalArgs a;
    fill_eval_args(h, &a);
    a.pos = pos;
    a.rec = pr.rec;
    a.perm = pr.perm;
    a.phase = pr.phase;
    a.n_pos = n_pos;
    set_outputs(h, a, val, grad, lap);
    const bool lt = h->separate_lap != 0;
    const int th = h->block_threads;
    switch (h->storage) {
    case QMCSPL_F64: return lt ? launch_typed<double, true>(a, th, st) : launch_typed<double, false>(a, th, st);
    case QMCSPL_F32: return lt ? launch_typed<float, true>(a, th, st) : launch_typed<float, false>(a, th, st);
    case QMCSPL_DF64: return lt ? launch_typed<DF64Tag, true>(a, th, st) : launch_typed<DF64Tag, false>(a, th, st);
    default:
        return lt ? launch_typed<__nv_bfloat16, true>(a, th, st) : launch_typed<__nv_bfloat16, false>(a, th, st);
    }
}

int launch_batched(int n_cells, const Handle* const* hs, const double* const* pos, const Prepared* pr,
                   const long long* n_pos, void* const* val, void* const* grad, void* const* lap,
                   int launch, int threads, cudaStream_t st)
{
    thread_local BatchArgs B;   // about 16 KB: kept off the stack, one per calling thread
    // QMCSPL_BATCH_AUTO: cells of at least kLargeLaunchRounds rounds of warp tasks (512-thread
    // blocks on every SM) get their own launch, the others share one batched launch;
    // QMCSPL_BATCH_SINGLE: every cell in the batched launch; QMCSPL_BATCH_SPLIT: every cell alone
    int nb = 0;
    B.start[0] = 0;
    for (int c = 0; c < n_cells; ++c) {
        EvalArgs& a = B.cell[nb];
        fill_eval_args(hs[c], &a);
        a.pos = pos[c];
        a.rec = pr[c].rec;
        a.perm = pr[c].perm;
        a.phase = pr[c].phase;
        a.n_pos = n_pos[c];
        set_outputs(hs[c], a, val[c], grad[c], lap[c]);
        const int gpw = 32 >> a.lanes_log2;
        const long long warps = (a.n_pos * a.tiles + gpw - 1) / gpw;
        const bool alone = launch == QMCSPL_BATCH_SPLIT || (launch == QMCSPL_BATCH_AUTO && large_launch(warps, QMCSPL_EVAL_THREADS));
        if (alone) {
            if (warps == 0) continue;
            const int rc = launch_bspline_vgl(hs[c], pos[c], pr[c], n_pos[c], val[c], grad[c], lap[c], st);
            if (rc != QMCSPL_OK) return rc;
            continue;
        }
        B.start[nb + 1] = B.start[nb] + warps;
        ++nb;
    }
    B.n_cells = nb;
    if (nb == 0 || B.start[nb] == 0) return QMCSPL_OK;
    const bool lt = hs[0]->separate_lap != 0;
    switch (hs[0]->storage) {
    case QMCSPL_DF64:
        return lt ? launch_batched_typed<DF64Tag, true>(B, threads, st) : launch_batched_typed<DF64Tag, false>(B, threads, st);
    case QMCSPL_F64:
        return lt ? launch_batched_typed<double, true>(B, threads, st) : launch_batched_typed<double, false>(B, threads, st);
    case QMCSPL_F32:
        return lt ? launch_batched_typed<float, true>(B, threads, st) : launch_batched_typed<float, false>(B, threads, st);
    default:
        return lt ? launch_batched_typed<__nv_bfloat16, true>(B, threads, st)
                  : launch_batched_typed<__nv_bfloat16, false>(B, threads, st);
    }
}

}  // namespace qmcspl

// ax_dfl.cuh -- FP64-accurate element operator in float pairs, by whole
// folded lines (orders whose N+1 is odd, N+1 <= 11).
//
// The arithmetic is the compensated float-pair arithmetic of ax_df.cuh; the
// data flow is the one of ax_bfp.cuh: every 1-D contraction takes a whole line
// into registers, folds it into even and odd parts (the GLL derivative matrix
// and its transpose are centro-antisymmetric, M[N-i][N-l] = -M[i][l]),
//     e_l = x_l + x_{N-l},  o_l = x_l - x_{N-l}          (l < H = (N+1)/2),
//     a_i = sum_l A_il e_l + M_{i,H} x_H,  b_i = sum_l B_il o_l,
//     y_i = a_i + b_i,  y_{N-i} = b_i - a_i              (i < H),
//     y_H = sum_l M_{H,l} o_l,
// with A_il = (M_il + M_{i,N-l})/2, B_il = (M_il - M_{i,N-l})/2: 40 product
// terms a line at N = 8 instead of 81, and one shared-memory access a value and
// stage instead of one a product.  The tables are constant-bank operands.
#pragma once

#include "ax_df.cuh"
#include "common.cuh"

template <int NP>
struct DflCfg {
    static constexpr int H = NP / 2;
    static constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
    static constexpr bool OK = NP % 2 == 1 && NP <= 11;
    static constexpr int LS = NP;            // odd line stride: no bank conflicts without padding
    static constexpr int SLAB = NP2 * LS;    // pairs per slab
};

#define DFL_HMAX 6
// Index 0: D (gradient), 1: D^T.  A[.][i][H] is the middle column M_{i,H};
// B[.][H] is the middle row.
struct DflTabs {
    dfp A[2][DFL_HMAX][DFL_HMAX], B[2][DFL_HMAX][DFL_HMAX];
};

// y = M x along one line (N+1 even: without the middle column and row).
template <int NP, int DIR>
__device__ __forceinline__ void dfl_line(const dfp (&x)[NP], dfp (&y)[NP], const DflTabs &T)
{
    constexpr int H = NP / 2;
    dfp e[H], o[H];
#pragma unroll
    for (int l = 0; l < H; ++l) {
        const dfp b = x[NP - 1 - l];
        e[l] = df_sum(x[l], b);
        o[l] = df_sum(x[l], {-b.hi, -b.lo});
    }
#pragma unroll
    for (int i = 0; i < H; ++i) {
        dfacc a = df_mul(T.A[DIR][i][0], e[0]), b = df_mul(T.B[DIR][i][0], o[0]);
#pragma unroll
        for (int l = 1; l < H; ++l) {
            df_mad(a, T.A[DIR][i][l], e[l]);
            df_mad(b, T.B[DIR][i][l], o[l]);
        }
        if constexpr (NP % 2 == 1) df_mad(a, T.A[DIR][i][H], x[H]);
        const dfp av = df_raw(a), bv = df_raw(b);
        y[i] = df_sum(av, bv);
        y[NP - 1 - i] = df_sum(bv, {-av.hi, -av.lo});
    }
    if constexpr (NP % 2 == 1) {
        dfacc b = df_mul(T.B[DIR][H][0], o[0]);
#pragma unroll
        for (int l = 1; l < H; ++l) df_mad(b, T.B[DIR][H][l], o[l]);
        y[H] = df_raw(b);
    }
}

// One element; the interface of ax_bfp_element.  red: one word, zero between
// elements.
template <int NP, class Load, class Store, class After, class Sync>
__device__ __forceinline__ void ax_dfl_element(const Load &load, const Store &store,
                                               const dfp *__restrict__ geo, dfp h1, dfp h2,
                                               const DflTabs &T, dfp *__restrict__ slab, unsigned *red,
                                               int tid, bool active, const After &after_load,
                                               const Sync &sync)
{
    using C = DflCfg<NP>;
    constexpr int NP2 = C::NP2, NP3 = C::NP3, LS = C::LS, SL = C::SLAB;
    dfp *su = slab, *sA = slab + SL, *sB = sA + SL;
    const int i = tid % NP, j = tid / NP;
    double xu[NP];
    if (active) {
        unsigned m = 0;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            xu[k] = load(k * NP2 + tid);
            m = max(m, (unsigned)df_bexp(xu[k]));
        }
        atomicMax(red, m);
    }
    sync();
    after_load();
    const unsigned bmax = *red;
    const int E = bmax > 0 ? (int)bmax - 1023 : 0;
    dfp ru[NP];
    if (active) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            ru[k] = df_split_scaled(xu[k], E);
            su[(k * NP + j) * LS + i] = ru[k];
        }
    }
    sync();
    if (tid == 0) *red = 0u;
    dfp gt[NP];
    if (active) {
        dfp x[NP], y[NP];
        const int row = (j * NP + i) * LS;
#pragma unroll
        for (int l = 0; l < NP; ++l) x[l] = su[row + l];
        dfl_line<NP, 0>(x, y, T);
#pragma unroll
        for (int l = 0; l < NP; ++l) sA[row + l] = y[l];
#pragma unroll
        for (int l = 0; l < NP; ++l) x[l] = su[(j * NP + l) * LS + i];
        dfl_line<NP, 0>(x, y, T);
#pragma unroll
        for (int l = 0; l < NP; ++l) sB[(j * NP + l) * LS + i] = y[l];
        dfl_line<NP, 0>(ru, gt, T);
    }
    sync();
    // geometric factors (column owner)
    if (active) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int p = k * NP2 + tid, q = (k * NP + j) * LS + i;
            const dfp ur = sA[q], us = sB[q], ut = gt[k];
            const dfp g11 = geo[0 * NP3 + p], g22 = geo[1 * NP3 + p], g33 = geo[2 * NP3 + p];
            const dfp g12 = geo[3 * NP3 + p], g13 = geo[4 * NP3 + p], g23 = geo[5 * NP3 + p];
            dfacc vr = df_mul(g11, ur), vs = df_mul(g12, ur), vt = df_mul(g13, ur);
            df_mad(vr, g12, us); df_mad(vr, g13, ut);
            df_mad(vs, g22, us); df_mad(vs, g23, ut);
            df_mad(vt, g23, us); df_mad(vt, g33, ut);
            sA[q] = df_raw(vr);
            sB[q] = df_raw(vs);
            gt[k] = df_raw(vt);
        }
    }
    sync();
    dfp wt[NP];
    if (active) {
        dfp x[NP], y[NP];
        const int row = (j * NP + i) * LS;
#pragma unroll
        for (int l = 0; l < NP; ++l) x[l] = sA[row + l];
        dfl_line<NP, 1>(x, y, T);
#pragma unroll
        for (int l = 0; l < NP; ++l) sA[row + l] = y[l];
#pragma unroll
        for (int l = 0; l < NP; ++l) x[l] = sB[(j * NP + l) * LS + i];
        dfl_line<NP, 1>(x, y, T);
#pragma unroll
        for (int l = 0; l < NP; ++l) sB[(j * NP + l) * LS + i] = y[l];
        dfl_line<NP, 1>(gt, wt, T);
    }
    sync();
    if (active) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int p = k * NP2 + tid, q = (k * NP + j) * LS + i;
            dfacc s = {wt[k].hi, wt[k].lo};
            df_add(s, sA[q]);
            df_add(s, sB[q]);
            const dfacc bu = df_mul(geo[6 * NP3 + p], ru[k]);
            dfacc o = df_mul(h1, df_raw(s));
            df_mad(o, h2, df_raw(bu));
            store(p, df_join_scaled(df_raw(o), E));
        }
    }
}

// Host: the folded tables from the FP64 derivative matrix D (row-major n x n, n <= 11).
static inline void ax_dfl_tables(int n, const double *D, DflTabs *T)
{
    const int H = n / 2;
    auto pair = [](double v) {
        const float h = (float)v;
        return dfp{h, (float)(v - (double)h)};
    };
    for (int dir = 0; dir < 2; ++dir) {
        auto M = [&](int i, int l) { return dir == 0 ? D[i * n + l] : D[l * n + i]; };
        for (int i = 0; i <= H; ++i)
            for (int l = 0; l < H; ++l) {
                T->A[dir][i][l] = pair(0.5 * (M(i, l) + M(i, n - 1 - l)));
                T->B[dir][i][l] = pair(0.5 * (M(i, l) - M(i, n - 1 - l)));
            }
        for (int i = 0; i < H; ++i) T->A[dir][i][H] = pair(M(i, H));
    }
}

// ax_line32.cuh -- FP32 element operator by whole lines.
//
// The same operator as ax.cuh (w = h1 sum_a D_a^T G_ab D_b u + h2 B u on one
// element, thread (i, j) owning column u[.][j][i]), arranged so that shared
// memory is touched once per value and stage instead of once per product:
// every 1-D contraction takes a whole line into registers (the t line is the
// thread's own column; the r line (j' = i, k' = j) and the s line (i' = i,
// k' = j) come from a slab), multiplies it by D held in constant memory (the
// unrolled indices make every entry a constant-bank operand of its FMA) and
// writes the whole result line back.  At N = 7 that is about 13 shared-memory
// accesses a node instead of 35.
//
// Slab layout: row (k, j) starts at k * KS + j * LS.  For NP a multiple of 4
// rows are 16-byte aligned and read as float4; the pads put the rows of eight
// consecutive threads, and the s lines of a warp, on distinct banks (NP = 8:
// row stride 12 and plane stride 104 words).  Otherwise rows have an odd
// stride.
#pragma once

#include "common.cuh"

// D row-major, stride NP.
struct LineTab32 {
    float d[SEM_NPMAX * SEM_NPMAX];
};

template <int NP>
struct Line32Cfg {
    static constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
    static constexpr bool V4 = (NP % 4) == 0;
    static constexpr int LS = (NP % 8) == 0 ? NP + 4 : V4 ? NP : (NP | 1);
    static constexpr int KS = NP * LS + ((NP % 8) == 0 ? 8 : V4 ? 4 : 0);
    static constexpr int SLAB = NP * KS;  // floats (a multiple of 4 when V4)
};

template <int NP>
__device__ __forceinline__ void line32_read_row(const float *row, float (&x)[NP])
{
    if constexpr (Line32Cfg<NP>::V4) {
#pragma unroll
        for (int l = 0; l < NP; l += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(row + l);
            x[l] = v.x; x[l + 1] = v.y; x[l + 2] = v.z; x[l + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int l = 0; l < NP; ++l) x[l] = row[l];
    }
}

template <int NP>
__device__ __forceinline__ void line32_write_row(float *row, const float (&y)[NP])
{
    if constexpr (Line32Cfg<NP>::V4) {
#pragma unroll
        for (int l = 0; l < NP; l += 4)
            *reinterpret_cast<float4 *>(row + l) = make_float4(y[l], y[l + 1], y[l + 2], y[l + 3]);
    } else {
#pragma unroll
        for (int l = 0; l < NP; ++l) row[l] = y[l];
    }
}

// y = D x (TR = false) or D^T x (TR = true), y_i summed in order of l.
template <int NP, bool TR>
__device__ __forceinline__ void line32_mul(const float (&x)[NP], float (&y)[NP], const LineTab32 &T)
{
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        float s = T.d[TR ? i : i * NP] * x[0];
#pragma unroll
        for (int l = 1; l < NP; ++l) s = fmaf(T.d[TR ? l * NP + i : i * NP + l], x[l], s);
        y[i] = s;
    }
}

// One element.  load(k) -> float (u at node k * NP^2 + tid), store(k, w, u).
// geo: [7][NP^3].  slab: three slabs.  after_load() runs on every thread once
// the column is in registers.  Every thread of the group calls it; sync() is
// the group's barrier (four per element; the next element's first slab write
// comes after every read of this one but those of the last stage, which read
// other slabs).
template <int NP, class Load, class Store, class After, class Sync>
__device__ __forceinline__ void ax_line32_element(const Load &load, const Store &store,
                                                  const float *__restrict__ geo, float h1, float h2,
                                                  const LineTab32 &T, float *__restrict__ slab, int tid,
                                                  bool active, const After &after_load, const Sync &sync)
{
    using C = Line32Cfg<NP>;
    constexpr int NP2 = C::NP2, NP3 = C::NP3, LS = C::LS, KS = C::KS;
    float *su = slab, *sA = slab + C::SLAB, *sB = sA + C::SLAB;
    const int i = tid % NP, j = tid / NP;
    const int col = j * LS + i;         // own column: + k * KS
    const int row = j * KS + i * LS;    // r line (k' = j, j' = i)
    const int sln = j * KS + i;         // s line (k' = j, i' = i): + l * LS
    float ru[NP], gt[NP];
    if (active) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            ru[k] = load(k);
            su[k * KS + col] = ru[k];
        }
    }
    after_load();
    sync();
    if (active) {
        float x[NP], y[NP];
        line32_read_row<NP>(su + row, x);
        line32_mul<NP, false>(x, y, T);
        line32_write_row<NP>(sA + row, y);
#pragma unroll
        for (int l = 0; l < NP; ++l) x[l] = su[sln + l * LS];
        line32_mul<NP, false>(x, y, T);
#pragma unroll
        for (int l = 0; l < NP; ++l) sB[sln + l * LS] = y[l];
        line32_mul<NP, false>(ru, gt, T);
    }
    sync();
    if (active) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int p = k * NP2 + tid, q = k * KS + col;
            const float ur = sA[q], us = sB[q], ut = gt[k];
            const float g11 = geo[0 * NP3 + p], g22 = geo[1 * NP3 + p], g33 = geo[2 * NP3 + p];
            const float g12 = geo[3 * NP3 + p], g13 = geo[4 * NP3 + p], g23 = geo[5 * NP3 + p];
            sA[q] = h1 * (g11 * ur + g12 * us + g13 * ut);
            sB[q] = h1 * (g12 * ur + g22 * us + g23 * ut);
            gt[k] = h1 * (g13 * ur + g23 * us + g33 * ut);
        }
    }
    sync();
    float wt[NP];
    if (active) {
        float x[NP], y[NP];
        line32_read_row<NP>(sA + row, x);
        line32_mul<NP, true>(x, y, T);
        line32_write_row<NP>(sA + row, y);
#pragma unroll
        for (int l = 0; l < NP; ++l) x[l] = sB[sln + l * LS];
        line32_mul<NP, true>(x, y, T);
#pragma unroll
        for (int l = 0; l < NP; ++l) sB[sln + l * LS] = y[l];
        line32_mul<NP, true>(gt, wt, T);
    }
    sync();
    if (active) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int q = k * KS + col;
            const float bm = geo[6 * NP3 + k * NP2 + tid];
            store(k, fmaf(h2 * bm, ru[k], (sA[q] + sB[q]) + wt[k]), ru[k]);
        }
    }
}

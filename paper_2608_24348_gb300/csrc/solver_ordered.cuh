// solver_ordered.cuh -- the FP64 Jacobi-PCG of Taylor-Green steps with the PCG pressure
// solver: every sum in one fixed order, a node a thread.
//
// The default pressure tolerance (1e-4, absolute) stops CG after ten to twenty
// iterations on a residual that is mostly the noise of the step before it.  Such
// an iterate follows the last bits of everything that enters it: with the
// operator's quantisation, one changed bit in 1e-4 of the velocities moves the
// pressure of the next step by 1e-10 of itself, and a small velocity component
// by 2e-9 to 8e-9 (N = 7, 24^3 and 32^3 elements; 8e-8 at N = 8).  The solver of
// solver.cuh is faster (5.4 ms a launch against 6.8 at 32^3, N = 7; half the
// time at 16^3) but sums in another order; runs that are to repeat to 1e-9 therefore keep this one.
// Every FP64 solve of such a step takes this solver, whatever its tolerance, but a
// relative one below 1e-11 (native FP64 operator); where the tolerance ends the
// iteration on the solution itself, the iterates agree to 1e-10 with either solver,
// and this one costs up to twice the time.  Steps with GMRES use solver.cuh.
//
// Work items: groups of NE elements, chunks of 256 unique nodes on SEM_UQ_ROWS
// rows, chunks of 256 local nodes; they are dealt to the CTAs in turn.  The last
// CTA to arrive at the barrier of a phase sums the CTAs' partials and advances
// every problem (the phases are those of solver.cuh, but A also updates x and
// keeps r at every copy, and XUPD adds the last alpha p).
#pragma once

#include "solver.cuh"

namespace ordered {

#define SEM_UQ_ROWS 4
constexpr size_t RED_BYTES = 2048;  // reduction words of the block-floating-point element phases

template <int NP>
constexpr int group_elems()
{
    if constexpr (NP % 2 == 0)
        return BfpCfg<NP>::NE;
    else
        return AxDfCfg<NP>::NE;
}

template <int NP>
__device__ __forceinline__ int64_t phase_items(const ProbDesc &P, int ph)
{
    switch (ph) {
        case PH_JAC: case PH_FINAL: case PH_SHIFT: case PH_XUPD:
            return (P.nL + SEM_SOLVE_THREADS - 1) / SEM_SOLVE_THREADS;
        case PH_JACGS: case PH_R0: case PH_C: {
            const GsDesc &d = P.mesh.d;
            const int64_t nxch = (d.ngx + SEM_SOLVE_THREADS - 1) / SEM_SOLVE_THREADS;
            const int64_t rows = (int64_t)d.ngy * d.ngz;
            return nxch * ((rows + SEM_UQ_ROWS - 1) / SEM_UQ_ROWS);
        }
        case PH_AX0: case PH_A:
            return (P.E + group_elems<NP>() - 1) / group_elems<NP>();
        default:
            return 0;
    }
}

// Adds the block sum of v[0..2] into dst[0..2] (thread 0); all threads call.
__device__ __forceinline__ void block_accumulate(double v[3], double *s_red, double *dst)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        double s = warp_sum(v[k]);
        if (lane == 0) s_red[warp * 3 + k] = s;
        v[k] = 0.0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 0; k < 3; ++k) {
            double s = 0.0;
            for (int w = 0; w < SEM_SOLVE_THREADS / 32; ++w) s += s_red[w * 3 + k];
            dst[k] += s;
        }
    }
    __syncthreads();
}

// Element items.  KIND 0: w = A x;  KIND 1: x += alpha p, p = z + beta p, w = A p, <p,w>.
template <int NP, int KIND>
__device__ __forceinline__ void elem_item_bfp(const ProbDesc &P, double alpha, double beta, int first,
                                              int64_t g, unsigned char *smem, double &acc)
{
    using C = BfpCfg<NP>;
    static_assert(8 * C::NE * sizeof(unsigned) <= RED_BYTES, "reduction words");
    unsigned *red = reinterpret_cast<unsigned *>(smem);
    dfp *slabs = reinterpret_cast<dfp *>(smem + RED_BYTES);
    const int grp = threadIdx.x / C::NP2;
    const bool inrange = grp < C::NE;
    // threads beyond the last whole element take part in the barriers only
    const int tid = inrange ? (int)threadIdx.x - grp * C::NP2 : -1;
    const int gs = inrange ? grp : 0;
    const int64_t e = g * C::NE + grp;
    const bool active = inrange && e < P.E;
    const int64_t off = (active ? e : 0) * C::NP3;
    const dfp *geo = P.geodf + (active ? e : 0) * 7 * C::NP3;
    const float h1h = (float)P.h1, h2h = (float)P.h2;
    const dfp H1 = {h1h, (float)(P.h1 - (double)h1h)}, H2 = {h2h, (float)(P.h2 - (double)h2h)};
    if (threadIdx.x == 0) geo_prefetch<NP>(P.geodf, g * C::NE, C::NE, P.E, 8);
    const BfpTabs &T = c_tabs[NP].bfp;
    const auto sync = [] { __syncthreads(); };
    dfp *slab = slabs + (size_t)gs * 3 * C::SLAB;
    if (KIND == 0) {
        const double *x = P.x + off;
        double *w = P.w + off;
        auto load = [&](int q) { return __ldcg(x + q); };
        auto store = [&](int q, double v) { w[q] = v; };
        ax_bfp_element<NP, false>(load, store, geo, H1, H2, T, slab, red + gs * 8, tid, active, [] {}, sync);
    } else {
        const double *r = P.r + off, *mi = P.minv + off;
        double *p = P.p + off, *w = P.w + off, *x = P.x + off;
        auto load = [&](int q) {
            double pn = __ldcg(mi + q) * __ldcg(r + q);
            if (!first) {
                const double po = __ldcg(p + q);
                x[q] = fma(alpha, po, __ldcg(x + q));
                pn = fma(beta, po, pn);
            }
            p[q] = pn;
            return pn;
        };
        auto store = [&](int q, double v) {
            w[q] = v;
            acc = fma(__ldcg(p + q), v, acc);
        };
        ax_bfp_element<NP, false>(load, store, geo, H1, H2, T, slab, red + gs * 8, tid, active, [] {}, sync);
    }
}

template <int NP, int KIND>
__device__ __forceinline__ void elem_item_df(const ProbDesc &P, double alpha, double beta, int first,
                                             int64_t g, unsigned char *smem, double &acc)
{
    using C = AxDfCfg<NP>;
    dfp *sm = reinterpret_cast<dfp *>(smem);
    dfp *sD = sm, *sDT = sm + NP * NP;
    int *sexp = reinterpret_cast<int *>(sm + 2 * NP * NP + (size_t)C::NE * 3 * C::NP3);
    const int grp = threadIdx.x / C::NP2;
    const int tid = threadIdx.x - grp * C::NP2;
    const bool inrange = grp < C::NE;
    const int64_t e = g * C::NE + grp;
    const bool active = inrange && e < P.E;
    dfp *su = sm + 2 * NP * NP + (size_t)(inrange ? grp : 0) * 3 * C::NP3;
    dfp *svr = su + C::NP3, *svs = svr + C::NP3;
    const int64_t off = (active ? e : 0) * C::NP3;
    const dfp *geo = P.geodf + (active ? e : 0) * 7 * C::NP3;
    const float h1h = (float)P.h1, h2h = (float)P.h2;
    const dfp H1 = {h1h, (float)(P.h1 - (double)h1h)}, H2 = {h2h, (float)(P.h2 - (double)h2h)};
    if (threadIdx.x == 0) geo_prefetch<NP>(P.geodf, g * C::NE, C::NE, P.E, 8);
    ax_df_load_D<NP>(P.Ddf, sD, sDT);
    int *myexp = sexp + (inrange ? grp : 0);
    if (KIND == 0) {
        const double *x = P.x + off;
        double *w = P.w + off;
        auto load = [&](int q) { return __ldcg(x + q); };
        auto store = [&](int q, double v) { w[q] = v; };
        ax_df_element<NP>(load, store, geo, H1, H2, sD, sDT, su, svr, svs, myexp, tid, active);
    } else {
        const double *r = P.r + off, *mi = P.minv + off;
        double *p = P.p + off, *w = P.w + off, *x = P.x + off;
        auto load = [&](int q) {
            double pn = __ldcg(mi + q) * __ldcg(r + q);
            if (!first) {
                const double po = __ldcg(p + q);
                x[q] = fma(alpha, po, __ldcg(x + q));
                pn = fma(beta, po, pn);
            }
            p[q] = pn;
            return pn;
        };
        auto store = [&](int q, double v) {
            w[q] = v;
            acc = fma(__ldcg(p + q), v, acc);
        };
        ax_df_element<NP>(load, store, geo, H1, H2, sD, sDT, su, svr, svs, myexp, tid, active);
    }
}

template <int NP, int KIND>
__device__ __forceinline__ void elem_item(const ProbDesc &P, double alpha, double beta, int first, int64_t g,
                                          unsigned char *smem, double &acc)
{
    if constexpr (NP % 2 == 0)
        elem_item_bfp<NP, KIND>(P, alpha, beta, first, g, smem, acc);
    else
        elem_item_df<NP, KIND>(P, alpha, beta, first, g, smem, acc);
}

// y/z copies of one row (gy, gz) of unique nodes: local offsets without the x part.
struct RowCopies {
    int m;
    int64_t off[4];
};

__device__ __forceinline__ void row_copies(const GsDesc &d, int row, RowCopies &R)
{
    const int gy = row % d.ngy, gz = row / d.ngy;
    int ey[2], iy[2], ez[2], iz[2];
    const int my = gs_copies_1d(gy, d.N, d.nely, d.py, ey, iy);
    const int mz = gs_copies_1d(gz, d.N, d.nelz, d.pz, ez, iz);
    const int64_t n3 = (int64_t)d.n * d.n * d.n;
    R.m = 0;
    for (int c = 0; c < mz; ++c)
        for (int b = 0; b < my; ++b)
            R.off[R.m++] = ((int64_t)ey[b] + (int64_t)d.nely * ez[c]) * d.nelx * n3 +
                           (int64_t)(iz[c] * d.n + iy[b]) * d.n;
}

// Copy k (y/z part) x a (x part) of a unique node; valid when k < R.m, a < mx.
#define UQ_FOR_COPIES(R, mx, xo, BODY)                              \
    _Pragma("unroll") for (int k_ = 0; k_ < 4; ++k_)                \
        _Pragma("unroll") for (int a_ = 0; a_ < 2; ++a_)            \
            if (k_ < (R).m && a_ < (mx)) {                          \
                const int64_t cp = (R).off[k_] + (xo)[a_];          \
                BODY;                                               \
            }

__device__ __forceinline__ void uniq_item(const ProbDesc &P, const PState &S, int ph, int64_t item,
                                          double v[3])
{
    const GsDesc &d = P.mesh.d;
    const int nxch = (d.ngx + SEM_SOLVE_THREADS - 1) / SEM_SOLVE_THREADS;
    const int it32 = (int)item;  // unique-node items fit in 32 bits (checked at setup)
    const int rg = it32 / nxch;
    const int gx = (it32 - rg * nxch) * SEM_SOLVE_THREADS + threadIdx.x;
    const int rows = d.ngy * d.ngz;
    if (gx >= d.ngx) return;
    const int64_t n3 = (int64_t)d.n * d.n * d.n;
    int ex[2], ix[2];
    const int mx = gs_copies_1d(gx, d.N, d.nelx, d.px, ex, ix);
    const int64_t xo[2] = {ex[0] * n3 + ix[0], mx > 1 ? ex[1] * n3 + ix[1] : 0};
    constexpr int RU = SEM_UQ_ROWS;
    RowCopies R[RU];
    bool ok[RU];
#pragma unroll
    for (int r = 0; r < RU; ++r) {
        const int row = rg * RU + r;
        ok[r] = row < rows;
        if (ok[r]) row_copies(d, row, R[r]);
        else R[r].m = 0;
    }
    switch (ph) {
        case PH_JACGS: {
            if (S.jac) {  // the Jacobi inverse is kept from an earlier solve: only sum b
#pragma unroll
                for (int r = 0; r < RU; ++r)
                    if (ok[r]) v[0] += __ldcg(P.b + R[r].off[0] + xo[0]);
                break;
            }
            double s[RU], bv[RU];
#pragma unroll
            for (int r = 0; r < RU; ++r) {
                s[r] = 0.0;
                bv[r] = 0.0;
                if (!ok[r]) continue;
                UQ_FOR_COPIES(R[r], mx, xo, s[r] += __ldcg(P.minv + cp));
                bv[r] = __ldcg(P.b + R[r].off[0] + xo[0]);
            }
#pragma unroll
            for (int r = 0; r < RU; ++r) {
                if (!ok[r]) continue;
                const double rinv = 1.0 / s[r];
                UQ_FOR_COPIES(R[r], mx, xo, P.minv[cp] = rinv);
                v[0] += bv[r];
            }
        } break;
        case PH_R0: {
            double s[RU], bv[RU], mv[RU];
#pragma unroll
            for (int r = 0; r < RU; ++r) {
                s[r] = 0.0;
                bv[r] = mv[r] = 0.0;
                if (!ok[r]) continue;
                UQ_FOR_COPIES(R[r], mx, xo, s[r] += __ldcg(P.w + cp));
                const int64_t f = R[r].off[0] + xo[0];
                bv[r] = __ldcg(P.b + f) - S.bmean;
                mv[r] = __ldcg(P.minv + f);
            }
#pragma unroll
            for (int r = 0; r < RU; ++r) {
                if (!ok[r]) continue;
                const double rv = bv[r] - s[r];
                UQ_FOR_COPIES(R[r], mx, xo, P.r[cp] = rv);
                v[0] = fma(rv, rv, v[0]);
                v[1] = fma(rv, mv[r] * rv, v[1]);
                v[2] = fma(bv[r], bv[r], v[2]);
            }
        } break;
        case PH_C: {
            double s[RU], r0[RU], mv[RU];
#pragma unroll
            for (int r = 0; r < RU; ++r) {
                s[r] = r0[r] = mv[r] = 0.0;
                if (!ok[r]) continue;
                UQ_FOR_COPIES(R[r], mx, xo, s[r] += __ldcg(P.w + cp));
                const int64_t f = R[r].off[0] + xo[0];
                r0[r] = __ldcg(P.r + f);
                mv[r] = __ldcg(P.minv + f);
            }
#pragma unroll
            for (int r = 0; r < RU; ++r) {
                if (!ok[r]) continue;
                const double rv = r0[r] - S.alpha * s[r];
                UQ_FOR_COPIES(R[r], mx, xo, P.r[cp] = rv);
                v[0] = fma(rv, rv, v[0]);
                v[1] = fma(rv, mv[r] * rv, v[1]);
            }
        } break;
        default: break;
    }
}

__device__ __forceinline__ void local_item(const ProbDesc &P, const PState &S, int ph, int64_t chunk,
                                           double v[3])
{
    const int64_t q = chunk * SEM_SOLVE_THREADS + threadIdx.x;
    if (q >= P.nL) return;
    const int n = P.n, n3 = n * n * n;
    const int64_t e = q / n3;
    const int l = (int)(q - e * n3);
    switch (ph) {
        case PH_JAC: {
            const int i = l % n, j = (l / n) % n, k = l / (n * n);
            const double *g = P.geo64 + e * 7 * n3;
            const double *D = P.D64;
            double s = 0.0;
            for (int t = 0; t < n; ++t) {
                const double a = D[t * n + i], b = D[t * n + j], c = D[t * n + k];
                s += a * a * g[0 * n3 + (k * n + j) * n + t];
                s += b * b * g[1 * n3 + (k * n + t) * n + i];
                s += c * c * g[2 * n3 + (t * n + j) * n + i];
            }
            const double di = D[i * n + i], dj = D[j * n + j], dk = D[k * n + k];
            s += 2.0 * (di * dj * g[3 * n3 + l] + di * dk * g[4 * n3 + l] + dj * dk * g[5 * n3 + l]);
            P.minv[q] = P.h1 * s + P.h2 * g[6 * n3 + l];
        } break;
        case PH_XUPD:
            P.x[q] = fma(S.alpha, __ldcg(P.p + q), __ldcg(P.x + q));
            break;
        case PH_FINAL:
            v[0] = fma(P.geo64[(e * 7 + 6) * n3 + l], __ldcg(P.x + q), v[0]);
            break;
        case PH_SHIFT:
            P.x[q] = __ldcg(P.x + q) - S.shift;
            break;
        default: break;
    }
}

static __device__ void advance(const SolveParams<8> &prm, const ProbDesc &P, PState &S, const double *red)
{
    const int ph = S.phase;
    auto finish = [&](int status) {
        S.status = status;
        S.phase = P.singular ? PH_FINAL : PH_DONE;
    };
    // after a C phase the last alpha p is not yet in x
    auto finish_pending = [&](int status) {
        S.status = status;
        S.phase = PH_XUPD;
    };
    switch (ph) {
        case PH_JAC: S.phase = PH_JACGS; break;
        case PH_JACGS:
            S.bmean = P.singular ? red[0] / (double)P.nG : 0.0;
            S.phase = PH_AX0;
            break;
        case PH_AX0: S.phase = PH_R0; break;
        case PH_R0: {
            S.bnorm = sqrt(red[2]);
            S.rnorm = sqrt(red[0]);
            S.target = prm.abs_tol ? prm.tol : prm.tol * S.bnorm;
            if (!isfinite(S.rnorm) || !isfinite(S.bnorm)) { finish(SEM_ERR_BREAKDOWN); break; }
            if (S.rnorm <= S.target) { finish(SEM_OK); break; }
            if (prm.maxit <= 0) { finish(SEM_ERR_NOT_CONVERGED); break; }
            S.rz = red[1];
            S.first = 1;
            S.beta = 0.0;
            S.phase = PH_A;
        } break;
        case PH_A: {
            const double pw = red[0];
            if (!(pw > 0.0) || !isfinite(pw)) { finish(SEM_ERR_BREAKDOWN); break; }
            S.alpha = S.rz / pw;
            S.phase = PH_C;
        } break;
        case PH_C: {
            S.iters += 1;
            S.rnorm = sqrt(red[0]);
            if (!isfinite(S.rnorm)) { finish_pending(SEM_ERR_BREAKDOWN); break; }
            if (S.rnorm <= S.target) { finish_pending(SEM_OK); break; }
            if (S.iters >= prm.maxit) { finish_pending(SEM_ERR_NOT_CONVERGED); break; }
            S.beta = red[1] / S.rz;
            S.rz = red[1];
            S.first = 0;
            S.phase = PH_A;
        } break;
        case PH_FINAL: S.shift = red[0] / P.volume; S.phase = PH_SHIFT; break;
        case PH_SHIFT: S.phase = PH_DONE; break;
        case PH_XUPD: S.phase = P.singular ? PH_FINAL : PH_DONE; break;
        default: S.phase = PH_DONE; break;
    }
}

template <int NP>
__global__ void __launch_bounds__(SEM_SOLVE_THREADS, 2)
    k_solve_ordered(const __grid_constant__ SolveParams<8> prm)
{
    constexpr int MAXP = 8;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double s_part[MAXP][3];
    __shared__ double s_red[SEM_SOLVE_THREADS / 32 * 3];
    __shared__ int s_phase[MAXP];
    __shared__ long long s_offs[MAXP + 1];
    __shared__ double s_alpha[MAXP], s_beta[MAXP], s_bmean[MAXP], s_shift[MAXP];
    __shared__ int s_first[MAXP], s_jac[MAXP];
    __shared__ int s_last, s_stop;
    __shared__ unsigned s_gen;
    const int np = prm.nprob;
    SyncState *sync = prm.sync;
    if constexpr (NP % 2 == 0)  // reduction words of the block-floating-point element phases
        for (int t = threadIdx.x; t < RED_BYTES / 4; t += blockDim.x) reinterpret_cast<unsigned *>(smem)[t] = 0u;

    for (int step = 0;; ++step) {
        // ---- schedule of this step
        if (threadIdx.x == 0) {
            long long o = 0;
            for (int p = 0; p < np; ++p) {
                int ph;
                if (step == 0) {
                    const ProbDesc &P = prm.prob[p];
                    s_jac[p] = jac_kept(P);
                    ph = s_jac[p] ? PH_JACGS : PH_JAC;
                    // (CTAs that read the word after this find it incomplete as well)
                    if (blockIdx.x == 0 && !s_jac[p]) *P.jac_dev = 0u;
                } else {
                    ph = ((volatile PState *)prm.st)[p].phase;
                }
                s_phase[p] = ph;
                s_offs[p] = o;
                o += phase_items<NP>(prm.prob[p], ph);
            }
            s_offs[np] = o;
            s_stop = (step > 0 && ((volatile int *)&sync->finished)[0]) ||
                     ((volatile int *)&sync->err)[0];
        }
        for (int p = threadIdx.x; p < np; p += blockDim.x) {
            const volatile PState *S = prm.st + p;
            s_alpha[p] = S->alpha;
            s_beta[p] = S->beta;
            s_bmean[p] = S->bmean;
            s_shift[p] = S->shift;
            s_first[p] = S->first;
            s_part[p][0] = s_part[p][1] = s_part[p][2] = 0.0;
        }
        __syncthreads();
        if (s_stop) break;

        // ---- work items
        const long long total = s_offs[np];
        double v[3] = {0.0, 0.0, 0.0};
        double acc = 0.0;
        int cur = -1;
        for (long long it = blockIdx.x; it < total; it += gridDim.x) {
            int p = 0;
            while (p + 1 < np && s_offs[p + 1] <= it) ++p;
            if (p != cur) {
                if (cur >= 0) {
                    v[0] += acc;
                    acc = 0.0;
                    block_accumulate(v, s_red, s_part[cur]);
                }
                cur = p;
            }
            const ProbDesc &P = prm.prob[p];
            const int ph = s_phase[p];
            const int64_t local = it - s_offs[p];
            PState S;
            S.alpha = s_alpha[p];
            S.beta = s_beta[p];
            S.bmean = s_bmean[p];
            S.shift = s_shift[p];
            S.jac = s_jac[p];
            if (ph == PH_AX0) {
                elem_item<NP, 0>(P, 0.0, 0.0, 1, local, smem, acc);
            } else if (ph == PH_A) {
                elem_item<NP, 1>(P, S.alpha, S.beta, s_first[p], local, smem, acc);
            } else if (ph == PH_JAC || ph == PH_FINAL || ph == PH_SHIFT || ph == PH_XUPD) {
                local_item(P, S, ph, local, v);
            } else {
                uniq_item(P, S, ph, local, v);
            }
        }
        if (cur >= 0) {
            v[0] += acc;
            block_accumulate(v, s_red, s_part[cur]);
        }

        // ---- publish partials, reducing barrier
        double *part = prm.partials + (size_t)blockIdx.x * MAXP * 3;
        for (int t = threadIdx.x; t < np * 3; t += blockDim.x) part[t] = s_part[t / 3][t % 3];
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            s_gen = ((volatile unsigned *)&sync->gen)[0];
            const unsigned arrived = atomicAdd(&sync->count, 1u);
            s_last = (arrived == gridDim.x - 1);
        }
        __syncthreads();
        if (s_last) {
            __threadfence();
            // fixed-order reduction of every (problem, value) pair: one warp each
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
            for (int pk = warp; pk < np * 3; pk += SEM_SOLVE_THREADS / 32) {
                const int p = pk / 3, k = pk % 3;
                double s = 0.0;
                if (k < phase_nvals(s_phase[p]))
                    for (int b = lane; b < (int)gridDim.x; b += 32)
                        s += __ldcg(prm.partials + ((size_t)b * MAXP + p) * 3 + k);
                s = warp_sum(s);
                if (lane == 0) s_part[p][k] = s;
            }
            __syncthreads();
            for (int p = threadIdx.x; p < np; p += blockDim.x) {
                PState S = prm.st[p];
                S.phase = s_phase[p];
                // (every CTA has read the word before it arrived here)
                if (S.phase == PH_JACGS && !s_jac[p]) *prm.prob[p].jac_dev = jac_bits(prm.prob[p]);
                advance(prm, prm.prob[p], S, s_part[p]);
                prm.st[p] = S;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                int fin = 1;
                for (int p = 0; p < np; ++p) fin &= (prm.st[p].phase == PH_DONE);
                sync->finished = fin;
                sync->count = 0;
                __threadfence();
                atomicAdd(&sync->gen, 1u);
            }
        } else if (threadIdx.x == 0) {
            const unsigned long long t0 = sem_globaltimer();
            while (ld_acquire_u32(&sync->gen) == s_gen) {
                if (((volatile int *)&sync->err)[0]) break;
                if ((long long)(sem_globaltimer() - t0) > prm.timeout_ns) {
                    atomicExch(&sync->err, SEM_ERR_TIMEOUT);
                    break;
                }
                __nanosleep(128);
            }
            __threadfence();
        }
        __syncthreads();
    }
}

template <int NP>
constexpr size_t smem_bytes()
{
    if constexpr (NP % 2 == 0)
        return RED_BYTES + ax_bfp_smem_bytes_ne<NP, BfpCfg<NP>::NE>();
    else
        return ax_df_smem_bytes<NP>();
}

// Host launcher (cooperative, grid sized for co-residency).
template <int NP>
int launch(const SolveParams<8> &prm, int num_sms, cudaStream_t s)
{
    auto kern = k_solve_ordered<NP>;
    const size_t smem = smem_bytes<NP>();
    static std::atomic<unsigned> attr{0};
    SEM_CUDA(sem_smem_attr(kern, smem, attr));
    int per_sm = 0;
    SEM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, SEM_SOLVE_THREADS, smem));
    if (per_sm < 1) return SEM_ERR_ARG;
    long long grid = (long long)per_sm * num_sms, most = 1;
    for (int p = 0; p < prm.nprob; ++p) {
        const long long m = (prm.prob[p].nL + SEM_SOLVE_THREADS - 1) / SEM_SOLVE_THREADS;
        if (m > most) most = m;
    }
    if (grid > most) grid = most;
    if (grid * 8 * 3 > prm.partials_cap) return SEM_ERR_ARG;
    void *args[] = {(void *)&prm};
    SEM_CUDA(cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)grid), dim3(SEM_SOLVE_THREADS), args,
                                         smem, s));
    return SEM_OK;
}

}  // namespace ordered

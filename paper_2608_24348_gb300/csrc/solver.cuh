// solver.cuh -- persistent, cooperative Jacobi-PCG / FP64 iterative refinement.
//
// One launch runs a whole solve (or a batch of independent solves).  Every
// problem carries a small state machine; all problems advance together in
// "grid steps".  In a step each problem executes the work items of its
// current phase (element groups, unique nodes or local nodes), every CTA
// publishes its FP64 partial sums, and a grid barrier ends the step.  Behind
// the barrier every CTA sums the published partials in the same fixed order
// and advances its own copy of every state machine (in shared memory), so the
// decision costs one exchange and is the same everywhere (deterministic).
// Every wait is bounded in time; a CTA that gives up raises SEM_ERR_TIMEOUT
// and the whole grid exits.
//
// Phases of one problem (Sec. 1.1: CG with Jacobi; Sec. 2: dot products and
// norms reduced in fp64):
//   JAC    local   minv = local diagonal of A
//   JACGS  unique  minv = 1/dssum(minv);  sum b  (mean removal when h2 == 0)
//   AX0    element w = A x                                      (FP64)
//   R0     unique  r = b' - dssum(w); w <- z = minv r; <r,r>, <r,z>, <b',b'>
//   A      element p = z + beta p; w <- A p; <p,w>
//   C      unique  r -= alpha dssum(w); y += alpha p (x += alpha p in the first
//                  X_DIRECT iterations); w <- z = minv r; <r,r>, <r,z>
//   XUPD   unique  x += y                                       (after the last C)
//   R64    unique  r = b' - dssum(w); <r,r>, <b',b'>            (refinement)
//   INIT32 unique  r32 = r / ||r||; d = 0; w32 <- z32; <r32,r32>, <r32,z32>
//   A32    element p32 = z32 + beta p32; w32 <- A32 p32; <p32,w32>
//   C32    unique  r32 -= alpha dssum(w32); d += alpha p32; w32 <- z32; <r32,r32>, <r32,z32>
//   UPD    unique  p = x (kept until the next FP64 residual accepts the step);
//                  x += ||r|| d
//   XREST  local   x = p: a refinement step that raised the FP64 residual is
//                  undone, so a solve never returns an iterate worse than the
//                  one it had before that step
//   FINAL  local   sum B x              (h2 == 0: remove the B-weighted mean)
//   SHIFT  local   x -= sum(B x) / sum(B)
// The inner product <a,b> = sum_local a b / mult is evaluated over unique
// nodes, where it is a plain sum; <p, dssum(Ap)> equals sum_local p (Ap)
// for a continuous p, which lets the element phase produce it directly.
//
// Where each vector lives: z and A p share one E-vector (w): the unique phase
// gathers every copy of A p and puts z in their place, the element phase reads
// its element's z and puts A p there.  r, y (the sum of the corrections; d in
// FP32) and the preconditioner are read and written at the first copy of every
// unique node only.  So the element phase, whose arithmetic dominates, has two
// input streams (z, p) instead of the four of a fused x and p update, and the
// solution's update rides in the streaming phase: 144 bytes a node and
// iteration in FP64.
//
// Element phases copy the next element's two input columns into shared memory
// with asynchronous copies (cp.async; every thread copies and reads only its
// own column, so no barrier guards them) while the current element is in
// flight, and synchronise per element group (a named barrier over the group's
// warps), so the groups of a CTA do not move in step.  Unique phases map one
// thread to a few consecutive nodes of one element's row.  A CTA of the line
// phases fills its multiprocessor (512 threads of 128 registers in FP64, 768 of
// 80 in FP32), so a barrier has 152 arrivals and the redundant sums behind it
// run once a multiprocessor.
#pragma once

#include <string.h>

#include "ax.cuh"
#include "ax_bfp.cuh"
#include "ax_df.cuh"
#include "ax_dfl.cuh"
#include "ax_line32.cuh"
#include "ax_tc.cuh"
#include "common.cuh"
#include "sum3.cuh"
#include "tma.cuh"
#include "uniq.cuh"

#define SEM_MAXP 64
// Threads of a CTA whose element phases are not line phases (see solve_threads).
#define SEM_SOLVE_THREADS 256

// Which element operators a solver kernel carries (keeps each kernel's
// register budget to what its mode needs).
// MODE_F64 evaluates the FP64 operator on the FP32 pipes (block-floating-point
// or float pairs); MODE_F64N uses native FP64 arithmetic.
enum SolveMode { MODE_F64 = 0, MODE_F32 = 1, MODE_TC = 2, MODE_F64N = 3 };

enum SolvePhase {
    PH_JAC = 0, PH_JACGS, PH_AX0, PH_R0, PH_A, PH_C, PH_R64, PH_INIT32, PH_A32, PH_C32, PH_UPD,
    PH_FINAL, PH_SHIFT, PH_XUPD, PH_XREST, PH_DONE
};

struct ProbDesc {
    int n, NE, NE32, singular;  // NE: elements per group (CUDA cores); NE32: inner operator
    int tc;                     // inner path of a MODE_TC launch: 0 FP32 CUDA cores, 1 BF16, 2 FP16,
                                // 3 FP16 x2, 4 BF16 x3 tensor cores
    int jac_cached;             // an earlier launch was to leave this problem's Jacobi inverse in minv
                                // (and minv32 if mixed); *jac_dev says whether it did
    int vec;                    // b and x are aligned for vector accesses
    int jac_shared;             // an earlier problem of the launch makes (or keeps) the inverse in minv
    int64_t E, nL, nG;
    UqMesh mesh;
    FastDiv dn3;
    double volume, h1, h2;
    const double *geo64;
    const float *geo32;
    const dfp *geodf;
    const double *D64;
    const float *D32;
    const dfp *Ddf;
    const double *b;
    double *x;
    double *r, *p, *w, *minv;
    double *y;          // the sum of the corrections; null: x is updated in every iteration instead
    unsigned *jac_dev;  // bit 0: minv, bit 1: minv32 hold a whole inverse (null: never kept)
    float *r32, *p32, *w32, *d32, *minv32;
};

struct PState {
    int phase, iters, outer, inner_iters, status, first;
    int jac;  // the Jacobi inverse was there when the launch began
    // rnorm: its square while an FP64 solve is between two C phases
    double rz, alpha, beta, bnorm, rnorm, target, bmean, scale, prev_rnorm, inner_target, shift;
};

struct SyncState {
    unsigned count, gen;
    int err, finished;
};

template <int MAXP>
struct SolveParams {
    int nprob, mixed, abs_tol, maxit, max_outer;
    double tol, inner_tol;
    long long timeout_ns;
    SyncState *sync;
    PState *st;
    double *partials;       // two buffers of [MAXP * 3][gridDim]
    long long partials_cap; // doubles that fit
    unsigned char order[MAXP]; // the problems by polynomial order
    ProbDesc prob[MAXP];
};

// ---------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------

__device__ __forceinline__ unsigned long long sem_globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_add_u32(unsigned *p, unsigned v)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Phases whose sums are gathered in floats (Sum3).
__device__ __forceinline__ bool phase_floats(int ph)
{
    return ph == PH_A32 || ph == PH_C32 || ph == PH_INIT32;
}

// Bits of *P.jac_dev that a solve of P needs and a whole JACGS phase leaves.  A
// launch that times out before that leaves zero: the next one makes the inverse.
__device__ __forceinline__ unsigned jac_bits(const ProbDesc &P) { return P.minv32 ? 3u : 1u; }

__device__ __forceinline__ bool jac_kept(const ProbDesc &P)
{
    return P.jac_cached && (*(const volatile unsigned *)P.jac_dev & jac_bits(P)) == jac_bits(P);
}

__host__ __device__ __forceinline__ int phase_nvals(int ph)
{
    switch (ph) {
        case PH_JACGS: return 1;
        case PH_R0: return 3;
        case PH_A: case PH_A32: return 1;
        case PH_C: case PH_C32: case PH_R64: case PH_INIT32: return 2;
        case PH_FINAL: return 1;
        default: return 0;
    }
}

// FP32 dot products accumulated on the FP32 pipes: every product exact
// (TwoProd), every sum error-free (TwoSum), the errors gathered in A.e -- the
// compensated dot product of Ogita, Rump & Oishi, as accurate as summing the
// exact products in twice FP32 precision.  GB300 runs FP64 at 1/58 of the
// FP32 rate, so the per-node FP64 multiply-add (and two conversions) this
// replaces cost more issue time than the ten FP32 operations here.
__device__ __forceinline__ void dot2_acc(dfacc &A, float a, float b)
{
    const float p = __fmul_rn(a, b);
    const float ep = __fmaf_rn(a, b, -p);
    const float s = __fadd_rn(A.s, p);
    const float bv = __fsub_rn(s, A.s);
    const float t = __fadd_rn(__fsub_rn(A.s, __fsub_rn(s, bv)), __fsub_rn(p, bv));
    A.s = s;
    A.e = __fadd_rn(A.e, __fadd_rn(t, ep));
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The sum of a thread's values by halves: the additions of one level are
// independent, and FP64 additions are slow to return on this part.
template <int N>
__device__ __forceinline__ double tree_sum(double (&t)[N])
{
#pragma unroll
    for (int m = N; m > 1; m = (m + 1) / 2)
#pragma unroll
        for (int j = 0; j < m / 2; ++j) t[j] += t[j + (m + 1) / 2];
    return t[0];
}

// A lane's L2 prefetch of the geometric factors of the element group it is
// about to work on (elements [e0, e0 + ne) of a [E][7][NP^3] array of
// wb-byte words): the operator reads them after its gradient stage, about
// half an element phase later.  (A whole group ahead let L2 evict the element
// phase's output before the gather read it.)
template <int NP>
__device__ __forceinline__ void geo_prefetch(const void *geo, int64_t e0, int ne, int64_t E, int wb)
{
    constexpr int64_t N3 = NP * NP * NP;
    if (e0 >= E) return;
    const int64_t e1 = e0 + ne < E ? e0 + ne : E;
    l2_prefetch_span(geo, e0 * 7 * N3 * wb, e1 * 7 * N3 * wb);
}

// ---------------------------------------------------------------------------
// element phases
// ---------------------------------------------------------------------------

// Element groups of the staged phases: GE elements on GT threads (whole
// warps), the smallest GT that keeps about 80 % of its lanes busy.
__host__ __device__ constexpr int grp_threads(int np)
{
    return np <= 4 ? 32 : np == 8 ? 64 : (np == 5 || np == 6 || np == 10 || np == 11) ? 128 : 256;
}
__host__ __device__ constexpr int grp_elems(int np) { return grp_threads(np) / (np * np); }

template <int NP, int TH>
struct GrpCfg {
    static constexpr int GT = grp_threads(NP), GE = grp_elems(NP);
    static constexpr int NG = TH / GT;  // groups per CTA
    static constexpr int NE = NG * GE;  // elements per CTA
};

// Barrier over one element group of a CTA of TH threads.
template <int GT, int TH>
struct GrpSync {
    int grp;
    __device__ __forceinline__ void operator()() const
    {
        if constexpr (GT == TH)
            __syncthreads();
        else if constexpr (GT == 32)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(GT) : "memory");
    }
};

// The calling thread's place in its element group.
template <int NP>
struct GrpThread {
    int grp, ge, tid;  // tid: column owner 0 .. NP^2 - 1, or -1 (takes part in the barriers only)
    __device__ __forceinline__ GrpThread()
    {
        constexpr int GT = grp_threads(NP), GE = grp_elems(NP);
        grp = threadIdx.x / GT;
        const int lt = threadIdx.x - grp * GT;
        ge = lt / (NP * NP);
        tid = ge < GE ? lt - ge * NP * NP : -1;
        if (tid < 0) ge = 0;
    }
};

// One problem's place in a step: its portions are dealt to slots, a slot being
// one group of warps, slot k on CTA k % ncta: a problem smaller than the
// machine spreads over the multiprocessors before it fills any of them, and the
// last round of a larger one leaves every multiprocessor about as many busy
// groups.  The next problem of the step goes on where the last one ended: rot
// counts slots of one warp.
struct Deal {
    unsigned cta, ncta, rot;
    // the first portion of group grp of a CTA that has ng groups of wpg warps;
    // the group's next ones follow ncta * ng apart
    __device__ __forceinline__ unsigned first(unsigned grp, unsigned wpg, unsigned ng) const
    {
        const unsigned n = ncta * ng;
        unsigned s = grp * ncta + cta;
        if (rot) s += n - (rot % ncta + ncta * (rot / ncta / wpg)) % n;
        return s < n ? s : s - n;
    }
    // the next problem's start after this one dealt out `portions`
    __device__ __forceinline__ unsigned after(unsigned portions, unsigned wpg, unsigned ng, unsigned nw) const
    {
        const unsigned n = ncta * ng;
        const unsigned s = (rot % ncta + ncta * (rot / ncta / wpg) + portions) % n;
        return (s % ncta + (s / ncta) * wpg * ncta) % (ncta * nw);
    }
};

// FP64-accurate phases stage two columns (z, p) per thread and keep the new p
// for the inner product in a third where the shared memory allows it.
template <int NP>
constexpr bool stage_keep_p()
{
    return NP <= 8;
}

template <int NP, int TH>
__host__ __device__ constexpr size_t stage64_bytes()
{
    return sizeof(double) * (stage_keep_p<NP>() ? 3 : 2) * NP * TH;
}

template <int NP, int TH>
__host__ __device__ constexpr size_t elem32_smem_bytes()
{
    return sizeof(float) * ((size_t)GrpCfg<NP, TH>::NE * 3 * Line32Cfg<NP>::SLAB + 2 * NP * TH);
}

// Shared memory of one low-register element, a multiple of 16 bytes.
template <int NP>
__host__ __device__ constexpr size_t lowreg_smem_bytes()
{
    return (ax_df_lowreg_smem_bytes<NP>() + 15) / 16 * 16;
}

// Tables of the line operators, one copy per translation unit and order
// (constant-bank operands in the unrolled contractions): the FP32 operator's, and
// the FP64-accurate one's for the order's parity.  Filled at context setup,
// outside any stream capture, by solver_upload_tables.
struct SolveTabs {
    LineTab32 l;
    union {
        BfpTabs bfp;
        DflTabs dfl;
    };
};
static __constant__ SolveTabs c_tabs[SEM_NPMAX + 1];

// A32: p32 = z32 + beta p32, w32 <- A32 p32, <p32, w32>, by whole lines.
template <int NP, int TH>
__device__ __forceinline__ void phase_a32(const ProbDesc &P, double beta, int first, const Deal &deal,
                                          unsigned char *smem, Sum3 &sum)
{
    using G = GrpCfg<NP, TH>;
    constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
    const GrpThread<NP> th;
    const GrpSync<G::GT, TH> sync{th.grp};
    float *slabs = reinterpret_cast<float *>(smem);
    float *slab = slabs + (size_t)(th.grp * G::GE + th.ge) * 3 * Line32Cfg<NP>::SLAB;
    float *sz = slabs + (size_t)G::NE * 3 * Line32Cfg<NP>::SLAB + threadIdx.x;
    float *sp = sz + NP * TH;
    const float b32 = (float)beta, h1 = (float)P.h1, h2 = (float)P.h2;
    const int E = (int)P.E, ngr = (E + G::GE - 1) / G::GE;
    auto fetch = [&](int g) {
        const int e = g * G::GE + th.ge;
        if (g < ngr && th.tid >= 0 && e < E) {
            const size_t off = (size_t)e * NP3 + th.tid;
#pragma unroll
            for (int k = 0; k < NP; ++k) cp_async4(sz + k * TH, P.w32 + off + k * NP2);
            if (!first)
#pragma unroll
                for (int k = 0; k < NP; ++k) cp_async4(sp + k * TH, P.p32 + off + k * NP2);
        }
    };
    const int stride = (int)deal.ncta * G::NG;
    int g = th.grp < G::NG ? (int)deal.first(th.grp, G::GT / 32, G::NG) : ngr;
    fetch(g);
    for (; g < ngr; g += stride) {
        const int e = g * G::GE + th.ge;
        const bool active = th.tid >= 0 && e < E;
        if (threadIdx.x % G::GT == 0) geo_prefetch<NP>(P.geo32, (int64_t)g * G::GE, G::GE, E, 4);
        const size_t off = (size_t)(active ? e : 0) * NP3 + th.tid;
        cp_async_wait_all();
        dfacc dot = {0.f, 0.f};
        auto load = [&](int k) {
            float pn = sz[k * TH];
            if (!first) pn = fmaf(b32, sp[k * TH], pn);
            P.p32[off + k * NP2] = pn;
            return pn;
        };
        auto store = [&](int k, float v, float u) {
            P.w32[off + k * NP2] = v;
            dot2_acc(dot, u, v);
        };
        ax_line32_element<NP>(load, store, P.geo32 + (size_t)(active ? e : 0) * 7 * NP3, h1, h2,
                              c_tabs[NP].l, slab, th.tid, active, [&] { fetch(g + stride); }, sync);
        sum3_add(sum, dot.s, dot.e, 0.f);
    }
}

// D: the FP64 derivative matrix, np x np row-major (host).
static inline int solver_upload_tables(int np, const double *D)
{
    if (np < 2 || np > SEM_NPMAX || !D) return SEM_ERR_ARG;
    SolveTabs T;
    memset(&T, 0, sizeof(T));
    for (int t = 0; t < np * np; ++t) T.l.d[t] = (float)D[t];
    if (np % 2 == 0) ax_bfp_tables(np, D, &T.bfp);
    else if (np <= 11) ax_dfl_tables(np, D, &T.dfl);
    SEM_CUDA(cudaMemcpyToSymbol(c_tabs, &T, sizeof(T), (size_t)np * sizeof(T)));
    return SEM_OK;
}

// Dynamic shared memory of an FP64-accurate line phase: eight reduction words
// an element (the first zeroed at the start of every phase), the slabs, the
// staged columns.
template <int NP, int TH>
constexpr size_t line64_red_bytes()
{
    return 8 * sizeof(unsigned) * GrpCfg<NP, TH>::NE;
}

template <int NP>
constexpr bool solve_bfp()
{
    return BfpCfg<NP>::OK && NP <= 12;
}
template <int NP>
constexpr bool solve_dfl()
{
    return DflCfg<NP>::OK;
}
template <int NP>
constexpr size_t line64_slab_pairs()
{
    return 3 * (size_t)(solve_bfp<NP>() ? BfpCfg<NP>::SLAB : NP * NP * NP);
}
template <int NP, int TH>
constexpr size_t line64_smem_bytes()
{
    return line64_red_bytes<NP, TH>() + sizeof(dfp) * GrpCfg<NP, TH>::NE * line64_slab_pairs<NP>() + stage64_bytes<NP, TH>();
}

// FP64-accurate element phases on the FP32 pipes by whole lines
// (block-floating-point pairs for even N+1 <= 12, float pairs for odd N+1 <=
// 11).  AX0: w = A x;  A: p = z + beta p, w <- A p, <p, w>.
template <int NP, int TH>
__device__ __forceinline__ void phase_a64(const ProbDesc &P, bool ax0, double beta, int first, const Deal &deal,
                                          unsigned char *smem, double &acc)
{
    using G = GrpCfg<NP, TH>;
    constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
    const GrpThread<NP> th;
    const GrpSync<G::GT, TH> sync{th.grp};
    const int slot = th.grp * G::GE + th.ge;
    unsigned *red = reinterpret_cast<unsigned *>(smem) + 8 * slot;
    dfp *slabs = reinterpret_cast<dfp *>(smem + line64_red_bytes<NP, TH>());
    dfp *slab = slabs + (size_t)slot * line64_slab_pairs<NP>();
    double *sz = reinterpret_cast<double *>(slabs + G::NE * line64_slab_pairs<NP>()) + threadIdx.x;
    double *sp = sz + NP * TH;
    double *sn = sp + NP * TH;  // the new p (stage_keep_p)
    const float h1h = (float)P.h1, h2h = (float)P.h2;
    const dfp H1 = {h1h, (float)(P.h1 - (double)h1h)}, H2 = {h2h, (float)(P.h2 - (double)h2h)};
    const int E = (int)P.E, ngr = (E + G::GE - 1) / G::GE;
    const double *zsrc = ax0 ? P.x : P.w;
    const bool add_p = !ax0 && !first;
    auto fetch = [&](int g) {
        const int e = g * G::GE + th.ge;
        if (g < ngr && th.tid >= 0 && e < E) {
            const size_t off = (size_t)e * NP3 + th.tid;
#pragma unroll
            for (int k = 0; k < NP; ++k) cp_async8(sz + k * TH, zsrc + off + k * NP2);
            if (add_p)
#pragma unroll
                for (int k = 0; k < NP; ++k) cp_async8(sp + k * TH, P.p + off + k * NP2);
        }
    };
    if (th.tid == 0 && th.grp < G::NG) *red = 0u;
    if (th.grp < G::NG) sync();
    const int stride = (int)deal.ncta * G::NG;
    int g = th.grp < G::NG ? (int)deal.first(th.grp, G::GT / 32, G::NG) : ngr;
    fetch(g);
    for (; g < ngr; g += stride) {
        const int e = g * G::GE + th.ge;
        const bool active = th.tid >= 0 && e < E;
        if (threadIdx.x % G::GT == 0) geo_prefetch<NP>(P.geodf, (int64_t)g * G::GE, G::GE, E, 8);
        const size_t off = (size_t)(active ? e : 0) * NP3;
        const dfp *geo = P.geodf + (size_t)(active ? e : 0) * 7 * NP3;
        cp_async_wait_all();
        auto load = [&](int q) {
            const int k = (q - th.tid) / NP2;  // a constant after unrolling
            double pn = sz[k * TH];
            if (ax0) return pn;
            if (add_p) pn = fma(beta, sp[k * TH], pn);
            if (stage_keep_p<NP>()) sn[k * TH] = pn;
            P.p[off + q] = pn;
            return pn;
        };
        auto store = [&](int q, double v) {
            P.w[off + q] = v;
            if (!ax0) {
                const int k = (q - th.tid) / NP2;
                acc = fma(stage_keep_p<NP>() ? sn[k * TH] : __ldcg(P.p + off + q), v, acc);
            }
        };
        auto next = [&] { fetch(g + stride); };
        if constexpr (solve_bfp<NP>())
            ax_bfp_element<NP, false>(load, store, geo, H1, H2, c_tabs[NP].bfp, slab, red, th.tid, active,
                                      next, sync);
        else
            ax_dfl_element<NP>(load, store, geo, H1, H2, c_tabs[NP].dfl, slab, red, th.tid, active, next,
                               sync);
    }
}

// FP64-accurate w = A x with the low-register float-pair operator (mixed
// modes: the FP64 residual of each refinement step), one element per 256
// threads of the CTA.
template <int NP, int TH>
__device__ __forceinline__ void phase_ax0_lowreg(const ProbDesc &P, const Deal &deal, unsigned char *smem)
{
    constexpr int NP3 = NP * NP * NP, NG = TH / SEM_SOLVE_THREADS;
    const float h1h = (float)P.h1, h2h = (float)P.h2;
    const dfp H1 = {h1h, (float)(P.h1 - (double)h1h)}, H2 = {h2h, (float)(P.h2 - (double)h2h)};
    const int grp = threadIdx.x / SEM_SOLVE_THREADS;
    const GrpSync<SEM_SOLVE_THREADS, TH> sync{grp};
    smem += grp * lowreg_smem_bytes<NP>();
    for (int64_t e = deal.first(grp, SEM_SOLVE_THREADS / 32, NG); e < P.E; e += deal.ncta * NG) {
        const double *x = P.x + e * NP3;
        double *w = P.w + e * NP3;
        auto load = [&](int q) { return __ldcg(x + q); };
        auto store = [&](int q, double v) { w[q] = v; };
        ax_df_element_lowreg<NP>(load, store, P.geodf + e * 7 * NP3, H1, H2, P.Ddf, smem,
                                 threadIdx.x % SEM_SOLVE_THREADS, SEM_SOLVE_THREADS, sync);
    }
}

// Loads of a phase without staging: the input of node q (z + beta p, kept as
// the new p, in phase A; x in AX0).
__device__ __forceinline__ double a_input(const ProbDesc &P, bool ax0, double beta, int first, size_t q)
{
    if (ax0) return __ldcg(P.x + q);
    double pn = __ldcg(P.w + q);
    if (!first) pn = fma(beta, __ldcg(P.p + q), pn);
    P.p[q] = pn;
    return pn;
}

// FP64-accurate element phases of the largest orders (float pairs, D in shared
// memory), one group of 256/NP^2 elements per CTA.
template <int NP>
__device__ __forceinline__ void elem_item_df(const ProbDesc &P, bool ax0, double beta, int first, int64_t g,
                                             unsigned char *smem, double &acc)
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
    const size_t off = (size_t)(active ? e : 0) * C::NP3;
    const dfp *geo = P.geodf + (active ? e : 0) * 7 * C::NP3;
    const float h1h = (float)P.h1, h2h = (float)P.h2;
    const dfp H1 = {h1h, (float)(P.h1 - (double)h1h)}, H2 = {h2h, (float)(P.h2 - (double)h2h)};
    if (threadIdx.x == 0) geo_prefetch<NP>(P.geodf, g * C::NE, C::NE, P.E, 8);
    ax_df_load_D<NP>(P.Ddf, sD, sDT);
    int *myexp = sexp + (inrange ? grp : 0);
    auto load = [&](int q) { return a_input(P, ax0, beta, first, off + q); };
    auto store = [&](int q, double v) {
        P.w[off + q] = v;
        if (!ax0) acc = fma(__ldcg(P.p + off + q), v, acc);
    };
    ax_df_element<NP>(load, store, geo, H1, H2, sD, sDT, su, svr, svs, myexp, tid, active);
}

// Native FP64 element phases.
template <int NP>
__device__ __forceinline__ void elem_item_native(const ProbDesc &P, bool ax0, double beta, int first,
                                                 int64_t g, unsigned char *smem, double &acc)
{
    using C = AxCfg<NP>;
    double *sm = reinterpret_cast<double *>(smem);
    double *sD = sm, *sDT = sm + NP * NP;
    const int grp = threadIdx.x / C::NP2;
    const int tid = threadIdx.x - grp * C::NP2;
    const bool inrange = grp < C::NE;
    const int64_t e = g * C::NE + grp;
    const bool active = inrange && e < P.E;
    double *su = sm + 2 * NP * NP + (size_t)(inrange ? grp : 0) * 3 * C::NP3;
    double *svr = su + C::NP3, *svs = svr + C::NP3;
    const size_t off = (size_t)(active ? e : 0) * C::NP3;
    const double *geo = P.geo64 + (active ? e : 0) * 7 * C::NP3;
    ax_load_D<NP, double>(P.D64, sD, sDT);
    auto load = [&](int q) { return a_input(P, ax0, beta, first, off + q); };
    auto store = [&](int q, double v, double u) {
        P.w[off + q] = v;
        if (!ax0) acc = fma(u, v, acc);
    };
    ax_element<NP, double>(load, store, geo, P.h1, P.h2, sD, sDT, su, svr, svs, tid, active);
}

// TC inner operator (16-bit tensor-core contractions, FP32 vectors).  tc: 1
// BF16, 2 FP16 (plain rounding); 3 FP16 x2, 4 BF16 x3 (split operands, N+1 <= 8).
template <int NP>
__device__ __forceinline__ void elem_item_tc(const ProbDesc &P, double beta, int first, int64_t g, int tc,
                                             unsigned char *smem, Sum3 &sum)
{
    const float b32 = (float)beta;
    dfacc dot = {0.f, 0.f};
    auto load = [&](int64_t q) {
        float pn = __ldcg(P.w32 + q);
        if (!first) pn = fmaf(b32, __ldcg(P.p32 + q), pn);
        P.p32[q] = pn;
        return pn;
    };
    auto store = [&](int64_t q, float v, float u) {
        P.w32[q] = v;
        dot2_acc(dot, u, v);
    };
    if (tc == 3)
        ax_tc_split_group<NP, true>(load, store, P.geo32, P.D32, (float)P.h1, (float)P.h2, P.E, g, smem);
    else if (tc == 4)
        ax_tc_split_group<NP, false>(load, store, P.geo32, P.D32, (float)P.h1, (float)P.h2, P.E, g, smem);
    else
        ax_tc_group<NP>(load, store, P.geo32, P.D32, (float)P.h1, (float)P.h2, P.E, g, tc == 2, smem);
    sum3_add(sum, dot.s, dot.e, 0.f);
}

// Whether the element phases of order NP in MODE are line phases (A32 always is).
template <int NP, int MODE>
constexpr bool line_mode()
{
    return MODE == MODE_F32 || (MODE == MODE_F64 && (solve_bfp<NP>() || solve_dfl<NP>()));
}

// This CTA's share of an element phase; returns the next problem's rot.
template <int NP, int MODE, int TH>
__device__ __forceinline__ unsigned phase_elem_np(const ProbDesc &P, int ph, double beta, int first,
                                                  const Deal &deal, unsigned char *smem, double &acc, Sum3 &dot)
{
    const bool ax0 = ph == PH_AX0;
    if constexpr (MODE == MODE_F64 && (solve_bfp<NP>() || solve_dfl<NP>())) {
        phase_a64<NP, TH>(P, ax0, beta, first, deal, smem, acc);
    } else if (MODE == MODE_F32 && !ax0) {
        if constexpr (MODE == MODE_F32) phase_a32<NP, TH>(P, beta, first, deal, smem, dot);
    } else if (MODE == MODE_TC && !ax0 && P.tc == 0) {  // each problem of the launch has its own inner path
        if constexpr (MODE == MODE_TC) phase_a32<NP, TH>(P, beta, first, deal, smem, dot);
    } else if ((MODE == MODE_F32 || MODE == MODE_TC) && ax0) {
        if constexpr (MODE == MODE_F32 || MODE == MODE_TC) phase_ax0_lowreg<NP, TH>(P, deal, smem);
        constexpr int NG = TH / SEM_SOLVE_THREADS;
        return deal.after((unsigned)P.E, SEM_SOLVE_THREADS / 32, NG, TH / 32);
    } else {
        // whole CTAs take groups of elements in turn
        const int ne = MODE == MODE_TC ? P.NE32 : P.NE;
        const int64_t items = (P.E + ne - 1) / ne;
        for (int64_t g = deal.first(0, 1, 1); g < items; g += deal.ncta) {
            if constexpr (MODE == MODE_F64) elem_item_df<NP>(P, ax0, beta, first, g, smem, acc);
            if constexpr (MODE == MODE_F64N) elem_item_native<NP>(P, ax0, beta, first, g, smem, acc);
            if constexpr (MODE == MODE_TC) elem_item_tc<NP>(P, beta, first, g, P.tc, smem, dot);
        }
        return deal.after((unsigned)(items % deal.ncta), 1, 1, TH / 32);
    }
    using G = GrpCfg<NP, TH>;
    return deal.after((unsigned)((P.E + G::GE - 1) / G::GE), G::GT / 32, G::NG, TH / 32);
}

// ---------------------------------------------------------------------------
// unique-node and local-node phases
// ---------------------------------------------------------------------------

// Iterations that update x themselves (FP64 modes); later ones gather their
// corrections in y, at the owned nodes alone, and x += y follows once at the end
// (740 iterations at 16^3 elements, N = 7: 31 us a C phase against 37).  A solve
// of few iterations saves that last pass.
constexpr int X_DIRECT = 4;

// Chunk t of a unique phase.  v: FP64 sums; sum: the sums of the FP32 phases
// (converting them to FP64 once a chunk cost more FP64 operations than an FP64
// phase has).
template <int NP, int MODE>
__device__ __forceinline__ void uniq_item(const ProbDesc &P, const PState &S, int ph, unsigned t, double v[3],
                                          Sum3 sum[2])
{
    constexpr int CH = UqCfg<NP>::CH;
    dfacc d[2] = {{0.f, 0.f}, {0.f, 0.f}};  // the chunk's own
    constexpr bool MIXED = MODE == MODE_F32 || MODE == MODE_TC;
    const UqChunk U = uq_chunk<NP>(P.mesh, t);
    if constexpr (!MIXED) {
        if (ph == PH_C || ph == PH_R0) {
            // C: r -= alpha dssum(w), y += alpha p;  R0: r = (b - mean) - dssum(w)
            const bool c = ph == PH_C;
            const double alpha = c ? S.alpha : 1.0, shift = S.bmean;
            double s[CH], r0[CH], mv[CH], po[CH], yo[CH];
#pragma unroll
            for (int i = 0; i < CH; ++i) r0[i] = yo[i] = po[i] = 0.0;
            uq_gather(P.w, U, s, [&] {
                uq_ldv(P.minv + U.f, mv);
                if (c) {
                    uq_ldv(P.r + U.f, r0);
                    uq_ldv(P.p + U.f, po);
                    if (P.y && S.iters > X_DIRECT) uq_ldv(P.y + U.f, yo);
                } else {
                    uq_ldu(P.b + U.f, r0, U.own, P.vec);
                }
            });
            if (!c)
#pragma unroll
                for (int i = 0; i < CH; ++i) r0[i] -= shift;
            // (slots past the owned nodes carry junk; nothing reads them)
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                if (!c && i < U.own) v[2] = fma(r0[i], r0[i], v[2]);
                r0[i] = fma(-alpha, s[i], r0[i]);
                s[i] = mv[i] * r0[i];
                yo[i] = fma(alpha, po[i], yo[i]);
                if (i < U.own) {
                    v[0] = fma(r0[i], r0[i], v[0]);
                    v[1] = fma(r0[i], s[i], v[1]);
                }
            }
            uq_stv(P.r + U.f, r0, CH);
            uq_scatter(P.w, U, s);
            if (c && P.y && S.iters >= X_DIRECT)
                uq_stv(P.y + U.f, yo, CH);
            else if (c)
                uq_update<CH>(P.x, U, P.vec, [&](int i, double xv) { return fma(alpha, po[i], xv); });
            return;
        }
        if (ph == PH_XUPD) {
            double yv[CH];
            uq_ldv(P.y + U.f, yv);
            uq_update<CH>(P.x, U, P.vec, [&](int i, double xv) { return xv + yv[i]; });
            return;
        }
    } else {
        if (ph == PH_C32) {
            const float a = (float)S.alpha;
            float s[CH], r0[CH], mv[CH], po[CH], dv[CH];
            uq_gather(P.w32, U, s, [&] {
                uq_ldv(P.r32 + U.f, r0);
                uq_ldv(P.minv32 + U.f, mv);
                uq_ldv(P.p32 + U.f, po);
                uq_ldv(P.d32 + U.f, dv);
            });
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                r0[i] = r0[i] - a * s[i];
                s[i] = mv[i] * r0[i];
                dv[i] = fmaf(a, po[i], dv[i]);
                if (i < U.own) {
                    dot2_acc(d[0], r0[i], r0[i]);
                    dot2_acc(d[1], r0[i], s[i]);
                }
            }
            uq_stv(P.r32 + U.f, r0, CH);
            uq_stv(P.d32 + U.f, dv, CH);
            uq_scatter(P.w32, U, s);
            sum3_add(sum[0], d[0].s, d[0].e, 0.f);
            sum3_add(sum[1], d[1].s, d[1].e, 0.f);
            return;
        }
        if (ph == PH_R64) {
            double s[CH], bv[CH];
            uq_gather(P.w, U, s, [&] { uq_ldu(P.b + U.f, bv, U.own, P.vec); });
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                bv[i] -= S.bmean;
                s[i] = bv[i] - s[i];
                if (i < U.own) {
                    v[0] = fma(s[i], s[i], v[0]);
                    v[1] = fma(bv[i], bv[i], v[1]);
                }
            }
            uq_stv(P.r + U.f, s, CH);
            return;
        }
        if (ph == PH_INIT32) {
            double r[CH];
            float mv[CH], z[CH], rv[CH], zero[CH];
            uq_ldv(P.r + U.f, r);
            uq_ldv(P.minv32 + U.f, mv);
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                rv[i] = (float)(r[i] / S.scale);
                z[i] = mv[i] * rv[i];
                zero[i] = 0.f;
                if (i < U.own) {
                    dot2_acc(d[0], rv[i], rv[i]);
                    dot2_acc(d[1], rv[i], z[i]);
                }
            }
            uq_stv(P.r32 + U.f, rv, CH);
            uq_stv(P.d32 + U.f, zero, CH);
            uq_scatter(P.w32, U, z);
            sum3_add(sum[0], d[0].s, d[0].e, 0.f);
            sum3_add(sum[1], d[1].s, d[1].e, 0.f);
            return;
        }
        if (ph == PH_UPD) {
            // the FP64 p vector is unused by refinement: it keeps x until the
            // next residual accepts the step
            float dv[CH];
            uq_ldv(P.d32 + U.f, dv);
            uq_each<CH>(U, [&](unsigned q, int i) {
                const double xv = __ldcg(P.x + q);
                P.p[q] = xv;
                P.x[q] = fma(S.scale, (double)dv[i], xv);
            });
            return;
        }
    }
    if (ph == PH_JACGS) {
        if (P.singular)
#pragma unroll
            for (int i = 0; i < CH; ++i)
                if (i < U.own) v[0] += __ldcg(P.b + U.f + i);
        if (S.jac || P.jac_shared) return;  // only the sum of b
        double s[CH];
        uq_gather(P.minv, U, s, [] {});
#pragma unroll
        for (int i = 0; i < CH; ++i) s[i] = 1.0 / s[i];
        uq_scatter(P.minv, U, s);
        if (P.minv32) {
            float f[CH];
#pragma unroll
            for (int i = 0; i < CH; ++i) f[i] = (float)s[i];
            uq_scatter(P.minv32, U, f);
        }
    }
}

__device__ __forceinline__ void local_item(const ProbDesc &P, const PState &S, int ph, unsigned q, double v[3])
{
    const int n = P.n, n3 = (int)P.dn3.d;
    const unsigned e = fd_div(q, P.dn3);
    const int l = (int)(q - e * n3);
    switch (ph) {
        case PH_JAC: {
            const int i = l % n, j = (l / n) % n, k = l / (n * n);
            const double *g = P.geo64 + (size_t)e * 7 * n3;
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
        case PH_XREST:
            P.x[q] = __ldcg(P.p + q);
            break;
        case PH_FINAL:
            v[0] = fma(P.geo64[((size_t)e * 7 + 6) * n3 + l], __ldcg(P.x + q), v[0]);
            break;
        case PH_SHIFT:
            P.x[q] = __ldcg(P.x + q) - S.shift;
            break;
        default: break;
    }
}

// ---------------------------------------------------------------------------
// per-problem state machine (run by one thread of every CTA between steps)
// ---------------------------------------------------------------------------

// Whether sqrt(rr) <= target; the square root is only taken near the target.
__device__ __forceinline__ bool norm_met(double rr, double target)
{
    const double t2 = target * target;
    if (t2 > 1e-290 && rr > t2 * (1.0 + 1e-12)) return false;
    return sqrt(rr) <= target;
}

template <int MAXP>
__device__ void advance(const SolveParams<MAXP> &prm, const ProbDesc &P, PState &S, const double *red)
{
    const int ph = S.phase;
    const int tail = P.singular ? PH_FINAL : PH_DONE;
    auto finish = [&](int status) {
        S.status = status;
        S.phase = tail;
    };
    // after C phases past the first X_DIRECT the correction y is not yet in x
    auto finish_y = [&](int status) {
        S.status = status;
        S.phase = (P.y && S.iters > X_DIRECT) ? PH_XUPD : tail;
    };
    switch (ph) {
        case PH_JAC: S.phase = PH_JACGS; break;
        case PH_JACGS:
            S.bmean = P.singular ? red[0] / (double)P.nG : 0.0;
            S.phase = PH_AX0;
            break;
        case PH_AX0: S.phase = prm.mixed ? PH_R64 : PH_R0; break;
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
            if (!(pw > 0.0) || !isfinite(pw)) {
                if (S.iters > 0) S.rnorm = sqrt(S.rnorm);  // (phase C keeps its square)
                finish_y(SEM_ERR_BREAKDOWN);
                break;
            }
            S.alpha = S.rz / pw;
            S.phase = PH_C;
        } break;
        case PH_C: {
            S.iters += 1;
            const double rr = red[0];
            const bool met = norm_met(rr, S.target);
            if (!isfinite(rr) || met || S.iters >= prm.maxit) {
                S.rnorm = sqrt(rr);
                finish_y(!isfinite(rr) ? SEM_ERR_BREAKDOWN : met ? SEM_OK : SEM_ERR_NOT_CONVERGED);
                break;
            }
            S.rnorm = rr;  // squared until the solve ends
            S.beta = red[1] / S.rz;
            S.rz = red[1];
            S.first = 0;
            S.phase = PH_A;
        } break;
        case PH_R64: {
            const double rn = sqrt(red[0]);
            if (S.outer == 0) {
                S.bnorm = sqrt(red[1]);
                S.target = prm.abs_tol ? prm.tol : prm.tol * S.bnorm;
            }
            if (rn <= S.target) { S.rnorm = rn; finish(SEM_OK); break; }
            // a step that did not lower the FP64 residual (or made it non-finite)
            // is undone: x returns to the iterate before it
            if (S.outer > 0 && !(rn <= S.prev_rnorm)) {
                S.rnorm = S.prev_rnorm;
                S.status = SEM_ERR_NOT_CONVERGED;
                S.phase = PH_XREST;
                break;
            }
            S.rnorm = rn;
            if (!isfinite(rn) || !isfinite(S.bnorm)) { finish(SEM_ERR_BREAKDOWN); break; }
            if (S.outer >= prm.max_outer || S.iters >= prm.maxit) { finish(SEM_ERR_NOT_CONVERGED); break; }
            if (S.outer > 0 && rn > 0.5 * S.prev_rnorm) { finish(SEM_ERR_NOT_CONVERGED); break; }
            S.prev_rnorm = rn;
            S.scale = rn;
            S.phase = PH_INIT32;
        } break;
        case PH_INIT32: {
            // the inner solve needs to reduce its residual only as far as the
            // outer target requires (with a factor 2 margin), never further
            // than inner_tol
            double rel = 0.5 * S.target / S.rnorm;
            if (rel < prm.inner_tol) rel = prm.inner_tol;
            if (rel > 0.5) rel = 0.5;
            S.inner_target = rel * sqrt(red[0]);
            S.rz = red[1];
            S.first = 1;
            S.beta = 0.0;
            S.inner_iters = 0;
            S.phase = (red[0] > 0.0) ? PH_A32 : PH_UPD;
        } break;
        case PH_A32: {
            const double pw = red[0];
            if (!(pw > 0.0) || !isfinite(pw)) { S.phase = PH_UPD; break; }
            S.alpha = S.rz / pw;
            S.phase = PH_C32;
        } break;
        case PH_C32: {
            S.iters += 1;
            S.inner_iters += 1;
            if (!isfinite(red[0]) || norm_met(red[0], S.inner_target) || S.iters >= prm.maxit) {
                S.phase = PH_UPD;
                break;
            }
            S.beta = red[1] / S.rz;
            S.rz = red[1];
            S.first = 0;
            S.phase = PH_A32;
        } break;
        case PH_UPD: S.outer += 1; S.phase = PH_AX0; break;
        case PH_FINAL: S.shift = red[0] / P.volume; S.phase = PH_SHIFT; break;
        case PH_SHIFT: S.phase = PH_DONE; break;
        case PH_XUPD: case PH_XREST: S.phase = tail; break;
        default: S.phase = PH_DONE; break;
    }
}

// ---------------------------------------------------------------------------
// the persistent kernel
// ---------------------------------------------------------------------------

enum PhaseKind { KIND_ELEM, KIND_UNIQ, KIND_LOCAL };

__host__ __device__ __forceinline__ int phase_kind(int ph)
{
    switch (ph) {
        case PH_AX0: case PH_A: case PH_A32: return KIND_ELEM;
        case PH_JAC: case PH_XREST: case PH_FINAL: case PH_SHIFT: return KIND_LOCAL;
        default: return KIND_UNIQ;
    }
}

constexpr size_t sem_max_sz(size_t a, size_t b) { return a > b ? a : b; }

// Dynamic shared memory of the element phases of one order and mode on TH threads.
template <int NP, int MODE, int TH>
constexpr size_t solve_smem_np()
{
    return MODE == MODE_F64N ? ax_smem_bytes<NP, double>()
           : MODE == MODE_F64 ? (line_mode<NP, MODE>() ? line64_smem_bytes<NP, TH>() : ax_df_smem_bytes<NP>())
           : MODE == MODE_F32 ? sem_max_sz(elem32_smem_bytes<NP, TH>(), TH / SEM_SOLVE_THREADS * lowreg_smem_bytes<NP>())
                              : sem_max_sz(sem_max_sz(ax_tc_smem_bytes<NP>(), ax_tc_split_smem_bytes<NP>()),
                                           sem_max_sz(lowreg_smem_bytes<NP>(), elem32_smem_bytes<NP, TH>()));
}

template <int MODE, int TH, int... NPs>
struct SmemMax;
template <int MODE, int TH>
struct SmemMax<MODE, TH> {
    static constexpr size_t v = 0;
};
template <int MODE, int TH, int NP0, int... NPs>
struct SmemMax<MODE, TH, NP0, NPs...> {
    static constexpr size_t v = sem_max_sz(solve_smem_np<NP0, MODE, TH>(), SmemMax<MODE, TH, NPs...>::v);
};

// Static shared memory of the kernel (states, sums, reduction words).
template <int MAXP, int TH, bool FLOATS>
constexpr size_t solve_static_smem()
{
    return MAXP * (sizeof(PState) + 3 * sizeof(double)) + 64 + TH / 8 +
           (FLOATS && MAXP * (TH / 32) > TH ? MAXP * 3 * (TH / 32) : 3 * TH) * sizeof(double);
}

// Threads of a CTA: one CTA that fills its multiprocessor for the line phases
// (512 threads of 128 registers in FP64, 768 of 80 in FP32) where the shared
// memory allows it; 256 (two resident) for the others, whose element groups
// are whole CTAs.
template <int MAXP, int MODE, int... NPs>
constexpr int solve_threads()
{
    constexpr int big = MODE == MODE_F32 ? 768 : 512;
    return (line_mode<NPs, MODE>() && ...) &&
                   SmemMax<MODE, big, NPs...>::v + solve_static_smem<MAXP, big, MODE == MODE_F32>() <= 227 * 1024
               ? big
               : SEM_SOLVE_THREADS;
}

template <int MODE, int TH, int... NPs>
struct PhaseDispatch;

template <int MODE, int TH, int NP0, int... NPs>
struct PhaseDispatch<MODE, TH, NP0, NPs...> {
    // This CTA's share of P's phase; returns the next problem's rot.
    __device__ __forceinline__ static unsigned run(const ProbDesc &P, const PState &S, int kind, const Deal &deal,
                                                   unsigned char *smem, double v[3], Sum3 d[2])
    {
        if constexpr (sizeof...(NPs) > 0)
            if (P.n != NP0) return PhaseDispatch<MODE, TH, NPs...>::run(P, S, kind, deal, smem, v, d);
        if (kind == KIND_ELEM)
            return phase_elem_np<NP0, MODE, TH>(P, S.phase, S.beta, S.first, deal, smem, v[0], d[0]);
        // unique phases: warps take 32 chunks in turn
        constexpr unsigned NW = TH / 32;
        const unsigned units = uq_units<NP0>(P.mesh), portions = (units + 31) / 32;
        for (unsigned g = deal.first(threadIdx.x / 32, 1, NW); g < portions; g += deal.ncta * NW) {
            const unsigned t = g * 32 + (threadIdx.x & 31);
            if (t < units) uniq_item<NP0, MODE>(P, S, S.phase, t, v, d);
        }
        return deal.after(portions, 1, NW, NW);
    }
    // Portions (groups of elements or four warps of chunks, the larger) of P.
    static unsigned portions(const ProbDesc &P)
    {
        if constexpr (sizeof...(NPs) > 0)
            if (P.n != NP0) return PhaseDispatch<MODE, TH, NPs...>::portions(P);
        const unsigned ge = line_mode<NP0, MODE>() ? GrpCfg<NP0, TH>::GE : (unsigned)P.NE;
        const unsigned a = ((unsigned)P.E + ge - 1) / ge, b = (uq_units<NP0>(P.mesh) + 127) / 128;
        return a > b ? a : b;
    }
};

template <int MAXP, int MODE, int TH, int... NPs>
__global__ void __launch_bounds__(TH, TH > SEM_SOLVE_THREADS ? 1 : 2)
    k_solve(const __grid_constant__ SolveParams<MAXP> prm)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ PState s_st[MAXP];
    __shared__ double s_sum[MAXP][3];
    // Sums of a problem's phase over the CTA: [value][thread], or, in an FP32 launch
    // (of several problems, or of more than 256 threads), [problem][value][warp].
    constexpr bool FLOATS = MODE == MODE_F32 || MODE == MODE_TC;
    constexpr int NW = TH / 32;
    constexpr int RED = FLOATS && MAXP * NW > TH ? MAXP * 3 * NW : 3 * TH;
    __shared__ double s_red[RED];
    __shared__ int s_fail;
    // Kept in shared memory so that no register holds them through an element
    // phase, which needs every register that it can get: the step, and each
    // warp's copy of the next problem's start.
    __shared__ unsigned s_step, s_rot[NW];
    const int np = prm.nprob;
    SyncState *sync = prm.sync;
    const unsigned grid = gridDim.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int p = threadIdx.x; p < np; p += TH) {
        PState S;
        memset(&S, 0, sizeof(S));
        const ProbDesc &P = prm.prob[p];
        S.jac = jac_kept(P);
        // (the sum of b that JACGS makes is only needed to remove its mean)
        S.phase = !S.jac ? PH_JAC : P.singular ? PH_JACGS : PH_AX0;
        s_st[p] = S;
        // (CTAs that read the word after this find it incomplete as well)
        if (blockIdx.x == 0 && !S.jac && !P.jac_shared && P.jac_dev) *P.jac_dev = 0u;
    }
    if (threadIdx.x == 0) s_step = 0;
    __syncthreads();
    auto partials = [&] { return prm.partials + (size_t)(s_step & 1) * MAXP * 3 * grid; };

    for (;;) {
        // ---- this CTA's share of every problem's phase; its sums are published
        bool all_done = true;
        int layout = -1;  // how the last element phase laid the shared memory out
        if (MAXP > 1 && lane == 0) s_rot[warp] = 0;
        for (int o = 0; o < (MAXP == 1 ? 1 : np); ++o) {
            const int p = MAXP == 1 ? 0 : prm.order[o];
            const PState &S = s_st[p];
            if (S.phase == PH_DONE) continue;
            all_done = false;
            const ProbDesc &P = prm.prob[p];
            const int kind = phase_kind(S.phase);
            if (MAXP > 1 && kind == KIND_ELEM) {
                const int want = P.n * 16 + P.tc * 2 + (S.phase == PH_AX0);
                if (layout >= 0 && layout != want) __syncthreads();
                layout = want;
            }
            double v[3] = {0.0, 0.0, 0.0};
            Sum3 d[2] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
            if (kind != KIND_LOCAL) {
                if (MAXP > 1) __syncwarp();
                const Deal deal = {blockIdx.x, grid, MAXP == 1 ? 0u : s_rot[warp]};
                const unsigned rot = PhaseDispatch<MODE, TH, NPs...>::run(P, S, kind, deal, smem, v, d);
                if (MAXP > 1) {
                    __syncwarp();
                    if (lane == 0) s_rot[warp] = rot;
                }
            } else if (S.phase != PH_JAC || !P.jac_shared) {
                for (unsigned q = blockIdx.x * TH + threadIdx.x; q < (unsigned)P.nL; q += grid * TH)
                    local_item(P, S, S.phase, q, v);
            }
            const int nv = phase_nvals(s_st[p].phase);
            if (nv == 0) continue;
            if (FLOATS && (np > 1 || TH > SEM_SOLVE_THREADS)) {
                // no barrier between the problems of an FP32 launch: a warp sums
                // its lanes' values and leaves the sums for the end of the step
                if (phase_floats(s_st[p].phase)) {
                    const double t = warp_sum3(d, lane);
                    if (lane % 16 == 0 && (int)lane / 16 < nv) s_red[(p * 3 + lane / 16) * NW + warp] = t;
                } else {
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        if (k < nv) {
                            const double t = warp_sum(v[k]);
                            if (lane == 0) s_red[(p * 3 + k) * NW + warp] = t;
                        }
                }
                continue;
            }
            // one warp per value sums the CTA's TH in a fixed order
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (k < nv)
                    s_red[k * TH + threadIdx.x] =
                        FLOATS && k < 2 && phase_floats(s_st[p].phase) ? sum3_value(d[k]) : v[k];
            __syncthreads();
            if ((int)warp < nv) {
                double t[NW];
#pragma unroll
                for (int j = 0; j < NW; ++j) t[j] = s_red[warp * TH + lane + 32 * j];
                const double s = warp_sum(tree_sum(t));
                if (lane == 0) partials()[(size_t)(p * 3 + warp) * grid + blockIdx.x] = s;
            }
            if (np > 1) __syncthreads();  // (s_red is written again)
        }
        if (all_done) break;

        if (FLOATS && (np > 1 || TH > SEM_SOLVE_THREADS)) {
            __syncthreads();
            for (int pk = warp; pk < np * 3; pk += NW) {
                const int p = pk / 3, k = pk - 3 * p;
                if (k < phase_nvals(s_st[p].phase)) {
                    const double t = warp_sum((int)lane < NW ? s_red[pk * NW + lane] : 0.0);
                    if (lane == 0) partials()[(size_t)pk * grid + blockIdx.x] = t;
                }
            }
        }

        // ---- grid barrier: the count reaches (steps so far + 1) * grid
        __syncthreads();
        if (threadIdx.x == 0) {
            s_fail = 0;
            red_release_add_u32(&sync->count, 1u);
            const unsigned goal = (s_step + 1u) * grid;
            const unsigned long long t0 = sem_globaltimer();
            for (unsigned spin = 0; (int)(ld_acquire_u32(&sync->count) - goal) < 0; ++spin) {
                if ((spin & 15u) != 0u) continue;
                if (((volatile int *)&sync->err)[0]) {
                    s_fail = 1;
                    break;
                }
                if ((long long)(sem_globaltimer() - t0) > prm.timeout_ns) {
                    atomicExch(&sync->err, SEM_ERR_TIMEOUT);
                    s_fail = 1;
                    break;
                }
            }
        }
        __syncthreads();
        if (s_fail) break;

        // ---- every CTA sums the partials in the same fixed order, one warp a value
        // (eight loads in flight a lane: one at a time their latencies added up to
        // 3 us a phase)
        for (int pk = warp; pk < np * 3; pk += NW) {
            const int p = pk / 3, k = pk - 3 * p;
            if (k < phase_nvals(s_st[p].phase)) {
                const double *src = partials() + (size_t)pk * grid;
                double s = 0.0;
                for (unsigned b0 = 0; b0 < grid; b0 += 256) {
                    double t[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const unsigned b = b0 + 32 * j + lane;
                        t[j] = b < grid ? __ldcg(src + b) : 0.0;
                    }
                    s += tree_sum(t);
                }
                s = warp_sum(s);
                if (lane == 0) s_sum[p][k] = s;
            }
        }
        __syncthreads();
        for (int p = threadIdx.x; p < np; p += TH)
            if (s_st[p].phase != PH_DONE) {
                const ProbDesc &P = prm.prob[p];
                // (every CTA has read the word before its first barrier)
                if (blockIdx.x == 0 && s_st[p].phase == PH_JACGS && !s_st[p].jac && !P.jac_shared && P.jac_dev)
                    *P.jac_dev = jac_bits(P);
                advance<MAXP>(prm, P, s_st[p], s_sum[p]);
            }
        if (threadIdx.x == 0) s_step += 1;
        __syncthreads();
    }
    // the final states, once (after a time-out: the states at the last whole step)
    __syncthreads();
    if (blockIdx.x == 0)
        for (int p = threadIdx.x; p < np; p += TH) {
            // (a solve that timed out between two C phases still keeps the norm's square)
            if ((s_st[p].phase == PH_A || s_st[p].phase == PH_C) && s_st[p].iters > 0)
                s_st[p].rnorm = sqrt(s_st[p].rnorm);
            prm.st[p] = s_st[p];
        }
}

// Host launcher (cooperative, grid sized for co-residency and no larger than
// the element and unique phases can use).
template <int MAXP, int MODE, int... NPs>
int launch_solve(const SolveParams<MAXP> &prm, int num_sms, cudaStream_t s)
{
    constexpr int TH = solve_threads<MAXP, MODE, NPs...>();
    auto kern = k_solve<MAXP, MODE, TH, NPs...>;
    const size_t smem = SmemMax<MODE, TH, NPs...>::v;
    static std::atomic<unsigned> attr{0};
    SEM_CUDA(sem_smem_attr(kern, smem, attr));
    int per_sm = 0;
    SEM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TH, smem));
    if (per_sm < 1) return SEM_ERR_ARG;
    long long most = 0;
    for (int p = 0; p < prm.nprob; ++p) most += PhaseDispatch<MODE, TH, NPs...>::portions(prm.prob[p]);
    long long grid = (long long)per_sm * num_sms;
    const long long fit = prm.partials_cap / (2 * MAXP * 3);
    if (grid > most) grid = most;
    if (grid > fit) grid = fit;
    if (grid < 1) grid = 1;
    void *args[] = {(void *)&prm};
    SEM_CUDA(cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)grid), dim3(TH), args, smem, s));
    return SEM_OK;
}

// Maximum grid the solver may use (sizes the partials buffer).
#define SEM_SOLVE_MAX_GRID_PER_SM 8

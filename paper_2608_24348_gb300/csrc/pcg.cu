// pcg.cu -- host side of the persistent PCG / iterative-refinement solver.
#include <stddef.h>
#include <string.h>

#include <vector>

#include "solver.cuh"

GsDesc sem_gs_desc(const sem_ctx *c);  // ops.cu
int sem_alloc_ws(sem_ctx *c, int slot);  // setup.cu

// Per-order kernels (solve_npXX.cu), up to 8 problems of one order.
#define SEM_DECL_NP(NPV) int sem_solve_launch_np##NPV(const SolveParams<8> &, int, int, cudaStream_t);
SEM_DECL_NP(2) SEM_DECL_NP(3) SEM_DECL_NP(4) SEM_DECL_NP(5) SEM_DECL_NP(6) SEM_DECL_NP(7)
SEM_DECL_NP(8) SEM_DECL_NP(9) SEM_DECL_NP(10) SEM_DECL_NP(11) SEM_DECL_NP(12) SEM_DECL_NP(13)
SEM_DECL_NP(14) SEM_DECL_NP(15) SEM_DECL_NP(16)
#undef SEM_DECL_NP
// Mixed-order kernel for N in {5, 7, 9} (solve_multi.cu), up to 64 problems.
int sem_solve_launch_multi(const SolveParams<SEM_MAXP> &, int, int, cudaStream_t);

#define SEM_DECL_TAB(NPV) int sem_solve_tables_np##NPV(const double *);
SEM_DECL_TAB(2) SEM_DECL_TAB(3) SEM_DECL_TAB(4) SEM_DECL_TAB(5) SEM_DECL_TAB(6) SEM_DECL_TAB(7)
SEM_DECL_TAB(8) SEM_DECL_TAB(9) SEM_DECL_TAB(10) SEM_DECL_TAB(11) SEM_DECL_TAB(12) SEM_DECL_TAB(13)
SEM_DECL_TAB(14) SEM_DECL_TAB(15) SEM_DECL_TAB(16)
#undef SEM_DECL_TAB
int sem_solve_tables_multi(int np, const double *D);

// The ordered solver of Taylor-Green steps (solver_ordered.cuh), N + 1 <= 10.
#define SEM_DECL_ORD(U)                                                        \
    int sem_solve_ordered_##U(const SolveParams<8> &, int, int, cudaStream_t); \
    int sem_solve_ordered_tables_##U(int, const double *);
SEM_DECL_ORD(a) SEM_DECL_ORD(b) SEM_DECL_ORD(c)
#undef SEM_DECL_ORD
typedef int (*ordered_fn)(const SolveParams<8> &, int, int, cudaStream_t);
typedef int (*ordered_tab_fn)(int, const double *);
static const ordered_fn k_ordered[3] = {sem_solve_ordered_c, sem_solve_ordered_a, sem_solve_ordered_b};  // n % 3
static const ordered_tab_fn k_ordered_tab[3] = {sem_solve_ordered_tables_c, sem_solve_ordered_tables_a,
                                                sem_solve_ordered_tables_b};

// The ordered solver's constant memory (even N + 1 <= 10), as sem_solve_upload_tables;
// at stepper setup, since only its steps use it.
int sem_solve_upload_ordered(const sem_ctx *c)
{
    return c->n % 2 == 0 && c->n <= 10 ? k_ordered_tab[c->n % 3](c->n, c->hD) : SEM_OK;
}

// Fills the constant memory of the solver kernels that serve the context's
// order (the per-order unit and, for N + 1 in {6, 8, 10}, the mixed-order
// unit) with the tables made from its derivative matrix, on the current device.
int sem_solve_upload_tables(const sem_ctx *c)
{
    typedef int (*tab_fn)(const double *);
    static const tab_fn f[17] = {nullptr, nullptr, sem_solve_tables_np2, sem_solve_tables_np3,
                                 sem_solve_tables_np4, sem_solve_tables_np5, sem_solve_tables_np6,
                                 sem_solve_tables_np7, sem_solve_tables_np8, sem_solve_tables_np9,
                                 sem_solve_tables_np10, sem_solve_tables_np11, sem_solve_tables_np12,
                                 sem_solve_tables_np13, sem_solve_tables_np14, sem_solve_tables_np15,
                                 sem_solve_tables_np16};
    if (c->n < 2 || c->n > 16) return SEM_ERR_ARG;
    int rc = f[c->n](c->hD);
    if (rc == SEM_OK && (c->n == 6 || c->n == 8 || c->n == 10)) rc = sem_solve_tables_multi(c->n, c->hD);
    return rc;
}

typedef int (*launch8_fn)(const SolveParams<8> &, int, int, cudaStream_t);
static const launch8_fn k_launch8[17] = {
    nullptr, nullptr, sem_solve_launch_np2, sem_solve_launch_np3, sem_solve_launch_np4,
    sem_solve_launch_np5, sem_solve_launch_np6, sem_solve_launch_np7, sem_solve_launch_np8,
    sem_solve_launch_np9, sem_solve_launch_np10, sem_solve_launch_np11, sem_solve_launch_np12,
    sem_solve_launch_np13, sem_solve_launch_np14, sem_solve_launch_np15, sem_solve_launch_np16};

struct SolveStateHost {
    SyncState sync;
    PState st[SEM_MAXP];
};

int sem_solve_state_bytes() { return (int)sizeof(SolveStateHost); }

size_t sem_partials_bytes(int num_sms)
{
    return sizeof(double) * (size_t)num_sms * SEM_SOLVE_MAX_GRID_PER_SM * SEM_MAXP * 3;
}

extern "C" void sem_solve_opts_default(sem_solve_opts *o)
{
    if (!o) return;
    o->tol = 1e-10;
    o->abs_tol = 0;
    o->maxit = 20000;
    o->inner = SEM_F64;
    o->inner_tol = 1e-4;
    o->max_outer = 50;
    o->wait_timeout_s = 0.0;
}

static int ne_for(int n) { return (256 / (n * n)) > 0 ? 256 / (n * n) : 1; }

// Element groups of the TC path use one warp per element.
static int TcNE(int n) { return n <= 8 ? 8 : 4; }

// Inner path of SEM_F32_TUNED per order (sem_tune_inner): 0 FP32 CUDA cores,
// 1 split FP16 tensor cores.
static int g_inner_path[SEM_NMAX + 1];

// Tensor-core path of a problem of order N (n = N + 1) for an inner dtype: 0
// = none (FP32 CUDA cores or no inner solve), else ProbDesc::tc.
static int inner_tc_of(sem_dtype inner, int n)
{
    switch (inner) {
        case SEM_BF16_TC: return 1;
        case SEM_F16_TC: return 2;
        case SEM_F16X2_TC: return 3;
        case SEM_BF16X3_TC: return 4;
        case SEM_F32_TUNED: return (n - 1 <= SEM_NMAX && g_inner_path[n - 1] == 1 && n <= 8) ? 3 : 0;
        default: return 0;
    }
}

// Whether a solve with these options takes the context's order (the tensor-core
// inner operators end at N + 1 = 10, their split-operand forms at 8).
bool sem_pcg_accepts(const sem_ctx *c, const sem_solve_opts &o)
{
    const bool split = o.inner == SEM_F16X2_TC || o.inner == SEM_BF16X3_TC;
    const bool tc = split || o.inner == SEM_BF16_TC || o.inner == SEM_F16_TC;
    return !tc || c->n <= (split ? 8 : 10);
}

// Problem p on the same context and coefficients as an earlier problem q of the
// launch takes q's Jacobi inverse instead of making (and keeping) its own.
static bool share_jacobi(const ProbDesc &q, ProbDesc &d, const sem_ctx *cq, const sem_ctx *c)
{
    if (cq != c || q.h1 != d.h1 || q.h2 != d.h2) return false;
    d.minv = q.minv;
    d.minv32 = q.minv32;
    d.jac_cached = q.jac_cached;
    d.jac_dev = q.jac_dev;
    d.jac_shared = 1;
    return true;
}

// Fills d for a solve on workspace ws; the Jacobi inverse is recomputed unless
// ws still holds the one of (h1, h2) (and its FP32 copy when mixed), and ws
// records what the launch leaves in minv / minv32 (the launch that finds them
// incomplete, because the one that was to make them timed out, makes them).  first .. first + nfirst:
// the launch's earlier problems and their contexts, one of which may share its
// Jacobi inverse.
static void fill_desc(const sem_ctx *c, sem_ws &ws, const double *b, double *x, double h1,
                      double h2, bool mixed, int tc, ProbDesc &d, const ProbDesc *first = nullptr,
                      sem_ctx *const *fctx = nullptr, int nfirst = 0)
{
    memset(&d, 0, sizeof(d));
    d.n = c->n;
    d.NE = ne_for(c->n);
    d.tc = tc;
    d.NE32 = tc ? TcNE(c->n) : d.NE;
    d.singular = (h2 == 0.0);
    d.E = c->E;
    d.nL = c->nL;
    d.nG = c->nG;
    d.mesh = uq_mesh(sem_gs_desc(c));
    d.dn3 = fast_div((unsigned)(d.n * d.n * d.n));
    d.volume = c->volume;
    d.h1 = h1;
    d.h2 = h2;
    d.geo64 = c->geo64;
    d.geo32 = c->geo32;
    d.geodf = (const dfp *)c->geodf;
    d.D64 = c->tab64 + 2 * c->n;
    d.D32 = c->tab32 + 2 * c->n;
    d.Ddf = (const dfp *)c->tabdf;
    d.b = b;
    d.x = x;
    d.r = ws.r;
    d.p = ws.p;
    d.w = ws.w;
    d.minv = ws.minv;
    d.y = ws.b;
    d.vec = ((uintptr_t)b | (uintptr_t)x) % 32 == 0;
    if (mixed) {
        d.r32 = ws.r32;
        d.p32 = ws.p32;
        d.w32 = ws.w32;
        d.d32 = ws.d32;
        d.minv32 = ws.minv32;
    }
    d.jac_dev = c->jac_dev + (&ws - c->ws);
    for (int q = 0; q < nfirst; ++q)
        if (share_jacobi(first[q], d, fctx[q], c)) return;
    d.jac_cached = ws.jac_ok && ws.jac_h1 == h1 && ws.jac_h2 == h2 && (!mixed || ws.jac32_ok);
    if (!d.jac_cached) {
        ws.jac_ok = 1;
        ws.jac_h1 = h1;
        ws.jac_h2 = h2;
        ws.jac32_ok = mixed;
    }
}

template <int MAXP>
static void fill_common(SolveParams<MAXP> &p, sem_ctx *owner, const sem_solve_opts &o, int nprob)
{
    p.nprob = nprob;
    p.mixed = o.inner != SEM_F64 && o.inner != SEM_F64_NATIVE;
    p.abs_tol = o.abs_tol;
    p.maxit = o.maxit;
    p.max_outer = o.max_outer;
    p.tol = o.tol;
    p.inner_tol = o.inner_tol;
    const double tmo = o.wait_timeout_s > 0 ? o.wait_timeout_s : 10.0;
    p.timeout_ns = (long long)(tmo * 1e9);
    SolveStateHost *S = (SolveStateHost *)owner->solve_dev;
    p.sync = &S->sync;
    p.st = S->st;
    p.partials = (double *)owner->partials;
    p.partials_cap = (long long)(sem_partials_bytes(owner->num_sms) / sizeof(double));
}

static int validate_opts(const sem_solve_opts &o)
{
    if (!(o.tol >= 0) || o.maxit < 0 || o.max_outer < 0) return SEM_ERR_ARG;
    if (o.inner < SEM_F64 || o.inner > SEM_F32_TUNED) return SEM_ERR_ARG;
    const bool mixed = o.inner != SEM_F64 && o.inner != SEM_F64_NATIVE;
    if (mixed && !(o.inner_tol > 0 && o.inner_tol < 1)) return SEM_ERR_ARG;
    return SEM_OK;
}

// Plain FP64 PCG to a relative tolerance below 1e-11 runs on the native
// FP64 operator: the float-pair and block-floating-point operators of
// SEM_F64 carry a relative error of a few 1e-13 per application, the size
// of such a residual, and on a singular (periodic Poisson) problem their
// error on the constant mode can end the solve with <p,Ap> <= 0.
static bool tight_f64(const sem_solve_opts &o) { return o.inner == SEM_F64 && !o.abs_tol && o.tol < 1e-11; }

// Enqueue one launch for problems `idx` (all on owner's state buffers).
// ordered: with the solver of solver_ordered.cuh.
static int enqueue(sem_ctx *owner, const sem_solve_opts &o, const ProbDesc *d, int np,
                   cudaStream_t s, bool ordered = false)
{
    SEM_CUDA(cudaMemsetAsync(owner->solve_dev, 0, sizeof(SolveStateHost), s));
    bool any_tc = false;
    for (int p = 0; p < np; ++p) any_tc |= (d[p].tc != 0);
    const bool tight = tight_f64(o);
    const int mode = tight ? MODE_F64N
                     : o.inner == SEM_F64 ? MODE_F64
                     : o.inner == SEM_F64_NATIVE ? MODE_F64N
                     : (o.inner == SEM_F32 || (o.inner == SEM_F32_TUNED && !any_tc)) ? MODE_F32 : MODE_TC;
    bool same = true;
    for (int p = 1; p < np; ++p) same &= (d[p].n == d[0].n);
    int rc;
    if (same && np <= 8) {
        SolveParams<8> prm;
        memset(&prm, 0, sizeof(prm));
        fill_common(prm, owner, o, np);
        for (int p = 0; p < np; ++p) {
            prm.prob[p] = d[p];
            prm.order[p] = (unsigned char)p;
        }
        rc = ordered ? k_ordered[d[0].n % 3](prm, d[0].n, owner->num_sms, s)
                     : k_launch8[d[0].n](prm, mode, owner->num_sms, s);
    } else {
        SolveParams<SEM_MAXP> *prm = new SolveParams<SEM_MAXP>();
        fill_common(*prm, owner, o, np);
        for (int p = 0; p < np; ++p) prm->prob[p] = d[p];
        for (int n = 2, o = 0; n <= SEM_NPMAX; ++n)
            for (int p = 0; p < np; ++p)
                if (d[p].n == n) prm->order[o++] = (unsigned char)p;
        rc = sem_solve_launch_multi(*prm, mode, owner->num_sms, s);
        delete prm;
    }
    if (rc) return rc;
    SEM_CUDA(cudaMemcpyAsync(owner->solve_host, owner->solve_dev, sizeof(SolveStateHost),
                             cudaMemcpyDeviceToHost, s));
    return SEM_OK;
}

static void read_info(const sem_ctx *owner, int p, sem_solve_info *info)
{
    const SolveStateHost *H = (const SolveStateHost *)owner->solve_host;
    const PState &S = H->st[p];
    info->status = H->sync.err ? H->sync.err : S.status;
    info->iters = S.iters;
    info->outer_iters = S.outer;
    info->final_rnorm = S.rnorm;
    info->bnorm = S.bnorm;
}

extern "C" int sem_last_solve_info(sem_ctx *c, sem_solve_info *info)
{
    if (!c || !info) return SEM_ERR_ARG;
    read_info(c, 0, info);
    return SEM_OK;
}

// A launch that failed to enqueue left the workspaces' Jacobi vectors as they
// were: forget what fill_desc recorded for them.
static int jac_forget(sem_ctx *c, int rc)
{
    if (rc != SEM_OK)
        for (int k = 0; k < 8; ++k) c->ws[k].jac_ok = c->ws[k].jac32_ok = 0;
    return rc;
}

// Device-pointer solve used by the stepper.
int sem_pcg_solve_dev(sem_ctx *c, int slot, const double *b, double *x, double h1, double h2,
                      const sem_solve_opts &o, cudaStream_t s)
{
    const bool mixed = o.inner != SEM_F64 && o.inner != SEM_F64_NATIVE;
    if (!sem_pcg_accepts(c, o)) return SEM_ERR_ARG;
    ProbDesc d;
    fill_desc(c, c->ws[slot], b, x, h1, h2, mixed, inner_tc_of(o.inner, c->n), d);
    return jac_forget(c, enqueue(c, o, &d, 1, s));
}

// Several device-pointer solves on one context (workspace slots slot0 and up) in
// one launch.  ordered: FP64 solves take solver_ordered.cuh.
int sem_pcg_solve_dev_batch(sem_ctx *c, int np, const double *const *b, double *const *x, double h1,
                            double h2, const sem_solve_opts &o, cudaStream_t s, int slot0, bool ordered)
{
    if (np < 1 || np > 4 || slot0 < 0 || slot0 + np > 8) return SEM_ERR_ARG;
    for (int p = 0; p < np; ++p)
        if (!c->ws[slot0 + p].r) return SEM_ERR_ARG;
    const bool mixed = o.inner != SEM_F64 && o.inner != SEM_F64_NATIVE;
    if (!sem_pcg_accepts(c, o)) return SEM_ERR_ARG;
    ordered = ordered && o.inner == SEM_F64 && !tight_f64(o) && c->n <= 10;
    ProbDesc d[8];
    sem_ctx *const cs[8] = {c, c, c, c, c, c, c, c};
    for (int p = 0; p < np; ++p)  // (the ordered solver's problems make a Jacobi inverse each)
        fill_desc(c, c->ws[slot0 + p], b[p], x[p], h1, h2, mixed, inner_tc_of(o.inner, c->n), d[p], d, cs,
                  ordered ? 0 : p);
    return jac_forget(c, enqueue(c, o, d, np, s, ordered));
}

// Device address of the solver state of problem p of the last launch (iters, status).
const void *sem_solve_state_ptr(const sem_ctx *c, int p, int *iters_off, int *status_off)
{
    SolveStateHost *S = (SolveStateHost *)c->solve_dev;
    *iters_off = (int)offsetof(PState, iters);
    *status_off = (int)offsetof(PState, status);
    return &S->st[p];
}

const void *sem_solve_sync_ptr(const sem_ctx *c)
{
    return &((SolveStateHost *)c->solve_dev)->sync;
}

extern "C" int sem_pcg_solve(sem_ctx *c, const double *b, double *x, double h1, double h2,
                             const sem_solve_opts *opts, sem_solve_info *info, void *stream)
{
    if (!c || !b || !x) return SEM_ERR_ARG;
    sem_solve_opts o;
    sem_solve_opts_default(&o);
    if (opts) o = *opts;
    int rc = validate_opts(o);
    if (rc) return rc;
    if (!(h1 >= 0) || !(h2 >= 0) || (h1 == 0 && h2 == 0)) return SEM_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = sizeof(double) * c->nL;
    const void *bd;
    void *xd;
    int bh, xh;
    rc = sem_stage_in(c, b, bytes, 0, s, &bd, &bh);
    if (rc) return rc;
    const void *xin;
    rc = sem_stage_in(c, x, bytes, 1, s, &xin, &xh);
    if (rc) return rc;
    xd = (void *)xin;
    rc = sem_pcg_solve_dev(c, 0, (const double *)bd, (double *)xd, h1, h2, o, s);
    if (rc) return rc;
    if (xh) SEM_CUDA(cudaMemcpyAsync(x, xd, bytes, cudaMemcpyDeviceToHost, s));
    if (info || bh || xh) SEM_CUDA(cudaStreamSynchronize(s));
    if (info) {
        read_info(c, 0, info);
        return info->status;
    }
    return SEM_OK;
}

extern "C" int sem_pcg_solve_batched(int nprob, sem_ctx *const *ctxs, const double *const *b,
                                     double *const *x, const double *h1, const double *h2,
                                     const sem_solve_opts *opts, sem_solve_info *infos,
                                     void *stream)
{
    if (nprob < 1 || nprob > SEM_MAXP || !ctxs || !b || !x || !h1 || !h2) return SEM_ERR_ARG;
    sem_solve_opts o;
    sem_solve_opts_default(&o);
    if (opts) o = *opts;
    int rc = validate_opts(o);
    if (rc) return rc;
    const bool mixed = o.inner != SEM_F64 && o.inner != SEM_F64_NATIVE;
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<ProbDesc> d(nprob);
    std::vector<int> slot(nprob, 0);
    for (int p = 0; p < nprob; ++p) {
        sem_ctx *c = ctxs[p];
        if (!c || !b[p] || !x[p]) return SEM_ERR_ARG;
        if (!(h1[p] >= 0) || !(h2[p] >= 0) || (h1[p] == 0 && h2[p] == 0)) return SEM_ERR_ARG;
        if (!sem_pcg_accepts(c, o)) return SEM_ERR_ARG;
        if (!sem_is_device_ptr(b[p]) || !sem_is_device_ptr(x[p])) return SEM_ERR_ARG;
        for (int q = 0; q < p; ++q) slot[p] += (ctxs[q] == c);
        if (slot[p] >= 4) return SEM_ERR_ARG;
        if (!c->ws[slot[p]].r) {  // first use of a repeated context: one more workspace
            rc = sem_alloc_ws(c, slot[p]);
            if (rc) return rc;
        }
        fill_desc(c, c->ws[slot[p]], b[p], x[p], h1[p], h2[p], mixed, inner_tc_of(o.inner, c->n), d[p],
                  d.data(), ctxs, p);
    }
    sem_ctx *owner = ctxs[0];
    bool multi_ok = true, same = true;
    for (int p = 0; p < nprob; ++p) {
        multi_ok &= (d[p].n == 6 || d[p].n == 8 || d[p].n == 10);
        same &= (d[p].n == d[0].n);
    }
    if ((same && nprob <= 8) || multi_ok) {
        rc = enqueue(owner, o, d.data(), nprob, s);
        if (rc) {
            for (int p = 0; p < nprob; ++p) jac_forget(ctxs[p], rc);
            return rc;
        }
        if (infos) {
            SEM_CUDA(cudaStreamSynchronize(s));
            int worst = SEM_OK;
            for (int p = 0; p < nprob; ++p) {
                read_info(owner, p, &infos[p]);
                if (infos[p].status != SEM_OK && worst == SEM_OK) worst = infos[p].status;
            }
            return worst;
        }
        return SEM_OK;
    }
    // other order mixes: one launch per problem, in order
    int worst = SEM_OK;
    for (int p = 0; p < nprob; ++p) {
        if (d[p].jac_shared) {  // made by an earlier launch, or again by this one
            d[p].jac_shared = 0;
            d[p].jac_cached = 1;
        }
        rc = enqueue(owner, o, &d[p], 1, s);
        if (rc) {
            for (int q = 0; q < nprob; ++q) jac_forget(ctxs[q], rc);
            return rc;
        }
        if (infos) {
            SEM_CUDA(cudaStreamSynchronize(s));
            read_info(owner, 0, &infos[p]);
            if (infos[p].status != SEM_OK && worst == SEM_OK) worst = infos[p].status;
        }
    }
    return infos ? worst : SEM_OK;
}

// ---------------------------------------------------------------------------
// Autotuner of the inner path (SEM_F32_TUNED)
// ---------------------------------------------------------------------------

__global__ void k_tune_rhs(double *b, double *x, int64_t n)
{
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= n) return;
    b[q] = (double)((q * 7 + 3) % 11) - 5.0;
    x[q] = 0.0;
}

extern "C" int sem_set_inner_path(int N, int path)
{
    if (N < 1 || N > SEM_NMAX || path < 0 || path > 1 || (path == 1 && N > 7)) return SEM_ERR_ARG;
    g_inner_path[N] = path;
    return SEM_OK;
}

extern "C" int sem_tune_inner(sem_ctx *c, int iters, double *ms, int *best)
{
    if (!c || !best || c->nL == 0) return SEM_ERR_ARG;
    if (iters < 1) iters = 30;
    if (ms) ms[0] = ms[1] = -1.0;
    double *b = nullptr, *x = nullptr;
    if (cudaMalloc(&b, sizeof(double) * c->nL) != cudaSuccess) return SEM_ERR_NOMEM;
    if (cudaMalloc(&x, sizeof(double) * c->nL) != cudaSuccess) {
        cudaFree(b);
        return SEM_ERR_NOMEM;
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = SEM_OK;
    double t[2] = {-1.0, -1.0};
    const int ncand = c->N <= 7 ? 2 : 1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) rc = SEM_ERR_CUDA;
    for (int cand = 0; cand < ncand && rc == SEM_OK; ++cand) {
        // `iters` inner iterations of one refinement step (tolerances out of reach)
        sem_solve_opts o;
        sem_solve_opts_default(&o);
        o.inner = cand == 0 ? SEM_F32 : SEM_F16X2_TC;
        o.tol = 0.0;
        o.inner_tol = 1e-30;
        o.maxit = iters;
        o.max_outer = 1;
        float best_ms = 1e30f;
        for (int rep = 0; rep < 2 && rc == SEM_OK; ++rep) {
            k_tune_rhs<<<(unsigned)sem_ceil_div(c->nL, 256), 256>>>(b, x, c->nL);
            if (cudaEventRecord(e0, 0) != cudaSuccess) { rc = SEM_ERR_CUDA; break; }
            rc = sem_pcg_solve_dev(c, 0, b, x, 1.0, 1.0, o, 0);
            if (rc) break;
            if (cudaEventRecord(e1, 0) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess) {
                rc = SEM_ERR_CUDA;
                break;
            }
            float f = 0.f;
            cudaEventElapsedTime(&f, e0, e1);
            if (rep > 0 && f < best_ms) best_ms = f;  // the first run is a warm-up
        }
        if (rc == SEM_OK) t[cand] = best_ms / iters;
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(b);
    cudaFree(x);
    if (rc) return rc;
    const int bi = (ncand == 2 && t[1] >= 0 && t[1] < t[0]) ? 1 : 0;
    if (ms) {
        ms[0] = t[0];
        ms[1] = t[1];
    }
    *best = bi;
    return sem_set_inner_path(c->N, bi);
}

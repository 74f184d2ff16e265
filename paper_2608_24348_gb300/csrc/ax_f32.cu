// ax_f32.cu -- FP32 stand-alone element operator: direct-load kernel and a
// bulk-copy (TMA) staged kernel.
//
// The staged kernel streams each element group's two contiguous blocks -- the
// u slab (NE (N+1)^3 values) and the element-blocked geometry (7 NE (N+1)^3)
// -- into a two-stage shared-memory ring with cp.async.bulk; while the block
// computes group g the copy of its next group is in flight, so the kernel
// keeps enough bytes moving without needing many resident warps.
#include <stdint.h>
#include <string.h>

#include "ax_launch.cuh"
#include "ax_line32.cuh"
#include "tma.cuh"

// Tile shape of the staged kernel: about TH threads per block (whole
// elements of NP^2 threads) and ST ring stages.
template <int NP, int TH, int ST>
struct TmaAxCfg {
    static constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
    static constexpr int NE = (TH / NP2) > 0 ? TH / NP2 : 1;
    static constexpr int THREADS = NE * NP2;
    static constexpr int STAGES = ST;
    static constexpr size_t U_BYTES = sizeof(float) * NE * NP3;
    static constexpr size_t G_BYTES = sizeof(float) * 7 * NE * NP3;
    static constexpr size_t STAGE_BYTES = U_BYTES + G_BYTES;
    static constexpr size_t WORK_OFF = STAGES * STAGE_BYTES;
    static constexpr size_t WORK_BYTES = sizeof(float) * (2 * NP2 + (size_t)NE * 3 * NP3);
    static constexpr size_t BAR_OFF = (WORK_OFF + WORK_BYTES + 15) / 16 * 16;
    static constexpr size_t SMEM = BAR_OFF + 16 * STAGES;
    // every block copy must be a multiple of 16 bytes
    static constexpr bool OK = (NP3 * sizeof(float)) % 16 == 0 && SMEM <= 227 * 1024;
};

template <int NP, int TH, int ST>
__global__ void __launch_bounds__(TmaAxCfg<NP, TH, ST>::THREADS)
    k_ax_tma(const float *__restrict__ u, float *__restrict__ w, const float *__restrict__ geo,
             const float *__restrict__ D, float h1, float h2, int64_t E, int *err, long long timeout_ns)
{
    using T = TmaAxCfg<NP, TH, ST>;
    using C = T;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + T::BAR_OFF);
    float *work = reinterpret_cast<float *>(smem + T::WORK_OFF);
    float *sD = work, *sDT = work + NP * NP;
    const int grp = threadIdx.x / C::NP2, tid = threadIdx.x - grp * C::NP2;
    float *su = work + 2 * NP * NP + (size_t)grp * 3 * C::NP3;
    float *svr = su + C::NP3, *svs = svr + C::NP3;
    const int64_t groups = (E + C::NE - 1) / C::NE;

    auto issue = [&](int s, int64_t g) {
        const int64_t e0 = g * C::NE;
        const int64_t ne = (E - e0) < C::NE ? (E - e0) : C::NE;
        const uint32_t ub = (uint32_t)(ne * C::NP3 * sizeof(float));
        const uint32_t gb = (uint32_t)(7 * ne * C::NP3 * sizeof(float));
        unsigned char *st = smem + (size_t)s * T::STAGE_BYTES;
        mbar_expect_tx(&bar[s], ub + gb);
        bulk_g2s(st, u + e0 * C::NP3, ub, &bar[s]);
        bulk_g2s(st + T::U_BYTES, geo + e0 * 7 * C::NP3, gb, &bar[s]);
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < T::STAGES; ++s) mbar_init(&bar[s], 1);
        mbar_fence_init();
    }
    ax_load_D<NP, float>(D, sD, sDT);
    __syncthreads();
    if (threadIdx.x == 0)
        for (int s = 0; s < T::STAGES; ++s) {
            const int64_t g = blockIdx.x + (int64_t)s * gridDim.x;
            if (g < groups) issue(s, g);
        }
    int64_t it = 0;
    bool failed = false;
    for (;; ++it) {
        const int64_t g = blockIdx.x + it * gridDim.x;
        if (g >= groups) break;
        const int s = (int)(it % T::STAGES);
        const uint32_t parity = (uint32_t)((it / T::STAGES) & 1);
        const bool ok = mbar_wait_bounded(&bar[s], parity, timeout_ns);
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        const unsigned char *st = smem + (size_t)s * T::STAGE_BYTES;
        const float *su_stage = reinterpret_cast<const float *>(st) + (size_t)grp * C::NP3;
        const float *geo_stage = reinterpret_cast<const float *>(st + T::U_BYTES) + (size_t)grp * 7 * C::NP3;
        const int64_t e = g * C::NE + grp;
        const bool active = grp < C::NE && e < E;
        float *we = w + (active ? e : 0) * C::NP3;
        auto load = [&](int p) { return su_stage[p]; };
        auto store = [&](int p, float v, float) { we[p] = v; };
        ax_element<NP, float>(load, store, geo_stage, h1, h2, sD, sDT, su, svr, svs, tid, active);
        // the stage is free again (ax_element ends with a block barrier)
        if (threadIdx.x == 0) {
            const int64_t g2 = g + (int64_t)T::STAGES * gridDim.x;
            if (g2 < groups) {
                fence_proxy_async_smem();
                issue(s, g2);
            }
        }
    }
    if (failed && threadIdx.x == 0) {
        atomicExch(err, SEM_ERR_TIMEOUT);
        // wait (bounded) for this block's copies still in flight before exiting
        for (int64_t k = it; k < it + T::STAGES; ++k) {
            const int64_t g = blockIdx.x + k * gridDim.x;
            if (g >= groups) break;
            mbar_wait_bounded(&bar[k % T::STAGES], (uint32_t)((k / T::STAGES) & 1), timeout_ns);
        }
    }
}

template <int NP, int TH, int ST>
static int launch_tma(const sem_ctx *c, const float *u, float *w, float h1, float h2, cudaStream_t s)
{
    using T = TmaAxCfg<NP, TH, ST>;
    if constexpr (!T::OK) {
        return SEM_ERR_ARG;
    } else {
        auto kern = k_ax_tma<NP, TH, ST>;
        static std::atomic<unsigned> attr{0};
        SEM_CUDA(sem_smem_attr(kern, T::SMEM, attr));
        int per_sm = 0;
        SEM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, T::THREADS, T::SMEM));
        if (per_sm < 1) return SEM_ERR_ARG;
        const int64_t groups = sem_ceil_div(c->E, T::NE);
        int64_t grid = (int64_t)per_sm * c->num_sms;
        if (grid > groups) grid = groups;
        kern<<<(unsigned)grid, T::THREADS, T::SMEM, s>>>(u, w, c->geo32, c->tab32 + 2 * c->n, h1, h2, c->E,
                                                         (int *)c->err_dev, 2000000000LL);
        SEM_CHECK_LAUNCH();
        return SEM_OK;
    }
}

// The line operator (ax_line32.cuh): the next element group's u copied into shared
// memory by asynchronous copies (every thread its own column), groups synchronised
// by themselves.  Bound: FP32 issue and HBM alike (36 bytes a node); 0.1055 ms at
// 32^3 elements, N = 7 (0.1209 by the staged form above, 0.089 the bytes alone).
//
// Blocks of 256 threads, or of the whole warps of one element for N >= 11, whose
// columns fill 256 threads badly.  Registers decide between the latency of one
// element (a whole line and its result want NP^2 / 2 or so) and the elements in
// flight: blocks an SM by order, measured at one to four (us; in brackets direct
// loads or, N = 7 and 9, the staged form, which the smallest meshes took before):
//  - N = 8: three, 77.6 at 13824 elements (two 93.7, four 83.3), 5.2 at 252 (four 6.4) [145, 5.5]
//  - N = 9: three, 113 at 13824 (two 132, four 136) [145]
//  - N = 10: two, 90.2 at 8000 (one 143, three 97.5), 5.2 at 125 [189, 5.7]
//  - N = 11: three blocks of 160, 132 at 8000 (256 threads, one block: 305) [198]
//  - N = 12: two blocks of 192, 109 at 3840 (256 threads, one block: 176) [148]
//  - N = 13: two blocks of 224 above six elements an SM, 90.8 at 1872 (one 105); one
//    below, 31.6 at 648 (two 34.2) [144, 29.3]
//  - others: four, or one (N >= 14: 128 registers spill).
// A mesh that one block an SM holds (two at N = 9) takes two blocks' registers at
// N = 2, 6, 7 and 9, since only its latency counts: N = 2, 36 elements 2.5 (four 2.7)
// [2.6]; N = 6, 648 elements 4.4 (four 4.9) [4.4]; N = 7, 36 elements 3.6 (3.8) [3.6];
// N = 9, 252 elements 5.3 (three 6.0, four 7.3) [5.4].  Direct loads stay ahead at N = 2
// above 4000 elements (15.0 against 16.5 at 65536) and N = 13 below 900 (29.3 against
// 31.6 at 648).  The staged form's and the direct loads' error is three times that of
// whole lines (1.2e-7 against 4.2e-8 of the result at N = 7).
template <int NP>
struct L32Shape {
    static constexpr int NP2 = NP * NP;
    static constexpr int GT = NP <= 4    ? 32
                              : NP == 8  ? 64
                              : NP >= 12 ? (NP2 + 31) / 32 * 32
                              : (NP == 5 || NP == 6 || NP == 10 || NP == 11) ? 128 : 256;
    static constexpr int TB = NP >= 12 ? GT : 256;
    static constexpr int GE = GT / NP2, NG = TB / GT, NE = NG * GE;
    static constexpr size_t SMEM = sizeof(float) * ((size_t)NE * 3 * Line32Cfg<NP>::SLAB + NP * TB);
    // blocks an SM (registers), for large meshes and for small ones
    static constexpr int MINB = NP == 9 || NP == 10 || NP == 12 ? 3 : NP == 11 || NP == 13 || NP == 14 ? 2 : NP >= 15 ? 1 : 4;
    static constexpr int MINB_SMALL = NP == 3 || NP == 7 || NP == 8 || NP == 10 ? 2 : NP == 14 ? 1 : MINB;
    // the largest small mesh, in elements an SM: a block's worth, N = 9 two blocks', N = 13 six
    static constexpr int SMALL = NP == 14 ? 6 : NP == 10 ? 4 : NE;
};

template <int NP, int MINB>
__global__ void __launch_bounds__(L32Shape<NP>::TB, MINB)
    k_ax_line32(const float *__restrict__ u, float *__restrict__ w, const float *__restrict__ geo,
                const __grid_constant__ LineTab32 T, float h1, float h2, int64_t E)
{
    using S = L32Shape<NP>;
    constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
    extern __shared__ __align__(16) unsigned char smem[];
    const int grp = threadIdx.x / S::GT, lt = threadIdx.x - grp * S::GT;
    const int ge = lt / NP2 < S::GE ? lt / NP2 : 0, tid = lt / NP2 < S::GE ? lt - ge * NP2 : -1;
    float *slab = reinterpret_cast<float *>(smem) + (size_t)(grp * S::GE + ge) * 3 * Line32Cfg<NP>::SLAB;
    float *su = reinterpret_cast<float *>(smem) + (size_t)S::NE * 3 * Line32Cfg<NP>::SLAB + threadIdx.x;
    auto sync = [&] {
        if constexpr (S::GT == S::TB)
            __syncthreads();
        else if constexpr (S::GT == 32)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(S::GT) : "memory");
    };
    const int64_t groups = (E + S::GE - 1) / S::GE, stride = (int64_t)gridDim.x * S::NG;
    auto fetch = [&](int64_t g) {
        const int64_t e = g * S::GE + ge;
        if (g < groups && tid >= 0 && e < E) {
#pragma unroll
            for (int k = 0; k < NP; ++k) cp_async4(su + k * S::TB, u + e * NP3 + k * NP2 + tid);
        }
    };
    int64_t g = (int64_t)grp * gridDim.x + blockIdx.x;
    fetch(g);
    for (; g < groups; g += stride) {
        const int64_t e0 = g * S::GE, e = e0 + ge;
        const bool active = tid >= 0 && e < E;
        if (lt == 0)
            l2_prefetch_span(geo, e0 * 7 * NP3 * 4, (e0 + S::GE < E ? e0 + S::GE : E) * 7 * NP3 * 4);
        float *we = w + (active ? e : 0) * NP3 + tid;
        cp_async_wait_all();
        auto load = [&](int k) { return su[k * S::TB]; };
        auto store = [&](int k, float v, float) { we[k * NP2] = v; };
        ax_line32_element<NP>(load, store, geo + (active ? e : 0) * 7 * NP3, h1, h2, T, slab, tid, active,
                              [&] { fetch(g + stride); }, sync);
    }
}

template <int NP, int MINB>
static int launch_line32_regs(const sem_ctx *c, const float *u, float *w, float h1, float h2, cudaStream_t s)
{
    using S = L32Shape<NP>;
    static std::atomic<unsigned> attr{0};
    SEM_CUDA(sem_smem_attr(k_ax_line32<NP, MINB>, S::SMEM, attr));
    int per_sm = 0;
    SEM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ax_line32<NP, MINB>, S::TB, S::SMEM));
    if (per_sm < 1) return SEM_ERR_ARG;
    const int64_t groups = sem_ceil_div(c->E, S::GE);
    int64_t grid = (int64_t)per_sm * c->num_sms;
    if (grid > groups) grid = groups;
    LineTab32 T;
    memset(&T, 0, sizeof(T));
    for (int t = 0; t < NP * NP; ++t) T.d[t] = (float)c->hD[t];
    k_ax_line32<NP, MINB><<<(unsigned)grid, S::TB, S::SMEM, s>>>(u, w, c->geo32, T, h1, h2, c->E);
    SEM_CHECK_LAUNCH();
    return SEM_OK;
}

template <int NP>
static int launch_line32(const sem_ctx *c, const float *u, float *w, float h1, float h2, cudaStream_t s)
{
    using S = L32Shape<NP>;
    if constexpr (S::MINB_SMALL != S::MINB)
        // (of the whole mesh, so that a call on host buffers, in chunks, does the same)
        if ((int64_t)c->nelx * c->nely * c->nelz <= (int64_t)S::SMALL * c->num_sms)
            return launch_line32_regs<NP, S::MINB_SMALL>(c, u, w, h1, h2, s);
    return launch_line32_regs<NP, S::MINB>(c, u, w, h1, h2, s);
}

// Variants of the FP32 operator (see sem_tune_ax): 0 whole lines, 1 staged
// 256 threads x 2 stages, 2 staged 128 threads x 3 stages.
int sem_launch_ax_f32_variant(const sem_ctx *c, int variant, const float *u, float *w, float h1,
                              float h2, cudaStream_t s)
{
    const int n = c->n;
    const bool staged_ok = ((uintptr_t)u % 16) == 0 && c->err_dev && (n == 4 || n == 6 || n == 8 || n == 10);
    if (variant != 0 && staged_ok) {
        switch (n * 8 + variant) {
            case 4 * 8 + 1: return launch_tma<4, 256, 2>(c, u, w, h1, h2, s);
            case 6 * 8 + 1: return launch_tma<6, 256, 2>(c, u, w, h1, h2, s);
            case 8 * 8 + 1: return launch_tma<8, 256, 2>(c, u, w, h1, h2, s);
            case 10 * 8 + 1: return launch_tma<10, 256, 2>(c, u, w, h1, h2, s);
            case 4 * 8 + 2: return launch_tma<4, 128, 3>(c, u, w, h1, h2, s);
            case 6 * 8 + 2: return launch_tma<6, 128, 3>(c, u, w, h1, h2, s);
            case 8 * 8 + 2: return launch_tma<8, 128, 3>(c, u, w, h1, h2, s);
            case 10 * 8 + 2: return launch_tma<10, 128, 3>(c, u, w, h1, h2, s);
            default: break;
        }
    }
    SEM_DISPATCH_NP(n, return launch_line32<NP>(c, u, w, h1, h2, s));
    return SEM_ERR_ARG;
}

// The operator with the three directions' products of a node summed in turn (the
// order of ax_element), whatever variant is in force.  The multigrid V-cycle uses
// it: its FP32 rounding passes through GMRES into the solution at the level of
// the pressure tolerance, so a change of summation order there would change the
// stepper's results by far more than FP64 rounding.
int sem_launch_ax_f32_columns(const sem_ctx *c, const float *u, float *w, float h1, float h2, cudaStream_t s)
{
    const float *tab = c->tab32 + 2 * c->n;
    switch (c->n) {
        case 4: return launch_tma<4, 256, 2>(c, u, w, h1, h2, s);
        case 6: return launch_tma<6, 256, 2>(c, u, w, h1, h2, s);
        case 8: return launch_tma<8, 128, 3>(c, u, w, h1, h2, s);
        case 10: return launch_tma<10, 128, 3>(c, u, w, h1, h2, s);
        case 2: return launch_ax<2, float>(c, u, w, c->geo32, tab, h1, h2, s);
        case 3: return launch_ax<3, float>(c, u, w, c->geo32, tab, h1, h2, s);
        case 5: return launch_ax<5, float>(c, u, w, c->geo32, tab, h1, h2, s);
        case 7: return launch_ax<7, float>(c, u, w, c->geo32, tab, h1, h2, s);
        case 9: return launch_ax<9, float>(c, u, w, c->geo32, tab, h1, h2, s);
        default: return SEM_ERR_ARG;
    }
}

// ax_dfl.cu -- stand-alone FP64-accurate sem_ax for odd N+1 <= 11: float pairs
// by whole folded lines (ax_dfl.cuh).
//
// Bound: FP32 issue (about 560 operations a node at N = 8; 72 bytes a node).
// 256/(N+1)^2 elements a block, u of the next elements copied into shared
// memory by asynchronous copies (every thread its own column) while the current
// ones are in flight.  It replaces the unfolded form whose contractions read
// every operand of every product from shared memory; sem_ax at N = 8, 18 x 21 x
// 17 elements (4.7 M nodes): 212 us before, 157 us.
#include <stdlib.h>

#include "ax_dfl.cuh"
#include "common.cuh"
#include "tma.cuh"

template <int NP>
struct DflShape {
    static constexpr int NE = 256 / (NP * NP);
    static constexpr int THREADS = NE * NP * NP;
    static constexpr size_t STAGE_OFF = sizeof(dfp) * NE * 3 * DflCfg<NP>::SLAB;
    static constexpr size_t RED_OFF = STAGE_OFF + sizeof(double) * NP * THREADS;
    static constexpr size_t SMEM = RED_OFF + sizeof(unsigned) * NE;
};

struct DflBlockSync {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

template <int NP>
__global__ void __launch_bounds__(DflShape<NP>::THREADS, 2)
    k_ax_dfl(const double *__restrict__ u, double *__restrict__ w, const dfp *__restrict__ geo,
             const __grid_constant__ DflTabs T, dfp h1, dfp h2, int64_t E)
{
    using S = DflShape<NP>;
    constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dfp *slabs = reinterpret_cast<dfp *>(smem_raw);
    double *su = reinterpret_cast<double *>(smem_raw + S::STAGE_OFF) + threadIdx.x;
    unsigned *red = reinterpret_cast<unsigned *>(smem_raw + S::RED_OFF);
    const int grp = threadIdx.x / NP2, tid = threadIdx.x - grp * NP2;
    if (tid == 0) red[grp] = 0u;
    auto fetch = [&](int64_t e0) {
        if (e0 + grp < E) {
            const double *src = u + (e0 + grp) * NP3 + tid;
#pragma unroll
            for (int k = 0; k < NP; ++k) cp_async8(su + k * S::THREADS, src + k * NP2);
        }
    };
    const int64_t stride = (int64_t)gridDim.x * S::NE;
    int64_t e0 = (int64_t)blockIdx.x * S::NE;
    fetch(e0);
    __syncthreads();
    for (; e0 < E; e0 += stride) {
        if (threadIdx.x == 0)
            l2_prefetch_span(geo, e0 * 7 * NP3 * 8, (e0 + S::NE < E ? e0 + S::NE : E) * 7 * NP3 * 8);
        const int64_t e = e0 + grp;
        const bool active = e < E;
        double *we = w + (active ? e : 0) * NP3;
        cp_async_wait_all();
        auto load = [&](int p) { return su[(p - tid) / NP2 * S::THREADS]; };
        auto store = [&](int p, double v) { we[p] = v; };
        ax_dfl_element<NP>(load, store, geo + (active ? e : 0) * 7 * NP3, h1, h2, T,
                           slabs + (size_t)grp * 3 * DflCfg<NP>::SLAB, red + grp, tid, active,
                           [&] { fetch(e0 + stride); }, DflBlockSync());
    }
}

template <int NP>
static int launch_dfl(const sem_ctx *c, const double *u, double *w, double h1, double h2, cudaStream_t s)
{
    using S = DflShape<NP>;
    if (!c->dfl_tabs) return SEM_ERR_ARG;
    static std::atomic<unsigned> attr{0};
    SEM_CUDA(sem_smem_attr(k_ax_dfl<NP>, S::SMEM, attr));
    int per_sm = 0;
    SEM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ax_dfl<NP>, S::THREADS, S::SMEM));
    if (per_sm < 1) return SEM_ERR_ARG;
    const int64_t groups = sem_ceil_div(c->E, S::NE);
    int64_t grid = (int64_t)per_sm * c->num_sms;
    if (grid > groups) grid = groups;
    const float a = (float)h1, b = (float)h2;
    const dfp H1 = {a, (float)(h1 - (double)a)}, H2 = {b, (float)(h2 - (double)b)};
    k_ax_dfl<NP><<<(unsigned)grid, S::THREADS, S::SMEM, s>>>(u, w, (const dfp *)c->geodf,
                                                             *(const DflTabs *)c->dfl_tabs, H1, H2, c->E);
    SEM_CHECK_LAUNCH();
    return SEM_OK;
}

// SEM_ERR_ARG where the order has no such kernel.
int sem_launch_ax_dfl(const sem_ctx *c, const double *u, double *w, double h1, double h2, cudaStream_t s)
{
    switch (c->n) {
        case 3: return launch_dfl<3>(c, u, w, h1, h2, s);
        case 5: return launch_dfl<5>(c, u, w, h1, h2, s);
        case 7: return launch_dfl<7>(c, u, w, h1, h2, s);
        case 9: return launch_dfl<9>(c, u, w, h1, h2, s);
        case 11: return launch_dfl<11>(c, u, w, h1, h2, s);
        default: return SEM_ERR_ARG;
    }
}

int sem_make_dfl_tabs(sem_ctx *c)
{
    if (c->n % 2 == 0 || c->n > 11) return SEM_OK;
    DflTabs *T = (DflTabs *)calloc(1, sizeof(DflTabs));
    if (!T) return SEM_ERR_NOMEM;
    ax_dfl_tables(c->n, c->hD, T);
    c->dfl_tabs = T;
    return SEM_OK;
}

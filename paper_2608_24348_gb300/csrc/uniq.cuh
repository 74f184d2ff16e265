// uniq.cuh -- passes over the unique nodes of the structured box.
//
// A pass that gathers every copy of a node (the direct-stiffness sum and what
// is fused with it) gives a thread a chunk of CH consecutive nodes of one
// element's row (fixed j, k), so that whole vectors are loaded and stored (one
// 32-byte access an array at N+1 = 8 in FP64) and the index arithmetic is paid
// once a chunk instead of once a node; per node it was most of the time of such
// a pass (the solver's FP32 update at 24^3 elements, N = 7: 83 us a node at a
// time, 40 us in chunks of four).
//
// Node counts stay below 2^31 (the geometry of 2^31 nodes would not fit the
// device), so offsets are 32-bit.
#pragma once

#include "common.cuh"
#include "gs.cuh"

// Unsigned division by a launch constant d (Granlund & Montgomery 1994, the
// round-up form): exact for every x < 2^31.
struct FastDiv {
    unsigned d, m, s;
};

static inline FastDiv fast_div(unsigned d)
{
    FastDiv f = {d, 0, 0};
    while ((1ull << f.s) < d) ++f.s;
    f.m = (unsigned)((((1ull << f.s) - d) << 32) / d + 1);
    return f;
}

__device__ __forceinline__ unsigned fd_div(unsigned x, const FastDiv &f)
{
    return (__umulhi(x, f.m) + x) >> f.s;
}

// Copies of index g along one direction in units of order N (gs_copies_1d on
// unsigned numbers; the same order of copies).
__device__ __forceinline__ int uq_copies(unsigned g, unsigned N, int nel, int periodic, unsigned ce[2],
                                         unsigned ci[2])
{
    const unsigned e = g / N, i = g - e * N;  // (N is a constant after inlining)
    ce[0] = e;
    ci[0] = i;
    ce[1] = e - 1;
    ci[1] = N;
    if (i != 0) return 1;
    if (periodic) {
        if (e == 0) ce[1] = nel - 1;
        return 2;
    }
    if ((int)e == nel) {  // the far boundary plane: the last node of the last element
        ce[0] = e - 1;
        ci[0] = N;
        return 1;
    }
    return e > 0 ? 2 : 1;
}

// The mesh of a pass.
struct UqMesh {
    GsDesc d;
    FastDiv ngy, nelx;
};

static inline UqMesh uq_mesh(const GsDesc &d)
{
    return {d, fast_div((unsigned)d.ngy), fast_div((unsigned)d.nelx)};
}

template <int NP>
struct UqCfg {
    static constexpr int CH = NP % 4 == 0 ? 4 : NP % 2 == 0 ? 2 : NP % 3 == 0 ? 3 : NP <= 7 ? NP : 1;
    static constexpr int NC = NP / CH;  // chunks a row
};

// Values that an access to a chunk takes at once (uq_ldv, uq_stv): a vector has to
// be aligned to as many.  An E-vector's offset into a larger array is a multiple of
// its length, which for even N+1 is a multiple of this, but for odd N+1 may be odd.
template <int NP>
__host__ __device__ constexpr int uq_width()
{
    constexpr int CH = UqCfg<NP>::CH;
    return CH == 4 || CH == 2 ? CH : 1;
}

// The copies of a chunk: offset f of its first node in the first row (the
// owner's), distances dy, dz to the rows of the neighbours that share it, and
// distance dl from f to the left neighbour's copy of that node (only the first
// node of an element's row has one; the last node, i = N, belongs to the right
// neighbour except at a far boundary plane).  Offsets add modulo 2^32.  own:
// nodes of the chunk that this thread owns.  The copies of a node in the order
// row, y row, z row, yz row, the own element before the left one -- the order in
// which sem_dssum sums them.
struct UqChunk {
    unsigned f, dl, dy, dz;
    bool hl, hy, hz;
    int own;
};

template <int NP>
__host__ __device__ __forceinline__ unsigned uq_units(const UqMesh &M)
{
    return (unsigned)UqCfg<NP>::NC * (unsigned)M.d.ngy * (unsigned)M.d.nelx * (unsigned)M.d.ngz;
}

// Chunk t: the chunks of a row, then the rows gy (consecutive rows of an
// element are contiguous), then the elements along x, then gz.
template <int NP>
__device__ __forceinline__ UqChunk uq_chunk(const UqMesh &M, unsigned t)
{
    constexpr unsigned CH = UqCfg<NP>::CH, NC = UqCfg<NP>::NC, N = NP - 1, N2 = NP * NP, N3 = N2 * NP;
    const GsDesc &d = M.d;
    const unsigned u = t / NC, c = t - u * NC;
    const unsigned v = fd_div(u, M.ngy), gy = u - v * M.ngy.d;
    const unsigned gz = fd_div(v, M.nelx), ex = v - gz * M.nelx.d;
    const unsigned ny = (unsigned)d.nelx * N3, nz = ny * (unsigned)d.nely;
    unsigned e[2], i[2];
    UqChunk U;
    U.hy = uq_copies(gy, N, d.nely, d.py, e, i) > 1;
    U.f = ex * N3 + c * CH + e[0] * ny + i[0] * NP;
    U.dy = (e[1] - e[0]) * ny + (i[1] - i[0]) * NP;
    U.hz = uq_copies(gz, N, d.nelz, d.pz, e, i) > 1;
    U.f += e[0] * nz + i[0] * N2;
    U.dz = (e[1] - e[0]) * nz + (i[1] - i[0]) * N2;
    U.hl = c == 0 && (ex > 0 || d.px);
    U.dl = N - (ex > 0 ? N3 : 0u - ((unsigned)d.nelx - 1) * N3);
    U.own = c == NC - 1 && (d.px || ex + 1 < (unsigned)d.nelx) ? CH - 1 : CH;
    return U;
}

// Loads of the unique phases.  Volatile: the compiler keeps them where they
// are written, a chunk's loads ahead of the first use of one.  Whole-sector
// vectors go to L2 only; smaller ones may find their sector in L1 (the grid
// barrier's acquire has dropped what an earlier phase left there).
__device__ __forceinline__ double uq_ld(const double *a)
{
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(a));
    return v;
}
__device__ __forceinline__ float uq_ld(const float *a)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(a));
    return v;
}

template <int CH>
__device__ __forceinline__ void uq_ldv(const double *a, double (&v)[CH])
{
    if constexpr (CH == 4) {
        asm volatile("ld.global.cg.v4.f64 {%0, %1, %2, %3}, [%4];"
                     : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(a));
    } else if constexpr (CH == 2) {
        asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "l"(a));
    } else {
#pragma unroll
        for (int i = 0; i < CH; ++i) v[i] = uq_ld(a + i);
    }
}
template <int CH>
__device__ __forceinline__ void uq_ldv(const float *a, float (&v)[CH])
{
    if constexpr (CH == 4) {
        asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(a));
    } else if constexpr (CH == 2) {
        asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "l"(a));
    } else {
#pragma unroll
        for (int i = 0; i < CH; ++i) v[i] = uq_ld(a + i);
    }
}

// Stores of the first `own` values (the whole vector where all are owned).
template <int CH>
__device__ __forceinline__ void uq_stv(double *a, const double (&v)[CH], int own)
{
    if (CH == 4 && own == CH) {
        if constexpr (CH == 4)
            asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(a), "d"(v[0]), "d"(v[1]), "d"(v[2]),
                         "d"(v[3]) : "memory");
    } else if (CH == 2 && own == CH) {
        if constexpr (CH == 2) *reinterpret_cast<double2 *>(a) = make_double2(v[0], v[1]);
    } else {
#pragma unroll
        for (int i = 0; i < CH; ++i)
            if (i < own) a[i] = v[i];
    }
}
template <int CH>
__device__ __forceinline__ void uq_stv(float *a, const float (&v)[CH], int own)
{
    if (CH == 4 && own == CH) {
        if constexpr (CH == 4) *reinterpret_cast<float4 *>(a) = make_float4(v[0], v[1], v[2], v[3]);
    } else if (CH == 2 && own == CH) {
        if constexpr (CH == 2) *reinterpret_cast<float2 *>(a) = make_float2(v[0], v[1]);
    } else {
#pragma unroll
        for (int i = 0; i < CH; ++i)
            if (i < own) a[i] = v[i];
    }
}

// s = the sums over every copy of the chunk's nodes.  (Adding the zero of an
// absent left copy leaves the sum as it is.)  more(): further loads of the
// caller, issued behind the first ones.
template <typename T, int CH, class More>
__device__ __forceinline__ void uq_gather(const T *a, const UqChunk &U, T (&s)[CH], const More &more)
{
    T ty[CH], tz[CH], l0 = T(0), ly = T(0), lz = T(0);
    uq_ldv(a + U.f, s);
    if (U.hl) l0 = uq_ld(a + (U.f + U.dl));
    more();
    if (U.hy) {
        uq_ldv(a + (U.f + U.dy), ty);
        if (U.hl) ly = uq_ld(a + (U.f + U.dy + U.dl));
    }
    if (U.hz) {
        uq_ldv(a + (U.f + U.dz), tz);
        if (U.hl) lz = uq_ld(a + (U.f + U.dz + U.dl));
    }
    s[0] += l0;
    if (U.hy) {
#pragma unroll
        for (int i = 0; i < CH; ++i) s[i] += ty[i];
        s[0] += ly;
    }
    if (U.hz) {
        const unsigned o = U.f + U.dy + U.dz;
        if (U.hy) {
            uq_ldv(a + o, ty);
            ly = U.hl ? uq_ld(a + (o + U.dl)) : T(0);
        }
#pragma unroll
        for (int i = 0; i < CH; ++i) s[i] += tz[i];
        s[0] += lz;
        if (U.hy) {
#pragma unroll
            for (int i = 0; i < CH; ++i) s[i] += ty[i];
            s[0] += ly;
        }
    }
}

// Every copy of the chunk's nodes takes its value.
template <typename T, int CH>
__device__ __forceinline__ void uq_scatter(T *a, const UqChunk &U, const T (&z)[CH])
{
    auto row = [&](unsigned o) {
        uq_stv(a + o, z, U.own);
        if (U.hl) a[o + U.dl] = z[0];
    };
    row(U.f);
    if (U.hy) row(U.f + U.dy);
    if (U.hz) {
        row(U.f + U.dz);
        if (U.hy) row(U.f + U.dy + U.dz);
    }
}

// Loads of a chunk of a caller's vector, whose alignment is only known at run
// time (vec); nodes past the owned ones give 0 or what lies there.
template <int CH>
__device__ __forceinline__ void uq_ldu(const double *a, double (&v)[CH], int own, bool vec)
{
    if (vec) {
        uq_ldv(a, v);
    } else {
#pragma unroll
        for (int i = 0; i < CH; ++i) v[i] = i < own ? uq_ld(a + i) : 0.0;
    }
}

// a = f(node, a) at every copy of the chunk's nodes of a caller's vector, two
// rows at a time with their loads ahead of the stores.
template <int CH, class F>
__device__ __forceinline__ void uq_update(double *a, const UqChunk &U, bool vec, const F &f)
{
#pragma unroll 1
    for (int z = 0; z < (U.hz ? 2 : 1); ++z) {
        const unsigned o0 = U.f + (z ? U.dz : 0u), o1 = o0 + U.dy;
        double v0[CH], v1[CH], l0 = 0.0, l1 = 0.0;
        uq_ldu(a + o0, v0, U.own, vec);
        if (U.hl) l0 = uq_ld(a + (o0 + U.dl));
        if (U.hy) {
            uq_ldu(a + o1, v1, U.own, vec);
            if (U.hl) l1 = uq_ld(a + (o1 + U.dl));
        }
        auto put = [&](unsigned o, double (&v)[CH], double l) {
#pragma unroll
            for (int i = 0; i < CH; ++i) v[i] = f(i, v[i]);
            if (vec) {
                uq_stv(a + o, v, U.own);
            } else {
#pragma unroll
                for (int i = 0; i < CH; ++i)
                    if (i < U.own) a[o + i] = v[i];
            }
            if (U.hl) a[o + U.dl] = f(0, l);
        };
        put(o0, v0, l0);
        if (U.hy) put(o1, v1, l1);
    }
}

// f(offset, node) for every copy of the chunk's nodes.
template <int CH, class F>
__device__ __forceinline__ void uq_each(const UqChunk &U, const F &f)
{
    for (int r = 0; r < 4; ++r) {
        if (((r & 1) && !U.hy) || ((r & 2) && !U.hz)) continue;
        const unsigned o = U.f + (r & 1 ? U.dy : 0u) + (r & 2 ? U.dz : 0u);
#pragma unroll
        for (int i = 0; i < CH; ++i)
            if (i < U.own) f(o + i, i);
        if (U.hl) f(o + U.dl, 0);
    }
}

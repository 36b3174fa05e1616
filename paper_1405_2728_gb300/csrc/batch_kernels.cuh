// Descriptors and kernels of the grouped batch (batch.cu): each grouped kernel
// runs one stage of the minimiser iteration over the work items of all problems
// still running.  They are compiled in translation units of their own
// (group_*.cu), which hand batch.cu their addresses.
#pragma once

#include "common.cuh"
#include "field_kernels.cuh"

namespace {

// the FFT arithmetic of a group's fields, and its y-z stage
template <typename T> using FA = typename fft_of<T>::type;
template <typename T, int PZ, int L, bool SEP>
__device__ __forceinline__ void yz_of(const Geom &g, const FieldPtrs<T> &P, int tid, int nth, int kx)
{
    if constexpr (!is_fx<FA<T>>) yz_body<PZ, L>(g, P, tid, nth, kx);
    else if constexpr (L == 0 && !(SEP && PZ == 1)) yz_body_fx<PZ, -1, (SEP || PZ == 1)>(g, P, tid, nth, kx);
}
// double grids of several layers with scales per component: a kernel of their own (SEP), launched if a batch has one, as
// both kinds in one kernel spill 2 KB a thread
template <typename T> __host__ __device__ inline bool group_sep(const Geom &g) { return is_fx<FA<T>> && g.sep && g.Pz > 1; }

// one problem of a grouped launch, as the grouped kernels read it
template <typename T>
struct GFilm {
    Geom g;
    FieldPtrs<T> P;
    int nth_xf, nth_x, nth_yz;   // working threads of the three stages (the problem's own launch shapes)
    int gx_x, nblk_x;            // x-inverse grid: CTAs along y, CTAs in all
    int first[3], count[3];      // the problem's work items of each stage (x-forward, y-z, x-inverse)
};

// Problems still running in this iteration, as a compacted work list: the
// grouped kernels are persistent and walk virtual item indices 0 ..
// prefix[s][nact] - 1 of stage s; index v belongs to films[a] for the a with
// prefix[s][a] <= v < prefix[s][a + 1].  Layout in device memory:
// nact, films[nf], prefix[3][nf + 1] (ints).
struct GActive {
    int *base;
    int nf;
    __device__ int &nact() const { return base[0]; }
    __device__ int *films() const { return base + 1; }
    __device__ int *prefix(int s) const { return base + 1 + nf + s * (nf + 1); }
};

struct GItem { int film, bx, by; };

template <typename T>
__device__ __forceinline__ void load_film(GFilm<T> &f, const GFilm<T> *src)
{
    const int nw = (int)(sizeof(GFilm<T>) / sizeof(int));
    for (int i = threadIdx.x; i < nw; i += blockDim.x)
        reinterpret_cast<int *>(&f)[i] = reinterpret_cast<const int *>(src)[i];
    __syncthreads();
}

// the work item behind virtual index v of stage s (binary search over the
// active problems' prefix sums)
__device__ __forceinline__ GItem active_item(const GActive &A, const int *first, const GItem *items, int s, int v)
// first[s * nf + f]: where problem f's items start in stage s's item array
{
    const int *pre = A.prefix(s);
    int lo = 0, hi = A.nact() - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pre[mid] <= v) lo = mid; else hi = mid - 1;
    }
    const int f = A.films()[lo];
    return items[first[s * A.nf + f] + (v - pre[lo])];
}

// Persistent grouped kernels: CTA b takes virtual items b, b + gridDim.x, ...
// of the problems still running.  Items of a stage are independent, so the
// order does not matter; the shared memory is reused item after item.
#define MM_GROUP_LOOP(STAGE)                                                                  \
    __shared__ __align__(16) GFilm<T> f;                                                      \
    const int total = A.prefix(STAGE)[A.nact()];                                              \
    for (int v = blockIdx.x; v < total; v += gridDim.x) {                                    \
        __syncthreads();                                                                      \
        const GItem it = active_item(A, first_of, items, STAGE, v);                           \
        load_film(f, films + it.film);

template <typename T>
__global__ void __launch_bounds__(768) k_xfwd_group(const GFilm<T> *films, const GItem *items, const int *first_of,
                                                    GActive A)
{
    MM_GROUP_LOOP(0)
        switch (lx_of(f.g.Hx)) {
#define C(L) case L: xfwd_body<T, FA<T>, true, L>(f.g, f.P, threadIdx.x, f.nth_xf, it.bx, it.by); break;
            MM_LX_CASES(C)
#undef C
        }
    }
}

// Block fixed point takes the code for any row length, odd parts included, here: integer results do
// not depend on the instance, and its compiled lengths in one kernel with
// three layer counts took four minutes to build.
template <typename T, bool SEP>
__global__ void __launch_bounds__(YZBound<T>::v) k_yz_group(const GFilm<T> *films, const GItem *items,
                                                            const int *first_of, GActive A)
{
    MM_GROUP_LOOP(1)
    if (group_sep<T>(f.g) != SEP) continue;
    switch (f.g.Pz * 1024 + (is_fx<FA<T>> ? 0 : ly_of(f.g.Py))) {
#define C(L) case 1 * 1024 + L: yz_of<T, 1, L, SEP>(f.g, f.P, threadIdx.x, f.nth_yz, it.bx); break; \
             case 4 * 1024 + L: yz_of<T, 4, L, SEP>(f.g, f.P, threadIdx.x, f.nth_yz, it.bx); break; \
             case 8 * 1024 + L: yz_of<T, 8, L, SEP>(f.g, f.P, threadIdx.x, f.nth_yz, it.bx); break;
        MM_LY_CASES(C)
#undef C
    }
    }
}

template <typename T>
__global__ void __launch_bounds__(768) k_xinv_group(const GFilm<T> *films, const GItem *items, const int *first_of,
                                                    GActive A)
{
    MM_GROUP_LOOP(2)
        const int bid = it.by * f.gx_x + it.bx;
        switch (lx_of(f.g.Hx)) {
#define C(L) case L: xinv_body<T, FA<T>, MODE_MIN, L>(f.g, f.P, 0.0, 0.0, 0.0, 0, 0, threadIdx.x, f.nth_x, it.bx, it.by, \
                                                    bid, f.nblk_x); break;
            MM_LX_CASES(C)
#undef C
        }
    }
}

} // namespace

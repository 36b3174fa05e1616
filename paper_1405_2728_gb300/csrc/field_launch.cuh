// Host-side launchers of the field kernels for one precision (field type T,
// FFT arithmetic F), and the entry points each precision's translation unit
// exports: the three precisions are compiled in separate units so that the
// library builds in parallel.
#pragma once

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "fft.cuh"
#include "field_kernels.cuh"

namespace {

// ---------------------------------------------------------------------------
// host-side launch helpers
// ---------------------------------------------------------------------------
template <typename T, typename F, bool MIN>
cudaError_t launch_xfwd(const Geom &g, const FieldPtrs<T, F> &P, cudaStream_t s)
{
    const dim3 grid((g.ny + g.TYF - 1) / g.TYF, g.nz);
    const int thr = threads_xf<T>(g);
    const size_t sm = smem_xf_t<T>(g);
    switch (lx_of(g.Hx)) {
#define C(L) case L: k_xfwd<T, F, MIN, L><<<grid, thr, sm, s>>>(g, P); break;
        MM_LX_CASES(C)
#undef C
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename T, typename F, int MODE>
cudaError_t launch_xinv(const Geom &g, const FieldPtrs<T, F> &P, cudaStream_t s, const double *hext,
                        cudaGraphConditionalHandle h, int use_cond)
{
    const dim3 grid((g.ny + g.TY - 1) / g.TY, g.nz);
    const int thr = threads_x<T>(g);
    const size_t sm = smem_x_t<T>(g);
    const double h0 = hext ? hext[0] : 0.0, h1 = hext ? hext[1] : 0.0, h2 = hext ? hext[2] : 0.0;
    switch (lx_of(g.Hx)) {
#define C(L) case L: k_xinv<T, F, MODE, L><<<grid, thr, sm, s>>>(g, P, h0, h1, h2, h, use_cond); break;
        MM_LX_CASES(C)
#undef C
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// the film y-z kernel: float, or block fixed point (yz_fixed.cu), whose
// buffers and scales do not depend on the field type
template <int PZ> cudaError_t launch_yz(const Geom &g, const FieldPtrs<float> &P, cudaStream_t s)
{
    switch (ly_of(g.Py)) {
#define C(L) case L: k_yz<PZ, L><<<g.C, threads_yz<float>(g), smem_yz_t<float>(g), s>>>(g, P); break;
        MM_LY_CASES(C)
#undef C
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename T, typename F>
cudaError_t launch_yz_any(const Geom &g, const FieldPtrs<T, F> &P, cudaStream_t s)
{
    if constexpr (is_fx<F>) {
        FieldPtrs<double, fx> Q;
        memset((void *)&Q, 0, sizeof Q);
        Q.W = P.W; Q.Nhat = P.Nhat; Q.tw_py = P.tw_py;
        Q.fe1 = P.fe1; Q.fe2 = P.fe2; Q.fek = P.fek;
        return mm_yz_fixed(g, Q, s);
    } else {
        switch (g.Pz) {
        case 1: return launch_yz<1>(g, P, s);
        case 4: return launch_yz<4>(g, P, s);
        case 8: return launch_yz<8>(g, P, s);
        default: return cudaErrorInvalidValue;  // Pz = 2 does not occur (nz = 1 gives 1, nz = 2 gives 4)
        }
    }
}

// the bulk layout's passes exist for double and float (double-word problems
// are film-layout only: the planner refuses bulk grids for them)
template <typename T, typename F>
constexpr bool has_bulk = !std::is_same<T, dfloat>::value;

// the y-z stage: the film kernel, or the three passes of the bulk layout
template <typename T, typename F>
cudaError_t launch_conv(const Geom &g, const FieldPtrs<T, F> &P, cudaStream_t s)
{
    if constexpr (has_bulk<T, F>) {
        if (g.bulk) return mm_bulk_conv(g, P, s, -1);
    }
    return launch_yz_any<T, F>(g, P, s);
}

// dynamic shared memory limits of the instances this geometry launches
template <typename T, typename F> cudaError_t configure_t(const Geom &g, size_t sxf, size_t sx, size_t syz)
{
    cudaError_t e = cudaSuccess;
    switch (lx_of(g.Hx)) {
#define C(L)                                                                                     \
    case L:                                                                                      \
        if ((e = smem_attr(k_xfwd<T, F, false, L>, sxf)) || (e = smem_attr(k_xfwd<T, F, true, L>, sxf)) || \
            (e = smem_attr(k_xinv<T, F, MODE_HEFF, L>, sx)) || (e = smem_attr(k_xinv<T, F, MODE_ENERGY, L>, sx)) || \
            (e = smem_attr(k_xinv<T, F, MODE_MIN, L>, sx)))                                      \
            return e;                                                                            \
        break;
        MM_LX_CASES(C)
#undef C
    default: return cudaErrorInvalidValue;
    }
    if (g.bulk) return cudaSuccess;
    if constexpr (is_fx<F>) {
        return mm_yz_fixed_configure(g, syz);
    } else {
        switch (ly_of(g.Py)) {
#define C(L)                                                                                     \
    case L:                                                                                      \
        if (g.Pz == 1) return smem_attr(k_yz<1, L>, syz);                                        \
        if (g.Pz == 4) return smem_attr(k_yz<4, L>, syz);                                        \
        if (g.Pz == 8) return smem_attr(k_yz<8, L>, syz);                                        \
        return cudaErrorInvalidValue;
            MM_LY_CASES(C)
#undef C
        }
        return cudaErrorInvalidValue;
    }
}

// Launch-shape autotuner: time every admissible rows-per-tile of the
// x-forward kernel, every rows-per-batch RB of the y-z kernel, and every
// rows-per-tile of the x-inverse kernel (the three are independent: the spectrum
// layout does not depend on them), on this problem's own buffers (MM_TUNE_REPS
// repetitions, best taken: candidates within a few percent of each other
// otherwise swap places from run to run); keep the fastest of each.  The
// kernels run in their minimiser modes on a state past its first iteration, so
// that the step and the step-size sums are part of what is timed, and on a
// tilted unit field: the block fixed point's work depends on the values (of an
// all-zero row nothing is converted, and equal scales are not shifted).
#define MM_TUNE_REPS 5
template <typename T> __global__ void k_tune_field(T *m, long N)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
        const unsigned h = (unsigned)i * 2654435761u;   // a scrambled cell number: tilts up to 0.1
        const float y = (float)(h >> 16) * (0.2f / 65536.0f) - 0.1f, z = (float)(h & 0xffffu) * (0.2f / 65536.0f) - 0.1f;
        const float s = rsqrtf(1.0f + y * y + z * z);
        m[i] = T(s);
        m[N + i] = T(y * s);
        m[2 * N + i] = T(z * s);
    }
}
template <typename T, typename F> cudaError_t autotune_t(mm_problem *p, const int *tys, int nty, const int *rbs, int nrb,
                                             cudaStream_t s)
{
    Geom g = p->g;
    typedef typename io_of<T>::type IO;
    FieldPtrs<T, F> P = make_ptrs<T, F>(p);
    P.m_src = (const IO *)p->mbuf[0];
    P.H_out = (IO *)p->gbuf[0];
    cudaEvent_t a, b;
    cudaError_t e;
    MinState ms;
    memset(&ms, 0, sizeof ms);
    ms.k = 1;
    ms.tau = ms.tau0 = 1e-9;
    ms.tauf = 1e-9f;
    ms.tauw = dfloat(1e-9);
    ms.max_iter = 1L << 40;
    ms.status = MMS_RUNNING;
    // iterate 0 in mbuf[0], which the x-forward kernel steps from (with the zeroed gradient)
    k_tune_field<T><<<mm_grid_for(g.N, 256, 8), 256, 0, s>>>((T *)p->mbuf[0], g.N);
    if ((e = cudaGetLastError())) return e;
    if ((e = cudaMemcpyAsync(p->st, &ms, sizeof ms, cudaMemcpyHostToDevice, s)) || (e = cudaStreamSynchronize(s)))
        return e;
    if ((e = cudaEventCreate(&a))) return e;
    if ((e = cudaEventCreate(&b))) { cudaEventDestroy(a); return e; }
    // best of n candidates: set(i) takes one, before() runs untimed, run() is timed
    auto best_of = [&](int n, auto set, auto before, auto run) {
        float best = 1e30f;
        int at = 0;
        for (int i = 0; i < n && !e; ++i) {
            set(i);
            float tmin = 1e30f;
            for (int r = 0; r < MM_TUNE_REPS && !e; ++r) {
                if ((e = before())) break;
                cudaEventRecord(a, s);
                e = run();
                cudaEventRecord(b, s);
                if (e || (e = cudaEventSynchronize(b))) break;
                float t = 0;
                cudaEventElapsedTime(&t, a, b);
                if (t < tmin) tmin = t;
            }
            if (tmin < best) { best = tmin; at = i; }
        }
        set(at);
    };
    auto nothing = [] { return cudaSuccess; };
    auto xfwd = [&] { return launch_xfwd<T, F, true>(g, P, s); };
    best_of(nty, [&](int i) { g.TYF = tys[i]; g.ltyf = mm_ilog2(g.TYF); }, nothing, xfwd);
    if (!g.bulk) best_of(nrb, [&](int i) { g.RB = rbs[i]; }, xfwd, [&] { return launch_yz_any<T, F>(g, P, s); });
    // the x-inverse kernel after the others, as in an iteration: alone it finds its inputs in L2.  (512 x 256 x 4 double-word:
    // timed alone 4 rows won, 87 to 90 us in the iteration, where 1 or 2 take 85.)  Large grids, whose inputs do not fit there, run
    // the others once: an iteration of theirs takes milliseconds.
    auto others = [&] {
        const cudaError_t r = xfwd();
        return r ? r : launch_conv<T, F>(g, P, s);
    };
    const bool chain = g.N <= 1L << 20;
    if (!e) e = others();
    best_of(nty, [&](int i) { g.TY = tys[i]; g.lty = mm_ilog2(g.TY); }, [&] { return chain ? others() : cudaSuccess; },
            [&] { return launch_xinv<T, F, MODE_MIN>(g, P, s, nullptr, 0, 0); });
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    const size_t bytes = 3 * (size_t)g.N * p->esz;
    for (int i = 0; i < 2; ++i) {
        if (!e) e = cudaMemsetAsync(p->mbuf[i], 0, bytes, s);
        if (!e) e = cudaMemsetAsync(p->gbuf[i], 0, bytes, s);
    }
    if (!e) e = cudaMemsetAsync(p->st, 0, sizeof(MinState), s);
    if (!e) e = cudaMemsetAsync(p->counter, 0, 64, s);
    if (!e) p->g = g;
    return e;
}

// Field chain for MODE_HEFF / MODE_ENERGY on caller-provided m (and H).
template <typename T, typename F>
cudaError_t heff_chain_t(mm_problem *p, const void *m, void *H, const double *hext, int mode, cudaStream_t s,
                         double hscale)
{
    const Geom &g = p->g;
    typedef typename io_of<T>::type IO;
    FieldPtrs<T, F> P = make_ptrs<T, F>(p);
    P.m_src = (const IO *)m;
    P.H_out = (IO *)H;
    P.hscale = hscale;
    cudaError_t e = launch_xfwd<T, F, false>(g, P, s);
    if (e) return e;
    if ((e = launch_conv<T, F>(g, P, s))) return e;
    if (mode == MODE_HEFF) return launch_xinv<T, F, MODE_HEFF>(g, P, s, hext, 0, 0);
    return launch_xinv<T, F, MODE_ENERGY>(g, P, s, hext, 0, 0);
}

template <typename T, typename F>
cudaError_t min_body_t(mm_problem *p, cudaGraphConditionalHandle h, cudaStream_t s, int use_cond)
{
    const Geom &g = p->g;
    FieldPtrs<T, F> P = make_ptrs<T, F>(p);
    cudaError_t e = launch_xfwd<T, F, true>(g, P, s);
    if (e) return e;
    if ((e = launch_conv<T, F>(g, P, s))) return e;
    return launch_xinv<T, F, MODE_MIN>(g, P, s, nullptr, h, use_cond);
}

template <typename T, typename F>
cudaError_t stage_times_t(mm_problem *p, int reps, double *ms, cudaStream_t s)
{
    const Geom &g = p->g;
    FieldPtrs<T, F> P = make_ptrs<T, F>(p);
    const int nst = g.bulk ? 5 : 3;
    cudaEvent_t ev[6];
    for (int i = 0; i <= nst; ++i)
        if (cudaEventCreate(&ev[i])) return cudaGetLastError();
    double acc[5] = {0, 0, 0, 0, 0};
    cudaError_t e = cudaSuccess;
    for (int r = 0; r < reps && !e; ++r) {
        int i = 0;
        cudaEventRecord(ev[i++], s);
        launch_xfwd<T, F, true>(g, P, s);
        cudaEventRecord(ev[i++], s);
        if (g.bulk) {
            if constexpr (has_bulk<T, F>) {
                for (int pass = 0; pass < 3; ++pass) {
                    mm_bulk_conv(g, P, s, pass);
                    cudaEventRecord(ev[i++], s);
                }
            }
        } else {
            launch_yz_any<T, F>(g, P, s);
            cudaEventRecord(ev[i++], s);
        }
        launch_xinv<T, F, MODE_MIN>(g, P, s, nullptr, 0, 0);
        cudaEventRecord(ev[i++], s);
        if ((e = cudaGetLastError())) break;
        if ((e = cudaEventSynchronize(ev[nst]))) break;
        for (int k = 0; k < nst; ++k) {
            float t = 0;
            cudaEventElapsedTime(&t, ev[k], ev[k + 1]);
            acc[k] += t;
        }
    }
    for (int i = 0; i <= nst; ++i) cudaEventDestroy(ev[i]);
    for (int i = 0; i < nst; ++i) ms[i] = acc[i] / (reps > 0 ? reps : 1);
    return e;
}

} // namespace

// Entry points of one precision, defined by its translation unit with
// MM_DEFINE_FIELD_ENTRIES(suffix, T, F).
#define MM_DEFINE_FIELD_ENTRIES(SFX, T, F)                                                                     \
    cudaError_t mm_fields_configure_##SFX(const Geom &g, size_t sxf, size_t sx, size_t syz)                   \
    {                                                                                                          \
        return configure_t<T, F>(g, sxf, sx, syz);                                                             \
    }                                                                                                          \
    cudaError_t mm_fields_autotune_##SFX(mm_problem *p, const int *tys, int nty, const int *rbs, int nrb,       \
                                         cudaStream_t s)                                                       \
    {                                                                                                          \
        return autotune_t<T, F>(p, tys, nty, rbs, nrb, s);                                                     \
    }                                                                                                          \
    cudaError_t mm_fields_chain_##SFX(mm_problem *p, const void *m, void *H, const double *hext, int mode,     \
                                      cudaStream_t s, double hscale)                                          \
    {                                                                                                          \
        return heff_chain_t<T, F>(p, m, H, hext, mode, s, hscale);                                             \
    }                                                                                                          \
    cudaError_t mm_fields_min_body_##SFX(mm_problem *p, cudaGraphConditionalHandle h, cudaStream_t s,          \
                                         int use_cond)                                                         \
    {                                                                                                          \
        return min_body_t<T, F>(p, h, s, use_cond);                                                            \
    }                                                                                                          \
    cudaError_t mm_fields_stage_times_##SFX(mm_problem *p, int reps, double *ms, cudaStream_t s)              \
    {                                                                                                          \
        return stage_times_t<T, F>(p, reps, ms, s);                                                            \
    }

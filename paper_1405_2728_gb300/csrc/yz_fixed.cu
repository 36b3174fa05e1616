// The film y-z kernel in block fixed point (MM_FP64 and MM_F32X2), in a
// translation unit of its own: it does not depend on the field type.
#include "common.cuh"
#include "fft.cuh"
#include "field_kernels.cuh"

namespace {

// One layer never has all components coupled.  With more, a grid of one column or
// row or of very flat cells is the exception, and takes the code for any length.
template <int PZ> cudaError_t launch(const Geom &g, const FieldPtrs<double, fx> &P, cudaStream_t s)
{
    if (PZ > 1 && g.sep) {
        k_yz_fx<PZ, -1, true><<<g.C, threads_yz<double>(g), smem_yz_t<double>(g), s>>>(g, P);
        return cudaGetLastError();
    }
    switch (ly_of(g.Py)) {
#define C(L) case L: k_yz_fx<PZ, L, PZ == 1><<<g.C, threads_yz<double>(g), smem_yz_t<double>(g), s>>>(g, P); break;
        MM_LY_CASES(C)
#undef C
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int PZ> cudaError_t configure(const Geom &g, size_t smem)
{
    if (PZ > 1 && g.sep) return smem_attr(k_yz_fx<PZ, -1, true>, smem);
    switch (ly_of(g.Py)) {
#define C(L) case L: return smem_attr(k_yz_fx<PZ, L, PZ == 1>, smem);
        MM_LY_CASES(C)
#undef C
    }
    return cudaErrorInvalidValue;
}

} // namespace

// Pz = 2 does not occur (nz = 1 gives 1, nz = 2 gives 4)
cudaError_t mm_yz_fixed(const Geom &g, const FieldPtrs<double, fx> &P, cudaStream_t s)
{
    return g.Pz == 1 ? launch<1>(g, P, s) : (g.Pz == 4 ? launch<4>(g, P, s) : (g.Pz == 8 ? launch<8>(g, P, s) : cudaErrorInvalidValue));
}
cudaError_t mm_yz_fixed_configure(const Geom &g, size_t smem)
{
    return g.Pz == 1 ? configure<1>(g, smem) : (g.Pz == 4 ? configure<4>(g, smem) : (g.Pz == 8 ? configure<8>(g, smem) : cudaErrorInvalidValue));
}

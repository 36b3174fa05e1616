// Host build of the shared-memory layouts of the block fixed-point rows, of rows with an odd part and of the twiddle
// tables (csrc/fft.cuh), for tests/test_index_host_fixed.py; nothing here runs on a GPU.
#include "../paper_1405_2728_gb300/csrc/fft.cuh"

extern "C" {
int h_spos_fx(int i) { return spos<fxc>(i); }
int h_row_stride_fx(int L) { return row_stride_fx(L); }
int h_pidx(int i) { return pidx(i); }
int h_row_stride(int L, int esz) { return row_stride(L, esz); }
int h_tpos_fx(int t, int L) { return tpos<fxmc>(t, L); }
int h_tpos_float(int t, int L) { return tpos<float2>(t, L); }
int h_tw_slots(int n) { return tw_slots(n); }
// rpos of a float row of a kernel compiled for length L (-1: none is)
int h_rpos_float(int L, int i)
{
    switch (lb_of(L)) {
#define C(N) case N: return rpos<float2, N>(i);
        MM_LC_POW2(C) MM_LB_ODD(C)
#undef C
    }
    return -1;
}
int h_compiled(int L, int which) { return which == 0 ? lx_of(L) : (which == 1 ? ly_of(L) : lb_of(L)); }
}

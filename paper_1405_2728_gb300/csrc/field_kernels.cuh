// Field kernels of one H_eff evaluation (and of the minimiser iteration),
// written as device bodies parameterised by the CTA's coordinates and its
// number of working threads, plus the single-problem kernels that call them.
// Included by heff.cu (single problems) and batch.cu (grouped launches over
// many problems), so both run the same arithmetic.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "fft.cuh"

namespace {

template <typename T> __device__ __forceinline__ T ldg(const T *p) { return __ldg(p); }
template <> __device__ __forceinline__ dfloat ldg(const dfloat *p)
{
    const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
    return dfloat(v.x, v.y);
}
// complex loads through the read-only path (ld_nc) or cached in L2 only (ld_cg)
template <typename V> __device__ __forceinline__ V ld_nc(const V *p) { return __ldg(p); }
template <typename V> __device__ __forceinline__ V ld_cg(const V *p) { return __ldcg(p); }
template <> __device__ __forceinline__ fxc ld_nc(const fxc *p)
{
    const longlong2 v = __ldg(reinterpret_cast<const longlong2 *>(p));
    return fxc{fx(v.x), fx(v.y)};
}
template <> __device__ __forceinline__ fxc ld_cg(const fxc *p)
{
    const longlong2 v = __ldcg(reinterpret_cast<const longlong2 *>(p));
    return fxc{fx(v.x), fx(v.y)};
}
template <typename F> constexpr bool is_fx = std::is_same<F, fx>::value;
// a value of the FFT arithmetic F read back in the field type T
template <typename T, typename F> __device__ __forceinline__ T to_field(F v) { return (T)v; }
// a caller's value (double for double-word fields) in the field type T, and back
template <typename T> __device__ __forceinline__ T from_io(typename io_of<T>::type v) { return (T)v; }
template <typename T> __device__ __forceinline__ typename io_of<T>::type to_io(T v) { return v; }
template <> __device__ __forceinline__ double to_io<dfloat>(dfloat v) { return df_to_double(v); }
// 1/sqrt(x) in the field type (the double and float steps divide by sqrt)
template <typename T> __device__ __forceinline__ T inv_sqrt(T x) { return (T)1 / sqrt(x); }
template <> __device__ __forceinline__ dfloat inv_sqrt<dfloat>(dfloat x) { return df_rsqrt(x); }
// 1/|m| of the renormalisation after a midpoint step (float: the fast
// reciprocal square root, ~2 ulp; double-word: one Newton step, ~2^-47)
__device__ __forceinline__ float renorm_scale(float s) { return rsqrtf(s); }
__device__ __forceinline__ dfloat renorm_scale(dfloat s) { return df_rsqrt(s); }

// a product that is not contracted into a sum: the same rounded value wherever it is used
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ dfloat mul_rn(dfloat a, dfloat b) { return a * b; }

// ordered bits of |x|'s high part, at or above those of infinity if x is not finite
__device__ __forceinline__ int magnitude(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ int magnitude(dfloat x) { return __float_as_int(x.hi) & 0x7fffffff; }
__device__ __forceinline__ int magnitude(float) { return 0; }   // floats keep their own scale

// real element x of a padded complex row holding Px reals
// (of a kernel compiled for LC)
template <typename T, int LC, typename V> __device__ __forceinline__ T &rel(V *row, int x)
{
    return reinterpret_cast<T *>(row + rpos<V, LC>(x >> 1))[x & 1];
}

// Rows of a field [3][nz][ny][nx] copied asynchronously into shared memory:
// dst [3][nrows][nx] receives rows y = ylo .. ylo + nrows - 1 of plane z
// (rows outside 0..ny-1 are skipped) in 16-byte chunks (the planner checked
// that rows start on 16-byte boundaries).
template <typename T>
__device__ __forceinline__ void stage_rows(T *dst, const T *__restrict__ src, const Geom &g, int z, int ylo,
                                           int nrows, int tid, int nth)
{
    constexpr int CH = 16 / sizeof(T);
    const int nx = g.nx, nc = g.fd_nc.d;
    const int tot = 3 * nrows * nc;
    const long plane = (long)z * g.ny * nx;
    if (tid >= nth) return;
    for (int q = tid; q < tot; q += nth) {
        const int rr = g.fd_nc.div(q), ch = q - rr * nc;  // rr = c * nrows + r
        const int c = (rr >= nrows) + (rr >= 2 * nrows), r = rr - c * nrows, y = ylo + r;
        if (y < 0 || y >= g.ny) continue;
        cp_async16(dst + (long)rr * nx + ch * CH, src + c * g.N + plane + (long)y * nx + ch * CH);
    }
}

// byte offset of the staging area of k_xinv (after the FFT rows and the
// twiddles, 16-byte aligned); it holds (15 TY + 6) rows of nx values
template <typename T> __host__ __device__ __forceinline__ size_t stage_offset(const Geom &g)
{
    return ((size_t)(3 * g.TY * g.rsx + g.Px) * 2 * sizeof(T) + 15) & ~(size_t)15;
}

// ---------------------------------------------------------------------------
// k_xfwd
// ---------------------------------------------------------------------------
// The kernel bodies take the CTA's coordinates and its number of working
// threads nth as arguments: a single problem launches them with its own
// grid (nth = blockDim.x); a batch launches one grid over the work items of
// many problems with blockDim.x the largest nth, and the threads at or above
// a problem's nth only take part in the barriers.  Loops start at tt, the
// thread index, or past every bound for those idle threads.
#define MM_IDLE_START (1 << 30)
template <typename T, typename F, bool MIN, int LX>
__device__ __forceinline__ void xfwd_body(const Geom &g, const FieldPtrs<T, F> &P, const int tid, const int nth,
                                          const int bx, const int by)
{
    typedef typename cvec<F>::type V;
    typedef typename twvec<F>::type TW;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *S = reinterpret_cast<V *>(smem_raw);
    const int tt = tid < nth ? tid : MM_IDLE_START;
    const int TY = g.TYF, y0 = bx * TY, z = by;
    const int nx = g.nx, ny = g.ny, Px = g.Px;
    const long N = g.N;
    TW *tw = reinterpret_cast<TW *>(S + 3 * TY * g.rsx);  // Px twiddles exp(-2 pi i t / Px)
    for (int i = tt; i < Px; i += nth) tw[tpos<TW>(i, g.Hx)] = P.tw_px[i];
    __shared__ int s_max[3 * MM_MAX_TILE];   // block fixed point: high words of the rows' largest values
    if constexpr (is_fx<F>) {
        if (tid < 3 * TY) s_max[tid] = 0;
    }

    typedef typename io_of<T>::type IO;
    const T *src = nullptr;        // minimiser mode: the iterate buffers
    const IO *src_io = nullptr;    // otherwise the caller's m
    T *dst = nullptr;
    const T *gp = nullptr;
    T tau = 0;
    int step_kind = 0;
    if (MIN) {
        const MinState *st = P.st;
        const long k = st->k;
        const int cur = st->base ^ (int)(k & 1);
        if (k > 0) {
            src = cur ? P.mbuf[0] : P.mbuf[1];
            dst = cur ? P.mbuf[1] : P.mbuf[0];
            gp = ((k - 1) & 1) ? P.gbuf[1] : P.gbuf[0];
            tau = pick<T>(st->tau, st->tauf, st->tauw);
            step_kind = st->step_kind;
        } else {
            src = cur ? P.mbuf[1] : P.mbuf[0];
        }
    } else {
        src_io = P.m_src;
    }
    // load (and step) the tile; row (c, yl) holds Px reals
#pragma unroll(sizeof(T) == 4 ? 2 : 1)
    for (int e = tt; e < TY * nx; e += nth) {
        const int yl = g.fd_nx.div(e), x = e - yl * nx, y = y0 + yl;
        T m0 = 0, m1 = 0, m2 = 0;
        if (y < ny) {
            const long n = ((long)z * ny + y) * nx + x;
            if constexpr (MIN) {
                m0 = ldg(src + n); m1 = ldg(src + N + n); m2 = ldg(src + 2 * N + n);
            } else {
                m0 = from_io<T>(ldg(src_io + n)); m1 = from_io<T>(ldg(src_io + N + n));
                m2 = from_io<T>(ldg(src_io + 2 * N + n));
            }
            if (MIN && dst) {
                const T g0 = ldg(gp + n), g1 = ldg(gp + N + n), g2 = ldg(gp + 2 * N + n);
                if (step_kind == MM_STEP_CAYLEY) {
                    const T q = (T)0.25 * tau * tau * (g0 * g0 + g1 * g1 + g2 * g2);
                    const T a = (T)1 - q, inv = (T)1 / ((T)1 + q);
                    m0 = (a * m0 - tau * g0) * inv;
                    m1 = (a * m1 - tau * g1) * inv;
                    m2 = (a * m2 - tau * g2) * inv;
                    if constexpr (!std::is_same<T, double>::value) {
                        // the closed form keeps |m| = 1 exactly in exact arithmetic;
                        // its rounding drifts ~1e-7 per step in float and ~1e-14 in
                        // double-word arithmetic, so those paths renormalise (the
                        // double path keeps the pure midpoint form, ~1e-16 per step)
                        const T r = renorm_scale(m0 * m0 + m1 * m1 + m2 * m2);
                        m0 *= r; m1 *= r; m2 *= r;
                    }
                } else {
                    m0 -= tau * g0; m1 -= tau * g1; m2 -= tau * g2;
                    const T inv = inv_sqrt(m0 * m0 + m1 * m1 + m2 * m2);
                    m0 *= inv; m1 *= inv; m2 *= inv;
                }
                dst[n] = m0; dst[N + n] = m1; dst[2 * N + n] = m2;
            }
        }
        if constexpr (is_fx<F>) {  // as they are, until the rows' scales are known
            rel<T, LX>(S + (0 * TY + yl) * g.rsx, x) = m0;
            rel<T, LX>(S + (1 * TY + yl) * g.rsx, x) = m1;
            rel<T, LX>(S + (2 * TY + yl) * g.rsx, x) = m2;
        } else {
            rel<F, LX>(S + (0 * TY + yl) * g.rsx, x) = F(m0);
            rel<F, LX>(S + (1 * TY + yl) * g.rsx, x) = F(m1);
            rel<F, LX>(S + (2 * TY + yl) * g.rsx, x) = F(m2);
        }
    }
    int e1 = 0;
    if constexpr (is_fx<F>) {
        // The scale 2^s of a row's three components, or with Geom::sep of each: the largest value becomes 2^57 .. 2^58
        // (one up to 1 + 2^-8 counts as 1, so that unit vectors and their rounding share one scale); non-finite
        // components are taken as zero and flagged.  By row, because the tile is chosen by timing and results must not
        // depend on it.  The Gx threads that transform a row convert it.
        constexpr bool DW = std::is_same<T, dfloat>::value;
        constexpr int inf = DW ? 0x7f800000 : 0x7ff00000, mant = DW ? 23 : 20, bias = DW ? 126 : 1022;
        __syncthreads();
        const int row = tid / g.Gx, j = tid - row * g.Gx;
        const bool act = row < 3 * TY;
        V *const R = S + row * g.rsx;
        int top = 0;
        if (act) {
            for (int x = j; x < nx; x += g.Gx) top = max(top, magnitude(rel<T, LX>(R, x)));
            if (top) atomicMax(&s_max[row], top);
        }
        __syncthreads();
        if (act) {
            auto finite = [&](int t) { return t < inf ? t : 0; };
            const int own = s_max[row], yl = row & (TY - 1);
            int all = own;   // the largest of those that share the scale, finite or not
            top = finite(own);
            if (!g.sep) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    all = max(all, s_max[c * TY + yl]);
                    top = max(top, finite(s_max[c * TY + yl]));
                }
            }
            const int top_e = ((top - (1 << (mant - 8))) >> mant) - bias, sc = min(58 - top_e, DW ? 150 : 1000);
            e1 = fx_pack(top > 0 ? -sc - 1 : FX_ZERO, all < inf ? 0 : 1);
            const float scalef = DW ? fx_pow2f(sc - 28) : 0.0f;
            const bool use = top > 0 && own < inf;
            for (int x = j; x < nx; x += g.Gx) {
                const T a = rel<T, LX>(R, x);
                fx q(0);
                if (use) {
                    if constexpr (DW) q = fx_from(a, scalef);
                    else q = fx(__double2ll_rn(fx_ldexp(a, sc)));
                }
                rel<fx, LX>(R, x) = q;
            }
        }
    }
    const int npad = Px - nx;
    for (int e = tt; e < 3 * TY * npad; e += nth) {
        const int row = g.fd_padx.div(e), x = nx + (e - row * npad);
        rel<F, LX>(S + row * g.rsx, x) = F(0);
    }
    __syncthreads();

    // complex FFT of length Hx of the packed rows (upper half zero)
    {
        const int row = tid / g.Gx, j = tid - row * g.Gx;
        const bool act = row < 3 * TY;
        if constexpr (is_fx<F>) {
            unsigned none = 0;
            const int sh = fft_row_fx<false, true, false, 2, LX, false>(S + (act ? row : 0) * g.rsx, g.Hx, g.lhx, j,
                                                                        tw, act, 0, 64, none);
            const int c = row >> g.ltyf, y = y0 + (row & (TY - 1));
            if (act && j == 0 && y < ny && (c == 0 || g.sep)) P.fe1[(z * ny + y) * (g.sep ? 3 : 1) + c] = e1 + fx_pack(sh, 0);
        } else {
            fft_row<false, true, false, 2, LX>(S + (act ? row : 0) * g.rsx, g.Hx, g.lhx, j, tw, act);
        }
    }

    // unpack to the real-input spectrum X[k], k = 0..Hx, and store transposed.
    // With sum = Z[k] + Z*[Hx-k], dif = Z[k] - Z*[Hx-k] and w = exp(-2 pi i k / Px):
    // X[k] = (sum - i w dif) / 2 and, from the same two values (w^Hx = -1),
    // X[Hx-k] = (sum* - i (w dif)*) / 2; one item per pair k = 0..Hx/2.
    const int Hx = g.Hx, hh = Hx >> 1;
    for (int e = tt; e < TY * 3 * (hh + 1); e += nth) {
        const int c = e % 3, rest = e / 3, yl = rest & (TY - 1), k = rest >> g.ltyf;
        const int y = y0 + yl;
        const V *row = S + (c * TY + yl) * g.rsx;
        const V Zk = row[rpos<V, LX>(k)];
        const V Zm = cconj(row[rpos<V, LX>(k == 0 ? 0 : Hx - k)]);
        if constexpr (is_fx<F>) {  // 2 X is stored: |Zk|, |Zm| < 2^60.5, so |2 X| < 2^62
            const V sum = cadd(Zk, Zm), wd = fx_cmul<false>(csub(Zk, Zm), tw[tpos<TW>(k, g.Hx)], 0);
            if (y < ny) {
                P.W[(((long)k * g.nz + z) * ny + y) * 3 + c] = V{sum.x + wd.y, sum.y - wd.x};
                if (Hx - k != k)
                    P.W[(((long)(Hx - k) * g.nz + z) * ny + y) * 3 + c] = V{sum.x - wd.y, -(sum.y + wd.x)};
            }
            continue;
        } else {
        const V sum = cadd(Zk, Zm), dif = csub(Zk, Zm);
        const V wd = cmul(tw[tpos<TW>(k, g.Hx)], dif);
        if (y < ny) {
            V X;
            X.x = F(0.5) * (sum.x + wd.y);
            X.y = F(0.5) * (sum.y - wd.x);
            P.W[(((long)k * g.nz + z) * ny + y) * 3 + c] = X;
            if (Hx - k != k) {
                X.x = F(0.5) * (sum.x - wd.y);
                X.y = F(0.5) * (-sum.y - wd.x);
                P.W[(((long)(Hx - k) * g.nz + z) * ny + y) * 3 + c] = X;
            }
        }
        }
    }
}

template <typename T, typename F, bool MIN, int LX>
__global__ void __launch_bounds__(768) k_xfwd(Geom g, FieldPtrs<T, F> P)
{
    xfwd_body<T, F, MIN, LX>(g, P, threadIdx.x, blockDim.x, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------------------
// k_yz
// ---------------------------------------------------------------------------
// The fixed-point kernel runs fewer, fatter threads (128 registers, two CTAs an
// SM); the y rows are then transformed in batches of RB rows.  384 threads of
// 80 registers took 156 us at 512 x 256 x 4 where 256 took 141: the z
// convolution then keeps too few coefficients in flight.
template <typename T> struct YZBound { static constexpr int v = sizeof(T) == 8 ? 256 : 768; };

// Block fixed point: the z convolution of one (kx, ky), NZM layers.  The
// tensor's xz and yz transforms are imaginary, so with i m_z in the place of
// m_z and -i H_z in that of H_z its matrix is real,
//   [xx xy xz; xy yy yz; xz yz -zz],
// and the real and the imaginary part are convolved apart, by two threads: half
// the values and sums a thread, within the 128 registers that two CTAs of 256
// threads (16 warps an SM) leave.
// Along z the tensor is a Toeplitz matrix, even (xx, yy, zz, xy) or odd (xz,
// yz) in z - z', so with up_j = m_j + m_{NZM-1-j} and um_j = m_j - m_{NZM-1-j} the
// sums S_i and differences D_i of the outputs i and NZM-1-i come from half-size
// products: 8 multiplications a component pair for 4 layers instead of 16
// (even) or 12 (odd).  Outputs carry a factor 2 for NZM > 1.
// The coefficients, combinations of the tensor at the z offsets K0 .. K3, are
// stored [coefficient][ky], 4 NE + 2 NO of them (k_tensor_fixed):
//  even  S: [K0+K3 K1+K2; K1+K2 K0+K1] up,  D: the same with minus, um
//  odd   S: [K3 K2-K1; K1+K2 K1] um,        D: [-K3 -(K1+K2); K1-K2 -K1] up
// so that each is loaded where it is used.
template <int NZM> struct ZConv {
    static constexpr int H = NZM > 1 ? NZM / 2 : 1;
    static constexpr int NE = NZM == 1 ? 1 : (NZM == 2 ? 2 : 6), NO = NZM == 1 ? 0 : (NZM == 2 ? 1 : 4);
    int2 up[3][H], um[3][H];   // split words, [component][j]
    const fxm *K;              // this (kx, ky)'s first coefficient
    int kst;

    // n coefficients from the table's index `first`
    template <int N> __device__ __forceinline__ void load(fxm (&k)[N], int first) const
    {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int2 w = __ldg(reinterpret_cast<const int2 *>(K + (long)(first + i) * kst));
            k[i] = fxm{w.x, w.y};
        }
    }
    // an even component's coefficients k from source b, into S_i (D false) or D_i
    template <bool D> __device__ __forceinline__ void even(fxdot &a, const fxm (&k)[NE], bool neg, int b, int i) const
    {
#pragma unroll
        for (int j = 0; j < H; ++j)
            a.mad(D ? um[b][j] : up[b][j], fxk(fxk(k[NZM == 1 ? 0 : (NZM == 2 ? D : (D ? 3 : 0) + i + j)]), neg));
    }
    // an odd one's
    template <bool D> __device__ __forceinline__ void odd(fxdot &a, const fxm (&k)[NO ? NO : 1], int b, int i) const
    {
        if constexpr (NZM > 1) {
#pragma unroll
            for (int j = 0; j < H; ++j) {
                // NZM = 4: rows (K3, -(K1-K2)), (K1+K2, K1) of S; (-K3, -(K1+K2)), (K1-K2, -K1) of D
                const int at = NZM == 2 ? 0 : (i == j ? 3 * i : (D ? 1 + j : 2 - j));
                const bool neg = NZM == 2 ? D : (D ? !(i == 1 && j == 0) : (i == 0 && j == 1));
                a.mad(D ? up[b][j] : um[b][j], fxk(fxk(k[at]), neg));
            }
        }
    }
    // outputs of component comp from two components of one parity and one of the other: store(layer, value).  Their
    // coefficients are loaded together: the loads come from L2, and one at a time they would be waited for.
    template <int COMP, typename St> __device__ __forceinline__ void output(St store) const
    {
        constexpr int XZ = 4 * NE, YZ = 4 * NE + NO;
        fxm e0[NE], e1[NE], o0[NO ? NO : 1], o1[NO ? NO : 1];
        if constexpr (COMP == 0) { load(e0, 0); load(e1, 3 * NE); if constexpr (NO > 0) load(o0, XZ); }
        if constexpr (COMP == 1) { load(e0, 3 * NE); load(e1, NE); if constexpr (NO > 0) load(o0, YZ); }
        if constexpr (COMP == 2) { load(e0, 2 * NE); if constexpr (NO > 0) { load(o0, XZ); load(o1, YZ); } }
#pragma unroll
        for (int i = 0; i < H; ++i) {
            fx sd[2];
#pragma unroll
            for (int w = 0; w < (NZM > 1 ? 2 : 1); ++w) {
                fxdot t;
                t.zero();
                auto add = [&](auto D) {
                    if constexpr (COMP < 2) {
                        even<D.value>(t, e0, false, 0, i);
                        even<D.value>(t, e1, false, 1, i);
                        odd<D.value>(t, o0, 2, i);
                    } else {
                        odd<D.value>(t, o0, 0, i);
                        odd<D.value>(t, o1, 1, i);
                        even<D.value>(t, e0, true, 2, i);
                    }
                };
                if (w) add(std::true_type()); else add(std::false_type());
                sd[w] = t.value();
            }
            if constexpr (NZM == 1) {
                store(0, sd[0]);
            } else {
                store(i, sd[0] + sd[1]);
                store(NZM - 1 - i, sd[0] - sd[1]);
            }
        }
    }
};

// The same stage in block fixed point (F = fx), one scale per x-frequency, or
// with SEP one per x-frequency and component.  The plane is brought to full
// magnitude when it is loaded, before the inverse transform and when it is
// stored; the z convolution, where the tensor scales each frequency differently,
// has a scale per ky, which components that the tensor couples share.
template <int PZ, int LY, bool SEP>
__device__ __forceinline__ void yz_body_fx(const Geom &g, const FieldPtrs<double, fx> &P, const int tid, const int nth,
                                           const int kx)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fxc *S = reinterpret_cast<fxc *>(smem_raw);
    constexpr int NS = SEP ? 3 : 1;
    __shared__ int s_e[NS], s_top[NS];
    // magnitudes in and out, sums of the frequencies' scales over the largest, flags
    __shared__ unsigned s_r[3 * NS + 1];
    unsigned *s_in = s_r, *s_out = s_r + NS, *s_sum = s_r + 2 * NS, *s_fl = s_r + 3 * NS;
    const int tt = tid < nth ? tid : MM_IDLE_START;
    const int ny = g.ny, nz = g.nz, Py = g.Py, nrow = 3 * nz;
    fxc *Wk = P.W + (long)kx * nrow * ny;
    fxmc *tw = reinterpret_cast<fxmc *>(S + nrow * g.rsy);
    signed char *s_sc = reinterpret_cast<signed char *>(tw + Py);  // [2][NS][Py]: scale and top bit of every ky
    load_twiddles_async(tw, P.tw_py, Py, Py, tt, nth);
    if (tid < NS) { s_e[tid] = FX_ZERO; s_top[tid] = FX_ZERO; }
    if (tid < 3 * NS + 1) s_r[tid] = 0;
    __syncthreads();

    // Wk[z][y][c] -> row (c, z); the first loads are issued before the rows' scales are looked at
    constexpr int PF = LY == 0 ? 2 : 4;   // (short rows: fewer instructions to fetch)
    const int tot = nrow * ny;
    fxc v[PF];
    auto load = [&](int e0) {
#pragma unroll
        for (int i = 0; i < PF; ++i)
            if (e0 + i * nth < tot) v[i] = ld_cg(Wk + e0 + i * nth);
    };
    if (tt < tot) load(tt);
    fx_cta_scales<NS>(P.fe1, nz * ny, NS, tt, nth, s_e, s_fl);
    __syncthreads();
    FxMags<NS> mags;
    for (int e0 = tt; e0 < tot;) {
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int e = e0 + i * nth;
            if (e >= tot) break;
            const int c = e % 3, rest = e / 3, zz = g.fd_ny.div(rest), y = rest - zz * ny;
            v[i] = fx_down(v[i], s_e[SEP ? c : 0] - fx_exp(P.fe1[SEP ? e : rest]));
            mags.or_in(c, fx_mag(v[i]));
            S[(c * nz + zz) * g.rsy + spos<fxc>(y)] = v[i];
        }
        e0 += PF * nth;
        if (e0 < tot) load(e0);
    }
    mags.cta_or(s_in);
    const int npad = Py - ny;
    for (int e = tt; e < nrow * npad; e += nth) {
        const int row = g.fd_pady.div(e), y = ny + (e - row * npad);
        S[row * g.rsy + spos<fxc>(y)] = czero<fxc>();
    }
    cp_async_wait_all();
    __syncthreads();
    const int rb = tid / g.Gy, j = tid - rb * g.Gy;  // row within a batch of g.RB rows
    const bool act = rb < g.RB;
    auto comp = [&](int r) { return SEP ? (r >= nz) + (r >= 2 * nz) : 0; };  // of a row
    int sh = 0, pre[NS];
#pragma unroll
    for (int c = 0; c < NS; ++c) pre[c] = 59 - fx_bits(s_in[c]);
    unsigned none = 0;
    for (int r0 = 0; r0 < nrow; r0 += g.RB) {
        const int r = act ? r0 + rb : 0;
        sh = fft_row_fx<false, true, false, 1, LY, false>(S + r * g.rsy, Py, g.lpy, j, tw, act, fx_of(pre, comp(r)), 64,
                                                          none);
    }
    // z convolution: inputs of a ky below 2^59, so sums and differences below
    // 2^60; outputs below 2^60 (the tensor's terms of an output sum to less
    // than 2^62 units, and the factor 2)
    constexpr int NZM = PZ > 1 ? PZ / 2 : 1;
    const int hy = Py / 2, kst = hy + 1;
    constexpr int NC = 4 * ZConv<NZM>::NE + 2 * ZConv<NZM>::NO;
    const FxCouple couple{g.nx > 1 && ny > 1, NZM > 1 && g.nx > 1, NZM > 1 && ny > 1};
    int eb[NS], d[NS], top[NS];   // a component's scale where it is mixed, its own over that, the largest output
#pragma unroll
    for (int c = 0; c < NS; ++c) {
        eb[c] = d[c] = s_e[c] - pre[c] + sh + (SEP ? g.tsc[c] : 0);
        top[c] = FX_ZERO;
    }
    couple.join(eb);
#pragma unroll
    for (int c = 0; c < NS; ++c) d[c] -= eb[c];
    for (int u = tt; u < 2 * Py; u += nth) {
        // a pair of lanes per ky: part 0 the real parts (of m_x, m_y and i m_z), part 1 the imaginary ones
        const int ky = u >> 1, part = u & 1, kyr = ky <= hy ? ky : Py - ky;
        const int left = 2 * Py - (u & ~31);
        const unsigned lanes = left >= 32 ? 0xffffffffu : (1u << left) - 1;
        fx *col = &S[spos<fxc>(ky)].x;                 // this ky's column; rows are 2 g.rsy values apart
        const int at[3] = {part, part, 1 - part};      // where the part lies in a component's complex value
        const bool flip[3] = {false, ky > hy, part == 0};  // xy and yz are odd in ky; i m_z and -i H_z
        ZConv<NZM> z;
        z.K = P.Nhat + (long)kx * NC * kst + kyr;
        z.kst = kst;
        int sc[NS];
        {
            fx m[3][NZM];
            FxMags<NS> mk;
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int n = 0; n < NZM; ++n) {
                    m[c][n] = n < nz ? col[2 * (c * nz + n) * g.rsy + at[c]] : fx(0);
                    mk.or_in(c, fx_mag(m[c][n]));
                }
#pragma unroll
            for (int c = 0; c < NS; ++c) sc[c] = fx_bits(mk.v[c] | __shfl_xor_sync(lanes, mk.v[c], 1)) + d[c];
            couple.join(sc);
#pragma unroll
            for (int c = 0; c < NS; ++c) sc[c] = 59 - sc[c];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
#pragma unroll
                for (int n = 0; n < NZM; ++n) {
                    m[c][n] = fx_scale(m[c][n], sc[SEP ? c : 0] + d[SEP ? c : 0]);
                    if (flip[c]) m[c][n] = -m[c][n];
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int i = 0; i < ZConv<NZM>::H; ++i) {
                    const fx a = m[c][i], b = m[c][NZM - 1 - i];
                    z.up[c][i] = fx_split(NZM > 1 ? a + b : a);
                    z.um[c][i] = fx_split(a - b);
                }
        }
        unsigned mag = 0;
        auto put = [&](int c, int n, fx r) {
            if (n >= nz) return;
            if (c == 1 ? flip[1] : (c == 2 && part == 1)) r = -r;
            mag |= fx_mag(r);
            col[2 * (c * nz + n) * g.rsy + at[c]] = r;
        };
        auto done = [&](int c) {
            // values of this ky and component: stored * 2^-sc, below 2^tk
            const int tk = fx_bits(mag | __shfl_xor_sync(lanes, mag, 1)) - sc[c];
            if (part == 0) {
                s_sc[c * Py + ky] = (signed char)sc[c];
                s_sc[(NS + c) * Py + ky] = (signed char)tk;
            }
            top[c] = max(top[c], tk);
            mag = 0;
        };
        z.template output<0>([&](int n, fx r) { put(0, n, r); });
        if (SEP) done(0);
        z.template output<1>([&](int n, fx r) { put(1, n, r); });
        if (SEP) done(SEP ? 1 : 0);
        z.template output<2>([&](int n, fx r) { put(2, n, r); });
        done(SEP ? 2 : 0);
    }
#pragma unroll
    for (int c = 0; c < NS; ++c) fx_cta_max(&s_top[c], top[c]);
    __syncthreads();
    // no partial sum of an inverse transform exceeds the sum of the largest moduli over ky
    unsigned sum[NS];
#pragma unroll
    for (int c = 0; c < NS; ++c) sum[c] = 0;
    for (int ky = tt; ky < Py; ky += nth) {
#pragma unroll
        for (int c = 0; c < NS; ++c) sum[c] += ((1u << 18) >> min(s_top[c] - s_sc[(NS + c) * Py + ky], 18)) + 1;
    }
#pragma unroll
    for (int c = 0; c < NS; ++c) fx_cta_add(&s_sum[c], sum[c]);
    __syncthreads();
    int t[NS], post[NS];
#pragma unroll
    for (int c = 0; c < NS; ++c) {
        pre[c] = 58 - s_top[c];
        t[c] = max(0, fx_log2_up(s_sum[c]) - 18);
    }
    mags = FxMags<NS>();
    for (int r0 = 0; r0 < nrow; r0 += g.RB) {
        const int r = act ? r0 + rb : 0, c = comp(r);
        unsigned mag = 0;
        fft_row_fx<true, false, true, 1, LY, true, true>(S + r * g.rsy, Py, g.lpy, j, tw, act, fx_of(pre, c), fx_of(t, c),
                                                         mag, s_sc + c * Py);
        mags.or_in(c, mag);
    }
    mags.cta_or(s_out);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NS; ++c) post[c] = 60 - fx_bits(s_out[c]);
    for (int i = tt; i < tot; i += nth) {
        const int c = i % 3, rest = i / 3, zz = g.fd_ny.div(rest), y = rest - zz * ny;
        Wk[i] = fx_scale(S[(c * nz + zz) * g.rsy + spos<fxc>(y)], fx_of(post, c));
    }
    if (tid < NS) {
        // with one layer the field along z depends on m_z alone, the others on m_x and m_y alone
        const int c = tid, fl = (int)*s_fl, hit = nz > 1 ? 7 : (c == 2 ? 4 : 3);
        const int e = fx_of(eb, c) + P.fek[kx] - (NZM > 1 ? 1 : 0) + fx_cum(fx_log(Py), fx_of(t, c)) - fx_of(pre, c) -
                      fx_of(post, c) + (SEP ? g.tsc[c] : 0);
        P.fe2[kx * NS + c] = fx_pack(e, (SEP ? fl & hit : fl) ? 1 : 0);
    }
}

template <int PZ, int LY>
__device__ __forceinline__ void yz_body(const Geom &g, const FieldPtrs<float> &P, const int tid, const int nth,
                                        const int kx)
{
    typedef float F;
    typedef float2 V;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *S = reinterpret_cast<V *>(smem_raw);
    const int tt = tid < nth ? tid : MM_IDLE_START;
    const int ny = g.ny, nz = g.nz, Py = g.Py;
    const int nrow = 3 * nz;
    V *Wk = P.W + (long)kx * nrow * ny;
    V *tw = S + nrow * g.rsy;
    load_twiddles_async(tw, P.tw_py, Py, Py, tt, nth);

    // Wk[z][y][c] -> row (c, z); PF loads per thread in flight before use
    constexpr int PF = 8;
    const int tot = nrow * ny;
    for (int e0 = tt; e0 < tot; e0 += PF * nth) {
        V v[PF];
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int e = e0 + i * nth;
            if (e < tot) v[i] = ld_cg(Wk + e);
        }
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int e = e0 + i * nth;
            if (e >= tot) break;
            const int c = e % 3, rest = e / 3, zz = g.fd_ny.div(rest), y = rest - zz * ny;
            S[(c * nz + zz) * g.rsy + rpos<V, LY>(y)] = v[i];
        }
    }
    const int npad = Py - ny;
    for (int e = tt; e < nrow * npad; e += nth) {
        const int row = g.fd_pady.div(e), y = ny + (e - row * npad);
        S[row * g.rsy + rpos<V, LY>(y)] = czero<V>();
    }
    cp_async_wait_all();
    __syncthreads();
    const int rb = tid / g.Gy, j = tid - rb * g.Gy;  // row within a batch of g.RB rows
    const bool act = rb < g.RB;
    for (int r0 = 0; r0 < nrow; r0 += g.RB)
        fft_row<false, true, false, 1, LY>(S + (act ? r0 + rb : 0) * g.rsy, Py, g.lpy, j, tw, act);

    // per ky: the z direction as a direct convolution (films have nz <= 4).
    // With the tensor transformed along x and y only, K(kx, ky, dz), the
    // field is H^_a(z) = sum_b sum_z' K_ab(z - z') m^_b(z') -- the same sums
    // the zero-padded z-FFT, product and inverse z-FFT would form, in fewer
    // operations and with no twiddles.  K_xx, K_yy, K_zz, K_xy are real and
    // even in dz, K_xz and K_yz imaginary and odd in dz (and zero at dz = 0);
    // K_xy, K_yz are odd in ky.  Stored for dz = 0 .. NZM-1 (zero beyond
    // nz - 1, so that every load is unconditional) as
    // [kx][dz][component][ky <= Py/2], scaled by -Ms/(Px Py).
    constexpr int NZM = PZ > 1 ? PZ / 2 : 1;  // nz <= NZM
    const int hy = Py / 2, kst = hy + 1;
    const F *Kk = P.Nhat + (long)kx * NZM * 6 * kst;
    for (int ky = tt; ky < Py; ky += nth) {
        const int pky = rpos<V, LY>(ky);
        const int kyr = ky <= hy ? ky : Py - ky;
        const bool flip = ky > hy;
        V mz[3][NZM], hz[3][NZM];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int n = 0; n < NZM; ++n) {
                mz[c][n] = (n < nz) ? S[(c * nz + n) * g.rsy + pky] : czero<V>();
                hz[c][n] = czero<V>();
            }
#pragma unroll
        for (int dz = 0; dz < NZM; ++dz) {
            const F *kd = Kk + (long)dz * 6 * kst + kyr;
            const F kxx = ldg(kd), kyy = ldg(kd + kst), kzz = ldg(kd + 2 * kst);
            const F kxy0 = ldg(kd + 3 * kst), kxz = ldg(kd + 4 * kst), kyz0 = ldg(kd + 5 * kst);
            const F kxy = flip ? -kxy0 : kxy0, kyz = flip ? -kyz0 : kyz0;
#pragma unroll
            for (int z = 0; z < NZM; ++z)
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    // source z' = z - dz (side 0) or z + dz (side 1); K(z - z') of the
                    // odd components is +K(dz) for z' < z and -K(dz) for z' > z
                    if (side == 1 && dz == 0) continue;
                    const int zp = side ? z + dz : z - dz;
                    if (zp < 0 || zp >= NZM) continue;
                    const V a = mz[0][zp], b = mz[1][zp], c = mz[2][zp];
                    hz[0][z].x += kxx * a.x + kxy * b.x; hz[0][z].y += kxx * a.y + kxy * b.y;
                    hz[1][z].x += kxy * a.x + kyy * b.x; hz[1][z].y += kxy * a.y + kyy * b.y;
                    hz[2][z].x += kzz * c.x;             hz[2][z].y += kzz * c.y;
                    if (dz > 0) {  // i * (+-k) * m = (-+k m.y, +-k m.x)
                        const F sxz = side ? -kxz : kxz, syz = side ? -kyz : kyz;
                        hz[0][z].x -= sxz * c.y;             hz[0][z].y += sxz * c.x;
                        hz[1][z].x -= syz * c.y;             hz[1][z].y += syz * c.x;
                        hz[2][z].x -= sxz * a.y + syz * b.y; hz[2][z].y += sxz * a.x + syz * b.x;
                    }
                }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int zz = 0; zz < NZM; ++zz)
                if (zz < nz) S[(c * nz + zz) * g.rsy + pky] = hz[c][zz];
    }
    __syncthreads();
    for (int r0 = 0; r0 < nrow; r0 += g.RB)
        fft_row<true, false, true, 1, LY>(S + (act ? r0 + rb : 0) * g.rsy, Py, g.lpy, j, tw, act);

    for (int e = tt; e < nrow * ny; e += nth) {
        const int c = e % 3, rest = e / 3, zz = g.fd_ny.div(rest), y = rest - zz * ny;
        Wk[e] = S[(c * nz + zz) * g.rsy + rpos<V, LY>(y)];
    }
}

template <int PZ, int LY>
__global__ void __launch_bounds__(YZBound<float>::v, 1) k_yz(Geom g, FieldPtrs<float> P)
{
    yz_body<PZ, LY>(g, P, threadIdx.x, blockDim.x, blockIdx.x);
}

template <int PZ, int LY, bool SEP>
__global__ void __launch_bounds__(YZBound<double>::v, 2) k_yz_fx(Geom g, FieldPtrs<double, fx> P)
{
    yz_body_fx<PZ, LY, SEP>(g, P, threadIdx.x, blockDim.x, blockIdx.x);
}

// ---------------------------------------------------------------------------
// reductions
// ---------------------------------------------------------------------------
// Slots of the per-CTA partial sums.  In MODE_MIN: s.s, s.y, y.y,
// max |m x H|^2, energy density sum, sum m.  In MODE_ENERGY: m.H_demag,
// m.H_exchange, K(1 - (m.u)^2), m.H_ext, -, sum m.
enum { SL_SS = 0, SL_SY = 1, SL_YY = 2, SL_T2 = 3, SL_ET = 4, SL_MX = 5, SL_MY = 6, SL_MZ = 7, NSL = 8 };
enum { SL_ED = 0, SL_EEX = 1, SL_EAN = 2, SL_EZ = 3 };
static_assert(NSL <= RED_NSLOT, "partials buffer holds RED_NSLOT doubles per CTA");
static_assert(NSL % 2 == 0 && RED_NSLOT % 2 == 0, "the last CTA reads the partials in 16-byte pairs");

// accumulator: double on the double path, a compensated float pair on the float path
template <typename T> struct Acc;
template <> struct Acc<double> {
    double v;
    __device__ __forceinline__ void zero() { v = 0.0; }
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void add_prod(double a, double b) { v += a * b; }
    __device__ __forceinline__ void add(const Acc &o) { v += o.v; }
    __device__ __forceinline__ void maxv(double x) { v = fmax(v, x); }
    __device__ __forceinline__ void maxv(const Acc &o) { v = fmax(v, o.v); }
    __device__ __forceinline__ Acc shfl_xor(int o) const { Acc r; r.v = __shfl_xor_sync(0xffffffffu, v, o); return r; }
    __device__ __forceinline__ double value() const { return v; }
};
template <> struct Acc<float> {
    float hi, lo;
    __device__ __forceinline__ void zero() { hi = 0.f; lo = 0.f; }
    __device__ __forceinline__ void add(float x)
    {
        const float s = hi + x, bb = s - hi;
        lo += (hi - (s - bb)) + (x - bb);
        hi = s;
    }
    // a * b added exactly: the product is split into its rounded value and
    // the rounding error (exact with one FMA: Dekker's TwoProduct in the form
    // of Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26 (2005) 1955)
    __device__ __forceinline__ void add_prod(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        const float e = fmaf(a, b, -p);
        add(p);
        lo += e;
    }
    __device__ __forceinline__ void add(const Acc &o) { add(o.hi); lo += o.lo; }
    __device__ __forceinline__ void maxv(float x) { hi = fmaxf(hi, x); }
    __device__ __forceinline__ void maxv(const Acc &o) { hi = fmaxf(hi, o.hi); }
    __device__ __forceinline__ Acc shfl_xor(int o) const
    {
        Acc r;
        r.hi = __shfl_xor_sync(0xffffffffu, hi, o);
        r.lo = __shfl_xor_sync(0xffffffffu, lo, o);
        return r;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// double-word accumulator of the MM_F32X2 fields: per-cell products and sums
// in double-word arithmetic (relative rounding a few units of 2^-48 per
// operation), converted to double for the sums across CTAs
template <> struct Acc<dfloat> {
    dfloat v;
    __device__ __forceinline__ void zero() { v = dfloat(0.0f, 0.0f); }
    __device__ __forceinline__ void add(dfloat x) { v = v + x; }
    __device__ __forceinline__ void add_prod(dfloat a, dfloat b) { v = v + a * b; }
    __device__ __forceinline__ void add(const Acc &o) { v = v + o.v; }
    __device__ __forceinline__ void maxv(dfloat x)
    {
        if (x.hi > v.hi || (x.hi == v.hi && x.lo > v.lo)) v = x;
    }
    __device__ __forceinline__ void maxv(const Acc &o) { maxv(o.v); }
    __device__ __forceinline__ Acc shfl_xor(int o) const
    {
        Acc r;
        r.v.hi = __shfl_xor_sync(0xffffffffu, v.hi, o);
        r.v.lo = __shfl_xor_sync(0xffffffffu, v.lo, o);
        return r;
    }
    __device__ __forceinline__ double value() const { return df_to_double(v); }
};

__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// b into a: the maximum for the torque slot of the minimiser, a sum otherwise
template <int MODE, typename A> __device__ __forceinline__ void fold(A &a, const A &b, int slot)
{
    if (MODE == MODE_MIN && slot == SL_T2) a.maxv(b);
    else a.add(b);
}

// The NSL = 8 slots of every working thread of the CTA reduced to totals, slot s
// in lane s of warp 0 (in the return value; other lanes and warps get
// something else).  In a warp, each exchange halves the slots a lane is in
// charge of along with the lanes, 4 + 2 + 1 + 1 + 1 additions instead of 8 x 5;
// FP64 instructions are what a small film's reduction waits for.  nw working
// warps; `sm`: NSL values a warp of shared memory, free for use; two barriers,
// all threads of the CTA take part.
template <int MODE, typename A>
__device__ __forceinline__ A reduce_slots(A (&r)[NSL], A *sm, const int tid, const int nth)
{
    static_assert(NSL == 8, "three exchanges leave one slot a lane");
    const int lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
    int slot = 0;
#pragma unroll
    for (int n = 4, o = 16; n >= 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
        slot += up ? n : 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const A give = up ? r[i] : r[n + i];
            A keep = up ? r[n + i] : r[i];
            fold<MODE>(keep, give.shfl_xor(o), slot + i);
            r[i] = keep;
        }
    }
    fold<MODE>(r[0], r[0].shfl_xor(2), slot);
    fold<MODE>(r[0], r[0].shfl_xor(1), slot);
    if (warp < nw && (lane & 3) == 0) sm[warp * NSL + slot] = r[0];
    __syncthreads();
    A t;
    t.zero();
    if (warp == 0) {
        const int s = lane & 7;
        for (int w = lane >> 3; w < nw; w += 4) fold<MODE>(t, sm[w * NSL + s], s);
        fold<MODE>(t, t.shfl_xor(8), s);
        fold<MODE>(t, t.shfl_xor(16), s);
    }
    __syncthreads();
    return t;
}

// Finish the evaluation from the totals (warp 0; `mine`: the total of slot `lane`
// in lanes 0 .. 7).  The quotients and roots are taken by one lane each, in one
// division and one square root: one after another they took several
// microseconds of dependent FP64 instructions.
template <int MODE>
__device__ __forceinline__ void finish_iteration(const Geom &g, double mine, MinState *st,
                                                 cudaGraphConditionalHandle h, int use_cond, int body_kernels)
{
    const int lane = threadIdx.x & 31;
    double tot[NSL];
#pragma unroll
    for (int s = 0; s < NSL; ++s) tot[s] = __shfl_sync(0xffffffffu, mine, s);
    const double V = g.dx * g.dy * g.dz, Ms = g.Ms, cE = MM_MU0 * Ms * V;
    const double ss = tot[SL_SS], sy = tot[SL_SY], yy = tot[SL_YY];
    enum { Q_TAU1 = 0, Q_TAU2 = 1, Q_ROOT = 2, Q_TORQUE = 3, Q_TMAX = 4, Q_M = SL_MX };
    const bool min = MODE == MODE_MIN;
    const double num = lane == Q_TAU1 || lane == Q_ROOT ? ss : (lane == Q_TAU2 ? sy : (lane < SL_MX ? tot[SL_T2] : mine));
    const double den = lane == Q_TAU1 ? sy
                       : (lane == Q_TAU2 || lane == Q_ROOT ? yy : (lane == Q_TORQUE ? Ms * Ms : (lane == Q_TMAX ? 1.0 : (double)g.N)));
    const double quot = num / den;
    const double root = min ? sqrt(quot) : 0.0;
    double q[NSL];
#pragma unroll
    for (int s = 0; s < NSL; ++s) q[s] = __shfl_sync(0xffffffffu, min && s >= Q_ROOT && s <= Q_TMAX ? root : quot, s);
    if (lane != 0) return;
    st->mavg[0] = q[SL_MX];
    st->mavg[1] = q[SL_MY];
    st->mavg[2] = q[SL_MZ];
    if (MODE == MODE_ENERGY) {
        const double Ed = -0.5 * cE * tot[SL_ED], Eex = -0.5 * cE * tot[SL_EEX];
        const double Ean = V * tot[SL_EAN], Ez = -cE * tot[SL_EZ];
        st->energy[0] = Ed; st->energy[1] = Eex; st->energy[2] = Ean; st->energy[3] = Ez;
        st->energy[4] = Ed + Eex + Ean + Ez;
        return;
    }
    const long k = st->k;
    const double tmax = q[Q_TMAX];
    st->max_torque = q[Q_TORQUE];
    st->bb[0] = k > 0 ? ss : 0.0;
    st->bb[1] = k > 0 ? sy : 0.0;
    st->bb[2] = k > 0 ? yy : 0.0;
    st->energy[4] = -0.5 * cE * tot[SL_ET];
    st->evals = k + 1;
    st->launches += body_kernels;
    if (k == 0) st->t_start_ns = globaltimer_ns();
    int stop = 1;
    const bool finite = isfinite(tmax) && isfinite(st->energy[4]) &&
                        (k == 0 || (isfinite(ss) && isfinite(sy) && isfinite(yy)));
    if (!finite) {
        st->status = MMS_NONFINITE;
    } else if (tmax < st->tol_abs) {
        st->status = MMS_CONVERGED;
    } else if (k >= st->max_iter) {
        st->status = MMS_MAXITER;
    } else if (st->timeout_ns && globaltimer_ns() - st->t_start_ns > st->timeout_ns) {
        st->status = MMS_TIMEOUT;
    } else {
        double tau;
        if (k == 0) {
            tau = st->tau0;
        } else {
            if (st->tau_rule == MM_TAU_ADAPTIVE)   // tau^2 when cos^2(s, y) < kappa, else tau^1
                tau = (sy * sy < st->kappa * (ss * yy)) ? q[Q_TAU2] : q[Q_TAU1];
            else                                   // alternation: tau^1 on odd k, tau^2 on even k
                tau = (k & 1) ? q[Q_TAU1] : q[Q_TAU2];
            if (!(isfinite(tau) && tau > 0.0)) tau = q[Q_ROOT];
            if (!(isfinite(tau) && tau > 0.0)) tau = st->tau0;
        }
        st->tau = tau;
        st->tauf = (float)tau;
        st->tauw = dfloat(tau);
        st->k = k + 1;
        stop = 0;
    }
    if (use_cond) cudaGraphSetConditional(h, stop ? 0u : 1u);
}

// ---------------------------------------------------------------------------
// k_xinv
// ---------------------------------------------------------------------------
// bid: this CTA's slot among the problem's nblk CTAs (partial sums, completion count)
template <typename T, typename F, int MODE, int LX>
__device__ __forceinline__ void xinv_body(const Geom &g, const FieldPtrs<T, F> &P, double hx0, double hx1, double hx2,
                                          cudaGraphConditionalHandle h, int use_cond, const int tid, const int nth,
                                          const int bx, const int by, const int bid, const int nblk)
{
    typedef typename cvec<F>::type V;
    typedef typename twvec<F>::type TW;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *S = reinterpret_cast<V *>(smem_raw);
    const int tt = tid < nth ? tid : MM_IDLE_START;
    const int TY = g.TY, y0 = bx * TY, z = by;
    const int nx = g.nx, ny = g.ny, nz = g.nz, Hx = g.Hx;
    const long N = g.N;
    TW *tw = reinterpret_cast<TW *>(S + 3 * TY * g.rsx);
    // block fixed point: the x-frequencies' largest scale and the sum of their scales over the largest, per component,
    // and the flags; the magnitude of each row and the scale of its transform, by row for the reason given in xfwd_body
    __shared__ int s_e[3];
    __shared__ unsigned s_r[4];
    __shared__ unsigned s_mag[3 * MM_MAX_TILE];
    __shared__ double s_scale[3 * MM_MAX_TILE];
    unsigned *s_fl = s_r, *s_sum = s_r + 1;
    unsigned mag = 0;
    const int *fe2 = nullptr;
    const int ns = g.sep ? 3 : 1, fst = ns * g.nzb;   // ints from one x-frequency's scales to the next's
    const bool sep = g.sep;
    auto own = [&](int c) { return sep ? c : 0; };   // which of the scales is a component's
    if constexpr (is_fx<F>) {
        fe2 = P.fe2 + ns * (z / g.ZB);
        if (tid < 3) s_e[tid] = FX_ZERO;
        if (tid < 4) s_r[tid] = 0;
        if (tid < 3 * TY) s_mag[tid] = 0;
        __syncthreads();
        if (sep) fx_cta_scales<3>(fe2, g.C, fst, tt, nth, s_e, s_fl);
        else fx_cta_scales<1>(fe2, g.C, fst, tt, nth, s_e, s_fl);
    }

    MinState *st = P.st;
    long k = 0;
    int cur = 0;
    typedef typename io_of<T>::type IO;
    constexpr bool FROM_T = MODE == MODE_MIN || std::is_same<T, IO>::value;
    const T *m = nullptr;       // m in the field type (the iterate, or the caller's m of that type)
    const IO *mio = nullptr;    // the caller's m when it is of another type (converted per load)
    const T *mp = nullptr, *gq = nullptr;
    if (MODE == MODE_MIN) {
        k = st->k;
        cur = st->base ^ (int)(k & 1);
        m = cur ? P.mbuf[1] : P.mbuf[0];
        mp = cur ? P.mbuf[0] : P.mbuf[1];
        gq = (k & 1) ? P.gbuf[0] : P.gbuf[1];  // g_{k-1}
    } else if constexpr (std::is_same<T, IO>::value) {
        m = P.m_src;
    } else {
        mio = P.m_src;
    }
    auto mval = [&](long i) -> T {
        if constexpr (FROM_T) return m[i];
        else return from_io<T>(mio[i]);
    };
    // the float kernel stages the local terms' inputs -- m on planes z-1, z,
    // z+1 (rows y0-1 .. y0+TY on its own plane), m_{k-1} and g_{k-1} -- with
    // cp.async now; they arrive while the inverse x-FFT runs
    const bool stg = sizeof(T) == 4 && MODE == MODE_MIN && g.stage;
    T *SG = reinterpret_cast<T *>(smem_raw + stage_offset<T>(g));
    const int oZm = 3 * (TY + 2) * nx, oZp = oZm + 3 * TY * nx, oMP = oZp + 3 * TY * nx, oGQ = oMP + 3 * TY * nx;
    load_twiddles_async(tw, P.tw_px, g.Px, g.Hx, tt, nth);
    cp_async_commit();
    if (stg) {
        stage_rows(SG, m, g, z, y0 - 1, TY + 2, tid, nth);
        if (z > 0) stage_rows(SG + oZm, m, g, z - 1, y0, TY, tid, nth);
        if (z < nz - 1) stage_rows(SG + oZp, m, g, z + 1, y0, TY, tid, nth);
        if (k > 0) {
            stage_rows(SG + oMP, mp, g, z, y0, TY, tid, nth);
            stage_rows(SG + oGQ, gq, g, z, y0, TY, tid, nth);
        }
    }
    cp_async_commit();

    // complex-to-real preprocessing: Z[k] = (X[k] + X*[Hx-k]) + i conj(w^k) (X[k] - X*[Hx-k]).
    // With sum and dif the two brackets and t = conj(w^k) dif, Z[k] = sum + i t and
    // (w^Hx = -1) Z[Hx-k] = sum* + i t*: one item per pair k = 0..Hx/2 loads X[k] and
    // X[Hx-k] once.  The loads of PF items per thread are issued before any is used.
    // A thread's items are all of one row (c, yl): it takes every ks-th k.
    constexpr int PF = sizeof(V) == 8 ? 8 : 4;
    const int hh = Hx >> 1, ks = nth / (3 * TY), k0 = tid / (3 * TY), q = tid - k0 * 3 * TY, c = q % 3, yl = q / 3;
    const bool mine = k0 < ks;
    const long strideK = (long)3 * nz * ny;
    V *const row = S + (c * TY + yl) * g.rsx;
    const V *const Wrow = P.W + ((long)z * ny + y0 + yl) * 3 + c;
    for (int g0 = 0; g0 <= hh; g0 += PF * ks) {  // trip count uniform over the CTA (barrier inside)
        V xa[PF], xb[PF];
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int kk = g0 + k0 + i * ks;
            xa[i] = czero<V>(); xb[i] = czero<V>();
            if (mine && kk <= hh && y0 + yl < ny) {
                xa[i] = ld_nc(Wrow + (long)kk * strideK);
                xb[i] = ld_nc(Wrow + (long)(Hx - kk) * strideK);
            }
        }
        if (g0 == 0) {  // the twiddles (first commit group) are needed from here on
            cp_async_wait_group<1>();
            __syncthreads();
            if constexpr (is_fx<F>) {
                unsigned sum[3] = {0, 0, 0};
                for (int i = tt; i < g.C; i += nth) {
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        if (a == 0 || sep) sum[a] += ((1u << 18) >> min(s_e[a] - fx_exp(fe2[i * fst + a]), 18)) + 1;
                }
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    if (a == 0 || sep) fx_cta_add(&s_sum[a], sum[a]);
            }
        }
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int kk = g0 + k0 + i * ks;
            if (!mine || kk > hh) break;
            V Z;
            V Xk = xa[i], Xm = cconj(xb[i]);
            if constexpr (is_fx<F>) {  // components below 2^60: |Z| < 2^62
                Xk = fx_down(Xk, s_e[own(c)] - fx_exp(fe2[kk * fst + own(c)]));
                Xm = fx_down(Xm, s_e[own(c)] - fx_exp(fe2[(Hx - kk) * fst + own(c)]));
            }
            const V sum = cadd(Xk, Xm), dif = csub(Xk, Xm);
            V t;
            if constexpr (is_fx<F>) t = fx_cmul<true>(dif, tw[tpos<TW>(kk, g.Hx)], 0);
            else t = cmulc(dif, tw[tpos<TW>(kk, g.Hx)]);  // conj(w^k) dif
            Z.x = sum.x - t.y;
            Z.y = sum.y + t.x;
            row[rpos<V, LX>(kk)] = Z;
            if constexpr (is_fx<F>) mag |= fx_mag(Z);
            if (kk != 0 && Hx - kk != kk) {
                Z.x = sum.x + t.y;
                Z.y = t.x - sum.y;
                row[rpos<V, LX>(Hx - kk)] = Z;
                if constexpr (is_fx<F>) mag |= fx_mag(Z);
            }
        }
    }
    constexpr bool DW = std::is_same<T, dfloat>::value;
    if constexpr (is_fx<F>) {
        if (mine && mag) atomicOr(&s_mag[c * TY + yl], mag);
    }
    __syncthreads();
    // the moduli of a row sum to at most 2^62 times the frequencies' scales over the largest
    auto bound = [&](int r) { return max(0, fx_log2_up(s_sum[own(r >> g.lty)]) - 18 + 62 - fx_bits(s_mag[r])); };
    if constexpr (is_fx<F>) {
        if (tid < 3 * TY) {
            // one unit of the row's values after its transform, in A/m (of double-words in two factors below the range of one)
            const int e = s_e[own(tid >> g.lty)] + fx_cum(fx_log(Hx), bound(tid)) - (58 - fx_bits(s_mag[tid]));
            if constexpr (DW)
                *reinterpret_cast<float2 *>(&s_scale[tid]) = make_float2(fx_pow2f(e < -100 ? e + 64 : e),
                                                                         e < -100 ? 5.42101086e-20f : 1.0f);   // 2^-64
            else
                s_scale[tid] = fx_pow2(e);
        }
    }
    {
        const int row = tid / g.Gx, j = tid - row * g.Gx;
        const bool act = row < 3 * TY;
        if constexpr (is_fx<F>) {
            const int r = act ? row : 0;
            unsigned none = 0;
            fft_row_fx<true, false, true, 2, LX, false>(S + r * g.rsx, Hx, g.lhx, j, tw, act, 58 - fx_bits(s_mag[r]),
                                                        bound(r), none);
        } else {
            fft_row<true, false, true, 2, LX>(S + (act ? row : 0) * g.rsx, Hx, g.lhx, j, tw, act);
        }
    }
    int bad = 0;
    if constexpr (is_fx<F>) bad = sep || !*s_fl ? (int)*s_fl : 7;
    cp_async_wait_all();
    if (stg) __syncthreads();

    // local terms
    T he0, he1, he2;
    if (MODE == MODE_MIN) {
        he0 = pick<T>(st->Hext[0], st->Hextf[0], st->Hextw[0]);
        he1 = pick<T>(st->Hext[1], st->Hextf[1], st->Hextw[1]);
        he2 = pick<T>(st->Hext[2], st->Hextf[2], st->Hextw[2]);
    } else {
        he0 = (T)hx0; he1 = (T)hx1; he2 = (T)hx2;
    }
    const T cx = pick<T>(g.cex_x, g.fcex_x, g.wcex[0]), cy = pick<T>(g.cex_y, g.fcex_y, g.wcex[1]),
            cz = pick<T>(g.cex_z, g.fcex_z, g.wcex[2]);
    const T can = pick<T>(g.can, g.fcan, g.wcan);
    const T Kuni = pick<T>(g.K, g.fK, g.wK), ux = pick<T>(g.u[0], g.fu[0], g.wu[0]),
            uy = pick<T>(g.u[1], g.fu[1], g.wu[1]), uz = pick<T>(g.u[2], g.fu[2], g.wu[2]);
    const T hs = (T)P.hscale;
    const T canK = mul_rn(can, Kuni);
    Acc<T> red[NSL];
#pragma unroll
    for (int s = 0; s < NSL; ++s) red[s].zero();

    for (int e = tt; e < TY * nx; e += nth) {
        const int yl = g.fd_nx.div(e), x = e - yl * nx, y = y0 + yl;
        if (y >= ny) continue;
        const long n = ((long)z * ny + y) * nx + x;
        T d0, d1, d2;
        if constexpr (is_fx<F>) {
            const fx q0 = rel<F, LX>(S + (0 * TY + yl) * g.rsx, x), q1 = rel<F, LX>(S + (1 * TY + yl) * g.rsx, x),
                     q2 = rel<F, LX>(S + (2 * TY + yl) * g.rsx, x);
            if constexpr (DW) {
                dfloat *d[3] = {&d0, &d1, &d2};
                const fx q[3] = {q0, q1, q2};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float2 f = *reinterpret_cast<const float2 *>(&s_scale[c * TY + yl]);
                    *d[c] = fx_to_dfloat(q[c], f.x);
                    if (f.y != 1.0f) { d[c]->hi *= f.y; d[c]->lo *= f.y; }
                }
            } else {
                d0 = __ll2double_rn(q0.v) * s_scale[yl];
                d1 = __ll2double_rn(q1.v) * s_scale[TY + yl];
                d2 = __ll2double_rn(q2.v) * s_scale[2 * TY + yl];
            }
            if (bad) {  // uniform over the CTA
                T nan;
                if constexpr (DW) nan = dfloat(__int_as_float(0x7fc00000), 0.0f);
                else nan = __longlong_as_double(0x7ff8000000000000ll);
                if (bad & 1) d0 = nan;
                if (bad & 2) d1 = nan;
                if (bad & 4) d2 = nan;
            }
        } else {
            d0 = to_field<T>(rel<F, LX>(S + (0 * TY + yl) * g.rsx, x));
            d1 = to_field<T>(rel<F, LX>(S + (1 * TY + yl) * g.rsx, x));
            d2 = to_field<T>(rel<F, LX>(S + (2 * TY + yl) * g.rsx, x));
        }
        // exchange: sum over present neighbours of (m_j - m_i) / d^2 (free faces)
        T m0, m1, m2, e0 = 0, e1 = 0, e2 = 0;
        if (stg) {
            const int cs = (TY + 2) * nx, ct = TY * nx;    // component strides of the staged rows
            const T *r0 = SG + (yl + 1) * nx + x;          // this cell, component 0
            m0 = r0[0]; m1 = r0[cs]; m2 = r0[2 * cs];
            if (x > 0)      { e0 += cx * (r0[-1] - m0);  e1 += cx * (r0[cs - 1] - m1);  e2 += cx * (r0[2 * cs - 1] - m2); }
            if (x < nx - 1) { e0 += cx * (r0[1] - m0);   e1 += cx * (r0[cs + 1] - m1);  e2 += cx * (r0[2 * cs + 1] - m2); }
            if (y > 0)      { e0 += cy * (r0[-nx] - m0); e1 += cy * (r0[cs - nx] - m1); e2 += cy * (r0[2 * cs - nx] - m2); }
            if (y < ny - 1) { e0 += cy * (r0[nx] - m0);  e1 += cy * (r0[cs + nx] - m1); e2 += cy * (r0[2 * cs + nx] - m2); }
            const T *rz = SG + yl * nx + x;
            if (z > 0)      { const T *q = rz + oZm; e0 += cz * (q[0] - m0); e1 += cz * (q[ct] - m1); e2 += cz * (q[2 * ct] - m2); }
            if (z < nz - 1) { const T *q = rz + oZp; e0 += cz * (q[0] - m0); e1 += cz * (q[ct] - m1); e2 += cz * (q[2 * ct] - m2); }
        } else {
            if constexpr (FROM_T) {
                m0 = ldg(m + n); m1 = ldg(m + N + n); m2 = ldg(m + 2 * N + n);
            } else {
                m0 = from_io<T>(ldg(mio + n)); m1 = from_io<T>(ldg(mio + N + n)); m2 = from_io<T>(ldg(mio + 2 * N + n));
            }
            if (x > 0)      { e0 += cx * (mval(n - 1) - m0);  e1 += cx * (mval(N + n - 1) - m1);  e2 += cx * (mval(2 * N + n - 1) - m2); }
            if (x < nx - 1) { e0 += cx * (mval(n + 1) - m0);  e1 += cx * (mval(N + n + 1) - m1);  e2 += cx * (mval(2 * N + n + 1) - m2); }
            if (y > 0)      { e0 += cy * (mval(n - nx) - m0); e1 += cy * (mval(N + n - nx) - m1); e2 += cy * (mval(2 * N + n - nx) - m2); }
            if (y < ny - 1) { e0 += cy * (mval(n + nx) - m0); e1 += cy * (mval(N + n + nx) - m1); e2 += cy * (mval(2 * N + n + nx) - m2); }
            const long sxy = (long)nx * ny;
            if (z > 0)      { e0 += cz * (mval(n - sxy) - m0); e1 += cz * (mval(N + n - sxy) - m1); e2 += cz * (mval(2 * N + n - sxy) - m2); }
            if (z < nz - 1) { e0 += cz * (mval(n + sxy) - m0); e1 += cz * (mval(N + n + sxy) - m1); e2 += cz * (mval(2 * N + n + sxy) - m2); }
        }
        // uniaxial anisotropy
        const T Kv = P.Kc ? from_io<T>(P.Kc[n]) : Kuni;
        T u0, u1, u2;
        if (P.uc) { u0 = from_io<T>(P.uc[n]); u1 = from_io<T>(P.uc[N + n]); u2 = from_io<T>(P.uc[2 * N + n]); }
        else { u0 = ux; u1 = uy; u2 = uz; }
        const T mu = m0 * u0 + m1 * u1 + m2 * u2;
        const T kc = P.Kc ? mul_rn(can, Kv) : canK;
        const T ka = kc * mu;
        const T H0 = d0 + e0 + ka * u0 + he0;
        const T H1 = d1 + e1 + ka * u1 + he1;
        const T H2 = d2 + e2 + ka * u2 + he2;
        if (MODE == MODE_HEFF) {
            P.H_out[n] = to_io(hs * H0); P.H_out[N + n] = to_io(hs * H1); P.H_out[2 * N + n] = to_io(hs * H2);
            continue;
        }
        red[SL_MX].add(m0); red[SL_MY].add(m1); red[SL_MZ].add(m2);
        if (MODE == MODE_ENERGY) {
            if constexpr (sizeof(T) == 4) {
                // float path: every per-cell product enters its sum exactly
                red[SL_ED].add_prod(m0, d0); red[SL_ED].add_prod(m1, d1); red[SL_ED].add_prod(m2, d2);
                red[SL_EEX].add_prod(m0, e0); red[SL_EEX].add_prod(m1, e1); red[SL_EEX].add_prod(m2, e2);
                red[SL_EAN].add_prod(Kv, (T)1 - mu * mu);
                red[SL_EZ].add_prod(m0, he0); red[SL_EZ].add_prod(m1, he1); red[SL_EZ].add_prod(m2, he2);
            } else {
                red[SL_ED].add(m0 * d0 + m1 * d1 + m2 * d2);
                red[SL_EEX].add(m0 * e0 + m1 * e1 + m2 * e2);
                red[SL_EAN].add(Kv * ((T)1 - mu * mu));
                red[SL_EZ].add(m0 * he0 + m1 * he1 + m2 * he2);
            }
            continue;
        }
        // projected gradient g = m x (m x H) = (m.H) m - |m|^2 H (the triple
        // product identity; orthogonal to m for any |m|, which keeps the
        // midpoint step norm-preserving even as rounding moves |m| off 1)
        const T mh = m0 * H0 + m1 * H1 + m2 * H2;
        const T mm = m0 * m0 + m1 * m1 + m2 * m2;
        const T g0 = mh * m0 - mm * H0, g1 = mh * m1 - mm * H1, g2 = mh * m2 - mm * H2;
        red[SL_T2].maxv(g0 * g0 + g1 * g1 + g2 * g2);  // |m x H|^2 = |g|^2 for |m| = 1
        // energy density / (mu0 Ms V), times -2: m.H + m.H_ext - 2 K/(mu0 Ms), complete
        // in every cell and with the field's own rounded 2 K/(mu0 Ms): a hard magnet's
        // terms cancel to a small part of K there, and sums of them apart would not
        const T mhe = m0 * he0 + m1 * he1 + m2 * he2;
        if constexpr (sizeof(T) == 4) {
            red[SL_ET].add_prod(m0, H0); red[SL_ET].add_prod(m1, H1); red[SL_ET].add_prod(m2, H2);
            red[SL_ET].add_prod(m0, he0); red[SL_ET].add_prod(m1, he1); red[SL_ET].add_prod(m2, he2);
            red[SL_ET].add(-kc);
        } else {
            red[SL_ET].add((mh + mhe) - kc);
        }
        T *gout = (k & 1) ? P.gbuf[1] : P.gbuf[0];
        if (k > 0) {
            T p0, p1, p2, q0, q1, q2;
            if (stg) {
                const int sn = yl * nx + x, ct = TY * nx;
                p0 = SG[oMP + sn]; p1 = SG[oMP + ct + sn]; p2 = SG[oMP + 2 * ct + sn];
                q0 = SG[oGQ + sn]; q1 = SG[oGQ + ct + sn]; q2 = SG[oGQ + 2 * ct + sn];
            } else {
                p0 = mp[n]; p1 = mp[N + n]; p2 = mp[2 * N + n];
                q0 = gq[n]; q1 = gq[N + n]; q2 = gq[2 * N + n];
            }
            const T s0 = m0 - p0, s1 = m1 - p1, s2 = m2 - p2;
            const T y0v = g0 - q0, y1v = g1 - q1, y2v = g2 - q2;
            if constexpr (sizeof(T) == 4) {
                // float path: exact products, compensated sums (the step size
                // needs s.y, a difference of nearly equal sums near convergence)
                red[SL_SS].add_prod(s0, s0); red[SL_SS].add_prod(s1, s1); red[SL_SS].add_prod(s2, s2);
                red[SL_SY].add_prod(s0, y0v); red[SL_SY].add_prod(s1, y1v); red[SL_SY].add_prod(s2, y2v);
                red[SL_YY].add_prod(y0v, y0v); red[SL_YY].add_prod(y1v, y1v); red[SL_YY].add_prod(y2v, y2v);
            } else {
                red[SL_SS].add(s0 * s0 + s1 * s1 + s2 * s2);
                red[SL_SY].add(s0 * y0v + s1 * y1v + s2 * y2v);
                red[SL_YY].add(y0v * y0v + y1v * y1v + y2v * y2v);
            }
        }
        gout[n] = g0; gout[N + n] = g1; gout[2 * N + n] = g2;
    }
    if (MODE == MODE_HEFF) return;

    // CTA reduction, in shared memory that the FFT rows no longer need
    __syncthreads();
    const int warp = tid >> 5, lane = tid & 31;
    {
        const Acc<T> t = reduce_slots<MODE>(red, reinterpret_cast<Acc<T> *>(smem_raw), tid, nth);
        if (warp == 0 && lane < NSL) P.partials[(long)bid * RED_NSLOT + lane] = t.value();
    }
    // the last CTA to arrive finishes the evaluation
    __shared__ int s_last;
    if (warp == 0) {
        __syncwarp();
        if (lane == 0) {
            __threadfence();
            s_last = (atomicAdd(P.counter, 1u) == (unsigned)nblk - 1);
        }
    }
    __syncthreads();
    if (s_last) {   // no early return: a persistent batch CTA goes on to its next work item
        // thread t sums the partials of CTAs t, t + nth, ...: a fixed order, so
        // the result does not depend on which CTA came last
        __threadfence();
        Acc<double> v[NSL];
#pragma unroll
        for (int s = 0; s < NSL; ++s) v[s].zero();
        for (int b = tt; b < nblk; b += nth) {
            double2 x[NSL / 2];
#pragma unroll
            for (int q = 0; q < NSL / 2; ++q)
                x[q] = __ldcg(reinterpret_cast<const double2 *>(P.partials + (long)b * RED_NSLOT) + q);
#pragma unroll
            for (int s = 0; s < NSL; ++s) {
                Acc<double> xs;
                xs.v = (s & 1) ? x[s / 2].y : x[s / 2].x;
                fold<MODE>(v[s], xs, s);
            }
        }
        const Acc<double> t = reduce_slots<MODE>(v, reinterpret_cast<Acc<double> *>(smem_raw), tid, nth);
        if (warp == 0) {
            finish_iteration<MODE>(g, t.v, st, h, use_cond, g.nbody);
            if (lane == 0) *P.counter = 0u;
        }
    }
}

template <typename T, typename F, int MODE, int LX>
__global__ void __launch_bounds__(768) k_xinv(Geom g, FieldPtrs<T, F> P, double hx0, double hx1, double hx2,
                                              cudaGraphConditionalHandle h, int use_cond)
{
    xinv_body<T, F, MODE, LX>(g, P, hx0, hx1, hx2, h, use_cond, threadIdx.x, blockDim.x, blockIdx.x, blockIdx.y,
                           blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y);
}

// ---------------------------------------------------------------------------
// launch shapes and buffers of a problem's field kernels
// ---------------------------------------------------------------------------
template <typename T, typename F = typename fft_of<T>::type> FieldPtrs<T, F> make_ptrs(mm_problem *p)
{
    typedef typename cvec<F>::type V;
    typedef typename twvec<F>::type TW;
    const Geom &g = p->g;
    FieldPtrs<T, F> P;
    P.m_src = nullptr; P.H_out = nullptr;
    P.mbuf[0] = (T *)p->mbuf[0]; P.mbuf[1] = (T *)p->mbuf[1];
    P.gbuf[0] = (T *)p->gbuf[0]; P.gbuf[1] = (T *)p->gbuf[1];
    P.W = (V *)p->W; P.W2 = (V *)p->W2; P.Nhat = (const typename coef<F>::type *)p->Nhat;
    P.tw_px = (const TW *)p->tw_px; P.tw_py = (const TW *)p->tw_py; P.tw_pz = (const TW *)p->tw_pz;
    P.fe1 = p->fexp;
    P.fea = p->fexp + 3 * (long)g.nz * g.ny;
    P.feb = P.fea + 3 * (long)g.C * g.nzb;
    P.fe2 = P.feb + 3 * (long)g.C * g.nkb;
    P.fek = P.fe2 + 3 * (long)g.C * g.nzb;   // mm_scale_fek
    typedef typename io_of<T>::type IO;
    P.Kc = (const IO *)p->Kc; P.uc = (const IO *)p->uc;
    P.partials = p->partials; P.st = p->st; P.counter = p->counter;
    P.hscale = 1.0;
    return P;
}

static inline int round32(int n) { return (n + 31) & ~31; }
template <typename T> int threads_x(const Geom &g) { return round32(3 * g.TY * g.Gx); }
template <typename T> int threads_xf(const Geom &g) { return round32(3 * g.TYF * g.Gx); }
template <typename T> size_t smem_xf_t(const Geom &g)
{
    typedef typename cvec<typename fft_of<T>::type>::type V;
    return (size_t)3 * g.TYF * g.rsx * sizeof(V) + (size_t)g.Px * sizeof(V);
}
template <typename T> int threads_yz(const Geom &g) { return round32(g.RB * g.Gy); }

template <typename T> size_t smem_x_t(const Geom &g)
{
    typedef typename cvec<typename fft_of<T>::type>::type V;
    size_t rows = (size_t)3 * g.TY * g.rsx * sizeof(V) + (size_t)g.Px * sizeof(V);
    if (sizeof(T) == 4 && g.stage) rows = stage_offset<T>(g) + (size_t)(15 * g.TY + 6) * g.nx * sizeof(T);
    const size_t stage = (size_t)NSL * (threads_x<T>(g) / 32) * 8;   // reduce_slots: 8-byte values
    return rows > stage ? rows : stage;
}
template <typename T> size_t smem_yz_t(const Geom &g)
{
    typedef typename cvec<typename fft_of<T>::type>::type V;
    // rows and Py twiddles,
    // and the block fixed-point kernel two bytes per y-frequency and component
    return ((size_t)3 * g.nz * g.rsy + g.Py) * sizeof(V) + (sizeof(T) == 4 ? 0 : (g.sep ? 6 : 2) * (size_t)g.Py);
}

// The field kernels are compiled for a set of FFT row lengths (template
// parameter LX of the x kernels, LY of the y-z kernel; MM_LX_CASES,
// MM_LY_CASES) and once for any power of two (0); the launchers pick the
// instance (lx_of, ly_of).

// the bytes a launch needs must fit the common cap, which every kernel is given
template <typename K> cudaError_t smem_attr(K *f, size_t bytes)
{
    if (bytes > (size_t)MM_SMEM_CAP) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, MM_SMEM_CAP);
}

} // namespace

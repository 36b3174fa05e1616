// Bulk layout of the demagnetisation convolution (Section 3's zero-padded
// FFT convolution for three-dimensional samples).
//
// The film kernels k_yz and k_yz_fx hold a whole padded y-z plane of one x-frequency in
// shared memory, which bounds nz * Py.  Bulk samples (a cube of 256^3 cells
// pads to 512 x 512 x 512, one of 160^3 to 320^3) split that stage into three passes through HBM:
//
//  k_ypass<fwd>  per (kx, ZB z-planes): FFT along y of the three components,
//                zero padding ny -> Py, W[kx][z][y][c] -> W2[kx][z][ky][c];
//  k_zconv       per (kx, KB y-frequencies): FFT along z (padding nz -> Pz),
//                the product with the symmetric 3x3 tensor spectrum
//                (H^ = -Ms N^ m^, normalisation folded into N^), inverse FFT
//                along z keeping the first nz values, in place in W2;
//  k_ypass<inv>  inverse FFT along y keeping the first ny rows, W2 -> W.
//
// The x passes (k_xfwd with the minimiser step, k_xinv with the local terms
// and the step-size sums) are the film kernels unchanged.  Shared-memory rows
// use the swizzled or padded Stockham layout of fft.cuh.
#include "common.cuh"
#include "fft.cuh"

namespace {

// log2 of a power of two (ZB, KB)
__device__ __forceinline__ int log2_of(int p) { return 31 - __clz(p); }

template <typename V> __device__ __forceinline__ V load_cg(const V *p) { return __ldcg(p); }
template <> __device__ __forceinline__ fxc load_cg(const fxc *p)
{
    const longlong2 v = __ldcg(reinterpret_cast<const longlong2 *>(p));
    return fxc{fx(v.x), fx(v.y)};
}

template <typename T> struct BulkBound { static constexpr int v = sizeof(T) == 8 ? 256 : 512; };
// two CTAs of the z pass per SM: without the bound its odd radices take 121
// registers (float: 682 -> 550 us at 160^3), and in fixed point one CTA of 384
// threads and 127 registers had an SM to itself (64^3: 121 -> 102 us)
constexpr int Z_CTAS = 2;
// the y passes' register bound: 168 in fixed point (128: y-forward 28.5 -> 32.5 us)
template <typename T> constexpr int Y_BOUND = sizeof(T) == 8 ? 384 : 512;

// In block fixed point (double fields, F = fx) every CTA of a pass brings its
// block to full magnitude when it loads it and when it stores it, component by
// component, with the scales of a block per (kx, ZB planes) after the y passes
// and per (kx, KB y-frequencies) after the z convolution.
template <typename T, bool INV, int LY>
__global__ void __launch_bounds__(Y_BOUND<T>) k_ypass(Geom g, FieldPtrs<T> P)
{
    typedef typename FieldPtrs<T>::V V;
    typedef typename FieldPtrs<T>::TW TW;
    constexpr bool FX = std::is_same<V, fxc>::value;
    __shared__ int s_e[3];
    __shared__ unsigned s_r[7];  // flags, magnitudes in and out
    unsigned *s_fl = s_r, *s_in = s_r + 1, *s_out = s_r + 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *S = reinterpret_cast<V *>(smem_raw);
    const int tid = threadIdx.x, nth = blockDim.x;
    const int ny = g.ny, nz = g.nz, Py = LY ? fft_length(LY) : g.Py, ZB = g.ZB, rs = g.rsy;
    const int kx = blockIdx.x, z0 = blockIdx.y * ZB;
    const int zb = min(ZB, nz - z0);
    TW *tw = reinterpret_cast<TW *>(S + 3 * ZB * rs);
    load_twiddles_async(tw, P.tw_py, Py, Py, tid, nth);
    FxMags<3> mags;
    const int *scales = nullptr;   // of the values read: of every (z, y) row of W, or of KB y-frequencies of W2
    const bool sep = g.sep;
    const int ns = sep ? 3 : 1;
    auto own = [&](int c) { return sep ? c : 0; };   // which of the scales is a component's
    if constexpr (FX) {
        if (tid < 3) s_e[tid] = FX_ZERO;
        if (tid < 7) s_r[tid] = 0;
        __syncthreads();
        scales = INV ? P.feb + (long)kx * g.nkb * ns : P.fe1 + (long)z0 * ny * ns;
        const int n = INV ? g.nkb : zb * ny;
        if (sep) fx_cta_scales<3>(scales, n, 3, tid, nth, s_e, s_fl);
        else fx_cta_scales<1>(scales, n, 1, tid, nth, s_e, s_fl);
        __syncthreads();
    }
    const long first = (long)kx * nz + z0;  // first (kx, z) row pair of this CTA
    const int lin = INV ? Py : ny;           // input length per (z, c) row
    const V *src = INV ? P.W2 + first * Py * 3 : P.W + first * ny * 3;
    // [zl][y][c] -> row (c, zl); PF loads per thread in flight before use
    constexpr int PF = sizeof(T) == 4 ? 8 : 4;
    const int tot = zb * lin * 3;
    for (int e0 = tid; e0 < tot; e0 += PF * nth) {
        V v[PF];
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int e = e0 + i * nth;
            if (e < tot) v[i] = load_cg(src + e);
        }
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int e = e0 + i * nth;
            if (e >= tot) break;
            const int c = e % 3, rest = e / 3, zl = INV ? rest / Py : g.fd_ny.div(rest), y = rest - zl * lin;
            if constexpr (FX) {
                v[i] = fx_down(v[i], s_e[own(c)] - fx_exp(scales[(INV ? y >> log2_of(g.KB) : rest) * ns + own(c)]));
                mags.or_in(own(c), fx_mag(v[i]));
            }
            S[(c * ZB + zl) * rs + rpos<V, LY>(y)] = v[i];
        }
    }
    if (!INV) {
        const int npad = Py - ny;
        for (int e = tid; e < 3 * ZB * npad; e += nth) {
            const int r = g.fd_pady.div(e), y = ny + (e - r * npad);
            S[r * rs + rpos<V, LY>(y)] = czero<V>();
        }
    }
    auto cta_mags = [&](unsigned *dst) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (c == 0 || sep) fx_cta_or(dst + c, mags.v[c]);
    };
    if constexpr (FX) cta_mags(s_in);
    cp_async_wait_all();
    __syncthreads();
    const int Gy = g.Gy, RB = g.RBY;
    const int rb = tid / Gy, j = tid - rb * Gy;
    int sh = 0, pre[3] = {0, 0, 0}, post[3] = {0, 0, 0};
    if constexpr (FX) {
#pragma unroll
        for (int c = 0; c < 3; ++c) pre[c] = (INV ? 58 : 59) - fx_bits(s_in[own(c)]);
    }
    mags = FxMags<3>();
    for (int r0 = 0; r0 < 3 * ZB; r0 += RB) {
        const int r = r0 + rb;
        const bool act = rb < RB && r < 3 * ZB && (r % ZB) < zb;
        if constexpr (FX) {
            const int c = act ? own(r >> log2_of(ZB)) : 0;
            unsigned mag = 0;
            sh = fft_row_fx<INV, !INV, INV, 1, LY, true>(S + (act ? r : 0) * rs, Py, g.lpy, j, tw, act, fx_of(pre, c), 64,
                                                         mag);
            mags.or_in(c, mag);
        } else
            fft_row<INV, !INV, INV, 1, LY>(S + (act ? r : 0) * rs, Py, g.lpy, j, tw, act);
    }
    if constexpr (FX) cta_mags(s_out);
    __syncthreads();
    if constexpr (FX) {
#pragma unroll
        for (int c = 0; c < 3; ++c) post[c] = 60 - fx_bits(s_out[own(c)]);
        if (tid < ns)
            (INV ? P.fe2 : P.fea)[((long)kx * g.nzb + blockIdx.y) * ns + tid] =
                fx_pack(s_e[tid] - fx_of(pre, tid) + sh - fx_of(post, tid), *s_fl >> tid & 1);
    }
    const int lout = INV ? ny : Py;
    V *dst = INV ? P.W + first * ny * 3 : P.W2 + first * Py * 3;
    for (int e = tid; e < zb * lout * 3; e += nth) {
        const int c = e % 3, rest = e / 3, zl = INV ? g.fd_ny.div(rest) : rest / Py, y = rest - zl * lout;
        V r = S[(c * ZB + zl) * rs + rpos<V, LY>(y)];
        if constexpr (FX) r = fx_scale(r, fx_of(post, c));
        dst[e] = r;
    }
}

// SEP: block fixed point with scales per component (Geom::sep)
template <typename T, int LZ, bool SEP>
__global__ void __launch_bounds__(BulkBound<T>::v, Z_CTAS) k_zconv(Geom g, FieldPtrs<T> P)
{
    typedef typename FieldPtrs<T>::V V;
    typedef typename FieldPtrs<T>::TW TW;
    constexpr bool FX = std::is_same<V, fxc>::value;
    constexpr int NS = SEP ? 3 : 1;
    __shared__ int s_e[NS], s_top[NS];
    // magnitudes in and out, sums of the frequencies' scales over the largest, flags
    __shared__ unsigned s_r[3 * NS + 1];
    unsigned *s_in = s_r, *s_out = s_r + NS, *s_sum = s_r + 2 * NS, *s_fl = s_r + 3 * NS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *S = reinterpret_cast<V *>(smem_raw);
    const int tid = threadIdx.x, nth = blockDim.x;
    const int nz = g.nz, Py = g.Py, Pz = LZ > 0 ? fft_length(LZ) : g.Pz, KB = g.KB, rs = g.rsz, lkb = log2_of(KB);
    const int kx = blockIdx.x, ky0 = blockIdx.y * KB;
    const int kb = min(KB, Py - ky0);
    TW *tw = reinterpret_cast<TW *>(S + 3 * KB * rs);
    load_twiddles_async(tw, P.tw_pz, Pz, Pz, tid, nth);
    FxMags<NS> mags;
    const int *scales = nullptr;
    if constexpr (FX) {
        if (tid < NS) { s_e[tid] = FX_ZERO; s_top[tid] = FX_ZERO; }
        if (tid < 3 * NS + 1) s_r[tid] = 0;
        __syncthreads();
        scales = P.fea + (long)kx * g.nzb * NS;
        fx_cta_scales<NS>(scales, g.nzb, NS, tid, nth, s_e, s_fl);
        __syncthreads();
    }
    // i = z * kb + kyl: a whole block of KB = 2^lkb frequencies, or the last one
    auto split = [&](int i, int &kyl, int &z) {
        if (kb == KB) { z = i >> lkb; kyl = i & (KB - 1); }
        else { z = i / kb; kyl = i - z * kb; }
    };
    // W2[kx][z][ky0 + kyl][c], z < nz -> row (c, kyl), element z; PF loads
    // per thread in flight before use
    V *base = P.W2 + ((long)kx * nz * Py + ky0) * 3;
    const long zs = (long)Py * 3;
    constexpr int PF = sizeof(T) == 4 ? 8 : 4;
    const int tot = nz * kb * 3;
    for (int e0 = tid; e0 < tot; e0 += PF * nth) {
        V v[PF];
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int e = e0 + i * nth;
            if (e < tot) {
                const int c = e % 3;
                int kyl, z;
                split(e / 3, kyl, z);
                v[i] = load_cg(base + (long)z * zs + kyl * 3 + c);
            }
        }
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int e = e0 + i * nth;
            if (e >= tot) break;
            const int c = e % 3;
            int kyl, z;
            split(e / 3, kyl, z);
            if constexpr (FX) {
                v[i] = fx_down(v[i], s_e[SEP ? c : 0] - fx_exp(scales[(z >> log2_of(g.ZB)) * NS + (SEP ? c : 0)]));
                mags.or_in(c, fx_mag(v[i]));
            }
            S[(c * KB + kyl) * rs + rpos<V, LZ>(z)] = v[i];
        }
    }
    const int npad = Pz - nz;
    for (int e = tid; e < 3 * KB * npad; e += nth) {
        const int r = g.fd_padz.div(e), z = nz + (e - r * npad);
        S[r * rs + rpos<V, LZ>(z)] = czero<V>();
    }
    if constexpr (FX) mags.cta_or(s_in);
    cp_async_wait_all();
    __syncthreads();
    const int Gz = g.Gz, RB = g.RBZ;
    const int rb = tid / Gz, j = tid - rb * Gz;
    signed char *s_sc = reinterpret_cast<signed char *>(tw + tw_slots(Pz));  // [2][NS][KB][Pz]: scale and top bit of a frequency
    signed char *s_tk = s_sc + NS * KB * Pz;
    int sh = 0, pre[NS], t[NS], post[NS];
    if constexpr (FX) {
#pragma unroll
        for (int c = 0; c < NS; ++c) pre[c] = 59 - fx_bits(s_in[c]);
    }
    for (int r0 = 0; r0 < 3 * KB; r0 += RB) {
        const int r = r0 + rb;
        const bool act = rb < RB && r < 3 * KB && (r % KB) < kb;
        if constexpr (FX) {
            unsigned none = 0;
            sh = fft_row_fx<false, true, false, 1, LZ, false>(S + (act ? r : 0) * rs, Pz, g.lpz, j, tw, act,
                                                              fx_of(pre, act ? r >> lkb : 0), 64, none);
        } else {
            fft_row<false, true, false, 1, LZ>(S + (act ? r : 0) * rs, Pz, g.lpz, j, tw, act);
        }
    }
    __syncthreads();
    int eb[NS], d[NS], top[NS];   // a component's scale where it is mixed, its own over that, the largest output
    const FxCouple couple{g.nx > 1 && g.ny > 1, g.nx > 1 && nz > 1, g.ny > 1 && nz > 1};
    if constexpr (FX) {
#pragma unroll
        for (int c = 0; c < NS; ++c) {
            eb[c] = d[c] = s_e[c] - pre[c] + sh + (SEP ? g.tsc[c] : 0);
            top[c] = FX_ZERO;
        }
        couple.join(eb);
#pragma unroll
        for (int c = 0; c < NS; ++c) d[c] -= eb[c];
    }
    // tensor product per (ky, kz); octant storage [kx][kzr][kyr][6] with the
    // off-diagonal signs of the reflected frequencies
    const int hy = Py / 2, hz = Pz / 2;
    const typename coef<typename fft_of<T>::type>::type *Nk = P.Nhat + (long)kx * (hz + 1) * (hy + 1) * 6;
    for (int e = tid; e < kb * Pz; e += nth) {
        int kyl, kz;
        split(e, kyl, kz);
        const int ky = ky0 + kyl;
        const int kyr = ky <= hy ? ky : Py - ky, kzr = kz <= hz ? kz : Pz - kz;
        const auto *n6 = Nk + ((long)kzr * (hy + 1) + kyr) * 6;
        V *a0 = S + (0 * KB + kyl) * rs + rpos<V, LZ>(kz);
        V *a1 = S + (1 * KB + kyl) * rs + rpos<V, LZ>(kz);
        V *a2 = S + (2 * KB + kyl) * rs + rpos<V, LZ>(kz);
        if constexpr (FX) {
            // one scale per frequency and coupled components: inputs below 2^59, outputs below 2^59
            auto element = [&](int c, bool neg) {
                const int2 w = __ldg(reinterpret_cast<const int2 *>(n6 + c));
                return fxk(fxk(fxm{w.x, w.y}), neg);
            };
            const fxk k[6] = {element(0, false), element(1, false), element(2, false), element(3, ky > hy),
                              element(4, kz > hz), element(5, (ky > hy) != (kz > hz))};
            fxc m0 = *a0, m1 = *a1, m2 = *a2;
            auto mags_of = [](const fxc &x, const fxc &y, const fxc &z) {
                FxMags<NS> k;
                k.or_in(0, fx_mag(x)); k.or_in(1, fx_mag(y)); k.or_in(2, fx_mag(z));
                return k;
            };
            const FxMags<NS> mk = mags_of(m0, m1, m2);
            int sc[NS];
#pragma unroll
            for (int c = 0; c < NS; ++c) sc[c] = fx_bits(mk.v[c]) + d[c];
            couple.join(sc);
#pragma unroll
            for (int c = 0; c < NS; ++c) sc[c] = 59 - sc[c];
            constexpr int c1 = SEP ? 1 : 0, c2 = SEP ? 2 : 0;
            m0 = fx_scale(m0, sc[0] + d[0]); m1 = fx_scale(m1, sc[c1] + d[c1]); m2 = fx_scale(m2, sc[c2] + d[c2]);
            auto row = [&](const fxk &p, const fxk &q, const fxk &r, fx x, fx y, fx z) {
                fxdot h;
                h.zero();
                h.mad(fx_split(x), p);
                h.mad(fx_split(y), q);
                h.mad(fx_split(z), r);
                return h.value();
            };
            const fxc h0{row(k[0], k[3], k[4], m0.x, m1.x, m2.x), row(k[0], k[3], k[4], m0.y, m1.y, m2.y)};
            const fxc h1{row(k[3], k[1], k[5], m0.x, m1.x, m2.x), row(k[3], k[1], k[5], m0.y, m1.y, m2.y)};
            const fxc h2{row(k[4], k[5], k[2], m0.x, m1.x, m2.x), row(k[4], k[5], k[2], m0.y, m1.y, m2.y)};
            const FxMags<NS> hk = mags_of(h0, h1, h2);
#pragma unroll
            for (int c = 0; c < NS; ++c) {
                const int tk = fx_bits(hk.v[c]) - sc[c];
                s_sc[(c * KB + kyl) * Pz + kz] = (signed char)sc[c];
                s_tk[(c * KB + kyl) * Pz + kz] = (signed char)tk;
                top[c] = max(top[c], tk);
            }
            *a0 = h0; *a1 = h1; *a2 = h2;
        } else {
        const T sy = ky <= hy ? (T)1 : (T)-1, sz = kz <= hz ? (T)1 : (T)-1;
        // six floats from an 8-byte boundary
        const float2 *n2 = reinterpret_cast<const float2 *>(n6);
        const float2 n01 = __ldg(n2), n23 = __ldg(n2 + 1), n45 = __ldg(n2 + 2);
        const T nxx = n01.x, nyy = n01.y, nzz = n23.x;
        const T nxy = sy * n23.y, nxz = sz * n45.x, nyz = sy * sz * n45.y;
        const V m0 = *a0, m1 = *a1, m2 = *a2;
        V h0, h1, h2;
        h0.x = nxx * m0.x + nxy * m1.x + nxz * m2.x; h0.y = nxx * m0.y + nxy * m1.y + nxz * m2.y;
        h1.x = nxy * m0.x + nyy * m1.x + nyz * m2.x; h1.y = nxy * m0.y + nyy * m1.y + nyz * m2.y;
        h2.x = nxz * m0.x + nyz * m1.x + nzz * m2.x; h2.y = nxz * m0.y + nyz * m1.y + nzz * m2.y;
        *a0 = h0; *a1 = h1; *a2 = h2;
        }
    }
    if constexpr (FX) {
#pragma unroll
        for (int c = 0; c < NS; ++c) fx_cta_max(&s_top[c], top[c]);
    }
    __syncthreads();
    if constexpr (FX) {
        // no partial sum of an inverse transform exceeds the sum of the largest moduli over kz
        unsigned sum[NS];
#pragma unroll
        for (int c = 0; c < NS; ++c) sum[c] = 0;
        for (int e = tid; e < Pz; e += nth) {
#pragma unroll
            for (int c = 0; c < NS; ++c) {
                int tk = FX_ZERO;
                for (int kyl = 0; kyl < kb; ++kyl) tk = max(tk, (int)s_tk[(c * KB + kyl) * Pz + e]);
                sum[c] += ((1u << 18) >> min(s_top[c] - tk, 18)) + 1;
            }
        }
#pragma unroll
        for (int c = 0; c < NS; ++c) fx_cta_add(&s_sum[c], sum[c]);
        __syncthreads();
        mags = FxMags<NS>();
#pragma unroll
        for (int c = 0; c < NS; ++c) {
            pre[c] = 58 - s_top[c];
            t[c] = max(0, fx_log2_up(s_sum[c]) - 18);
        }
    }
    for (int r0 = 0; r0 < 3 * KB; r0 += RB) {
        const int r = r0 + rb;
        const bool act = rb < RB && r < 3 * KB && (r % KB) < kb;
        if constexpr (FX) {
            const int c = SEP && act ? r >> lkb : 0;
            unsigned mag = 0;
            fft_row_fx<true, false, true, 1, LZ, true, true>(S + (act ? r : 0) * rs, Pz, g.lpz, j, tw, act, fx_of(pre, c),
                                                             fx_of(t, c), mag,
                                                             s_sc + (c * KB + (act ? r & (KB - 1) : 0)) * Pz);
            mags.or_in(c, mag);
        } else {
            fft_row<true, false, true, 1, LZ>(S + (act ? r : 0) * rs, Pz, g.lpz, j, tw, act);
        }
    }
    if constexpr (FX) mags.cta_or(s_out);
    __syncthreads();
    if constexpr (FX) {
#pragma unroll
        for (int c = 0; c < NS; ++c) post[c] = 60 - fx_bits(s_out[c]);
        if (tid < NS) {
            const int c = tid, e = fx_of(eb, c) + P.fek[kx] + fx_cum(fx_log(Pz), fx_of(t, c)) - fx_of(pre, c) -
                                   fx_of(post, c) + (SEP ? g.tsc[c] : 0);
            P.feb[((long)kx * g.nkb + blockIdx.y) * NS + c] = fx_pack(e, *s_fl ? 1 : 0);  // the tensor mixes all components
        }
    }
    for (int e = tid; e < nz * kb * 3; e += nth) {
        const int c = e % 3;
        int kyl, z;
        split(e / 3, kyl, z);
        V r = S[(c * KB + kyl) * rs + rpos<V, LZ>(z)];
        if constexpr (FX) r = fx_scale(r, fx_of(post, c));
        base[(long)z * zs + kyl * 3 + c] = r;
    }
}

inline int round32(int n) { return (n + 31) & ~31; }

template <typename T> size_t smem_y_t(const Geom &g, int zb)
{
    typedef typename cvec<T>::type V;
    return ((size_t)3 * zb * g.rsy + tw_slots(g.Py)) * sizeof(V);
}
template <typename T> size_t smem_z_t(const Geom &g, int kb)
{
    typedef typename cvec<T>::type V;
    // and two bytes per frequency (and component) of a block fixed-point transform
    return ((size_t)3 * kb * g.rsz + tw_slots(g.Pz)) * sizeof(V) +
           (sizeof(T) == 8 ? (size_t)(g.sep ? 6 : 2) * kb * g.Pz : 0);
}

template <typename T> cudaError_t bulk_conv_t(const Geom &g, const FieldPtrs<T> &P, cudaStream_t s, int pass)
{
    const dim3 gy(g.C, (g.nz + g.ZB - 1) / g.ZB), gz(g.C, (g.Py + g.KB - 1) / g.KB);
    const int ty = round32(g.RBY * g.Gy), tz = round32(g.RBZ * g.Gz);
    const size_t sy = smem_y_t<T>(g, g.ZB), sz = smem_z_t<T>(g, g.KB);
    const int ly = lb_of(g.Py), lz = lb_of(g.Pz);
    if (pass < 0 || pass == 0) {
        switch (ly) {
#define C(L) case L: k_ypass<T, false, L><<<gy, ty, sy, s>>>(g, P); break;
            MM_LB_CASES(C)
#undef C
        default: return cudaErrorInvalidValue;
        }
    }
    if (pass < 0 || pass == 1) {
        if constexpr (sizeof(T) == 8) {
            if (g.sep) k_zconv<T, -1, true><<<gz, tz, sz, s>>>(g, P);  // rare: the code for any length
        }
        if (sizeof(T) == 4 || !g.sep) {
            switch (lz) {
#define C(L) case L: k_zconv<T, L, false><<<gz, tz, sz, s>>>(g, P); break;
                MM_LB_CASES(C)
#undef C
            default: return cudaErrorInvalidValue;
            }
        }
    }
    if (pass < 0 || pass == 2) {
        switch (ly) {
#define C(L) case L: k_ypass<T, true, L><<<gy, ty, sy, s>>>(g, P); break;
            MM_LB_CASES(C)
#undef C
        default: return cudaErrorInvalidValue;
        }
    }
    return cudaGetLastError();
}

// the bytes a launch needs must fit the common cap, which every kernel is given
template <typename F> cudaError_t smem_attr(F *f, size_t bytes)
{
    if (bytes > (size_t)MM_SMEM_CAP) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, MM_SMEM_CAP);
}

template <typename T> cudaError_t configure_t(const Geom &g)
{
    cudaError_t e = cudaSuccess;
    const size_t sy = smem_y_t<T>(g, g.ZB), sz = smem_z_t<T>(g, g.KB);
    switch (lb_of(g.Py)) {
#define C(L) case L: if ((e = smem_attr(k_ypass<T, false, L>, sy)) || (e = smem_attr(k_ypass<T, true, L>, sy))) return e; break;
        MM_LB_CASES(C)
#undef C
    }
    if constexpr (sizeof(T) == 8) {
        if (g.sep) return smem_attr(k_zconv<T, -1, true>, sz);
    }
    switch (lb_of(g.Pz)) {
#define C(L) case L: return smem_attr(k_zconv<T, L, false>, sz);
        MM_LB_CASES(C)
#undef C
    }
    return cudaErrorInvalidValue;
}

} // namespace

cudaError_t mm_bulk_conv(const Geom &g, const FieldPtrs<double> &P, cudaStream_t s, int pass)
{
    return bulk_conv_t<double>(g, P, s, pass);
}
cudaError_t mm_bulk_conv(const Geom &g, const FieldPtrs<float> &P, cudaStream_t s, int pass)
{
    return bulk_conv_t<float>(g, P, s, pass);
}

size_t mm_bulk_smem_y(const mm_problem *p, int zb)
{
    return p->precision == MM_FP64 ? smem_y_t<double>(p->g, zb) : smem_y_t<float>(p->g, zb);
}
size_t mm_bulk_smem_z(const mm_problem *p, int kb)
{
    return p->precision == MM_FP64 ? smem_z_t<double>(p->g, kb) : smem_z_t<float>(p->g, kb);
}
int mm_bulk_thread_bound(const mm_problem *p)
{
    return p->precision == MM_FP64 ? BulkBound<double>::v : BulkBound<float>::v;
}
int mm_bulk_thread_bound_y(const mm_problem *p)
{
    return p->precision == MM_FP64 ? Y_BOUND<double> : Y_BOUND<float>;
}
cudaError_t mm_bulk_configure(const mm_problem *p)
{
    return p->precision == MM_FP64 ? configure_t<double>(p->g) : configure_t<float>(p->g);
}

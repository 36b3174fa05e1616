// Block fixed-point arithmetic of the MM_FP64 and MM_F32X2 convolution: 64-bit integers
// with power-of-two scales per block of values (a row, an x-frequency), run on
// the integer pipes.
//
// Why: this GPU has 2 FP64 lanes per SM (measured 1.68 FMA per clock and SM),
// against 42 64-bit integer additions and 24-32 wide multiply-adds per clock
// and SM.  A radix-8 butterfly with its twiddles is 84 FP64 instructions, 50
// clocks of an SM, or about 6 clocks in this arithmetic.  Precision: an FFT's
// error is relative to the norm of its row, and a value here carries up to 58
// bits below the largest value of its block, where a double carries 53.
//
// A value is v * 2^e with e held per block.  Twiddles are multipliers of type
// fxm: hi * 2^32 + lo with a signed low word, in units of 2^-61.  Their
// products with a value leave out the low x low partial product, at most 2
// units of the result before its scaling, and are rounded.  The tensor is held
// in units of 2^-62 and multiplied exactly (fxdot).
// Bounds: values stay below 2^62 in magnitude wherever they are multiplied,
// and below 2^63 everywhere (see the callers' scaling).
#pragma once

#include <cuda_runtime.h>

// a value (aligned like the double it takes the place of)
struct __align__(8) fx {
    long long v;
    fx() = default;
    __host__ __device__ constexpr fx(long long x) : v(x) {}
    __host__ __device__ constexpr fx(int x) : v(x) {}
};
struct __align__(16) fxc {
    fx x, y;
};
// a multiplier: a twiddle in units of 2^-61 or a tensor element in units of 2^-62
struct __align__(8) fxm {
    int lo, hi;
};
struct __align__(16) fxmc {
    fxm x, y;
};

// The three components have scales of their own where they are not all mixed by
// the tensor, or unequally (Geom::sep): a component is then as accurate as its own size allows.
// (With one scale for the three, the in-plane field of a one-layer film
// magnetised along z with a tilt of 1e-8 was off by 1e-8 of itself.)  Where all
// are mixed, a field component gathers the rounding of the largest in any
// arithmetic, and they share one.
// Scale of a block as the kernels hand it on: e * 4 + flag.  Non-finite inputs
// have no place in a block; their component is taken as zero and flagged (1),
// and comes out as NaN where the field would.
#define FX_ZERO (-100000)   // exponent of an all-zero block
__host__ __device__ __forceinline__ constexpr int fx_pack(int e, int flags) { return e * 4 + flags; }
__host__ __device__ __forceinline__ constexpr int fx_exp(int p) { return p >> 2; }
__host__ __device__ __forceinline__ constexpr int fx_flags(int p) { return p & 3; }

__host__ __device__ constexpr fxm fx_multiplier(long long q)
{
    // signed low word, never -2^31, so that a multiplier can be negated word by word
    const int lo = (int)(unsigned)(unsigned long long)q;
    return lo == (int)0x80000000u ? fxm{lo + 1, (int)((q >> 32) + 1)} : fxm{lo, (int)((q - lo) >> 32)};
}

#ifdef __CUDACC__
// double-word value * 2^s, s = 58 - E, for |hi| <= (1 + 2^-8) 2^E, on the FP32
// pipes (f = 2^(30 - E)): the high part to 2^-28 of its integer unit exactly,
// the low part (at most 2^34 units) to a multiple of 16 units
__device__ __forceinline__ fx fx_from(dfloat a, float f)
{
    const float h = __fmul_rn(a.hi, f);
    const int i = __float2int_rn(h);
    const float rest = __fmul_rn(__fsub_rn(h, (float)i), 268435456.0f);                 // 2^28
    const float low = __fmul_rn(__fmul_rn(a.lo, f), 16777216.0f);                       // 2^24
    return fx(((long long)i << 28) + __float2int_rn(rest) + ((long long)__float2int_rn(low) << 4));
}
__device__ __forceinline__ fx operator+(fx a, fx b) { return fx(a.v + b.v); }
__device__ __forceinline__ fx operator-(fx a, fx b) { return fx(a.v - b.v); }
__device__ __forceinline__ fx operator-(fx a) { return fx(-a.v); }

// signed high word of the split v = hi * 2^32 + (signed) lo
__device__ __forceinline__ int fx_hi(fx a) { return (int)(a.v >> 32) + (int)((unsigned)a.v >> 31); }
__device__ __forceinline__ int fx_lo(fx a) { return (int)a.v; }

// sum of products of values and twiddles: P holds the high x high products
// (units of 2^64), c the cross products (units of 2^32)
struct fxacc {
    long long P, c;
    // value(sh) drops `sh` further bits (0..3): the rounding constant enters here
    __device__ __forceinline__ void zero(int sh) { P = 0; c = 1ll << (28 + sh); }
    __device__ __forceinline__ void mad(int ah, int al, int bh, int bl)
    {
        P += (long long)ah * bh;
        c += (long long)ah * bl;
        c += (long long)al * bh;
    }
    // (P 2^32 + c) >> (29 + sh)
    __device__ __forceinline__ fx value(int sh) const
    {
        const long long h = P + (c >> 32);
        const unsigned w0 = (unsigned)c, w1 = (unsigned)h, w2 = (unsigned)(h >> 32);
        const unsigned lo = __funnelshift_rc(w0, w1, 29 + sh), hi = __funnelshift_rc(w1, w2, 29 + sh);
        return fx((long long)(((unsigned long long)hi << 32) | lo));
    }
};

// a tensor element (units of 2^-62) split for fxdot, and its negative
struct fxk {
    int hi, lo, lo3;
    __device__ __forceinline__ explicit fxk(fxm k) : hi(k.hi), lo(k.lo), lo3(k.lo >> 3) {}
    __device__ __forceinline__ fxk(const fxk &k, bool neg)
        : hi(neg ? -k.hi : k.hi), lo(neg ? -k.lo : k.lo), lo3(neg ? -k.lo3 : k.lo3) {}
};
// sum of up to 8 products of values below 2^60 and tensor elements, the low x
// low products included (q, in units of 2^-27 of a unit)
struct fxdot {
    long long P, c;
    int q;
    __device__ __forceinline__ void zero() { P = 0; c = 1ll << 29; q = 0; }
    __device__ __forceinline__ void mad(int2 a, const fxk &b)  // a: (low, high) words of a split value
    {
        P += (long long)a.y * b.hi;
        c += (long long)a.y * b.lo;
        c += (long long)a.x * b.hi;
        q += __mulhi(a.x, b.lo3);
    }
    __device__ __forceinline__ fx value() const
    {
        const long long d = c + ((long long)q << 3), h = P + (d >> 32);
        const unsigned w0 = (unsigned)d, w1 = (unsigned)h, w2 = (unsigned)(h >> 32);
        const unsigned lo = __funnelshift_r(w0, w1, 30), hi = __funnelshift_r(w1, w2, 30);
        return fx((long long)(((unsigned long long)hi << 32) | lo));
    }
};
__device__ __forceinline__ int2 fx_split(fx a) { return make_int2(fx_lo(a), fx_hi(a)); }

// a * b for a constant b, |b| <= 1 (rounded)
__device__ __forceinline__ fx fx_mulc(fxm b, fx a)
{
    fxacc s;
    s.zero(0);
    s.mad(fx_hi(a), fx_lo(a), b.hi, b.lo);
    return s.value(0);
}

// a * w (CONJ: a * conj(w)) divided by 2^sh, sh in 0..3
template <bool CONJ> __device__ __forceinline__ fxc fx_cmul(fxc a, fxmc w, int sh)
{
    const int xh = fx_hi(a.x), xl = fx_lo(a.x), yh = fx_hi(a.y), yl = fx_lo(a.y);
    fxacc re, im;
    re.zero(sh);
    im.zero(sh);
    re.mad(xh, xl, w.x.hi, w.x.lo);
    im.mad(yh, yl, w.x.hi, w.x.lo);
    if (CONJ) {
        re.mad(yh, yl, w.y.hi, w.y.lo);
        im.mad(xh, xl, -w.y.hi, -w.y.lo);
    } else {
        re.mad(yh, yl, -w.y.hi, -w.y.lo);
        im.mad(xh, xl, w.y.hi, w.y.lo);
    }
    fxc r;
    r.x = re.value(sh);
    r.y = im.value(sh);
    return r;
}

// v / 2^s rounded to nearest, ties to even, s >= 0: rounding ties up shifts the mean of a row by up to a quarter of a
// unit, which the next transform gathers in one cell
__device__ __forceinline__ fx fx_shr(fx a, int s)
{
    return s ? fx((a.v + ((1ll << (s - 1)) - 1) + ((a.v >> s) & 1)) >> s) : a;
}
// v * 2^d, d of either sign (uniform over a block); large right shifts give 0
__device__ __forceinline__ fx fx_scale(fx a, int d)
{
    if (d >= 0) return fx(a.v << d);
    return d > -62 ? fx_shr(a, -d) : fx(0);
}
__device__ __forceinline__ fxc fx_scale(fxc a, int d)
{
    fxc r;
    r.x = fx_scale(a.x, d);
    r.y = fx_scale(a.y, d);
    return r;
}
// v / 2^s rounded, s >= 0 (fx_scale's right shift alone: half the code where small
// films wait for instructions)
__device__ __forceinline__ fxc fx_down(fxc a, int s)
{
    if (s == 0) return a;
    if (s > 61) return fxc{fx(0), fx(0)};
    return fxc{fx_shr(a.x, s), fx_shr(a.y, s)};
}
// bits of the high word's magnitude, to be OR-ed over a block; with b the
// number of bits of the result, every |v| of the block is below 2^(32 + b) + 1
__device__ __forceinline__ unsigned fx_mag(fx a)
{
    const int h = (int)(a.v >> 32);
    return (unsigned)(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned fx_mag(fxc a) { return fx_mag(a.x) | fx_mag(a.y); }
// v * f as a double-word, f a power of two: the high word's leading 24 bits,
// then what they leave with the low word
__device__ __forceinline__ dfloat fx_to_dfloat(fx a, float f)
{
    const int h = fx_hi(a);
    const float top = (float)h;
    const float rest = fmaf((float)(h - (int)top), 4294967296.0f, (float)fx_lo(a));     // 2^32
    return df_fast2sum(__fmul_rn(__fmul_rn(top, 65536.0f), __fmul_rn(f, 65536.0f)), __fmul_rn(rest, f));
}

// OR (or maximum, or sum) over the CTA into *dst in shared memory; a barrier makes it visible
__device__ __forceinline__ void fx_cta_or(unsigned *dst, unsigned v)
{
    v = __reduce_or_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0 && v) atomicOr(dst, v);
}
__device__ __forceinline__ void fx_cta_max(int *dst, int v)
{
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMax(dst, v);
}
__device__ __forceinline__ void fx_cta_add(unsigned *dst, unsigned v)
{
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicAdd(dst, v);
}
// N = 3: one value per component, added to by component number; N = 1: one for all
template <int N> struct FxMags {
    unsigned v[N];
    __device__ __forceinline__ FxMags()
    {
#pragma unroll
        for (int c = 0; c < N; ++c) v[c] = 0;
    }
    __device__ __forceinline__ void or_in(int c, unsigned x)
    {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] |= N == 1 || c == i ? x : 0;
    }
    __device__ __forceinline__ void cta_or(unsigned *dst) const
    {
#pragma unroll
        for (int c = 0; c < N; ++c) fx_cta_or(dst + c, v[c]);
    }
};
// element c of a register array (N = 1: the one for all components)
template <int N> __device__ __forceinline__ int fx_of(const int (&a)[N], int c)
{
    if constexpr (N == 1) return a[0];
    else return c == 0 ? a[0] : (c == 1 ? a[1] : a[2]);
}
// Largest exponents and the flags (bit c) of the scales p[i * stride + c], i < n,
// c < N, over the CTA; a barrier makes them visible
template <int N> __device__ __forceinline__ void fx_cta_scales(const int *p, int n, long stride, int tt, int nth, int *s_e,
                                                               unsigned *s_fl)
{
    int e[N];
#pragma unroll
    for (int c = 0; c < N; ++c) e[c] = FX_ZERO;
    unsigned fl = 0;
    for (int i = tt; i < n; i += nth) {
#pragma unroll
        for (int c = 0; c < N; ++c) {
            const int q = p[i * stride + c];
            e[c] = max(e[c], fx_exp(q));
            fl |= (unsigned)fx_flags(q) << c;
        }
    }
#pragma unroll
    for (int c = 0; c < N; ++c) fx_cta_max(s_e + c, e[c]);
    fx_cta_or(s_fl, fl);
}
// Components that the tensor couples (pairs of axes that both have more than
// one cell) share a scale where they are mixed: the largest of theirs.  All
// pairs are coupled, one, or none.
struct FxCouple {
    bool xy, xz, yz;
    __device__ __forceinline__ void join(int (&e)[3]) const
    {
        const int a = e[0], b = e[1], c = e[2];
        e[0] = max(a, max(xy ? b : a, xz ? c : a));
        e[1] = max(b, max(xy ? a : b, yz ? c : b));
        e[2] = max(c, max(xz ? a : c, yz ? b : c));
    }
    __device__ __forceinline__ void join(int (&)[1]) const {}
};
// least t >= 0 with 2^t >= v
__device__ __forceinline__ int fx_log2_up(unsigned v) { return v > 1 ? 32 - __clz((int)(v - 1)) : 0; }
__device__ __forceinline__ int fx_bits(unsigned mag) { return 64 - __clz((int)mag); }  // 32 + bits of mag

__device__ __forceinline__ float fx_pow2f(int e)
{
    return e < -126 ? 0.0f : __int_as_float((min(e, 127) + 127) << 23);
}
// x * 2^e by its exponent bits; 0 for results below the normal numbers (and for x = 0)
__device__ __forceinline__ double fx_ldexp(double x, int e)
{
    const int hi = __double2hiint(x), old = (hi >> 20) & 0x7ff;
    return old == 0 || old + e <= 0 ? 0.0 : __hiloint2double(hi + (e << 20), __double2loint(x));
}
// 2^e as a double, 0 below the smallest normal power
__device__ __forceinline__ double fx_pow2(int e)
{
    if (e < -1022) return 0.0;
    return __longlong_as_double((long long)(min(e, 1023) + 1023) << 52);
}
#endif

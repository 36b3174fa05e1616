// Shared-memory FFT building blocks for the zero-padded demagnetisation
// convolution (the "FFT accelerated convolution" of Section 3).
//
// A row of L complex values, L = 2^l or 2^l times 3, 5 or 25 with l >= 3,
// lives in shared memory and is transformed in place by G = max(1, L/8)
// threads with self-sorting Stockham passes (Stockham; Cochran et al., Proc.
// IEEE 55 (1967) 1664): an optional first pass of radix 2 or 4, then radix-8
// passes, then the odd radices.  Each thread keeps one radix-8 butterfly (or
// two radix-4 or -5, three radix-3, four radix-2 ones) in registers per pass;
// a barrier separates the loads of a pass from its stores, which makes the
// in-place update safe.  Twiddles come from a table tw[t] = exp(-2 pi i t/L')
// read with stride ts = L'/L.
//
// Zero padding is exploited where the convolution needs it:
//  HALF_IN : the upper half of the input is known to be zero, so the first
//            pass reads half of its inputs and skips the arithmetic on zeros;
//  HALF_OUT: only the lower half of the output is wanted, so the last pass
//            computes and stores only those values.
#pragma once

#include "common.cuh"

template <typename V> __device__ __forceinline__ V czero() { V r; r.x = 0; r.y = 0; return r; }

// Rows in shared memory are stored with one padding element after every 8:
// element i lives at pidx(i).  Stockham stores of radix 8 and strides 1 or 8
// then spread over all banks instead of hitting one bank group.
__host__ __device__ __forceinline__ int pidx(int i) { return i + (i >> 3); }
// shared-memory footprint (elements) of a padded row of length L, plus one
// element so that consecutive rows start in different banks
__host__ __device__ __forceinline__ int padded_row(int L) { return L + (L >> 3) + 1; }

// Row layout by element size.  16-byte elements (double2) use the padding
// above: each Stockham pass then takes the minimum number of shared-memory
// wavefronts.  8-byte elements (float2) are served 16 per wavefront; with
// the padding a warp's 32 consecutive elements span 36 slots, which costs 3
// to 4 wavefronts instead of 2.  They use an XOR swizzle instead, within
// aligned groups of 16 elements: bits 4-6 of the index are XORed into
// bits 0-3 (bit 6 into bit 3).  In a bank simulation of the radix-8
// Stockham passes this keeps unit-stride loads, the stride-8 stores of the
// first pass and the grouped stores of the later passes at 2 wavefronts
// (L = 512, 4096).  It is a permutation of every aligned group of 16, so a
// row of L elements needs only L slots, plus one between rows.
// Block fixed-point rows (16-byte elements, 8 per wavefront) are swizzled
// within aligned groups of 8 for the same reason, which leaves room for the
// twiddles of the y-z kernel beside its rows: 12 rows of 512 and the table take
// 105 KiB, two CTAs an SM.
template <typename V> __host__ __device__ __forceinline__ int spos(int i)
{
    if constexpr (std::is_same<V, fxc>::value) return i ^ ((i >> 3) & 7);
    else if constexpr (sizeof(V) == 8) return i ^ (((i >> 4) & 7) | (((i >> 6) & 1) << 3));
    else return i + (i >> 3);
}
// (rows of a length with an odd part are padded like 16-byte ones: rpos)
__host__ __device__ __forceinline__ int row_stride(int L, int esz)
{
    return esz == 8 && (L & (L - 1)) == 0 ? L + 1 : padded_row(L);
}
// Element i of a row of a kernel compiled for LC.  The swizzle of a power of two
// is linear over XOR, so a pass takes one XOR per access.  A length with an odd
// part has offsets that share bits, which costs about five integer instructions an
// access, in kernels bound by those; padding has constant offsets there.  160^3
// cells, FP32 z pass: 533 us swizzled and with divisions by runtime block sizes, 445 without both.
template <typename V, int LC> __host__ __device__ __forceinline__ int rpos(int i)
{
    if constexpr (sizeof(V) == 8 && LC > 16) return pidx(i);
    else return spos<V>(i);
}

// the same for block fixed-point rows
__host__ __device__ __forceinline__ int row_stride_fx(int L) { return (L <= 8 ? L : (L + 7) / 8 * 8) + 1; }

// L = 2^l (times an odd part): l
__host__ __device__ constexpr int pow2_part(int L)
{
    int l = 0;
    while (!((L >> l) & 1)) ++l;
    return l;
}

// Twiddle t of a table in shared memory lives at tpos(t, L), L the row length.
// A pass reads multiples of L/(Ns R) r; unswizzled, the eight different ones of
// a pass with Ns = 8 over a power of two lie 128 bytes apart, in one bank group
// (512 x 256 x 4, two measurements: FP32 y-z kernel 37 and 38.5 -> 32.5 us,
// x-forward 20.7 and 20.4 -> 19.5 us).  Lengths with an odd part
// spread by themselves.  Double tables (the tensor setup) stay in global
// memory, in order.
template <typename W> __host__ __device__ __forceinline__ int tpos(int t, int L)
{
    if constexpr (std::is_same<W, double2>::value) return t;
    else if (L & (L - 1)) return t;
    else if constexpr (std::is_same<W, fxmc>::value) return spos<fxc>(t);
    else return spos<W>(t);
}

// slots of such a table of n: whole swizzle groups
__host__ __device__ constexpr int tw_slots(int n) { return n <= 16 ? n : (n + 15) / 16 * 16; }

// copy a twiddle table of n complex values for rows of length L into shared memory (threads tid of
// nth), issued as asynchronous copies (8 or 16 bytes per element); complete at cp_async_wait_all() of each thread, then a barrier
template <typename W>
__device__ __forceinline__ void load_twiddles_async(W *dst, const W *src, int n, int L, int tid, int nth)
{
    for (int i = tid; i < n; i += nth) {
        if constexpr (sizeof(W) == 16) cp_async16(dst + tpos<W>(i, L), src + i);
        else cp_async8(dst + tpos<W>(i, L), src + i);
    }
}

// 2-point DFT
template <bool HIN, typename V> __device__ __forceinline__ void dft2(V &a0, V &a1)
{
    if (HIN) { a1 = a0; return; }
    V t = a0;
    a0 = cadd(t, a1);
    a1 = csub(t, a1);
}

// 4-point DFT, forward uses -i, inverse +i; outputs in natural order
template <bool INV, bool HIN, typename V> __device__ __forceinline__ void dft4(V &x0, V &x1, V &x2, V &x3)
{
    V t0, t1, t2, t3;
    if (HIN) {           // x2 = x3 = 0
        t0 = x0; t1 = x0; t2 = x1; t3 = cmul_mi<INV>(x1);
    } else {
        t0 = cadd(x0, x2); t1 = csub(x0, x2);
        t2 = cadd(x1, x3); t3 = cmul_mi<INV>(csub(x1, x3));
    }
    x0 = cadd(t0, t2);
    x2 = csub(t0, t2);
    x1 = cadd(t1, t3);
    x3 = csub(t1, t3);
}

// 8-point DFT by one radix-2 decimation-in-frequency split into two 4-point
// DFTs: u_n = a_n + a_{n+4}, v_n = (a_n - a_{n+4}) W^n, X_{2k} = DFT4(u)_k,
// X_{2k+1} = DFT4(v)_k, W = exp(-+ i pi/4).
template <bool INV, bool HIN, typename V> __device__ __forceinline__ void dft8(V *a)
{
    typedef decltype(a[0].x) T;
    const T r = (T)0.70710678118654752440084436210484903928;
    V u0, u1, u2, u3, d0, d1, d2, d3;
    if (HIN) {
        u0 = a[0]; u1 = a[1]; u2 = a[2]; u3 = a[3];
        d0 = a[0]; d1 = a[1]; d2 = a[2]; d3 = a[3];
    } else {
        u0 = cadd(a[0], a[4]); d0 = csub(a[0], a[4]);
        u1 = cadd(a[1], a[5]); d1 = csub(a[1], a[5]);
        u2 = cadd(a[2], a[6]); d2 = csub(a[2], a[6]);
        u3 = cadd(a[3], a[7]); d3 = csub(a[3], a[7]);
    }
    V v1, v2, v3;
    if (INV) {
        v1.x = r * (d1.x - d1.y); v1.y = r * (d1.x + d1.y);
        v2.x = -d2.y;             v2.y = d2.x;
        v3.x = -r * (d3.x + d3.y); v3.y = r * (d3.x - d3.y);
    } else {
        v1.x = r * (d1.x + d1.y); v1.y = r * (d1.y - d1.x);
        v2.x = d2.y;              v2.y = -d2.x;
        v3.x = r * (d3.y - d3.x); v3.y = -r * (d3.x + d3.y);
    }
    dft4<INV, false>(u0, u1, u2, u3);
    dft4<INV, false>(d0, v1, v2, v3);
    a[0] = u0; a[1] = d0; a[2] = u1; a[3] = v1;
    a[4] = u2; a[5] = v2; a[6] = u3; a[7] = v3;
}

template <int R, bool INV, bool HIN, typename V> __device__ __forceinline__ void dftR(V *a)
{
    if constexpr (R == 2) dft2<HIN>(a[0], a[1]);
    else if constexpr (R == 4) dft4<INV, HIN>(a[0], a[1], a[2], a[3]);
    else dft8<INV, HIN>(a);
}

// r times i (inverse) or -i (forward) added to and taken from u: the outputs
// n and R - n of an odd-length DFT
template <bool INV, typename V> __device__ __forceinline__ void odd_pair(V u, V r, V &lo, V &hi)
{
    const V w = cmul_mi<INV>(r);
    lo = cadd(u, w);
    hi = csub(u, w);
}
template <typename V, typename T> __device__ __forceinline__ V caxpy(V a, T c, V b)
{
    V r;
    r.x = a.x + c * b.x;
    r.y = a.y + c * b.y;
    return r;
}
// 3-point and 5-point DFTs from the sums and differences of a_n and a_{R-n}
template <bool INV, typename V> __device__ __forceinline__ void dft3(V *a)
{
    typedef decltype(a[0].x) T;
    const T s = (T)0.86602540378443864676372317075294;
    const V t = cadd(a[1], a[2]), d = csub(a[1], a[2]);
    const V u = caxpy(a[0], (T)-0.5, t);
    V r;
    r.x = s * d.x; r.y = s * d.y;
    a[0] = cadd(a[0], t);
    odd_pair<INV>(u, r, a[1], a[2]);
}
template <bool INV, typename V> __device__ __forceinline__ void dft5(V *a)
{
    typedef decltype(a[0].x) T;
    const T c1 = (T)0.30901699437494742410229341718282, c2 = (T)-0.80901699437494742410229341718282;
    const T s1 = (T)0.95105651629515357211643933337938, s2 = (T)0.58778525229247312916870595463907;
    const V t1 = cadd(a[1], a[4]), t2 = cadd(a[2], a[3]), d1 = csub(a[1], a[4]), d2 = csub(a[2], a[3]);
    const V u1 = caxpy(caxpy(a[0], c1, t1), c2, t2), u2 = caxpy(caxpy(a[0], c2, t1), c1, t2);
    V r1, r2;
    r1.x = s1 * d1.x + s2 * d2.x; r1.y = s1 * d1.y + s2 * d2.y;
    r2.x = s2 * d1.x - s1 * d2.x; r2.y = s2 * d1.y - s1 * d2.y;
    a[0] = cadd(a[0], cadd(t1, t2));
    odd_pair<INV>(u1, r1, a[1], a[4]);
    odd_pair<INV>(u2, r2, a[2], a[3]);
}

// One Stockham pass of odd radix R (3 or 5) over a row of length L: L/R
// butterflies, thread j takes j, j + G, ...  Ns is a power of two or L/R.  With
// HOUT only the outputs below L/2 are stored.
template <int R, bool INV, bool HOUT, typename V>
__device__ __forceinline__ void stockham_odd(V *row, int L, int Ns, int j, int G, const V *__restrict__ tw, int ts,
                                             bool active)
{
    constexpr int NB = (8 + R - 1) / R;
    V v[NB * R];
#pragma unroll
    for (int i = 0; i < NB * R; ++i) v[i] = czero<V>();
    const int LR = L / R, tstep0 = (L / (Ns * R)) * ts;
    if (active) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int b = j + q * G;
            if (b >= LR) break;
            const int step = tstep0 * (Ns == LR ? b : b & (Ns - 1));
#pragma unroll
            for (int r = 0; r < R; ++r) {
                v[q * R + r] = row[(LR & 7) ? pidx(b + r * LR) : pidx(b) + r * (LR + (LR >> 3))];
                if (r > 0) {
                    const V w = tw[tpos<V>(r * step, L)];
                    v[q * R + r] = INV ? cmulc(v[q * R + r], w) : cmul(v[q * R + r], w);
                }
            }
            if constexpr (R == 3) dft3<INV>(&v[q * R]);
            else dft5<INV>(&v[q * R]);
        }
    }
    __syncthreads();
    if (active) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int b = j + q * G;
            if (b >= LR) break;
            const int k = Ns == LR ? b : b & (Ns - 1);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i0 = (b - k) * R + k, i = i0 + r * Ns;
                if (!HOUT || 2 * i < L) row[(Ns & 7) ? pidx(i) : pidx(i0) + r * (Ns + (Ns >> 3))] = v[q * R + r];
            }
        }
    }
    __syncthreads();
}

// One Stockham pass of radix R over a row of length L (Ns = product of the
// radices of the previous passes).  Thread j handles butterflies j + q G,
// q < 8/R.  Caller guarantees visibility of the row before the call; the
// pass ends with a barrier.
//
// Padded offsets in closed form (Ns, R, LR = L/R powers of two): butterfly b
// reads elements b + r LR, whose padded offsets are pidx(b) + r (LR + LR/8)
// when 8 divides LR; it writes elements (b - k) R + k + r Ns, k = b mod Ns,
// whose padded offsets are 9 (b - k) + k + k/8 + r Ns + (r Ns)/8 for R = 8
// (and likewise with (b - k) R for R < 8), since k < Ns and Ns divides or is
// a multiple of 8.
template <int R, bool INV, bool HIN, bool HOUT, bool PAD = false, typename V>
__device__ __forceinline__ void stockham_pass(V *row, int L, int Ns, int j, int G,
                                              const V *__restrict__ tw, int ts, bool active)
{
    constexpr int NB = 8 / R;
    constexpr bool XOR = sizeof(V) == 8 && !PAD;   // a swizzled float row (PAD: length with an odd part)
    V v[8];
    const int LR = L / R;
    const int ld9 = LR + (LR >> 3);       // padded stride between the inputs of a butterfly (8 | LR)
    const int tstep0 = (L / (Ns * R)) * ts;
    if (active) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int b = j + q * G;
            const int p0 = XOR ? spos<V>(b) : pidx(b);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (HIN && r >= R / 2) { v[q * R + r] = czero<V>(); continue; }
                if constexpr (XOR) v[q * R + r] = row[p0 ^ spos<V>(r * LR)];   // b < LR
                else v[q * R + r] = row[(LR & 7) ? pidx(b + r * LR) : p0 + r * ld9];
            }
            if (Ns > 1) {
                const int step = tstep0 * (b & (Ns - 1));
                int t = step;
#pragma unroll
                for (int r = 1; r < R; ++r, t += step) {
                    const V w = tw[tpos<V>(t, L)];
                    v[q * R + r] = INV ? cmulc(v[q * R + r], w) : cmul(v[q * R + r], w);
                }
            }
            dftR<R, INV, HIN>(&v[q * R]);
        }
    } else {
        // (defined for idle threads too: in a loop over rows an undefined value would be carried round it, 32 registers
        // and more a pass)
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = czero<V>();
    }
    __syncthreads();
    if (active) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int b = j + q * G;
            const int k = b & (Ns - 1);
            const int hi = (b - k) * R;                  // multiple of 8 when R == 8
            const int s0 = XOR ? spos<V>(hi + k) : ((R == 8) ? hi + (hi >> 3) + k + (k >> 3) : 0);
#pragma unroll
            for (int r = 0; r < (HOUT ? R / 2 : R); ++r) {
                const int rn = r * Ns;
                if constexpr (XOR) row[s0 ^ spos<V>(rn)] = v[q * R + r];       // hi + k has no bits of rn
                else row[(R == 8) ? s0 + rn + (rn >> 3) : pidx(hi + k + rn)] = v[q * R + r];
            }
        }
    }
    __syncthreads();
}

// In-place FFT of one shared-memory row of length L, 2^logL times 1, 3, 5 or
// 25 (forward: exp(-i...), inverse: exp(+i...), unnormalised).  Every thread of the CTA
// must call this with the same L (it contains barriers); thread j in [0, G)
// of the row's group works on it.  Threads with active == false (padding
// threads of the CTA) only take part in the barriers.  The caller
// synchronises before the call so that the row's contents are visible; the
// row is final after return.  Twiddles: tw[t * TS] = exp(-2 pi i t / L).
//
// fft_row_n takes L at run time; fft_row_c<LOGL> is the same sequence of
// passes with L a compile-time constant, so that every offset, stride and
// pass count folds into the instructions.  Kernels are instantiated for the
// common lengths (template parameter LC of fft_row) and the host launches
// the matching instance.
template <bool INV, bool HIN, bool HOUT, int TS, bool ODD, typename V>
__device__ __forceinline__ void fft_row_n(V *row, int L, int logL, int j, const V *__restrict__ tw, bool active)
{
    if (L == 1) return;
    if (L < 8) {
        // G == 1: the single thread of the row does the whole transform.  The
        // barriers stay outside the branches so that every thread of a warp
        // executes the same barrier instruction.
        V a[4];
        if (active) {
            a[0] = row[0];
            a[1] = (HIN && L == 2) ? czero<V>() : row[1];
            if (L == 2) {
                dft2<HIN>(a[0], a[1]);
            } else {
                a[2] = HIN ? czero<V>() : row[2];
                a[3] = HIN ? czero<V>() : row[3];
                dft4<INV, HIN>(a[0], a[1], a[2], a[3]);
            }
        }
        __syncthreads();
        if (active) {
            row[0] = a[0];
            if (L == 2) {
                if (!HOUT) row[1] = a[1];
            } else {
                row[1] = a[1];
                if (!HOUT) { row[2] = a[2]; row[3] = a[3]; }
            }
        }
        __syncthreads();
        return;
    }
    const int G = L >> 3;
    const int rem = logL % 3;
    const int n8 = logL / 3;
    int odd = ODD ? L >> logL : 1;
    int Ns = 1;
    bool first = true;
    if (rem == 1) {
        stockham_pass<2, INV, HIN, false>(row, L, Ns, j, G, tw, TS, active);
        Ns = 2; first = false;
    } else if (rem == 2) {
        stockham_pass<4, INV, HIN, false>(row, L, Ns, j, G, tw, TS, active);
        Ns = 4; first = false;
    }
    for (int p = 0; p < n8; ++p) {
        const bool last = (p == n8 - 1) && odd == 1;
        if (first && HIN) {
            if (last && HOUT) stockham_pass<8, INV, true, true>(row, L, Ns, j, G, tw, TS, active);
            else stockham_pass<8, INV, true, false>(row, L, Ns, j, G, tw, TS, active);
        } else {
            if (last && HOUT) stockham_pass<8, INV, false, true>(row, L, Ns, j, G, tw, TS, active);
            else stockham_pass<8, INV, false, false>(row, L, Ns, j, G, tw, TS, active);
        }
        Ns <<= 3;
        first = false;
    }
    if constexpr (ODD) {
        if (odd == 25) {
            stockham_odd<5, INV, false>(row, L, Ns, j, G, tw, TS, active);
            Ns *= 5;
            odd = 5;
        }
        if (odd == 5) stockham_odd<5, INV, HOUT>(row, L, Ns, j, G, tw, TS, active);
        else if (odd == 3) stockham_odd<3, INV, HOUT>(row, L, Ns, j, G, tw, TS, active);
    }
}

template <int L, bool INV, bool HIN, bool HOUT, int TS, typename V>
__device__ __forceinline__ void fft_row_c(V *row, int j, const V *__restrict__ tw, bool active)
{
    static_assert(L >= 8 && L % 8 == 0, "compile-time rows have at least 8 elements");
    constexpr int LOGL = pow2_part(L), odd = L >> LOGL, G = L >> 3, rem = LOGL % 3, n8 = LOGL / 3;
    constexpr int NS0 = rem == 1 ? 2 : (rem == 2 ? 4 : 1);
    if constexpr (rem == 1) stockham_pass<2, INV, HIN, false, (odd > 1)>(row, L, 1, j, G, tw, TS, active);
    if constexpr (rem == 2) stockham_pass<4, INV, HIN, false, (odd > 1)>(row, L, 1, j, G, tw, TS, active);
#pragma unroll
    for (int p = 0; p < n8; ++p) {
        const int Ns = NS0 << (3 * p);
        const bool last = (p == n8 - 1) && odd == 1, first = (p == 0 && rem == 0);
        if (first && HIN) {
            if (last && HOUT) stockham_pass<8, INV, true, true, (odd > 1)>(row, L, Ns, j, G, tw, TS, active);
            else stockham_pass<8, INV, true, false, (odd > 1)>(row, L, Ns, j, G, tw, TS, active);
        } else {
            if (last && HOUT) stockham_pass<8, INV, false, true, (odd > 1)>(row, L, Ns, j, G, tw, TS, active);
            else stockham_pass<8, INV, false, false, (odd > 1)>(row, L, Ns, j, G, tw, TS, active);
        }
    }
    if constexpr (odd == 25) stockham_odd<5, INV, false>(row, L, L / 25, j, G, tw, TS, active);
    if constexpr (odd == 25 || odd == 5) stockham_odd<5, INV, HOUT>(row, L, L / 5, j, G, tw, TS, active);
    if constexpr (odd == 3) stockham_odd<3, INV, HOUT>(row, L, L / 3, j, G, tw, TS, active);
}

// LC > 0: the kernel was compiled for rows of length 2^LC, or LC above 16
// (L, logL unused); LC == 0: any power of two; LC == -1: any length
constexpr int fft_length(int LC) { return LC > 16 ? LC : 1 << LC; }
template <bool INV, bool HIN, bool HOUT, int TS, int LC, typename V>
__device__ __forceinline__ void fft_row(V *row, int L, int logL, int j, const V *__restrict__ tw, bool active)
{
    if constexpr (LC > 0) fft_row_c<fft_length(LC), INV, HIN, HOUT, TS>(row, j, tw, active);
    else fft_row_n<INV, HIN, HOUT, TS, LC < 0>(row, L, logL, j, tw, active);
}

// ---------------------------------------------------------------------------
// The same transforms in block fixed point (fixed.cuh)
// ---------------------------------------------------------------------------
// Scaling: the first pass takes its inputs times 2^pre, which the caller
// chooses so that their components stay below 2^58 (2^59 with HIN, whose
// first pass adds half as many).  A value after passes of total radix 2^q is
// a sum of at most 2^q inputs, and at most 2^t times the largest input when
// the caller knows that all inputs of a row together are no larger (t >= log2 L
// says nothing).  Moduli then stay below 2^61.5 when
// fx_cum(q, t) = max(0, min(q, t) - 3) bits have been shifted out by then; each
// later pass folds its share into the rounding of the twiddle products.
// Sums of two such values stay below 2^63.
// With VAR, element i of the row is scaled by 2^(pre - var[i]) instead.
// fft_row_fx returns the bits shifted out in all; `mag` collects the magnitude
// bits of the outputs (fx_mag).
__host__ __device__ __forceinline__ constexpr int fx_cum(int q, int t)
{
    const int m = q < t ? q : t;
    return m > 3 ? m - 3 : 0;
}

// q of a whole row of length L
__host__ __device__ constexpr int fx_log(int L)
{
    const int l = pow2_part(L), odd = L >> l;
    return l + (odd == 25 ? 5 : (odd == 5 ? 3 : (odd == 3 ? 2 : 0)));
}

template <bool INV, bool HIN> __device__ __forceinline__ void dft8_fx(fxc *a)
{
    // sqrt(1/2) in units of 2^-61
    constexpr fxm r = fx_multiplier(1630477228166597777ll);
    fxc u0, u1, u2, u3, d0, d1, d2, d3;
    if (HIN) {
        u0 = a[0]; u1 = a[1]; u2 = a[2]; u3 = a[3];
        d0 = a[0]; d1 = a[1]; d2 = a[2]; d3 = a[3];
    } else {
        u0 = cadd(a[0], a[4]); d0 = csub(a[0], a[4]);
        u1 = cadd(a[1], a[5]); d1 = csub(a[1], a[5]);
        u2 = cadd(a[2], a[6]); d2 = csub(a[2], a[6]);
        u3 = cadd(a[3], a[7]); d3 = csub(a[3], a[7]);
    }
    fxc v1, v2, v3;
    if (INV) {
        v1.x = fx_mulc(r, d1.x - d1.y); v1.y = fx_mulc(r, d1.x + d1.y);
        v2.x = -d2.y;                   v2.y = d2.x;
        v3.x = fx_mulc(r, -(d3.x + d3.y)); v3.y = fx_mulc(r, d3.x - d3.y);
    } else {
        v1.x = fx_mulc(r, d1.x + d1.y); v1.y = fx_mulc(r, d1.y - d1.x);
        v2.x = d2.y;                    v2.y = -d2.x;
        v3.x = fx_mulc(r, d3.y - d3.x); v3.y = fx_mulc(r, -(d3.x + d3.y));
    }
    dft4<INV, false>(u0, u1, u2, u3);
    dft4<INV, false>(d0, v1, v2, v3);
    a[0] = u0; a[1] = d0; a[2] = u1; a[3] = v1;
    a[4] = u2; a[5] = v2; a[6] = u3; a[7] = v3;
}

template <int R, bool INV, bool HIN, bool HOUT, bool FIRST, bool MAG, bool VAR>
__device__ __forceinline__ void stockham_pass_fx(fxc *row, int L, int Ns, int j, int G, const fxmc *__restrict__ tw,
                                                 int ts, bool active, int sh, unsigned &mag,
                                                 const signed char *var)
{
    constexpr int NB = 8 / R;
    fxc v[8];
    const int LR = L / R;
    const int tstep0 = (L / (Ns * R)) * ts;
    if (active) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int b = j + q * G;
            const int p0 = spos<fxc>(b);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (HIN && r >= R / 2) { v[q * R + r] = czero<fxc>(); continue; }
                v[q * R + r] = row[(LR & 63) ? spos<fxc>(b + r * LR) : p0 + r * LR];
            }
            if (FIRST && VAR) {
#pragma unroll
                for (int r = 0; r < (HIN ? R / 2 : R); ++r)
                    v[q * R + r] = fx_scale(v[q * R + r], sh - var[b + r * LR]);
            } else if (FIRST && sh > 0) {
#pragma unroll
                for (int r = 0; r < (HIN ? R / 2 : R); ++r) {
                    v[q * R + r].x.v <<= sh;
                    v[q * R + r].y.v <<= sh;
                }
            }
            if (FIRST && !VAR && sh < 0) {
#pragma unroll
                for (int r = 0; r < (HIN ? R / 2 : R); ++r) v[q * R + r] = fx_scale(v[q * R + r], sh);
            }
            if (!FIRST) {
                const int step = tstep0 * (b & (Ns - 1));
                v[q * R].x = fx_shr(v[q * R].x, sh);
                v[q * R].y = fx_shr(v[q * R].y, sh);
                int t = step;
#pragma unroll
                for (int r = 1; r < R; ++r, t += step) v[q * R + r] = fx_cmul<INV>(v[q * R + r], tw[tpos<fxmc>(t, L)], sh);
            }
            if constexpr (R == 8) dft8_fx<INV, HIN>(&v[q * R]);
            else dftR<R, INV, HIN>(&v[q * R]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = czero<fxc>();
    }
    __syncthreads();
    if (active) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int b = j + q * G;
            const int k = b & (Ns - 1);
            const int i0 = (b - k) * R + k, p0 = spos<fxc>(i0);
#pragma unroll
            for (int r = 0; r < (HOUT ? R / 2 : R); ++r) {
                const int rn = r * Ns;
                row[(Ns & 63) ? spos<fxc>(i0 + rn) : p0 + rn] = v[q * R + r];
                if (MAG) mag |= fx_mag(v[q * R + r]);
            }
        }
    }
    __syncthreads();
}

// a + c1 t1 + c2 t2 (constants in units of 2^-61)
__device__ __forceinline__ fx fx_axpy2(fx a, fxm c1, fx t1, fxm c2, fx t2)
{
    fxacc s;
    s.zero(0);
    s.mad(fx_hi(t1), fx_lo(t1), c1.hi, c1.lo);
    s.mad(fx_hi(t2), fx_lo(t2), c2.hi, c2.lo);
    return a + s.value(0);
}
template <bool INV> __device__ __forceinline__ void dft3_fx(fxc *a)
{
    constexpr fxm s = fx_multiplier(1996918623117814388ll);   // sqrt(3)/2
    const fxc t = cadd(a[1], a[2]), d = csub(a[1], a[2]);
    const fxc u{a[0].x - fx_shr(t.x, 1), a[0].y - fx_shr(t.y, 1)}, r{fx_mulc(s, d.x), fx_mulc(s, d.y)};
    a[0] = cadd(a[0], t);
    odd_pair<INV>(u, r, a[1], a[2]);
}
template <bool INV> __device__ __forceinline__ void dft5_fx(fxc *a)
{
    constexpr fxm c1 = fx_multiplier(712544676207699905ll), c2 = fx_multiplier(-1865466180814546881ll);  // cos(2 pi n/5)
    constexpr fxm s1 = fx_multiplier(2192987019466309470ll), s2 = fx_multiplier(1355340514917506542ll);  // sin(2 pi n/5)
    constexpr fxm n1{-s1.lo, -s1.hi};
    const fxc t1 = cadd(a[1], a[4]), t2 = cadd(a[2], a[3]), d1 = csub(a[1], a[4]), d2 = csub(a[2], a[3]);
    const fxc u1{fx_axpy2(a[0].x, c1, t1.x, c2, t2.x), fx_axpy2(a[0].y, c1, t1.y, c2, t2.y)};
    const fxc u2{fx_axpy2(a[0].x, c2, t1.x, c1, t2.x), fx_axpy2(a[0].y, c2, t1.y, c1, t2.y)};
    const fxc r1{fx_axpy2(fx(0), s1, d1.x, s2, d2.x), fx_axpy2(fx(0), s1, d1.y, s2, d2.y)};
    const fxc r2{fx_axpy2(fx(0), s2, d1.x, n1, d2.x), fx_axpy2(fx(0), s2, d1.y, n1, d2.y)};
    a[0] = cadd(a[0], cadd(t1, t2));
    odd_pair<INV>(u1, r1, a[1], a[4]);
    odd_pair<INV>(u2, r2, a[2], a[3]);
}
template <int R, bool INV, bool HOUT, bool MAG>
__device__ __forceinline__ void stockham_odd_fx(fxc *row, int L, int Ns, int j, int G, const fxmc *__restrict__ tw, int ts,
                                                bool active, int sh, unsigned &mag)
{
    constexpr int NB = (8 + R - 1) / R;
    fxc v[NB * R];
#pragma unroll
    for (int i = 0; i < NB * R; ++i) v[i] = czero<fxc>();
    const int LR = L / R, tstep0 = (L / (Ns * R)) * ts;
    if (active) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int b = j + q * G;
            if (b >= LR) break;
            const int step = tstep0 * (Ns == LR ? b : b & (Ns - 1));
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const fxc a = row[spos<fxc>(b + r * LR)];
                v[q * R + r] = r ? fx_cmul<INV>(a, tw[tpos<fxmc>(r * step, L)], sh) : fxc{fx_shr(a.x, sh), fx_shr(a.y, sh)};
            }
            if constexpr (R == 3) dft3_fx<INV>(&v[q * R]);
            else dft5_fx<INV>(&v[q * R]);
        }
    }
    __syncthreads();
    if (active) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int b = j + q * G;
            if (b >= LR) break;
            const int k = Ns == LR ? b : b & (Ns - 1);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = (b - k) * R + k + r * Ns;
                if (!HOUT || 2 * i < L) {
                    row[spos<fxc>(i)] = v[q * R + r];
                    if (MAG) mag |= fx_mag(v[q * R + r]);
                }
            }
        }
    }
    __syncthreads();
}

// one pass of a row: FIRST with the scale `pre`, later ones with their share of the shift
template <int R, bool INV, bool HIN, bool HOUT, bool FIRST, bool MAG, bool VAR>
__device__ __forceinline__ void fx_pass(fxc *row, int L, int Ns, int j, int G, const fxmc *tw, int ts, bool active,
                                        int pre, int q, int t, unsigned &mag, const signed char *var)
{
    const int lr = R == 8 ? 3 : (R == 4 ? 2 : 1);
    const int sh = FIRST ? pre : fx_cum(q, t) - fx_cum(q - lr, t);
    stockham_pass_fx<R, INV, HIN, HOUT, FIRST, MAG, VAR>(row, L, Ns, j, G, tw, ts, active, sh, mag, var);
}

template <bool INV, bool HIN, bool HOUT, int TS, int LC, bool MAG, bool VAR = false>
__device__ __forceinline__ int fft_row_fx(fxc *row, int L, int logL, int j, const fxmc *__restrict__ tw, bool active,
                                          int pre, int t, unsigned &mag, const signed char *var = nullptr)
{
    if constexpr (LC > 0) {
        constexpr int LL = fft_length(LC), LG = pow2_part(LL), odd = LL >> LG, G = LL >> 3, rem = LG % 3, n8 = LG / 3;
        constexpr int NS0 = rem == 1 ? 2 : (rem == 2 ? 4 : 1);
        if constexpr (rem == 1) fx_pass<2, INV, HIN, false, true, false, VAR>(row, LL, 1, j, G, tw, TS, active, pre, 1, t, mag, var);
        if constexpr (rem == 2) fx_pass<4, INV, HIN, false, true, false, VAR>(row, LL, 1, j, G, tw, TS, active, pre, 2, t, mag, var);
#pragma unroll
        for (int p = 0; p < n8; ++p) {
            const int Ns = NS0 << (3 * p), q = rem + 3 * (p + 1);
            const bool last = (p == n8 - 1) && odd == 1, first = (p == 0 && rem == 0);
            if (first && last) fx_pass<8, INV, HIN, HOUT, true, MAG, VAR>(row, LL, Ns, j, G, tw, TS, active, pre, q, t, mag, var);
            else if (first) fx_pass<8, INV, HIN, false, true, false, VAR>(row, LL, Ns, j, G, tw, TS, active, pre, q, t, mag, var);
            else if (last) fx_pass<8, INV, false, HOUT, false, MAG, false>(row, LL, Ns, j, G, tw, TS, active, pre, q, t, mag, var);
            else fx_pass<8, INV, false, false, false, false, false>(row, LL, Ns, j, G, tw, TS, active, pre, q, t, mag, var);
        }
        if constexpr (odd == 25) {
            stockham_odd_fx<5, INV, false, false>(row, LL, LL / 25, j, G, tw, TS, active, fx_cum(LG + 3, t) - fx_cum(LG, t), mag);
            stockham_odd_fx<5, INV, HOUT, MAG>(row, LL, LL / 5, j, G, tw, TS, active, fx_cum(LG + 5, t) - fx_cum(LG + 3, t), mag);
        }
        if constexpr (odd == 5)
            stockham_odd_fx<5, INV, HOUT, MAG>(row, LL, LL / 5, j, G, tw, TS, active, fx_cum(LG + 3, t) - fx_cum(LG, t), mag);
        if constexpr (odd == 3)
            stockham_odd_fx<3, INV, HOUT, MAG>(row, LL, LL / 3, j, G, tw, TS, active, fx_cum(LG + 2, t) - fx_cum(LG, t), mag);
        return fx_cum(LG + (odd == 25 ? 5 : (odd == 5 ? 3 : (odd == 3 ? 2 : 0))), t);
    } else {
        if (L < 8) {
            fxc a[4];
            if (active) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    a[i] = czero<fxc>();
                    if (i < L && !(HIN && 2 * i >= L && L > 1)) a[i] = fx_scale(row[i], VAR ? pre - var[i] : pre);
                }
                if (L == 2) dft2<false>(a[0], a[1]);
                if (L == 4) dft4<INV, false>(a[0], a[1], a[2], a[3]);
            }
            __syncthreads();
            if (active) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i < L && !(HOUT && 2 * i >= L && L > 1)) {
                        row[i] = a[i];
                        if (MAG) mag |= fx_mag(a[i]);
                    }
            }
            __syncthreads();
            return 0;
        }
        const int G = L >> 3, rem = logL % 3, n8 = logL / 3;
        int Ns = 1, q = 0, odd = LC < 0 ? L >> logL : 1;
        if (rem == 1) { fx_pass<2, INV, HIN, false, true, false, VAR>(row, L, 1, j, G, tw, TS, active, pre, 1, t, mag, var); Ns = 2; q = 1; }
        else if (rem == 2) { fx_pass<4, INV, HIN, false, true, false, VAR>(row, L, 1, j, G, tw, TS, active, pre, 2, t, mag, var); Ns = 4; q = 2; }
        for (int p = 0; p < n8; ++p) {
            const bool last = p == n8 - 1 && odd == 1, first = q == 0;
            q += 3;
            if (first && last) fx_pass<8, INV, HIN, HOUT, true, MAG, VAR>(row, L, Ns, j, G, tw, TS, active, pre, q, t, mag, var);
            else if (first) fx_pass<8, INV, HIN, false, true, false, VAR>(row, L, Ns, j, G, tw, TS, active, pre, q, t, mag, var);
            else if (last) fx_pass<8, INV, false, HOUT, false, MAG, false>(row, L, Ns, j, G, tw, TS, active, pre, q, t, mag, var);
            else fx_pass<8, INV, false, false, false, false, false>(row, L, Ns, j, G, tw, TS, active, pre, q, t, mag, var);
            Ns <<= 3;
        }
        // the odd passes: q bits rounded up from the radices so far (40 = 8 x 5: 6; 25 x 2^l: l + 5)
        if constexpr (LC < 0) {
            if (odd == 25) {
                stockham_odd_fx<5, INV, false, false>(row, L, Ns, j, G, tw, TS, active, fx_cum(q + 3, t) - fx_cum(q, t), mag);
                q += 3;
                Ns *= 5;
                const int q2 = logL + 5;
                stockham_odd_fx<5, INV, HOUT, MAG>(row, L, Ns, j, G, tw, TS, active, fx_cum(q2, t) - fx_cum(q, t), mag);
                q = q2;
            } else if (odd == 5) {
                stockham_odd_fx<5, INV, HOUT, MAG>(row, L, Ns, j, G, tw, TS, active, fx_cum(q + 3, t) - fx_cum(q, t), mag);
                q += 3;
            } else if (odd == 3) {
                stockham_odd_fx<3, INV, HOUT, MAG>(row, L, Ns, j, G, tw, TS, active, fx_cum(q + 2, t) - fx_cum(q, t), mag);
                q += 2;
            }
        }
        return fx_cum(q, t);
    }
}

// Row lengths with compiled code: the powers of two 64 .. 1024 in every kernel,
// and the lengths with an odd part that the planner gives an axis (LC of
// fft_row; X(LC)): the x rows hold half the padded length, the y-z kernel of
// films the whole one, and the passes of bulk grids have all of them.
#define MM_LC_POW2(X) X(6) X(7) X(8) X(9) X(10)
#define MM_LX_ODD(X) X(160) X(192) X(320) X(384)
#define MM_LY_ODD(X) X(320) X(384) X(640) X(768)
#define MM_LB_ODD(X) X(80) X(96) X(160) X(192) X(200) X(320) X(384) X(400) X(640) X(768) X(800)
#define MM_LX_CASES(X) X(0) MM_LC_POW2(X) MM_LX_ODD(X)
#define MM_LY_CASES(X) X(0) MM_LC_POW2(X) MM_LY_ODD(X)
#define MM_LB_CASES(X) X(0) MM_LC_POW2(X) MM_LB_ODD(X)
__host__ __device__ inline int lc_pow2(int L, int other)
{
    return L >= 64 && L <= 1024 && (L & (L - 1)) == 0 ? pow2_part(L) : other;
}
#define MM_LC_OF(name, ODD, other)           \
    __host__ __device__ inline int name(int L) \
    {                                         \
        switch (L) {                          \
            ODD(MM_LC_CASE) return L;         \
        }                                     \
        return lc_pow2(L, other);             \
    }
#define MM_LC_CASE(N) case N:
MM_LC_OF(lx_of, MM_LX_ODD, 0)
MM_LC_OF(ly_of, MM_LY_ODD, 0)
MM_LC_OF(lb_of, MM_LB_ODD, 0)

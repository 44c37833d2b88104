// fixed_fft.cuh -- FP64 line transforms in 64-bit fixed point.
//
// GB300 issues FP64 at 1/36 of the rate of a 64-bit integer add or of a
// 32 x 32 + 64 multiply-add (measured, lanes per clock and SM: DFMA and DADD
// 1.66, add.s64 60, mad.wide.s32 58), so an FP64 line transform is bound by
// FP64 issue (row DCT of 8 fields at N = 2048: 1.82 ms for 0.54 GB moved).
// Here a line is converted to 64-bit fixed point with one power-of-two scale
// of its own, transformed with integer adds and multiply-adds, and converted
// back:
//   scale    the line's largest magnitude goes to 2^59 .. 2^60, so every FP64
//            value within 2^-7 of it is represented exactly and the others
//            to 2^-60 of it;
//   growth   the sum of |re| + |im| over the line bounds every intermediate of
//            the transform.  It is taken per lane (the values that one lane
//            transforms in registers) and per line: the line is shifted right
//            by s0 before the first in-register pass so that no lane can
//            exceed 2^60, and by sh more at the twiddles between the passes,
//            so that the line cannot.  Localised lines and sparse spectra
//            (most of this scheme's: the interface, the low modes) need
//            neither; a dense line shifts by log2 of its length in all;
//   twiddles 64-bit constants with 62 fractional bits (error 2^-63; FP64
//            twiddles carry 2^-54), products rounded at the last bit.
// The error is thus a few units of 2^-60 of the line's L1 norm, below that of
// the FP64 butterflies it replaces (their rounding: 2^-53 per pass relative
// to the line's 2-norm).
//
// Range: a complex product takes components below 2^61.  A non-finite input
// value makes its whole line NaN (as the FP64 transform does).  Subnormal
// values and scales beyond the FP64 range on the way back are exact up to
// FP64's own rounding (to_double).
//
// The line layout is that of warp_fft.cuh: M = E G complex values on G lanes,
// an E-point DFT in registers, twiddle, transpose through the line's
// shared-memory buffer, G-point DFTs; for G = R E the split second pass.
#pragma once
#include "dct_device.cuh"
#include "warp_fft.cuh"
#include "bounds.cuh"

namespace ccm {
namespace xf {

struct fx { long long v; };
__device__ __forceinline__ fx operator+(fx a, fx b) { return fx{a.v + b.v}; }
__device__ __forceinline__ fx operator-(fx a, fx b) { return fx{a.v - b.v}; }
__device__ __forceinline__ fx operator-(fx a) { return fx{-a.v}; }
using cx = cplx<fx>;

// ------------------------------------------------------------------ products
// A factor w (|w| <= 2^62, 62 fractional bits) as w = h 2^32 + l with l a
// signed word; h and -h, -l fit 32 bits.
struct Fac { int h, l; };
__host__ __device__ constexpr Fac fac(long long w) {
    return Fac{(int)((w + 0x80000000LL) >> 32), (int)(w & 0xffffffffLL)};
}
struct CFac { Fac x, y; };              // re, im

// cos(2 pi j / 64) with 62 fractional bits
__host__ __device__ constexpr long long cos64(int j) {
    j &= 63;
    if (j > 32) j = 64 - j;
    const bool neg = j > 16;
    if (neg) j = 32 - j;
    long long v = 0;
    switch (j) {
        case 0: v = 0x4000000000000000LL; break;
        case 1: v = 0x3fb11b47a24a4b3cLL; break;
        case 2: v = 0x3ec52f9feeb96056LL; break;
        case 3: v = 0x3d3e82ad8c5bb4bbLL; break;
        case 4: v = 0x3b20d79e651a8c51LL; break;
        case 5: v = 0x387165e3017b61a4LL; break;
        case 6: v = 0x3536cc521d434606LL; break;
        case 7: v = 0x317900d62a2e816aLL; break;
        case 8: v = 0x2d413cccfe779921LL; break;
        case 9: v = 0x2899e64a123bac30LL; break;
        case 10: v = 0x238e76735cd190d9LL; break;
        case 11: v = 0x1e2b5d3806f63b1eLL; break;
        case 12: v = 0x187de2a6aea962d2LL; break;
        case 13: v = 0x1294062ed59f05a9LL; break;
        case 14: v = 0x0c7c5c1e34d3055bLL; break;
        case 15: v = 0x0645e9af0a6d0af8LL; break;
        default: v = 0; break;
    }
    return neg ? -v : v;
}
constexpr long long kSqrtHalf = 0x2d413cccfe779921LL;

// round(a w / 2^62) for complex a (components below 2^61) and |w| <= 1, CONJ:
// times conj(w).  The low x low products are left out (under one unit), the
// cross products round to nearest.
template <bool CONJ>
__device__ __forceinline__ cx cmulf(cx a, CFac w) {
    constexpr long long half = 1LL << 29;
    const int xl = (int)a.x.v, yl = (int)a.y.v;
    const int xh = (int)(a.x.v >> 32) + (int)((unsigned)xl >> 31), yh = (int)(a.y.v >> 32) + (int)((unsigned)yl >> 31);
    const int x4 = xh * 4, y4 = yh * 4;
    const int wyh = CONJ ? -w.y.h : w.y.h, wyl = CONJ ? -w.y.l : w.y.l;
    long long cr = half + (long long)xh * w.x.l;
    cr += (long long)xl * w.x.h;
    cr += (long long)yh * -wyl;
    cr += (long long)yl * -wyh;
    long long re = (cr >> 30) + (long long)x4 * w.x.h;
    re += (long long)y4 * -wyh;
    long long ci = half + (long long)xh * wyl;
    ci += (long long)xl * wyh;
    ci += (long long)yh * w.x.l;
    ci += (long long)yl * w.x.h;
    long long im = (ci >> 30) + (long long)x4 * wyh;
    im += (long long)y4 * w.x.h;
    return mk(fx{re}, fx{im});
}
__device__ __forceinline__ fx mulf(fx a, Fac w) {
    const int l = (int)a.v, h = (int)(a.v >> 32) + (int)((unsigned)l >> 31);
    long long c = (1LL << 29) + (long long)h * w.l;
    c += (long long)l * w.h;
    return fx{(c >> 30) + (long long)(h * 4) * w.h};
}

// x W_R^i, W_R = exp(-2 pi i / R) (INV: conjugate); i and R are compile-time
// constants after unrolling
template <int R, bool INV>
__device__ __forceinline__ cx twidx(cx x, int i) {
    const int j = (i * (64 / R)) & 63;
    if (j == 0) return x;
    if (j == 16) return INV ? mk(-x.y, x.x) : mk(x.y, -x.x);
    if (j == 32) return mk(-x.x, -x.y);
    if (j == 48) return INV ? mk(x.y, -x.x) : mk(-x.y, x.x);
    constexpr Fac h = fac(kSqrtHalf);
    if (j == 8) return INV ? mk(mulf(x.x - x.y, h), mulf(x.x + x.y, h)) : mk(mulf(x.x + x.y, h), mulf(x.y - x.x, h));
    if (j == 24) return INV ? mk(mulf(-(x.x + x.y), h), mulf(x.x - x.y, h)) : mk(mulf(x.y - x.x, h), mulf(-(x.x + x.y), h));
    return cmulf<!INV>(x, CFac{fac(cos64(j)), fac(cos64(j + 48))});     // exp(+i ...), conjugated for the forward one
}

// Radix-2 decimation in frequency on v[OFF .. OFF + R): natural input, output
// v[OFF + r] = X[bitrev_R(r)].
template <int R, bool INV, int OFF>
struct DIFX {
    static __device__ __forceinline__ void run(cx* v) {
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            const cx a = v[OFF + i], b = v[OFF + i + R / 2];
            v[OFF + i] = a + b;
            v[OFF + i + R / 2] = twidx<R, INV>(a - b, i);
        }
        DIFX<R / 2, INV, OFF>::run(v);
        DIFX<R / 2, INV, OFF + R / 2>::run(v);
    }
};
template <bool INV, int OFF> struct DIFX<1, INV, OFF> { static __device__ __forceinline__ void run(cx*) {} };

// ------------------------------------------------------------------ line shapes
// M = E G.  32 values per lane at most (128 registers of data); from M = 2048
// on a line spans two and four warps (split second pass).
template <int M> struct Shape;
template <> struct Shape<32>   { static constexpr int E = 8,  G = 4;   };
template <> struct Shape<64>   { static constexpr int E = 8,  G = 8;   };
template <> struct Shape<128>  { static constexpr int E = 16, G = 8;   };
template <> struct Shape<256>  { static constexpr int E = 16, G = 16;  };
template <> struct Shape<512>  { static constexpr int E = 32, G = 16;  };
template <> struct Shape<1024> { static constexpr int E = 32, G = 32;  };
template <> struct Shape<2048> { static constexpr int E = 32, G = 64;  };
template <> struct Shape<4096> { static constexpr int E = 32, G = 128; };

// LINES lines per CTA: eight (one 64-byte segment of eight rows in the
// transposed writes), fewer where their buffers no longer fit.  A buffer is
// the padded transpose plus what makes its length odd in units of 16 bytes
// modulo 128, so that the same element of eight lines lies in distinct banks.
template <int M> struct Geo {
    static constexpr int E = Shape<M>::E, G = Shape<M>::G, J = E >= G ? E / G : 1, R = G > E ? G / E : 1;
    static constexpr int N = 2 * M, HI = E / 2;            // HI pairs per lane
    static constexpr int LINES = M <= 1024 ? 8 : M == 2048 ? 4 : 2;
    static constexpr int THREADS = LINES * G;
    static constexpr int W = G > 32 ? G / 32 : 1;          // warps per line
    static constexpr int P = E >= G ? G + 1 : G + R;       // transpose row
    static constexpr int BUF = ((E * P + 7) / 8) * 8 + 1;
    static constexpr size_t SMEM = (size_t)LINES * BUF * sizeof(cx);
    static_assert(THREADS % 32 == 0, "whole warps");
};

template <int M> __device__ __forceinline__ void lane_of(int& n2, int& slot) {
    constexpr int G = Geo<M>::G;
    n2 = threadIdx.x % G;
    slot = threadIdx.x / G;
}
// Barrier of one line's lanes (named barrier 1 + slot where it spans warps).
template <int M> __device__ __forceinline__ void sync_line(int slot) { wf::line_sync<Geo<M>::G>(slot); }

// Per-line words shared by the line's lanes (and read by the whole CTA).
template <int M> struct LineSm {
    unsigned red[Geo<M>::LINES][Geo<M>::W];
    float redf[Geo<M>::LINES][Geo<M>::W];
    int ex[Geo<M>::LINES];             // value = fixed * 2^ex; kBad: a non-finite line
};
constexpr int kBad = 0x40000000;

template <int M> __device__ __forceinline__ unsigned line_max(unsigned x, int slot, LineSm<M>& sm) {
    constexpr int G = Geo<M>::G, W = Geo<M>::W;
#pragma unroll
    for (int o = (G < 32 ? G : 32) / 2; o > 0; o >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
    if constexpr (W > 1) {
        sync_line<M>(slot);
        if ((threadIdx.x & 31) == 0) sm.red[slot][(threadIdx.x >> 5) % W] = x;
        sync_line<M>(slot);
#pragma unroll
        for (int w = 0; w < W; ++w) x = max(x, sm.red[slot][w]);
    }
    return x;
}
template <int M> __device__ __forceinline__ float line_sum(float x, int slot, LineSm<M>& sm) {
    constexpr int G = Geo<M>::G, W = Geo<M>::W;
#pragma unroll
    for (int o = (G < 32 ? G : 32) / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if constexpr (W > 1) {
        sync_line<M>(slot);
        if ((threadIdx.x & 31) == 0) sm.redf[slot][(threadIdx.x >> 5) % W] = x;
        sync_line<M>(slot);
        x = sm.redf[slot][0];
#pragma unroll
        for (int w = 1; w < W; ++w) x += sm.redf[slot][w];
    }
    return x;
}

// ------------------------------------------------------------------ conversions
// High word without the sign: orders magnitudes, 0x7ff00000 and above are
// infinities and NaN.
__device__ __forceinline__ unsigned mag_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// x in fixed point with the line's largest exponent em (biased, >= 1) at
// 2^59 .. 2^60: x 2^(1082 - em), rounded to nearest (ties away from zero).
__device__ __forceinline__ fx to_fixed(double x, int em) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    int e = (int)((hi >> 20) & 0x7ffu);
    const unsigned m = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
    e = max(e, 1);
    const unsigned long long t = ((unsigned long long)m << 42) | ((unsigned long long)lo << 10);   // below 2^63
    const long long q = (long long)(((t >> min(2 + em - e, 63)) + 1) >> 1);
    const long long s = (int)hi >> 31;
    return fx{(q ^ s) - s};
}

// v 2^ex rounded to nearest (ties away from zero)
__device__ __forceinline__ double to_double(fx v, int ex) {
    const long long s = v.v >> 63;
    unsigned long long q = (unsigned long long)((v.v ^ s) - s);
    const int lz = __clzll((long long)q);
    int e = ex - lz + 63 + 1022;                       // biased exponent - 1
    double r = 0.0;
    if (q) {
        q <<= lz;
        if (e >= 0 && e < 2045) {
            const unsigned long long b = ((unsigned long long)(unsigned)e << 52) + (q >> 11) + ((q >> 10) & 1);
            r = __longlong_as_double((long long)(b | ((unsigned long long)s & 0x8000000000000000ull)));
        } else {                                       // beyond FP64's normal range
            r = scalbn((double)(v.v), max(-4000, min(4000, ex)));
        }
    }
    return r;
}
// v 2^(ex + p) of a line with exponent ex
__device__ __forceinline__ double line_double(fx v, int ex, int p = 0) {
    return ex == kBad ? __longlong_as_double(0x7ff8000000000000ll) : to_double(v, ex + p);
}

// ------------------------------------------------------------------ scaling
// v: this lane's E values, components below 2^60.6.  Shifts the line right by
// s0 (returned through ex, which it is added to) so that no lane's first pass
// can exceed 2^60, and sets sh, the further shift at the twiddles that keeps
// the line below 2^60 (ex also counts it).
template <int M>
__device__ __forceinline__ void fit_line(cx* v, int slot, LineSm<M>& sm, int& ex, int& sh) {
    constexpr int E = Geo<M>::E;
    unsigned acc = 0;                                  // lane sum of |re| + |im| in units of 2^38, rounded up
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const int a = (int)(v[i].x.v >> 32), b = (int)(v[i].y.v >> 32);
        acc += (unsigned)(abs(a) >> 6) + (unsigned)(abs(b) >> 6) + 2u;
    }
    const int top = 32 - __clz((int)line_max<M>(acc, slot, sm));        // lane sums below 2^top
    const float tot = line_sum<M>((float)acc, slot, sm) * 1.001f;
    const int s0 = max(0, top - 22);
    const int et = ((__float_as_int(tot) >> 23) & 0xff) - 126;          // line sum below 2^et
    sh = max(0, et - 22 - s0);
    if (s0 > 0) {
        const long long h = 1LL << (s0 - 1);
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = mk(fx{(v[i].x.v + h) >> s0}, fx{(v[i].y.v + h) >> s0});
    }
    ex += s0 + sh;
}

// ------------------------------------------------------------------ line transform
__device__ __forceinline__ CFac ld_fac(const int4* __restrict__ t) {
    const int4 q = __ldg(t);
    return CFac{Fac{q.x, q.y}, Fac{q.z, q.w}};
}
__device__ __forceinline__ cx shift_cx(cx a, int sh, long long h) { return mk(fx{(a.x.v + h) >> sh}, fx{(a.y.v + h) >> sh}); }

// The unnormalised DFT of the line (value G n1 + n2 in v[n1] of lane n2);
// the result lies in buf in natural order, visible to the line's lanes.
// tw2[k1 G + n2] = W_M^{n2 k1}.
template <int M, bool INV>
__device__ __forceinline__ void fft_line(cx* v, cx* buf, const int4* __restrict__ tw2, int n2, int slot, int sh) {
    using Gm = Geo<M>;
    constexpr int E = Gm::E, G = Gm::G, P = Gm::P;
    DIFX<E, INV, 0>::run(v);
    const long long h = (1LL << sh) >> 1;
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const int k1 = wf::bitrev<E>(r);
        cx u = v[r];
        if (k1) u = cmulf<INV>(u, ld_fac(tw2 + k1 * G + n2));
        buf[k1 * P + n2] = shift_cx(u, sh, h);
    }
    sync_line<M>(slot);
    if constexpr (E >= G) {
        constexpr int J = Gm::J;
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int m = 0; m < G; ++m) v[j * G + m] = buf[(n2 * J + j) * P + m];
        sync_line<M>(slot);
        DIFX<G, INV, 0>::run(v);
        if constexpr (J == 2) DIFX<G, INV, (J == 2 ? G : 0)>::run(v);
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int r = 0; r < G; ++r) buf[(n2 * J + j) + E * wf::bitrev<G>(r)] = v[j * G + r];
    } else {
        // each G-point row on R adjacent lanes (fourstep_split in warp_fft.cuh has the formula)
        constexpr int R = Gm::R;
        constexpr unsigned FULL = 0xffffffffu;
        const int k1 = n2 / R, q = n2 % R;
#pragma unroll
        for (int t = 0; t < E; ++t) v[t] = buf[k1 * P + R * t + q];
        sync_line<M>(slot);
        DIFX<E, INV, 0>::run(v);
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int k = wf::bitrev<E>(r);
            cx u = cmulf<INV>(v[r], ld_fac(tw2 + k * G + E * q));       // W_G^{q k}
            cx p = mk(fx{__shfl_xor_sync(FULL, u.x.v, R / 2)}, fx{__shfl_xor_sync(FULL, u.y.v, R / 2)});
            if constexpr (R == 2) {
                buf[k1 + E * (k + E * q)] = q ? p - u : u + p;
            } else {
                u = (q & 2) ? p - u : u + p;
                p = mk(fx{__shfl_xor_sync(FULL, u.x.v, 1)}, fx{__shfl_xor_sync(FULL, u.y.v, 1)});
                const cx a = (q & 1) ? p : u, b = (q & 1) ? u : p;
                const cx wb = (q & 2) ? (INV ? mk(-b.y, b.x) : mk(b.y, -b.x)) : b;
                buf[k1 + E * (k + E * (((q & 1) << 1) | (q >> 1)))] = (q & 1) ? a - wb : a + wb;
            }
        }
    }
    sync_line<M>(slot);
}

// ------------------------------------------------------------------ DCT pairs
// Factors of the pair (k, M-k), k = 0 .. M/2 (see PairTw in warp_fft.cuh), as
// factors of at most 1; the powers of two that bring them to size are folded
// into the line's exponent:
//   wn = e^{-2 pi i k/N}; forward a = f_k e^{-i pi k/2N}, b = f e^{-i pi/4} e^{+i pi k/2N};
//   inverse the conjugates (f_k, f below).
// Forward: c_k / 2 = f_k 2^-pf, inverse: s_k / 2 = f'_k 2^-pi.
struct PairTab {
    const int4* __restrict__ wn;
    const int4* __restrict__ a;
    const int4* __restrict__ b;
    int p;                              // the power of two
};
struct Quad64 { fx xk, xNk, xMk, xMpk; };

__device__ __forceinline__ Quad64 post_pair(cx A, cx B, const PairTab& t, int k) {
    const cx P = mk(A.x + B.x, A.y - B.y), Q = mk(A.x - B.x, A.y + B.y);
    const cx U = cmulf<false>(Q, ld_fac(t.wn + k));
    const cx S = mk(P.x + U.y, P.y - U.x), R = mk(P.x - U.y, -(P.y + U.x));
    const cx s = cmulf<false>(S, ld_fac(t.a + k)), r = cmulf<false>(R, ld_fac(t.b + k));
    return Quad64{s.x, -s.y, r.x, -r.y};
}
__device__ __forceinline__ void pre_pair(const Quad64& X, const PairTab& t, int k, cx& zk, cx& zMk) {
    const cx V = cmulf<false>(mk(X.xk, -X.xNk), ld_fac(t.a + k));
    const cx Y = cmulf<false>(mk(X.xMk, -X.xMpk), ld_fac(t.b + k));
    const cx s = mk(V.x + Y.x, V.y - Y.y), d = mk(V.x - Y.x, V.y + Y.y);
    const cx u = cmulf<true>(d, ld_fac(t.wn + k));
    zk = mk(s.x - u.y, s.y + u.x);
    zMk = mk(s.x + u.y, u.x - s.y);
}

// Pair items of a line: item k in [1, M/2) holds the modes k, N-k, M-k, M+k;
// item 0 holds the modes 0, M/2, M, N-M/2 (the pairs 0 and M/2), so that the
// M/2 items hold each of the N modes once.
template <int M> __device__ __forceinline__ int item_mode(int k, int u) {
    constexpr int N = 2 * M;
    const int hi = k == 0 ? (u == 1 ? M / 2 : u == 3 ? N - M / 2 : u == 0 ? 0 : M) : 0;
    return k == 0 ? hi : u == 0 ? k : u == 1 ? N - k : u == 2 ? M - k : M + k;
}
// The four modes of item k from the natural-order spectrum z (a second turn
// of the loop for item 0: one copy of the code).
template <int M> __device__ __forceinline__ Quad64 post_item(const cx* z, const PairTab& t, int k) {
    const cx A = z[k], B = z[k == 0 ? M / 2 : M - k];
    Quad64 q = post_pair(A, k == 0 ? A : B, t, k);
    if (k == 0) {
        const Quad64 h = post_pair(B, B, t, M / 2);
        q.xNk = h.xk;
        q.xMpk = h.xNk;
    }
    return q;
}
template <int M> __device__ __forceinline__ void pre_item(const Quad64& X, const PairTab& t, int k, cx* z) {
    cx a, b;
    if (k != 0) {
        pre_pair(X, t, k, a, b);
        z[k] = a;
        z[M - k] = b;
    } else {
        pre_pair(Quad64{X.xk, fx{0}, X.xMk, X.xMk}, t, 0, a, b);
        z[0] = a;
        pre_pair(Quad64{X.xNk, X.xMpk, X.xNk, X.xMpk}, t, M / 2, a, b);
        z[M / 2] = a;
    }
}

// Forward half-length transform of a real line at x (global, 16-byte aligned;
// v[m] = (x[4m], x[4m+2]), v[M-1-m] = (x[4m+3], x[4m+1])): the natural-order
// spectrum in buf, its exponent in sm.ex[slot] and returned.  DST: the line is
// multiplied by (-1)^i, and by -1 on odd rows (the DST as a DCT).
template <int M, bool DST>
__device__ __forceinline__ int forward_line(const double* __restrict__ x, cx* buf, const int4* __restrict__ tw2, int n2,
                                             int slot, LineSm<M>& sm, bool odd_row) {
    constexpr int E = Geo<M>::E, G = Geo<M>::G;
    cx v[E];
    int ex, sh;
    bool bad;
    {
        double d[2 * E];
        unsigned mx = 0;
        const double2* x2 = reinterpret_cast<const double2*>(x);
#pragma unroll
        for (int i = 0; i < E / 2; ++i) {
            const double2 q0 = __ldg(x2 + 2 * (G * i + n2)), q1 = __ldg(x2 + 2 * (G * i + n2) + 1);
            d[2 * i] = q0.x;
            d[2 * i + 1] = q1.x;
            if constexpr (G <= 32) {
                d[2 * (E - 1 - i)] = __shfl_xor_sync(0xffffffffu, q1.y, G - 1);
                d[2 * (E - 1 - i) + 1] = __shfl_xor_sync(0xffffffffu, q0.y, G - 1);
            } else {
                d[2 * (E - 1 - i)] = __ldg(x + 4 * (G * i + (G - 1 - n2)) + 3);
                d[2 * (E - 1 - i) + 1] = __ldg(x + 4 * (G * i + (G - 1 - n2)) + 1);
            }
        }
#pragma unroll
        for (int i = 0; i < 2 * E; ++i) mx = max(mx, mag_hi(d[i]));
        mx = line_max<M>(mx, slot, sm);
        bad = mx >= 0x7ff00000u;
        const int em = max((int)(mx >> 20), 1);
        ex = em - 1082;
#pragma unroll
        for (int i = 0; i < E; ++i) {
            v[i] = mk(to_fixed(d[2 * i], em), to_fixed(d[2 * i + 1], em));
            if constexpr (DST) {               // (-1)^i: even columns in the first half of z, odd ones in the second
                const bool neg = odd_row != (i >= E / 2);
                if (neg) v[i] = mk(-v[i].x, -v[i].y);
            }
        }
    }
    fit_line<M>(v, slot, sm, ex, sh);
    fft_line<M, false>(v, buf, tw2, n2, slot, sh);
    if (bad) ex = kBad;
    if (n2 == 0) sm.ex[slot] = ex;
    return ex;
}

// Inverse: the line's modes X (items k = n2 + G i, four values each, in
// orthonormal DCT coefficients) to the natural-order samples in buf (sample m:
// x[4m], x[4m+2]; sample M-1-m: x[4m+3], x[4m+1]); the exponent in sm.ex[slot]
// and returned.
template <int M>
__device__ __forceinline__ int inverse_line(double (&X)[2 * Geo<M>::E], cx* buf, const int4* __restrict__ tw2,
                                             const PairTab& ti, int n2, int slot, LineSm<M>& sm) {
    constexpr int E = Geo<M>::E, G = Geo<M>::G;
    unsigned mx = 0;
#pragma unroll
    for (int i = 0; i < 2 * E; ++i) mx = max(mx, mag_hi(X[i]));
    mx = line_max<M>(mx, slot, sm);
    const bool bad = mx >= 0x7ff00000u;
    const int em = max((int)(mx >> 20), 1);
    // room for the pairs: a sample of z is at most 4 sqrt(2) times the largest mode
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
        const Quad64 q{to_fixed(X[4 * i], em + 2), to_fixed(X[4 * i + 1], em + 2), to_fixed(X[4 * i + 2], em + 2),
                       to_fixed(X[4 * i + 3], em + 2)};
        pre_item<M>(q, ti, n2 + G * i, buf);
    }
    int ex = em + 2 - 1082 + ti.p, sh;
    sync_line<M>(slot);
    cx v[E];
#pragma unroll
    for (int i = 0; i < E; ++i) v[i] = buf[G * i + n2];
    sync_line<M>(slot);
    fit_line<M>(v, slot, sm, ex, sh);
    fft_line<M, true>(v, buf, tw2, n2, slot, sh);
    if (bad) ex = kBad;
    if (n2 == 0) sm.ex[slot] = ex;
    return ex;
}

// x[4m .. 4m+3] from the natural-order samples
template <int M> __device__ __forceinline__ vec4<double> unpack_item(const cx* z, int m, int ex) {
    const cx a = z[m], b = z[M - 1 - m];
    return {line_double(a.x, ex), line_double(b.y, ex), line_double(a.y, ex), line_double(b.x, ex)};
}

// 1 / d for d > 0 well inside the FP64 range: hardware seed (20 bits or more)
// and one cubically convergent Newton step (e = 1 - d r, r (1 + e + e^2)),
// error below 2 units in the last place; plain division otherwise.
__device__ __forceinline__ double recip(double d) {
    const unsigned h = (unsigned)__double2hiint(d);
    if (h - 0x02000000u >= 0x7b000000u) return 1.0 / d;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    double e = fma(-d, r, 1.0);
    e = fma(e, e, e);
    return fma(r, e, r);
}

}  // namespace xf
}  // namespace ccm

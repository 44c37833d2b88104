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
//            exceed 2^60, and by more at the twiddles between the passes,
//            so that the line cannot.  Localised lines and sparse spectra
//            (most of this scheme's: the interface, the low modes) need
//            neither; a dense line shifts by log2 of its length in all, on
//            long lines in both later passes by what each can add: a
//            shift's rounding grows by the square root of the length still to
//            be transformed, and all of it at the first twiddle left dense
//            lines of N = 4096 and 8192 further off than FP64 ones (8192: 1.2e-15
//            against 4.1e-16 .. 4.9e-16);
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
// Line layout: M = A C D complex values on G = M / A lanes, A = 16 per lane
// (8 and 4 on short lines, whose grids leave most of the chip idle: there a
// lane's own chain of instructions is the kernel's time): an A-point DFT in registers, twiddle, then on
// each row of B = C D values a C-point and a D-point DFT, exchanged through the
// line's shared-memory buffer (D = 1: one exchange).  Sixteen values are 64
// registers of data, so sixteen warps fit an SM; with 32 (two exchanges fewer)
// eight fit and the kernels waited on instruction latency and, in the ones
// with the longest unrolled code, on instruction fetch (ncu, N = 2048: issue
// slots 39 % busy in the row kernel, 15 - 21 % in the others).
#pragma once
#include "dct_device.cuh"
#include "warp_fft.cuh"
#include "bounds.cuh"
#include "fixed_ops.h"

namespace ccm {
namespace xf {

struct fx { long long v; };
__device__ __forceinline__ fx operator+(fx a, fx b) { return fx{a.v + b.v}; }
__device__ __forceinline__ fx operator-(fx a, fx b) { return fx{a.v - b.v}; }
__device__ __forceinline__ fx operator-(fx a) { return fx{-a.v}; }
using cx = cplx<fx>;

// ------------------------------------------------------------------ products
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

// One level of a radix-2 decimation in frequency on v[OFF .. OFF + R)
template <int R, bool INV, int OFF>
__device__ __forceinline__ void level(cx* v) {
#pragma unroll
    for (int i = 0; i < R / 2; ++i) {
        const cx a = v[OFF + i], b = v[OFF + i + R / 2];
        v[OFF + i] = a + b;
        v[OFF + i + R / 2] = twidx<R, INV>(a - b, i);
    }
}

// Radix-2 decimation in frequency on v[OFF .. OFF + R): natural input, output
// v[OFF + r] = X[bitrev_R(r)].
template <int R, bool INV, int OFF>
struct DIFX {
    static __device__ __forceinline__ void run(cx* v) {
        level<R, INV, OFF>(v);
        DIFX<R / 2, INV, OFF>::run(v);
        DIFX<R / 2, INV, OFF + R / 2>::run(v);
    }
};
template <bool INV, int OFF> struct DIFX<1, INV, OFF> { static __device__ __forceinline__ void run(cx*) {} };

// ------------------------------------------------------------------ line shapes
template <int M> struct Shape;
template <> struct Shape<32>   { static constexpr int A = 4,  C = 4,  D = 2;  };
template <> struct Shape<64>   { static constexpr int A = 4,  C = 4,  D = 4;  };
template <> struct Shape<128>  { static constexpr int A = 8,  C = 4,  D = 4;  };
template <> struct Shape<256>  { static constexpr int A = 8,  C = 4,  D = 8;  };
template <> struct Shape<512>  { static constexpr int A = 16, C = 4,  D = 8;  };
template <> struct Shape<1024> { static constexpr int A = 16, C = 8,  D = 8;  };
template <> struct Shape<2048> { static constexpr int A = 16, C = 16, D = 8;  };
template <> struct Shape<4096> { static constexpr int A = 16, C = 16, D = 16; };

// LINES lines per CTA: eight (one 64-byte segment of eight rows in the
// transposed writes), fewer where their buffers no longer fit.  Rows of the
// exchanges are P = B + 1 values apart (odd, so that eight rows' values of one
// column lie in distinct banks), and so, modulo eight, are the buffers.
template <int M> struct Geo {
    static constexpr int A = Shape<M>::A, C = Shape<M>::C, D = Shape<M>::D, B = C * D, E = A, G = M / A;
    static_assert(A * B == M && A % C == 0 && A % D == 0, "line shape");
    static constexpr int N = 2 * M;
    static constexpr int LINES = M <= 1024 ? 8 : M == 2048 ? 4 : 2;
    static constexpr int THREADS = LINES * G;
    static constexpr int W = G > 32 ? G / 32 : 1;          // warps per line
    static constexpr int P = B + 1;
    static constexpr int BUF = ((A * P + 7) / 8) * 8 + 1;
    static constexpr size_t SMEM = (size_t)LINES * BUF * sizeof(cx);
    static constexpr int MINB = 512 / THREADS > 4 ? 4 : 512 / THREADS;       // at most 128 registers
    static constexpr bool STAGED = M >= 1024;              // shifts in both passes (shorter lines: all at the first twiddle)
    static constexpr int LOG_C = C == 4 ? 2 : C == 8 ? 3 : 4;
    static_assert(1 << LOG_C == C, "");
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
    // mantissa at bit 62 as two words, right by 2 + em - e, rounded by the last shift
    unsigned H = __funnelshift_l(lo, m, 10), Lw = lo << 10;
    const int r = min(2 + em - e, 63);
    if (r >= 32) { Lw = H; H = 0; }
    Lw = __funnelshift_r(Lw, H, r);                    // shift counts modulo 32
    H >>= r & 31;
    const long long q = (long long)(((((unsigned long long)H << 32) | Lw) + 1) >> 1);
    const long long s = (int)hi >> 31;
    return fx{(q ^ s) - s};
}

// Beyond FP64's normal range (kept out of line: its conversions would be
// executed ahead of the branch, on the FP64 pipe).
static __device__ __noinline__ double to_double_far(long long v, int ex) { return scalbn((double)v, max(-4000, min(4000, ex))); }

// v 2^ex rounded to nearest (ties away from zero)
__device__ __forceinline__ double to_double(fx v, int ex) {
    const long long s8 = v.v >> 63, u = (v.v ^ s8) - s8;
    const unsigned h = (unsigned)(u >> 32), l = (unsigned)u;
    const unsigned n = h ? h : l, m = h ? l : 0;
    const int lz = __clz((int)n), e = (h ? ex : ex - 32) - lz + 63 + 1022;   // biased exponent - 1
    if (n != 0 && (unsigned)e >= 2045u) return to_double_far(v.v, ex);
    const unsigned H = __funnelshift_l(m, n, lz), Lw = m << (lz & 31);
    const unsigned long long b = (((unsigned long long)((unsigned)e << 20) + (H >> 11)) << 32 | __funnelshift_r(Lw, H, 11)) + ((Lw >> 10) & 1);
    const unsigned long long z = n ? b | ((unsigned long long)s8 & 0x8000000000000000ull) : 0;
    return __longlong_as_double((long long)z);
}
// v 2^(ex + p) of a line with exponent ex
__device__ __forceinline__ double line_double(fx v, int ex, int p = 0) {
    return ex == kBad ? __longlong_as_double(0x7ff8000000000000ll) : to_double(v, ex + p);
}

// ------------------------------------------------------------------ scaling
// v 2^-sh rounded to nearest, ties to even (sh < 32).  Ties are frequent at
// small shifts; rounded up, they moved every value of a line by a quarter of
// a unit, which the transform gathers in its zero mode (psi's mean drifted by
// 2e-16 a step at N = 2048).
__device__ __forceinline__ fx shift_fx(fx a, int sh) {
    const int odd = (int)__funnelshift_r((unsigned)a.v, (unsigned)(a.v >> 32), sh) & (sh ? 1 : 0);
    return fx{(a.v + (((1LL << sh) - 1) >> 1) + odd) >> sh};
}
__device__ __forceinline__ cx shift_cx(cx a, int sh) { return mk(shift_fx(a.x, sh), shift_fx(a.y, sh)); }

// DIFX<Z> with a shift after its second level, the last one with products.  A
// product by W_8 takes values of modulus below 2^60.5, so the inputs are below
// 2^58 (Z = 16: four are added before it) or 2^59 (Z = 8: two), or their whole sum
// is below 2^60: that part of the shift (kPre bits) comes before.
template <int Z> constexpr int kPre = Z == 16 ? 2 : 1;
template <int Z, bool INV>
__device__ __forceinline__ void dif_shift(cx* v, int sh) {
    static_assert(Z == 8 || Z == 16, "");
    level<Z, INV, 0>(v);
    level<Z / 2, INV, 0>(v);
    level<Z / 2, INV, Z / 2>(v);
    if (sh) {
#pragma unroll
        for (int i = 0; i < Z; ++i) v[i] = shift_cx(v[i], sh);
    }
    DIFX<Z / 4, INV, 0>::run(v);
    DIFX<Z / 4, INV, Z / 4>::run(v);
    DIFX<Z / 4, INV, Z / 2>::run(v);
    DIFX<Z / 4, INV, 3 * (Z / 4)>::run(v);
}

// v: this lane's E values, components below 2^62.  Shifts the line right by
// s0 (returned through ex, which it is added to) so that no lane's first pass
// can exceed 2^60, and sets the further shifts (ex also counts them): sh.x at
// the first twiddle for the second pass, a sum over C lanes, and sh.y for the
// last one, most of it between that one's levels.
template <int M>
__device__ __forceinline__ void fit_line(cx* v, int slot, LineSm<M>& sm, int& ex, int2& sh) {
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
    const int e2 = Geo<M>::STAGED ? min(et, top + Geo<M>::LOG_C) : et;
    sh.x = max(0, e2 - 22 - s0);
    sh.y = max(0, et - 22 - s0 - sh.x);
    if (s0 > 0) {
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = shift_cx(v[i], s0);
    }
    ex += s0 + sh.x + sh.y;
}

// ------------------------------------------------------------------ line transform
__device__ __forceinline__ CFac ld_fac(const int4* __restrict__ t) {
    const int4 q = __ldg(t);
    return CFac{Fac{q.x, q.y}, Fac{q.z, q.w}};
}

// The unnormalised DFT of the line (value G n1 + n2 in v[n1] of lane n2);
// the result lies in buf in natural order, visible to the line's lanes.
// tw: W_M^{n2 k1} at k1 G + n2, then (D > 1) W_B^{d kc} at kc D + d.
//   1. A-point DFT over n1, times W_M^{n2 k1}, to row k1 of the buffer;
//   2. C-point DFTs over c of the row's values D c + d, times W_B^{d kc}, back
//      to the slots they came from (D = 1: to natural order, k1 + A kc);
//   3. D-point DFTs over d of D kc + d, to natural order k1 + A (kc + C kd).
// Lanes run along d in step 2 and along k1 in the last step: both reads and
// the natural-order write are free of bank conflicts.
template <int M, bool INV>
__device__ __forceinline__ void fft_line(cx* v, cx* buf, const int4* __restrict__ tw, int n2, int slot, int2 sh) {
    using Gm = Geo<M>;
    constexpr int A = Gm::A, C = Gm::C, D = Gm::D, G = Gm::G, P = Gm::P;
    DIFX<A, INV, 0>::run(v);
#pragma unroll
    for (int r = 0; r < A; ++r) {
        const int k1 = wf::bitrev<A>(r);
        cx u = v[r];
        if (k1) u = cmulf<INV>(u, ld_fac(tw + k1 * G + n2));
        buf[k1 * P + n2] = shift_cx(u, sh.x);
    }
    sync_line<M>(slot);
    const int pre = Gm::STAGED ? min(sh.y, kPre<D>) : 0;        // of sh.y, before the last pass
    if constexpr (D > 1) {
        const int4* __restrict__ t3 = tw + M;
#pragma unroll
        for (int j = 0; j < A / C; ++j) {
            const int q = n2 + G * j, d = q % D;
            cx* row = buf + (q / D) * P + d;
            cx u[C];
#pragma unroll
            for (int c = 0; c < C; ++c) u[c] = row[D * c];
            DIFX<C, INV, 0>::run(u);
#pragma unroll
            for (int r = 0; r < C; ++r) {
                const int kc = wf::bitrev<C>(r);
                if (kc) u[r] = cmulf<INV>(u[r], ld_fac(t3 + kc * D + d));
                if (Gm::STAGED && pre) u[r] = shift_cx(u[r], pre);
                row[D * kc] = u[r];
            }
        }
        sync_line<M>(slot);
    }
    constexpr int Z = D > 1 ? D : C;              // the last DFT
#pragma unroll
    for (int j = 0; j < A / Z; ++j) {
        const int q = n2 + G * j, k1 = q % A, kc = q / A;     // D = 1: kc = 0
#pragma unroll
        for (int d = 0; d < Z; ++d) v[j * Z + d] = buf[k1 * P + Z * kc + d];
    }
    sync_line<M>(slot);
#pragma unroll
    for (int j = 0; j < A / Z; ++j) {
        const int q = n2 + G * j, k1 = q % A, kc = q / A;
        if constexpr (Gm::STAGED) dif_shift<Z, INV>(v + j * Z, sh.y - pre);
        else DIFX<Z, INV, 0>::run(v + j * Z);
#pragma unroll
        for (int r = 0; r < Z; ++r) {
            const int kd = wf::bitrev<Z>(r);
            buf[k1 + A * (D > 1 ? kc + C * kd : kd)] = v[j * Z + r];
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

// Slots: a line's N modes as M complex values, slot i = (X[i], X[N-i]) for
// i >= 1 and slot 0 = (X[0], X[M]).  The pair k fills the slots k and M-k;
// item k = 0 .. M/2 - 1 is the pair k and, for k = 0, the pairs 0 and M/2
// (slots 0 and M/2).
template <int M> __device__ __forceinline__ int slot_mode(int i, int c) {
    return c == 0 ? i : i == 0 ? M : 2 * M - i;
}
template <int M> __device__ __forceinline__ int item_slot2(int k) { return k == 0 ? M / 2 : M - k; }

// The two slots of item k from the natural-order spectrum z (a second turn
// for item 0).
template <int M> __device__ __forceinline__ void post_item(const cx* z, const PairTab& t, int k, cx& s1, cx& s2) {
    const cx A = z[k], B = z[item_slot2<M>(k)];
    const Quad64 q = post_pair(A, k == 0 ? A : B, t, k);
    s1 = mk(q.xk, q.xNk);
    s2 = mk(q.xMk, q.xMpk);
    if (k == 0) {
        const Quad64 h = post_pair(B, B, t, M / 2);
        s1.y = q.xMk;
        s2 = mk(h.xk, h.xNk);
    }
}
template <int M> __device__ __forceinline__ void pre_item(cx s1, cx s2, const PairTab& t, int k, cx* z) {
    cx a, b;
    if (k != 0) {
        pre_pair(Quad64{s1.x, s1.y, s2.x, s2.y}, t, k, a, b);
    } else {
        cx c;
        pre_pair(Quad64{s1.x, fx{0}, s1.y, s1.y}, t, 0, a, c);
        pre_pair(Quad64{s2.x, s2.y, s2.x, s2.y}, t, M / 2, b, c);
    }
    z[k] = a;
    z[item_slot2<M>(k)] = b;
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
    int ex;
    int2 sh;
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

// Inverse: the line's modes in buf as slots of doubles (orthonormal DCT
// coefficients; mx: the largest mag_hi of this lane's) to the natural-order
// samples in buf (sample m: x[4m], x[4m+2]; sample M-1-m: x[4m+3], x[4m+1]);
// the exponent in sm.ex[slot] and returned.  OWN: every lane has filled the
// slots of its own items k = n2 + G i itself.
template <int M, bool OWN>
__device__ __forceinline__ int inverse_line(unsigned mx, cx* buf, const int4* __restrict__ tw, const PairTab& ti, int n2,
                                            int slot, LineSm<M>& sm) {
    constexpr int E = Geo<M>::E, G = Geo<M>::G;
    mx = line_max<M>(mx, slot, sm);
    if constexpr (!OWN) sync_line<M>(slot);
    const bool bad = mx >= 0x7ff00000u;
    const int em = max((int)(mx >> 20), 1);
    // Room for the pairs: with modes below 2^59 the second product takes a sum of two values below 2^59.5, and a sample
    // of z is below 2^61.5.  The bits left are what the small modes of a line with a large mean are rounded by.
#pragma unroll 1
    for (int i = 0; i < E / 2; ++i) {
        const int k = n2 + G * i;
        const double2 p = reinterpret_cast<const double2*>(buf)[k], q = reinterpret_cast<const double2*>(buf)[item_slot2<M>(k)];
        pre_item<M>(mk(to_fixed(p.x, em + 1), to_fixed(p.y, em + 1)), mk(to_fixed(q.x, em + 1), to_fixed(q.y, em + 1)), ti, k,
                    buf);
    }
    int ex = em + 1 - 1082 + ti.p;
    int2 sh;
    sync_line<M>(slot);
    cx v[E];
#pragma unroll
    for (int i = 0; i < E; ++i) v[i] = buf[G * i + n2];
    sync_line<M>(slot);
    fit_line<M>(v, slot, sm, ex, sh);
    fft_line<M, true>(v, buf, tw, n2, slot, sh);
    if (bad) ex = kBad;
    if (n2 == 0) sm.ex[slot] = ex;
    return ex;
}

// x[4m .. 4m+3] from the natural-order samples
template <int M> __device__ __forceinline__ vec4<double> unpack_item(const cx* z, int m, int ex) {
    const cx a = z[m], b = z[M - 1 - m];
    return {line_double(a.x, ex), line_double(b.y, ex), line_double(a.y, ex), line_double(b.x, ex)};
}

}  // namespace xf
}  // namespace ccm

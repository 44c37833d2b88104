// wide_kernels.cuh -- FP32 kernels on the lines of wide_fft.cuh: the
// Neumann / Dirichlet solver (N = 64 .. 8192), the preconditioner of the
// classical scheme, and the periodic solver (N = 64 .. 4096).
#pragma once
#include "step_kernels.cuh"
#include "wide_fft.cuh"
#include "wide_ops.h"

namespace ccm {
namespace lf {

// Forward DCT-II along x of LINES rows of field blockIdx.y, transposed write
// out[f][kx][y0 + r].  n: values per array (index checks).
template <int M, bool DST>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
kl_row_fwd(const float* __restrict__ in, float* __restrict__ out, const float2* __restrict__ tw, PairTab tf,
           const int* __restrict__ dskip, size_t fstride, size_t n) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N;
    if (dskip && dskip[blockIdx.y]) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    cf* bufs = reinterpret_cast<cf*>(smraw);
    int n2, slot;
    lane_of<M>(n2, slot);
    const size_t f0 = blockIdx.y * fstride;
    const int y0 = blockIdx.x * Gm::LINES;
    forward_line<M, DST>(in + CCM_IXW(f0 + (size_t)(y0 + slot) * N, N, n), bufs + (size_t)slot * Gm::BUF, tw, n2, slot,
                         (y0 + slot) & 1);
    __syncthreads();
    write_modes<M, Gm::LINES>(bufs, out + f0 + y0, tf, f0 + y0, n);
}

// v / (c0 + s (c1 + c2 s)), s = ex + ey, with the divisor in double-float
// arithmetic (TwoSum / FMA products, relative error about 2^-44): the quotient
// is that of an FP64 divisor to within its FP32 rounding, without the FP64
// instructions (eight per value).
struct DivCoef { float2 c0, c1, c2; };           // high and low parts
__device__ __forceinline__ void divisor(float2 ex, float2 ey, const DivCoef& c, float& dh, float& dl) {
    float sh, sl;
    two_sum(ex.x, ey.x, sh, sl);
    sl += ex.y + ey.y;
    // t = c2 s + c1
    float p = c.c2.x * sh, e = fmaf(c.c2.x, sh, -p);
    e = fmaf(c.c2.x, sl, fmaf(c.c2.y, sh, e));
    float th, tl;
    two_sum(p, c.c1.x, th, tl);
    tl += e + c.c1.y;
    // d = t s + c0
    p = th * sh;
    e = fmaf(th, sh, -p);
    e = fmaf(th, sl, fmaf(tl, sh, e));
    two_sum(p, c.c0.x, dh, dl);
    dl += e + c.c0.y;
}
__device__ __forceinline__ float div_mode(float v, float2 ex, float2 ey, const DivCoef& c) {
    float dh, dl;
    divisor(ex, ey, c, dh, dl);
    const float r = __frcp_rn(dh);
    const float q = v * r;
    return fmaf(fmaf(-q, dl, fmaf(-q, dh, v)), r, q);
}

// LINES spectral rows (contiguous over y): forward DCT along y, division by
// c0 + c1 s + c2 s^2, inverse DCT, transposed write out[y][kx].  ev
// holds the eigenvalues times a power of two and c the coefficients times its
// inverse powers; dcoef: coefficients formed on the device (FP64), brought to
// that scale by s1 and s2.
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
kl_col_solve(const float* __restrict__ in, float* __restrict__ out, const float2* __restrict__ tw, PairTab tf,
             PairTab ti, const float2* __restrict__ ev, DivCoef c, const double* __restrict__ dcoef, double s1,
             double s2, const int* __restrict__ dskip, size_t fstride) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, E = Gm::E, G = Gm::G;
    if (dskip && dskip[blockIdx.y]) return;
    if (dcoef) {
        auto pair = [](double x) { const float h = (float)x; return make_float2(h, (float)(x - (double)h)); };
        c.c0 = pair(dcoef[0]); c.c1 = pair(dcoef[1] * s1); c.c2 = pair(dcoef[2] * s2);
    }
    extern __shared__ __align__(16) unsigned char smraw[];
    cf* bufs = reinterpret_cast<cf*>(smraw);
    int n2, slot;
    lane_of<M>(n2, slot);
    cf* buf = bufs + (size_t)slot * Gm::BUF;
    const int x0 = blockIdx.x * Gm::LINES, kx = x0 + slot;
    forward_line<M, false>(in + CCM_IXW(blockIdx.y * fstride + (size_t)kx * N, N, gridDim.y * fstride), buf, tw, n2, slot, false);
    const float2 ex = __ldg(ev + kx);
#pragma unroll 2
    for (int j = 0; j < E / 2; ++j) {
        const int k = n2 + G * j, i2 = item_slot2<M>(k);
        cf s1, s2;
        post_item<M>(buf, tf, k, s1, s2);
        s1.x = div_mode(s1.x, ex, __ldg(ev + slot_mode<M>(k, 0)), c);
        s1.y = div_mode(s1.y, ex, __ldg(ev + slot_mode<M>(k, 1)), c);
        s2.x = div_mode(s2.x, ex, __ldg(ev + slot_mode<M>(i2, 0)), c);
        s2.y = div_mode(s2.y, ex, __ldg(ev + slot_mode<M>(i2, 1)), c);
        pre_item<M>(s1, s2, ti, k, buf);               // the slots this item read
    }
    sync_line<M>(slot);
    inverse_line<M>(buf, tw, n2, slot);
    __syncthreads();
    write_samples<M, Gm::LINES>(bufs, out + blockIdx.y * fstride + x0, blockIdx.y * fstride + x0, gridDim.y * fstride);
}

// Inverse DCT along x of LINES rows (in place allowed).  DST: times (-1)^(i+j).
template <int M, bool DST>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
kl_row_inv(const float* in, float* out, const float2* __restrict__ tw, PairTab ti, const int* __restrict__ dskip,
           size_t fstride) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, E = Gm::E, G = Gm::G;
    if (dskip && dskip[blockIdx.y]) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    int n2, slot;
    lane_of<M>(n2, slot);
    cf* buf = reinterpret_cast<cf*>(smraw) + (size_t)slot * Gm::BUF;
    const int y = blockIdx.x * Gm::LINES + slot;
    const size_t o = blockIdx.y * fstride + (size_t)y * N, n = gridDim.y * fstride;
    const float* row = in + CCM_IXW(o, N, n);
#pragma unroll
    for (int j = 0; j < E / 2; ++j) {
        const int k = n2 + G * j, i2 = item_slot2<M>(k);
        pre_item<M>(mk(row[k], row[slot_mode<M>(k, 1)]), mk(row[i2], row[slot_mode<M>(i2, 1)]), ti, k, buf);
    }
    sync_line<M>(slot);
    inverse_line<M>(buf, tw, n2, slot);
#pragma unroll
    for (int j = 0; j < E / 2; ++j) {
        const int m = n2 + G * j;
        if (!CCM_OKW(o + 4 * m, 4, n)) continue;
        const cf a = buf[m], b = buf[M - 1 - m];
        const float s = DST && (y & 1) ? -1.f : 1.f;    // x = 4m is even: signs (+, -, +, -) times (-1)^y
        *reinterpret_cast<float4*>(out + o + 4 * m) =
            DST ? make_float4(s * a.x, -s * b.y, s * a.y, -s * b.x) : make_float4(a.x, b.y, a.y, b.x);
    }
}

// ------------------------------------------------------------------ periodic solver
// The field is real: a row of N = 2M values is the complex line x[2m] + i x[2m+1]
// of length M, its spectrum the pairs (k, M-k)
//   X[k] = E + W O, X[M-k] = conj(E - W O), W = e^{-2 pi i k/N},
//   E = (Z[k] + conj Z[M-k])/2, O = (Z[k] - conj Z[M-k])/(2i),
// and only the columns kx = 0 .. M-1 are transformed along y (complex lines of
// length N), the real rows X[0] and X[M] together as the column X[0] + i X[M].
// Half the lines and half the traffic of full-length complex transforms, but for
// the last pass (kp_row_inv).

// Row spectra of LINES rows, written transposed: outc[kx N + y].
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
kp_row_fwd(const float* __restrict__ in, float2* __restrict__ outc, const float2* __restrict__ tw, PairTab t) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, E = Gm::E, G = Gm::G, R2 = Gm::LINES / 2;
    extern __shared__ __align__(16) unsigned char smraw[];
    cf* bufs = reinterpret_cast<cf*>(smraw);
    int n2, slot;
    lane_of<M>(n2, slot);
    const int y0 = blockIdx.x * Gm::LINES;
    {
        const float2* x = reinterpret_cast<const float2*>(in + CCM_IXW((size_t)(y0 + slot) * N, N, (size_t)N * N));
        cf v[E];
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = ld_c(x + G * i + n2);
        fft_line<M, false, true>(v, bufs + (size_t)slot * Gm::BUF, tw, n2, slot);
    }
    __syncthreads();
#pragma unroll 1
    for (int q = threadIdx.x; q < R2 * (M / 2); q += Gm::THREADS) {
        const int r2 = q % R2, k = q / R2;
        const cf w = mk(__ldg(t.wa + k).x, __ldg(t.wa + k).y);
        cf a[2], b[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const cf* z = bufs + (size_t)(2 * r2 + r) * Gm::BUF;
            const cf A = z[k], B = z[item_slot2<M>(k)];
            if (k == 0) {
                a[r] = mk(A.x + A.y, A.x - A.y);              // X[0] and X[M]
                b[r] = mk(B.x, -B.y);                         // X[M/2] = conj Z[M/2]
            } else {
                const cf e = mk(0.5f * (A.x + B.x), 0.5f * (A.y - B.y)), o = mk(0.5f * (A.y + B.y), 0.5f * (B.x - A.x));
                a[r] = mk(fmaf(w.x, o.x, fmaf(-w.y, o.y, e.x)), fmaf(w.x, o.y, fmaf(w.y, o.x, e.y)));       // e + w o
                b[r] = mk(fmaf(-w.x, o.x, fmaf(w.y, o.y, e.x)), fmaf(w.x, o.y, fmaf(w.y, o.x, -e.y)));      // conj(e - w o)
            }
        }
        const size_t oa = (size_t)k * N + y0 + 2 * r2, ob = (size_t)item_slot2<M>(k) * N + y0 + 2 * r2;
        if (CCM_OKW(oa, 2, (size_t)M * N)) *reinterpret_cast<float4*>(outc + oa) = make_float4(a[0].x, a[0].y, a[1].x, a[1].y);
        if (CCM_OKW(ob, 2, (size_t)M * N)) *reinterpret_cast<float4*>(outc + ob) = make_float4(b[0].x, b[0].y, b[1].x, b[1].y);
    }
}

// 1 / (c0 + s (c1 + c2 s)) rounded to FP32, times sc (a power of two)
__device__ __forceinline__ float recip_mode(float2 ex, float2 ey, const DivCoef& c, float sc) {
    float dh, dl;
    divisor(ex, ey, c, dh, dl);
    const float r = __frcp_rn(dh);
    return sc * fmaf(r, fmaf(-r, dl, fmaf(-r, dh, 1.0f)), r);
}

// LINES columns kx of N complex values (Geo of line length N): FFT along y,
// division, inverse FFT, transposed write outc[y (N/2) + kx].  sc: the
// normalisation 1 / N^2 of the two inverse passes.
template <int N>
__global__ void __launch_bounds__(Geo<N>::THREADS, Geo<N>::MINB)
kp_col(const float2* __restrict__ inc, float2* __restrict__ outc, const float2* __restrict__ tw,
       const float2* __restrict__ ev, DivCoef c, float sc) {
    using Gm = Geo<N>;
    constexpr int M = N / 2, E = Gm::E, G = Gm::G, R2 = Gm::LINES / 2;
    extern __shared__ __align__(16) unsigned char smraw[];
    cf* bufs = reinterpret_cast<cf*>(smraw);
    int n2, slot;
    lane_of<N>(n2, slot);
    cf* buf = bufs + (size_t)slot * Gm::BUF;
    const int x0 = blockIdx.x * Gm::LINES, kx = x0 + slot;
    {
        cf v[E];
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = ld_c(inc + CCM_IX((size_t)kx * N + G * i + n2, (size_t)M * N));
        fft_line<N, false, true>(v, buf, tw, n2, slot);
    }
    const float2 ex = __ldg(ev + kx);
    if (kx != 0) {
#pragma unroll 2
        for (int i = 0; i < E; ++i) {
            const int k = G * i + n2;
            buf[k] = scale(buf[k], recip_mode(ex, __ldg(ev + k), c, sc));
        }
    } else {
        // Z = P + i Q with P, Q the spectra of the real columns X[0], X[M]: pairs (k, N-k)
        const float2 eM = __ldg(ev + M);
#pragma unroll 1
        for (int k = n2; k <= M; k += G) {
            const int m = (N - k) & (N - 1);
            const cf A = buf[k], B = buf[m];
            const cf P = mk(0.5f * (A.x + B.x), 0.5f * (A.y - B.y)), Q = mk(0.5f * (A.y + B.y), 0.5f * (B.x - A.x));
            const float2 ey = __ldg(ev + k);
            const cf p = scale(P, recip_mode(ex, ey, c, sc)), q = scale(Q, recip_mode(eM, ey, c, sc));
            buf[k] = mk(p.x - q.y, p.y + q.x);
            if (m != k) buf[m] = mk(p.x + q.y, q.x - p.y);
        }
    }
    sync_line<N>(slot);
    inverse_line<N, true>(buf, tw, n2, slot);
    __syncthreads();
#pragma unroll 2
    for (int q = threadIdx.x; q < R2 * N; q += Gm::THREADS) {
        const int r2 = q % R2, y = q / R2;
        const cf a = bufs[(size_t)(2 * r2) * Gm::BUF + y], b = bufs[(size_t)(2 * r2 + 1) * Gm::BUF + y];
        const size_t o = (size_t)y * M + x0 + 2 * r2;
        if (CCM_OKW(o, 2, (size_t)M * N)) *reinterpret_cast<float4*>(outc + o) = make_float4(a.x, a.y, b.x, b.y);
    }
}

// Inverse of kp_row_fwd: LINES rows inc[y (N/2) + kx] to real rows out[y N + x],
// as full complex lines (Geo of line length N) whose imaginary part is dropped.
// Half-length lines (as in the forward pass) are half the work but carry all of
// the transform's rounding in the result instead of half of its variance: with
// them the solve was 1.12 times as far off as with full-length transforms
// throughout (N = 32 .. 4096, up to 1.33 where the divisor damps the noise of
// the earlier passes).
template <int N>
__global__ void __launch_bounds__(Geo<N>::THREADS, Geo<N>::MINB)
kp_row_inv(const float2* __restrict__ inc, float* __restrict__ out, const float2* __restrict__ tw) {
    using Gm = Geo<N>;
    constexpr int M = N / 2, E = Gm::E, G = Gm::G;
    extern __shared__ __align__(16) unsigned char smraw[];
    int n2, slot;
    lane_of<N>(n2, slot);
    cf* buf = reinterpret_cast<cf*>(smraw) + (size_t)slot * Gm::BUF;
    const int y = blockIdx.x * Gm::LINES + slot;
    const float2* row = inc + CCM_IXW((size_t)y * M, M, (size_t)M * N);
#pragma unroll
    for (int j = 0; j < E / 2; ++j) {
        const int k = n2 + G * j;
        const cf A = ld_c(row + k);
        buf[k] = k == 0 ? mk(A.x, 0.f) : A;                   // row 0 holds X[0] + i X[M]
        buf[k == 0 ? M : N - k] = k == 0 ? mk(A.y, 0.f) : conj_(A);
    }
    sync_line<N>(slot);
    inverse_line<N, true>(buf, tw, n2, slot);
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const size_t o = (size_t)y * N + G * i + n2;
        if (CCM_OK(o, (size_t)N * N)) out[o] = buf[G * i + n2].x;
    }
}

}  // namespace lf
}  // namespace ccm

// fixed_kernels.cuh -- FP64 kernels on the fixed-point line transforms of
// fixed_fft.cuh (N = 64 .. 8192): the step's four transform kernels, with the
// data flow of the block-FFT kernels of step_kernels.cuh, and the three of
// the Neumann / Dirichlet solver (spectral_solve.cu, and the preconditioner
// of the classical scheme).
//
// Spectra: spec[kx][f][4 k + u], f = f0' S H Q K P g0' L_P, item k = 0 .. M/2 - 1,
// u its four modes (fixed_fft.cuh, item_mode): every access to them is 32
// contiguous bytes per lane.  isig = 1/sigma and itau = 1/tau are tables in
// the same order (they depend on the parameters only; evaluating them costs
// ten FP64 instructions a mode in each of two kernels, reading them 16 bytes).
#pragma once
#include "step_kernels.cuh"
#include "fixed_fft.cuh"
#include "fixed_ops.h"

namespace ccm {
namespace xf {

inline PairTab pair_fwd(const Tables& t) {
    const int n = t.M / 2 + 1;
    return PairTab{t.mem + t.M, t.mem + t.M + n, t.mem + t.M + 2 * n, -t.pf};
}
inline PairTab pair_inv(const Tables& t) {
    const int n = t.M / 2 + 1;
    return PairTab{t.mem + t.M, t.mem + t.M + 3 * n, t.mem + t.M + 4 * n, -t.pi};
}

// ------------------------------------------------------------------ forward rows
// Forward DCT-II along x of LINES rows of field blockIdx.y, written
// transposed: out[f][kx][y0 + r].  n: values per array (index checks).
template <int M, bool DST>
__global__ void __launch_bounds__(Geo<M>::THREADS)
kx_row_fwd(const double* __restrict__ in, double* __restrict__ out, const int4* __restrict__ tw2, PairTab tf,
           const int* __restrict__ dskip, size_t fstride, size_t n) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, L = Gm::LINES;
    if (dskip && dskip[blockIdx.y]) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    cx* bufs = reinterpret_cast<cx*>(smraw);
    int n2, slot;
    lane_of<M>(n2, slot);
    const size_t f0 = blockIdx.y * fstride;
    const int y0 = blockIdx.x * L;
    forward_line<M, DST>(in + CCM_IXW(f0 + (size_t)(y0 + slot) * N, N, n), bufs + (size_t)slot * Gm::BUF, tw2, n2, slot, sm,
                         (y0 + slot) & 1);
    __syncthreads();
    for (int q = threadIdx.x; q < L * (M / 2); q += Gm::THREADS) {
        const int r = q % L, k = q / L, ex = sm.ex[r];
        const Quad64 X = post_item<M>(bufs + (size_t)r * Gm::BUF, tf, k);
        const fx v[4] = {X.xk, X.xNk, X.xMk, X.xMpk};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const size_t o = f0 + (size_t)item_mode<M>(k, u) * N + y0 + r;
            if (CCM_OK(o, n)) out[o] = line_double(v[u], ex, tf.p);
        }
    }
}

// ------------------------------------------------------------------ forward columns and Gram sums
// The sixteen Gram sums of one mode (f0' f0' is not needed: the slot stays 0).
__device__ __forceinline__ void gram_mode(double (&acc)[16], const double (&v)[NF], double isig, double itau) {
    int p = 0;
#pragma unroll
    for (int b = 1; b < 5; ++b) {
        const double w = v[b] * isig;
        acc[p] = fma(v[0], w, acc[p]);
        ++p;
#pragma unroll
        for (int a = 1; a <= b; ++a) {
            acc[p] = fma(v[a], w, acc[p]);
            ++p;
        }
    }
    const double w = v[5] * itau;
    acc[14] = fma(v[6], w, acc[14]);
    acc[15] = fma(v[7], w, acc[15]);
}
// Order of acc above -> column of a partial row (a <= b over f0' S H Q K row by row, PG, PL)
__device__ __forceinline__ int gram_col(int p) {
    // p: (0,1) (1,1) | (0,2) (1,2) (2,2) | (0,3) (1,3) (2,3) (3,3) | (0,4) .. (4,4) | PG PL
    if (p >= 14) return p + 1;
    const int b = p < 2 ? 1 : p < 5 ? 2 : p < 9 ? 3 : 4;
    const int a = p - (b == 1 ? 0 : b == 2 ? 2 : b == 3 ? 5 : 9);
    return a * 5 - a * (a - 1) / 2 + (b - a);
}
// Block sum of the sixteen accumulators into a partial row.  Recursive
// halving: at each of four exchanges a lane keeps half of its values (15
// additions and a last one, instead of 80 for sixteen butterfly sums).
template <int THREADS>
__device__ __forceinline__ void gram_store(double (&acc)[16], double* __restrict__ row, double* __restrict__ sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int idx = 0;
#pragma unroll
    for (int h = 8; h >= 1; h >>= 1) {
        const bool up = lane & h;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double give = up ? acc[i] : acc[i + h], keep = up ? acc[i + h] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, h);
        }
        if (up) idx += h;
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 16);
    __syncthreads();
    if (lane < 16) sm[warp * 16 + idx] = acc[0];
    __syncthreads();
    if (threadIdx.x < 16) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) s += sm[w * 16 + threadIdx.x];
        row[gram_col(threadIdx.x)] = s;
    }
    if (threadIdx.x == 16) row[0] = 0.0;
}
__device__ __forceinline__ vec4<double> ldq(const double* __restrict__ p) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    return {a.x, a.y, b.x, b.y};
}

// Forward DCT-II along y of the eight fields of a spectral row kx (one line
// per lane group), the spectra and the Gram sums; each CTA takes the rows
// blockIdx.x, blockIdx.x + gridDim.x, ... and leaves one partial row.
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS)
kx_col_gram(const double* __restrict__ in, double* __restrict__ spec, double* __restrict__ part,
            const int4* __restrict__ tw2, PairTab tf, const double* __restrict__ isig, const double* __restrict__ itau) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N;
    static_assert(Gm::LINES == NF, "one line per field");
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    cx* bufs = reinterpret_cast<cx*>(smraw);
    int n2, slot;
    lane_of<M>(n2, slot);
    const size_t NN = (size_t)N * N;
    double acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.0;
    for (int kx = blockIdx.x; kx < N; kx += gridDim.x) {
        forward_line<M, false>(in + CCM_IXW(slot * NN + (size_t)kx * N, N, NF * NN), bufs + (size_t)slot * Gm::BUF, tw2, n2,
                               slot, sm, false);
        __syncthreads();
        for (int k = threadIdx.x; k < M / 2; k += Gm::THREADS) {
            double v[4][NF];
            double* srow = spec + CCM_IXW((size_t)kx * NF * N, NF * N, NF * NN) + 4 * k;
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const Quad64 q = post_item<M>(bufs + (size_t)f * Gm::BUF, tf, k);
                const int ex = sm.ex[f];
                v[0][f] = line_double(q.xk, ex, tf.p); v[1][f] = line_double(q.xNk, ex, tf.p);
                v[2][f] = line_double(q.xMk, ex, tf.p); v[3][f] = line_double(q.xMpk, ex, tf.p);
                if (f != 5) st4(srow + (size_t)f * N, vec4<double>{v[0][f], v[1][f], v[2][f], v[3][f]});
            }
            const vec4<double> ws = ldq(isig + (size_t)kx * N + 4 * k), wt = ldq(itau + (size_t)kx * N + 4 * k);
            gram_mode(acc, v[0], ws.a, wt.a);
            gram_mode(acc, v[1], ws.b, wt.b);
            gram_mode(acc, v[2], ws.c, wt.c);
            gram_mode(acc, v[3], ws.d, wt.d);
        }
        __syncthreads();
    }
    gram_store<Gm::THREADS>(acc, part + (size_t)blockIdx.x * NRED2, reinterpret_cast<double*>(smraw));
}

// Lines too long for eight buffers per CTA (M >= 2048): the spectra of LINES
// rows of field blockIdx.y, and the Gram sums from them in a second kernel.
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS)
kx_col_fwd(const double* __restrict__ in, double* __restrict__ spec, const int4* __restrict__ tw2, PairTab tf) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    int n2, slot;
    lane_of<M>(n2, slot);
    cx* buf = reinterpret_cast<cx*>(smraw) + (size_t)slot * Gm::BUF;
    const size_t NN = (size_t)N * N;
    const int f = blockIdx.y, kx = blockIdx.x * Gm::LINES + slot;
    const int ex = forward_line<M, false>(in + CCM_IXW(f * NN + (size_t)kx * N, N, NF * NN), buf, tw2, n2, slot, sm, false);
    double* srow = spec + CCM_IXW(((size_t)kx * NF + f) * N, N, NF * NN);
    for (int k = n2; k < M / 2; k += Gm::G) {
        const Quad64 q = post_item<M>(buf, tf, k);
        st4(srow + 4 * k, vec4<double>{line_double(q.xk, ex, tf.p), line_double(q.xNk, ex, tf.p),
                                       line_double(q.xMk, ex, tf.p), line_double(q.xMpk, ex, tf.p)});
    }
}
constexpr int kGramThreads = 256;
static __global__ void __launch_bounds__(kGramThreads)
kx_gram_rows(const double* __restrict__ spec, double* __restrict__ part, int N, const double* __restrict__ isig,
             const double* __restrict__ itau) {
    __shared__ double sm[kGramThreads / 32 * 16];
    double acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.0;
    for (int kx = blockIdx.x; kx < N; kx += gridDim.x)
        for (int j = threadIdx.x; j < N; j += kGramThreads) {
            double v[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) v[f] = __ldg(spec + ((size_t)kx * NF + f) * N + j);
            gram_mode(acc, v, __ldg(isig + (size_t)kx * N + j), __ldg(itau + (size_t)kx * N + j));
        }
    gram_store<kGramThreads>(acc, part + (size_t)blockIdx.x * NRED2, sm);
}

// isig, itau in the order of the spectra
template <int M> __device__ __forceinline__ int slot_mode(int j) { return item_mode<M>(j >> 2, j & 3); }
template <int M>
__global__ void kx_weights(const double* __restrict__ ev, SpecCoef sc, double* __restrict__ isig, double* __restrict__ itau) {
    constexpr size_t N = 2 * M;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < N * N; q += (size_t)gridDim.x * blockDim.x) {
        const double s = ev[q / N] + ev[slot_mode<M>((int)(q % N))];
        isig[q] = recip(fma(fma(sc.C3, s, sc.C2), s, sc.C1));
        itau[q] = recip(fma(sc.lam, s, sc.Ct));
    }
}

// ------------------------------------------------------------------ recovery and inverse columns
// Transposed write of the LINES natural-order lines of a CTA: out[y][x0 + r].
template <int M>
__device__ __forceinline__ void write_transposed(const cx* bufs, const LineSm<M>& sm, double* __restrict__ out, size_t base,
                                                 int x0, size_t n) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, L = Gm::LINES;
    for (int q = threadIdx.x; q < L * (M / 2); q += Gm::THREADS) {
        const int r = q % L, m = q / L;
        const vec4<double> v = unpack_item<M>(bufs + (size_t)r * Gm::BUF, m, sm.ex[r]);
        const size_t o = base + (size_t)(4 * m) * N + x0 + r;
        if (CCM_OK(o + 3 * (size_t)N, n)) {
            out[o] = v.a;
            out[o + N] = v.b;
            out[o + 2 * (size_t)N] = v.c;
            out[o + 3 * (size_t)N] = v.d;
        }
    }
}

// LINES spectral rows of field blockIdx.y (0: phi, 1: psi): recovery
// combination, inverse DCT along y, transposed write out[f][y][kx].
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS)
kx_comb_icol(const double* __restrict__ spec, double* __restrict__ out, const int4* __restrict__ tw2, PairTab ti,
             const double* __restrict__ isig, const double* __restrict__ itau, const DevScalars* __restrict__ dsc) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, E = Gm::E, G = Gm::G;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    cx* bufs = reinterpret_cast<cx*>(smraw);
    int n2, slot;
    lane_of<M>(n2, slot);
    const size_t NN = (size_t)N * N;
    const int f = blockIdx.y, x0 = blockIdx.x * Gm::LINES, kx = x0 + slot;
    const double* s = spec + CCM_IXW((size_t)kx * NF * N, NF * N, NF * NN);
    double X[2 * E];
    if (f == 0) {
        const double aS = -dsc->alpha[0], aH = -dsc->alpha[1], aQ = -dsc->alpha[2], aK = -dsc->alpha[3];
#pragma unroll
        for (int i = 0; i < E / 2; ++i) {
            const int o = 4 * (n2 + G * i);
            const vec4<double> v0 = ldq(s + o), v1 = ldq(s + N + o), v2 = ldq(s + 2 * N + o), v3 = ldq(s + 3 * N + o),
                               v4 = ldq(s + 4 * N + o), w = ldq(isig + (size_t)kx * N + o);
            X[4 * i] = fma(aK, v4.a, fma(aQ, v3.a, fma(aH, v2.a, fma(aS, v1.a, v0.a)))) * w.a;
            X[4 * i + 1] = fma(aK, v4.b, fma(aQ, v3.b, fma(aH, v2.b, fma(aS, v1.b, v0.b)))) * w.b;
            X[4 * i + 2] = fma(aK, v4.c, fma(aQ, v3.c, fma(aH, v2.c, fma(aS, v1.c, v0.c)))) * w.c;
            X[4 * i + 3] = fma(aK, v4.d, fma(aQ, v3.d, fma(aH, v2.d, fma(aS, v1.d, v0.d)))) * w.d;
        }
    } else {
        const double aL = dsc->alpha[4];
#pragma unroll
        for (int i = 0; i < E / 2; ++i) {
            const int o = 4 * (n2 + G * i);
            const vec4<double> v6 = ldq(s + 6 * N + o), v7 = ldq(s + 7 * N + o), w = ldq(itau + (size_t)kx * N + o);
            X[4 * i] = fma(aL, v7.a, v6.a) * w.a;
            X[4 * i + 1] = fma(aL, v7.b, v6.b) * w.b;
            X[4 * i + 2] = fma(aL, v7.c, v6.c) * w.c;
            X[4 * i + 3] = fma(aL, v7.d, v6.d) * w.d;
        }
    }
    inverse_line<M>(X, bufs + (size_t)slot * Gm::BUF, tw2, ti, n2, slot, sm);
    __syncthreads();
    write_transposed<M>(bufs, sm, out, f * NN, x0, 2 * NN);
}

// ------------------------------------------------------------------ inverse rows
// This lane's modes of a row in natural order.
template <int M> __device__ __forceinline__ void load_modes(double (&X)[2 * Geo<M>::E], const double* row, int n2) {
#pragma unroll
    for (int i = 0; i < Geo<M>::E / 2; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) X[4 * i + u] = row[item_mode<M>(n2 + Geo<M>::G * i, u)];
}

// Inverse DCT along x of LINES rows of field blockIdx.y and
// u^{n+1} = u_bar + du.
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS)
kx_irow(const double* __restrict__ in, double* __restrict__ phi_new, double* __restrict__ psi_new,
        const int4* __restrict__ tw2, PairTab ti, const double* __restrict__ phn, const double* __restrict__ pho,
        const double* __restrict__ psn, const double* __restrict__ pso, int bdf1) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, E = Gm::E, G = Gm::G;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    int n2, slot;
    lane_of<M>(n2, slot);
    cx* buf = reinterpret_cast<cx*>(smraw) + (size_t)slot * Gm::BUF;
    const size_t NN = (size_t)N * N;
    const int f = blockIdx.y, y = blockIdx.x * Gm::LINES + slot;
    double X[2 * E];
    load_modes<M>(X, in + CCM_IXW(f * NN + (size_t)y * N, N, 2 * NN), n2);
    const int ex = inverse_line<M>(X, buf, tw2, ti, n2, slot, sm);
    const double* un = f ? psn : phn;
    const double* uo = f ? pso : pho;
    double* u = f ? psi_new : phi_new;
    for (int m = n2; m < M / 2; m += G) {
        const size_t o = CCM_IXW((size_t)y * N + 4 * m, 4, NN);
        const vec4<double> d = unpack_item<M>(buf, m, ex), a = ld4(un + o), b = ld4(uo + o);
        st4(u + o, vec4<double>{bar_add(a.a, b.a, d.a, 0.0, bdf1 != 0), bar_add(a.b, b.b, d.b, 0.0, bdf1 != 0),
                                bar_add(a.c, b.c, d.c, 0.0, bdf1 != 0), bar_add(a.d, b.d, d.d, 0.0, bdf1 != 0)});
    }
}

// ------------------------------------------------------------------ solver
// LINES spectral rows (contiguous over y): forward DCT along y, division by
// c0 + c1 s + c2 s^2, inverse DCT, transposed write out[y][kx].
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS)
kx_col_solve(const double* __restrict__ in, double* __restrict__ out, const int4* __restrict__ tw2, PairTab tf, PairTab ti,
             const double* __restrict__ ev, double c0, double c1, double c2, const double* __restrict__ dcoef,
             const int* __restrict__ dskip, size_t fstride) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, E = Gm::E, G = Gm::G;
    if (dskip && dskip[blockIdx.y]) return;
    if (dcoef) { c0 = dcoef[0]; c1 = dcoef[1]; c2 = dcoef[2]; }   // coefficients formed on the device
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    cx* bufs = reinterpret_cast<cx*>(smraw);
    int n2, slot;
    lane_of<M>(n2, slot);
    cx* buf = bufs + (size_t)slot * Gm::BUF;
    const int x0 = blockIdx.x * Gm::LINES, kx = x0 + slot;
    const int ex = forward_line<M, false>(in + blockIdx.y * fstride + (size_t)kx * N, buf, tw2, n2, slot, sm, false);
    const double evx = ev[kx];
    double X[2 * E];
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
        const int k = n2 + G * i;
        const Quad64 q = post_item<M>(buf, tf, k);
        const fx v[4] = {q.xk, q.xNk, q.xMk, q.xMpk};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const double s = evx + __ldg(ev + item_mode<M>(k, u));
            X[4 * i + u] = line_double(v[u], ex, tf.p) * recip(c0 + s * (c1 + c2 * s));
        }
    }
    inverse_line<M>(X, buf, tw2, ti, n2, slot, sm);    // writes only the slots this lane has read before its first barrier
    __syncthreads();
    write_transposed<M>(bufs, sm, out, blockIdx.y * fstride, x0, ~(size_t)0);
}

// Inverse DCT along x of LINES rows (in place allowed).  DST: times (-1)^(i+j).
template <int M, bool DST>
__global__ void __launch_bounds__(Geo<M>::THREADS)
kx_row_inv(const double* in, double* out, const int4* __restrict__ tw2, PairTab ti, const int* __restrict__ dskip,
           size_t fstride) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, E = Gm::E, G = Gm::G;
    if (dskip && dskip[blockIdx.y]) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    int n2, slot;
    lane_of<M>(n2, slot);
    cx* buf = reinterpret_cast<cx*>(smraw) + (size_t)slot * Gm::BUF;
    const int y = blockIdx.x * Gm::LINES + slot;
    const size_t o = blockIdx.y * fstride + (size_t)y * N;
    double X[2 * E];
    load_modes<M>(X, in + o, n2);
    const int ex = inverse_line<M>(X, buf, tw2, ti, n2, slot, sm);
    for (int m = n2; m < M / 2; m += G) {
        vec4<double> v = unpack_item<M>(buf, m, ex);
        if (DST) {                                     // x = 4m is even: signs (+, -, +, -) times (-1)^y
            const double s = (y & 1) ? -1.0 : 1.0;
            v.a *= s; v.b *= -s; v.c *= s; v.d *= -s;
        }
        st4(out + o + 4 * m, v);
    }
}

}  // namespace xf
}  // namespace ccm

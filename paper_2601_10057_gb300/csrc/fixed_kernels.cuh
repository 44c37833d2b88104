// fixed_kernels.cuh -- FP64 kernels on the fixed-point line transforms of
// fixed_fft.cuh (N = 64 .. 8192): the step's four transform kernels, with the
// data flow of the block-FFT kernels of step_kernels.cuh, and the three of
// the Neumann / Dirichlet solver (spectral_solve.cu, and the preconditioner
// of the classical scheme).
//
// Spectra: spec[kx][f][2 i + c], f = f0' S H Q K P g0' L_P, in the slot order of
// fixed_fft.cuh: sixteen contiguous bytes per slot.  isig = 1/sigma and itau =
// 1/tau are tables in the same order (they depend on the parameters only;
// evaluating them costs ten FP64 instructions a mode in each of two kernels,
// reading them 16 bytes).
#pragma once
#include "step_kernels.cuh"
#include "fixed_fft.cuh"
#include "fixed_ops.h"

namespace ccm {
namespace xf {

inline PairTab pair_fwd(const Tables& t) {
    const int n = t.M / 2 + 1;
    return PairTab{t.mem + 2 * t.M, t.mem + 2 * t.M + n, t.mem + 2 * t.M + 2 * n, -t.pf};
}
inline PairTab pair_inv(const Tables& t) {
    const int n = t.M / 2 + 1;
    return PairTab{t.mem + 2 * t.M, t.mem + 2 * t.M + 3 * n, t.mem + 2 * t.M + 4 * n, -t.pi};
}

// ------------------------------------------------------------------ forward rows
// Forward DCT-II along x of LINES rows of field blockIdx.y, written
// transposed: out[f][kx][y0 + r].  n: values per array (index checks).
template <int M, bool DST>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
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
#pragma unroll 1
    for (int q = threadIdx.x; q < L * (M / 2); q += Gm::THREADS) {
        const int r = q % L, k = q / L, ex = sm.ex[r];
        cx s[2];
        post_item<M>(bufs + (size_t)r * Gm::BUF, tf, k, s[0], s[1]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = u ? item_slot2<M>(k) : k;
            const size_t o0 = f0 + (size_t)slot_mode<M>(i, 0) * N + y0 + r, o1 = f0 + (size_t)slot_mode<M>(i, 1) * N + y0 + r;
            if (CCM_OK(o0, n)) out[o0] = line_double(s[u].x, ex, tf.p);
            if (CCM_OK(o1, n)) out[o1] = line_double(s[u].y, ex, tf.p);
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
__device__ __forceinline__ double2 ld2(const double* __restrict__ p) { return __ldg(reinterpret_cast<const double2*>(p)); }

// Forward DCT-II along y of the eight fields of a spectral row kx (one line
// per lane group), the spectra and the Gram sums; each CTA takes the rows
// blockIdx.x, blockIdx.x + gridDim.x, ... and leaves one partial row.  The
// post-process turns each line's buffer into doubles in place (every item
// writes the two slots it read), and the Gram sums read the eight fields'
// slots from there.
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
kx_col_gram(const double* __restrict__ in, double* __restrict__ spec, double* __restrict__ part,
            const int4* __restrict__ tw2, PairTab tf, const double* __restrict__ isig, const double* __restrict__ itau) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, G = Gm::G;
    static_assert(Gm::LINES == NF, "one line per field");
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    cx* bufs = reinterpret_cast<cx*>(smraw);
    int n2, slot;
    lane_of<M>(n2, slot);
    cx* buf = bufs + (size_t)slot * Gm::BUF;
    const size_t NN = (size_t)N * N;
    double acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.0;
    for (int kx = blockIdx.x; kx < N; kx += gridDim.x) {
        const int ex = forward_line<M, false>(in + CCM_IXW(slot * NN + (size_t)kx * N, N, NF * NN), buf, tw2, n2, slot, sm, false);
        double* srow = spec + CCM_IXW(((size_t)kx * NF + slot) * N, N, NF * NN);
#pragma unroll 1
        for (int k = n2; k < M / 2; k += G) {
            cx s[2];
            post_item<M>(buf, tf, k, s[0], s[1]);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int i = u ? item_slot2<M>(k) : k;
                const double2 d = make_double2(line_double(s[u].x, ex, tf.p), line_double(s[u].y, ex, tf.p));
                reinterpret_cast<double2*>(buf)[i] = d;
                if (slot != 5) reinterpret_cast<double2*>(srow)[i] = d;        // P^ enters the Gram sums only
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int i = threadIdx.x; i < M; i += Gm::THREADS) {
            const double2 ws = ld2(isig + (size_t)kx * N + 2 * i), wt = ld2(itau + (size_t)kx * N + 2 * i);
            double a[NF], b[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const double2 d = reinterpret_cast<const double2*>(bufs + (size_t)f * Gm::BUF)[i];
                a[f] = d.x;
                b[f] = d.y;
            }
            gram_mode(acc, a, ws.x, wt.x);
            gram_mode(acc, b, ws.y, wt.y);
        }
        __syncthreads();
    }
    gram_store<Gm::THREADS>(acc, part + (size_t)blockIdx.x * NRED2, reinterpret_cast<double*>(smraw));
}

// Lines too long for eight buffers per CTA (M >= 2048): the spectra of LINES
// rows of field blockIdx.y, and the Gram sums from them in a second kernel.
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
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
#pragma unroll 1
    for (int k = n2; k < M / 2; k += Gm::G) {
        cx s[2];
        post_item<M>(buf, tf, k, s[0], s[1]);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            reinterpret_cast<double2*>(srow)[u ? item_slot2<M>(k) : k] =
                make_double2(line_double(s[u].x, ex, tf.p), line_double(s[u].y, ex, tf.p));
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
            for (int f = 0; f < NF; ++f) v[f] = __ldg(spec + CCM_IX(((size_t)kx * NF + f) * N + j, (size_t)NF * N * N));
            gram_mode(acc, v, __ldg(isig + (size_t)kx * N + j), __ldg(itau + (size_t)kx * N + j));
        }
    gram_store<kGramThreads>(acc, part + (size_t)blockIdx.x * NRED2, sm);
}

// isig, itau in the order of the spectra
template <int M>
__global__ void kx_weights(const double* __restrict__ ev, SpecCoef sc, double* __restrict__ isig, double* __restrict__ itau) {
    constexpr size_t N = 2 * M;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < N * N; q += (size_t)gridDim.x * blockDim.x) {
        const double s = ev[q / N] + ev[slot_mode<M>((int)(q % N) >> 1, (int)(q & 1))];
        isig[q] = 1.0 / fma(fma(sc.C3, s, sc.C2), s, sc.C1);
        itau[q] = 1.0 / fma(sc.lam, s, sc.Ct);
    }
}

// ------------------------------------------------------------------ recovery and inverse columns
// Transposed write of the LINES natural-order lines of a CTA: out[y][x0 + r].
template <int M>
__device__ __forceinline__ void write_transposed(const cx* bufs, const LineSm<M>& sm, double* __restrict__ out, size_t base,
                                                 int x0, size_t n) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, L = Gm::LINES;
#pragma unroll 1
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
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
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
    cx* buf = bufs + (size_t)slot * Gm::BUF;
    unsigned mx = 0;
    auto put = [&](int i, double x, double y) {
        reinterpret_cast<double2*>(buf)[i] = make_double2(x, y);
        mx = max(mx, max(mag_hi(x), mag_hi(y)));
    };
    if (f == 0) {
        const double aS = -dsc->alpha[0], aH = -dsc->alpha[1], aQ = -dsc->alpha[2], aK = -dsc->alpha[3];
#pragma unroll 4
        for (int j = 0; j < E; ++j) {
            const int i = n2 + G * j;
            const double2 v0 = ld2(s + 2 * i), v1 = ld2(s + N + 2 * i), v2 = ld2(s + 2 * N + 2 * i), v3 = ld2(s + 3 * N + 2 * i),
                          v4 = ld2(s + 4 * N + 2 * i), w = ld2(isig + (size_t)kx * N + 2 * i);
            put(i, fma(aK, v4.x, fma(aQ, v3.x, fma(aH, v2.x, fma(aS, v1.x, v0.x)))) * w.x,
                fma(aK, v4.y, fma(aQ, v3.y, fma(aH, v2.y, fma(aS, v1.y, v0.y)))) * w.y);
        }
    } else {
        const double aL = dsc->alpha[4];
#pragma unroll 8
        for (int j = 0; j < E; ++j) {
            const int i = n2 + G * j;
            const double2 v6 = ld2(s + 6 * N + 2 * i), v7 = ld2(s + 7 * N + 2 * i), w = ld2(itau + (size_t)kx * N + 2 * i);
            put(i, fma(aL, v7.x, v6.x) * w.x, fma(aL, v7.y, v6.y) * w.y);
        }
    }
    inverse_line<M, false>(mx, buf, tw2, ti, n2, slot, sm);
    __syncthreads();
    write_transposed<M>(bufs, sm, out, f * NN, x0, 2 * NN);
}

// ------------------------------------------------------------------ inverse rows
// A row's modes (natural order, global) to slots of doubles in buf; returns
// the largest mag_hi of this lane's.
template <int M> __device__ __forceinline__ unsigned load_modes(cx* buf, const double* row, int n2) {
    unsigned mx = 0;
#pragma unroll 8
    for (int j = 0; j < Geo<M>::E; ++j) {
        const int i = n2 + Geo<M>::G * j;
        const double x = row[i], y = row[slot_mode<M>(i, 1)];
        reinterpret_cast<double2*>(buf)[i] = make_double2(x, y);
        mx = max(mx, max(mag_hi(x), mag_hi(y)));
    }
    return mx;
}

// Inverse DCT along x of LINES rows of field blockIdx.y and
// u^{n+1} = u_bar + du.
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
kx_irow(const double* __restrict__ in, double* __restrict__ phi_new, double* __restrict__ psi_new,
        const int4* __restrict__ tw2, PairTab ti, const double* __restrict__ phn, const double* __restrict__ pho,
        const double* __restrict__ psn, const double* __restrict__ pso, int bdf1) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, G = Gm::G;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    int n2, slot;
    lane_of<M>(n2, slot);
    cx* buf = reinterpret_cast<cx*>(smraw) + (size_t)slot * Gm::BUF;
    const size_t NN = (size_t)N * N;
    const int f = blockIdx.y, y = blockIdx.x * Gm::LINES + slot;
    const unsigned mx = load_modes<M>(buf, in + CCM_IXW(f * NN + (size_t)y * N, N, 2 * NN), n2);
    const int ex = inverse_line<M, false>(mx, buf, tw2, ti, n2, slot, sm);
    const double* un = f ? psn : phn;
    const double* uo = f ? pso : pho;
    double* u = f ? psi_new : phi_new;
#pragma unroll 2
    for (int m = n2; m < M / 2; m += G) {
        const size_t o = CCM_IXW((size_t)y * N + 4 * m, 4, NN);
        const vec4<double> d = unpack_item<M>(buf, m, ex), a = ld4(un + o), b = ld4(uo + o);
        // u_bar + du without the FP32 path's correction term (an FP64 addition less)
        auto add = [&](double p, double q, double x) { return (bdf1 ? p : fma(p - q, 1.0 / 3.0, p)) + x; };
        st4(u + o, vec4<double>{add(a.a, b.a, d.a), add(a.b, b.b, d.b), add(a.c, b.c, d.c), add(a.d, b.d, d.d)});
    }
}

// ------------------------------------------------------------------ solver
// LINES spectral rows (contiguous over y): forward DCT along y, division by
// c0 + c1 s + c2 s^2, inverse DCT, transposed write out[y][kx].
template <int M>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
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
    const size_t n = gridDim.y * fstride;
    const int ex = forward_line<M, false>(in + CCM_IXW(blockIdx.y * fstride + (size_t)kx * N, N, n), buf, tw2, n2, slot, sm, false);
    const double evx = ev[kx];
    unsigned mx = 0;
#pragma unroll 1
    for (int j = 0; j < E / 2; ++j) {
        const int k = n2 + G * j;
        cx z[2];
        post_item<M>(buf, tf, k, z[0], z[1]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = u ? item_slot2<M>(k) : k;
            const double sx = evx + __ldg(ev + slot_mode<M>(i, 0)), sy = evx + __ldg(ev + slot_mode<M>(i, 1));
            const double x = line_double(z[u].x, ex, tf.p) / (c0 + sx * (c1 + c2 * sx));
            const double y = line_double(z[u].y, ex, tf.p) / (c0 + sy * (c1 + c2 * sy));
            reinterpret_cast<double2*>(buf)[i] = make_double2(x, y);
            mx = max(mx, max(mag_hi(x), mag_hi(y)));
        }
    }
    inverse_line<M, true>(mx, buf, tw2, ti, n2, slot, sm);
    __syncthreads();
    write_transposed<M>(bufs, sm, out, blockIdx.y * fstride, x0, n);
}

// Inverse DCT along x of LINES rows (in place allowed).  DST: times (-1)^(i+j).
template <int M, bool DST>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
kx_row_inv(const double* in, double* out, const int4* __restrict__ tw2, PairTab ti, const int* __restrict__ dskip,
           size_t fstride) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, G = Gm::G;
    if (dskip && dskip[blockIdx.y]) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ LineSm<M> sm;
    int n2, slot;
    lane_of<M>(n2, slot);
    cx* buf = reinterpret_cast<cx*>(smraw) + (size_t)slot * Gm::BUF;
    const int y = blockIdx.x * Gm::LINES + slot;
    const size_t o = blockIdx.y * fstride + (size_t)y * N, n = gridDim.y * fstride;
    const unsigned mx = load_modes<M>(buf, in + CCM_IXW(o, N, n), n2);
    const int ex = inverse_line<M, false>(mx, buf, tw2, ti, n2, slot, sm);
#pragma unroll 2
    for (int m = n2; m < M / 2; m += G) {
        vec4<double> v = unpack_item<M>(buf, m, ex);
        if (DST) {                                     // x = 4m is even: signs (+, -, +, -) times (-1)^y
            const double s = (y & 1) ? -1.0 : 1.0;
            v.a *= s; v.b *= -s; v.c *= s; v.d *= -s;
        }
        if (CCM_OKW(o + 4 * m, 4, n)) st4(out + o + 4 * m, v);
    }
}

}  // namespace xf
}  // namespace ccm

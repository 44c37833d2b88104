// wide_step.cuh -- FP32 step kernels on the lines of wide_fft.cuh: recovery +
// inverse columns and inverse rows (N = 128 .. 8192), and the forward passes of
// N = 8192.
//
// The inverse kernels wait on memory, and on warp-level lines (32 or 64 values
// per lane, 72 - 128 registers) they held 16 - 24 warps per SM; with sixteen
// values per lane 32 warps fit: N = 2048 recovery 61 -> 45 us, inverse rows
// 40 -> 30; N = 8192 1112 -> 743, 839 -> 395.  The recovery kernel takes one field per CTA (the phi CTAs,
// five spectra, come first, the lighter psi CTAs fill the tail).
#pragma once
#include "warp_kernels.cuh"
#include "wide_fft.cuh"

namespace ccm {
namespace lf {

// Exact (double-float) sum over the G lanes of one line: inside the warp for
// G <= 32; for G = 32 W each of the W warps sums its part, the parts go
// through `sm` (W float2 per line slot) and every warp adds them in the same
// order.
template <int G>
__device__ __forceinline__ double line_sum_exact(float hi, float lo, int slot, float2* sm) {
    if constexpr (G <= 32) {
        return group_sum_exact<G>(hi, lo);
    } else {
        constexpr int W = G / 32;
        const float2 h = group_sum_df<32>(hi, lo);
        const int part = (threadIdx.x >> 5) % W;
        if ((threadIdx.x & 31) == 0) sm[W * slot + part] = h;
        wf::line_sync<G>(slot);
        float2 a = sm[W * slot];
#pragma unroll
        for (int w = 1; w < W; ++w) {
            const float2 b = sm[W * slot + w];
            df_add2(a.x, a.y, b.x, b.y);
        }
        wf::line_sync<G>(slot);        // the slots may be written again by a later call
        return (double)a.x + (double)a.y;
    }
}

// ------------------------------------------------------------------ forward rows
// 4096-point lines: clusters of two CTAs of four rows each (write_modes_pair).
// Shorter lines take the warp-level kernels of warp_kernels.cuh, which move a
// line through shared memory once less: measured at N = 8192 row 1894 us with
// 64 x 64 lines on two warps, 1995 on wide lines with 16-byte segments, 1610
// with the cluster; column pass 2022 -> 1300; but N = 4096 row 294 (warp) / 374
// (cluster), column 338 / 349, N = 2048 row 63 / 81, column 64 / 82.
template <int M> struct FwdGeo {
    static constexpr int LINES = 4, CLUSTER = 2;
    static constexpr int THREADS = LINES * Geo<M>::G;
    static constexpr size_t SMEM = (size_t)LINES * Geo<M>::BUF * sizeof(cf);
    static constexpr int MINB = 1024 / THREADS;
};

// Forward DCT-II along x of four rows of field blockIdx.y per CTA, eight per
// cluster, transposed write.
template <int M>
__global__ void __launch_bounds__(FwdGeo<M>::THREADS, FwdGeo<M>::MINB)
kl_row(const float* __restrict__ in, float* __restrict__ out, const float2* __restrict__ tw, PairTab tf) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N;
    extern __shared__ __align__(16) unsigned char smraw[];
    cf* bufs = reinterpret_cast<cf*>(smraw);
    int n2, slot;
    lane_of<M>(n2, slot);
    const size_t NN = (size_t)N * N, f0 = blockIdx.y * NN;
    const int y = blockIdx.x * FwdGeo<M>::LINES + slot, y0 = (blockIdx.x & ~1) * FwdGeo<M>::LINES;
    forward_line<M, false>(in + CCM_IXW(f0 + (size_t)y * N, N, NF * NN), bufs + (size_t)slot * Gm::BUF, tw, n2, slot, false);
    write_modes_pair<M>(bufs, out + f0 + y0, tf, f0 + y0, NF * NN);
}

// ------------------------------------------------------------------ forward columns and Gram sums
// Sixteen of the seventeen Gram sums of a mode, f0' f0' left out (not used by
// the solve; its column stays 0): for b = 1 .. 4 the products with a = 0 .. b,
// then PG, PL.  psi only / phi only for the split column pass.
template <bool PHI, bool PSI>
__device__ __forceinline__ void gram_mode(float (&acc)[16], const float (&v)[NF], float isig, float itau) {
    if constexpr (PHI) {
        int p = 0;
#pragma unroll
        for (int b = 1; b < 5; ++b) {
            const float w = v[b] * isig;
#pragma unroll
            for (int a = 0; a <= b; ++a) { acc[p] = fmaf(v[a], w, acc[p]); ++p; }
        }
    }
    if constexpr (PSI) {
        const float w = v[5] * itau;
        acc[14] = fmaf(v[6], w, acc[14]);
        acc[15] = fmaf(v[7], w, acc[15]);
    }
}
// Accumulator p -> column of a partial row (a <= b over f0' S H Q K row by row, PG, PL)
__device__ __forceinline__ int gram_col(int p) {
    if (p >= 14) return p + 1;
    const int b = p < 2 ? 1 : p < 5 ? 2 : p < 9 ? 3 : 4, a = p - (b == 1 ? 0 : b == 2 ? 2 : b == 3 ? 5 : 9);
    return a * 5 - a * (a - 1) / 2 + (b - a);
}
// Block sums into a partial row of float pairs: FP32 over a warp by recursive
// halving (16 values in 16 exchanges), double-float over the warps.
template <int THREADS>
__device__ __forceinline__ void gram_store(float (&acc)[16], float2* __restrict__ row, float* __restrict__ sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int idx = 0;
#pragma unroll
    for (int h = 8; h >= 1; h >>= 1) {
        const bool up = lane & h;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float give = up ? acc[i] : acc[i + h], keep = up ? acc[i + h] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, h);
        }
        if (up) idx += h;
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 16);
    __syncthreads();                                   // the line buffers are free
    if (lane < 16) sm[warp * 16 + idx] = acc[0];
    __syncthreads();
    if (threadIdx.x < 16) {
        float hi = 0.f, lo = 0.f;
#pragma unroll 8
        for (int w = 0; w < THREADS / 32; ++w) df_add(hi, lo, sm[w * 16 + threadIdx.x]);
        row[gram_col(threadIdx.x)] = make_float2(hi, lo);
    }
    if (threadIdx.x == 16) row[0] = make_float2(0.f, 0.f);
}

// Columns: the eight lines of a spectral row do not fit a CTA, so they go four
// at a time through five buffers: first P, g0', L_P and K, whose psi sums are
// formed before f0', S, H, Q take places beside K.
template <int M> struct ColGeo {
    static constexpr int LINES = 4, COLS = 5;
    static constexpr int THREADS = LINES * Geo<M>::G;
    static constexpr size_t SMEM = (size_t)COLS * Geo<M>::BUF * sizeof(cf);
};

// Post-process of a line in place (slots of modes) and its spectrum in pair
// order (SpecRow: float4 of modes k, N-k, M-k, M+k for k = 0 .. M/2; pair 0 holds
// X[0], 0, X[M], X[M], pair M/2 its two modes twice); dst null: not stored.
template <int M> __device__ __forceinline__ void post_line(cf* buf, const PairTab& tf, float* dst, int n2) {
#pragma unroll 2
    for (int k = n2; k < M / 2; k += Geo<M>::G) {
        cf s1, s2;
        post_item<M>(buf, tf, k, s1, s2);
        buf[k] = s1;
        buf[item_slot2<M>(k)] = s2;
        if (dst) {
            float4* d = reinterpret_cast<float4*>(dst);
            d[k] = k == 0 ? make_float4(s1.x, 0.f, s1.y, s1.y) : make_float4(s1.x, s1.y, s2.x, s2.y);
            if (k == 0) d[M / 2] = make_float4(s2.x, s2.y, s2.x, s2.y);
        }
    }
}
// Gram sums over the slots of a spectral row; buffer of field f: bufs + pos[f] BUF
template <int M, bool PHI, bool PSI>
__device__ __forceinline__ void gram_slots(float (&acc)[16], const cf* bufs, const int (&pos)[NF], float evx,
                                           const float* __restrict__ evf, const SpecCoefF& sc) {
#pragma unroll 1
    for (int i = threadIdx.x; i < M; i += ColGeo<M>::THREADS) {
        float a[NF], b[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            if (f < 5 ? !PHI : !PSI) { a[f] = b[f] = 0.f; continue; }
            const cf z = bufs[(size_t)pos[f] * Geo<M>::BUF + i];
            a[f] = z.x;
            b[f] = z.y;
        }
        const float s0 = evx + __ldg(evf + slot_mode<M>(i, 0)), s1 = evx + __ldg(evf + slot_mode<M>(i, 1));
        // correctly rounded reciprocals (the same values as 1.0f / x)
        gram_mode<PHI, PSI>(acc, a, PHI ? __frcp_rn(sc.C1 + s0 * (sc.C2 + sc.C3 * s0)) : 0.f, PSI ? __frcp_rn(sc.Ct + sc.lam * s0) : 0.f);
        gram_mode<PHI, PSI>(acc, b, PHI ? __frcp_rn(sc.C1 + s1 * (sc.C2 + sc.C3 * s1)) : 0.f, PSI ? __frcp_rn(sc.Ct + sc.lam * s1) : 0.f);
    }
}

// Forward DCT-II along y of the eight fields of spectral row kx, the spectra
// and the Gram sums.
template <int M>
__global__ void __launch_bounds__(ColGeo<M>::THREADS, 1)
kl_col(const float* __restrict__ in, float* __restrict__ spec, double* __restrict__ part, const float2* __restrict__ tw,
       PairTab tf, const float* __restrict__ evf, SpecCoefF sc) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N;
    extern __shared__ __align__(16) unsigned char smraw[];
    cf* bufs = reinterpret_cast<cf*>(smraw);
    const int kx = blockIdx.x;
    int n2, slot;
    lane_of<M>(n2, slot);
    const size_t NN = (size_t)N * N;
    const float evx = __ldg(evf + kx);
    float acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.f;
    float* srow = spec + CCM_IXW((size_t)kx * SpecRow<M>::KS, SpecRow<M>::KS, (size_t)N * SpecRow<M>::KS);
    auto line = [&](int f, int p) {
        cf* buf = bufs + (size_t)p * Gm::BUF;
        forward_line<M, false>(in + CCM_IXW(f * NN + (size_t)kx * N, N, NF * NN), buf, tw, n2, slot, false);
        post_line<M>(buf, tf, f == 5 ? nullptr : srow + (size_t)(f < 5 ? f : f - 1) * SpecRow<M>::FO, n2);   // P^: Gram sums only
    };
    constexpr int pos[NF] = {0, 1, 2, 4, 3, 0, 1, 2};     // buffer of each field
    line(slot < 3 ? 5 + slot : 4, slot);
    __syncthreads();
    gram_slots<M, false, true>(acc, bufs, pos, evx, evf, sc);
    __syncthreads();
    line(slot, slot < 3 ? slot : 4);
    __syncthreads();
    gram_slots<M, true, false>(acc, bufs, pos, evx, evf, sc);
    __syncthreads();
    gram_store<ColGeo<M>::THREADS>(acc, reinterpret_cast<float2*>(part) + (size_t)kx * NRED2, reinterpret_cast<float*>(smraw));
}

// ------------------------------------------------------------------ recovery and inverse columns
// LINES spectral rows of one field: recovery combination and divide, inverse
// DCT along y, transposed write out[f][y][kx].  Block b: field b / (N / LINES).
template <int M, bool GRP = false>
__global__ void __launch_bounds__(Geo<M>::THREADS, Geo<M>::MINB)
kl_comb(const float* __restrict__ spec, float* __restrict__ out, const float2* __restrict__ tw, PairTab ti,
        const float* __restrict__ evf, const float4* __restrict__ evp, SpecCoefF sc, DevScalars* __restrict__ dsc,
        int anchor_mass, const __grid_constant__ GroupArgs<GRP> ga, int bps) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, E = Gm::E, G = Gm::G, NB = N / Gm::LINES;
    extern __shared__ __align__(16) unsigned char smraw[];
    cf* bufs = reinterpret_cast<cf*>(smraw);
    const size_t NN = (size_t)N * N;
    int bx = blockIdx.x;
    if constexpr (GRP) {          // grouped launch
        const int sim = blockIdx.x / bps;
        bx = blockIdx.x - sim * bps;
        const BatchArgs& A = ga.a[sim];
        spec = A.bufA; out = A.bufB; tw = A.tww; ti = A.tiw; evf = A.evf; evp = A.evp; sc = A.sf; dsc = A.sc;
    }
    int n2, slot;
    lane_of<M>(n2, slot);
    const int f = bx / NB, x0 = (bx % NB) * Gm::LINES, kx = x0 + slot;
    cf* buf = bufs + (size_t)slot * Gm::BUF;
    const float evx = __ldg(evf + kx);
    const size_t base = CCM_IXW((size_t)kx * SpecRow<M>::KS, SpecRow<M>::KS, (size_t)N * SpecRow<M>::KS);
    constexpr size_t FS = SpecRow<M>::FO;
    auto put = [&](int k, const Quad<float>& X) {
        cf zk, zMk;
        wf::pre_pair_lean(X, ld_pair(ti, k), zk, zMk);
        buf[k] = zk;
        if (k > 0) buf[M - k] = zMk;
    };
    if (f == 0) {
        const float aS = (float)dsc->alpha[0], aH = (float)dsc->alpha[1], aQ = (float)dsc->alpha[2], aK = (float)dsc->alpha[3];
#pragma unroll 2
        for (int k = n2; k <= M / 2; k += G) {
            const float4 e4 = __ldg(evp + k);
            const float* src = spec + base + 4 * k;
            const float4 f0 = __ldg(reinterpret_cast<const float4*>(src));
            const float4 f1 = __ldg(reinterpret_cast<const float4*>(src + FS));
            const float4 f2 = __ldg(reinterpret_cast<const float4*>(src + 2 * FS));
            const float4 f3 = __ldg(reinterpret_cast<const float4*>(src + 3 * FS));
            const float4 f4 = __ldg(reinterpret_cast<const float4*>(src + 4 * FS));
            auto comb = [&](float a0, float a1, float a2, float a3, float a4, float ev) {
                const float s = evx + ev;
                return (a0 - aS * a1 - aH * a2 - aQ * a3 - aK * a4) * __frcp_rn(sc.C1 + s * (sc.C2 + sc.C3 * s));
            };
            put(k, Quad<float>{comb(f0.x, f1.x, f2.x, f3.x, f4.x, e4.x), comb(f0.y, f1.y, f2.y, f3.y, f4.y, e4.y),
                               comb(f0.z, f1.z, f2.z, f3.z, f4.z, e4.z), comb(f0.w, f1.w, f2.w, f3.w, f4.w, e4.w)});
        }
    } else {
        const float aL = (float)dsc->alpha[4];
#pragma unroll 4
        for (int k = n2; k <= M / 2; k += G) {
            const float4 e4 = __ldg(evp + k);
            const float* src = spec + base + 4 * k;
            const float4 f6 = __ldg(reinterpret_cast<const float4*>(src + 5 * FS));
            const float4 f7 = __ldg(reinterpret_cast<const float4*>(src + 6 * FS));
            auto comb = [&](float a6, float a7, float ev) {
                return (a6 + aL * a7) * __frcp_rn(sc.Ct + sc.lam * (evx + ev));
            };
            Quad<float> X{comb(f6.x, f7.x, e4.x), comb(f6.y, f7.y, e4.y), comb(f6.z, f7.z, e4.z), comb(f6.w, f7.w, e4.w)};
            // d_psi has zero mean (mass conservation); the zero mode is set exactly and the stored mean kept with the anchor
            if (anchor_mass && kx == 0 && k == 0) X.xk = 0.f;
            put(k, X);
        }
    }
    sync_line<M>(slot);
    inverse_line<M>(buf, tw, n2, slot);
    if (anchor_mass && f == 1 && x0 == 0) {
        // the zero-mean psi increment's kx = 0 column should sum to 0 over y; record what the
        // FP32 transform left (removed in the inverse row kernel).  Every line of the block takes part in the sum.
        __shared__ float2 lsum[Gm::LINES * (G > 32 ? G / 32 : 1)];
        float dhi = 0.f, dlo = 0.f;
#pragma unroll 1
        for (int m = n2; m < M / 2; m += G) {
            const cf a = buf[m], b = buf[M - 1 - m];
            df_add(dhi, dlo, a.x); df_add(dhi, dlo, b.y); df_add(dhi, dlo, a.y); df_add(dhi, dlo, b.x);
        }
        const double dsum = line_sum_exact<G>(dhi, dlo, slot, lsum);
        if (slot == 0 && n2 == 0) dsc->dc_col = dsum;
    }
    if constexpr (Gm::LINES == 4) {                       // comb_cluster: two CTAs
        write_samples_pair<M>(bufs, out + f * NN + (size_t)(x0 & ~7), f * NN + (size_t)(x0 & ~7), 2 * NN);
    } else {
        __syncthreads();
        write_samples<M, Gm::LINES>(bufs, out + f * NN + x0, f * NN + x0, 2 * NN);
    }
}
template <int M> __host__ __device__ constexpr int comb_cluster() { return Geo<M>::LINES == 4 ? 2 : 1; }

// Rows per CTA of the inverse row kernel: four (the lines are independent;
// smaller CTAs leave less of a last wave idle), two at M = 4096.
template <int M> struct RowGeo {
    static constexpr int G = Geo<M>::G;
    static constexpr int LINES = M == 4096 ? 2 : G < 8 ? 8 : 4;
    static constexpr int THREADS = LINES * G;
    static constexpr size_t SMEM = (size_t)LINES * Geo<M>::BUF * sizeof(cf);
    static constexpr int MINB = 1024 / THREADS > 16 ? 16 : 1024 / THREADS;
    static_assert(THREADS % 32 == 0, "whole warps");
};

// Inverse DCT along x of LINES rows of one field and u^{n+1} = u_bar + du with
// the compensated (and, for psi, error-feedback and mass-anchored) final
// rounding (bar_add, bar_add_fb).  Block b: field b / (N / LINES).
template <int M, bool GRP = false>
__global__ void __launch_bounds__(RowGeo<M>::THREADS, RowGeo<M>::MINB)
kl_irow(const float* __restrict__ in, float* __restrict__ phi_new, float* __restrict__ psi_new,
        const float2* __restrict__ tw, PairTab ti, const float* __restrict__ phn, const float* __restrict__ pho,
        const float* __restrict__ psn, const float* __restrict__ pso, int bdf1, const DevScalars* __restrict__ dsc,
        int anchor_mass, const __grid_constant__ GroupArgs<GRP> ga, int bps) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, E = Gm::E, G = Gm::G, L = RowGeo<M>::LINES, NB = N / L;
    int bx = blockIdx.x;
    if constexpr (GRP) {          // grouped launch
        const int sim = blockIdx.x / bps;
        bx = blockIdx.x - sim * bps;
        const BatchArgs& A = ga.a[sim];
        in = A.bufB; phi_new = A.phi_new; psi_new = A.psi_new; tw = A.tww; ti = A.tiw;
        phn = A.phn; pho = A.pho; psn = A.psn; pso = A.pso; dsc = A.sc;
    }
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ float2 lsum[L * (G > 32 ? G / 32 : 1)];
    int n2, slot;
    lane_of<M>(n2, slot);
    cf* buf = reinterpret_cast<cf*>(smraw) + (size_t)slot * Gm::BUF;
    const size_t NN = (size_t)N * N;
    const int fld = bx / NB, y = (bx % NB) * L + slot;
    const float* row = in + CCM_IXW(fld * NN + (size_t)y * N, N, 2 * NN);
    const float x0 = __ldg(row);                          // the row's DC coefficient
#pragma unroll 4
    for (int k = n2; k <= M / 2; k += G) {
        const Quad<float> X{__ldg(row + k), k > 0 ? __ldg(row + N - k) : 0.f, __ldg(row + M - k), __ldg(row + M + k)};
        cf zk, zMk;
        wf::pre_pair_lean(X, ld_pair(ti, k), zk, zMk);
        buf[k] = zk;
        if (k > 0) buf[M - k] = zMk;
    }
    sync_line<M>(slot);
    inverse_line<M>(buf, tw, n2, slot);
    const size_t roff = (size_t)y * N;
    const float4* un = reinterpret_cast<const float4*>((fld == 0 ? phn : psn) + roff);
    const float4* uo = reinterpret_cast<const float4*>((fld == 0 ? pho : pso) + roff);
    float* dst = (fld == 0 ? phi_new : psi_new) + roff;
    const bool b1 = bdf1 != 0;
    if (fld == 0 || !anchor_mass) {                       // uniform over the CTA
#pragma unroll 4
        for (int j = 0; j < E / 2; ++j) {
            const int m = n2 + G * j;
            if (!CCM_OKW(roff + 4 * m, 4, NN)) continue;
            const cf a = buf[m], b = buf[M - 1 - m];
            const float4 p = __ldg(un + m), q = __ldg(uo + m);
            *reinterpret_cast<float4*>(dst + 4 * m) =
                make_float4(bar_add(p.x, q.x, a.x, 0.f, b1), bar_add(p.y, q.y, b.y, 0.f, b1),
                            bar_add(p.z, q.z, a.y, 0.f, b1), bar_add(p.w, q.w, b.x, 0.f, b1));
        }
        return;
    }
    // psi: the row's increments should sum to sqrt(N) x0; the residual of the FP32 transform and the column residual
    // dc_col are removed, with the mean anchor, in the final rounding (error feedback along each lane's values, the
    // lanes' remaining errors, summed exactly over the row, folded into the row's first value with one dithered rounding,
    // so that the stored row sums to its exact value within about one ulp)
    const uint32_t step = (uint32_t)dsc->steps;           // dither key (graph replays read it here)
    float rhi = 0.f, rlo = 0.f;
#pragma unroll 1
    for (int j = 0; j < E / 2; ++j) {
        const int m = n2 + G * j;
        const cf a = buf[m], b = buf[M - 1 - m];
        df_add(rhi, rlo, a.x); df_add(rhi, rlo, b.y); df_add(rhi, rlo, a.y); df_add(rhi, rlo, b.x);
    }
    const double rsum = line_sum_exact<G>(rhi, rlo, slot, lsum);
    const double sN = sqrt((double)N);
    const float an = (float)(dsc->anchor - sN * dsc->dc_col / ((double)N * N) + (sN * (double)x0 - rsum) / (double)N);
    float carry = 0.f, first = 0.f;
#pragma unroll 4
    for (int j = 0; j < E / 2; ++j) {
        const int m = n2 + G * j;
        if (!CCM_OKW(roff + 4 * m, 4, NN)) continue;
        const cf a = buf[m], b = buf[M - 1 - m];
        const float4 p = __ldg(un + m), q = __ldg(uo + m);
        float4 o;
        o.x = bar_add_fb(p.x, q.x, a.x, an, b1, carry);
        o.y = bar_add_fb(p.y, q.y, b.y, an, b1, carry);
        o.z = bar_add_fb(p.z, q.z, a.y, an, b1, carry);
        o.w = bar_add_fb(p.w, q.w, b.x, an, b1, carry);
        if (j == 0) first = o.x;
        *reinterpret_cast<float4*>(dst + 4 * m) = o;
    }
    const double rest = line_sum_exact<G>(carry, 0.f, slot, lsum);
    if (n2 == 0) dst[0] = dither_round(first, (float)rest, dither_key(step, (uint32_t)roff) | 1u);
}

}  // namespace lf
}  // namespace ccm

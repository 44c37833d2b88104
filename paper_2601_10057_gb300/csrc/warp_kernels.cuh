// warp_kernels.cuh -- FP32 forward passes built on the warp-level line FFT
// (N = 2M in 128 .. 4096).  Same data flow as the block-FFT kernels of
// step_kernels.cuh:
//   kw_rowdct_T    forward DCT-II along x, transposed write (RT rows per CTA)
//   kw_coldct_gram forward DCT-II along y of the 8 fields of KC spectral rows,
//                  Gram partial sums and the spectra (post-processed from all
//                  8 line buffers at once, so no staging copy)
// The recovery and inverse row kernels, and all passes of 4096-point lines, are
// in wide_step.cuh.
// Every warp owns one line buffer per lane group (32 / G lines per warp).
#pragma once
#include "step_kernels.cuh"
#include "warp_fft.cuh"

namespace ccm {

constexpr int kWarps = 8;

// Pair-ordered spectra of the warp path: for each spectral row kx and each
// of the 7 stored fields (f0', S, H, Q, K, g0', L_P), the float4 of modes
// (k, N-k, M-k, M+k) for each pair k = 0 .. M/2, i.e. a row of
// RS = 4 (M/2 + 1) = N + 4 floats (16-byte aligned).  The layout is kx-major:
// the 7 field rows of one kx are contiguous (stride KS = 7 RS), so the
// recovery kernel reads each CTA's rows as one contiguous block and the
// column kernel writes each kx as one.
template <int M> struct SpecRow {
    static constexpr int RS = 4 * (M / 2 + 1);
    static constexpr size_t FO = (size_t)RS;          // next field, same kx
    static constexpr size_t KS = (size_t)7 * RS;      // next kx
};

template <int M> struct WGeo {
    static constexpr int E = wf::Shape<M>::E, G = wf::Shape<M>::G;
    static constexpr int LPW = 32 / G;                  // lines per warp
    static constexpr int SLOTS = kWarps * LPW;          // line buffers per CTA
    // complex per buffer: unpadded, XOR-swizzled transpose (M + 2), so that
    // three 8-line CTAs of the forward kernels fit the 196 KB shared-memory
    // configuration
    static constexpr int BUF = wf::buf_len<M, true>();
    static constexpr size_t buf_bytes() { return (size_t)SLOTS * BUF * sizeof(cplx<float>); }
};

// ------------------------------------------------------------------ kw_rowdct_T
// SLOTS rows of field blockIdx.y per CTA (one line per lane group).  Each
// line's natural-order half-length spectrum stays in its buffer; the DCT
// post-process reads it from there pair by pair while writing the transposed
// output, so the buffers double as the staging area of that write.
template <int M, bool GRP = false>
__global__ void __launch_bounds__(kWarps * 32, M <= 1024 ? 3 : 1)
kw_rowdct_T(const float* __restrict__ in, float* __restrict__ out,
            const cplx<float>* __restrict__ tw2, wf::PairTwTab twF, int ahead,
            const __grid_constant__ GroupArgs<GRP> ga, int bps) {
    using Gm = WGeo<M>;
    constexpr int N = 2 * M, E = Gm::E, RT = Gm::SLOTS;
    extern __shared__ __align__(16) unsigned char smraw[];
    cplx<float>* bufs = reinterpret_cast<cplx<float>*>(smraw);
    const size_t NN = (size_t)N * N;
    int bx = blockIdx.x;
    if constexpr (GRP) {          // grouped launch (no prefetch ahead)
        const int sim = blockIdx.x / bps;
        bx = blockIdx.x - sim * bps;
        const BatchArgs& A = ga.a[sim];
        in = A.bufA; out = A.bufB; tw2 = A.tw2; twF = A.twF; ahead = 0;
    }
    const int f = blockIdx.y, y0 = bx * RT;
    {   // rows of the CTA one residency ahead
        const int t = blockIdx.y * gridDim.x + blockIdx.x + ahead;
        if (ahead > 0 && t < (int)(gridDim.x * gridDim.y) && threadIdx.x < RT)
            prefetch_l2(in + (t / gridDim.x) * NN + (size_t)((t % gridDim.x) * RT + threadIdx.x) * N, N * sizeof(float));
    }
    int n2, slot;
    wf::lane_geo<M>(n2, slot);
    cplx<float>* buf = bufs + (size_t)slot * Gm::BUF;
    {
        cplx<float> v[E];
        wf::pack_fwd_global<M>(in + CCM_IXW(f * NN + (size_t)(y0 + slot) * N, N, NF * NN), v, n2);
        wf::fourstep<float, M, true>(v, buf, tw2, n2);
    }
    __syncthreads();
    // DCT post-process fused into the transposed write.  Item (r4, k) takes
    // the pair k (slots k and M-k of the natural-order spectra) of the rows
    // 4 r4 .. 4 r4 + 3 and writes its four modes k, N-k, M-k, M+k, each as one
    // float4 of the four rows; the item k = 0 also takes the pair M/2, so
    // that every item loads eight slots and stores four float4 (pair 0 gives
    // the modes 0 and M, pair M/2 the modes M/2 and 3M/2).  Consecutive
    // threads take the two halves of one 32-byte row segment when R4 = 2.
    const float2* stage = reinterpret_cast<const float2*>(bufs);
    constexpr int BC = Gm::BUF;                      // float2 per line buffer
    float* dst = out + f * NN + y0;
    constexpr int R4 = RT / 4;
    static_assert(RT % 4 == 0, "rows of a CTA in groups of four");
    auto put = [&](int mode, int r4, float a, float b, float c, float d) {
        if (CCM_OKW(f * NN + y0 + (size_t)mode * N + 4 * r4, 4, NF * NN))
            *reinterpret_cast<float4*>(dst + (size_t)mode * N + 4 * r4) = make_float4(a, b, c, d);
    };
    for (int q = threadIdx.x; q < R4 * (M / 2); q += blockDim.x) {
        const int r4 = q % R4, k = q / R4;
        const float2* sp = stage + (size_t)(4 * r4) * BC;
        const int ka = k == 0 ? M / 2 : M - k;       // second slot: M - k, or the pair M/2
        cplx<float> A[4], B[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float2 a = sp[(size_t)r * BC + k], b = sp[(size_t)r * BC + ka];
            A[r] = mk(a.x, a.y);
            B[r] = mk(b.x, b.y);
        }
        if (k == 0) {
            const wf::PairTw t0 = wf::load_pair_tw<false>(twF, 0), th = wf::load_pair_tw<false>(twF, M / 2);
            Quad<float> X[4], Y[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                X[r] = wf::post_pair_lean(A[r], A[r], t0);
                Y[r] = wf::post_pair_lean(B[r], B[r], th);
            }
            put(0, r4, X[0].xk, X[1].xk, X[2].xk, X[3].xk);
            put(M, r4, X[0].xMk, X[1].xMk, X[2].xMk, X[3].xMk);
            put(M / 2, r4, Y[0].xk, Y[1].xk, Y[2].xk, Y[3].xk);
            put(N - M / 2, r4, Y[0].xNk, Y[1].xNk, Y[2].xNk, Y[3].xNk);
        } else {
            const wf::PairTw t = wf::load_pair_tw<false>(twF, k);
            Quad<float> X[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) X[r] = wf::post_pair_lean(A[r], B[r], t);
            put(k, r4, X[0].xk, X[1].xk, X[2].xk, X[3].xk);
            put(N - k, r4, X[0].xNk, X[1].xNk, X[2].xNk, X[3].xNk);
            put(M - k, r4, X[0].xMk, X[1].xMk, X[2].xMk, X[3].xMk);
            put(M + k, r4, X[0].xMpk, X[1].xMpk, X[2].xMpk, X[3].xMpk);
        }
    }
}

// ------------------------------------------------------------------ kw_coldct_gram
template <int M, bool GRP = false>
__global__ void __launch_bounds__(kWarps * 32, M <= 1024 ? 3 : 1)
kw_coldct_gram(const float* __restrict__ in, float* __restrict__ spec, double* __restrict__ part,
               const cplx<float>* __restrict__ tw2, wf::PairTwTab twF,
               const float* __restrict__ evf, const float4* __restrict__ evp, SpecCoefF sc,
               const __grid_constant__ GroupArgs<GRP> ga, int bps) {
    using Gm = WGeo<M>;
    constexpr int N = 2 * M, G = Gm::G, E = Gm::E, KC = Gm::SLOTS / NF;
    extern __shared__ __align__(16) unsigned char smraw[];
    cplx<float>* bufs = reinterpret_cast<cplx<float>*>(smraw);
    const size_t NN = (size_t)N * N;
    int bx = blockIdx.x;
    if constexpr (GRP) {          // grouped launch
        const int sim = blockIdx.x / bps;
        bx = blockIdx.x - sim * bps;
        const BatchArgs& A = ga.a[sim];
        in = A.bufB; spec = A.bufA; part = A.part2; tw2 = A.tw2; twF = A.twF; evf = A.evf; evp = A.evp; sc = A.sf;
    }
    const int kx0 = bx * KC;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int n2, slot;                                        // line = (kc, field)
    wf::lane_geo<M>(n2, slot);
    const int kc = slot / NF, f = slot % NF;
    {
        cplx<float> v[E];
        wf::pack_fwd_global<M>(in + CCM_IXW(f * NN + (size_t)(kx0 + kc) * N, N, NF * NN), v, n2);
        wf::fourstep<float, M, true>(v, bufs + (size_t)slot * Gm::BUF, tw2, n2);
    }
    __syncthreads();
    float acc[NRED2];
#pragma unroll
    for (int i = 0; i < NRED2; ++i) acc[i] = 0.f;
    static_assert(KC * NF <= 32, "one lane per (column, field) of the pair M/2");
    if (warp == kWarps - 1) {
        // pair M/2 (modes M/2 and 3M/2 only) of every column by the last warp,
        // one lane per (column, field), so that the loop below gives every
        // thread the same number of pairs; lane 8c adds the column's Gram terms
        const int c = lane >> 3, g = lane & 7;
        float xm = 0.f, x3 = 0.f;
        if (c < KC) {
            const cplx<float>* b = bufs + (size_t)(c * NF + g) * Gm::BUF;
            const Quad<float> X = wf::post_pair_lean(b[M / 2], b[M / 2], wf::load_pair_tw<false>(twF, M / 2));
            xm = X.xk;
            x3 = X.xNk;
            if (g != 5)
                *reinterpret_cast<float4*>(spec + (size_t)(kx0 + c) * SpecRow<M>::KS + (size_t)(g < 5 ? g : g - 1) * SpecRow<M>::FO +
                                           4 * (M / 2)) = make_float4(xm, x3, xm, x3);
        }
#pragma unroll 1
        for (int mode = 0; mode < 2; ++mode) {       // M/2, then 3M/2
            float v[NF];
#pragma unroll
            for (int u = 0; u < NF; ++u) v[u] = __shfl_sync(0xffffffffu, mode ? x3 : xm, (lane & ~7) + u);
            if (g == 0 && c < KC) {
                const float4 eh = evp[M / 2];
                const float sm = evf[kx0 + c] + (mode ? eh.y : eh.x);
                gram_accumulate(acc, v, __frcp_rn(sc.C1 + sm * (sc.C2 + sc.C3 * sm)), __frcp_rn(sc.Ct + sc.lam * sm));
            }
        }
    }
    for (int q = threadIdx.x; q < KC * (M / 2); q += blockDim.x) {
        const int c = q / (M / 2), k = q % (M / 2);
        const int kx = kx0 + c;
        Quad<float> X[NF];
        const wf::PairTw tw = wf::load_pair_tw<false>(twF, k);
#pragma unroll
        for (int g = 0; g < NF; ++g) {
            const cplx<float>* b = bufs + (size_t)(c * NF + g) * Gm::BUF;
            X[g] = wf::post_pair_lean(b[k], b[(M - k) & (M - 1)], tw);
        }
        const float evx = evf[kx];
        const float4 e4 = evp[k];
        const float ev_u[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (!pair_mode_valid(u, k, M)) continue;
            const float s = evx + ev_u[u];
            // correctly rounded reciprocals (the same values as 1.0f / x)
            const float isig = __frcp_rn(sc.C1 + s * (sc.C2 + sc.C3 * s));
            const float itau = __frcp_rn(sc.Ct + sc.lam * s);
            float v[NF];
#pragma unroll
            for (int g = 0; g < NF; ++g)
                v[g] = (u == 0) ? X[g].xk : (u == 1) ? X[g].xNk : (u == 2) ? X[g].xMk : X[g].xMpk;
            gram_accumulate(acc, v, isig, itau);
        }
        // spectra in pair order: slot u of pair k holds mode k, N-k, M-k, M+k
        // (k = 0: no mode N, slot 3 repeats mode M; k = M/2, above: slots 2, 3
        // repeat modes M/2, 3M/2), one float4 per field
        float* dst = spec + (size_t)kx * SpecRow<M>::KS + 4 * k;
#pragma unroll
        for (int g = 0; g < NF; ++g) {
            if (g == 5) continue;
            if (!CCM_OKW((size_t)kx * SpecRow<M>::KS + 4 * k + (size_t)(g < 5 ? g : g - 1) * SpecRow<M>::FO, 4,
                         (size_t)N * SpecRow<M>::KS)) continue;
            float4 o = make_float4(X[g].xk, k == 0 ? 0.f : X[g].xNk, X[g].xMk, X[g].xMpk);
            if (k == 0) o.w = o.z;
            *reinterpret_cast<float4*>(dst + (size_t)(g < 5 ? g : g - 1) * SpecRow<M>::FO) = o;
        }
    }
    __syncthreads();       // the line buffers are free: their start holds the block reduction
    block_sum_store_part<NRED2, float>(acc, reinterpret_cast<float2*>(part) + (size_t)bx * NRED2,
                                       reinterpret_cast<double*>(smraw));
}

}  // namespace ccm

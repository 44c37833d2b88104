// wide_fft.cuh -- FP32 lines of M complex values on M / A lanes (A = 16 values
// each, 8 and 4 on short lines, see Shape), for kernels that want many warps per
// SM: the standalone solver and the classical preconditioner at every length,
// the step's recovery and inverse-row kernels from N = 128 on, and its forward
// kernels at N = 8192.
//
// The line layout is that of fixed_fft.cuh (M = A C D, two exchanges through
// the line's buffer, lines on a part of a warp to eight warps).  warp_fft.cuh keeps a line
// on one warp with up to 64 values per lane: fewer exchanges, and the faster
// one in the step's forward kernels up to N = 4096 (wide_step.cuh has both times).
#pragma once
#include <cooperative_groups.h>
#include "dct_device.cuh"
#include "warp_fft.cuh"
#include "bounds.cuh"

namespace ccm {
namespace lf {

using cf = cplx<float>;

template <int M> struct Shape;
template <> struct Shape<32>   { static constexpr int A = 4,  C = 4,  D = 2;  };
template <> struct Shape<64>   { static constexpr int A = 4,  C = 4,  D = 4;  };
template <> struct Shape<128>  { static constexpr int A = 8,  C = 4,  D = 4;  };
template <> struct Shape<256>  { static constexpr int A = 8,  C = 4,  D = 8;  };
template <> struct Shape<512>  { static constexpr int A = 16, C = 4,  D = 8;  };
template <> struct Shape<1024> { static constexpr int A = 16, C = 8,  D = 8;  };
template <> struct Shape<2048> { static constexpr int A = 16, C = 16, D = 8;  };
template <> struct Shape<4096> { static constexpr int A = 16, C = 16, D = 16; };

// Transpose rows are P = B + 1 values apart (odd: the last pass reads one
// column of sixteen rows per half-warp).  Eight lines per CTA (32-byte
// segments in the transposed writes), four at M = 4096 (1024 threads).
template <int M> struct Geo {
    static constexpr int A = Shape<M>::A, C = Shape<M>::C, D = Shape<M>::D, B = C * D, E = A, G = M / A;
    static_assert(A * B == M && A % C == 0 && A % D == 0, "line shape");
    static constexpr int N = 2 * M;
    static constexpr int LINES = M <= 2048 ? 8 : 4;
    static constexpr int THREADS = LINES * G;
    static constexpr int P = B + 1, BUF = ((A * P + 3) / 4) * 4 + 2;
    static constexpr size_t SMEM = (size_t)LINES * BUF * sizeof(cf);
    static constexpr int MINB = 1024 / THREADS > 8 ? 8 : 1024 / THREADS;      // 64 registers
    static_assert(THREADS % 32 == 0 && THREADS <= 1024, "whole warps");
};

template <int M> __device__ __forceinline__ void lane_of(int& n2, int& slot) {
    n2 = threadIdx.x % Geo<M>::G;
    slot = threadIdx.x / Geo<M>::G;
}
template <int M> __device__ __forceinline__ void sync_line(int slot) { wf::line_sync<Geo<M>::G>(slot); }

__device__ __forceinline__ cf ld_c(const float2* __restrict__ t) {
    const float2 w = __ldg(t);
    return mk(w.x, w.y);
}

// x W_R^i, W_R = exp(-2 pi i / R) (INV: conjugate), with the constants as a high
// and a low part.  Their rounding is the same in every line; a 16-point DFT has
// more of them than the radix-8 passes of the block-level transforms, and with
// rounded ones a line of 2048 or 4096 values was 3 - 6 % further off than theirs.
template <int R, bool INV>
__device__ __forceinline__ cf twid(cf x, int i) {
    static_assert(R <= 16, "");
    const int j = (i * (32 / R)) & 31;                 // below 16
    if (j == 0) return x;
    if (j == 8) return INV ? mk(-x.y, x.x) : mk(x.y, -x.x);
    double c, s;
    wf::w32(j, c, s);
    const float ch = (float)c, cl = (float)(c - (double)ch);
    if (j == 4 || j == 12) {
        auto mul = [&](float t) { return fmaf(t, ch, t * cl); };
        const float p = mul(x.x + x.y), m = mul(x.x - x.y);      // c = +-sqrt(1/2); j = 4: (p, -m), j = 12: (m, p)
        if (j == 4) return INV ? mk(m, p) : mk(p, -m);
        return INV ? mk(p, -m) : mk(m, p);
    }
    const float sh = (float)s, sl = (float)(s - (double)sh);
    auto dot = [](float a, float h, float l, float b, float g, float k) { return fmaf(a, h, fmaf(b, g, fmaf(a, l, b * k))); };
    return INV ? mk(dot(x.x, ch, cl, x.y, -sh, -sl), dot(x.y, ch, cl, x.x, sh, sl))
               : mk(dot(x.x, ch, cl, x.y, sh, sl), dot(x.y, ch, cl, x.x, -sh, -sl));
}
// In-register radix-2 decimation in frequency on v[OFF .. OFF + R): natural
// input, output v[OFF + r] = X[bitrev_R(r)].
template <int R, bool INV, int OFF>
struct DIF {
    static __device__ __forceinline__ void run(cf* v) {
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            const cf a = v[OFF + i], b = v[OFF + i + R / 2];
            v[OFF + i] = a + b;
            v[OFF + i + R / 2] = twid<R, INV>(a - b, i);
        }
        DIF<R / 2, INV, OFF>::run(v);
        DIF<R / 2, INV, OFF + R / 2>::run(v);
    }
};
template <bool INV, int OFF> struct DIF<1, INV, OFF> { static __device__ __forceinline__ void run(cf*) {} };

// x times the table's entry q (INV: its conjugate); LO: with the entry's low part, lo values further on
template <bool INV, bool LO>
__device__ __forceinline__ cf twiddle(cf x, const float2* __restrict__ t, int q, int lo) {
    const cf w = ld_c(t + q);
    if constexpr (!LO) return INV ? cmulc(x, w) : cmul(x, w);
    const cf l = ld_c(t + q + lo);
    const float wy = INV ? -w.y : w.y, ly = INV ? -l.y : l.y;
    return mk(fmaf(x.x, w.x, fmaf(-x.y, wy, fmaf(x.x, l.x, -x.y * ly))), fmaf(x.y, w.x, fmaf(x.x, wy, fmaf(x.y, l.x, x.x * ly))));
}

// The unnormalised DFT of a line (fixed_fft.cuh, fft_line, has the passes).
// LO: the tables' low parts as well (the periodic solver).
template <int M, bool INV, bool LO = false>
__device__ __forceinline__ void fft_line(cf* v, cf* buf, const float2* __restrict__ tw, int n2, int slot) {
    using Gm = Geo<M>;
    constexpr int A = Gm::A, C = Gm::C, D = Gm::D, G = Gm::G, P = Gm::P;
    DIF<A, INV, 0>::run(v);
#pragma unroll
    for (int r = 0; r < A; ++r) {
        const int k1 = wf::bitrev<A>(r);
        cf u = v[r];
        if (k1) u = twiddle<INV, LO>(u, tw, k1 * G + n2, 2 * M);
        buf[k1 * P + n2] = u;
    }
    sync_line<M>(slot);
    if constexpr (D > 1) {
        const float2* __restrict__ t3 = tw + M;
#pragma unroll
        for (int j = 0; j < A / C; ++j) {
            const int q = n2 + G * j, d = q % D;
            cf* row = buf + (q / D) * P + d;
            cf u[C];
#pragma unroll
            for (int c = 0; c < C; ++c) u[c] = row[D * c];
            DIF<C, INV, 0>::run(u);
#pragma unroll
            for (int r = 0; r < C; ++r) {
                const int kc = wf::bitrev<C>(r);
                if (kc) u[r] = twiddle<INV, LO>(u[r], t3, kc * D + d, 2 * M);
                row[D * kc] = u[r];
            }
        }
        sync_line<M>(slot);
    }
    constexpr int Z = D > 1 ? D : C;
#pragma unroll
    for (int j = 0; j < A / Z; ++j) {
        const int q = n2 + G * j, k1 = q % A, kc = q / A;
#pragma unroll
        for (int d = 0; d < Z; ++d) v[j * Z + d] = buf[k1 * P + Z * kc + d];
    }
    sync_line<M>(slot);
#pragma unroll
    for (int j = 0; j < A / Z; ++j) {
        const int q = n2 + G * j, k1 = q % A, kc = q / A;
        DIF<Z, INV, 0>::run(v + j * Z);
#pragma unroll
        for (int r = 0; r < Z; ++r) {
            const int kd = wf::bitrev<Z>(r);
            buf[k1 + A * (D > 1 ? kc + C * kd : kd)] = v[j * Z + r];
        }
    }
    sync_line<M>(slot);
}

// Forward half-length transform of a real line x (16-byte aligned): natural-
// order spectrum in buf.  The reordered line (v[m] = (x[4m], x[4m+2]),
// v[M-1-m] = (x[4m+3], x[4m+1])) is staged in buf.  DST: times (-1)^i, and -1 on odd rows.
template <int M, bool DST>
__device__ __forceinline__ void forward_line(const float* __restrict__ x, cf* buf, const float2* __restrict__ tw, int n2,
                                             int slot, bool odd_row) {
    constexpr int E = Geo<M>::E, G = Geo<M>::G;
    {
        float4 q[E / 2];
#pragma unroll
        for (int i = 0; i < E / 2; ++i) q[i] = __ldcg(reinterpret_cast<const float4*>(x) + (G * i + n2));
#pragma unroll
        for (int i = 0; i < E / 2; ++i) {
            const int m = G * i + n2;
            const float s = DST && odd_row ? -1.f : 1.f;
            buf[m] = DST ? mk(s * q[i].x, s * q[i].z) : mk(q[i].x, q[i].z);
            buf[M - 1 - m] = DST ? mk(-s * q[i].w, -s * q[i].y) : mk(q[i].w, q[i].y);
        }
    }
    sync_line<M>(slot);
    cf v[E];
#pragma unroll
    for (int i = 0; i < E; ++i) v[i] = buf[G * i + n2];
    sync_line<M>(slot);
    fft_line<M, false>(v, buf, tw, n2, slot);
}

// Slots and items as in fixed_fft.cuh: slot i = (X[i], X[N-i]), slot 0 = (X[0],
// X[M]); item k fills the slots k and M-k (k = 0: 0 and M/2).
template <int M> __device__ __forceinline__ int slot_mode(int i, int c) { return c == 0 ? i : i == 0 ? M : 2 * M - i; }
template <int M> __device__ __forceinline__ int item_slot2(int k) { return k == 0 ? M / 2 : M - k; }

// Factors of the pair k (wf::PairTw) from two tables: (wn, a) and b.
struct PairTab { const float4* __restrict__ wa; const float2* __restrict__ b; };
__device__ __forceinline__ wf::PairTw ld_pair(const PairTab& t, int k) {
    const float4 u = __ldg(t.wa + k);
    const float2 b = __ldg(t.b + k);
    return wf::PairTw{u.x, u.y, u.z, u.w, b.x, b.y};
}

template <int M> __device__ __forceinline__ void post_item(const cf* z, const PairTab& t, int k, cf& s1, cf& s2) {
    const cf A = z[k], B = z[item_slot2<M>(k)];
    const Quad<float> q = wf::post_pair_lean(A, k == 0 ? A : B, ld_pair(t, k));
    s1 = mk(q.xk, q.xNk);
    s2 = mk(q.xMk, q.xMpk);
    if (k == 0) {
        const Quad<float> h = wf::post_pair_lean(B, B, ld_pair(t, M / 2));
        s1.y = q.xMk;
        s2 = mk(h.xk, h.xNk);
    }
}
template <int M> __device__ __forceinline__ void pre_item(cf s1, cf s2, const PairTab& t, int k, cf* z) {
    cf a, b;
    if (k != 0) {
        wf::pre_pair_lean(Quad<float>{s1.x, s1.y, s2.x, s2.y}, ld_pair(t, k), a, b);
    } else {
        cf c;
        wf::pre_pair_lean(Quad<float>{s1.x, 0.f, s1.y, s1.y}, ld_pair(t, 0), a, c);
        wf::pre_pair_lean(Quad<float>{s2.x, s2.y, s2.x, s2.y}, ld_pair(t, M / 2), b, c);
    }
    z[k] = a;
    z[item_slot2<M>(k)] = b;
}

// Inverse transform of the line whose pre-processed values lie in buf
// (visible to the line's lanes) to natural-order samples in buf.
template <int M, bool LO = false>
__device__ __forceinline__ void inverse_line(cf* buf, const float2* __restrict__ tw, int n2, int slot) {
    constexpr int E = Geo<M>::E, G = Geo<M>::G;
    cf v[E];
#pragma unroll
    for (int i = 0; i < E; ++i) v[i] = buf[G * i + n2];
    sync_line<M>(slot);
    fft_line<M, true, LO>(v, buf, tw, n2, slot);
}

// ------------------------------------------------------------------ transposed writes
// The modes of the CTA's LINES lines (natural-order spectra in bufs) to
// dst[mode N + r], four rows per 16-byte store (kw_rowdct_T has the scheme).
// lim: values of the array at dst (index checks), o0: dst's index in it.
template <int M, int LINES>
__device__ __forceinline__ void write_modes(const cf* bufs, float* __restrict__ dst, const PairTab& t, size_t o0, size_t lim) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, R4 = LINES / 4;
    auto put = [&](int mode, int r4, float a, float b, float c, float d) {
        if (CCM_OKW(o0 + (size_t)mode * N + 4 * r4, 4, lim))
            *reinterpret_cast<float4*>(dst + (size_t)mode * N + 4 * r4) = make_float4(a, b, c, d);
    };
#pragma unroll 1
    for (int q = threadIdx.x; q < R4 * (M / 2); q += blockDim.x) {
        const int r4 = q % R4, k = q / R4;
        cf s1[4], s2[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) post_item<M>(bufs + (size_t)(4 * r4 + r) * Gm::BUF, t, k, s1[r], s2[r]);
        const int i2 = item_slot2<M>(k);
        put(slot_mode<M>(k, 0), r4, s1[0].x, s1[1].x, s1[2].x, s1[3].x);
        put(slot_mode<M>(k, 1), r4, s1[0].y, s1[1].y, s1[2].y, s1[3].y);
        put(slot_mode<M>(i2, 0), r4, s2[0].x, s2[1].x, s2[2].x, s2[3].x);
        put(slot_mode<M>(i2, 1), r4, s2[0].y, s2[1].y, s2[2].y, s2[3].y);
    }
}
// The samples of the CTA's lines to dst[y N + r] (o0, lim as above).
template <int M, int LINES>
__device__ __forceinline__ void write_samples(const cf* bufs, float* __restrict__ dst, size_t o0, size_t lim) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N, R4 = LINES / 4;
#pragma unroll 1
    for (int q = threadIdx.x; q < R4 * (M / 2); q += blockDim.x) {
        const int r4 = q % R4, m = q / R4;
        cf a[4], b[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const cf* z = bufs + (size_t)(4 * r4 + r) * Gm::BUF;
            a[r] = z[m];
            b[r] = z[M - 1 - m];
        }
        if (!CCM_OKW(o0 + (size_t)(4 * m + 3) * N + 4 * r4, 4, lim)) continue;
        float* d = dst + (size_t)(4 * m) * N + 4 * r4;
        *reinterpret_cast<float4*>(d) = make_float4(a[0].x, a[1].x, a[2].x, a[3].x);
        *reinterpret_cast<float4*>(d + N) = make_float4(b[0].y, b[1].y, b[2].y, b[3].y);
        *reinterpret_cast<float4*>(d + 2 * (size_t)N) = make_float4(a[0].y, a[1].y, a[2].y, a[3].y);
        *reinterpret_cast<float4*>(d + 3 * (size_t)N) = make_float4(b[0].x, b[1].x, b[2].x, b[3].x);
    }
}

// The same writes by a cluster of two CTAs of four lines each, which together
// hold eight rows: each CTA writes half of the modes (samples) of all eight,
// reading the other's four lines through distributed shared memory, so that a
// row segment is 32 bytes (a whole sector) where eight lines do not fit one
// CTA.  dst: the first of the eight rows.
template <int M>
__device__ __forceinline__ void write_modes_pair(cf* bufs, float* __restrict__ dst, const PairTab& t, size_t o0, size_t lim) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N;
    auto cl = cooperative_groups::this_cluster();
    const int rank = (int)cl.block_rank(), r4 = threadIdx.x & 1;
    const cf* z = cl.map_shared_rank(bufs, r4);
    cl.sync();
    auto put = [&](int mode, float a, float b, float c, float d) {
        if (CCM_OKW(o0 + (size_t)mode * N + 4 * r4, 4, lim))
            *reinterpret_cast<float4*>(dst + (size_t)mode * N + 4 * r4) = make_float4(a, b, c, d);
    };
#pragma unroll 1
    for (int q = threadIdx.x; q < M / 2; q += blockDim.x) {
        const int k = rank * (M / 4) + (q >> 1);
        cf s1[4], s2[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) post_item<M>(z + (size_t)r * Gm::BUF, t, k, s1[r], s2[r]);
        const int i2 = item_slot2<M>(k);
        put(slot_mode<M>(k, 0), s1[0].x, s1[1].x, s1[2].x, s1[3].x);
        put(slot_mode<M>(k, 1), s1[0].y, s1[1].y, s1[2].y, s1[3].y);
        put(slot_mode<M>(i2, 0), s2[0].x, s2[1].x, s2[2].x, s2[3].x);
        put(slot_mode<M>(i2, 1), s2[0].y, s2[1].y, s2[2].y, s2[3].y);
    }
    cl.sync();                                         // the other CTA may still read these lines
}
template <int M>
__device__ __forceinline__ void write_samples_pair(cf* bufs, float* __restrict__ dst, size_t o0, size_t lim) {
    using Gm = Geo<M>;
    constexpr int N = Gm::N;
    auto cl = cooperative_groups::this_cluster();
    const int rank = (int)cl.block_rank(), r4 = threadIdx.x & 1;
    const cf* zr = cl.map_shared_rank(bufs, r4);
    cl.sync();
#pragma unroll 1
    for (int q = threadIdx.x; q < M / 2; q += blockDim.x) {
        const int m = rank * (M / 4) + (q >> 1);
        cf a[4], b[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const cf* z = zr + (size_t)r * Gm::BUF;
            a[r] = z[m];
            b[r] = z[M - 1 - m];
        }
        if (!CCM_OKW(o0 + (size_t)(4 * m + 3) * N + 4 * r4, 4, lim)) continue;
        float* d = dst + (size_t)(4 * m) * N + 4 * r4;
        *reinterpret_cast<float4*>(d) = make_float4(a[0].x, a[1].x, a[2].x, a[3].x);
        *reinterpret_cast<float4*>(d + N) = make_float4(b[0].y, b[1].y, b[2].y, b[3].y);
        *reinterpret_cast<float4*>(d + 2 * (size_t)N) = make_float4(a[0].y, a[1].y, a[2].y, a[3].y);
        *reinterpret_cast<float4*>(d + 3 * (size_t)N) = make_float4(b[0].x, b[1].x, b[2].x, b[3].x);
    }
    cl.sync();
}

// Launch in clusters of `cluster` CTAs along x (1: a plain launch).
template <typename... KA, typename... A>
inline void launch_cluster(int cluster, void (*kernel)(KA...), dim3 grid, int threads, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);        // errors: cudaGetLastError, as after <<<>>>
}

}  // namespace lf
}  // namespace ccm

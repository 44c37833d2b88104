// fixed_m.cu -- the FP64 fixed-point line transforms of one line length
// M = FIXED_M (compiled once per length; fixed_ops.h).
#include <cmath>
#include "../../include/ccmsav.h"
#include "fixed_kernels.cuh"

#define FIXED_CAT2(a, b) a##b
#define FIXED_CAT(a, b) FIXED_CAT2(a, b)

namespace ccm {
namespace xf {
namespace {

constexpr int M = FIXED_M, N = 2 * M;
using Gm = Geo<M>;
constexpr int GRID = N / Gm::LINES;
constexpr bool FUSED_GRAM = Gm::LINES == NF;      // eight line buffers fit a CTA

int optin(const void* fn) {
    int dev = 0, lim = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return CCMSAV_ECUDA;
    if ((size_t)lim < Gm::SMEM + 1024) return CCMSAV_EINVAL;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::SMEM) == cudaSuccess ? CCMSAV_OK
                                                                                                                : CCMSAV_ECUDA;
}

int setup(int* gram_rows) {
    const void* fns[] = {(const void*)kx_row_fwd<M, false>, (const void*)kx_row_fwd<M, true>, (const void*)kx_comb_icol<M>,
                         (const void*)kx_irow<M>, (const void*)kx_col_solve<M>, (const void*)kx_row_inv<M, false>,
                         (const void*)kx_row_inv<M, true>};
    for (const void* f : fns)
        if (const int r = optin(f)) return r;
    int dev = 0, nsm = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return CCMSAV_ECUDA;
    if constexpr (FUSED_GRAM) {
        const void* f = (const void*)kx_col_gram<M>;
        if (const int r = optin(f)) return r;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f, Gm::THREADS, Gm::SMEM) != cudaSuccess) return CCMSAV_ECUDA;
    } else {
        if (const int r = optin((const void*)kx_col_fwd<M>)) return r;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, (const void*)kx_gram_rows, kGramThreads, 0) != cudaSuccess)
            return CCMSAV_ECUDA;
    }
    const int all = nsm * (per > 0 ? per : 1);
    *gram_rows = N < all ? N : all;
    return CCMSAV_OK;
}

// exp(i 2 pi j / n) in long double: products of a coarse and a fine table
struct Circle {
    static constexpr int F = 64;
    long n;
    long double cc[4 * N / F + 1], sc[4 * N / F + 1], cf[F], sf[F];
    explicit Circle(long n_) : n(n_) {
        const long double w = 2.0L * 3.14159265358979323846264338327950288L / (long double)n;
        for (int i = 0; i < F; ++i) { cf[i] = cosl(w * i); sf[i] = sinl(w * i); }
        for (long i = 0; i * F < n; ++i) { cc[i] = cosl(w * (i * F)); sc[i] = sinl(w * (i * F)); }
    }
    void at(long j, long double& c, long double& s) const {
        j %= n;
        const long a = j / F, b = j % F;
        c = cc[a] * cf[b] - sc[a] * sf[b];
        s = sc[a] * cf[b] + cc[a] * sf[b];
    }
};

int4 entry(long double x, long double y) {
    auto put = [](long double v, int& h, int& l) {
        long long q = llroundl(v * 4611686018427387904.0L);
        if ((int)(q & 0xffffffffLL) == (int)0x80000000) ++q;      // -l must fit a word
        const Fac f = fac(q);
        h = f.h; l = f.l;
    };
    int4 e;
    put(x, e.x, e.y);
    put(y, e.z, e.w);
    return e;
}

void fill(int4* t, int* pf, int* pi) {
    const Circle* w = new Circle(4L * N);                          // steps of pi / 2N
    long double c, s;
    for (int k1 = 0; k1 < Gm::A; ++k1)
        for (int n2 = 0; n2 < Gm::G; ++n2) {
            w->at(8L * ((long)n2 * k1 % M), c, s);                 // W_M = 8 steps
            t[k1 * Gm::G + n2] = entry(c, -s);
        }
    for (int kc = 0; kc < Gm::C; ++kc)
        for (int d = 0; d < Gm::D; ++d) {
            w->at(8L * Gm::A * ((long)d * kc % Gm::B), c, s);      // W_B = W_M^A
            t[M + kc * Gm::D + d] = entry(c, -s);
        }
    const int np = M / 2 + 1;
    int4 *wn = t + 2 * M, *fa = wn + np, *fb = fa + np, *ia = fb + np, *ib = ia + np;
    int lg = 0;
    while ((1 << lg) < N) ++lg;
    const long double h = sqrtl(0.5L);
    // forward: c_1/2 = sqrt(2/N)/2 = f 2^-pf, c_0/2 = sqrt(1/2) f 2^-pf
    const long double f1 = (lg - 1) % 2 == 0 ? 1.0L : h, f0 = h * f1;
    *pf = (lg - 1) / 2 + 1;
    // inverse: s_1/2 = 1/sqrt(2N) = g 2^-pi, s_0/2 = sqrt(2) g 2^-pi
    const long double g1 = lg % 2 == 0 ? h : 0.5L, g0 = lg % 2 == 0 ? 1.0L : h;
    *pi = lg / 2;
    for (int k = 0; k < np; ++k) {
        w->at(4L * k, c, s);                                       // 2 pi k / N
        wn[k] = entry(c, -s);
        w->at(k, c, s);                                            // pi k / 2N
        const long double fk = k ? f1 : f0, gk = k ? g1 : g0;
        fa[k] = entry(fk * c, -fk * s);
        ia[k] = entry(gk * c, gk * s);
        w->at(N / 2 - k, c, s);                                    // pi / 4 - pi k / 2N
        fb[k] = entry(f1 * c, -f1 * s);
        ib[k] = entry(g1 * c, g1 * s);
    }
    delete w;
}

void weights(const double* ev, const SpecCoef& sc, double* isig, double* itau, cudaStream_t st) {
    const long nb = ((long)N * N + 255) / 256;
    kx_weights<M><<<(int)(nb < 2432 ? nb : 2432), 256, 0, st>>>(ev, sc, isig, itau);
}
void row_step(const double* a, double* b, const Tables& t, cudaStream_t st) {
    kx_row_fwd<M, false><<<dim3(GRID, NF), Gm::THREADS, Gm::SMEM, st>>>(a, b, t.mem, pair_fwd(t), nullptr, (size_t)N * N,
                                                                       (size_t)NF * N * N);
}
void col_gram(const double* b, double* spec, double* part, const Tables& t, const double* isig, const double* itau, int rows,
              cudaStream_t st) {
    if constexpr (FUSED_GRAM) {
        kx_col_gram<M><<<rows, Gm::THREADS, Gm::SMEM, st>>>(b, spec, part, t.mem, pair_fwd(t), isig, itau);
    } else {
        kx_col_fwd<M><<<dim3(GRID, NF), Gm::THREADS, Gm::SMEM, st>>>(b, spec, t.mem, pair_fwd(t));
        kx_gram_rows<<<rows, kGramThreads, 0, st>>>(spec, part, N, isig, itau);
    }
}
void comb(const double* spec, double* b, const Tables& t, const double* isig, const double* itau, const DevScalars* sc,
          cudaStream_t st) {
    kx_comb_icol<M><<<dim3(GRID, 2), Gm::THREADS, Gm::SMEM, st>>>(spec, b, t.mem, pair_inv(t), isig, itau, sc);
}
void irow(const double* b, double* phi_new, double* psi_new, const Tables& t, const double* phn, const double* pho,
          const double* psn, const double* pso, int bdf1, cudaStream_t st) {
    kx_irow<M><<<dim3(GRID, 2), Gm::THREADS, Gm::SMEM, st>>>(b, phi_new, psi_new, t.mem, pair_inv(t), phn, pho, psn, pso, bdf1);
}
void solve(const double* f, double* u, double* scr, const Tables& t, const double* ev, const double c[3], const double* dcoef,
           const int* dskip, int nf, bool dst, cudaStream_t st) {
    const dim3 g(GRID, nf), b(Gm::THREADS);
    const size_t NN = (size_t)N * N;
    if (dst) kx_row_fwd<M, true><<<g, b, Gm::SMEM, st>>>(f, scr, t.mem, pair_fwd(t), dskip, NN, nf * NN);
    else kx_row_fwd<M, false><<<g, b, Gm::SMEM, st>>>(f, scr, t.mem, pair_fwd(t), dskip, NN, nf * NN);
    kx_col_solve<M><<<g, b, Gm::SMEM, st>>>(scr, u, t.mem, pair_fwd(t), pair_inv(t), ev, c[0], c[1], c[2], dcoef, dskip, NN);
    if (dst) kx_row_inv<M, true><<<g, b, Gm::SMEM, st>>>(u, u, t.mem, pair_inv(t), dskip, NN);
    else kx_row_inv<M, false><<<g, b, Gm::SMEM, st>>>(u, u, t.mem, pair_inv(t), dskip, NN);
}
int oob(unsigned* flag) {
    *flag = 0;
#ifdef CCMSAV_BOUNDS
    unsigned z = 0;
    if (cudaMemcpyFromSymbol(flag, g_oob_flag, sizeof(z)) != cudaSuccess || cudaMemcpyToSymbol(g_oob_flag, &z, sizeof(z)) != cudaSuccess)
        return CCMSAV_ECUDA;
#endif
    return CCMSAV_OK;
}

}  // namespace

extern const Ops FIXED_CAT(kFixedOps, FIXED_M);
const Ops FIXED_CAT(kFixedOps, FIXED_M){M,    setup, fill, weights, row_step, col_gram,
                                        comb, irow,  solve, oob};

}  // namespace xf
}  // namespace ccm

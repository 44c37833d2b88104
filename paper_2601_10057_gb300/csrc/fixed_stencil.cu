// fixed_stencil.cu -- coefficients and launches of the FP64 stencil in fixed
// point (fixed_stencil.cuh, fixed_ops.h).
#include <cmath>
#include <algorithm>
#include "../../include/ccmsav.h"
#include "fixed_stencil.cuh"

namespace ccm {
namespace xf {
namespace {

// Tiles: 64 x 32 cells (eight rows a thread) on large grids, smaller ones
// where those would leave SMs without a tile (N = 512: 128 tiles of 64 x 32).
template <typename F> auto with_tile(int N, F f) {
    if (N >= 2048) return f(std::integral_constant<int, 64>(), std::integral_constant<int, 32>());
    if (N >= 512) return f(std::integral_constant<int, 32>(), std::integral_constant<int, 16>());
    return f(std::integral_constant<int, 32>(), std::integral_constant<int, 8>());
}
constexpr int kTileY = 4;

Fac factor(double x) { return fac((long long)std::llround(std::ldexp(x, 62))); }
long long q60(double x) { return (long long)std::llround(std::ldexp(x, Q)); }
int exp_of(double x) {                   // |x| <= 2^e
    int e = 0;
    std::frexp(std::fabs(x), &e);
    return x == 0.0 ? 0 : e;
}

}  // namespace

bool make_stencil(const StencilCoef<double>& c, StencilFix& k) {
    const double coef[] = {c.C2, c.C3, c.Mth, c.betap, c.inv_h2, c.inv_eps, c.eps, c.lam, c.gin, c.gout, c.psin, c.psout, c.bin,
                           c.bout, c.M0, c.beta};
    for (double x : coef)
        if (!std::isfinite(x) || std::fabs(x) > 1e30) return false;
    if (!(std::fabs(c.beta) <= 1.0 && c.M0 >= 0.0 && c.M0 <= 1.0)) return false;
    k = StencilFix{};
    k.bdf1 = c.bdf1;
    // f0'
    const double f1 = c.C2 * (8.0 / 3.0) * c.inv_h2, f2 = c.C3 * (8.0 / 3.0) * c.inv_h2 * c.inv_h2, f3 = c.Mth * c.inv_h2;
    const int fe = exp_of(std::max(std::max(std::fabs(f1), std::fabs(f2)), std::fabs(f3))) + 2;
    k.f_lap = factor(std::ldexp(f1, -fe)); k.f_lap2 = factor(std::ldexp(f2, -fe));
    k.f_th = factor(std::ldexp(f3, -fe));
    k.bar = c.betap / 3.0;
    k.f_exp = fe - Q;
    // S, H, Q
    const int se = exp_of(c.inv_eps);
    k.s_c = factor(std::ldexp(c.inv_eps, -se)); k.s_exp = se - Q;
    k.beta = q60(c.beta);
    k.betaf = fac(k.beta);
    const double s34 = 1.0606601717798212866, hp = s34 * c.inv_eps, hl = s34 * c.eps * c.inv_h2;   // 3 sqrt2 / 4
    const int he = exp_of(std::max(hp, hl));
    k.h_p = factor(std::ldexp(hp, -he)); k.h_l = factor(std::ldexp(hl, -he)); k.h_exp = he - Q;
    const double qx = 2.0 * c.inv_eps2, qt = 3.0 * c.inv_h2;
    const int qe = exp_of(std::max(qx, qt)) + 1;
    k.q_x = factor(std::ldexp(qx, -qe)); k.q_t = factor(std::ldexp(qt, -qe)); k.q_exp = qe - Q;
    // P, K, I_Z: gamma/2 2^-pa <= 1/4, 2 gamma 2^-fa <= 1/2 (|u| <= 4 units: P' <= 2, f' <= 3)
    const int ga = exp_of(std::max(c.gin, c.gout));
    k.pa = ga + 1;
    k.p_in = factor(std::ldexp(c.gin, -k.pa - 1)); k.p_out = factor(std::ldexp(c.gout, -k.pa - 1));
    k.fa = ga + 2;
    k.f_in = factor(std::ldexp(c.gin, 1 - k.fa)); k.f_out = factor(std::ldexp(c.gout, 1 - k.fa));
    const double bm = std::max(std::fabs(c.bin), std::fabs(c.bout));
    k.fb = bm == 0.0 ? -2000 : exp_of(bm);
    k.qpi = factor(0.78539816339744830962);
    k.M0 = factor(c.M0);
    // g0' = lam kq Lap(psi^n - psi^{n-1}), kq = -2/3 (BDF1: 0); L_P
    k.g_c = c.bdf1 ? 0.0 : c.lam * (-2.0 / 3.0) * c.inv_h2;
    k.wV = c.quarter_inv_eps; k.wA = 3.0 * c.inv_h2; k.wB = c.inv_eps2;
    return true;
}

int stencil_setup(int N) {
    return with_tile(N, [&](auto tx, auto ty) {
        constexpr int X = decltype(tx)::value, Y = decltype(ty)::value;
        const void* f = (const void*)k_stencil_fixed<X, kTileY, Y>;
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fixed_stencil_smem<X, Y>()) != cudaSuccess ||
            cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 100) != cudaSuccess)
            return CCMSAV_ECUDA;
        return CCMSAV_OK;
    });
}
int stencil_rows(int N) {
    return with_tile(N, [&](auto tx, auto ty) { return (N / decltype(tx)::value) * (N / decltype(ty)::value); });
}
void stencil(const double* phn, const double* pho, const double* psn, const double* pso, double* out, double* part, int N,
             const StencilFix& k, const StencilCoef<double>& c, const DevScalars* sc, cudaStream_t st) {
    with_tile(N, [&](auto tx, auto ty) {
        constexpr int X = decltype(tx)::value, Y = decltype(ty)::value;
        k_stencil_fixed<X, kTileY, Y><<<dim3(N / X, N / Y), dim3(X, kTileY), fixed_stencil_smem<X, Y>(), st>>>(
            phn, pho, psn, pso, out, part, N, k, c, sc);
        return 0;
    });
}
int stencil_oob(unsigned* flag) {
    *flag = 0;
#ifdef CCMSAV_BOUNDS
    unsigned z = 0;
    if (cudaMemcpyFromSymbol(flag, g_oob_flag, sizeof(z)) != cudaSuccess || cudaMemcpyToSymbol(g_oob_flag, &z, sizeof(z)) != cudaSuccess)
        return CCMSAV_ECUDA;
#endif
    return CCMSAV_OK;
}

}  // namespace xf
}  // namespace ccm

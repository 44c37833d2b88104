// wide_m.cu -- the FP32 kernels on wide lines of one line length M = WIDE_M
// (compiled once per length; wide_ops.h).
#include <cmath>
#include "../../include/ccmsav.h"
#include "wide_kernels.cuh"

#define WIDE_CAT2(a, b) a##b
#define WIDE_CAT(a, b) WIDE_CAT2(a, b)

namespace ccm {
namespace lf {
namespace {

constexpr int M = WIDE_M, N = 2 * M;
using Gm = Geo<M>;
constexpr int GRID = N / Gm::LINES;

int setup() {
    const void* fns[] = {(const void*)kl_row_fwd<M, false>, (const void*)kl_row_fwd<M, true>, (const void*)kl_col_solve<M>,
                         (const void*)kl_row_inv<M, false>, (const void*)kl_row_inv<M, true>, (const void*)kp_row_fwd<M>,
                         (const void*)kp_col<M>, (const void*)kp_row_inv<M>};
    for (const void* f : fns)
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::SMEM) != cudaSuccess) return CCMSAV_ECUDA;
    return CCMSAV_OK;
}

float2 pair(double x) {
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}

void solve(const float* f, float* u, float* scr, const Tables& t, const double c[3], const double* dcoef, const int* dskip,
           int nf, bool dst, cudaStream_t st) {
    const dim3 g(GRID, nf), b(Gm::THREADS);
    const size_t NN = (size_t)N * N;
    const PairTab tf{t.pf, t.pfb}, ti{t.pi, t.pib};
    const double s1 = std::ldexp(1.0, t.shift), s2 = std::ldexp(1.0, 2 * t.shift);
    DivCoef d{};
    if (!dcoef) d = DivCoef{pair(c[0]), pair(c[1] * s1), pair(c[2] * s2)};
    if (dst) kl_row_fwd<M, true><<<g, b, Gm::SMEM, st>>>(f, scr, t.tw, tf, dskip, NN, nf * NN);
    else kl_row_fwd<M, false><<<g, b, Gm::SMEM, st>>>(f, scr, t.tw, tf, dskip, NN, nf * NN);
    kl_col_solve<M><<<g, b, Gm::SMEM, st>>>(scr, u, t.tw, tf, ti, t.ev, d, dcoef, s1, s2, dskip, NN);
    if (dst) kl_row_inv<M, true><<<g, b, Gm::SMEM, st>>>(u, u, t.tw, ti, dskip, NN);
    else kl_row_inv<M, false><<<g, b, Gm::SMEM, st>>>(u, u, t.tw, ti, dskip, NN);
}
void prow_fwd(const float* f, float2* outc, const Tables& t, cudaStream_t st) {
    kp_row_fwd<M><<<GRID, Gm::THREADS, Gm::SMEM, st>>>(f, outc, t.tw, PairTab{t.pf, t.pfb});
}
void pcol(const float2* inc, float2* outc, const Tables& t, const Tables& tev, const double c[3], cudaStream_t st) {
    const double s1 = std::ldexp(1.0, tev.shift), s2 = std::ldexp(1.0, 2 * tev.shift);
    // columns of length M: M / 2 of them
    kp_col<M><<<M / 2 / Gm::LINES, Gm::THREADS, Gm::SMEM, st>>>(inc, outc, t.tw, tev.ev,
                                                               DivCoef{pair(c[0]), pair(c[1] * s1), pair(c[2] * s2)},
                                                               1.0f / ((float)M * (float)M));
}
void prow_inv(const float2* inc, float* u, const Tables& t, cudaStream_t st) {
    kp_row_inv<M><<<M / Gm::LINES, Gm::THREADS, Gm::SMEM, st>>>(inc, u, t.tw);      // rows of length M
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

extern const Ops WIDE_CAT(kWideOps, WIDE_M);
const Ops WIDE_CAT(kWideOps, WIDE_M){M, Gm::A, Gm::C, Gm::D, setup, solve,
                                                      prow_fwd, pcol, prow_inv, oob};

}  // namespace lf
}  // namespace ccm

// wide_ops.h -- host interface of the FP32 kernels on wide lines
// (wide_kernels.cuh), compiled per line length M = N/2 (wide_m.cu, -DWIDE_M=M).
#pragma once
#include <cuda_runtime.h>

namespace ccm {
namespace lf {

// Tables of one solver (device): the twiddles of the two exchanges [2 M] and their low parts [2 M], the
// pair factors (PairTab) and the 1D eigenvalues times 2^-shift as
// (high, low) float pairs.
struct Tables {
    float2* tw = nullptr;
    float4* pf = nullptr;
    float4* pi = nullptr;
    float2* pfb = nullptr;              // the pairs' factors b
    float2* pib = nullptr;
    float2* ev = nullptr;
    int M = 0, shift = 0;
    double smin = 0.0, smax = 0.0;      // smallest and largest eigenvalue of -Lap_h (2D)
};

struct Ops {
    int M, A, C, D;
    int (*setup)();
    // u = (c0 - c1 Lap_h + c2 Lap_h^2)^{-1} f for nf fields (dst: Dirichlet); u may be f.  Coefficients
    // from c, or from the device (dcoef); dskip: fields to leave alone (both may be null).
    void (*solve)(const float* f, float* u, float* scr, const Tables& t, const double c[3], const double* dcoef,
                  const int* dskip, int nf, bool dst, cudaStream_t st);
    // periodic solver: the forward row pass of N = 2M (tables of M), the column pass of N = M
    // (tables of M and of the eigenvalues, tev) and the inverse row pass of N = M
    void (*prow_fwd)(const float* f, float2* outc, const Tables& t, cudaStream_t st);
    void (*pcol)(const float2* inc, float2* outc, const Tables& t, const Tables& tev, const double c[3], cudaStream_t st);
    void (*prow_inv)(const float2* inc, float* u, const Tables& t, cudaStream_t st);
    int (*oob)(unsigned* flag);         // index-check flag of the translation unit: read and cleared (CCMSAV_BOUNDS)
};

const Ops* wide_ops(int M);              // M = 32 .. 4096, else null
// he: the N eigenvalues in the transform's index order (null: twiddles only);
// smin: the smallest of them.  0 or a CCMSAV_E* code.
int make_tables(const Ops* o, Tables& t, const double* he, double smin, cudaStream_t st);
void free_tables(Tables& t);
// Whether the coefficients suit the FP32 pairs of the kernels: a non-negative
// c0 (no cancellation in the divisor) and a divisor within 1e-25 .. 1e25.
bool solve_ok(const Tables& t, const double c[3]);

}  // namespace lf
}  // namespace ccm

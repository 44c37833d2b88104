// fixed_ops.h -- host interface of the FP64 fixed-point line transforms
// (fixed_kernels.cuh).  The kernels of each line length M = N/2 are compiled
// in a translation unit of their own (fixed_m.cu with -DFIXED_M=M, so that
// they build in parallel); fixed_ops(M) returns its launch functions.
#pragma once
#include <cuda_runtime.h>

namespace ccm {
struct SpecCoef;
struct DevScalars;
template <typename T> struct StencilCoef;
namespace xf {

// A factor w (|w| <= 2^62, 62 fractional bits) as w = h 2^32 + l with l a
// signed word; h and -h, -l fit 32 bits.
struct Fac { int h, l; };
__host__ __device__ constexpr Fac fac(long long w) {
    return Fac{(int)((w + 0x80000000LL) >> 32), (int)(w & 0xffffffffLL)};
}

// Coefficients of the fixed-point stencil (fixed_stencil.cuh).  x_c: factors;
// _exp: exponents of the outputs (value = fixed 2^exp); long long: with 60
// fractional bits.  p_in, p_out: gamma/2 2^-pa; f_in, f_out: 2 gamma 2^-fa;
// |beta_in|, |beta_out| <= 2^fb.
struct StencilFix {
    int bdf1;
    int f_exp, s_exp, h_exp, q_exp, pa, fa, fb;
    Fac f_lap, f_lap2, f_th, s_c, betaf, h_p, h_l, q_x, q_t, M0, p_in, p_out, f_in, f_out, qpi;
    long long beta;
    double g_c, bar, wV, wA, wB;
};
// false: parameters outside the kernel's range (the caller takes k_stencil)
bool make_stencil(const StencilCoef<double>& c, StencilFix& k);
int stencil_setup(int N);                // shared-memory opt-in of the kernel for N x N fields
int stencil_rows(int N);                 // partial rows it writes
void stencil(const double* phn, const double* pho, const double* psn, const double* pso, double* out, double* part, int N,
             const StencilFix& k, const StencilCoef<double>& c, const DevScalars* sc, cudaStream_t st);
int stencil_oob(unsigned* flag);         // as Ops::oob

// Twiddle and pair tables of one line length (device, one allocation: the
// twiddles of the two exchanges [M each], then the pair tables wn, forward a, b, inverse a, b [M/2 + 1 each]; each
// entry a complex factor with 62 fractional bits as two (high, signed low)
// word pairs).
struct Tables {
    int4* mem = nullptr;
    int M = 0, pf = 0, pi = 0;          // powers of two of the forward and inverse DCT factors
};

struct Ops {
    int M;
    // opt in to the kernels' shared memory; *gram_rows: partial rows that col_gram leaves
    int (*setup)(int* gram_rows);
    // host values of the tables' 2 M + 5 (M/2 + 1) entries and the powers of two
    void (*fill)(int4* host, int* pf, int* pi);
    void (*weights)(const double* ev, const SpecCoef& sc, double* isig, double* itau, cudaStream_t st);
    // the four transform kernels of a step (fields in a, b as in SimImpl's bufA, bufB)
    void (*row_step)(const double* a, double* b, const Tables& t, cudaStream_t st);
    void (*col_gram)(const double* b, double* spec, double* part, const Tables& t, const double* isig, const double* itau,
                     int rows, cudaStream_t st);
    void (*comb)(const double* spec, double* b, const Tables& t, const double* isig, const double* itau,
                 const DevScalars* sc, cudaStream_t st);
    void (*irow)(const double* b, double* phi_new, double* psi_new, const Tables& t, const double* phn, const double* pho,
                 const double* psn, const double* pso, int bdf1, cudaStream_t st);
    // u = (c0 - c1 Lap_h + c2 Lap_h^2)^{-1} f for nf fields of N x N (Neumann; dst: Dirichlet); scr: nf fields.
    // u may be f.  dcoef: c0, c1, c2 on the device (may be null); dskip: fields to leave alone (may be null).
    void (*solve)(const double* f, double* u, double* scr, const Tables& t, const double* ev, const double c[3],
                  const double* dcoef, const int* dskip, int nf, bool dst, cudaStream_t st);
    int (*oob)(unsigned* flag);         // index-check flag of the translation unit: read and cleared (CCMSAV_BOUNDS)
};

// Launch functions of line length M, or null (M = 32 .. 4096 are built).
const Ops* fixed_ops(int M);
// Device tables of line length M on stream st (the host copy is complete on
// return); 0 or a CCMSAV_E* code.
int make_tables(const Ops* o, Tables& t, cudaStream_t st);
inline void free_tables(Tables& t) { cudaFree(t.mem); t = Tables{}; }

}  // namespace xf
}  // namespace ccm

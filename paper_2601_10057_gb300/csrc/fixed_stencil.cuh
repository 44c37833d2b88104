// fixed_stencil.cuh -- the FP64 stencil (k_stencil of step_kernels.cuh) in
// 64-bit fixed point.
//
// k_stencil<double> executes about 200 FP64 instructions a cell (1.47 ms at
// N = 2048; FP64 issues at 1.66 lanes a clock and SM).  The fields are of
// order one and enter through differences of neighbours, so this kernel holds
// them in fixed point with 60 fractional bits (range +-8): sums and
// differences are exact and cost two integer instructions, a product about
// twelve (36 lane-clocks are one FP64 instruction).
//   phi*, psi*, 3 phi_bar = 4 phi^n - phi^{n-1} and psi^n - psi^{n-1} are exact
//   up to the conversion of the levels (2^-61; FP64 rounds phi* and phi_bar to
//   2^-54), so are the Laplacians; Lap^2 is taken from Lap with 57 bits.
//   Coefficients of any size are normalised to a 62-bit factor and a power of
//   two, the powers applied when a result is converted to FP64.  g0' and L_P,
//   exact sums of differences that add up to zero over the grid, take their
//   coefficient in FP64: a product rounded at the last bit of the fixed-point
//   value is not conservative (psi 7e-14 off after two steps at N = 4096,
//   against 6e-16).  So does the term of f0' in phi_bar (beta > 0), which is the
//   same in every cell of a phase: at the scale of the Lap^2 term its rounding
//   moved phi's mean by 1.4e-13 a step (N = 2048, gamma_bend = 1, dt = 1e-4).
//   The nonlocal bending term uses the identity
//     h^2 [phi |grad phi|^2 - div(phi^2 grad phi)]
//       = -1/2 phi (sum_f d_f^2 + 2 phi h^2 Lap phi) - 1/2 sum_f +-d_f^3
//   over the four face differences d_f (+ east, north; - west, south): the
//   arithmetic face averages of phi^2 expand exactly.
// Each face is evaluated once: a thread takes RPT consecutive rows of a column
// and hands its north face on as the next row's south face, and takes its west
// face from the lane on its left (lane 0 evaluates it).
//
// Measured (one step, event times, no tile outside the range): N = 2048 1475 ->
// 397 us, N = 512 113 -> 39 us, N = 64 112 -> 15 us (the last two mostly from
// tiles small enough to give every SM one); now bound by instruction issue (61 %
// of the slots busy, DRAM 13 %).
//
// Concentrations are in a unit of their own (psi_unit, from psi_in, psi_out and
// the conserved mean), and the osmotic terms P, f_in, f_out of a tile scaled by
// the largest |psi* - psi_in|, |psi* - psi_out| in it: with 60 absolute bits and
// psi of size 1e-3 I_Z was off by 2e-11, at 1e-6 by 5e-6.
//
// Range: |phi*| <= 1.5, |phi_bar| < 4/3, |psi*| <= 3 units, face differences of phi*
// up to 1/4, of 3 phi_bar up to 1 and of the normalised flux up to 1.5,
// |psi^n - psi^{n-1}| <= 1/2 unit.  A CTA with a cell outside (steep profiles,
// diverging or non-finite states) evaluates its tile in FP64 (stencil_tile) after
// that.  A profile of four cells' width has differences of 0.18; evolving states
// of that width were found at 0.21 (N = 256), 0.24 - 0.34 (N = 128) and up to 0.75
// (N = 64, dt = 1e-4: most tiles of most steps, 57 us a step instead of 40).
#pragma once
#include "step_kernels.cuh"
#include "fixed_fft.cuh"
#include "fixed_ops.h"

namespace ccm {
namespace xf {

using ll = long long;

// ------------------------------------------------------------------ arithmetic
// a w / 2^62 rounded, |w| <= 2^62, any a
__device__ __forceinline__ ll mulc(ll a, Fac w) {
    const int l = (int)a, h = (int)(a >> 32) + (int)((unsigned)l >> 31);
    ll c = (1LL << 29) + (ll)h * w.l;
    c += (ll)l * w.h;
    return (c >> 30) + (ll)(((unsigned long long)((ll)h * w.h)) << 2);
}
__device__ __forceinline__ Fac split(ll a) {
    const int l = (int)a;
    return Fac{(int)(a >> 32) + (int)((unsigned)l >> 31), l};
}
// a b / 2^S rounded to about a unit
template <int S> __device__ __forceinline__ ll mulv(Fac a, Fac b) {
    static_assert(S > 33 && S <= 62, "");
    ll c = (1LL << (S - 33)) + (ll)a.h * b.l;
    c += (ll)a.l * b.h;
    return (c >> (S - 32)) + (ll)(((unsigned long long)((ll)a.h * b.h)) << (64 - S));
}
template <int S> __device__ __forceinline__ ll sqrv(Fac a) {
    // the low square counts here: it is never negative, left out it would bias every square
    const ll c = (ll)a.h * a.l + ((1LL << (S - 34)) + (__mulhi(a.l, a.l) >> 1));
    return (c >> (S - 33)) + (ll)(((unsigned long long)((ll)a.h * a.h)) << (64 - S));
}
constexpr int Q = 60;                             // fractional bits of the fields
constexpr ll kOne = 1LL << Q;

// x 2^-p with Q fractional bits, rounded; |x 2^-p| >= 4, infinities and NaN set
// bad.  |p| <= 900.
__device__ __forceinline__ ll to_q(double x, bool& bad, int p = 0) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ffu);
    bad |= e > 1024 + p;
    const unsigned m = (hi & 0xfffffu) | 0x100000u;     // subnormals and zero: far below the last bit
    unsigned H = __funnelshift_l(lo, m, 10), Lw = lo << 10;
    const int r = max(0, min(1024 + p - e, 63));        // mantissa at bit 62 -> 2 units, rounded by the last shift
    if (r >= 32) { Lw = H; H = 0; }
    Lw = __funnelshift_r(Lw, H, r);
    H >>= r & 31;
    const ll q = (ll)(((((unsigned long long)H << 32) | Lw) + 1) >> 1);
    const ll s = (int)hi >> 31;
    return (q ^ s) - s;
}
// |x| <= lim 2^-32 2^Q units of the high word
__device__ __forceinline__ bool outside(ll x, unsigned lim) { return (unsigned)(int)(x >> 32) + lim > 2 * lim; }
__host__ __device__ constexpr unsigned hi_of(double v) { return (unsigned)(v * (double)(1LL << (Q - 32))); }

// sin(pi phi/2) and cos(pi phi/2) with 62 bits for |phi| <= 2 (phi with Q):
// u = 1 - |phi|, cos(pi phi/2) = sin(pi u/2) (exactly 0 at phi = +-1) and
// sin(pi phi/2) = sign(phi) cos(pi u/2); with v = min(|u|, 1 - |u|) <= 1/2 both
// are Taylor polynomials in (pi v/2) (first omitted terms 2^-63 and 2^-68),
// exchanged for |u| > 1/2.
__device__ __forceinline__ void sincos_half_pi(ll phi, ll& sn, ll& cs) {
    const ll sp = phi >> 63;
    const ll u = kOne - ((phi ^ sp) - sp);
    const ll su = u >> 63;
    const ll au = (u ^ su) - su;
    const bool sw = au > kOne / 2;
    const ll v = (sw ? kOne - au : au) << (62 - Q);
    const Fac vf = split(v), w = split(sqrv<62>(vf));
    constexpr ll S[9] = {0x6487ed5110b4611aLL, 0x295779cc4b7ca57dLL, 0x519af19dd6ab875LL, 0x4cb4b3398af617LL, 0x2a0f0690fdcf0LL,
                         0xf183a7ef444LL, 0x3d1e869a03LL, 0xb7d6dcf9LL, 0x1aaec33LL};
    constexpr ll C[10] = {0x4000000000000000LL, 0x4ef4f326f9177969LL, 0x103c1f081b5ac3b3LL, 0x155d3c7e3cbffa0LL, 0xf0fa83448dd5dLL,
                          0x69b47ca8812aLL, 0x1f9d38a3764LL, 0x6db893d13LL, 0x120c62c3LL, 0x25418bLL};
    ll a = S[8], b = C[9];
#pragma unroll
    for (int k = 7; k >= 0; --k) a = S[k] - mulc(a, w);
#pragma unroll
    for (int k = 8; k >= 0; --k) b = C[k] - mulc(b, w);
    a = mulc(a, vf);
    const ll si = sw ? b : a, co = sw ? a : b;          // sin, cos of pi |u| / 2
    cs = (si ^ su) - su;
    sn = (co ^ sp) - sp;
}

// ------------------------------------------------------------------ kernel
template <int TX, int TYB> constexpr size_t fixed_stencil_smem() {
    return ((size_t)(TYB + 4) * (TX + 4) + 4 * (size_t)(TYB + 2) * (TX + 2)) * sizeof(ll);
}

struct Face { ll d, d2, d3, fl; };
// Face between two cells (value at the + side minus the - side): d, d^2 and d^3
// of phi*, the flux M(A phi*) dP; m: the face mobility (62 bits).
__device__ __forceinline__ Face face(ll pm, ll pp, ll Pm, ll Pp, Fac M0, ll& m) {
    Face f;
    f.d = pp - pm;
    const Fac df = split(f.d);
    f.d2 = sqrv<Q>(df);
    f.d3 = mulv<Q>(split(f.d2), df);
    const Fac av = split((pp + pm) >> 1);
    const Fac s = split(sqrv<Q>(av) - kOne);
    m = (1LL << 62) - (mulc(sqrv<Q>(s), M0) << 2);
    f.fl = mulc(Pp - Pm, split(m));
    return f;
}

// Binary exponent p of the unit of psi: the largest of |psi_in|, |psi_out| and of
// the conserved mean lies in 2^(p - 2) .. 2^(p - 1), whatever unit a
// concentration is given in (three units are six times it or more).  The largest
// |psi| is at least the mean, so a mean above 2^(p - 7) keeps the error of psi
// (2^-61 units) below that of FP64.  kNoUnit: smaller means (and units far from
// 1), which take the FP64 stencil.
constexpr int kNoUnit = 0x40000000;
__device__ __forceinline__ int psi_unit(double mean, double psin, double psout) {
    const int em = (int)(mag_hi(mean) >> 20), e = max(max((int)(mag_hi(psin) >> 20), (int)(mag_hi(psout) >> 20)), em);
    return em + 5 < e || e < 1021 - 300 || e > 1021 + 300 ? kNoUnit : e - 1021;
}

// Bitwise or of x over the CTA (two words); s: NW words of 64 bits, read after
// the next barrier by or_all.
__device__ __forceinline__ void or_warp(unsigned long long x, unsigned long long* s) {
    const unsigned l = __reduce_or_sync(0xffffffffu, (unsigned)x), h = __reduce_or_sync(0xffffffffu, (unsigned)(x >> 32));
    if ((threadIdx.x & 31) == 0) *s = ((unsigned long long)h << 32) | l;
}
template <int NW> __device__ __forceinline__ unsigned long long or_all(const unsigned long long* s) {
    unsigned long long x = s[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) x |= s[w];
    return x;
}
// Magnitude of x but for the last unit (one's complement), for or_warp
__device__ __forceinline__ unsigned long long mag_bits(ll x) { return (unsigned long long)(x ^ (x >> 63)); }
__device__ __forceinline__ ll shl(ll x, int s) { return (ll)((unsigned long long)x << s); }
// Left shift that brings values of those bits below 2^top
__device__ __forceinline__ int room(unsigned long long bits, int top) { return max(0, top - 64 + __clzll((ll)bits)); }

// One tile; false if a cell lies outside the range (what has been written is
// then to be written again).
template <int TX, int TY, int TYB>
__device__ __forceinline__ bool
fixed_tile(unsigned char* smraw, const double* __restrict__ phn, const double* __restrict__ pho, const double* __restrict__ psn,
           const double* __restrict__ pso, double* __restrict__ out, double* __restrict__ part, int N, const StencilFix& k,
           const StencilCoef<double>& c, const DevScalars* __restrict__ sc) {
    constexpr int W2 = TX + 4, W1 = TX + 2, H1 = TYB + 2, NT = TX * TY, RPT = TYB / TY, NW = NT / 32;
    ll* sbar = reinterpret_cast<ll*>(smraw);            // 3 phi_bar, [TYB+4][W2]
    ll* sph = sbar + (TYB + 4) * W2;                    // phi*, [H1][W1] each below
    ll* sP = sph + H1 * W1;                             // psi*, then P'
    ll* sdq = sP + H1 * W1;                             // psi^n - psi^{n-1}
    ll* slb = sdq + H1 * W1;                            // h^2 Lap 3 phi_bar / 8
    __shared__ longlong2 ssum[NW][4];                   // (value 2^27 and up, below)
    __shared__ ll smin[NW];
    const int bx = blockIdx.x, by = blockIdx.y, i0 = bx * TX, j0 = by * TYB;
    const int tid = threadIdx.y * TX + threadIdx.x;
    const size_t NN = (size_t)N * N;
    const bool two = !k.bdf1;
    const int pe = psi_unit(sc->mass_mode, c.psin, c.psout);
    if (pe == kNoUnit) return false;                    // the whole grid
    bool bad = false;
    const ll pin = to_q(c.psin, bad, pe), pout = to_q(c.psout, bad, pe);
    __shared__ unsigned long long soa[NW], sou[NW];
    unsigned long long oa = 0;                          // |phi*| - 1
    unsigned long long ou = 0;                          // psi* - psi_in and psi* - psi_out
    {   // halo load, as in stencil_tile
        constexpr int RH = TYB + 4, NR = RH / TY, NI = NR + 1, NB = NI < 4 ? NI : 4;
        static_assert(RH % TY == 0 && 4 * RH <= NT && TYB % TY == 0, "halo load mapping");
        const int cx_ = tid % TX, ty = tid / TX;
        const int gxc = reflect(i0 + cx_ - 2, N);
        const int ex_r = tid >> 2, ex_c = TX + (tid & 3);
        const bool ex_on = tid < 4 * RH;
        const int gxe = reflect(i0 + ex_c - 2, N);
#pragma unroll 1
        for (int u0 = 0; u0 < NI; u0 += NB) {
            double ra[NB], rb[NB], rc[NB], rd[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int u = u0 + b;
                const bool ex = u == NR;
                ra[b] = rb[b] = rc[b] = rd[b] = 0.0;
                if (u < NI && (!ex || ex_on)) {
                    const int lj = ex ? ex_r : ty + TY * u, li = ex ? ex_c : cx_;
                    const size_t g = (size_t)reflect(j0 + lj - 2, N) * N + (ex ? gxe : gxc);
                    ra[b] = phn[CCM_IX(g, NN)];
                    rb[b] = pho[CCM_IX(g, NN)];
                    if (lj >= 1 && lj <= TYB + 2 && li >= 1 && li <= TX + 2) {
                        rc[b] = psn[CCM_IX(g, NN)];
                        rd[b] = pso[CCM_IX(g, NN)];
                    }
                }
            }
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int u = u0 + b;
                const bool ex = u == NR;
                if (u < NI && (!ex || ex_on)) {
                    const int lj = ex ? ex_r : ty + TY * u, li = ex ? ex_c : cx_;
                    const ll a = to_q(ra[b], bad), d = two ? a - to_q(rb[b], bad) : 0;
                    const ll b3 = 3 * a + d, ps = a + d;
                    bad |= outside(b3, hi_of(4.0) - 1) || outside(ps, hi_of(1.5)) || outside(d, hi_of(2.0));
                    sbar[lj * W2 + li] = b3;
                    if (lj >= 1 && lj <= TYB + 2 && li >= 1 && li <= TX + 2) {
                        const int o = (lj - 1) * W1 + (li - 1);
                        const ll s = to_q(rc[b], bad, pe), du = two ? s - to_q(rd[b], bad, pe) : 0;
                        bad |= outside(s + du, hi_of(3.0)) || outside(du, hi_of(0.5));
                        ou |= mag_bits(s + du - pin) | mag_bits(s + du - pout);
                        const ll sg = ps >> 63;
                        oa |= mag_bits((ps ^ sg) - sg - kOne);
                        sph[o] = ps;
                        sP[o] = s + du;
                        sdq[o] = du;
                    }
                }
            }
        }
    }
    or_warp(oa, &soa[tid >> 5]);
    or_warp(ou, &sou[tid >> 5]);
    __syncthreads();
    // The SAV sums take phi^3 - phi and the face differences times 2^sa, phi^2 - 1 - beta times 2^sv, so that a tile
    // away from the interfaces (and a state without any) has its sums to the same relative accuracy as one across an
    // interface.  With | |phi*| - 1 | <= oa the three are at most 2.5 oa (|phi*| <= 3/2), 2 oa and 2.5 oa + |beta|; where
    // sa > 0 a tile holds one phase (differences below 1/4; across phases they are above 7/4, out of range).
    const unsigned long long oat = or_all<NW>(soa);
    const int sa = room(oat, 57), sv = room(3 * oat + 3 + (unsigned long long)llabs(k.beta), 59);
    // The osmotic terms of u = psi* - psi_in, psi* - psi_out (both exact, below 4): u times 2^su, below 1 where it can be,
    // P = P' 2^p_exp, f = gamma/2 u^2 + beta = f' 2^f_exp with |P'| <= 2, |f'| <= 3.
    const int su = room(or_all<NW>(sou), Q), fe0 = k.fa + 2 * (pe - su), f_exp = max(fe0, k.fb), fd = min(f_exp - fe0, 63);
    const int p_exp = k.pa + pe - su;
    const ll bin = to_q(c.bin, bad, f_exp), bout = to_q(c.bout, bad, f_exp);
    const ll half_fd = fd ? 1LL << (fd - 1) : 0;
    // one-halo region: h^2 Lap 3 phi_bar, P'; on the tile's own cells K and the I_Z term
    ll accZ = 0;
#pragma unroll 1
    for (int q = tid; q < W1 * H1; q += NT) {
        const int lj1 = q / W1, li1 = q % W1;
        const ll* b = sbar + (lj1 + 1) * W2 + li1 + 1;
        const ll C = b[0], dE = b[1] - C, dW = b[-1] - C, dN = b[W2] - C, dS = b[-W2] - C;
        bad |= outside(dE, hi_of(1.0)) || outside(dW, hi_of(1.0)) || outside(dN, hi_of(1.0)) || outside(dS, hi_of(1.0));
        slb[q] = (((dE + dW) + (dN + dS)) + 4) >> 3;
        const ll ui = shl(sP[q] - pin, su), uo = shl(sP[q] - pout, su);
        ll sp, cp;
        sincos_half_pi(sph[q], sp, cp);
        const Fac spf = split(sp);
        // P = (1 + p) gamma_in u_in / 2 + (1 - p) gamma_out u_out / 2
        const ll Pi = mulc(ui, k.p_in), Po = mulc(uo, k.p_out);
        sP[q] = (Pi + Po) + mulc(Pi - Po, spf);
        const int gi = i0 + li1 - 1, gj = j0 + lj1 - 1;
        if (lj1 >= 1 && lj1 <= TYB && li1 >= 1 && li1 <= TX && CCM_OK(4 * NN + (size_t)gj * N + gi, 8 * NN)) {
            const ll fi = ((mulc(sqrv<Q + 2>(split(ui)), k.f_in) + half_fd) >> fd) + bin;
            const ll fo = ((mulc(sqrv<Q + 2>(split(uo)), k.f_out) + half_fd) >> fd) + bout;
            const ll D = fi - fo;
            out[4 * NN + (size_t)gj * N + gi] = to_double(fx{mulc(mulc(D, split(cp)), k.qpi)}, f_exp - Q);
            accZ += (fi + fo + mulc(D, spf) + 8) >> 4;
        }
    }
    __syncthreads();
    const int gi = i0 + threadIdx.x, li = threadIdx.x + 1, lane = tid & 31;
    const int r0 = threadIdx.y * RPT;
    ll accV = 0, accA = 0, accB = 0, mmin = 1LL << 62;
    ll mN;
    Face S_;
    {
        const int o = (r0 + 1) * W1 + li;
        S_ = face(sph[o - W1], sph[o], sP[o - W1], sP[o], k.M0, mN);
    }
#pragma unroll 1
    for (int jj = r0; jj < r0 + RPT; ++jj) {
        const int o = (jj + 1) * W1 + li, gj = j0 + jj;
        const size_t g = (size_t)gj * N + gi;
        const ll pC = sph[o], PC = sP[o];
        ll mE;
        const Face E_ = face(pC, sph[o + 1], PC, sP[o + 1], k.M0, mE);
        const Face N_ = face(pC, sph[o + W1], PC, sP[o + W1], k.M0, mN);
        if (gi + 1 < N) mmin = min(mmin, mE);
        if (gj + 1 < N) mmin = min(mmin, mN);
        Face W_;
        W_.d = __shfl_up_sync(0xffffffffu, E_.d, 1);
        W_.d2 = __shfl_up_sync(0xffffffffu, E_.d2, 1);
        W_.d3 = __shfl_up_sync(0xffffffffu, E_.d3, 1);
        W_.fl = __shfl_up_sync(0xffffffffu, E_.fl, 1);
        if (lane == 0) {
            ll m;
            W_ = face(sph[o - 1], pC, sP[o - 1], PC, k.M0, m);
        }
        auto far = [&](const Face& f) { return outside(f.d, hi_of(0.25)) || outside(f.fl, hi_of(1.5)); };
        bad |= far(E_) || far(N_) || far(W_) || far(S_);
        const ll lapp = (E_.d - W_.d) + (N_.d - S_.d);
        const ll sd2 = (E_.d2 + W_.d2) + (N_.d2 + S_.d2);
        const Fac pf = split(pC);
        const ll p2 = sqrv<Q>(pf), p2m = p2 - kOne;
        const ll p3m = mulv<Q>(split(p2m), pf);
        const ll T = mulv<Q>(split(sd2 + 2 * mulv<Q>(split(lapp), pf)), pf) + ((E_.d3 - W_.d3) + (N_.d3 - S_.d3));
        const ll X = mulv<Q>(split(p3m), split(p2 + (p2m >> 1)));           // (phi^3 - phi)(3 phi^2 - 1)/2
        const ll dC = sdq[o];
        const ll lapd = ((sdq[o + 1] - dC) + (sdq[o - 1] - dC)) + ((sdq[o + W1] - dC) + (sdq[o - W1] - dC));
        const ll lC = slb[o];
        const ll lap2 = ((slb[o + 1] - lC) + (slb[o - 1] - lC)) + ((slb[o + W1] - lC) + (slb[o - W1] - lC));
        const ll bC = sbar[(jj + 2) * W2 + li + 1];
        const ll f0 = (mulc(lC, k.f_lap) - mulc(lap2, k.f_lap2)) - mulc(lapp, k.f_th);
        const ll vv = p2m - k.beta;
        if (CCM_OK(7 * NN + g, 8 * NN)) {
            double f = to_double(fx{f0}, k.f_exp);
            if (k.bar != 0.0) f = fma(-k.bar, to_double(fx{bC}, -Q), f);
            out[g] = f;
            out[NN + g] = to_double(fx{mulc(p3m - mulv<Q>(pf, k.betaf), k.s_c)}, k.s_exp);
            out[2 * NN + g] = to_double(fx{mulc(p3m, k.h_p) - mulc(lapp, k.h_l)}, k.h_exp);
            out[3 * NN + g] = to_double(fx{mulc(X, k.q_x) - mulc(T, k.q_t)}, k.q_exp);
            out[5 * NN + g] = to_double(fx{PC}, p_exp - Q);
            out[6 * NN + g] = to_double(fx{lapd}, pe - Q) * k.g_c;
            out[7 * NN + g] = to_double(fx{(E_.fl - W_.fl) + (N_.fl - S_.fl)}, p_exp - Q) * c.inv_h2;
        }
        // the terms of the SAV sums, scaled
        ll a2 = sd2;
        if (sa)
            a2 = (sqrv<Q>(split(shl(E_.d, sa))) + sqrv<Q>(split(shl(W_.d, sa)))) +
                 (sqrv<Q>(split(shl(N_.d, sa))) + sqrv<Q>(split(shl(S_.d, sa))));
        accV += (sqrv<Q>(split(shl(vv, sv))) + 8) >> 4;
        accA += (mulv<Q>(split(a2), split(p2)) + 8) >> 4;
        accB += (sqrv<Q>(split(shl(p3m, sa))) + 8) >> 4;
        S_ = N_;
    }
    // Warp sums of the threads' 56-bit sums (nine cells below 8 at most), exact and without overflow: in pieces of 27,
    // 27 and 10 bits, the upper two put together in units of 2^27.
    const ll v[4] = {accV, accA, accB, accZ};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned p0 = __reduce_add_sync(0xffffffffu, (unsigned)v[q] & 0x7ffffffu);
        const unsigned p1 = __reduce_add_sync(0xffffffffu, (unsigned)(v[q] >> 27) & 0x7ffffffu);
        const int p2 = __reduce_add_sync(0xffffffffu, (int)(v[q] >> 54));
        if (lane == 0) ssum[tid >> 5][q] = make_longlong2(((ll)p2 << 27) + p1, p0);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mmin = min(mmin, __shfl_xor_sync(0xffffffffu, mmin, o));
    if (lane == 0) smin[tid >> 5] = mmin;
    if (__syncthreads_or(bad)) return false;
    if (tid < NRED1) {
        double r = 0.0;
        auto sum = [&](int q, int e) {
            double s = 0.0;
            for (int w = 0; w < NW; ++w) s += to_double(fx{ssum[w][q].x}, e - 29) + to_double(fx{ssum[w][q].y}, e - 56);
            return s;
        };
        if (tid == 0) r = sum(0, -2 * sv) * k.wV;
        else if (tid == 1) r = sum(1, -2 * sa) * k.wA + sum(2, -2 * sa) * k.wB;
        else if (tid == 2) r = sum(3, f_exp);
        else if (tid == 8) {
            ll m = smin[0];
            for (int w = 1; w < NW; ++w) m = min(m, smin[w]);
            r = to_double(fx{m}, -62);
        }
        part[(size_t)(by * gridDim.x + bx) * NRED1 + tid] = r;
    }
    return true;
}

template <int TX, int TY, int TYB>
__global__ void __launch_bounds__(TX * TY, TX * TY <= 128 ? 4 : 2)
k_stencil_fixed(const double* __restrict__ phn, const double* __restrict__ pho, const double* __restrict__ psn,
                const double* __restrict__ pso, double* __restrict__ out, double* __restrict__ part, int N,
                const __grid_constant__ StencilFix k, const __grid_constant__ StencilCoef<double> c,
                const DevScalars* __restrict__ sc) {
    extern __shared__ __align__(16) unsigned char smraw[];
    // uniform over the CTA
    if (!fixed_tile<TX, TY, TYB>(smraw, phn, pho, psn, pso, out, part, N, k, c, sc))
        stencil_tile<double, TX, TY, TYB>(smraw, phn, pho, psn, pso, out, part, N, c, blockIdx.x, blockIdx.y, gridDim.x);
}

}  // namespace xf
}  // namespace ccm

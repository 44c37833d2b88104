// wide_ops.cu -- table of the FP32 wide-line kernels by line length and their
// device tables (wide_ops.h).
#include <cmath>
#include <vector>
#include "../../include/ccmsav.h"
#include "wide_ops.h"

namespace ccm {
namespace lf {

extern const Ops kWideOps32, kWideOps64, kWideOps128, kWideOps256, kWideOps512, kWideOps1024, kWideOps2048, kWideOps4096;

const Ops* wide_ops(int M) {
    switch (M) {
        case 32: return &kWideOps32;
        case 64: return &kWideOps64;
        case 128: return &kWideOps128;
        case 256: return &kWideOps256;
        case 512: return &kWideOps512;
        case 1024: return &kWideOps1024;
        case 2048: return &kWideOps2048;
        case 4096: return &kWideOps4096;
        default: return nullptr;
    }
}

int make_tables(const Ops* o, Tables& t, const double* he, double smin, cudaStream_t st) {
    const int M = o->M, N = 2 * M, G = M / o->A, B = o->C * o->D, np = M / 2 + 1;
    t.M = M;
    std::vector<float2> tw(4 * (size_t)M, make_float2(0.f, 0.f)), ev(N);
    auto root = [&](size_t at, double j, double n) {         // exp(-2 pi i j / n): high parts, the low parts 2 M further on
        const double c = std::cos(2.0 * M_PI * j / n), s = -std::sin(2.0 * M_PI * j / n);
        tw[at] = make_float2((float)c, (float)s);
        tw[at + 2 * (size_t)M] = make_float2((float)(c - (double)tw[at].x), (float)(s - (double)tw[at].y));
    };
    for (int k1 = 0; k1 < o->A; ++k1)
        for (int n2 = 0; n2 < G; ++n2) root((size_t)k1 * G + n2, (double)((long)n2 * k1 % M), M);
    for (int kc = 0; kc < o->C; ++kc)
        for (int d = 0; d < o->D; ++d) root((size_t)M + kc * o->D + d, (double)((long)d * kc % B), B);
    std::vector<float4> pf(np), pi(np);
    std::vector<float2> pfb(np), pib(np);
    const double c0 = std::sqrt(1.0 / N), c1 = std::sqrt(2.0 / N), s0 = 1.0 / (M * c0), s1 = 1.0 / (M * c1), q = M_PI / 4.0;
    for (int k = 0; k < np; ++k) {                           // wf::PairTw
        const double a = 2.0 * M_PI * k / N, th = M_PI * k / (2.0 * N), ck = k ? c1 : c0, sk = k ? s1 : s0;
        pf[k] = make_float4((float)std::cos(a), (float)(-std::sin(a)), (float)(0.5 * ck * std::cos(th)), (float)(-0.5 * ck * std::sin(th)));
        pi[k] = make_float4((float)std::cos(a), (float)(-std::sin(a)), (float)(0.5 * sk * std::cos(th)), (float)(0.5 * sk * std::sin(th)));
        pfb[k] = make_float2((float)(0.5 * c1 * std::cos(q - th)), (float)(-0.5 * c1 * std::sin(q - th)));
        pib[k] = make_float2((float)(0.5 * s1 * std::cos(q - th)), (float)(0.5 * s1 * std::sin(q - th)));
    }
    double mx = 0.0;
    for (int k = 0; he && k < N; ++k) mx = he[k] > mx ? he[k] : mx;
    std::frexp(mx, &t.shift);                                // eigenvalues 2^-shift below 1
    for (int k = 0; he && k < N; ++k) {
        const double x = std::ldexp(he[k], -t.shift);
        const float h = (float)x;
        ev[k] = make_float2(h, (float)(x - (double)h));
    }
    t.smin = 2.0 * smin;
    t.smax = 2.0 * mx;
    if (cudaMalloc(&t.tw, tw.size() * sizeof(float2)) != cudaSuccess || cudaMalloc(&t.pf, np * sizeof(float4)) != cudaSuccess ||
        cudaMalloc(&t.pi, np * sizeof(float4)) != cudaSuccess || cudaMalloc(&t.pfb, np * sizeof(float2)) != cudaSuccess ||
        cudaMalloc(&t.pib, np * sizeof(float2)) != cudaSuccess || cudaMalloc(&t.ev, N * sizeof(float2)) != cudaSuccess)
        return CCMSAV_ENOMEM;
    if (cudaMemcpyAsync(t.tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(t.pf, pf.data(), np * sizeof(float4), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(t.pi, pi.data(), np * sizeof(float4), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(t.pfb, pfb.data(), np * sizeof(float2), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(t.pib, pib.data(), np * sizeof(float2), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(t.ev, ev.data(), N * sizeof(float2), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return CCMSAV_ECUDA;
    return CCMSAV_OK;
}

void free_tables(Tables& t) {
    cudaFree(t.tw); cudaFree(t.pf); cudaFree(t.pi); cudaFree(t.pfb); cudaFree(t.pib); cudaFree(t.ev);
    t = Tables{};
}

bool solve_ok(const Tables& t, const double c[3]) {
    const double lo = c[0] + t.smin * (c[1] + c[2] * t.smin), hi = c[0] + t.smax * (c[1] + c[2] * t.smax);
    return c[0] >= 0.0 && lo > 1e-25 && hi < 1e25 && std::abs(t.shift) <= 300;
}

}  // namespace lf
}  // namespace ccm

// fixed_ops.cu -- table of the FP64 fixed-point line transforms by line
// length and the upload of their twiddle tables (fixed_ops.h).
#include <vector>
#include "../../include/ccmsav.h"
#include "fixed_ops.h"

namespace ccm {
namespace xf {

extern const Ops kFixedOps32, kFixedOps64, kFixedOps128, kFixedOps256, kFixedOps512, kFixedOps1024, kFixedOps2048,
    kFixedOps4096;

const Ops* fixed_ops(int M) {
    switch (M) {
        case 32: return &kFixedOps32;
        case 64: return &kFixedOps64;
        case 128: return &kFixedOps128;
        case 256: return &kFixedOps256;
        case 512: return &kFixedOps512;
        case 1024: return &kFixedOps1024;
        case 2048: return &kFixedOps2048;
        case 4096: return &kFixedOps4096;
        default: return nullptr;
    }
}

int make_tables(const Ops* o, Tables& t, cudaStream_t st) {
    t.M = o->M;
    const size_t n = 2 * (size_t)t.M + 5 * (size_t)(t.M / 2 + 1);
    std::vector<int4> h(n, int4{0, 0, 0, 0});
    o->fill(h.data(), &t.pf, &t.pi);
    if (cudaMalloc(&t.mem, n * sizeof(int4)) != cudaSuccess) { t.mem = nullptr; return CCMSAV_ENOMEM; }
    if (cudaMemcpyAsync(t.mem, h.data(), n * sizeof(int4), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return CCMSAV_ECUDA;
    return CCMSAV_OK;
}

}  // namespace xf
}  // namespace ccm

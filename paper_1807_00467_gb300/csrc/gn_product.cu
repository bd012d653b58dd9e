// Column-marching Gauss-Newton product of the NGF term and its Jacobi
// diagonal: the launches of the body in gn_product_body.cuh (the design is
// described there).
#include "gn_product_body.cuh"

namespace ngf {

namespace {

using namespace gnpk;

template <int RX, int RZ, bool DG>
__global__ void __launch_bounds__(kNT, 1) gn_product_kernel(const __grid_constant__ ColArgs a) {
    if (a.skip && *a.skip) return;   // uniform: every block reads the same flag
    extern __shared__ __align__(128) float smem[];
    __shared__ __align__(8) uint64_t bars[kStages];
    uint32_t pbits = 0;
    gn_product_body<RX, RZ, DG>(a, smem, bars, blockIdx.x, gridDim.x, a.chain != 0, true, pbits);
}

}  // namespace

bool gn_product_supported(const ColGeom &g) {
    if (!g.tma || g.rho[0] < 2 || g.rho[1] < 2 || g.m[2] > 256 || g.nxt * g.nyt > kNodeMax) return false;
    return (size_t)pc_smem(g).total * sizeof(float) <= 227u * 1024u;
}

cudaError_t launch_gn_product(const ColArgs &a0, bool diag, cudaStream_t st) {
    if (!gn_product_supported(a0.g)) return cudaErrorInvalidValue;
    ColArgs a = a0;
    const size_t smem = sizeof(float) * (size_t)pc_smem(a.g).total;
    const int ncols = a.g.nb[0] * a.g.nb[1] * a.g.nbz;
    // persistent CTAs (one per SM, columns strided by the grid) when every
    // column's step count is a whole number of ring cycles, else one column per CTA
    const int tail = a.g.n[2] - (a.g.nbz - 1) * a.g.TZ;
    a.chain = (a.g.TZ + 4) % kStages == 0 && (tail + 4) % kStages == 0;
    const int sms = device_sm_count();
    const int grid = a.chain ? (ncols < sms ? ncols : sms) : ncols;
    auto run = [&](auto kernel) {
        cudaError_t e = allow_max_dynamic_smem(kernel);
        if (e != cudaSuccess) return e;
        kernel<<<grid, kNT, smem, st>>>(a);
        return cudaGetLastError();
    };
#define NGF_PC(RX, RZ) (diag ? run(gn_product_kernel<RX, RZ, true>) : run(gn_product_kernel<RX, RZ, false>))
#define NGF_PX(RX)                           \
    switch (a.g.rho[2]) {                    \
        case 1: return NGF_PC(RX, 1);        \
        case 2: return NGF_PC(RX, 2);        \
        case 4: return NGF_PC(RX, 4);        \
        default: return NGF_PC(RX, 0);       \
    }
    switch (a.g.rho[0]) {
        case 2: NGF_PX(2)
        case 4: NGF_PX(4)
        default: NGF_PX(8)
    }
#undef NGF_PX
#undef NGF_PC
}

}  // namespace ngf

// Volume change control, Eqs. (7)-(9): the launches of the per-cell body of
// vcc_body.cuh (gradient and energy, Gauss-Newton product, its diagonal).

#include "vcc_body.cuh"

namespace ngf {

namespace {

using vcck::NC;

// Blocks per SM by the registers that two cells (F = float2) or one need
// without spills.  The diagonal, whose 24 sums per cell would not fit twice,
// takes one cell per thread.
template <int VM, typename F>
__global__ void __launch_bounds__(NC / vcck::VccSmem<F>::kLanes, VM == 1 || sizeof(F) == 4 ? 4 : 6)
    vcc_cell_kernel(const VccArgs a) {
    if (a.skip && *a.skip) return;   // uniform: every block reads the same flag
    __shared__ vcck::VccSmem<F> sm;
    vcck::vcc_cell_body<VM, F>(a, cuda_block(), sm);
}

}  // namespace

cudaError_t launch_vcc_cells(const VccArgs &a, cudaStream_t st) {
    dim3 grid(a.nb[0], a.nb[1], a.nb[2]);
    // Two cells per thread from more than one wave of one-cell blocks on (4 per
    // SM): gradient 88 against 105 us and GN product 97 against 103 us at
    // 129 x 129 x 65 nodes (8192 blocks), 43 / 49 and 46 / 48 us at 97 x 97 x 49
    // (3456); below, one cell per thread has the shorter chain: 8.4 against
    // 10.5 us at 17 x 17 x 13 (24 blocks), 10.5 / 10.9 us at 33 x 33 x 33 (256).
    // Both forms give the same bits.
    const bool two = (long)a.nb[0] * a.nb[1] * a.nb[2] > 4L * device_sm_count();
    if (a.diag) vcc_cell_kernel<2, float><<<grid, NC, 0, st>>>(a);
    else if (a.v && two) vcc_cell_kernel<1, float2><<<grid, NC / 2, 0, st>>>(a);
    else if (a.v) vcc_cell_kernel<1, float><<<grid, NC, 0, st>>>(a);
    else if (two) vcc_cell_kernel<0, float2><<<grid, NC / 2, 0, st>>>(a);
    else vcc_cell_kernel<0, float><<<grid, NC, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace ngf

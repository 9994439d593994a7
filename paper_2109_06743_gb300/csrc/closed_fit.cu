// Closed-form Newton fits of the 2D3V moment fitting (closed_newton.cuh): the
// double-float kernel of FP32 mode and the FP64 kernel of FP64 mode, for
// every velocity-block size (the block edge is a run-time number there).
#include "closed_newton.cuh"

namespace vl {

cudaError_t launch_closed_fit(const FitArgs& a, cudaStream_t st) {
    // at most 65535 x 65535 cells (vlasov_init): blocks and todo's entries fit 32 bits
    // long before memory does (a cell's fluid, moments and workspace take 1 kB)
    const long long blocks = (2 * a.ncell + 127) / 128;
    if (blocks < 1) return cudaSuccess;
    if (a.fp64) cf::closed_fit_kernel<double><<<(unsigned)blocks, 128, 0, st>>>(a);
    else cf::closed_fit_kernel<df2><<<(unsigned)blocks, 128, 0, st>>>(a);
    count_launch();
    return cudaGetLastError();
}

}  // namespace vl

// Dispatch of the 2D3V Newton fit kernels over the compiled velocity-block
// sizes and the two arithmetics (newton.cuh: double-float on the FP32 pipe;
// newton64.cuh: plain FP64); each size is instantiated in its own
// translation unit (newton_<N>.cu) so that the build compiles them in
// parallel. With a.ntodo the closed-form kernel (closed_fit.cu) runs first
// and these direct kernels take the fits it leaves.
#include "kernels.cuh"

namespace vl {

cudaError_t launch_newton_8(const FitArgs& a, cudaStream_t st);
cudaError_t launch_newton_12(const FitArgs& a, cudaStream_t st);
cudaError_t launch_newton_16(const FitArgs& a, cudaStream_t st);
cudaError_t launch_newton_20(const FitArgs& a, cudaStream_t st);
cudaError_t launch_newton_24(const FitArgs& a, cudaStream_t st);
cudaError_t launch_newton64_8(const FitArgs& a, cudaStream_t st);
cudaError_t launch_newton64_12(const FitArgs& a, cudaStream_t st);
cudaError_t launch_newton64_16(const FitArgs& a, cudaStream_t st);
cudaError_t launch_newton64_20(const FitArgs& a, cudaStream_t st);
cudaError_t launch_newton64_24(const FitArgs& a, cudaStream_t st);

cudaError_t launch_newton3d(const FitArgs& a, cudaStream_t st) {
    if (a.ntodo) {
        const cudaError_t e = launch_closed_fit(a, st);
        if (e != cudaSuccess) return e;
    }
    if (a.fp64) {
        switch (a.nv) {
            case 8: return launch_newton64_8(a, st);
            case 12: return launch_newton64_12(a, st);
            case 16: return launch_newton64_16(a, st);
            case 20: return launch_newton64_20(a, st);
            case 24: return launch_newton64_24(a, st);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (a.nv) {
        case 8: return launch_newton_8(a, st);
        case 12: return launch_newton_12(a, st);
        case 16: return launch_newton_16(a, st);
        case 20: return launch_newton_20(a, st);
        case 24: return launch_newton_24(a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace vl

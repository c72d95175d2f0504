// w5ct_adjoint64js.cu -- the adjoint sweep kernels for Real = double, WENO variant
// 0 (one translation unit per arithmetic type and variant, compiled in
// parallel).
#include "w5ct_adjoint.cuh"

namespace w5ct {

template <>
cudaError_t launch_adj_sweep<double, 0>(int axis, const AdjSweepArgs<double> &a, cudaStream_t s) {
    return launch_adj_sweep_impl<double, 0>(axis, a, s);
}

template <>
cudaError_t prepare_adj_sweep<double, 0>() {
    return prepare_adj_sweep_impl<double, 0>();
}

}  // namespace w5ct

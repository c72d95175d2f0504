// w5ct_adjoint32z.cu -- the adjoint sweep kernels for Real = float, WENO variant
// 1 (one translation unit per arithmetic type and variant, compiled in
// parallel).
#include "w5ct_adjoint.cuh"

namespace w5ct {

template <>
cudaError_t launch_adj_sweep<float, 1>(int axis, const AdjSweepArgs<float> &a, cudaStream_t s) {
    return launch_adj_sweep_impl<float, 1>(axis, a, s);
}

template <>
cudaError_t prepare_adj_sweep<float, 1>() {
    return prepare_adj_sweep_impl<float, 1>();
}

}  // namespace w5ct

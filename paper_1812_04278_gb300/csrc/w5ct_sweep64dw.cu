// w5ct_sweep64dw.cu -- the FP64 single-patch sweeps with the WENO part of
// every characteristic field's flux in double-word arithmetic
// (w5ct_physics.cuh, weno_field): the smoothness
// indicators, the nonlinear weights and the two interpolants of the LF-split
// differences run on the FP32 pipe, while the cell box, the eigenvectors,
// the projections, the split itself, the back-projection and every stored
// value stay in IEEE double.  A translation unit of its own so that it compiles in
// parallel with the other sweeps.
#include "w5ct_internal.h"

namespace w5ct {

cudaError_t launch_sweep_all_f64dw(int variant, const SweepArgs<double> (&a)[3], cudaStream_t s) {
    return variant == 0 ? AllSweeps<double, 0, true>::launch(a, s) : AllSweeps<double, 1, true>::launch(a, s);
}

cudaError_t prepare_sweeps_f64dw() {
    const cudaError_t e = AllSweeps<double, 0, true>::prepare();
    return e == cudaSuccess ? AllSweeps<double, 1, true>::prepare() : e;
}

}  // namespace w5ct

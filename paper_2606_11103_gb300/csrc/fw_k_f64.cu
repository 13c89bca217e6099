// FP64 state and arithmetic: the verification build of the same kernels.
#include "fw_launch.cuh"

namespace fwgb {
cudaError_t sweeps_f64(const fw_medium *m, cudaStream_t s, int which, int j)
{
    return launch_step_sweeps<double, double, double>(m, s, which, j);
}
cudaError_t image_step_f64(const fw_medium *m, const StepImages &im, const int *zero, int it, bool record, bool pdl,
                           cudaStream_t s)
{
    return launch_image_step<double, double>(m, im, zero, it, record, pdl, s);
}
}  // namespace fwgb

// FP32 state and FP32 memory variables.
#include "fw_launch.cuh"

namespace fwgb {
cudaError_t sweeps_f32(const fw_medium *m, cudaStream_t s, int which, int j)
{
    return launch_step_sweeps<float, float, float>(m, s, which, j);
}
cudaError_t image_step_f32(const fw_medium *m, const StepImages &im, const int *zero, int it, bool record, bool pdl,
                           cudaStream_t s)
{
    return launch_image_step<float, float>(m, im, zero, it, record, pdl, s);
}
__global__ void k_advance(int *d_it, int n)
{
    pdl_launch();
    pdl_wait();
    *d_it += n;
}
cudaError_t launch_advance(int *d_it, int n, bool pdl, cudaStream_t s)
{
    return launch_kernel(k_advance, dim3(1), dim3(1), 0, s, pdl, d_it, n);
}
bool vel_maps_f32(EncodeTiledFn encode, fw_medium *m) { return build_vel_maps_t<float, float, float>(encode, m); }
}  // namespace fwgb

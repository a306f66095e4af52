// Instantiations of the fused step kernel: Model B, FP32 populations, N = 2..8.
#include "step_kernel.cuh"

namespace nlbm {

cudaError_t launch_step_b_f32(int ns, const StepParams &p, int tx, int ty, cudaStream_t st)
{
    return launch_step_model<1, 0>(ns, p, tx, ty, st);
}

cudaError_t step_form_b_f32(int ns, const StepParams &p, int tx, StepForm *form, int *wave_rows)
{
    return step_form<1>(ns, p, tx, form, wave_rows);
}

}  // namespace nlbm

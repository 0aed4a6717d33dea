// Single-precision instantiations of the MHD bunch kernels.
#include "kernels_impl.cuh"

namespace mhd {

static const StepLaunch kStepF32[] = {
    StepInst<float, 3, 32, 8, 512>::entry(5.07f, 5.07f),
    StepInst<float, 3, 16, 16, 512>::entry(5.66f, 5.66f),
    StepInst<float, 3, 16, 16, 640>::entry(5.32f, 5.32f),
    StepInst<float, 3, 16, 8, 256, 2>::entry(3.5f, 4.5f),
    StepInst<float, 3, 8, 8, 128, 3>::entry(2.0f, 3.0f),
    StepInst<float, 3, 16, 16, 384>::entry(6.1f, 6.1f),
    StepInst<float, 3, 24, 8, 512>::entry(4.76f, 4.76f),
    StepInst<float, 2, 16, 16, 256>::entry(4.9f, 11.0f),
    StepInst<float, 2, 32, 8, 256>::entry(4.35f, 9.5f),
    StepInst<float, 1, 64, 1, 128>::entry(),
};

const PrecisionKernels& kernels_f32() {
    static const PrecisionKernels k{kStepF32, (int)(sizeof(kStepF32) / sizeof(kStepF32[0])), &launch_fill<float>,
                                    &launch_cfl<float>, &launch_adjoint<float>, AF_N,
                                    &launch_fill_interp<float>, &launch_cfl_patch<float>, &launch_fill_cfl<float>,
                                    &prepare_fill_cfl<float>};
    return k;
}

}  // namespace mhd

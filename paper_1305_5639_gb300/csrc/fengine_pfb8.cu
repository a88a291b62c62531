// F-engine instantiations with the fused polyphase filter bank of up to 8 taps
// (see fengine_kernel.cuh).
#include "fengine_kernel.cuh"

namespace corr {

corr_status fengine_run_pfb8(bool planar, const FShape &f, const float *win, int taps, const void *volt,
                             const float *scale, void *out, cudaStream_t st) {
    return launch_pfb<8>(planar, f, PfbArgs{win, taps}, volt, scale, out, st);
}

}  // namespace corr

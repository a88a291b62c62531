// Power pass of the F-engine with the fused polyphase filter bank, up to 4 and 8 taps
// (see fengine_kernel.cuh).
#include "fengine_kernel.cuh"

namespace corr {

corr_status fengine_run_pfb_power(const FShape &f, const float *win, int taps, const void *volt, double *power,
                                  cudaStream_t st) {
    const PfbArgs pfb{win, taps};
    return taps <= 4 ? launch_pfb_power<4>(f, pfb, volt, power, st) : launch_pfb_power<8>(f, pfb, volt, power, st);
}

}  // namespace corr

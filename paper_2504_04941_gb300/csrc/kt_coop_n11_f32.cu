// kt_coop_n11_f32.cu -- several lanes per cell, 11 unknowns with temperature, FP32-LU (TR-BDF2).
#include "kt_coop.cuh"

namespace kt {

int launch_coop_n11_f32(const LaunchArgs &a, const LaunchCfg &c, void *stream)
{
    return launch_g<11, true, true>(a, c, static_cast<cudaStream_t>(stream));
}

}  // namespace kt

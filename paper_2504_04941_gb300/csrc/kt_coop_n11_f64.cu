// kt_coop_n11_f64.cu -- several lanes per cell, 11 unknowns with temperature, FP64 form.
#include "kt_coop.cuh"

namespace kt {

int launch_coop_n11_f64(const LaunchArgs &a, const LaunchCfg &c, void *stream)
{
    return launch_g<11, true, false>(a, c, static_cast<cudaStream_t>(stream));
}

}  // namespace kt

// kt_coop_any_f64.cu -- several lanes per cell, any size up to 16 unknowns, FP64 form.
#include "kt_coop.cuh"

namespace kt {

int launch_coop_any_f64(const LaunchArgs &a, const LaunchCfg &c, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return a.nv.energy ? launch_t<kLaneMaxN, 16, true, false>(a, c, s)
                       : launch_t<kLaneMaxN, 16, false, false>(a, c, s);
}

}  // namespace kt

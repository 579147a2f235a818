// kt_coop_n3.cu -- four lanes per cell, 3 isothermal unknowns, both forms.
#include "kt_coop.cuh"

namespace kt {

int launch_coop_n3(const LaunchArgs &a, const LaunchCfg &c, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return c.form == KT_FORM_FP32LU ? launch_t<3, 4, false, true>(a, c, s) : launch_t<3, 4, false, false>(a, c, s);
}

}  // namespace kt

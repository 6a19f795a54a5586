// FP32 instantiations of the stage kernels for the HLL and HLLC face fluxes;
// a translation unit of its own so that it compiles in parallel with the others.
#include <cstring>

#include "dispatch.cuh"

namespace gpweno {

gpweno_status launch_stage_f32_var16(gpweno_plan p, const StageIO &io, cudaStream_t st)
{
    return launch_stage_T<float, kVarFlux>(p, io, st);
}

}  // namespace gpweno

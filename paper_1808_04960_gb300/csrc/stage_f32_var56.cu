// FP32 instantiations of the stage kernels with the smoothness indicators in their own scale for any face flux on grids with an external (halo) side;
// a translation unit of its own so that it compiles in parallel with the others.
#include <cstring>

#include "dispatch.cuh"

namespace gpweno {

gpweno_status launch_stage_f32_var56(gpweno_plan p, const StageIO &io, cudaStream_t st)
{
    return launch_stage_T<float, kVarRange | kVarFlux | kVarSlab>(p, io, st);
}

}  // namespace gpweno

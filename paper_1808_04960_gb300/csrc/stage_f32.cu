// FP32 instantiations of the stage kernels (bulk arithmetic in FP32; tables
// rounded from double-double).
#include <cstring>

#include "dispatch.cuh"

namespace gpweno {

gpweno_status launch_stage_f32(gpweno_plan p, const StageIO &io, cudaStream_t st)
{
    const int var = (p->opts.beta_mean ? kVarMean : 0) | (p->opts.scheme ? kVarFdFlux : 0) | (p->opts.ao ? kVarAo : 0) |
                    (has_external_side(p) ? kVarSlab : 0) | (p->opts.flux_form ? kVarFlux : 0) |
                    (p->opts.beta_mean || p->opts.ao || unit_scale_fits(p) ? 0 : kVarRange);
    switch (var) {
    case 0: return launch_stage_T<float, 0>(p, io, st);
    case kVarMean: return launch_stage_f32_var1(p, io, st);
    case kVarFdFlux: return launch_stage_f32_var2(p, io, st);
    case kVarFdFlux | kVarMean: return launch_stage_f32_var3(p, io, st);
    case kVarAo: return launch_stage_f32_var4(p, io, st);
    case kVarAo | kVarMean: return launch_stage_f32_var5(p, io, st);
    case kVarSlab: return launch_stage_f32_var8(p, io, st);
    case kVarFlux: return launch_stage_f32_var16(p, io, st);
    case kVarFlux | kVarMean: return launch_stage_f32_var17(p, io, st);
    case kVarFlux | kVarAo: return launch_stage_f32_var20(p, io, st);
    case kVarFlux | kVarAo | kVarMean: return launch_stage_f32_var21(p, io, st);
    case kVarFlux | kVarSlab: return launch_stage_f32_var24(p, io, st);
    case kVarRange:
    case kVarRange | kVarFlux: return launch_stage_f32_var48(p, io, st);
    case kVarRange | kVarSlab:
    case kVarRange | kVarFlux | kVarSlab: return launch_stage_f32_var56(p, io, st);
    case kVarRange | kVarFdFlux: return launch_stage_f32_var34(p, io, st);
    default: set_error("no kernels for scheme variant %d", var); return GPWENO_ERR_ARG;
    }
}

Tile2D choose_tile_f32(const gpweno_plan_s *p)
{
    return choose_tile(p->dims.n[0], p->dims.n[1], p->R, p->num_sms);
}

gpweno_status launch_max_rate_f32(gpweno_plan p, const void *U, cudaStream_t st)
{
    return launch_max_rate_T<float>(p, U, st);
}

}  // namespace gpweno

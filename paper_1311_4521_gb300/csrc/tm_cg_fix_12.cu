// tm_cg_fix_12.cu -- the solver's fixed-point FP64 hops for 12-real links.
#include "tm_cg_fix.cuh"

namespace twm {

cudaError_t cg_fx_stage_12(const tm_gauge *U, int stage, const void *in, const void *in_fx, void *t, void *q, void *out,
                           bool iterate, const Coef &k, const CgFxArgs &c, cudaStream_t s)
{
    const bool signs = U->geom.anti[1] || U->geom.anti[2] || U->geom.anti[3];
    return signs ? cg_fx_stage<12, true>(U, stage, in, in_fx, t, q, out, iterate, k, c, s)
                 : cg_fx_stage<12, false>(U, stage, in, in_fx, t, q, out, iterate, k, c, s);
}

}  // namespace twm

// tm_cg_fix.cuh -- the solver's FP64 hops with fixed-point link products
// (tm_fix.cuh): the launches of Q^dag Q on an FP64 handle, with the solver's
// reductions and its vector update in the epilogue as in k_cg_hop, and the
// temporaries between them in fixed point.
#pragma once

#include "tm_cg.cuh"
#include "tm_fix.cuh"
#include "tm_internal.h"

namespace twm {

// What a solver hop needs beyond FxArgs.
struct CgFxArgs {
    double *y, *r;            // HOP_UPDATE: solution (increment) and residual, packed FP64
    const void *pdir;         // and the search direction
    double *partials;
    CgScalars *s;
    int gate;
};

// Site i of an FP64 field that this thread has just stored.  Not through the
// read-only path of SpinorIO's loads, which is for memory that nothing writes
// during the kernel.
__device__ __forceinline__ void fx_read_back(const void *base, unsigned vh, unsigned i, Spinor<double> &s)
{
    const volatile double *b = static_cast<const double *>(base) + 2 * size_t(i);
#pragma unroll
    for (int c = 0; c < 12; ++c, b += 2 * size_t(vh)) s[c / 3][c % 3] = {b[0], b[1]};
}

template <int PI, int PO, int RECON, int MODE, bool HASX, bool SIGNS>
__global__ void __launch_bounds__(FX_BLOCK, 6) k_cg_fx_hop(const __grid_constant__ FxArgs A, const __grid_constant__ CgFxArgs C)
{
    __shared__ int4 slots[FxStage<RECON>::WORDS * FX_BLOCK];
    __shared__ unsigned words[12 * FX_BLOCK];
    if (gated(C.s, C.gate)) return;
    const unsigned vh = A.g.vh, site = blockIdx.x * FX_BLOCK + threadIdx.x, i = min(site, vh - 1);
    const FxStage<RECON> st{slots + threadIdx.x};
    const int4 *x0 = HASX ? static_cast<const int4 *>(A.x) + i : nullptr;
    // sites left to FP64 products read the fixed-point t as it is, and for a copy of p the FP64 p
    constexpr int PR = PO == FXF ? F64 : PI;
    Spinor<double> acc, xs, o;
    const FxVerdict verdict = fx_hop_site<PI, RECON, false, SIGNS>(A, i, st, FxSizes<FX_BLOCK>(words), x0, vh, acc);
    if (HASX) st.wait();   // on every path: no thread leaves with copies to its slots under way
    if (HASX) st.site(xs);
    epilogue(A.k, acc, HASX ? &xs : nullptr, o);
    // HOP_UPDATE does not store its result, but for a warp with a site that is looked at again (in a field that
    // serves nothing else)
    const bool on = site < vh;
    if (MODE != HOP_UPDATE || __any_sync(0xffffffffu, on && (verdict.slow || verdict.least < FX_LEAST))) {
        const bool replaced = fx_finish<PR, F64, PO, RECON, false, HASX>(A, i, on, verdict, o);
        if (MODE != HOP_PLAIN && replaced && on) fx_read_back(A.out, vh, i, o);
    }
    double nrm = 0.0;
    if (on) {
        if (MODE == HOP_NORM) nrm = norm2(o);
        if (MODE == HOP_UPDATE) {
            const double alpha = C.s->alpha;
            Spinor<double> pv, v;
            SpinorIO<F64>::load(C.pdir, vh, i, pv);
            SpinorIO<F64>::load(C.y, vh, i, v);
#pragma unroll
            for (int c = 0; c < 12; ++c) v[c / 3][c % 3] = fmadd(alpha, pv[c / 3][c % 3], v[c / 3][c % 3]);
            SpinorIO<F64>::store(C.y, vh, i, v);
            SpinorIO<F64>::load(C.r, vh, i, v);
#pragma unroll
            for (int c = 0; c < 12; ++c) v[c / 3][c % 3] = fmadd(-alpha, o[c / 3][c % 3], v[c / 3][c % 3]);
            SpinorIO<F64>::store(C.r, vh, i, v);
            nrm = norm2(v);
        }
    }
    if (MODE != HOP_PLAIN) reduce_finish<FX_BLOCK>(nrm, C.partials, C.s, MODE == HOP_NORM ? FIN_PAP : FIN_RR_UPDATE);
}

// The four launches of Q^dag Q: stage 0 in -> t, 1 t -> q (in re-read), 2 q
// -> t, 3 t -> out (q re-read).  in, q: packed FP64, with in_fx a fixed-point
// copy of in for stage 0; t: a fixed-point field.  (q as well in fixed point
// alone would cost its small components bits: beside kappa^2 H H they carry
// in itself.)  iterate: the solver's iteration, which reduces |q|^2 in stage
// 1 and applies its update in stage 3 (out: a field for the sites that stage
// 3 looks at again).
template <int RECON, bool SIGNS>
inline cudaError_t cg_fx_stage(const tm_gauge *U, int stage, const void *in, const void *in_fx, void *t, void *q, void *out,
                               bool iterate, const Coef &k, const CgFxArgs &c, cudaStream_t s)
{
    const Geom &g = U->geom;
    const unsigned grid = (g.vh + FX_BLOCK - 1) / FX_BLOCK;
    auto args = [&](const void *input, const void *x, void *output, const void *exact) {
        return FxArgs(g, U->map, k, 1 - (stage & 1), U->fx, U->links, input, x, output, exact);
    };
    switch (stage) {
    case 0:
        if (in_fx) k_cg_fx_hop<FXF, FXF, RECON, HOP_PLAIN, false, SIGNS><<<grid, FX_BLOCK, 0, s>>>(args(in_fx, nullptr, t, in), c);
        else k_cg_fx_hop<F64, FXF, RECON, HOP_PLAIN, false, SIGNS><<<grid, FX_BLOCK, 0, s>>>(args(in, nullptr, t, in), c);
        break;
    case 1:
        if (iterate) k_cg_fx_hop<FXF, F64, RECON, HOP_NORM, true, SIGNS><<<grid, FX_BLOCK, 0, s>>>(args(t, in, q, t), c);
        else k_cg_fx_hop<FXF, F64, RECON, HOP_PLAIN, true, SIGNS><<<grid, FX_BLOCK, 0, s>>>(args(t, in, q, t), c);
        break;
    case 2:
        k_cg_fx_hop<F64, FXF, RECON, HOP_PLAIN, false, SIGNS><<<grid, FX_BLOCK, 0, s>>>(args(q, nullptr, t, q), c);
        break;
    default:
        if (iterate) k_cg_fx_hop<FXF, F64, RECON, HOP_UPDATE, true, SIGNS><<<grid, FX_BLOCK, 0, s>>>(args(t, q, out, t), c);
        else k_cg_fx_hop<FXF, F64, RECON, HOP_PLAIN, true, SIGNS><<<grid, FX_BLOCK, 0, s>>>(args(t, q, out, t), c);
    }
    return cudaGetLastError();
}

// One translation unit per reconstruction (tm_cg_fix_18.cu, tm_cg_fix_12.cu).
cudaError_t cg_fx_stage_18(const tm_gauge *U, int stage, const void *in, const void *in_fx, void *t, void *q, void *out,
                           bool iterate, const Coef &k, const CgFxArgs &c, cudaStream_t s);
cudaError_t cg_fx_stage_12(const tm_gauge *U, int stage, const void *in, const void *in_fx, void *t, void *q, void *out,
                           bool iterate, const Coef &k, const CgFxArgs &c, cudaStream_t s);

}  // namespace twm

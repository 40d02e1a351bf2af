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

// Site i of a field that this thread has just stored.  Not through the
// read-only path of SpinorIO's loads, which is for memory that nothing writes
// during the kernel.
template <int P> __device__ __forceinline__ void fx_read_back(const void *base, unsigned vh, unsigned i, Spinor<double> &s)
{
    const volatile int4 *b = P == FXF ? fx_entry(static_cast<const int4 *>(base), FX_SPINOR_BLOCK, i)
                                      : static_cast<const int4 *>(base) + i;
    const int word = P == FXF ? static_cast<const volatile int *>(fx_words(base, vh))[i] : FX_RAW;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const volatile int4 &q = b[c * (P == FXF ? size_t(32) : size_t(vh))];
        const int4 v = make_int4(q.x, q.y, q.z, q.w);
        s[c / 3][c % 3] = P == FXF ? fx_component(v, word) : cpx<double>{__hiloint2double(v.y, v.x), __hiloint2double(v.w, v.z)};
    }
}

template <int PI, int PX, int PO, int RECON, int MODE, bool HASX, bool SIGNS>
__global__ void __launch_bounds__(FX_BLOCK, 6) k_cg_fx_hop(const __grid_constant__ FxArgs A, const __grid_constant__ CgFxArgs C)
{
    __shared__ int4 slots[FxStage<RECON>::WORDS * FX_BLOCK];
    if (gated(C.s, C.gate)) return;
    const unsigned vh = A.g.vh, site = blockIdx.x * FX_BLOCK + threadIdx.x, i = min(site, vh - 1);
    const FxStage<RECON> st{slots + threadIdx.x};
    const int4 *x0 = HASX && PX == F64 ? static_cast<const int4 *>(A.x) + i : nullptr;
    Spinor<double> acc, xs, o;
    const bool slow = fx_hop_site<PI, RECON, false, SIGNS>(A, i, st, x0, vh, acc);
    if (HASX && PX == F64) st.wait();   // on every path: no thread leaves with copies to its slots under way
    double nrm = 0.0;
    if (site < vh) {
        if (slow) {   // stored, then read back (HOP_UPDATE: from a field that serves nothing else)
            fx_slow_site<PI, PX, PO, RECON, false, HASX>(A, i);
            if (MODE != HOP_PLAIN) fx_read_back<PO>(A.out, vh, i, o);
        } else {
            if (HASX && PX == F64) {
                st.site(xs);
            } else if (HASX) {
                SpinorIO<PX>::load_raw(A.x, vh, i, xs);
            }
            epilogue(A.k, acc, HASX ? &xs : nullptr, o);
            if (MODE != HOP_UPDATE) SpinorIO<PO>::store(A.out, vh, i, o);
        }
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
// -> t, 3 t -> out (q re-read).  in: packed FP64, or with in_fx a fixed-point
// copy of it for stage 0.  t, q: fixed-point fields.  iterate: the solver's
// iteration, which reduces |q|^2 in stage 1 and applies its update in stage 3
// (out: a field for the sites that stage 3 computes with FP64 products).
template <int RECON, bool SIGNS>
inline cudaError_t cg_fx_stage(const tm_gauge *U, int stage, const void *in, const void *in_fx, void *t, void *q, void *out,
                               bool iterate, const Coef &k, const CgFxArgs &c, cudaStream_t s)
{
    const Geom &g = U->geom;
    const unsigned grid = (g.vh + FX_BLOCK - 1) / FX_BLOCK;
    FxArgs A{g, U->map, k, 1 - (stage & 1), static_cast<const FxEntry *>(U->fx), static_cast<const double2 *>(U->links),
             in, nullptr, t};
    switch (stage) {
    case 0:
        if (in_fx) {
            A.in = in_fx;
            k_cg_fx_hop<FXF, F64, FXF, RECON, HOP_PLAIN, false, SIGNS><<<grid, FX_BLOCK, 0, s>>>(A, c);
        } else {
            k_cg_fx_hop<F64, F64, FXF, RECON, HOP_PLAIN, false, SIGNS><<<grid, FX_BLOCK, 0, s>>>(A, c);
        }
        break;
    case 1:
        A.in = t;
        A.x = in;
        A.out = q;
        if (iterate) k_cg_fx_hop<FXF, F64, FXF, RECON, HOP_NORM, true, SIGNS><<<grid, FX_BLOCK, 0, s>>>(A, c);
        else k_cg_fx_hop<FXF, F64, FXF, RECON, HOP_PLAIN, true, SIGNS><<<grid, FX_BLOCK, 0, s>>>(A, c);
        break;
    case 2:
        A.in = q;
        k_cg_fx_hop<FXF, F64, FXF, RECON, HOP_PLAIN, false, SIGNS><<<grid, FX_BLOCK, 0, s>>>(A, c);
        break;
    default:
        A.in = t;
        A.x = q;
        A.out = out;
        if (iterate) k_cg_fx_hop<FXF, FXF, F64, RECON, HOP_UPDATE, true, SIGNS><<<grid, FX_BLOCK, 0, s>>>(A, c);
        else k_cg_fx_hop<FXF, FXF, F64, RECON, HOP_PLAIN, true, SIGNS><<<grid, FX_BLOCK, 0, s>>>(A, c);
    }
    return cudaGetLastError();
}

// One translation unit per reconstruction (tm_cg_fix_18.cu, tm_cg_fix_12.cu).
cudaError_t cg_fx_stage_18(const tm_gauge *U, int stage, const void *in, const void *in_fx, void *t, void *q, void *out,
                           bool iterate, const Coef &k, const CgFxArgs &c, cudaStream_t s);
cudaError_t cg_fx_stage_12(const tm_gauge *U, int stage, const void *in, const void *in_fx, void *t, void *q, void *out,
                           bool iterate, const Coef &k, const CgFxArgs &c, cudaStream_t s);

}  // namespace twm

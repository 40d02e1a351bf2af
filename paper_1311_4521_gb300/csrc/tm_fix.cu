// tm_fix.cu -- the FP64 hop with fixed-point link products (tm_fix.cuh): the
// limb copy of the links and the hop kernels.
#include "tm_fix.cuh"
#include "tm_internal.h"

// Resident CTAs of 64 threads per SM the fixed-point hops are compiled for:
// 6 (168 registers) measured fastest at 32^3x64: Q_tm 0.80 ms against 0.94
// (4) and 0.96 (7, whose 128 registers spill); the hop on FP64 fields 0.47
// against 0.56 ms (4).
#ifndef TM_FX_MINB
#define TM_FX_MINB 6
#endif

namespace twm {

// The limbs of every link from its FP64 storage, and whether all of them
// can be used (fx_link_ok; for 12-real links with the rebuilt third row):
// *unfit is set to 1 otherwise.  One thread per (parity, direction, site);
// integers only, so that the copy takes the time of its traffic (with FP64
// arithmetic it took 3 ms at 32^3x64, its 2.4 GB need 0.4).
template <int RECON>
__global__ void __launch_bounds__(128) k_fx_links(unsigned vh, const double2 *__restrict__ links, FxEntry *__restrict__ fx,
                                                  int *unfit)
{
    constexpr int NC = RECON / 2;
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x, blk = blockIdx.y;
    if (i >= vh) return;
    FxEntry u[9];
    bool ok = true;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const double2 v = ld_stream(links + (size_t(blk) * NC + k) * vh + i);
        // below 1 + 2^-20 and so finite
        ok = ok && (__double2hiint(v.x) & 0x7fffffff) < 0x3ff00001 && (__double2hiint(v.y) & 0x7fffffff) < 0x3ff00001;
        fx_split(v.x, 1025u, 0u, u[k].x, u[k].y);
        fx_split(v.y, 1025u, 0u, u[k].z, u[k].w);
    }
    if (RECON == 12 && ok) {
        u[6] = fx_minor(u[1], u[5], u[2], u[4]);
        u[7] = fx_minor(u[2], u[3], u[0], u[5]);
        u[8] = fx_minor(u[0], u[4], u[1], u[3]);
    }
    if (!ok || !fx_link_ok(u)) {
        *unfit = 1;
        return;
    }
    constexpr unsigned block = fx_link_block(RECON);
    FxEntry *o = fx_entry(fx + size_t(blk >> 2) * fx_blocks(vh) * (block / 16), block, i) + (blk & 3) * NC * 32;
#pragma unroll
    for (int k = 0; k < NC; ++k) st_stream(o + 32 * k, u[k]);
}

cudaError_t launch_fx_links(unsigned vh, int recon, const void *links, void *fx, int *unfit, cudaStream_t s)
{
    const dim3 grid((vh + 127) / 128, 8);
    if (recon == 18)
        k_fx_links<18><<<grid, 128, 0, s>>>(vh, static_cast<const double2 *>(links), static_cast<FxEntry *>(fx), unfit);
    else
        k_fx_links<12><<<grid, 128, 0, s>>>(vh, static_cast<const double2 *>(links), static_cast<FxEntry *>(fx), unfit);
    return cudaGetLastError();
}

// An FP64 field (packed or canonical) in fixed point.
template <int PI> __global__ void __launch_bounds__(128) k_fx_field(unsigned vh, const void *__restrict__ in, void *__restrict__ out)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= vh) return;
    Spinor<double> s;
    SpinorIO<PI>::load(in, vh, i, s);
    SpinorIO<FXF>::store(out, vh, i, s);
}

// The hop of k_hop / k_hop_io with fixed-point link products: input, re-read
// input and output each packed FP64, canonical FP64 or (input and output) a
// fixed-point field.
template <int PI, int PX, int PO, int RECON, bool DAG, bool HASX, bool SIGNS>
__global__ void __launch_bounds__(FX_BLOCK, TM_FX_MINB)
    k_fx_hop(const __grid_constant__ FxArgs A)
{
    __shared__ int4 slots[FxStage<RECON>::WORDS * FX_BLOCK];
    const Geom &g = A.g;
    const SiteMap &m = A.m;
    // the map's CTAs of m.block threads, laid end to end; threads past the end repeat the last site
    const unsigned v = blockIdx.x * FX_BLOCK + threadIdx.x, b = m.tiled ? v / m.block : 0u;
    const unsigned site = m.tiled ? (b < g.vh / m.block ? map_site(g, m, b, v - b * m.block) : g.vh) : v;
    const unsigned i = min(site, g.vh - 1);
    const FxStage<RECON> st{slots + threadIdx.x};
    const int4 *x0 = HASX ? static_cast<const int4 *>(A.x) + (PX == F64C ? size_t(i) * 12 : size_t(i)) : nullptr;
    Spinor<double> acc, xs, o;
    const bool slow = fx_hop_site<PI, RECON, DAG, SIGNS>(A, i, st, x0, PX == F64C ? 1 : g.vh, acc);
    if (site >= g.vh) return;
    if (slow) {
        fx_slow_site<PI, PX, PO, RECON, DAG, HASX>(A, i);
        return;
    }
    if (HASX) {
        st.wait();
        st.site(xs);
    }
    epilogue(A.k, acc, HASX ? &xs : nullptr, o);
    SpinorIO<PO>::store(A.out, g.vh, i, o);
}

static unsigned fx_grid(unsigned vh) { return (vh + FX_BLOCK - 1) / FX_BLOCK; }

template <int RECON>
static cudaError_t launch_f64_fields(const tm_gauge *U, bool dag, int p, const void *in, void *out, const void *x, const Coef &k,
                          cudaStream_t s, const SiteMap &m)
{
    auto kern = dag ? (x ? k_fx_hop<F64, F64, F64, RECON, true, true, true> : k_fx_hop<F64, F64, F64, RECON, true, false, true>)
                    : (x ? k_fx_hop<F64, F64, F64, RECON, false, true, true> : k_fx_hop<F64, F64, F64, RECON, false, false, true>);
    kern<<<fx_grid(U->geom.vh), FX_BLOCK, 0, s>>>(
        FxArgs{U->geom, m, k, p, static_cast<const FxEntry *>(U->fx), static_cast<const double2 *>(U->links), in, x, out});
    return cudaGetLastError();
}

cudaError_t launch_fx_hop(const tm_gauge *U, bool dag, int out_parity, const void *in, void *out, const void *x,
                          const Coef &k, cudaStream_t s, const SiteMap &m)
{
    return U->recon == 18 ? launch_f64_fields<18>(U, dag, out_parity, in, out, x, k, s, m)
                          : launch_f64_fields<12>(U, dag, out_parity, in, out, x, k, s, m);
}

size_t fx_copy_bytes(const tm_gauge *U) { return fx_link_bytes(U->geom.vh, U->recon); }

size_t fx_qtm_bytes(unsigned vh) { return 2 * align256(fx_field_bytes(vh)); }

template <int PI, int RECON>
static cudaError_t fx_qtm(const tm_gauge *U, bool stage_b, const void *in, void *tmp, void *out, const Coef &k, cudaStream_t s)
{
    const Geom &g = U->geom;
    const FxEntry *f = static_cast<const FxEntry *>(U->fx);
    const double2 *l = static_cast<const double2 *>(U->links);
    void *even = static_cast<char *>(tmp) + align256(fx_field_bytes(g.vh));
    const bool signs = g.anti[1] || g.anti[2] || g.anti[3];
    if (!stage_b) {
        auto kern = signs ? k_fx_hop<FXF, F64, FXF, RECON, false, false, true> : k_fx_hop<FXF, F64, FXF, RECON, false, false, false>;
        k_fx_field<PI><<<(g.vh + 127) / 128, 128, 0, s>>>(g.vh, in, even);
        kern<<<fx_grid(g.vh), FX_BLOCK, 0, s>>>(FxArgs{g, U->map, k, 1, f, l, even, nullptr, tmp});
    } else {
        auto kern = signs ? k_fx_hop<FXF, PI, PI, RECON, false, true, true> : k_fx_hop<FXF, PI, PI, RECON, false, true, false>;
        kern<<<fx_grid(g.vh), FX_BLOCK, 0, s>>>(FxArgs{g, U->map, k, 0, f, l, tmp, in, out});
    }
    return cudaGetLastError();
}

cudaError_t launch_fx_qtm(const tm_gauge *U, bool canonical, bool stage_b, const void *in, void *tmp, void *out,
                          const Coef &k, cudaStream_t s)
{
    if (U->recon == 18) return canonical ? fx_qtm<F64C, 18>(U, stage_b, in, tmp, out, k, s) : fx_qtm<F64, 18>(U, stage_b, in, tmp, out, k, s);
    return canonical ? fx_qtm<F64C, 12>(U, stage_b, in, tmp, out, k, s) : fx_qtm<F64, 12>(U, stage_b, in, tmp, out, k, s);
}

}  // namespace twm

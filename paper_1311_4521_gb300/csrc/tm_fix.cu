// tm_fix.cu -- the FP64 hop with fixed-point link products (tm_fix.cuh): the
// limb copy of the links and the hop kernels.
#include "tm_fix.cuh"
#include "tm_internal.h"

// Resident CTAs of 64 threads per SM the fixed-point hops are compiled for:
// 6 (168 registers) measured fastest at 32^3x64: when chosen, Q_tm 0.80 ms against 0.94
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
    unsigned bits = 0;   // of all entries, signs aside
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const double2 v = ld_stream(links + (size_t(blk) * NC + k) * vh + i);
        // below 1 + 2^-20 and so finite
        ok = ok && (__double2hiint(v.x) & 0x7fffffff) < 0x3ff00001 && (__double2hiint(v.y) & 0x7fffffff) < 0x3ff00001;
        bits |= unsigned((__double2hiint(v.x) | __double2hiint(v.y)) & 0x7fffffff) | unsigned(__double2loint(v.x) | __double2loint(v.y));
        fx_split_near(v.x, 1025u, u[k].x, u[k].y);
        fx_split_near(v.y, 1025u, u[k].z, u[k].w);
    }
    if (RECON == 12 && ok) {
        u[6] = fx_minor(u[1], u[5], u[2], u[4]);
        u[7] = fx_minor(u[2], u[3], u[0], u[5]);
        u[8] = fx_minor(u[0], u[4], u[1], u[3]);
    }
    if (!ok || !fx_link_ok(u, bits == 0)) {
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
// fixed-point field; PR is the format of the input that sites left to FP64
// products read (A.exact).
template <int PI, int PR, int PX, int PO, int RECON, bool DAG, bool HASX, bool SIGNS>
__global__ void __launch_bounds__(FX_BLOCK, TM_FX_MINB)
    k_fx_hop(const __grid_constant__ FxArgs A)
{
    __shared__ int4 slots[FxStage<RECON>::WORDS * FX_BLOCK];
    __shared__ unsigned words[12 * FX_BLOCK];
    const Geom &g = A.g;
    const SiteMap &m = A.m;
    // the map's CTAs of m.block threads, laid end to end; threads past the end repeat the last site
    const unsigned v = blockIdx.x * FX_BLOCK + threadIdx.x, b = m.tiled ? v / m.block : 0u;
    const unsigned site = m.tiled ? (b < g.vh / m.block ? map_site(g, m, b, v - b * m.block) : g.vh) : v;
    const unsigned i = min(site, g.vh - 1);
    const FxStage<RECON> st{slots + threadIdx.x};
    const int4 *x0 = HASX ? static_cast<const int4 *>(A.x) + (PX == F64C ? size_t(i) * 12 : size_t(i)) : nullptr;
    Spinor<double> acc, xs, o;
    const FxSizes<FX_BLOCK> sizes(words);
    const FxVerdict verdict = fx_hop_site<PI, RECON, DAG, SIGNS>(A, i, st, sizes, x0, PX == F64C ? 1 : g.vh, acc);
    if (HASX) st.wait();   // on every path: no thread leaves with copies to its slots under way
    if (HASX) st.site(xs);
    epilogue(A.k, acc, HASX ? &xs : nullptr, o);
    fx_finish<PR, PX, PO, RECON, DAG, HASX>(A, i, site < g.vh, verdict, o);
}

// The same hop with the 8 hops of a site dealt out to four warps, one
// direction each, for lattices whose sites do not fill the GPU: a CTA covers
// 32 sites.  The warps' integer sums, and the sums of absolute values, meet in
// shared memory, then warp w finishes spin w.  The site map is not used (results do not depend on it).
constexpr int FX_SPLIT = 128;
template <int RECON> constexpr size_t fx_split_bytes() { return sizeof(int4) * FxStage<RECON, FX_SPLIT>::WORDS * FX_SPLIT; }

template <int PI, int PX, int PO, int RECON, bool DAG, bool HASX, bool SIGNS>
__global__ void __launch_bounds__(FX_SPLIT, 3) k_fx_hop_split(const __grid_constant__ FxArgs A)
{
    extern __shared__ int4 dyn[];
    __shared__ int4 info[FX_SPLIT];
    __shared__ unsigned words[12 * FX_SPLIT];   // [12][4 directions][32]
    const Geom &g = A.g;
    const unsigned vh = g.vh, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned site = blockIdx.x * 32 + lane, i = min(site, vh - 1);
    const FxStage<RECON, FX_SPLIT> st{dyn + threadIdx.x};
    Nbrs n;
    neighbours(g, A.p, i, n);
    const FxLinks<RECON> src{A.fx, vh, i, A.p};
    FxSum t;
    unsigned long long d = 0;
    t.clear(FX_LOWEST_E);
    const FxSizes<FX_SPLIT> sizes(words);
    switch (w) {
    case 0: fx_start<PI, 0>(g, n, src, A.in, st); break;
    case 1: fx_start<PI, 2>(g, n, src, A.in, st); break;
    case 2: fx_start<PI, 4>(g, n, src, A.in, st); break;
    default: fx_start<PI, 6>(g, n, src, A.in, st);
    }
    double2 x[3];   // spin w of the re-read input
    if (HASX)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 *b = static_cast<const double2 *>(A.x);
            x[c] = ld_keep(PX == F64C ? b + size_t(i) * 12 + 3 * w + c : b + size_t(3 * w + c) * vh + i);
        }
    bool slow = false;
    if constexpr (PI == FXF) slow = fx_exponents(n, A.in, vh, t.e, d);
    switch (w) {
    case 0: fx_hops<PI, DAG, 0, 1, SIGNS>(g, n, src, A.in, st, nullptr, 0, d, t, sizes, slow); break;
    case 1: fx_hops<PI, DAG, 2, 3, SIGNS>(g, n, src, A.in, st, nullptr, 0, d, t, sizes, slow); break;
    case 2: fx_hops<PI, DAG, 4, 5, SIGNS>(g, n, src, A.in, st, nullptr, 0, d, t, sizes, slow); break;
    default: fx_hops<PI, DAG, 6, 7, SIGNS>(g, n, src, A.in, st, nullptr, 0, d, t, sizes, slow);
    }
    if constexpr (PI != FXF) {   // the directions' exponents and ranges meet first
        info[threadIdx.x] = make_int4(t.e, slow, 0, 0);
        __syncthreads();
        const int own = t.e;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int4 q = info[32 * v + lane];
            t.e = max(t.e, q.x);
            slow = slow || q.y;
        }
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                t.re[s][c] = fx_sar(t.re[s][c], t.e - own);
                t.im[s][c] = fx_sar(t.im[s][c], t.e - own);
            }
        sizes.sar(t.e - own);
    } else {
        __syncthreads();   // every warp has read its staged words
    }
    long long *part = reinterpret_cast<long long *>(dyn);   // [24][4 directions][32]
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            part[(6 * s + 2 * c) * FX_SPLIT + threadIdx.x] = t.re[s][c];
            part[(6 * s + 2 * c + 1) * FX_SPLIT + threadIdx.x] = t.im[s][c];
        }
    __syncthreads();
    constexpr int bits = PI == FXF ? FX_FIELD : FX_HALF;
    const bool up = w < 2;
    const cpx<double> a = up ? cpx<double>{A.k.d[0], A.k.d[1]} : cpx<double>{A.k.d[2], A.k.d[3]};
    const cpx<double> b = up ? cpx<double>{A.k.d[4], A.k.d[5]} : cpx<double>{A.k.d[6], A.k.d[7]};
    cpx<double> o[3];
    unsigned least2 = 0xffffffffu;   // of this warp's spin, re and im
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const long long *q = part + (6 * w + 2 * c) * FX_SPLIT + lane;
        const long long re = q[0] + q[32] + q[64] + q[96];
        const long long im = q[FX_SPLIT] + q[FX_SPLIT + 32] + q[FX_SPLIT + 64] + q[FX_SPLIT + 96];
        const cpx<double> hop = {fx_to_double(re, t.e, bits), fx_to_double(im, t.e, bits)};
        const volatile unsigned *z = words + (3 * w + c) * FX_SPLIT + lane;
        least2 = __vminu2(least2, z[0] + z[32] + z[64] + z[96]);
        o[c] = A.k.unit ? (up ? hop : -hop) : a * hop;
        if (HASX) o[c] = cmadd(b, cpx<double>{x[c].x, x[c].y}, o[c]);
    }
    // the spins' ranges and smallest sums meet; then all know what is to be done
    int least = int(min(least2 & 0xffffu, least2 >> 16));
    unsigned m = 0, any = 0;
    if (PO == FXF)
#pragma unroll
        for (int c = 0; c < 3; ++c) fx_range_of(o[c], m, any);
    __syncthreads();
    info[threadIdx.x] = make_int4(int(m), int(any), least, 0);
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int4 q = info[32 * v + lane];
        m = max(m, unsigned(q.x));
        any |= unsigned(q.y);
        least = min(least, q.z);
    }
    const FxVerdict verdict(slow, least, t.e, bits);
    bool again = verdict.least < FX_LEAST;
    if constexpr (PO == FXF) {
        const FxSite f(m, any);
        if (site < vh && !slow) {
#pragma unroll
            for (int c = 0; c < 3; ++c) f.store(A.out, i, 3 * w + c, o[c]);
            if (w == 0) f.store_word(A.out, vh, i);
        }
        again = again || !fx_stores(A, float(verdict.least), verdict.e, f);
    } else if (site < vh && !slow) {
        double2 *q = static_cast<double2 *>(A.out);
#pragma unroll
        for (int c = 0; c < 3; ++c)
            st_stream(PO == F64C ? q + size_t(i) * 12 + 3 * w + c : q + size_t(3 * w + c) * vh + i, make_double2(o[c].re, o[c].im));
    }
    __syncthreads();   // the spins' stores come before what may replace them
    if (w == 0) {
        const int todo = site >= vh ? FX_DONE : slow ? FX_SLOW : again ? FX_CHECK : FX_DONE;
        if (__any_sync(0xffffffffu, todo != FX_DONE)) fx_again<PI, PX, PO, RECON, DAG, HASX>(A, i, verdict.e, todo);
    }
}

// Lattices up to this many sites per parity take the split hop: as many as
// three of its CTAs per SM hold at once (3 x 152 x 32).  Measured in a graph,
// Q_tm whole / split in us: 8^4 27 / 16, 8^3x16 29 / 19, 10^3x20 32 / 26,
// 12^3x16 (13,824 sites) 30 / 27, 14x14x10x16 (15,680) 29 / 37, 12^3x24 34 /
// 40, 16^4 40 / 56 (more warps, but each repeats the neighbour arithmetic and
// the sums cross shared memory); with 12-real links 43 / 35 and 40 / 49 on
// either side of the line.
#ifndef TM_FX_SPLIT_SITES
#define TM_FX_SPLIT_SITES 14592
#endif

template <int PI, int PR, int PX, int PO, int RECON, bool DAG, bool HASX>
static cudaError_t fx_launch(const FxArgs &A, cudaStream_t s)
{
    const unsigned vh = A.g.vh;
    const bool signs = A.g.anti[1] || A.g.anti[2] || A.g.anti[3];
    if (vh <= TM_FX_SPLIT_SITES) {
        static_assert(!(HASX && PO == FXF), "fx_stores takes the hop alone");
        auto kern = k_fx_hop_split<PI, PX, PO, RECON, DAG, HASX, true>;
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(fx_split_bytes<RECON>()));
        if (e != cudaSuccess) return e;
        kern<<<(vh + 31) / 32, FX_SPLIT, fx_split_bytes<RECON>(), s>>>(A);
    } else {
        auto kern = signs ? k_fx_hop<PI, PR, PX, PO, RECON, DAG, HASX, true> : k_fx_hop<PI, PR, PX, PO, RECON, DAG, HASX, false>;
        kern<<<(vh + FX_BLOCK - 1) / FX_BLOCK, FX_BLOCK, 0, s>>>(A);
    }
    return cudaGetLastError();
}

template <int RECON>
static cudaError_t launch_f64_fields(const tm_gauge *U, bool dag, int p, const void *in, void *out, const void *x, const Coef &k,
                          cudaStream_t s, const SiteMap &m)
{
    const FxArgs A(U->geom, m, k, p, U->fx, U->links, in, x, out, in);
    if (dag) return x ? fx_launch<F64, F64, F64, F64, RECON, true, true>(A, s) : fx_launch<F64, F64, F64, F64, RECON, true, false>(A, s);
    return x ? fx_launch<F64, F64, F64, F64, RECON, false, true>(A, s) : fx_launch<F64, F64, F64, F64, RECON, false, false>(A, s);
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
    auto args = [&](const void *input, const void *x, void *output, const void *exact) {
        return FxArgs(g, U->map, k, stage_b ? 0 : 1, U->fx, U->links, input, x, output, exact);
    };
    if (stage_b) return fx_launch<FXF, FXF, PI, PI, RECON, false, true>(args(tmp, in, out, tmp), s);
    if (g.vh <= TM_FX_SPLIT_SITES) return fx_launch<PI, PI, F64, FXF, RECON, false, false>(args(in, nullptr, tmp, in), s);
    void *even = static_cast<char *>(tmp) + align256(fx_field_bytes(g.vh));
    k_fx_field<PI><<<(g.vh + 127) / 128, 128, 0, s>>>(g.vh, in, even);
    return fx_launch<FXF, PI, F64, FXF, RECON, false, false>(args(even, nullptr, tmp, in), s);
}

cudaError_t launch_fx_qtm(const tm_gauge *U, bool canonical, bool stage_b, const void *in, void *tmp, void *out,
                          const Coef &k, cudaStream_t s)
{
    if (U->recon == 18) return canonical ? fx_qtm<F64C, 18>(U, stage_b, in, tmp, out, k, s) : fx_qtm<F64, 18>(U, stage_b, in, tmp, out, k, s);
    return canonical ? fx_qtm<F64C, 12>(U, stage_b, in, tmp, out, k, s) : fx_qtm<F64, 12>(U, stage_b, in, tmp, out, k, s);
}

}  // namespace twm

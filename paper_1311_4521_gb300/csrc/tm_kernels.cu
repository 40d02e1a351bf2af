// tm_kernels.cu -- hopping-matrix kernels with fused twisted-mass epilogues,
// and the layout conversions between the canonical complex-double layouts
// and the packed component-major storage.
#include "tm_internal.h"

namespace twm {

bool make_geom(const int dims[4], const int bc[4], Geom &g)
{
    for (int d = 0; d < 4; ++d)
        if (dims[d] < 2 || (dims[d] & 1)) return false;
    double V = double(dims[0]) * dims[1] * dims[2] * dims[3];
    if (V >= 2147483648.0) return false;
    g.lx = dims[0];
    g.ly = dims[1];
    g.lz = dims[2];
    g.lt = dims[3];
    g.hx = dims[0] / 2;
    g.vh = unsigned(V / 2);
    g.sy = unsigned(g.hx);
    g.sz = g.sy * unsigned(g.ly);
    g.st = g.sz * unsigned(g.lz);
    for (int m = 0; m < 4; ++m) g.anti[m] = bc ? (bc[m] < 0) : 0;
    geom_set_divisors(g);
    return true;
}

Coef coef_plain() { return Coef{1, 0, 1, 0, 0, 0, 0, 0}; }

Coef coef_qtm_a(double mut)
{
    double d = 1.0 / (1.0 + mut * mut);
    // (1 - i mut) / (1 + mut^2) on spins 0,1 and (1 + i mut) / (1 + mut^2) on spins 2,3
    return Coef{d, -mut * d, d, mut * d, 0, 0, 0, 0};
}

Coef coef_qtm_b(double kappa, double mut)
{
    double k2 = kappa * kappa;
    // upper: -k2 hop + (1 + i mut) x ; lower: -( -k2 hop + (1 - i mut) x )
    return Coef{-k2, 0, k2, 0, 1.0, mut, -1.0, mut};
}

// The same pair with -kappa^2 moved into the first launch: it writes
// -kappa^2 M_oo^-1 H_oe x, and the second launch adds the hop of that with
// the coefficients +1 (upper) and -1 (lower), a sign instead of a multiply.
Coef coef_qtm_a_scaled(double kappa, double mut)
{
    double d = -kappa * kappa / (1.0 + mut * mut);
    return Coef{d, -mut * d, d, mut * d, 0, 0, 0, 0};
}

Coef coef_qtm_b_unit(double mut)
{
    Coef c{1.0, 0, -1.0, 0, 1.0, mut, -1.0, mut};
    c.unit = 1;
    return c;
}

// ------------------------------------------------------------------ hop
template <int P, int RECON, bool DAG, bool HASX>
__global__ void __launch_bounds__(128, TM_HOP_MINB(P)) k_hop(Geom g, int p, const typename LinkIO<P, RECON>::V *__restrict__ links,
                                             const void *__restrict__ in, void *__restrict__ out,
                                             const void *__restrict__ x, Coef k, SiteMap m)
{
    using R = typename SpinorIO<P>::R;
    const unsigned i = map_site(g, m, blockIdx.x, threadIdx.x);
    if (i >= g.vh) return;
    Spinor<R> acc, o;
    hop_site<P, RECON, DAG>(g, p, i, links, in, acc);
    if (HASX) {
        Spinor<R> xs;
        if constexpr (P == F16) {   // the re-read input's site norm folded into its coefficients
            const R xn = SpinorIO<P>::load_raw(x, g.vh, i, xs);
            epilogue(k, acc, &xs, o, xn);
        } else {
            SpinorIO<P>::load(x, g.vh, i, xs);
            epilogue(k, acc, &xs, o);
        }
    } else {
        epilogue(k, acc, static_cast<const Spinor<R> *>(nullptr), o);
    }
    SpinorIO<P>::store(out, g.vh, i, o);
}

// The two Q_tm launches of tm_Qtm_host for FP64 handles without fixed-point
// links, on the caller's canonical layout: launch A (PI = F64C) gathers its input from it, launch B
// re-reads it as x (PX = F64C) and writes its result in it (PO = F64C); the
// odd temporary between them stays component-major.  The per-site
// arithmetic is the hop's, so results equal tm_Qtm's on packed fields.
template <int PI, int PX, int PO, int RECON, bool HASX>
__global__ void __launch_bounds__(128, TM_HOP_MINB(F64))
    k_hop_io(Geom g, int p, const typename LinkIO<F64, RECON>::V *__restrict__ links, const void *__restrict__ in,
             void *__restrict__ out, const void *__restrict__ x, Coef k, SiteMap m)
{
    const unsigned i = map_site(g, m, blockIdx.x, threadIdx.x);
    if (i >= g.vh) return;
    Nbrs n;
    neighbours(g, p, i, n);
    GlobalLinks<F64, RECON> src{links, g.vh, i, p};
    Spinor<double> acc, o;
    hop_site_src<PI, false>(g, n, src, in, acc);
    if (HASX) {
        Spinor<double> xs;
        SpinorIO<PX>::load(x, g.vh, i, xs);
        epilogue(k, acc, &xs, o);
    } else {
        epilogue(k, acc, static_cast<const Spinor<double> *>(nullptr), o);
    }
    SpinorIO<PO>::store(out, g.vh, i, o);
}

template <int RECON>
static cudaError_t qtm_canonical(bool stage_b, const Geom &g, const SiteMap &m, const void *links, const void *in,
                                 void *tmp, void *out, const Coef &k, cudaStream_t s)
{
    using V = typename LinkIO<F64, RECON>::V;
    const V *l = static_cast<const V *>(links);
    const unsigned grid = map_grid(g, m);
    if (!stage_b) k_hop_io<F64C, F64, F64, RECON, false><<<grid, m.block, 0, s>>>(g, 1, l, in, tmp, nullptr, k, m);
    else k_hop_io<F64, F64C, F64C, RECON, true><<<grid, m.block, 0, s>>>(g, 0, l, tmp, out, in, k, m);
    return cudaGetLastError();
}

cudaError_t launch_qtm(const tm_gauge *U, bool fx, bool canonical, bool stage_b, const void *in, void *tmp, void *out,
                       const Coef &k, cudaStream_t s)
{
    const Geom &g = U->geom;
    if (g.vh == 0) return cudaSuccess;
    if (fx) return launch_fx_qtm(U, canonical, stage_b, in, tmp, out, k, s);
    if (!canonical) {
        return stage_b ? launch_hop(U, false, TM_EO, tmp, out, in, k, s) : launch_hop(U, false, TM_OE, in, tmp, nullptr, k, s);
    }
    if (U->recon == 18) return qtm_canonical<18>(stage_b, g, U->map, U->links, in, tmp, out, k, s);
    return qtm_canonical<12>(stage_b, g, U->map, U->links, in, tmp, out, k, s);
}

// The double-float hop with the 8 hops of a site dealt out to four warps, one
// direction each, for lattices whose sites do not fill the GPU: a CTA covers
// 32 sites.  A thread's 8 hops are a chain of some 27 us however few sites
// there are.  The warps' partial sums meet in shared memory, are added in the
// order of the directions, and warp w finishes spin w.  The site map is not
// used (results do not depend on it).
template <int RECON, bool DAG, bool HASX>
__global__ void __launch_bounds__(128, TM_HOP_MINB(F64X))
    k_hop_split(Geom g, int p, const typename LinkIO<F64X, RECON>::V *__restrict__ links, const void *__restrict__ in,
                void *__restrict__ out, const void *__restrict__ x, Coef k)
{
    __shared__ float4 part[12][128];   // [component][direction, site]
    const unsigned lane = threadIdx.x & 31, w = threadIdx.x >> 5, site = blockIdx.x * 32 + lane, i = min(site, g.vh - 1);
    float4 xv[3];   // spin w of the re-read input
    if (HASX)
#pragma unroll
        for (int c = 0; c < 3; ++c) xv[c] = ld_keep(static_cast<const float4 *>(x) + size_t(3 * w + c) * g.vh + i);
    {
        Nbrs n;
        neighbours(g, p, i, n);
        const GlobalLinks<F64X, RECON> src{links, g.vh, i, p};
        Spinor<dd> acc;
#pragma unroll
        for (int c = 0; c < 12; ++c) acc[c / 3][c % 3] = {dd(0.f), dd(0.f)};
        // one loop for all warps: four copies of it, one per direction, overflowed the
        // instruction cache (12^3x24, Q_tm: 86 us against 53)
        hop_site_rolled<F64X, DAG>(g, n, src, in, acc, int(2 * w), int(2 * w + 2));
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const cpx<dd> a = acc[c / 3][c % 3];
            part[c][threadIdx.x] = make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo);
        }
    }
    __syncthreads();
    if (site >= g.vh) return;
    const dd z(0.f);
    const int h = w < 2 ? 0 : 2;
    const cpx<dd> a = {k.get(h, z), k.get(h + 1, z)}, b = {k.get(h + 4, z), k.get(h + 5, z)};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        cpx<dd> hop = {z, z};
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const float4 q = part[3 * w + c][32 * v + lane];
            hop = hop + cpx<dd>{dd{q.x, q.y}, dd{q.z, q.w}};
        }
        cpx<dd> o = k.unit ? (w < 2 ? hop : -hop) : a * hop;
        if (HASX) o = cmadd(b, cpx<dd>{dd{xv[c].x, xv[c].y}, dd{xv[c].z, xv[c].w}}, o);
        st_stream(static_cast<float4 *>(out) + size_t(3 * w + c) * g.vh + i, make_float4(o.re.hi, o.re.lo, o.im.hi, o.im.lo));
    }
}

// Lattices that take it: up to 16000 sites per parity, and for 18-real links
// from the second wave of the whole hop (more than 2 x 152 CTAs of 128) to
// 160000.  In a graph, Q_tm whole / split in us, 18-real and 12-real links
// (whose warps each rebuild the rows they need): 8^4 51 / 17 and 70 / 25;
// 13,824 sites 50 / 21 and 65 / 33; 15,680 51 / 37 and 65 / 62; 17,280 52 / 38
// and 66 / 65 with the hop at 29.4 / 31.4; 40,960 65 / 58 and 76 / 107;
// 128,000 185 / 163; 160,000 210 / 204; 221,184 272 / 274.  Between the two
// ranges the whole hop is one wave of 24 to 26 us, and the split one ahead of
// it in a graph (20,736: 25 / 18) but not in turn with other launches:
// 12^3x24 and the unpacking of its result, one call after another, 36.9 on
// every run against 30, 37 and 41.
inline bool f64x_split(int recon, unsigned vh)
{
    return vh <= 16000 || (recon == 18 && vh > 2 * 152 * 128 && vh <= 160000);
}

template <int RECON>
static cudaError_t hop_split(const Geom &g, bool dag, int p, const void *links, const void *in, void *out, const void *x,
                             const Coef &k, cudaStream_t s)
{
    auto kern = dag ? (x ? k_hop_split<RECON, true, true> : k_hop_split<RECON, true, false>)
                    : (x ? k_hop_split<RECON, false, true> : k_hop_split<RECON, false, false>);
    kern<<<(g.vh + 31) / 32, 128, 0, s>>>(g, p, static_cast<const typename LinkIO<F64X, RECON>::V *>(links), in, out, x, k);
    return cudaGetLastError();
}

template <int P, int RECON>
static cudaError_t hop_dispatch(const Geom &g, bool dag, int p, const void *links, const void *in, void *out,
                                const void *x, const Coef &k, cudaStream_t s, const SiteMap &m)
{
    using V = typename LinkIO<P, RECON>::V;
    if constexpr (P == F64X)
        if (f64x_split(RECON, g.vh)) return hop_split<RECON>(g, dag, p, links, in, out, x, k, s);
    const V *l = static_cast<const V *>(links);
    const unsigned grid = map_grid(g, m);
    auto kern = dag ? (x ? k_hop<P, RECON, true, true> : k_hop<P, RECON, true, false>)
                    : (x ? k_hop<P, RECON, false, true> : k_hop<P, RECON, false, false>);
    kern<<<grid, m.block, 0, s>>>(g, p, l, in, out, x, k, m);
    return cudaGetLastError();
}

cudaError_t launch_hop(const tm_gauge *U, bool dag, int out_parity, const void *in, void *out, const void *x,
                       const Coef &k, cudaStream_t s, const SiteMap &m)
{
    const Geom &g = U->geom;
    if (g.vh == 0) return cudaSuccess;
    if (U->fx) return launch_fx_hop(U, dag, out_parity, in, out, x, k, s, m);
    const void *l = U->links;
    switch (U->prec * 100 + U->recon) {
    case F64 * 100 + 18: return hop_dispatch<F64, 18>(g, dag, out_parity, l, in, out, x, k, s, m);
    case F64 * 100 + 12: return hop_dispatch<F64, 12>(g, dag, out_parity, l, in, out, x, k, s, m);
    case F32 * 100 + 18: return hop_dispatch<F32, 18>(g, dag, out_parity, l, in, out, x, k, s, m);
    case F32 * 100 + 12: return hop_dispatch<F32, 12>(g, dag, out_parity, l, in, out, x, k, s, m);
    case F16 * 100 + 12: return hop_dispatch<F16, 12>(g, dag, out_parity, l, in, out, x, k, s, m);
    case F64X * 100 + 18: return hop_dispatch<F64X, 18>(g, dag, out_parity, l, in, out, x, k, s, m);
    case F64X * 100 + 12: return hop_dispatch<F64X, 12>(g, dag, out_parity, l, in, out, x, k, s, m);
    }
    return cudaErrorInvalidValue;
}

// ------------------------------------------------------------------ layouts
int link_nchunk(int prec, int recon)
{
    if (prec == F64 || prec == F64X) return recon == 18 ? 9 : 6;
    if (prec == F32) return recon == 18 ? 9 : 3;
    if (prec == F16 && recon == 12) return 3;
    return 0;
}

size_t link_chunk_bytes(int prec, int recon)
{
    if (prec == F64 || prec == F64X) return 16;
    if (prec == F32) return recon == 18 ? 8 : 16;
    if (prec == F16) return 8;
    return 0;
}

// One thread per (mu, lexicographic site) of the canonical U[mu][lex][3][3].
template <int P, int RECON>
__global__ void k_pack_gauge(Geom g, const double *__restrict__ U, typename LinkIO<P, RECON>::V *links)
{
    unsigned long long idx = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    unsigned long long V = 2ull * g.vh;
    if (idx >= 4 * V) return;
    int mu = int(idx / V);
    unsigned lex = unsigned(idx % V);
    unsigned x = lex % g.lx, r = lex / g.lx;
    unsigned y = r % g.ly;
    r /= g.ly;
    unsigned z = r % g.lz, t = r / g.lz;
    int p = (x + y + z + t) & 1;
    double m[18];
    for (int k = 0; k < 18; ++k) m[k] = U[idx * 18 + k];
    using L = LinkIO<P, RECON>;
    L::store(links + size_t(4 * p + mu) * L::NCHUNK * g.vh, g.vh, lex >> 1, m);
}

cudaError_t launch_pack_gauge(const Geom &g, int prec, int recon, const double *U, void *links, cudaStream_t s)
{
    unsigned long long n = 8ull * g.vh;
    unsigned grid = unsigned((n + 255) / 256);
#define TM_PACK(P, RC)                                                                                   \
    if (prec == P && recon == RC) {                                                                      \
        k_pack_gauge<P, RC><<<grid, 256, 0, s>>>(g, U, static_cast<typename LinkIO<P, RC>::V *>(links)); \
        return cudaGetLastError();                                                                       \
    }
    TM_PACK(F64, 18)
    TM_PACK(F64, 12)
    TM_PACK(F32, 18)
    TM_PACK(F32, 12)
    TM_PACK(F16, 12)
    TM_PACK(F64X, 18)
    TM_PACK(F64X, 12)
#undef TM_PACK
    return cudaErrorInvalidValue;
}

// Between the canonical layout (192 contiguous bytes per site) and the packed
// one, a CTA takes 64 sites through shared memory, so that both sides of the
// copy are coalesced.  Measured on 1,048,576 sites, FP32: pack 65 -> 59 us,
// unpack 187 -> 51 us, 5.9 TB/s (a thread per site used to write 16 bytes
// every 192, and to convert with the FP64 pipe).
constexpr int LB = 64, LS = 13;   // sites per CTA; stride of a staged site in 16-byte words (odd: no bank conflicts)

template <int P>
__global__ void __launch_bounds__(LB) k_pack_spinor(unsigned vh, const double *__restrict__ in, void *out)
{
    using R = typename SpinorIO<P>::R;
    __shared__ double2 stage[LB * LS];
    const unsigned i0 = blockIdx.x * LB, n = min(unsigned(LB), vh - i0), i = i0 + threadIdx.x;
    const double2 *src = reinterpret_cast<const double2 *>(in) + size_t(i0) * 12;
    for (unsigned k = threadIdx.x; k < 12 * n; k += LB) stage[k / 12 * LS + k % 12] = ld_stream(src + k);
    __syncthreads();
    if (i >= vh) return;
    Spinor<R> s;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const double2 v = stage[threadIdx.x * LS + c];
        s[c / 3][c % 3] = {to_R<R>(v.x), to_R<R>(v.y)};
    }
    SpinorIO<P>::store(out, vh, i, s);
}

template <int P>
__global__ void __launch_bounds__(LB) k_unpack_spinor(unsigned vh, const void *in, double *__restrict__ out)
{
    using R = typename SpinorIO<P>::R;
    __shared__ double2 stage[LB * LS];
    const unsigned i0 = blockIdx.x * LB, n = min(unsigned(LB), vh - i0), i = i0 + threadIdx.x;
    if (i < vh) {
        Spinor<R> s;
        SpinorIO<P>::load(in, vh, i, s);
#pragma unroll
        for (int c = 0; c < 12; ++c) stage[threadIdx.x * LS + c] = make_double2(widen(s[c / 3][c % 3].re), widen(s[c / 3][c % 3].im));
    }
    __syncthreads();
    double2 *dst = reinterpret_cast<double2 *>(out) + size_t(i0) * 12;
    for (unsigned k = threadIdx.x; k < 12 * n; k += LB) st_stream(dst + k, stage[k / 12 * LS + k % 12]);
}

cudaError_t launch_pack_spinor(unsigned vh, int prec, const double *in, void *out, cudaStream_t s)
{
    if (vh == 0) return cudaSuccess;
    unsigned grid = (vh + LB - 1) / LB;
    if (prec == F64) k_pack_spinor<F64><<<grid, LB, 0, s>>>(vh, in, out);
    else if (prec == F64X) k_pack_spinor<F64X><<<grid, LB, 0, s>>>(vh, in, out);
    else if (prec == F32) k_pack_spinor<F32><<<grid, LB, 0, s>>>(vh, in, out);
    else if (prec == F16) k_pack_spinor<F16><<<grid, LB, 0, s>>>(vh, in, out);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_unpack_spinor(unsigned vh, int prec, const void *in, double *out, cudaStream_t s)
{
    if (vh == 0) return cudaSuccess;
    unsigned grid = (vh + LB - 1) / LB;
    if (prec == F64) k_unpack_spinor<F64><<<grid, LB, 0, s>>>(vh, in, out);
    else if (prec == F64X) k_unpack_spinor<F64X><<<grid, LB, 0, s>>>(vh, in, out);
    else if (prec == F32) k_unpack_spinor<F32><<<grid, LB, 0, s>>>(vh, in, out);
    else if (prec == F16) k_unpack_spinor<F16><<<grid, LB, 0, s>>>(vh, in, out);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

}  // namespace twm

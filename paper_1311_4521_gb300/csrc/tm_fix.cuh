// tm_fix.cuh -- the FP64 hop with its link products in fixed point.
//
// The FP64 units issue 2 lanes per SM and clock here, the integer ones 32
// lanes of a 32 x 32 -> 64 bit multiply-add (measured: 4.1 cycles per warp
// and scheduler), and the link multiplies are 576 of the 840 FP64
// instructions of a site.  So they are done in integers: a hop's projected
// half-spinor becomes 12 numbers of 58 bits under a common exponent, the
// links are kept a second time as 58-bit fractions, and a real product is
// three multiply-adds of 29-bit limbs (the product of the low limbs, below
// 2^-58 of the largest, is left out).  The 8 hops are summed in 64-bit
// integers and converted to FP64 once; the epilogue stays in FP64.
//
// Precision: everything is held to a unit eta, 2^-57 of the largest component
// (as a power of two) that enters a site, where FP64 rounds every product and
// sum to 2^-53 of itself.  Links, stored fields and partial sums are rounded
// to nearest and low limbs are balanced, so that a component's hop is off by
// 1.44 eta rms (5.0 with truncation; against exact integers, random links).
// That is no more than FP64's own error of 0.34 2^-53 S rms, S the sum of the
// absolute products that enter the component, where S >= FX_LEAST 2^48 eta.
// Every hop adds up the |U h| of its 8 directions, which S is at least: a
// site with a component below that is looked at again (fx_again), with S
// itself, and computed with FP64 products from the FP64 input if it is so.
// So are sites with neighbours that are not finite or near the ends of the
// exponent range, and a gauge field with a link outside fx_link_ok.  Measured
// against 64-bit and longer arithmetic, Q_tm is off by 1.2e-16 (1.3e-16 with
// FP64 products).
//
// Measured (32^3x64, 18-real links, against FP64 products): Q_tm 3.04 -> 0.78
// ms, one hop 1.52 -> 0.49 ms; 8^4, split over warps: Q_tm 65 -> 19 us.
// What it took beyond the integers (Q_tm at 32^3x64): multiply-adds from
// plain C, not inline PTX 1.36 -> 1.02 ms; neighbours and links staged by
// cp.async one hop ahead, 12 warps per SM, 0.87; the fallback called with
// few words instead of with the site's sum 0.80.
#pragma once

#include <cmath>

#include "tm_device.cuh"

namespace twm {

constexpr int FX_LIMB = 29;            // bits of a limb
// Least sum of absolute products of a component, in units of 2^48 eta (512
// make the largest input component): 1.44 eta / (0.34 2^-53) = 136 of them.
// (Links that do not mix colours: 0.93 eta and 0.54, 55 of them.)
constexpr int FX_LEAST = 136;
// Least such sum, times the output's coefficient, of a component of an output
// that is stored in fixed point, relative to the power of two above the
// largest: rounding to 57 bits (0.29 units) against 0.35 2^-53 S.
constexpr float FX_LEAST_STORED = 0.052f;
constexpr unsigned FX_FMIN = 200, FX_FMAX = 1850;  // biased exponents taken here

// A spinor field of the library's own (the odd temporary of Q_tm) in fixed
// point: blocks of 32 sites, each 12 arrays of 32 int4 (re.hi, re.lo, im.hi,
// im.lo) so that a site's loads share one address and differ by constants,
// then a word per site with e in its lower half: component = (hi 2^29 + lo)
// 2^(e - 57), -2^28 <= lo <= 2^28, e the smallest exponent with every
// |component| < 2^e.  A site that does not fit, or whose small components
// would lose more than FP64 arithmetic gave them, holds its FP64 bits and the
// word FX_RAW.  (One array per component over all sites instead cost two
// 64-bit additions per load: 3800 against 4400 instructions a site.)
constexpr int FX_FIELD = 57, FX_HALF = 58;   // fraction bits of field components and of projected half-spinors
constexpr int FX_RAW = 0x7fffffff, FX_ZERO_E = -4000;
constexpr int FX_LOWEST_E = -5000;   // below FX_ZERO_E: a sum that has met nothing but zeros
constexpr unsigned FX_SPINOR_BLOCK = 12 * 32 * 16;
constexpr unsigned fx_link_block(int recon) { return 4 * (recon / 2) * 32 * 16; }   // 32 sites' links of 4 directions
TM_HD unsigned fx_blocks(unsigned vh) { return (vh + 31) / 32; }
TM_HD size_t fx_field_bytes(unsigned vh) { return size_t(FX_SPINOR_BLOCK + 128) * fx_blocks(vh); }
TM_HD size_t fx_link_bytes(unsigned vh, int recon) { return 2 * size_t(fx_link_block(recon)) * fx_blocks(vh); }
// Entry of site j in its block (of `block` bytes).
template <typename T> TM_HD T *fx_entry(T *base, unsigned block, unsigned j)
{
    return base + size_t(j >> 5) * (block / unsigned(sizeof(T))) + (j & 31u);
}

// One link entry as limbs: value = (hi 2^29 + lo) 2^-58, -2^28 <= lo <= 2^28;
// re in x, y and im in z, w.
typedef int4 FxEntry;

#if defined(__CUDACC__)

// acc + a b, 32 x 32 -> 64 bit: one multiply-add.  (As inline PTX the same
// sums were compiled to products and separate 64-bit additions: 5683
// against 3861 instructions a site, 1.36 against 1.02 ms for Q_tm at 32^3x64.)
__device__ __forceinline__ unsigned long long fx_mad(int a, int b, unsigned long long acc)
{
    return acc + (unsigned long long)((long long)a * b);
}
// arithmetic shift; amounts above 63 leave the sign
__device__ __forceinline__ long long fx_sar(long long v, int s)
{
    asm("shr.s64 %0, %0, %1;" : "+l"(v) : "r"(s));
    return v;
}

// The limbs of v (times -1 if nm is all ones): its mantissa with the leading
// bit at the top of 64 bits, shifted right by `from` less its biased exponent
// (and 3 more for the low limb).  The shifts saturate, so zeros and numbers
// far below the reference vanish.
__device__ __forceinline__ void fx_split(double v, unsigned from, unsigned nm, int &hi, int &lo)
{
    const unsigned hw = unsigned(__double2hiint(v)), lw = unsigned(__double2loint(v));
    const unsigned th = __funnelshift_l(lw, hw, 11) | 0x80000000u, tl = lw << 11;
    const unsigned s = from - ((hw >> 20) & 0x7ffu);
    unsigned mh, ml;
    asm("shr.u32 %0, %1, %2;" : "=r"(mh) : "r"(th), "r"(s));
    asm("{ .reg .b64 t; .reg .b32 d; mov.b64 t, {%1, %2}; shr.u64 t, t, %3; mov.b64 {%0, d}, t; }"
        : "=r"(ml) : "r"(tl), "r"(th), "r"(s + 3u));
    const int sg = int((unsigned(int(hw) >> 31) ^ nm) | 1u);
    hi = int(mh) * sg;
    lo = int(ml & 0x1fffffffu) * sg;
}

// The same to nearest, with a low limb between -2^28 and 2^28.
__device__ __forceinline__ void fx_split_near(double v, unsigned from, int &hi, int &lo)
{
    const unsigned hw = unsigned(__double2hiint(v)), lw = unsigned(__double2loint(v));
    const unsigned th = __funnelshift_l(lw, hw, 11) | 0x80000000u, tl = lw << 11;
    unsigned long long m;
    asm("{ .reg .b64 t; mov.b64 t, {%1, %2}; shr.u64 %0, t, %3; }" : "=l"(m) : "r"(tl), "r"(th), "r"(from + 2u - ((hw >> 20) & 0x7ffu)));
    m = ((m + 1) >> 1) + (1u << (FX_LIMB - 1));
    const int sg = int(unsigned(int(hw) >> 31) | 1u);
    hi = int(m >> FX_LIMB) * sg;
    lo = (int(unsigned(m) & ((1u << FX_LIMB) - 1)) - (1 << (FX_LIMB - 1))) * sg;
}

// v 2^(e - bits) in FP64
__device__ __forceinline__ double fx_to_double(long long v, int e, int bits)
{
    const double d = __ll2double_rn(v);
    const int add = v ? (e - bits) << 20 : 0;
    return __hiloint2double(__double2hiint(d) + add, __double2loint(d));
}

__device__ __forceinline__ const int *fx_words(const void *base, unsigned vh)
{
    return reinterpret_cast<const int *>(static_cast<const char *>(base) + size_t(FX_SPINOR_BLOCK) * fx_blocks(vh));
}

// Adds a component's high words without sign to a site's largest, and all its bits but signs.
__device__ __forceinline__ void fx_range_of(const cpx<double> &v, unsigned &m, unsigned &bits)
{
    const unsigned p = unsigned(__double2hiint(v.re)) & 0x7fffffffu, q = unsigned(__double2hiint(v.im)) & 0x7fffffffu;
    m = max(m, max(p, q));
    bits |= p | q | unsigned(__double2loint(v.re)) | unsigned(__double2loint(v.im));
}

// How a site is stored in a fixed-point field, from the range of its 12 components.
struct FxSite {
    bool raw;
    int e;
    unsigned from;
    __device__ __forceinline__ FxSite(unsigned m, unsigned bits)
    {
        const bool zero = bits == 0;
        const unsigned f = m >> 20;
        raw = !zero && (f < FX_FMIN || f > FX_FMAX);
        e = zero ? FX_ZERO_E : int(f) - 1022;
        from = zero ? 8000u : f + 4u;
    }
    __device__ __forceinline__ void store(void *base, unsigned i, int c, const cpx<double> &v) const
    {
        int4 o;
        fx_split_near(v.re, from, o.x, o.y);
        fx_split_near(v.im, from, o.z, o.w);
        if (raw) o = make_int4(__double2hiint(v.re), __double2loint(v.re), __double2hiint(v.im), __double2loint(v.im));
        st_stream(fx_entry(static_cast<int4 *>(base), FX_SPINOR_BLOCK, i) + 32 * c, o);
    }
    __device__ __forceinline__ void store_word(void *base, unsigned vh, unsigned i) const
    {
        st_stream(const_cast<int *>(fx_words(base, vh)) + i, raw ? FX_RAW : e & 0xffff);
    }
};

// A stored component of a site with word `word`, in FP64.
__device__ __forceinline__ cpx<double> fx_component(const int4 &v, int word)
{
    if (word == FX_RAW) return {__hiloint2double(v.x, v.y), __hiloint2double(v.z, v.w)};
    const int e = int(short(word & 0xffff));
    return {fx_to_double(((long long)v.x << FX_LIMB) + v.y, e, FX_FIELD),
            fx_to_double(((long long)v.z << FX_LIMB) + v.w, e, FX_FIELD)};
}

// Fixed-point fields read and written as FP64 sites.
template <> struct SpinorIO<FXF> {
    using R = double;
    __device__ static R load_raw(const void *base, unsigned vh, unsigned i, Spinor<R> &s)
    {
        const int4 *b = fx_entry(static_cast<const int4 *>(base), FX_SPINOR_BLOCK, i);
        const int word = fx_words(base, vh)[i];
#pragma unroll
        for (int c = 0; c < 12; ++c) s[c / 3][c % 3] = fx_component(b[32 * c], word);
        return R(1);
    }
    __device__ static void load(const void *base, unsigned vh, unsigned i, Spinor<R> &s) { load_raw(base, vh, i, s); }
    __device__ __forceinline__ static void store(void *base, unsigned vh, unsigned i, const Spinor<R> &s)
    {
        store_as(base, vh, i, s, false);
    }
    // The same, in FP64 bits if raw is set; returns how it was stored.
    __device__ __forceinline__ static FxSite store_as(void *base, unsigned vh, unsigned i, const Spinor<R> &s, bool raw)
    {
        unsigned m = 0, bits = 0;
#pragma unroll
        for (int c = 0; c < 12; ++c) fx_range_of(s[c / 3][c % 3], m, bits);
        FxSite f(m, bits);
        f.raw = f.raw || raw;
#pragma unroll
        for (int c = 0; c < 12; ++c) f.store(base, i, c, s[c / 3][c % 3]);
        f.store_word(base, vh, i);
        return f;
    }
};

// A site's sum: 64-bit integers in units of 2^(e - bits).
struct FxSum {
    long long re[4][3], im[4][3];
    int e;
    __device__ __forceinline__ void clear(int exponent)
    {
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int c = 0; c < 3; ++c) re[s][c] = im[s][c] = 0;
        e = exponent;
    }
};
// Two 16-bit sums, 2^s of the old units to a new one.
__device__ __forceinline__ unsigned fx_size_sar(unsigned v, int s)
{
    return s > 15 ? 0u : (v >> s) & ((0xffffu >> s) * 0x10001u);
}
// A site's sums of absolute values: per component those of the 8 hops in
// units of 2^48 of the sum's, re in the lower and im in the upper half of a
// word (a hop is below 2^59.4, so that a half holds the sum of 8).  They live
// in shared memory, 12 words of each thread: in registers they made the hop
// spill 200 to 350 bytes.
template <int BLOCK> struct FxSizes {
    unsigned at;   // shared-memory address of this thread's first word
    __device__ __forceinline__ explicit FxSizes(unsigned *words)
        : at(unsigned(__cvta_generic_to_shared(words + threadIdx.x)))
    {
#pragma unroll
        for (int c = 0; c < 12; ++c) set(c, 0u);
    }
    __device__ __forceinline__ void set(int c, unsigned v) const { asm volatile("st.shared.u32 [%0], %1;" ::"r"(at + 4 * BLOCK * c), "r"(v)); }
    __device__ __forceinline__ unsigned get(int c) const
    {
        unsigned v;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at + 4 * BLOCK * c));
        return v;
    }
    __device__ __forceinline__ void add(int c, unsigned v) const { asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(at + 4 * BLOCK * c), "r"(v)); }
    __device__ __forceinline__ void sar(int s) const
    {
// a loop: unrolled, the FP64 hop on 12-real links outgrew the instruction cache (0.93 against 0.85 ms at 32^3x64)
#pragma unroll 1
        for (int c = 0; c < 12; ++c) set(c, fx_size_sar(get(c), s));
    }
    __device__ __forceinline__ int least() const
    {
        unsigned m = get(0);
#pragma unroll
        for (int c = 1; c < 12; ++c) m = __vminu2(m, get(c));
        return int(min(m & 0xffffu, m >> 16));
    }
};

// A projected half-spinor as limbs (in units that the sum's exponent fixes).
struct FxHalf {
    int hi[2][3][2], lo[2][3][2];
};

// Adds (r, S A_mu^dag r) for one component r of the upper spin s: the lower
// spin that it feeds, times +-1 or +-i, as in accumulate().
template <int MU, int S, class Sizes>
__device__ __forceinline__ void fx_accumulate(int s, int c, long long re, long long im, FxSum &t, const Sizes &sizes)
{
    // the upper 16 bits of both absolute values (less one where negative)
    unsigned size, signs;
    asm("prmt.b32 %0, %1, %2, 0x7632;" : "=r"(size) : "r"(int(re >> 32)), "r"(int(im >> 32)));
    asm("prmt.b32 %0, %1, %1, 0xbb99;" : "=r"(signs) : "r"(size));
    size ^= signs;
    sizes.add(3 * s + c, size);
    sizes.add(3 * (2 + ((MU == 0 || MU == 3) ? s : 1 - s)) + c, (MU == 1 || MU == 3) ? __funnelshift_l(size, size, 16) : size);
    t.re[s][c] += re;
    t.im[s][c] += im;
    // lower spin 2 + k and its factor: MU 0: -s h_k; 1: s i h_(1-k); 2: s h1, -s h0; 3: s i h0, -s i h1
    const int k = (MU == 0 || MU == 3) ? s : 1 - s;
    const bool times_i = MU == 1 || MU == 3;
    bool minus = S < 0;
    if (MU == 0) minus = !minus;
    if (MU == 2 && s == 0) minus = !minus;
    if (MU == 3 && s == 1) minus = !minus;
    const long long a = times_i ? im : re, b = times_i ? re : im;   // i r = (-im, re)
    if (minus != times_i) t.re[2 + k][c] -= a;
    else t.re[2 + k][c] += a;
    if (minus) t.im[2 + k][c] -= b;
    else t.im[2 + k][c] += b;
}

// The fixed-point links: per origin parity blocks of 32 sites, each with one
// FxEntry array of 32 for every direction and stored complex entry.
template <int RECON> struct FxLinks {
    const FxEntry *links;
    unsigned vh, i;
    int p;
    template <int MU, bool FWD> __device__ __forceinline__ const FxEntry *at(const Nbrs &n) const
    {
        constexpr unsigned blk = fx_link_block(RECON);
        const FxEntry *b = links + size_t(FWD ? p : 1 - p) * fx_blocks(vh) * (blk / 16);
        return fx_entry(b, blk, FWD ? i : n.bwd[MU]) + MU * (RECON / 2) * 32;
    }
};

// One component of conj(row0 x row1): conj(a d - b c), as limbs.
__device__ __forceinline__ FxEntry fx_minor(const FxEntry &a, const FxEntry &d, const FxEntry &b, const FxEntry &c)
{
    unsigned long long hr = 0, mr = 1u << (FX_LIMB - 1), hi = 0, mi = 1u << (FX_LIMB - 1);   // rounded to nearest
    // re = a.re d.re - a.im d.im - b.re c.re + b.im c.im ; im = -(a.re d.im + a.im d.re - b.re c.im - b.im c.re)
    auto put = [](int xh, int xl, int yh, int yl, unsigned long long &h, unsigned long long &m) {
        h = fx_mad(xh, yh, h);
        m = fx_mad(xh, yl, m);
        m = fx_mad(xl, yh, m);
    };
    put(a.x, a.y, d.x, d.y, hr, mr);
    put(-a.z, -a.w, d.z, d.w, hr, mr);
    put(-b.x, -b.y, c.x, c.y, hr, mr);
    put(b.z, b.w, c.z, c.w, hr, mr);
    put(-a.x, -a.y, d.z, d.w, hi, mi);
    put(-a.z, -a.w, d.x, d.y, hi, mi);
    put(b.x, b.y, c.z, c.w, hi, mi);
    put(b.z, b.w, c.x, c.y, hi, mi);
    const long long re = (long long)hr + ((long long)mr >> FX_LIMB), im = (long long)hi + ((long long)mi >> FX_LIMB);
    FxEntry r;
    r.x = int((re + (1 << (FX_LIMB - 1))) >> FX_LIMB);
    r.y = int(re) - int(unsigned(r.x) << FX_LIMB);
    r.z = int((im + (1 << (FX_LIMB - 1))) >> FX_LIMB);
    r.w = int(im) - int(unsigned(r.z) << FX_LIMB);
    return r;
}

// Whether a link (as limbs, each component below 1 + 2^-20) can be used: every
// row's and column's sum of |re| + |im| at most 2.5 (sqrt(6) bounds it for a
// unitary matrix), which bounds a hop's product with a half-spinor below 2^58
// by 2.5 * 2^58 and the sum of the 8 by 1.25 * 2^62 < 2^63, and its largest
// component at least 1/16, or all of them zero (`zero`, by the bits of the
// entries: limbs are zero below 2^-58 too).
__device__ __forceinline__ bool fx_link_ok(const FxEntry (&u)[9], bool zero)
{
    constexpr int most = int(2.5 * (1 << FX_LIMB));   // limbs are below 2^30, so three entries sum below 2^32.6
    bool ok = true;
    int big = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        unsigned row = 0, col = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const FxEntry r = u[3 * a + b], c = u[3 * b + a];
            row += unsigned(abs(r.x) + abs(r.z)) >> 1;
            col += unsigned(abs(c.x) + abs(c.z)) >> 1;
            big = max(big, max(abs(r.x), abs(r.z)));
        }
        ok = ok && row <= unsigned(most) / 2 && col <= unsigned(most) / 2;
    }
    return ok && (big >= 1 << (FX_LIMB - 4) || zero);
}

// Staging of a hop's data: every thread copies its own neighbour site (12
// 16-byte words) and link (RECON / 2 words) to its own slots of shared
// memory with cp.async, one hop ahead of the arithmetic, so that the loads
// in flight take no registers and no thread waits for another.  The site's
// words are read into registers (projected) before the next hop's copies
// start, so they need one slot; the links need two.
constexpr int FX_BLOCK = 64;   // threads per CTA of the fixed-point hops
template <int RECON_, int BLOCK_ = FX_BLOCK> struct FxStage {
    static constexpr int RECON = RECON_, BLOCK = BLOCK_, NL = RECON / 2, WORDS = 12 + 2 * NL;
    int4 *slot;   // this thread's first word; word w at slot[w * BLOCK]
    __device__ __forceinline__ int4 spinor(int c) const { return slot[c * BLOCK]; }
    // the staged FP64 site
    __device__ __forceinline__ void site(Spinor<double> &s) const
    {
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const int4 v = spinor(c);
            s[c / 3][c % 3] = {__hiloint2double(v.y, v.x), __hiloint2double(v.w, v.z)};
        }
    }
    __device__ __forceinline__ int4 link(int q, int k) const { return slot[(12 + q * NL + k) * BLOCK]; }
    __device__ __forceinline__ void copy(int w, const void *src) const
    {
        const unsigned dst = unsigned(__cvta_generic_to_shared(slot + w * BLOCK));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    }
    // Starts the copies of one hop, the link into slot q: the words of the
    // site at s (sstride apart) and of the link at u.
    __device__ __forceinline__ void start(int q, const int4 *s, size_t sstride, const FxEntry *u) const
    {
#pragma unroll
        for (int c = 0; c < 12; ++c) copy(c, s + c * sstride);
#pragma unroll
        for (int k = 0; k < NL; ++k) copy(12 + q * NL + k, u + 32 * k);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    __device__ __forceinline__ void start_site(const int4 *s, size_t sstride) const
    {
#pragma unroll
        for (int c = 0; c < 12; ++c) copy(c, s + c * sstride);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    __device__ __forceinline__ void wait() const { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
};

// The link product of direction MU on x, aligned to the sum by a right shift
// of d, added to the sum.  A 32 x 32 -> 64 bit multiply-add takes 4 issue
// cycles of a scheduler, an addition 2 on another pipe, so complex products
// use three real ones: with w = ur + ui (ur - ui for the conjugate link of a
// backward hop) and K = w hr,
//     re = K -+ ui (hr + hi),   im = K + ur (hi - hr).
// Per sum the products with one low limb come first; shifted by a limb they
// join the sum of the high ones.  Both sums start from half of what their
// shift drops, which rounds to nearest at no cost; less one in every other
// hop, so that ties go up and down alike.  Intermediate sums may wrap, results
// do not.
template <int MU, int S, bool FWD, bool ALIGN, class Stage>
__device__ __forceinline__ void fx_apply(const Stage &st, int q, const FxHalf &x, int d, FxSum &t, const FxSizes<Stage::BLOCK> &sizes)
{
    const unsigned long long half = ALIGN ? ((1ull << d) - (FWD ? 1u : 0u)) >> 1 : 0ull;
    int sh[2][3], sl[2][3], dh[2][3], dl[2][3];   // -+(hr + hi) and hi - hr
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            sh[s][c] = FWD ? -x.hi[s][c][0] - x.hi[s][c][1] : x.hi[s][c][0] + x.hi[s][c][1];
            sl[s][c] = FWD ? -x.lo[s][c][0] - x.lo[s][c][1] : x.lo[s][c][0] + x.lo[s][c][1];
            dh[s][c] = x.hi[s][c][1] - x.hi[s][c][0];
            dl[s][c] = x.lo[s][c][1] - x.lo[s][c][0];
        }
    constexpr int RECON = Stage::RECON;
    FxEntry full[RECON == 12 ? 9 : 1];
    if constexpr (RECON == 12) {
#pragma unroll
        for (int k = 0; k < 6; ++k) full[k] = st.link(q, k);
        full[6] = fx_minor(full[1], full[5], full[2], full[4]);
        full[7] = fx_minor(full[2], full[3], full[0], full[5]);
        full[8] = fx_minor(full[0], full[4], full[1], full[3]);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        FxEntry u[3];
        int wh[3], wl[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int k = FWD ? 3 * a + b : 3 * b + a;
            u[b] = RECON == 12 ? full[RECON == 12 ? k : 0] : st.link(q, k);
            wh[b] = FWD ? u[b].x + u[b].z : u[b].x - u[b].z;
            wl[b] = FWD ? u[b].y + u[b].w : u[b].y - u[b].w;
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            unsigned long long k = 1u << (FX_LIMB - 1), re, im;
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                k = fx_mad(wh[b], x.lo[s][b][0], k);
                k = fx_mad(wl[b], x.hi[s][b][0], k);
            }
            re = im = k;
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                re = fx_mad(u[b].z, sl[s][b], re);
                im = fx_mad(u[b].x, dl[s][b], im);
                re = fx_mad(u[b].w, sh[s][b], re);
                im = fx_mad(u[b].y, dh[s][b], im);
            }
            k = half;
#pragma unroll
            for (int b = 0; b < 3; ++b) k = fx_mad(wh[b], x.hi[s][b][0], k);
            re = k + ((long long)re >> FX_LIMB);
            im = k + ((long long)im >> FX_LIMB);
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                re = fx_mad(u[b].z, sh[s][b], re);
                im = fx_mad(u[b].x, dh[s][b], im);
            }
            long long r = (long long)re, i = (long long)im;
            if (ALIGN) {
                r = fx_sar(r, d);
                i = fx_sar(i, d);
            }
            fx_accumulate<MU, S>(s, a, r, i, t, sizes);
        }
    }
}

// ---- input in fixed point (FXF)
// The projected half-spinor of the fixed-point site j: project() on limbs.
template <int MU, int S, class Stage> __device__ __forceinline__ void fx_project(const Stage &st, FxHalf &x)
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int4 p[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) p[s] = st.spinor(3 * s + c);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            // h_s = u_s + S (A_mu l)_s: the lower spin and its factor (1 or i, signed)
            const int4 l = p[2 + ((MU == 0 || MU == 3) ? s : 1 - s)];
            const bool times_i = MU == 1 || MU == 3;
            bool minus = S < 0;
            if (MU == 0 || MU == 1) minus = !minus;           // A_0 l = -l; A_1 l = (-i l1, -i l0)
            if (MU == 2 && s == 0) minus = !minus;            // A_2 l = (-l1, l0)
            if (MU == 3 && s == 0) minus = !minus;            // A_3 l = (-i l0, i l1)
            const int rh = times_i ? -l.z : l.x, rl = times_i ? -l.w : l.y;
            const int ih = times_i ? l.x : l.z, il = times_i ? l.y : l.w;
            x.hi[s][c][0] = minus ? p[s].x - rh : p[s].x + rh;
            x.lo[s][c][0] = minus ? p[s].y - rl : p[s].y + rl;
            x.hi[s][c][1] = minus ? p[s].z - ih : p[s].z + ih;
            x.lo[s][c][1] = minus ? p[s].w - il : p[s].w + il;
        }
    }
}

__device__ __forceinline__ void fx_negate(FxHalf &x, int sg)
{
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                x.hi[s][c][k] *= sg;
                x.lo[s][c][k] *= sg;
            }
}

// ---- input in FP64
// h (times -1 if neg) as limbs of 58 bits under the sum's exponent, which is
// raised (to one more than h needs) where h does not fit.
// bad: set by components that the integer path does not take.
template <bool FIRST, class Sizes>
__device__ __forceinline__ void fx_from_half(const Half<double> &h, bool neg, FxHalf &x, FxSum &t, const Sizes &sizes, bool &bad)
{
    unsigned m = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const unsigned a = unsigned(__double2hiint(h[s][c].re)) & 0x7fffffffu;
            const unsigned b = unsigned(__double2hiint(h[s][c].im)) & 0x7fffffffu;
            m = max(m, max(a, b));
        }
    const int e = int(m >> 20) - 1022;   // |h| < 2^e
    if (m < (FX_FMIN << 20)) {           // all zero, or too small for the integer path
        unsigned bits = m;
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int c = 0; c < 3; ++c) bits |= unsigned(__double2loint(h[s][c].re)) | unsigned(__double2loint(h[s][c].im));
        bad = bad || bits;
    } else {
        bad = bad || m >= (FX_FMAX + 1) << 20;
        if (e > t.e) {
            if (!FIRST) {   // before the first hop all sums are zero
                const int s = e + 1 - t.e;
#pragma unroll
                for (int sp = 0; sp < 4; ++sp)
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        t.re[sp][c] = fx_sar(t.re[sp][c], s);
                        t.im[sp][c] = fx_sar(t.im[sp][c], s);
                    }
                sizes.sar(s);
            }
            t.e = e + 1;
        }
    }
    const unsigned from = unsigned(t.e + 1022 + 3), nm = neg ? 0xffffffffu : 0u;
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            fx_split(h[s][c].re, from, nm, x.hi[s][c][0], x.lo[s][c][0]);
            fx_split(h[s][c].im, from, nm, x.hi[s][c][1], x.lo[s][c][1]);
        }
}

// ---- the 8 hops
// Starts the copies of hop K (2 mu, or 2 mu + 1 for the backward one).
template <int P, int K, class Stage>
__device__ __forceinline__ void fx_start(const Geom &g, const Nbrs &n, const FxLinks<Stage::RECON> &src, const void *in, const Stage &st)
{
    constexpr int MU = K >> 1;
    const unsigned j = K & 1 ? n.bwd[MU] : n.fwd[MU];
    const int4 *f = static_cast<const int4 *>(in);
    const FxEntry *u = src.template at<MU, !(K & 1)>(n);
    if (P == FXF) st.start(K & 1, fx_entry(f, FX_SPINOR_BLOCK, j), 32, u);
    else if (P == F64C) st.start(K & 1, f + size_t(j) * 12, 1, u);
    else st.start(K & 1, f + j, g.vh, u);
}

// Hops K to LAST.  SIGNS: whether directions other than time may
// have a boundary sign.
template <int P, bool DAG, int K, int LAST, bool SIGNS, bool FIRST = true, class Stage>
__device__ __forceinline__ void fx_hops(const Geom &g, const Nbrs &n, const FxLinks<Stage::RECON> &src, const void *in,
                                        const Stage &st, const int4 *x0, size_t xstride, unsigned long long d,
                                        FxSum &t, const FxSizes<Stage::BLOCK> &sizes, bool &bad)
{
    st.wait();
    constexpr int MU = K >> 1, q = K & 1;
    constexpr int S = (DAG ? +1 : -1) * (q ? -1 : 1);
    const bool neg = (MU == 0 || SIGNS) && (q ? n.wb[MU] : n.wf[MU]) && g.anti[MU];
    FxHalf x;
    if constexpr (P == FXF) {
        fx_project<MU, S>(st, x);
        if (MU == 0 || SIGNS) fx_negate(x, neg ? -1 : 1);
    } else {
        Spinor<double> s;
        Half<double> h;
        st.site(s);
        project<MU, S>(s, h);
        fx_from_half<FIRST>(h, neg, x, t, sizes, bad);
    }
    __syncwarp();   // the site's words are read before the next copies start
    if constexpr (K < LAST) fx_start<P, K + 1>(g, n, src, in, st);
    else if (x0) st.start_site(x0, xstride);
    fx_apply<MU, S, q == 0, P == FXF>(st, q, x, int(unsigned(d >> (8 * K)) & 0xffu), t, sizes);
    if constexpr (K < LAST) fx_hops<P, DAG, K + 1, LAST, SIGNS, false>(g, n, src, in, st, x0, xstride, d, t, sizes, bad);
}

// Everything a fixed-point hop launch needs; a kernel parameter that device
// functions read in place.
struct FxArgs {
    Geom g;
    SiteMap m;
    Coef k;
    int p;                  // output parity
    const FxEntry *fx;      // fixed-point links
    const double2 *links;   // FP64 links
    const void *in, *x;
    void *out;
    const void *exact;      // the FP64 field that `in` is a fixed-point copy of, else `in` itself
    // for a fixed-point output: a = scale 2^scale_e, the smaller of |re| + |im| of k's two factors of the hop
    float scale;
    int scale_e;
    FxArgs(const Geom &geom, const SiteMap &map, const Coef &coef, int parity, const void *fx_links, const void *fp64_links,
           const void *input, const void *reread, void *output, const void *exact_input)
        : g(geom), m(map), k(coef), p(parity), fx(static_cast<const FxEntry *>(fx_links)),
          links(static_cast<const double2 *>(fp64_links)), in(input), x(reread), out(output), exact(exact_input)
    {
        const double a = coef.unit ? 1.0 : std::fmin(std::fabs(coef.d[0]) + std::fabs(coef.d[1]),
                                                     std::fabs(coef.d[2]) + std::fabs(coef.d[3]));
        scale = float(std::frexp(a, &scale_e));
    }
};

// |v| 2^-e as a float that is zero only for v = 0 and good to 2^-20 from 2^-60 on.
__device__ __forceinline__ float fx_narrow(double v, int e)
{
    const unsigned hw = unsigned(__double2hiint(v)) & 0x7fffffffu;
    const int f = int(hw) - ((e + 896) << 20);
    const float r = f < (67 << 20) ? 0x1p-60f : __int_as_float(f << 3);
    return (hw | unsigned(__double2loint(v))) == 0u ? 0.f : r;
}

// Whether the result of a fixed-point hop, o = a hop, may be stored in fixed
// point (FxSite f), with `least` the smallest sum of absolute products of its
// components in units of 2^e: FX_LEAST_STORED.
__device__ __forceinline__ bool fx_stores(const FxArgs &A, float least, int e, const FxSite &f)
{
    if (f.raw || f.e == FX_ZERO_E) return true;
    const int up = max(min(e + A.scale_e - f.e, 60), -60);   // far less wherever it matters
    return least * A.scale * __int_as_float((127 + up) << 23) >= FX_LEAST_STORED;
}

// Component c of site j of a field that SpinorIO<P> describes.
template <int P> __device__ __forceinline__ cpx<double> fx_load(const void *base, unsigned vh, unsigned j, int c)
{
    const int4 *b = static_cast<const int4 *>(base);
    if (P == FXF) return fx_component(fx_entry(b, FX_SPINOR_BLOCK, j)[32 * c], fx_words(base, vh)[j]);
    const double2 v = ld_keep(reinterpret_cast<const double2 *>(base) + (P == F64C ? size_t(j) * 12 + c : size_t(c) * vh + j));
    return {v.x, v.y};
}

// The smallest nonzero sum of absolute products S that enters a component of
// the hop at site i, in units of 2^e (infinite if all are zero), from the
// FP64 input with FP64 projections; the products in single precision.
template <int PR, int RECON, bool DAG> __device__ __forceinline__ float fx_least_sum(const FxArgs &A, unsigned i, int e)
{
    Nbrs n;
    neighbours(A.g, A.p, i, n);
    const GlobalLinks<F64, RECON> src{A.links, A.g.vh, i, A.p};
    constexpr int SF = DAG ? +1 : -1, SB = -SF;
    float sum[4][3][2] = {};
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        const int mu = k >> 1;
        const bool fwd = (k & 1) == 0;
        unsigned j = 0;
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (m == mu) j = fwd ? n.fwd[m] : n.bwd[m];
        Spinor<double> s;
        Half<double> h;
        Link<double> u;
        SpinorIO<PR>::load_raw(A.exact, A.g.vh, j, s);
        switch (k) {
        case 0: project<0, SF>(s, h); src.template fwd<0>(n, u); break;
        case 1: project<0, SB>(s, h); src.template bwd<0>(n, u); break;
        case 2: project<1, SF>(s, h); src.template fwd<1>(n, u); break;
        case 3: project<1, SB>(s, h); src.template bwd<1>(n, u); break;
        case 4: project<2, SF>(s, h); src.template fwd<2>(n, u); break;
        case 5: project<2, SB>(s, h); src.template bwd<2>(n, u); break;
        case 6: project<3, SF>(s, h); src.template fwd<3>(n, u); break;
        default: project<3, SB>(s, h); src.template bwd<3>(n, u); break;
        }
        float w[3][3][2], v[2][3][2];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                w[a][b][0] = fx_narrow(fwd ? u[a][b].re : u[b][a].re, 0);
                w[a][b][1] = fx_narrow(fwd ? u[a][b].im : u[b][a].im, 0);
            }
#pragma unroll
        for (int sp = 0; sp < 2; ++sp)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[sp][c][0] = fx_narrow(h[sp][c].re, e);
                v[sp][c][1] = fx_narrow(h[sp][c].im, e);
            }
        // the lower spin that an upper one feeds, and whether times i (fx_accumulate)
        const bool cross = mu == 1 || mu == 2, times_i = mu == 1 || mu == 3;
#pragma unroll
        for (int sp = 0; sp < 2; ++sp)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                float re = 0.f, im = 0.f;
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    re += w[a][b][0] * v[sp][b][0] + w[a][b][1] * v[sp][b][1];
                    im += w[a][b][0] * v[sp][b][1] + w[a][b][1] * v[sp][b][0];
                }
                sum[sp][a][0] += re;
                sum[sp][a][1] += im;
                const float x = times_i ? im : re, y = times_i ? re : im;
                sum[2 + sp][a][0] += cross ? 0.f : x;
                sum[2 + sp][a][1] += cross ? 0.f : y;
                sum[3 - sp][a][0] += cross ? x : 0.f;
                sum[3 - sp][a][1] += cross ? y : 0.f;
            }
    }
    float least = __int_as_float(0x7f800000);
#pragma unroll
    for (int c = 0; c < 24; ++c) {
        const float v = sum[c / 6][c / 2 % 3][c & 1];
        if (v != 0.f) least = fminf(least, v);
    }
    return least;
}

// One site by a whole warp: a lane takes one of the 8 hops, one upper spin s,
// and the real or the imaginary parts.
template <int PR, int RECON, bool DAG> struct FxWarpSite {
    int k, mu, s, part;
    bool fwd, cross, times_i, plus, neg;   // the lower spin that s feeds is 1 - s; times i; projector's sign; boundary
    cpx<double> h[3];                      // the projected spin
    Link<double> u;
    __device__ __forceinline__ FxWarpSite(const FxArgs &A, unsigned i)
    {
        using L = LinkIO<F64, RECON>;
        const unsigned vh = A.g.vh, lane = threadIdx.x & 31;
        k = lane & 7, mu = k >> 1, s = (lane >> 3) & 1, part = lane >> 4;
        fwd = (k & 1) == 0, cross = mu == 1 || mu == 2, times_i = mu == 1 || mu == 3;
        plus = (DAG ? +1 : -1) * (fwd ? 1 : -1) > 0;
        Nbrs n;
        neighbours(A.g, A.p, i, n);
        unsigned j = 0, jb = 0;
        neg = false;
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (m == mu) {
                j = fwd ? n.fwd[m] : n.bwd[m];
                jb = fwd ? i : n.bwd[m];
                neg = (fwd ? n.wf[m] : n.wb[m]) && A.g.anti[m];
            }
        L::load(A.links + size_t(4 * (fwd ? A.p : 1 - A.p) + mu) * L::NCHUNK * vh, vh, jb, u);
        // h_s = u_s + f l, f = 1, -1, i or -i (fx_project)
        const bool toggle = mu < 2 || s == 0;
        const double f = plus != toggle ? 1.0 : -1.0;
        const int low = 2 + (cross ? 1 - s : s);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const cpx<double> a = fx_load<PR>(A.exact, vh, j, 3 * s + c), l = fx_load<PR>(A.exact, vh, j, 3 * low + c);
            h[c] = {a.re + f * (times_i ? -l.im : l.re), a.im + f * (times_i ? l.re : l.im)};
        }
    }
    __device__ __forceinline__ cpx<double> link(int a, int b) const { return fwd ? u[a][b] : conj(u[b][a]); }
    // The lane that holds this lane's share of a lower spin (and gives its own).
    __device__ __forceinline__ int partner() const { return (cross ? 8 : 0) | (times_i ? 16 : 0); }
};

// fx_least_sum of one site by a whole warp.
template <int PR, int RECON, bool DAG> __device__ __forceinline__ float fx_least_sum_warp(const FxArgs &A, unsigned i, int e)
{
    constexpr unsigned all = 0xffffffffu;
    const FxWarpSite<PR, RECON, DAG> w(A, i);
    float least = __int_as_float(0x7f800000), v[3][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float re = fx_narrow(w.h[c].re, e), im = fx_narrow(w.h[c].im, e);
        v[c][0] = w.part ? im : re;
        v[c][1] = w.part ? re : im;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float x = 0.f;
#pragma unroll
        for (int b = 0; b < 3; ++b) x += fx_narrow(w.link(a, b).re, 0) * v[b][0] + fx_narrow(w.link(a, b).im, 0) * v[b][1];
        float y = __shfl_xor_sync(all, x, w.partner());
#pragma unroll
        for (int o = 1; o < 8; o *= 2) {
            x += __shfl_xor_sync(all, x, o);
            y += __shfl_xor_sync(all, y, o);
        }
        if (x != 0.f) least = fminf(least, x);
        if (y != 0.f) least = fminf(least, y);
    }
    least = fminf(least, __shfl_xor_sync(all, least, 8));
    return fminf(least, __shfl_xor_sync(all, least, 16));
}

// Output site i with FP64 products, from the input to the stored result.
// Returns whether all its hops are finite; if not, nothing is stored (the
// order of the sums decides between NaN and infinities: fx_again's).
template <int PR, int PX, int PO, int RECON, bool DAG, bool HASX>
__device__ __forceinline__ bool fx_site_warp(const FxArgs &A, unsigned i)
{
    constexpr unsigned all = 0xffffffffu;
    const unsigned vh = A.g.vh;
    const FxWarpSite<PR, RECON, DAG> w(A, i);
    double x[3], y[3];
    bool finite = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double r = 0.0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const cpx<double> u = w.link(a, b);
            r += u.re * (w.part ? w.h[b].im : w.h[b].re);
            r += u.im * (w.part ? w.h[b].re : -w.h[b].im);
        }
        x[a] = w.neg ? -r : r;
        // as in accumulate(): what the lower spin gets of it, i r = (-im, re)
        const int to = w.cross ? 1 - w.s : w.s;
        bool minus = !w.plus;
        if (w.mu == 0 || (w.mu >= 2 && to == 1)) minus = !minus;
        if (w.times_i && w.part) minus = !minus;
        y[a] = __shfl_xor_sync(all, minus ? -x[a] : x[a], w.partner());
#pragma unroll
        for (int o = 1; o < 8; o *= 2) {
            x[a] += __shfl_xor_sync(all, x[a], o);
            y[a] += __shfl_xor_sync(all, y[a], o);
        }
        finite = finite && fabs(x[a]) <= 1.7976931348623157e308 && fabs(y[a]) <= 1.7976931348623157e308;
    }
    if (!__all_sync(all, finite)) return false;
    const int spin = (w.k == 0 ? 0 : 2) + w.s;   // of the lanes that store: parts re, hops 0 and 1
    const bool up = spin < 2;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double re = w.k == 0 ? x[a] : y[a], im = __shfl_xor_sync(all, re, 16);
        if (w.part || w.k > 1) continue;
        const cpx<double> hop = {re, im};
        const double *d = A.k.d + (up ? 0 : 2);
        cpx<double> o = A.k.unit ? (up ? hop : -hop) : cpx<double>{d[0], d[1]} * hop;
        if (HASX) o = cmadd(cpx<double>{d[4], d[5]}, fx_load<PX>(A.x, vh, i, 3 * spin + a), o);
        const int c = 3 * spin + a;
        if (PO == FXF) {
            st_stream(fx_entry(static_cast<int4 *>(A.out), FX_SPINOR_BLOCK, i) + 32 * c,
                      make_int4(__double2hiint(o.re), __double2loint(o.re), __double2hiint(o.im), __double2loint(o.im)));
            if (c == 0) st_stream(const_cast<int *>(fx_words(A.out, vh)) + i, FX_RAW);
        } else {
            st_stream(static_cast<double2 *>(A.out) + (PO == F64C ? size_t(i) * 12 + c : size_t(c) * vh + i), make_double2(o.re, o.im));
        }
    }
    return true;
}

// What is left to do at output site i after its fixed-point hop.
enum { FX_DONE = 0, FX_CHECK = 1, FX_SLOW = 2 };

// The few sites of a warp that are not done; every lane of the warp calls it.
// FX_CHECK: the stored fixed-point result, with 2^48 eta = 2^e, stays if every
// sum of absolute products is large enough (for a fixed-point output also for
// it to be stored so).  FX_SLOW and the others: computed with FP64 products,
// from the input to the stored result.  A call whose arguments are few words:
// passing the site's sum in and out cost 7 % of the kernel.
// Up to FX_FEW sites are done one by one by the whole warp.  By a lane each,
// the check is a chain of several us that every launch waited for somewhere
// (Q_tm on 16^4 69 us, now 40; on 8^4 45, now 16), and FP64 products a longer
// one (16^4, unit links, with such sites: 113 us, now 73).  With 16 a point
// source on 8^4 took 95 us against 84.  More are checked and computed by a
// lane each: checks one by one take 35 us per site of a warp and launch on
// 24^3x48, by all lanes at once 80.  Such fields have components of exactly
// zero, which only the check tells from small ones (Q_tm on a field of one
// spin, 24^3x48, links exp(0.3 i A): 1.45 ms unchecked, 0.45 checked), or
// components of very different size, for which it is spent in vain (1.58
// against 1.45 ms; 1.02 with FP64 products throughout).
constexpr int FX_FEW = 8;
template <int PR, int PX, int PO, int RECON, bool DAG, bool HASX>
__device__ __noinline__ void fx_again(const FxArgs &A, unsigned i, int e, int todo)
{
    constexpr unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    __syncwarp();   // results stored so far come before what other lanes replace
    unsigned check = __ballot_sync(all, todo == FX_CHECK);
    float least = 0.f;
    if (__popc(check) > FX_FEW) {
        if (todo == FX_CHECK) least = fx_least_sum<PR, RECON, DAG>(A, i, e);
        __syncwarp();
    } else {
        while (check) {
            const int q = __ffs(int(check)) - 1;
            check &= check - 1;
            const float of_q = fx_least_sum_warp<PR, RECON, DAG>(A, __shfl_sync(all, i, q), __shfl_sync(all, e, q));
            if (lane == q) least = of_q;
        }
    }
    if (todo == FX_CHECK) {
        bool stays = least >= float(FX_LEAST);
        if (PO == FXF) {
            const int word = static_cast<const volatile int *>(fx_words(A.out, A.g.vh))[i];
            FxSite f(0, 0);
            f.raw = word == FX_RAW;
            f.e = int(short(word & 0xffff));
            stays = stays && fx_stores(A, least, e, f);
        }
        if (stays) todo = FX_DONE;
    }
    unsigned slow = __ballot_sync(all, todo != FX_DONE);
    if (__popc(slow) <= FX_FEW) {
        while (slow) {
            const int q = __ffs(int(slow)) - 1;
            slow &= slow - 1;
            if (fx_site_warp<PR, PX, PO, RECON, DAG, HASX>(A, __shfl_sync(all, i, q)) && lane == q) todo = FX_DONE;
        }
    }
    if (todo == FX_DONE) return;
    Nbrs n;
    neighbours(A.g, A.p, i, n);
    GlobalLinks<F64, RECON> src{A.links, A.g.vh, i, A.p};
    Spinor<double> acc, xs, o;
    hop_site_src<PR, DAG>(A.g, n, src, A.exact, acc);
    if (HASX) SpinorIO<PX>::load(A.x, A.g.vh, i, xs);
    epilogue(A.k, acc, HASX ? &xs : nullptr, o);
    if constexpr (PO == FXF) SpinorIO<FXF>::store_as(A.out, A.g.vh, i, o, true);
    else SpinorIO<PO>::store(A.out, A.g.vh, i, o);
}

// The exponent of a site's sum, the largest of its 8 neighbours', and per hop
// a byte of d: the shift that aligns it.  Returns whether the integer path
// does not take the site.
__device__ __forceinline__ bool fx_exponents(const Nbrs &n, const void *in, unsigned vh, int &sum_e, unsigned long long &d)
{
    const int *word = fx_words(in, vh);
    int e[8];
    bool slow = false;
    sum_e = FX_ZERO_E;
#pragma unroll
    for (int m = 0; m < 8; ++m) e[m] = ld_keep(word + (m & 1 ? n.bwd[m >> 1] : n.fwd[m >> 1]));
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        slow = slow || e[m] == FX_RAW;
        e[m] = int(short(e[m] & 0xffff));
        sum_e = max(sum_e, e[m]);
    }
    d = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) d |= (unsigned long long)(unsigned(min(sum_e - e[m], 63))) << (8 * m);
    return slow;
}

// What is to be done with a site after its fixed-point hop.
struct FxVerdict {
    bool slow;    // the integer path does not take it: acc is not its hop
    int least;    // the smallest sum of absolute values of its 24 components,
    int e;        // in units of 2^e
    __device__ __forceinline__ FxVerdict(bool slow_, int least_, int sum_e, int bits)
        : slow(slow_), least(least_), e(sum_e - bits + 48)
    {
        if (sum_e <= FX_ZERO_E) least = 0x7fff;   // all neighbours zero
    }
};

// The hop at output site i; every thread of the warp calls it.  With x0 set,
// the 12 words at x0, xstride apart, are in the stage's site slot once its
// copies are waited for.
template <int P, int RECON, bool DAG, bool SIGNS>
__device__ __forceinline__ FxVerdict fx_hop_site(const FxArgs &A, unsigned i, const FxStage<RECON> &st,
                                                 const FxSizes<FX_BLOCK> &sizes, const int4 *x0, size_t xstride,
                                                 Spinor<double> &acc)
{
    const Geom &g = A.g;
    const void *in = A.in;
    Nbrs n;
    neighbours(g, A.p, i, n);
    const FxLinks<RECON> src{A.fx, g.vh, i, A.p};
    fx_start<P, 0>(g, n, src, in, st);
    FxSum t;
    unsigned long long d = 0;
    t.clear(P == FXF ? FX_ZERO_E : FX_LOWEST_E);
    bool slow = false;
    if constexpr (P == FXF) slow = fx_exponents(n, in, g.vh, t.e, d);
    fx_hops<P, DAG, 0, 7, SIGNS>(g, n, src, in, st, x0, xstride, d, t, sizes, slow);
    constexpr int bits = P == FXF ? FX_FIELD : FX_HALF;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            acc[s][c] = {fx_to_double(t.re[s][c], t.e, bits), fx_to_double(t.im[s][c], t.e, bits)};
    return FxVerdict(slow, sizes.least(), t.e, bits);
}

// Stores the result o of a site (if on) whose hop gave verdict v, or has it
// looked at again; every lane of the warp calls it.  Returns whether some
// lane's o may have been replaced.
template <int PR, int PX, int PO, int RECON, bool DAG, bool HASX>
__device__ __forceinline__ bool fx_finish(const FxArgs &A, unsigned i, bool on, const FxVerdict &v, const Spinor<double> &o)
{
    int todo = !on ? FX_DONE : v.slow ? FX_SLOW : v.least < FX_LEAST ? FX_CHECK : FX_DONE;
    if (on && !v.slow) {
        if constexpr (PO == FXF) {
            const FxSite f = SpinorIO<FXF>::store_as(A.out, A.g.vh, i, o, false);
            if (!fx_stores(A, float(v.least), v.e, f)) todo = FX_CHECK;
        } else {
            SpinorIO<PO>::store(A.out, A.g.vh, i, o);
        }
    }
    if (!__any_sync(0xffffffffu, todo != FX_DONE)) return false;
    fx_again<PR, PX, PO, RECON, DAG, HASX>(A, i, v.e, todo);
    __syncwarp();   // a site may have been stored by other lanes than its own
    return true;
}

#endif  // __CUDACC__

}  // namespace twm

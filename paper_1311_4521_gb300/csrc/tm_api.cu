// tm_api.cu -- the C ABI of include/tmhop.h: contexts, gauge handles,
// packed fields, the hopping matrix and Q_tm.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "tm_internal.h"

using namespace twm;

namespace {

tm_status fail(tm_ctx *ctx, tm_status st, const char *fmt, const char *detail = "")
{
    if (ctx) {
        char buf[512];
        snprintf(buf, sizeof buf, fmt, detail);
        ctx->err = buf;
    }
    return st;
}

tm_status cuda_fail(tm_ctx *ctx, cudaError_t e, const char *where)
{
    if (ctx) ctx->err = std::string(where) + ": " + cudaGetErrorString(e);
    return TM_ERR_CUDA;
}

#define TM_CUDA(ctx, call)                                     \
    do {                                                       \
        cudaError_t e_ = (call);                               \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_, #call); \
    } while (0)

// Makes the fixed-point copy of an FP64 handle's links (tm_fix.cuh) in the
// fx_room bytes at fx; the handle keeps it unless some
// link does not fit (the hops then use FP64 products).  Synchronises s.
cudaError_t make_fx_links(tm_gauge *h, void *fx, cudaStream_t s)
{
    int *flag = reinterpret_cast<int *>(static_cast<char *>(fx) + fx_copy_bytes(h)), unfit = 0;
    cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int), s);
    if (e == cudaSuccess) e = launch_fx_links(h->geom.vh, h->recon, h->links, fx, flag, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&unfit, flag, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && !unfit) h->fx = fx;
    return e;
}

// While it lives, this thread may allocate although a stream captures in
// global mode; such a call would otherwise fail and end that capture.
struct AllowAllocation {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    AllowAllocation() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~AllowAllocation() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

bool valid_prec(int p) { return p == TM_F64 || p == TM_F32 || p == TM_F16 || p == TM_F64X; }

}  // namespace

tm_status tm_ctx_scratch(tm_ctx *ctx, size_t bytes, void **ptr)
{
    if (ctx->scratch_bytes < bytes) {
        if (ctx->scratch) {
            cudaError_t e = cudaFree(ctx->scratch);
            ctx->scratch = nullptr;
            ctx->scratch_bytes = 0;
            if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFree(scratch)");
        }
        TM_CUDA(ctx, cudaMalloc(&ctx->scratch, bytes));
        ctx->scratch_bytes = bytes;
    }
    *ptr = ctx->scratch;
    return TM_OK;
}

tm_status tm_qtm_scratch(tm_ctx *ctx, const tm_gauge *U, cudaStream_t s, void **tmp, bool *fx)
{
    const size_t bytes = U->fx ? fx_qtm_bytes(U->geom.vh) : 0;
    if (ctx->fx_scratch_bytes < bytes) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        const cudaError_t q = cudaStreamIsCapturing(s, &capture);
        if (q != cudaSuccess) (void)cudaGetLastError();   // the default stream while another one captures
        if (q == cudaSuccess && capture == cudaStreamCaptureStatusNone) {
            // not part of a capture that this or another thread makes on another stream
            const AllowAllocation allow;
            if (ctx->fx_scratch) {
                const cudaError_t e = cudaFree(ctx->fx_scratch);
                ctx->fx_scratch = nullptr;
                ctx->fx_scratch_bytes = 0;
                if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFree(fixed-point scratch)");
            }
            const cudaError_t e = cudaMalloc(&ctx->fx_scratch, bytes);
            if (e == cudaSuccess) ctx->fx_scratch_bytes = bytes;
            else if (e != cudaErrorMemoryAllocation) return cuda_fail(ctx, e, "cudaMalloc(fixed-point scratch)");
            else (void)cudaGetLastError();   // not sticky
        }
    }
    *fx = bytes != 0 && ctx->fx_scratch_bytes >= bytes;
    if (!*fx) return tm_ctx_scratch(ctx, spinor_bytes(U->geom.vh, U->prec), tmp);
    *tmp = ctx->fx_scratch;
    return TM_OK;
}

tm_status tm_ctx_reduce_buffer(tm_ctx *ctx, size_t bytes, void **ptr)
{
    if (ctx->red_bytes < bytes) {
        if (ctx->red) {
            cudaError_t e = cudaFree(ctx->red);
            ctx->red = nullptr;
            ctx->red_bytes = 0;
            if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFree(reduce buffer)");
        }
        TM_CUDA(ctx, cudaMalloc(&ctx->red, bytes));
        ctx->red_bytes = bytes;
    }
    *ptr = ctx->red;
    return TM_OK;
}

extern "C" {

const char *tm_status_string(tm_status s)
{
    switch (s) {
    case TM_OK: return "ok";
    case TM_ERR_ARG: return "invalid argument";
    case TM_ERR_CUDA: return "CUDA error";
    case TM_ERR_NOT_CONVERGED: return "solver did not converge";
    case TM_ERR_NONFINITE: return "non-finite residual";
    case TM_ERR_TIMEOUT: return "device wait timed out";
    case TM_ERR_UNSUPPORTED: return "unsupported combination";
    }
    return "unknown status";
}

tm_status tm_ctx_create(tm_ctx **out, int device)
{
    if (!out) return TM_ERR_ARG;
    *out = nullptr;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) return TM_ERR_ARG;
    if (cudaSetDevice(device) != cudaSuccess) return TM_ERR_CUDA;
    tm_ctx *ctx = new tm_ctx;
    ctx->device = device;
    cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, device);
    if (const char *cache = getenv("TMHOP_TUNE_CACHE")) ctx->tune_cache = cache;
    *out = ctx;
    return TM_OK;
}

void tm_ctx_destroy(tm_ctx *ctx)
{
    if (!ctx) return;
    if (ctx->scratch) cudaFree(ctx->scratch);
    if (ctx->fx_scratch) cudaFree(ctx->fx_scratch);
    if (ctx->ws) cudaFree(ctx->ws);
    if (ctx->stage) cudaFree(ctx->stage);
    if (ctx->bq) cudaFree(ctx->bq);
    if (ctx->red) cudaFree(ctx->red);
    if (ctx->dev_status) cudaFree(ctx->dev_status);
    if (ctx->copy_in) cudaStreamDestroy(ctx->copy_in);
    if (ctx->copy_out) cudaStreamDestroy(ctx->copy_out);
    delete ctx;
}

const char *tm_last_error(const tm_ctx *ctx) { return ctx ? ctx->err.c_str() : "null context"; }

tm_status tm_ctx_check(tm_ctx *ctx)
{
    if (!ctx) return TM_ERR_ARG;
    if (!ctx->dev_status) return TM_OK;
    int v = 0;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(&v, ctx->dev_status, sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && v) e = cudaMemset(ctx->dev_status, 0, sizeof(int));
    if (e != cudaSuccess) return cuda_fail(ctx, e, "tm_ctx_check");
    if (v) return fail(ctx, TM_ERR_CUDA, "tm_ctx_check: a bounded wait of the staged batched hop ran out");
    return TM_OK;
}

tm_status tm_ctx_set_fixed_point(tm_ctx *ctx, int on)
{
    if (!ctx) return TM_ERR_ARG;
    ctx->fixed_point = on ? 1 : 0;
    return TM_OK;
}

tm_status tm_ctx_set_autotune(tm_ctx *ctx, int on)
{
    if (!ctx) return TM_ERR_ARG;
    ctx->autotune = on ? 1 : 0;
    return TM_OK;
}

size_t tm_ctx_tune_report(const tm_ctx *ctx, char *buf, size_t size)
{
    if (!ctx) return 0;
    std::string rep;
    for (const auto &kv : ctx->tuned) {
        char line[256];
        auto ms = ctx->tuned_ms.find(kv.first);
        auto band = ctx->tuned_band.find(kv.first);
        snprintf(line, sizeof line, "%s nrb=%d cap=%u ms3=%.4f band=%d\n", kv.first.c_str(), kv.second.first,
                 kv.second.second, ms == ctx->tuned_ms.end() ? 0.0 : double(ms->second),
                 band == ctx->tuned_band.end() ? 1 : band->second);
        rep += line;
    }
    for (const auto &kv : ctx->tuned_maps) rep += "hop/" + kv.first + " " + kv.second + "\n";
    if (buf && size > 0) {
        const size_t n = rep.size() < size - 1 ? rep.size() : size - 1;
        memcpy(buf, rep.data(), n);
        buf[n] = '\0';
    }
    return rep.size() + 1;
}

tm_status tm_ctx_trace(tm_ctx *ctx, void *const *events, int nevents)
{
    if (!ctx) return TM_ERR_ARG;
    ctx->trace.clear();
    if (!events) return TM_OK;
    if (nevents < 3) return fail(ctx, TM_ERR_ARG, "tm_ctx_trace: need at least 3 events");
    for (int k = 0; k < nevents; ++k) {
        if (!events[k]) {
            ctx->trace.clear();
            return fail(ctx, TM_ERR_ARG, "tm_ctx_trace: null event");
        }
        ctx->trace.push_back(static_cast<cudaEvent_t>(events[k]));
    }
    return TM_OK;
}

size_t tm_spinor_bytes(long vh, int prec)
{
    if (vh < 0 || !valid_prec(prec)) return 0;
    return spinor_bytes(unsigned(vh), prec);
}

tm_status tm_spinor_pack(tm_ctx *ctx, long vh, const double *in_dev, void *out_dev, int prec, void *stream)
{
    if (!ctx) return TM_ERR_ARG;
    if (vh < 0 || vh >= (1L << 31)) return fail(ctx, TM_ERR_ARG, "tm_spinor_pack: bad site count");
    if (!valid_prec(prec)) return fail(ctx, TM_ERR_ARG, "tm_spinor_pack: bad precision");
    if (vh > 0 && (bad_ptr(in_dev) || bad_ptr(out_dev))) return fail(ctx, TM_ERR_ARG, "tm_spinor_pack: null or misaligned pointer");
    TM_CUDA(ctx, launch_pack_spinor(unsigned(vh), prec, in_dev, out_dev, (cudaStream_t)stream));
    return TM_OK;
}

tm_status tm_spinor_unpack(tm_ctx *ctx, long vh, const void *in_dev, double *out_dev, int prec, void *stream)
{
    if (!ctx) return TM_ERR_ARG;
    if (vh < 0 || vh >= (1L << 31)) return fail(ctx, TM_ERR_ARG, "tm_spinor_unpack: bad site count");
    if (!valid_prec(prec)) return fail(ctx, TM_ERR_ARG, "tm_spinor_unpack: bad precision");
    if (vh > 0 && (bad_ptr(in_dev) || bad_ptr(out_dev))) return fail(ctx, TM_ERR_ARG, "tm_spinor_unpack: null or misaligned pointer");
    TM_CUDA(ctx, launch_unpack_spinor(unsigned(vh), prec, in_dev, out_dev, (cudaStream_t)stream));
    return TM_OK;
}

}  // extern "C"

static size_t link_bytes(const Geom &g, int prec, int reconstruct)
{
    return size_t(8) * link_nchunk(prec, reconstruct) * link_chunk_bytes(prec, reconstruct) * g.vh;
}

// Bytes for the fixed-point copy of an FP64 handle's links and its flag (make_fx_links).
static size_t fx_room(const tm_gauge *h) { return align256(fx_copy_bytes(h) + sizeof(int)); }

// Whether there is memory for the fixed-point copy of h's links beside what a
// program may still need: after it at least half of the device's memory is
// free, and 3 KiB per site of one parity, more than a solve on the lattice
// takes (workspace 1.6 KiB, of the full system another 1.3).  So the copies of
// all handles together never take the second half, and a lattice whose solve
// fits without a copy does not lose it to one.
static bool fx_fits(const tm_gauge *h)
{
    size_t left = 0, total = 0;
    if (cudaMemGetInfo(&left, &total) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return left >= fx_room(h) + std::max(total / 2, size_t(3072) * h->geom.vh);
}

static tm_status bad_format(int prec, int reconstruct)
{
    if (!valid_prec(prec) || (reconstruct != 12 && reconstruct != 18)) return TM_ERR_ARG;
    return prec == TM_F16 && reconstruct != 12 ? TM_ERR_UNSUPPORTED : TM_OK;
}

// A handle whose links live in memory of its own, or in the caller's (mem).
static tm_status create_gauge(tm_ctx *ctx, const char *name, const int dims[4], const double *U_dev, int prec,
                              int reconstruct, const int bc[4], void *mem, size_t mem_bytes, void *stream, tm_gauge **out)
{
    if (!ctx) return TM_ERR_ARG;
    auto refuse = [&](tm_status st, const char *why) { return tm_fail(ctx, st, std::string(name) + why); };
    if (!out || !dims || bad_ptr(U_dev) || !bc) return refuse(TM_ERR_ARG, ": null or misaligned pointer");
    *out = nullptr;
    if (const tm_status st = bad_format(prec, reconstruct))
        return refuse(st, st == TM_ERR_UNSUPPORTED ? ": TM_F16 links need reconstruct 12"
                          : valid_prec(prec)       ? ": reconstruct must be 12 or 18"
                                                   : ": bad precision");
    for (int m = 0; m < 4; ++m)
        if (bc[m] != 1 && bc[m] != -1) return refuse(TM_ERR_ARG, ": bc entries must be +1 or -1");
    Geom g;
    if (!make_geom(dims, bc, g)) return refuse(TM_ERR_ARG, ": extents must be even, >= 2, volume < 2^31");
    if (mem && mem_bytes < link_bytes(g, prec, reconstruct)) return refuse(TM_ERR_ARG, ": too little memory for the links");
    tm_gauge *h = new tm_gauge;
    h->ctx = ctx;
    memcpy(h->dims, dims, sizeof h->dims);
    memcpy(h->bc, bc, sizeof h->bc);
    h->prec = prec;
    h->recon = reconstruct;
    h->geom = g;
    h->bytes = link_bytes(g, prec, reconstruct);
    // the links, and for FP64 handles their fixed-point copy where there is memory
    const size_t copy = prec == TM_F64 && ctx->fixed_point ? fx_room(h) : 0;
    void *fx = nullptr;
    cudaError_t e = cudaSuccess;
    if (mem) {
        h->owns = false;
        h->links = mem;
        if (copy && mem_bytes >= align256(h->bytes) + copy) fx = static_cast<char *>(mem) + align256(h->bytes);
    } else {
        e = cudaMalloc(&h->links, h->bytes);
        if (e == cudaSuccess && copy && fx_fits(h)) {
            e = cudaMalloc(&fx, copy);
            if (e != cudaSuccess) fx = nullptr;
            if (e == cudaErrorMemoryAllocation) {
                (void)cudaGetLastError();   // not sticky
                e = cudaSuccess;
            }
        }
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (e == cudaSuccess) e = launch_pack_gauge(g, prec, reconstruct, U_dev, h->links, s);
    if (e == cudaSuccess && fx) e = make_fx_links(h, fx, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (h->owns && fx && !h->fx) cudaFree(fx);   // some link does not fit
    if (e != cudaSuccess) {
        if (e == cudaErrorMemoryAllocation) (void)cudaGetLastError();   // not sticky
        tm_gauge_destroy(h);
        return cuda_fail(ctx, e, name);
    }
    tm_apply_cached_map(ctx, h);
    *out = h;
    return TM_OK;
}

extern "C" {

tm_status tm_gauge_create(tm_ctx *ctx, const int dims[4], const double *U_dev, int prec, int reconstruct,
                          const int bc[4], void *stream, tm_gauge **out)
{
    return create_gauge(ctx, "tm_gauge_create", dims, U_dev, prec, reconstruct, bc, nullptr, 0, stream, out);
}

tm_status tm_gauge_create_in(tm_ctx *ctx, const int dims[4], const double *U_dev, int prec, int reconstruct,
                             const int bc[4], void *mem_dev, size_t bytes, void *stream, tm_gauge **out)
{
    if (!ctx) return TM_ERR_ARG;
    if (bad_ptr(mem_dev)) return fail(ctx, TM_ERR_ARG, "tm_gauge_create_in: null or misaligned memory");
    return create_gauge(ctx, "tm_gauge_create_in", dims, U_dev, prec, reconstruct, bc, mem_dev, bytes, stream, out);
}

size_t tm_gauge_storage_bytes(const int dims[4], int prec, int reconstruct)
{
    const int bc[4] = {1, 1, 1, 1};
    tm_gauge h;
    if (!dims || bad_format(prec, reconstruct) != TM_OK || !make_geom(dims, bc, h.geom)) return 0;
    h.recon = reconstruct;
    return align256(link_bytes(h.geom, prec, reconstruct)) + (prec == TM_F64 ? fx_room(&h) : 0);
}

void tm_gauge_destroy(tm_gauge *g)
{
    if (!g) return;
    if (g->owns && g->links) cudaFree(g->links);
    if (g->owns && g->fx) cudaFree(g->fx);
    if (g->links8) cudaFree(g->links8);
    delete g;
}

size_t tm_gauge_bytes(const tm_gauge *g) { return g ? g->bytes + (g->fx ? fx_copy_bytes(g) : 0) : 0; }

tm_status tm_hopping_eo(tm_ctx *ctx, const tm_gauge *U, void *out_dev, const void *in_dev, int dir, int dagger,
                        void *stream)
{
    if (!ctx) return TM_ERR_ARG;
    if (!U || bad_ptr(out_dev) || bad_ptr(in_dev)) return fail(ctx, TM_ERR_ARG, "tm_hopping_eo: null or misaligned pointer");
    if (dir != TM_EO && dir != TM_OE) return fail(ctx, TM_ERR_ARG, "tm_hopping_eo: dir must be TM_EO or TM_OE");
    if (out_dev == in_dev) return fail(ctx, TM_ERR_ARG, "tm_hopping_eo: out and in must not overlap");
    TM_CUDA(ctx, launch_hop(U, dagger != 0, dir, in_dev, out_dev, nullptr, coef_plain(), (cudaStream_t)stream));
    return TM_OK;
}

tm_status tm_Qtm(tm_ctx *ctx, const tm_gauge *U, void *out_e_dev, const void *in_e_dev, double kappa, double mu,
                 int sign, void *stream)
{
    if (!ctx) return TM_ERR_ARG;
    if (!U || bad_ptr(out_e_dev) || bad_ptr(in_e_dev)) return fail(ctx, TM_ERR_ARG, "tm_Qtm: null or misaligned pointer");
    if (sign != 1 && sign != -1) return fail(ctx, TM_ERR_ARG, "tm_Qtm: sign must be +1 or -1");
    if (out_e_dev == in_e_dev) return fail(ctx, TM_ERR_ARG, "tm_Qtm: out and in must not overlap");
    void *tmp = nullptr;
    bool fx = false;
    cudaStream_t s = (cudaStream_t)stream;
    tm_status st = tm_qtm_scratch(ctx, U, s, &tmp, &fx);
    if (st != TM_OK) return st;
    double mut = 2.0 * kappa * mu * sign;
    tm_trace_mark(ctx, 0, s);
    TM_CUDA(ctx, launch_qtm(U, fx, false, false, in_e_dev, tmp, out_e_dev, coef_qtm_a_scaled(kappa, mut), s));
    tm_trace_mark(ctx, 1, s);
    TM_CUDA(ctx, launch_qtm(U, fx, false, true, in_e_dev, tmp, out_e_dev, coef_qtm_b_unit(mut), s));
    tm_trace_mark(ctx, 2, s);
    return TM_OK;
}

}  // extern "C"

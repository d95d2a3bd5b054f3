// ge_api.cpp -- the C ABI declared in include/ge.h: argument checking,
// contexts and their device buffers, coefficients, kernel selection and
// launch sequencing.  Host code only; built with -ffp-contract=off so the
// coefficients are rounded exactly as written.
#include "ge.h"

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime_api.h>

#include <cmath>
#include <cstdlib>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>

#include "ge_internal.h"
#include "ge_prop.h"

namespace {

thread_local char g_last_error[512] = "";

ge_status fail(ge_status st, const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    std::vsnprintf(g_last_error, sizeof(g_last_error), fmt, ap);
    va_end(ap);
    return st;
}

ge_status cuda_fail(cudaError_t e, const char *what)
{
    if (e == cudaErrorMemoryAllocation)
        return fail(GE_ENOMEM, "%s: %s", what, cudaGetErrorString(e));
    return fail(GE_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

using ge::kDefaultDepthDf;
using ge::kDefaultDepthF32;
using ge::kDefaultDepthF64;
// Largest r the double-float kernel takes: the right-hand side reaches about
// (1 + 3r) times the data and must stay far inside the FP32 exponent range.
constexpr double kDfMaxR = 1048576.0;
constexpr int kMaxDepth = 1023;

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

size_t elem_size(ge_precision p) { return p == GE_F64 ? sizeof(double) : sizeof(float); }
int elems_per_row(ge_precision p) { return ge::kRowBytes / (int)elem_size(p); }

}  // namespace

namespace ge {
void set_last_error(const char *msg) { std::snprintf(g_last_error, sizeof(g_last_error), "%s", msg); }
}  // namespace ge

struct ge_ctx {
    CUtensorMap tmap[2];  // one per buffer (source of a tiled launch)
    int64_t n = 0;
    double r = 0, beta_l = 0, beta_r = 0;
    double onepg_lo = 0;  // low part of the scaled map's growth factor (see fill_coefficients)
    ge_precision prec = GE_F64;
    cudaStream_t stream = nullptr;
    int device = 0;
    int64_t n_rows = 0;  // 128-byte rows per buffer
    void *buf[2] = {nullptr, nullptr};
    int cur = 0;         // buffer holding the state
    int64_t step = 0;    // global step counter
    ge_kernel kernel = GE_KERNEL_AUTO;
    int depth = 0;
    int64_t width = 1;   // sub-domain width k
    int *err_dev = nullptr;
    int num_sms = 0;
    int tb_blocks_per_sm = 0;
    int tb_rounds_per_sm = 0;     // its cooperative form
    bool pooled = false;          // buf[0] comes from ctx_pool
    int tb_df_blocks_per_sm = 0;  // double-float kernel (GE_F64 contexts)
    ge::CanonCoef canon{};
    ge::TbParams tb{};   // launch-independent fields filled at creation
    ge::PropState prop{}; // composed steps (GE_KERNEL_AUTO)
};

namespace {

void fill_coefficients(ge_ctx *c)
{
    const double r = c->r;
    const double r2 = r * r;
    const double det = 1.0 + 2.0 * r;
    // Eqs. (cc)/(dd): numerator coefficients over the determinant 1 + 2r
    c->canon.c1 = (r + r2) / det;
    c->canon.c2 = (1.0 - r2) / det;
    c->canon.c3 = (r - r2) / det;
    c->canon.c4 = r2 / det;
    // Eqs. (aa)/(bb): r/(1+r) and (1-r)/(1+r)
    c->canon.s0 = r / (1.0 + r);
    c->canon.s1 = (1.0 - r) / (1.0 + r);
    c->canon.beta_l = c->beta_l;
    c->canon.beta_r = c->beta_r;

    ge::tb_fill_base(r, c->beta_l, c->beta_r, c->prec == GE_F64 ? 0 : (c->prec == GE_F32 ? 1 : 2), &c->tb,
                     &c->onepg_lo);
}

ge_status make_tensor_maps(ge_ctx *c)
{
    auto enc = tensor_map_encoder();
    if (!enc)
        return fail(GE_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
    const int K = elems_per_row(c->prec);
    for (int b = 0; b < 2; ++b) {
        cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)c->n_rows};
        cuuint64_t strides[1] = {(cuuint64_t)ge::kRowBytes};
        cuuint32_t box[2] = {(cuuint32_t)K, (cuuint32_t)ge::kTileRows};
        cuuint32_t estr[2] = {1, 1};
        CUresult r = enc(&c->tmap[b],
                         c->prec == GE_F64 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                         2, c->buf[b], dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS)
            return fail(GE_ECUDA, "cuTensorMapEncodeTiled failed (CUresult %d)", (int)r);
    }
    return GE_OK;
}

bool valid_prec(int p) { return p == GE_F64 || p == GE_F32 || p == GE_F32_COMP; }
bool valid_kernel(int k)
{
    return k == GE_KERNEL_AUTO || k == GE_KERNEL_CANONICAL || k == GE_KERNEL_ONESTEP ||
           k == GE_KERNEL_TEMPORAL || k == GE_KERNEL_TEMPORAL_DF;
}

void df_split(double x, float *pair) { ge::df_split_host(x, pair); }
int df_code_of(double x) { return ge::df_code_host(x); }

// Launch-independent fields of the double-float kernel.  The scaled map's
// growth per step is exactly 1 + g with g = g_hi + g_lo the pair the kernel
// holds; the host's scale mirror (growth_lo) and the singleton factor use
// that g.  Rescalings keep the FP32 headroom.
ge::TbParams df_params(const ge_ctx *c, double *growth_lo)
{
    ge::TbParams p = c->tb;
    const double r = c->r;
    df_split(2.0 * r, p.dfc[0]);
    p.df_gl = p.dfc[0][1] != 0.0f;
    const double g = (double)p.dfc[0][0] + (double)p.dfc[0][1];
    p.onepg = 1.0 + g;
    const double bb = p.onepg - 1.0;  // TwoSum: onepg + lo == 1 + g exactly
    *growth_lo = (1.0 - (p.onepg - bb)) + (g - bb);
    df_split((1.0 + g) * ((1.0 - r) / (1.0 + r)), p.dfc[1]);
    df_split(r, p.dfc[2]);
    df_split(1.0 - r, p.dfc[3]);
    const int every = (int)std::floor(GE_F32_HEADROOM / std::log2(1.0 + 2.0 * r));
    p.rescale_every = every < 1 ? 1 : every;
    p.df_code = c->err_dev + 32;
    return p;
}

// Depth of the tiled kernel from the tuning table named by GE_TUNE_TABLE
// (lines "<f64|f32|f32c> <n_min> <n_max> <depth>", '#' starts a comment,
// the first matching line wins, malformed lines are skipped); 0 = none.
int table_depth(ge_precision prec, int64_t n)
{
    const char *path = std::getenv("GE_TUNE_TABLE");
    if (!path || !*path)
        return 0;
    FILE *f = std::fopen(path, "r");
    if (!f)
        return 0;
    char line[256];
    int found = 0;
    while (!found && std::fgets(line, sizeof(line), f)) {
        char p[16];
        long long lo = 0, hi = 0;
        int d = 0;
        if (line[0] == '#' || std::sscanf(line, "%15s %lld %lld %d", p, &lo, &hi, &d) != 4)
            continue;
        const int pp = !std::strcmp(p, "f64") ? GE_F64 : !std::strcmp(p, "f32") ? GE_F32
                       : !std::strcmp(p, "f32c") ? GE_F32_COMP : -1;
        if (pp == (int)prec && n >= lo && n <= hi && d >= 1 && d <= kMaxDepth)
            found = d;
    }
    std::fclose(f);
    return found;
}

int effective_depth(const ge_ctx *c)
{
    if (c->depth)
        return c->depth;
    if (c->kernel == GE_KERNEL_TEMPORAL_DF)
        return kDefaultDepthDf;
    return (c->prec == GE_F64) ? kDefaultDepthF64 : kDefaultDepthF32;
}

// Where the tiled kernel runs (grid_cap aside).
ge::TbTarget tiled_target(const ge_ctx *c)
{
    ge::TbTarget t{};
    t.tmap[0] = &c->tmap[0];
    t.tmap[1] = &c->tmap[1];
    t.buf[0] = c->buf[0];
    t.buf[1] = c->buf[1];
    t.n = c->n;
    t.n_rows = c->n_rows;
    t.err = c->err_dev;
    t.tile_ctr = c->err_dev + 48;  // two tile-queue words (48, 49)
    return t;
}

// Advance `steps` steps with the tiled kernel, `depth` steps per launch
// (df: the double-float kernel, after its per-call prescale); the launches
// and the scale mirror are planned by ge::tb_run.
ge_status run_tiled(ge_ctx *c, int64_t steps, int depth, bool df = false)
{
    double growth_lo = c->onepg_lo;
    const ge::TbParams base = df ? df_params(c, &growth_lo) : c->tb;
    const int prec = c->prec == GE_F64 ? 0 : (c->prec == GE_F32 ? 1 : 2);
    if (df) {
        // the prescale 2^-e0 of this call: data and walls below 1 in magnitude
        const int wl = df_code_of(c->beta_l), wr = df_code_of(c->beta_r);
        cudaError_t e = ge::df_prescale(c->buf[c->cur], c->n, wl > wr ? wl : wr, c->err_dev + 32, c->stream);
        if (e != cudaSuccess)
            return cuda_fail(e, "double-float prescale launch");
    }
    ge::TbTarget t = tiled_target(c);
    t.grid_cap = (long long)c->num_sms * (df ? c->tb_df_blocks_per_sm : c->tb_blocks_per_sm);
    const cudaError_t e = ge::tb_run(t, base, growth_lo, df, prec, &c->cur, c->step, steps, depth, c->stream);
    if (e == cudaErrorInvalidValue)
        return fail(GE_EINVAL, "depth %d does not fit a tile", depth);
    if (e != cudaSuccess)
        return cuda_fail(e, "tiled GE kernel launch");
    return GE_OK;
}

// Composed steps (ge_prop.h); *taken = 0 when this call keeps the tiled kernel.
// build: only put the operators the call needs on the stream.
ge_status run_composed(ge_ctx *c, int64_t steps, int *taken, bool build = false)
{
    *taken = 0;
    // a requested stall times out tile loads: the tiled kernel's
    if (c->tb.stall > 0 || !ge::prop_takes(c->n, c->r, steps, c->prec == GE_F64 ? 0 : (c->prec == GE_F32 ? 1 : 2)))
        return GE_OK;
    ge::PropTarget t{};
    t.buf[0] = c->buf[0];
    t.buf[1] = c->buf[1];
    t.n = c->n;
    t.r = c->r;
    t.beta_l = c->beta_l;
    t.beta_r = c->beta_r;
    t.f64 = c->prec == GE_F64;
    t.num_sms = c->num_sms;
    t.err = c->err_dev;
    t.tiled = tiled_target(c);
    t.base = &c->tb;
    t.growth_lo = c->onepg_lo;
    t.prec = c->prec == GE_F64 ? 0 : (c->prec == GE_F32 ? 1 : 2);
    t.depth = effective_depth(c);
    t.rounds_grid = c->num_sms * c->tb_rounds_per_sm;
    const cudaError_t e = ge::prop_run(&c->prop, t, &c->cur, c->step, steps, taken, c->stream, build);
    return e == cudaSuccess ? GE_OK : cuda_fail(e, "composed-step kernel launch");
}

// General sub-domain width k (ge_sweep.cu): up to `depth` steps per launch on
// a tile in shared memory (multi), else, or where the width leaves too few
// units per tile, one launch per step.
ge_status run_sweep(ge_ctx *c, int64_t steps, bool multi, int depth)
{
    for (int64_t s = 0; s < steps;) {
        const int parity = (int)((c->step + s) & 1);
        cudaError_t e;
        if (multi) {
            const int want = (int)((steps - s) < depth ? (steps - s) : depth);
            int done = 0;
            if (c->prec == GE_F64)
                e = ge::launch_sweep_tb_f64(static_cast<const double *>(c->buf[c->cur]),
                                            static_cast<double *>(c->buf[c->cur ^ 1]), c->n, parity, c->width,
                                            want, c->canon, &done, c->stream);
            else
                e = ge::launch_sweep_tb_f32(static_cast<const float *>(c->buf[c->cur]),
                                            static_cast<float *>(c->buf[c->cur ^ 1]), c->n, parity, c->width,
                                            want, c->canon, &done, c->stream);
            if (e != cudaSuccess)
                return cuda_fail(e, "sub-domain sweep kernel launch");
            if (done > 0) {
                c->cur ^= 1;
                s += done;
                continue;
            }
        }
        if (c->prec == GE_F64)
            e = ge::launch_sweep_f64(static_cast<const double *>(c->buf[c->cur]),
                                     static_cast<double *>(c->buf[c->cur ^ 1]), c->n, parity, c->width,
                                     c->canon, c->stream);
        else
            e = ge::launch_sweep_f32(static_cast<const float *>(c->buf[c->cur]),
                                     static_cast<float *>(c->buf[c->cur ^ 1]), c->n, parity, c->width,
                                     c->canon, c->stream);
        if (e != cudaSuccess)
            return cuda_fail(e, "sub-domain sweep kernel launch");
        c->cur ^= 1;
        ++s;
    }
    return GE_OK;
}

ge_status run_canonical(ge_ctx *c, int64_t steps)
{
    for (int64_t s = 0; s < steps; ++s) {
        const int parity = (int)((c->step + s) & 1);
        cudaError_t e;
        if (c->prec == GE_F64)
            e = ge::launch_canon_f64(static_cast<const double *>(c->buf[c->cur]),
                                     static_cast<double *>(c->buf[c->cur ^ 1]), c->n, parity, c->canon,
                                     c->stream);
        else
            e = ge::launch_canon_f32(static_cast<const float *>(c->buf[c->cur]),
                                     static_cast<float *>(c->buf[c->cur ^ 1]), c->n, parity, c->canon,
                                     c->stream);
        if (e != cudaSuccess)
            return cuda_fail(e, "canonical GE kernel launch");
        c->cur ^= 1;
    }
    return GE_OK;
}

// A context's memory, from a pool of its own per device: cudaMalloc and
// cudaFree of 20 MB took 125 us of a one-shot solve's 495.  The pool keeps at
// most kPoolKeep bytes between contexts, and none once an allocation of the
// library fails (it is trimmed, and the allocation tried again); larger
// contexts, and streams that are being captured, use cudaMalloc.
constexpr size_t kPoolKeep = (size_t)64 << 20;

cudaMemPool_t ctx_pool(int device, bool make)
{
    static std::mutex lock;
    static cudaMemPool_t pool[64];
    static bool tried[64];
    if (device < 0 || device >= 64)
        return nullptr;
    std::lock_guard<std::mutex> hold(lock);
    if (!tried[device] && make) {
        tried[device] = true;
        cudaMemPoolProps p{};
        p.allocType = cudaMemAllocationTypePinned;
        p.location.type = cudaMemLocationTypeDevice;
        p.location.id = device;
        cuuint64_t keep = kPoolKeep;
        if (cudaMemPoolCreate(&pool[device], &p) != cudaSuccess) {
            pool[device] = nullptr;
            cudaGetLastError();
        } else if (cudaMemPoolSetAttribute(pool[device], cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            cudaMemPoolDestroy(pool[device]);
            pool[device] = nullptr;
            cudaGetLastError();
        }
    }
    return pool[device];
}

cudaError_t ctx_alloc(ge_ctx *c, char **mem, size_t bytes)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaMemPool_t pool = bytes <= kPoolKeep ? ctx_pool(c->device, true) : nullptr;
    if (pool && cudaStreamIsCapturing(c->stream, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
        if (cudaMallocFromPoolAsync(reinterpret_cast<void **>(mem), bytes, pool, c->stream) == cudaSuccess) {
            c->pooled = true;
            return cudaSuccess;
        }
        cudaGetLastError();
    }
    return ge::device_malloc(reinterpret_cast<void **>(mem), bytes);
}

// The context's memory is one allocation, buf[0].  Its stream's work, and a
// graph captured from it that runs on any other stream, may still use it:
// cudaFree waits for the device, but not for memory from a pool, so that is
// waited for here, on the context's device and without touching its stream
// (the caller may have destroyed it).  idle: nothing of the context can be
// running, and its stream is the caller's of this very call.
void release(ge_ctx *c, bool idle = false)
{
    if (!c)
        return;
    if (c->buf[0] && c->pooled && idle) {
        if (cudaFreeAsync(c->buf[0], c->stream) != cudaSuccess)
            cudaGetLastError();
    } else if (c->buf[0]) {
        int dev = c->device;
        cudaGetDevice(&dev);
        if (dev != c->device)
            cudaSetDevice(c->device);
        // (memory that may be in use is never given back)
        if (!c->pooled || cudaDeviceSynchronize() == cudaSuccess)
            cudaFree(c->buf[0]);
        if (dev != c->device)
            cudaSetDevice(dev);
    }
    if (c->prop.pins)
        c->prop.pins->drop();
    delete c;
}

// A stream of the library's own, for copies beside a context's stream.
cudaError_t side_stream(int device, cudaStream_t *s)
{
    static std::mutex lock;
    static cudaStream_t streams[64];
    if (device < 0 || device >= 64)
        return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> hold(lock);
    cudaError_t e = cudaSuccess;
    if (!streams[device])
        e = cudaStreamCreateWithFlags(&streams[device], cudaStreamNonBlocking);
    *s = streams[device];
    return e;
}

}  // namespace

cudaError_t ge::device_malloc(void **p, size_t bytes)
{
    cudaError_t e = cudaMalloc(p, bytes);
    int dev = 0;
    if (e != cudaErrorMemoryAllocation || cudaGetDevice(&dev) != cudaSuccess)
        return e;
    cudaMemPool_t pool = ctx_pool(dev, false);
    if (!pool)
        return e;
    cudaGetLastError();
    cudaMemPoolTrimTo(pool, 0);
    return cudaMalloc(p, bytes);
}

extern "C" {

const char *ge_status_str(ge_status s)
{
    switch (s) {
    case GE_OK: return "GE_OK";
    case GE_EINVAL: return "GE_EINVAL";
    case GE_ENOMEM: return "GE_ENOMEM";
    case GE_ECUDA: return "GE_ECUDA";
    case GE_ETIMEOUT: return "GE_ETIMEOUT";
    case GE_ENONFINITE: return "GE_ENONFINITE";
    }
    return "GE_UNKNOWN";
}

const char *ge_last_error(void) { return g_last_error; }

ge_status ge_create(ge_ctx **out, int64_t n, double r, double beta_l, double beta_r, ge_precision prec,
                    const void *u0_dev, void *stream)
{
    if (out == nullptr)
        return fail(GE_EINVAL, "ge_create: out is NULL");
    *out = nullptr;
    if (n < 1)
        return fail(GE_EINVAL, "ge_create: n = %lld, need n >= 1", (long long)n);
    if (!(r > 0.0) || !std::isfinite(r))
        return fail(GE_EINVAL, "ge_create: r = %g, need a finite r > 0", r);
    if (!std::isfinite(beta_l) || !std::isfinite(beta_r))
        return fail(GE_EINVAL, "ge_create: wall values must be finite");
    if (!valid_prec(prec))
        return fail(GE_EINVAL, "ge_create: unknown precision %d", (int)prec);
    const int K = elems_per_row(prec);
    const int64_t n_rows = (n + K - 1) / K;
    if (n_rows >= (1LL << 31) - 2 * ge::kTileRows)
        return fail(GE_EINVAL, "ge_create: n = %lld is too large", (long long)n);

    ge_ctx *c = new (std::nothrow) ge_ctx();
    if (c)
        c->prop.pins = ge::PropPins::make();
    if (!c || !c->prop.pins) {
        release(c);
        return fail(GE_ENOMEM, "ge_create: host allocation failed");
    }
    c->n = n;
    c->r = r;
    c->beta_l = beta_l;
    c->beta_r = beta_r;
    c->prec = prec;
    c->stream = static_cast<cudaStream_t>(stream);
    c->n_rows = n_rows;
    cudaError_t e = cudaGetDevice(&c->device);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, c->device);
    if (e != cudaSuccess) {
        release(c);
        return cuda_fail(e, "ge_create: device query");
    }
    // one allocation for the two buffers, the error words and the composed
    // steps' arrays (allocations and frees are most of a one-shot solve's
    // set-up); the arrays need no initial values
    const size_t bytes = ((size_t)n_rows * ge::kRowBytes + 255) & ~(size_t)255;
    char *mem = nullptr;
    e = ctx_alloc(c, &mem, 2 * bytes + 256 + ge::prop_bytes(n, prec == GE_F64));
    if (e != cudaSuccess) {
        release(c);
        return cuda_fail(e, "ge_create: device allocation");
    }
    c->buf[0] = mem;
    c->buf[1] = mem + bytes;
    c->err_dev = reinterpret_cast<int *>(mem + 2 * bytes);
    e = cudaMemsetAsync(mem, 0, 2 * bytes + 256, c->stream);
    if (e == cudaSuccess && u0_dev)
        e = cudaMemcpyAsync(c->buf[0], u0_dev, (size_t)n * elem_size(prec), cudaMemcpyDeviceToDevice,
                            c->stream);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        release(c);
        return cuda_fail(e, "ge_create: initialising buffers");
    }
    ge::prop_carve(&c->prop, reinterpret_cast<char *>(c->err_dev) + 256, n, prec == GE_F64);
    fill_coefficients(c);
    c->depth = table_depth(prec, n);
    ge_status st = make_tensor_maps(c);
    if (st != GE_OK) {
        release(c);
        return st;
    }
    const int prec_idx = prec == GE_F64 ? 0 : (prec == GE_F32 ? 1 : 2);
    e = ge::tb_occupancy(prec_idx, &c->tb_blocks_per_sm);
    if (e == cudaSuccess)
        e = ge::tb_rounds_occupancy(prec_idx, &c->tb_rounds_per_sm);
    if (e == cudaSuccess)
        e = ge::prop_prepare();
    if (e == cudaSuccess && prec == GE_F64) {
        e = ge::tb_df_occupancy(&c->tb_df_blocks_per_sm);
        if (e == cudaSuccess && c->tb_df_blocks_per_sm < 1)
            e = cudaErrorInvalidConfiguration;
    }
    if (e != cudaSuccess || c->tb_blocks_per_sm < 1) {
        release(c);
        return cuda_fail(e == cudaSuccess ? cudaErrorInvalidConfiguration : e,
                         "ge_create: tiled kernel occupancy");
    }
    *out = c;
    return GE_OK;
}

ge_status ge_set_kernel(ge_ctx *c, ge_kernel kernel, int32_t depth)
{
    if (!c)
        return fail(GE_EINVAL, "ge_set_kernel: ctx is NULL");
    if (!valid_kernel(kernel))
        return fail(GE_EINVAL, "ge_set_kernel: unknown kernel %d", (int)kernel);
    if (depth < 0 || depth > kMaxDepth)
        return fail(GE_EINVAL, "ge_set_kernel: depth %d outside 0..%d", (int)depth, kMaxDepth);
    if (kernel == GE_KERNEL_CANONICAL && c->prec == GE_F32_COMP)
        return fail(GE_EINVAL, "ge_set_kernel: the canonical kernel has no compensated variant");
    if (kernel == GE_KERNEL_TEMPORAL_DF && c->prec != GE_F64)
        return fail(GE_EINVAL, "ge_set_kernel: the double-float kernel needs a GE_F64 context");
    if (kernel == GE_KERNEL_TEMPORAL_DF && c->r > kDfMaxR)
        return fail(GE_EINVAL, "ge_set_kernel: the double-float kernel takes r <= 2^20 (r = %g)", c->r);
    c->kernel = kernel;
    c->depth = depth;
    return GE_OK;
}

ge_status ge_set_int_pipes(ge_ctx *c, int32_t on)
{
    if (!c || (on != 0 && on != 1))
        return fail(GE_EINVAL, "ge_set_int_pipes: NULL ctx or on not 0/1");
    c->tb.emu = on;
    return GE_OK;
}

ge_status ge_get_kernel(const ge_ctx *c, ge_kernel *kernel, int32_t *depth)
{
    if (!c || !kernel || !depth)
        return fail(GE_EINVAL, "ge_get_kernel: NULL argument");
    *kernel = c->kernel;
    *depth = effective_depth(c);
    return GE_OK;
}

ge_status ge_tune(ge_ctx *c, int64_t steps, int32_t *best_depth)
{
    if (!c || steps < 1)
        return fail(GE_EINVAL, "ge_tune: NULL ctx or steps < 1");
    if (c->width > 1 || c->kernel == GE_KERNEL_CANONICAL || c->kernel == GE_KERNEL_ONESTEP) {
        if (best_depth)
            *best_depth = effective_depth(c);
        return GE_OK;  // nothing to tune
    }
    ge::NvtxRange nvtx("ge_tune");
    static const int cand64[] = {24, 32, 48, 64, 96};
    static const int cand32[] = {64, 96, 128, 192, 256};
    static const int cand_df[] = {32, 48, 64, 96, 128};
    const bool df = c->kernel == GE_KERNEL_TEMPORAL_DF;
    const int *cand = df ? cand_df : (c->prec == GE_F64 ? cand64 : cand32);
    const size_t bytes = (size_t)c->n * elem_size(c->prec);
    void *saved = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = ge::device_malloc(&saved, bytes);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(saved, c->buf[c->cur], bytes, cudaMemcpyDeviceToDevice, c->stream);
    if (e == cudaSuccess)
        e = cudaEventCreate(&e0);
    if (e == cudaSuccess)
        e = cudaEventCreate(&e1);
    const int64_t step0 = c->step;
    double best = 1e300;
    int best_d = effective_depth(c);
    ge_status st = GE_OK;
    for (int i = 0; i < 5 && e == cudaSuccess && st == GE_OK; ++i) {
        // one untimed run (first use of the launch shape), then a timed one,
        // each from the saved state and step counter
        for (int rep = 0; rep < 2 && e == cudaSuccess && st == GE_OK; ++rep) {
            e = cudaMemcpyAsync(c->buf[c->cur], saved, bytes, cudaMemcpyDeviceToDevice, c->stream);
            c->step = step0;
            if (e == cudaSuccess && rep == 1)
                e = cudaEventRecord(e0, c->stream);
            if (e == cudaSuccess)
                st = run_tiled(c, steps, cand[i], df);
            if (e == cudaSuccess && st == GE_OK && rep == 1)
                e = cudaEventRecord(e1, c->stream);
        }
        float ms = 0.0f;
        if (e == cudaSuccess && st == GE_OK)
            e = cudaEventSynchronize(e1);
        if (e == cudaSuccess && st == GE_OK)
            e = cudaEventElapsedTime(&ms, e0, e1);
        if (e == cudaSuccess && st == GE_OK && ms < best) {
            best = ms;
            best_d = cand[i];
        }
    }
    // the state and the step counter as they were
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->buf[c->cur], saved, bytes, cudaMemcpyDeviceToDevice, c->stream);
    c->step = step0;
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(c->stream);
    if (e0)
        cudaEventDestroy(e0);
    if (e1)
        cudaEventDestroy(e1);
    if (saved)
        cudaFree(saved);
    if (st != GE_OK)
        return st;
    if (e != cudaSuccess)
        return cuda_fail(e, "ge_tune");
    c->depth = best_d;
    if (best_depth)
        *best_depth = best_d;
    return GE_OK;
}

ge_status ge_set_subdomain_width(ge_ctx *c, int64_t k)
{
    if (!c)
        return fail(GE_EINVAL, "ge_set_subdomain_width: ctx is NULL");
    if (k < 1)
        return fail(GE_EINVAL, "ge_set_subdomain_width: k = %lld, need k >= 1", (long long)k);
    if (k > 1 && c->prec == GE_F32_COMP)
        return fail(GE_EINVAL, "ge_set_subdomain_width: no compensated variant for k > 1");
    c->width = k;
    return GE_OK;
}

ge_status ge_step_n(ge_ctx *c, int64_t steps)
{
    ge::NvtxRange nvtx("ge_step_n");
    if (!c)
        return fail(GE_EINVAL, "ge_step_n: ctx is NULL");
    if (steps < 0)
        return fail(GE_EINVAL, "ge_step_n: steps = %lld < 0", (long long)steps);
    if (steps == 0)
        return GE_OK;
    ge_status st;
    if (c->width > 1) {
        const bool multi = c->kernel != GE_KERNEL_CANONICAL && c->kernel != GE_KERNEL_ONESTEP;
        st = run_sweep(c, steps, multi, c->depth ? c->depth : ge::sweep_tb_depth(c->n, c->width, (int)elem_size(c->prec), c->num_sms));
        if (st == GE_OK)
            c->step += steps;
        return st;
    }
    switch (c->kernel) {
    case GE_KERNEL_CANONICAL:
        st = run_canonical(c, steps);
        break;
    case GE_KERNEL_ONESTEP:
        st = run_tiled(c, steps, 1);
        break;
    case GE_KERNEL_TEMPORAL_DF:
        st = run_tiled(c, steps, effective_depth(c), true);
        break;
    default: {
        int taken = 0;
        st = c->kernel == GE_KERNEL_AUTO ? run_composed(c, steps, &taken) : GE_OK;
        if (st == GE_OK && !taken)
            st = run_tiled(c, steps, effective_depth(c));
    }
    }
    if (st == GE_OK)
        c->step += steps;
    return st;
}

ge_status ge_read_state(ge_ctx *c, void *out_dev)
{
    if (!c || !out_dev)
        return fail(GE_EINVAL, "ge_read_state: NULL argument");
    cudaError_t e = cudaMemcpyAsync(out_dev, c->buf[c->cur], (size_t)c->n * elem_size(c->prec),
                                    cudaMemcpyDeviceToDevice, c->stream);
    return e == cudaSuccess ? GE_OK : cuda_fail(e, "ge_read_state");
}

ge_status ge_write_state(ge_ctx *c, const void *in_dev, int64_t step_count)
{
    if (!c || !in_dev)
        return fail(GE_EINVAL, "ge_write_state: NULL argument");
    if (step_count < 0)
        return fail(GE_EINVAL, "ge_write_state: step_count < 0");
    cudaError_t e = cudaMemcpyAsync(c->buf[c->cur], in_dev, (size_t)c->n * elem_size(c->prec),
                                    cudaMemcpyDeviceToDevice, c->stream);
    if (e == cudaSuccess)  // a new state: earlier device failures no longer apply
        e = cudaMemsetAsync(c->err_dev, 0, sizeof(int), c->stream);
    if (e != cudaSuccess)
        return cuda_fail(e, "ge_write_state");
    c->step = step_count;
    return GE_OK;
}

ge_status ge_read_range(ge_ctx *c, int64_t offset, int64_t count, void *out_dev)
{
    if (!c || (!out_dev && count > 0))
        return fail(GE_EINVAL, "ge_read_range: NULL argument");
    if (offset < 0 || count < 0 || offset > c->n - count)
        return fail(GE_EINVAL, "ge_read_range: points [%lld, %lld) outside 0..%lld", (long long)offset,
                    (long long)(offset + count), (long long)c->n);
    if (count == 0)
        return GE_OK;
    const size_t es = elem_size(c->prec);
    cudaError_t e = cudaMemcpyAsync(out_dev, static_cast<const char *>(c->buf[c->cur]) + offset * es,
                                    (size_t)count * es, cudaMemcpyDeviceToDevice, c->stream);
    return e == cudaSuccess ? GE_OK : cuda_fail(e, "ge_read_range");
}

ge_status ge_write_range(ge_ctx *c, int64_t offset, int64_t count, const void *in_dev)
{
    if (!c || (!in_dev && count > 0))
        return fail(GE_EINVAL, "ge_write_range: NULL argument");
    if (offset < 0 || count < 0 || offset > c->n - count)
        return fail(GE_EINVAL, "ge_write_range: points [%lld, %lld) outside 0..%lld", (long long)offset,
                    (long long)(offset + count), (long long)c->n);
    if (count == 0)
        return GE_OK;
    const size_t es = elem_size(c->prec);
    cudaError_t e = cudaMemcpyAsync(static_cast<char *>(c->buf[c->cur]) + offset * es, in_dev, (size_t)count * es,
                                    cudaMemcpyDeviceToDevice, c->stream);
    return e == cudaSuccess ? GE_OK : cuda_fail(e, "ge_write_range");
}

ge_status ge_debug_stall(ge_ctx *c, int64_t cycles)
{
    if (!c || cycles < 0)
        return fail(GE_EINVAL, "ge_debug_stall: NULL ctx or cycles < 0");
    c->tb.stall = (long long)cycles;
    return GE_OK;
}

ge_status ge_get_step(const ge_ctx *c, int64_t *step_count)
{
    if (!c || !step_count)
        return fail(GE_EINVAL, "ge_get_step: NULL argument");
    *step_count = c->step;
    return GE_OK;
}

ge_status ge_sync(ge_ctx *c)
{
    if (!c)
        return fail(GE_EINVAL, "ge_sync: ctx is NULL");
    cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess)
        return cuda_fail(e, "ge_sync");
    int word = 0;
    e = cudaMemcpy(&word, c->err_dev, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess)
        return cuda_fail(e, "ge_sync: reading the device error word");
    if (word == ge::kDevTimeout)
        return fail(GE_ETIMEOUT, "a tile load did not complete within the wait limit");
    return GE_OK;
}

void ge_destroy(ge_ctx *c)
{
    if (!c)
        return;
    release(c);
}

ge_status ge_solve(int64_t n, double r, double beta_l, double beta_r, ge_precision prec, ge_kernel kernel,
                   int32_t depth, int64_t steps, const void *u0_host, void *u_out_host, void *stream)
{
    ge::NvtxRange nvtx("ge_solve");
    if (!u0_host || !u_out_host)
        return fail(GE_EINVAL, "ge_solve: NULL host buffer");
    if (steps < 0)
        return fail(GE_EINVAL, "ge_solve: steps < 0");
    ge_ctx *c = nullptr;
    ge_status st = ge_create(&c, n, r, beta_l, beta_r, prec, nullptr, stream);
    if (st != GE_OK)
        return st;
    const size_t bytes = (size_t)n * elem_size(prec);
    // the operators of composed steps do not depend on the data: they are
    // built while it is copied (145 us of kernels beside 65 us for 8 MB)
    int building = 0;
    cudaError_t e = cudaSuccess;
    st = ge_set_kernel(c, kernel, depth);
    if (st == GE_OK && c->kernel == GE_KERNEL_AUTO && steps > 0)
        st = run_composed(c, steps, &building, true);
    if (st == GE_OK) {
        cudaStream_t side = c->stream;
        cudaEvent_t copied = nullptr;
        if (building && (cudaEventCreateWithFlags(&copied, cudaEventDisableTiming) != cudaSuccess ||
                         side_stream(c->device, &side) != cudaSuccess)) {
            cudaGetLastError();
            side = c->stream;
        }
        e = cudaMemcpyAsync(c->buf[c->cur], u0_host, bytes, cudaMemcpyHostToDevice, side);
        if (e == cudaSuccess && side != c->stream) {
            e = cudaEventRecord(copied, side);
            if (e == cudaSuccess)
                e = cudaStreamWaitEvent(c->stream, copied, 0);
            if (e != cudaSuccess)
                cudaStreamSynchronize(side);
        }
        if (copied)
            cudaEventDestroy(copied);
        if (e != cudaSuccess) {
            ge_destroy(c);
            return cuda_fail(e, "ge_solve: host to device copy");
        }
        st = ge_step_n(c, steps);
    }
    if (st == GE_OK) {
        e = cudaMemcpyAsync(u_out_host, c->buf[c->cur], bytes, cudaMemcpyDeviceToHost, c->stream);
        if (e != cudaSuccess)
            st = cuda_fail(e, "ge_solve: device to host copy");
    }
    if (st == GE_OK)
        st = ge_sync(c);
    release(c, st == GE_OK);
    return st;
}

}  // extern "C"

// ge_prop_plan.cpp -- host-side planning of composed steps (ge_prop.h): how a
// call's steps are cut into operators, which operators a context keeps, and
// the launches.  Host code only; built with -ffp-contract=off so the
// coefficients are rounded exactly as written.
#include "ge_prop.h"

#include <algorithm>
#include <cmath>
#include <new>

namespace ge {

namespace {

constexpr long long kMinPoints = 16;
// mesh ratios far outside any use keep the step-by-step kernels
constexpr double kMinR = 1e-6, kMaxR = 1e6;
constexpr int kMaxChain = 8190;    // block steps per operator (the cone scan of a tile grows with it)

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// Bytes of the arrays of a context.
struct Sizes {
    int rcap, hs;
    size_t e, h, F, tab, hdr, x, list;
    Sizes(long long n, int f64)
    {
        const long long most = f64 ? kPropR64Max : kPropRMax;
        rcap = (int)((std::min(n, most) + 15) & ~15LL);
        hs = rcap + 8;
        e = align256((size_t)(2 * rcap + 16) * 8);
        h = align256((size_t)4 * hs * 8);
        F = align256((size_t)2 * hs * 8);
        tab = n < kPropTileMin ? 0 : align256(f64 ? kPropTab64 : kPropTab32);
        hdr = align256(sizeof(PropHeader));
        x = n < kPropTileMin ? 0 : align256((size_t)4 * (2 * rcap + 9) * 8) + 256;
        list = align256((size_t)(n / kPropBlk + 1) * sizeof(int));
    }
    size_t set() const { return e + h + F + tab + hdr; }
    size_t scratch() const { return 2 * (e + h); }
    size_t total() const { return kPropSets * set() + 2 * scratch() + x + list + 256; }
};

// Largest operator.  Its taps are a bell of standard deviation sqrt(2 r k)
// cut off at the cone k + 1, and the tap tables with the tile's digits have
// to fit one CTA's shared memory: r k <= 1512 (FP64: sigma 55, digits out to
// 9 sigma) or 7200 (FP32: sigma 120, four digits, out to 6.7 sigma); where
// the cone is the smaller, k <= 330 or 990 at any r.
int max_chain(double r, int f64, long long n)
{
    const double rk = f64 ? 1512.0 : 7200.0;
    double k = std::max(rk / r, f64 ? 330.0 : 990.0);
    k = std::min(k, (double)kMaxChain);
    k = std::min(k, (double)(n - 2));
    return (int)k & ~1;
}

// Reach of the FP64 taps: 12 standard deviations (the rest is below 2^-100).
// (At most 704 for FP64 and 1472 for FP32 by the limits above.)
int reach(double r, int k)
{
    const double s = 12.0 * std::sqrt(2.0 * r * (double)k) + 32.0;
    return (int)std::min((double)(k + 1), s);
}

// Reach of the digits (see max_chain), rounded up to whole blocks.
int halo_blocks(double r, int k, int f64)
{
    const double s = (f64 ? 9.2 : 7.0) * std::sqrt(2.0 * r * (double)k) + 24.0;
    const int w = (int)std::min((double)(k + 4), s);
    const int hb = (w + 15 + kPropBlk) / kPropBlk;
    return std::min(hb, f64 ? kPropHb64 : kPropHb32);
}

// Which blocks of a tile are left to dot products (PropRun::range, near).
// Values are held to 2^-63 (FP32: 2^-31) of 2^e, the power of two above the
// window's largest, and the rounding of that is smoothed as the values are:
// for taps of standard deviation d its root mean square shrinks by S =
// (2 sqrt(pi) d)^-1/2.  `range` keeps it below 2^-54 (2^-25) of a block's
// largest value, which storing the result may cost as well; where the results
// are looked at (PropHeader::keep), blocks of 2^-4 of that go on to there.
//   Past d = 48 points the steps one by one give a block the errors of the
// blocks beside it (where a smooth field crosses zero, say), and its results
// are looked at together with theirs.
void tile_range(double r, int k, int f64, int *range, int *near)
{
    const double d = std::sqrt(2.0 * r * (double)k);
    const bool bell = k >= 16.0 * r;
    const double s2 = bell ? std::min(1.0, 1.0 / (3.5449 * d)) : 1.0;
    *range = (f64 ? 8 : 5) + (int)std::floor(-0.5 * std::log2(s2));
    *near = bell && d >= 48.0 ? 1 : 0;
}

}  // namespace

PropPins *PropPins::make()
{
    PropPins *p = new (std::nothrow) PropPins();
    for (int i = 0; p && i < kPropSets; ++i)
        p->slot[i].owner = p;
    return p;
}

void PropPins::drop()
{
    if (owners.fetch_sub(1, std::memory_order_acq_rel) == 1)
        delete this;
}

void PropPins::pin(int i, cudaStream_t stream)
{
    Slot *s = &slot[i];
    s->graphs.fetch_add(1, std::memory_order_relaxed);
    owners.fetch_add(1, std::memory_order_relaxed);
    // (called from a thread of CUDA's, where no CUDA call is allowed)
    cudaHostFn_t gone = [](void *p) {
        Slot *s = static_cast<Slot *>(p);
        PropPins *owner = s->owner;
        s->graphs.fetch_sub(1, std::memory_order_release);
        owner->drop();
    };
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaGraph_t graph = nullptr;
    cudaUserObject_t object = nullptr;
    bool held = cudaStreamGetCaptureInfo(stream, &cap, nullptr, &graph, nullptr, nullptr, nullptr) == cudaSuccess && graph &&
                cudaUserObjectCreate(&object, s, gone, 1, cudaUserObjectNoDestructorSync) == cudaSuccess;
    if (held && cudaGraphRetainUserObject(graph, object, 1, cudaGraphUserObjectMove) != cudaSuccess) {
        s->graphs.fetch_add(1, std::memory_order_relaxed);
        owners.fetch_add(1, std::memory_order_relaxed);
        cudaUserObjectRelease(object, 1);
        held = false;
    }
    if (!held)
        cudaGetLastError();  // the operator stays the graph's for the context's life
}

size_t prop_bytes(long long n, int f64) { return Sizes(n, f64).total(); }

void prop_carve(PropState *st, void *mem, long long n, int f64)
{
    const Sizes z(n, f64);
    st->mem = mem;
    st->rcap = z.rcap;
    st->hs = z.hs;
    char *p = static_cast<char *>(mem);
    auto take = [&](size_t b) {
        char *q = p;
        p += b;
        return q;
    };
    for (PropSet &s : st->set) {
        s = PropSet{};
        s.e = reinterpret_cast<double *>(take(z.e)) + z.rcap + 8;
        s.h = reinterpret_cast<double *>(take(z.h));
        s.F = reinterpret_cast<double *>(take(z.F));
        s.tab = reinterpret_cast<unsigned char *>(take(z.tab));
        s.hdr = reinterpret_cast<PropHeader *>(take(z.hdr));
    }
    for (int i = 0; i < 2; ++i)
        st->scratch[i] = reinterpret_cast<double *>(take(z.scratch()));
    st->x = z.x ? reinterpret_cast<double *>(take(z.x)) : nullptr;
    st->list = reinterpret_cast<int *>(take(z.list));
    st->count = reinterpret_cast<int *>(take(256));
}

// Fewest steps a call takes this way: where a context's first call, which
// also builds the operator, is as fast as the tiled kernel's (us, r = 1,
// first call of a fresh context, this way / tiled):
//   dot products alone (n = 2000): FP64 8 steps 41 / 60; FP32 32 steps 54 /
//     53, 64 steps 60 / 69; compensated 32 steps 54 / 59;
//   tiles: FP64 16 steps 88 / 93 (n = 1e5), 92 / 134 (2^20), 452 / 582
//     (2^24), but 8 steps 432 / 419; FP32 128 steps 107 / 125 (2^20) but 150
//     / 115 (2^22) and 306 / 185 (2^24), where an FP32 tile's conversion
//     costs what 200 steps of the FP32 pipes do; compensated 64 steps 95 /
//     102 (2^20), 285 / 253 (2^24), 128 steps 308 / 441.
// Later calls take half of that or less at these step counts.
//   The compensated kernel rounds the state to FP32 where a launch ends, an
// operator where it ends: grids too short for operators of as many steps (n -
// 2 at most) keep the kernel (n = 19, r = 1e-4, 958 steps: 6.6e-8, composed
// 3.4e-7).
bool prop_takes(long long n, double r, long long steps, int prec)
{
    if (n < kMinPoints || r < kMinR || r > kMaxR)
        return false;
    if (prec == 2 && n < kDefaultDepthF32 + 2)
        return false;
    const bool tiles = n >= kPropTileMin;
    long long least;
    if (prec == 0)
        least = tiles ? 20 : 8;
    else if (prec == 1)
        least = tiles ? 128 + n * 192 / (1 << 24) : 48;
    else
        least = tiles ? 64 + n * 48 / (1 << 24) : 32;
    return steps >= least;
}

namespace {

// (high, low) double pair of x / y, y = yh + yl.
void dd_quot(double x, double yh, double yl, double *out)
{
    const double q = x / yh;
    const double rem = std::fma(-q, yh, x) - q * yl;
    out[0] = q;
    out[1] = rem / yh;
}

// (hi + lo) 2^64 for a sum in [0, 1), to the nearest below.
unsigned long long fraction(double hi, double lo)
{
    const double two64 = 18446744073709551616.0;
    const double s = hi * two64, w = std::floor(s);
    const double v = std::floor((s - w) + lo * two64);
    if (w >= two64)
        return v < 0.0 ? 0ull - (unsigned long long)-v : ~0ull;
    return v < 0.0 ? (unsigned long long)w - (unsigned long long)-v : (unsigned long long)w + (unsigned long long)v;
}

// Exponent code (code_of in ge_prop.cu: 0 for zero, else the biased exponent
// of the state's type, at least 1) of what a wall adds to a right-hand side.
int wall_code(double beta, double r, int f64)
{
    if (beta == 0.0)
        return 0;
    int e = 0;
    std::frexp(beta * std::max(1.0, r), &e);
    return f64 ? std::min(std::max(e + 1022, 1), 2046) : std::min(std::max(e + 126, 1), 254);
}

// Build an operator's arrays: a short chain step by step, then binary powering.
cudaError_t build_set(PropState *st, const PropTarget &t, PropSet &s, int pr, int hb, cudaStream_t stream)
{
    const double r = t.r;
    PropCoef c{};
    // 1 + 2r and 1 + r as exact pairs (2r is exact)
    const double d2 = 1.0 + 2.0 * r, b2 = d2 - 1.0, d2l = (1.0 - (d2 - b2)) + (2.0 * r - b2);
    const double d1 = 1.0 + r, b1 = d1 - 1.0, d1l = (1.0 - (d1 - b1)) + (r - b1);
    dd_quot(1.0, d2, d2l, c.al);
    dd_quot(2.0 * r, d2, d2l, c.be);
    // (1 - r) / (1 + r) = 2 / (1 + r) - 1
    double two[2];
    dd_quot(2.0, d1, d1l, two);
    const double k = two[0] - 1.0, kb = k - two[0];
    c.ka[0] = k;
    c.ka[1] = ((two[0] - (k - kb)) + (-1.0 - kb)) + two[1];

    c.be_frac = fraction(c.be[0], c.be[1]);
    c.ka_frac = k < 0.0 ? fraction(-c.ka[0], -c.ka[1]) : fraction(c.ka[0], c.ka[1]);

    const Sizes z(t.n, t.f64);
    PropLevel a{};
    a.hs = z.hs;
    auto arrays = [&](int i, double **e, double **el, double **h, double **hl) {
        char *p = reinterpret_cast<char *>(st->scratch[i]);
        *e = reinterpret_cast<double *>(p) + z.rcap + 8;
        *el = reinterpret_cast<double *>(p + z.e) + z.rcap + 8;
        *h = reinterpret_cast<double *>(p + 2 * z.e);
        *hl = reinterpret_cast<double *>(p + 2 * z.e + z.h);
    };
    double *in[4], *out[4];
    arrays(0, &in[0], &in[1], &in[2], &in[3]);
    arrays(1, &out[0], &out[1], &out[2], &out[3]);
    a.c = c;
    const int Rlim = reach(r, s.k);
    // the leading bits' chain step by step, then a doubling for each bit left
    int levels = 0;
    while ((s.k >> levels) > kPropShort)
        ++levels;
    int k1 = s.k >> levels;
    cudaError_t e = prop_launch_short(in[0], in[1], in[2], in[3], z.hs, k1, c, stream);
    // start parities each level's wall arrays are needed for, from the last
    // level back (a level reads those of its first and of its second half)
    int par[32];
    par[levels] = (1 << s.p0) | (1 << pr);
    for (int l = levels; l > 0; --l) {
        const int half = s.k >> (levels - l + 1), dl = (s.k >> (levels - l)) & 1;
        par[l - 1] = 0;
        for (int p = 0; p < 2; ++p)
            if ((par[l] >> p) & 1)
                par[l - 1] |= (1 << ((p + half + dl) & 1)) | (1 << ((p + dl) & 1));
    }
    auto set_in = [&] {
        a.e0 = in[0];
        a.el0 = k1 == s.k >> levels ? in[1] : nullptr;  // a doubling leaves FP64 taps
        a.h0 = in[2];
        a.hl0 = a.el0 ? in[3] : nullptr;
        a.k1 = k1;
        a.R1 = std::min(k1 + 1, Rlim);
    };
    for (int bit = levels - 1; bit >= 0 && e == cudaSuccess; --bit) {
        set_in();
        a.e1 = out[0];
        a.h1 = out[2];
        a.delta = (s.k >> bit) & 1;
        k1 = 2 * k1 + a.delta;
        a.R2 = std::min(k1 + 1, Rlim);
        a.par = par[levels - bit];
        e = prop_launch_level(a, stream);
        std::swap(in, out);
    }
    if (e != cudaSuccess)
        return e;
    set_in();
    a.e1 = s.e;
    a.h1 = s.h;
    a.par = par[levels];
    PropFinish f{};
    f.k = s.k;
    f.p0 = s.p0;
    f.entry = s.entry;
    f.exit = s.exit;
    f.r = r;
    f.x1 = (1.0 + r) / (1.0 + 2.0 * r);
    f.x2 = r / (1.0 + 2.0 * r);
    f.F = t.beta_l != 0.0 || t.beta_r != 0.0 ? s.F : nullptr;
    if (st->x) {
        f.x = st->x + 32;
        f.x_max = reinterpret_cast<unsigned long long *>(st->x);
        if ((e = cudaMemsetAsync(f.x_max, 0, 8, stream)) != cudaSuccess)
            return e;
    }
    e = prop_launch_finish(a, f, stream);
    if (e == cudaSuccess && f.x)
        e = prop_launch_digits(s, f, a.R1, t.prec, hb, stream);
    return e;
}

}  // namespace

cudaError_t prop_run(PropState *st, const PropTarget &t, int *cur, long long step0, long long steps, int *taken,
                     cudaStream_t stream, bool build_only)
{
    *taken = 0;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(stream, &cap);
    if (e != cudaSuccess)
        return e;
    const bool capturing = cap != cudaStreamCaptureStatusNone;
    const double r = t.r, det = 1.0 + 2.0 * r;
    const int p0 = (int)(step0 & 1), pr = p0 ^ (int)(t.n & 1);

    // entry, steps - 1 block steps, exit: `full` operators of k block steps
    // (k even, so every operator starts at parity p0) and a last one, with
    // the exit, of the rest
    const long long chain = steps - 1;
    const int kmax = max_chain(r, t.f64, t.n);
    if (kmax < 2)
        return cudaSuccess;
    const long long q = (chain + kmax - 1) / kmax;
    long long k = 2 * ((chain + 2 * q - 1) / (2 * q));
    if (k > kmax)
        k = kmax;
    long long full = q > 1 ? chain / k : 0;
    if (q > 1 && full * k == chain)
        --full;
    const int k_last = (int)(chain - full * k);

    // the operators this call needs, each in a slot of its own: the first
    // with the entry, the last with the exit, those between with neither
    struct Need {
        int k, entry, exit;
        PropSet *set;
        bool build;
        int hb;
        bool tiles;
    } need[3];
    int needs = 0;
    if (full > 0)
        need[needs++] = {(int)k, 1, 0, nullptr, false, 0, false};
    if (full > 1)
        need[needs++] = {(int)k, 0, 0, nullptr, false, 0, false};
    need[needs++] = {k_last, full == 0, 1, nullptr, false, 0, false};
    auto holds = [&](const PropSet &s, const Need &w) {
        return s.used && s.k == w.k && s.p0 == p0 && s.entry == w.entry && s.exit == w.exit;
    };
    for (int i = 0; i < needs; ++i)
        for (PropSet &s : st->set)
            if (holds(s, need[i]))
                need[i].set = &s;
    // a slot for each of the others, the least recently used: all of them
    // before any is given up
    for (int i = 0; i < needs; ++i) {
        if (need[i].set)
            continue;
        PropSet *s = nullptr;
        for (int z = 0; z < kPropSets; ++z) {
            PropSet &c = st->set[z];
            bool taken_here = st->pins->pinned(z);
            for (int j = 0; j < needs; ++j)
                taken_here = taken_here || need[j].set == &c;
            if (!taken_here && (!s || c.used < s->used))
                s = &c;
        }
        if (!s)
            return cudaSuccess;  // every slot belongs to a captured graph
        need[i].set = s;
        need[i].build = true;
    }
    for (int i = 0; i < needs; ++i) {
        PropSet &s = *need[i].set;
        if (need[i].build) {
            s.k = need[i].k;
            s.p0 = p0;
            s.entry = need[i].entry;
            s.exit = need[i].exit;
            s.valid = 0;
        }
        // arrays written inside a capture exist only once that graph runs:
        // outside one they count as missing
        need[i].build = !s.valid;
        s.used = ++st->clock;
    }
    const double x2 = r / det;
    for (int i = 0; i < needs; ++i) {
        Need &w = need[i];
        w.hb = halo_blocks(r, w.k, t.f64);
        // away from the walls by the digits' reach; below this size the dot
        // products of all rows take less time than a tile
        w.tiles = t.n >= kPropTileMin && t.n > 2LL * w.hb * kPropBlk + 4 * kPropBlk;
        if (w.build && (e = build_set(st, t, *w.set, pr, w.hb, stream)) != cudaSuccess)
            return e;
        if (capturing)
            st->pins->pin((int)(w.set - st->set), stream);
        else
            w.set->valid = 1;
    }
    *taken = 1;
    if (build_only)
        return cudaSuccess;
    if (need[0].tiles && (e = cudaMemsetAsync(st->count, 0, 2 * sizeof(int), stream)) != cudaSuccess)
        return e;
    for (long long i = 0; i <= full; ++i) {
        const Need &w = i == full ? need[needs - 1] : need[i == 0 ? 0 : 1];
        const PropSet &s = *w.set;
        PropRun a{};
        a.in = t.buf[*cur];
        a.out = t.buf[*cur ^ 1];
        a.n = t.n;
        a.r = r;
        a.x2 = x2;
        a.xs = 1.0 / (1.0 + r);
        a.fl = r * t.beta_l;
        a.fr = r * t.beta_r;
        a.bl = t.beta_l;
        a.br = t.beta_r;
        a.wall_l = wall_code(t.beta_l, r, t.f64);
        a.wall_r = wall_code(t.beta_r, r, t.f64);
        a.k = s.k;
        a.p0 = p0;
        a.pr = pr;
        a.entry = s.entry;
        a.exit = s.exit;
        a.R = reach(r, s.k);
        a.hs = st->hs;
        a.e = s.e;
        a.h = s.h;
        a.F = s.F;
        a.tab = s.tab;
        a.hdr = s.hdr;
        a.err = t.err;
        a.list = st->list;
        a.count = st->count + (i & 1);
        a.count_next = st->count + ((i + 1) & 1);
        long long items;
        if (w.tiles) {
            a.hb = w.hb;
            a.blk0 = a.hb;
            a.blk1 = t.n / kPropBlk - a.hb;
            a.per = t.f64 ? kPropRows64 - 2 * a.hb : kPropTileBlks;
            a.tiles = (a.blk1 - a.blk0 + a.per - 1) / a.per;
            tile_range(r, s.k, t.f64, &a.range, &a.near);
            a.rows_l = a.blk0 * kPropBlk;
            a.row_r = a.blk1 * kPropBlk;
            // listed blocks past which the whole grid step by step is sooner
            // done than their dot products: a block's 64 rows of 2 R taps at
            // 2e11 multiply-adds a second and 85 ns for its eight items' set-up
            // (3 us each on 304 CTAs), against the tiled kernel's rate and its
            // wall tiles' time a step
            const double rate = t.prec == 0 ? 8e11 : t.prec == 1 ? 1.8e13 : 5.8e12, wall = t.prec == 0 ? 4.4e-6 : 0.85e-6;
            const double tiled_s = std::max((double)t.n * s.k / rate, wall * s.k) + 20e-6;
            a.gate_min = (int)std::min(tiled_s / (128.0 * a.R / 2e11 + 85e-9), 2e9);
            const bool gated = a.gate_min < a.blk1 - a.blk0 &&
                               tb_plan_rounds(t.tiled, *t.base, t.growth_lo, t.prec, *cur, p0, s.k, s.entry, s.exit,
                                              t.depth, &st->rounds);
            if (gated) {
                st->rounds.barrier = st->count + 2;
                a.zero[0] = st->count + 2;
                a.zero[1] = t.tiled.tile_ctr;
                a.zero[2] = t.tiled.tile_ctr + 1;
            } else {
                a.gate_min = 2000000000;
            }
            if ((e = prop_launch_tiles(a, t.f64, t.num_sms, stream)) != cudaSuccess)
                return e;
            if (gated) {
                if ((e = launch_tb_rounds(t.prec, t.tiled.tmap[*cur], t.tiled.tmap[*cur ^ 1], st->rounds, a,
                                          t.rounds_grid, stream)) != cudaSuccess)
                    return e;
                *cur ^= 1;
                continue;
            }
            items = 2LL * t.num_sms;
        } else {
            a.rows_l = t.n;
            a.row_r = t.n;
            items = t.n / 8 + 1;
        }
        const int grid = (int)std::min<long long>(items, 8LL * t.num_sms);
        if ((e = prop_launch_dots(a, t.f64, grid, stream)) != cudaSuccess)
            return e;
        *cur ^= 1;
    }
    return cudaSuccess;
}

}  // namespace ge

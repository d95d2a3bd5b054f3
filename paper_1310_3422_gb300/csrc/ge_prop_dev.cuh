// ge_prop_dev.cuh -- rows of a composed operator as FP64 dot products, shared
// by the tiles' kernels (ge_prop.cu) and the step-by-step fallback (ge_tb.cu).
#pragma once

#include "ge_prop.h"

namespace ge {
namespace {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// z 2^e rounded to nearest even, for a normal result, on the integer pipes
// (the conversion instruction runs on the FP64 unit).
__device__ __forceinline__ double fixed_to_double(long long z, int e)
{
    const unsigned long long m = (unsigned long long)(z < 0 ? -z : z);
    const int lead = __clzll((long long)m);                 // 1 .. 63 (64 for zero)
    const unsigned long long w = m << (lead & 63);          // leading one at bit 63
    unsigned long long f = w >> 11;
    const unsigned low = (unsigned)w & 0x7ff;
    f += (low > 0x400 || (low == 0x400 && (f & 1))) ? 1 : 0;
    // exponent field of 2^(63 - lead + e), less the leading one's own unit
    f += (unsigned long long)(unsigned)(1023 + 62 - lead + e) << 52;
    if (m == 0)
        f = 0;
    return __longlong_as_double((long long)(f | ((unsigned long long)z & 0x8000000000000000ull)));
}

// The sum over a warp of P (1 or 2) values a lane, each to 2^-57 of the
// largest, rounded once.  As integers relative to the largest exponent, by
// three reductions of 27 bits each: FP64 additions in a tree round at each of
// its five levels, which was half of a short row's error (24 steps of rough
// data at r = 1: 1.3e-16 where the steps one by one err 1.1e-16), and take
// the FP64 unit 19 cycles each.  Sums that are not finite, or that could
// overflow or be subnormal, take the tree.
template <int P>
__device__ __forceinline__ double warp_sum_rounded_once(const double (&v)[P])
{
    static_assert(P == 1 || P == 2, "the sum of 32 P integers below 2^57 stays below 2^63");
    unsigned code = 0;
#pragma unroll
    for (int p = 0; p < P; ++p)
        code = max(code, ((unsigned)__double2hiint(v[p]) >> 20) & 0x7ff);
    const int ref = (int)__reduce_max_sync(0xffffffffu, code);
    if (ref < 64 || ref >= 2040)
        return warp_sum(P == 2 ? v[0] + v[P - 1] : v[0]);
    unsigned long long y = 0;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const unsigned long long u = (unsigned long long)__double_as_longlong(v[p]);
        const int e = (int)(u >> 52) & 0x7ff;
        unsigned long long m = (u & 0x000fffffffffffffull) | (e ? 0x0010000000000000ull : 0);
        // v = m 2^(e - 1075) = (m 2^(e - ref + 4)) 2^(ref - 1079)
        const int sh = (e ? e : 1) - ref + 4, n = -sh < 60 ? -sh : 60;
        m = sh >= 0 ? m << sh : (m + (1ull << (n - 1))) >> n;
        // (biased: 32 P times 2^59 / P is 2^64, no part of the sum)
        y += (1ull << 59) / P + ((long long)u < 0 ? 0 - m : m);
    }
    const unsigned a = __reduce_add_sync(0xffffffffu, (unsigned)y & 0x7ffffffu);
    const unsigned b = __reduce_add_sync(0xffffffffu, (unsigned)(y >> 27) & 0x7ffffffu);
    const unsigned c = __reduce_add_sync(0xffffffffu, (unsigned)(y >> 54));
    return fixed_to_double((long long)(a + ((unsigned long long)b << 27) + ((unsigned long long)c << 54)), ref - 1079);
}

// ---- reading the state ---------------------------------------------------

// Point j's right-hand side w = u + r (u_partner - u) (+ the wall terms), the
// groups those of parity 1 - p0 -- or the value itself after the first
// operator, when the buffer holds w.  (As (1 - r) u + r u_partner it would
// take the rounding of 1 - r, the same in every row, and of the first product.)
template <typename T>
__device__ __forceinline__ double load_w(const PropRun &P, long long j)
{
    const T *in = static_cast<const T *>(P.in);
    const double u = (double)in[j];
    if (!P.entry)
        return u;
    const long long m = ((j + 1 - P.p0) & 1) ? j - 1 : j + 1;
    double w = fma(P.r, (m >= 0 && m < P.n ? (double)in[m] : 0.0) - u, u);
    if (j == 0)
        w += P.fl;
    if (j == P.n - 1)
        w += P.fr;
    return w;
}

// ---- dot products --------------------------------------------------------

// A few rows of a CTA: the rows near the walls (or all rows of a small grid),
// and the blocks a tile left out.  The window of right-hand sides is staged
// in shared memory as doubles; a row's sum is the work of one warp, or of
// several where there are more warps than rows.  Bound by the FP64 unit (two
// taps' widths of multiply-adds a row; a warp's instruction takes an SM 19
// cycles) and, in a few rows, by latency: loads go out in batches.
//
// FP32 states take the same sum on pairs of FP32 numbers (high + low: taps,
// window and accumulator, the products' and sums' errors kept by the
// error-free transformations of Knuth and Dekker), 12 FP32 instructions a
// term and a fifth of FP64's time: 46 bits of the taps and the window, so the
// result's rounding to FP32 is all that shows.  (Plain FP32 sums are worse at
// r = 4 from rough data, where w is several times u: 2e-7.)  A window whose
// values could overflow or underflow takes the FP64 sum.
constexpr int kDotRows = 8, kEdgeRows = 8;

// Items start at multiples of their rows, or one row before: where the exit
// pairs an odd row with the next, so that no item needs a row of another's.
__host__ __device__ __forceinline__ int item_shift(const PropRun &P) { return P.exit && ((P.p0 + P.k) & 1) ? 1 : 0; }
__host__ __device__ __forceinline__ long long item_count(long long rows, int per, int shift)
{
    return rows > 0 ? (rows + shift + per - 1) / per : 0;
}

// How far right row i's sum reaches in k steps: k where the last step pairs
// the row with its right neighbour, else k - 1 (and the other way to the left).
__device__ __forceinline__ int reach_right(const PropRun &P, long long i)
{
    return ((i + P.p0 + P.k - 1) & 1) ? P.k - 1 : P.k;
}
constexpr int kDotWin = 2 * kPropRMax + 16;

template <int ROWS>
struct DotShared {
    double row[ROWS + 2];
    int bad[ROWS + 2];
    int code;  // FP32: largest exponent in the window
};

// a + b = t + err exactly.
__device__ __forceinline__ float two_sum(float a, float b, float &err)
{
    const float t = __fadd_rn(a, b), z = __fsub_rn(t, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(t, z)), __fsub_rn(b, z));
    return t;
}

// Right-hand sides of an FP32 state as pairs: u + r (u_partner - u).
__device__ __forceinline__ float2 load_w32(const PropRun &P, long long j, int &code)
{
    const float *in = static_cast<const float *>(P.in);
    const float u = in[j];
    int c = (int)(__float_as_uint(u) >> 23) & 0xff;
    float2 w = make_float2(u, 0.0f);
    if (P.entry) {
        const long long m = ((j + 1 - P.p0) & 1) ? j - 1 : j + 1;
        if (j == 0 || j == P.n - 1 || m < 0 || m >= P.n) {
            const double x = load_w<float>(P, j);
            w.x = (float)x;
            w.y = (float)(x - (double)w.x);
            const int cw = (int)(__float_as_uint(w.x) >> 23) & 0xff;
            c = cw > c ? cw : c;
        } else {
            const float v = in[m], r = (float)P.r, rl = (float)(P.r - (double)r);
            const int cv = (int)(__float_as_uint(v) >> 23) & 0xff;
            c = cv > c ? cv : c;
            float dl, e;
            const float d = two_sum(v, -u, dl), p = __fmul_rn(r, d);
            w.x = two_sum(u, p, e);
            w.y = __fadd_rn(e, __fmaf_rn(r, dl, __fmaf_rn(rl, d, __fmaf_rn(r, d, -p))));
        }
    }
    code = c > code ? c : code;
    return w;
}

// The running sum of a lane's terms, in FP64 or as a pair.
struct Sum64 {
    double s = 0.0;
    __device__ __forceinline__ void add(double t, double w) { s = fma(t, w, s); }
    __device__ __forceinline__ double value() const { return s; }
};
struct Sum32 {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float2 t, float2 w)
    {
        const float p = __fmul_rn(t.x, w.x);
        float e;
        s = two_sum(s, p, e);
        c = __fadd_rn(c, __fadd_rn(e, __fmaf_rn(t.y, w.x, __fmaf_rn(t.x, w.y, __fmaf_rn(t.x, w.x, -p)))));
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};
template <typename E>
struct SumOf;
template <>
struct SumOf<double> {
    using S = Sum64;
};
template <>
struct SumOf<float2> {
    using S = Sum32;
};
// What shared memory holds of a tap or a right-hand side, by the state's type.
template <typename T>
struct PairOf;
template <>
struct PairOf<double> {
    using E = double;
};
template <>
struct PairOf<float> {
    using E = float2;
};

// x is not finite, or large enough (r <= 1e6) for its right-hand side to
// overflow: an integer test, where load_w costs FP64 instructions.
__device__ __forceinline__ bool may_spoil(double x)
{
    return ((unsigned)__double2hiint(x) & 0x7ff00000u) >= (2047u - 24u) << 20;
}
__device__ __forceinline__ bool may_spoil(float x) { return (__float_as_uint(x) & 0x7f800000u) == 0x7f800000u; }

// An operator's taps and its two walls' arrays into dot_taps(R) elements of
// shared memory.  Every row of a CTA's items reads them: from global memory
// each row's sum was a chain of cache latencies (an item of four rows took
// 19,000 cycles, half of them waiting).
__host__ __device__ constexpr int dot_taps(int R) { return 2 * R + 1 + 4 * (R + 1); }
__device__ __forceinline__ double tap_as(double v, double) { return v; }
__device__ __forceinline__ float2 tap_as(double v, float2)
{
    // on the integer pipes (the conversions run on the FP64 unit): the high
    // part truncated, the low part the next 24 bits; taps are at most 1,
    // those below FP32's normal range count as zero
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    const int ex = (int)((u >> 52) & 0x7ff) - (1023 - 127);  // FP32 exponent field
    const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
    if (ex <= 24)
        return make_float2(0.0f, 0.0f);
    const unsigned hi = sign | ((unsigned)ex << 23) | ((unsigned)(u >> 29) & 0x7fffffu);
    // 2^(ex - 127) (1.low29 - 1) 2^-23, by subtracting the leading one
    const float one = __uint_as_float(sign | ((unsigned)(ex - 23) << 23));
    const float lo = __uint_as_float(sign | ((unsigned)(ex - 23) << 23) | (((unsigned)u >> 6) & 0x7fffffu));
    return make_float2(__uint_as_float(hi), __fsub_rn(lo, one));
}
template <int NT, typename E>
__device__ __forceinline__ void dot_stage(const PropRun &P, E *taps)
{
    const int R = P.R;
    const double *e = P.e - R, *h0 = P.h + P.p0 * 2 * P.hs, *h1 = P.h + P.pr * 2 * P.hs;
    for (int x0 = threadIdx.x; x0 < dot_taps(R); x0 += 8 * NT) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int x = x0 + u * NT, y = x - (2 * R + 1),
                      q = (y >= R + 1) + (y >= 2 * (R + 1)) + (y >= 3 * (R + 1)), z = y - q * (R + 1);
            v[u] = x >= dot_taps(R) ? 0.0 : __ldg(y < 0 ? e + x : (q < 2 ? h0 : h1) + (q & 1) * P.hs + z);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (x0 + u * NT < dot_taps(R))
                taps[x0 + u * NT] = tap_as(v[u], E{});
    }
}

// One lane's part of row i: of its 32 PARTS lanes, number x0.  w: the window,
// from point wlo on; taps: dot_stage's, or NULL for the global arrays.
template <typename E, int PARTS, bool STAGED>
__device__ __forceinline__ double row_part(const PropRun &P, const E *s_w, long long wlo, const E *taps, long long i,
                                           int x0)
{
    const int R = P.R, ph = (int)(i & 1), rev = (P.p0 ^ ph) & 1;
    const int right = reach_right(P, i), left = 2 * P.k - 1 - right;
    const long long jl = i - (left < R ? left : R) > 0 ? i - (left < R ? left : R) : 0;
    const long long jh = i + (right < R ? right : R) < P.n - 1 ? i + (right < R ? right : R) : P.n - 1;
    // two sums, of alternate terms
    typename SumOf<E>::S s[2];
    auto add = [&](int a, int end, auto tap, const E *w, int dw) {
        int x = a + x0;
#pragma unroll 4
        for (; x + 32 * PARTS < end; x += 64 * PARTS) {
            s[0].add(tap(x), w[dw * x]);
            s[1].add(tap(x + 32 * PARTS), w[dw * (x + 32 * PARTS)]);
        }
        if (x < end)
            s[0].add(tap(x), w[dw * x]);
    };
    auto get = [](const E *st, const double *gl, int x) {
        if constexpr (STAGED)
            return st[x];
        else
            return __ldg(gl + x);
    };
    {
        const int o = (int)(i - jl), se = rev ? -1 : 1;
        const E *e = STAGED ? taps + R + se * -o : nullptr;
        const double *g = P.e + se * -o;
        add(0, (int)(jh - jl) + 1, [&](int x) { return get(e, g, se * x); }, s_w + (jl - wlo), 1);
    }
    double f = 0.0;
    // the left wall: h_{i&1}(j + i - (i & 1)) for j >= 0
    const long long il = i - ph;
    if (il <= R) {
        const E *h = STAGED ? taps + 2 * R + 1 + ph * (R + 1) + il : nullptr;
        const double *g = P.h + (P.p0 * 2 + ph) * P.hs + il;
        const long long m = R - il < jh ? R - il : jh;
        add((int)jl, (int)m + 1, [&](int x) { return get(h, g, x); }, s_w - wlo, 1);
        if (x0 == 0 && P.bl != 0.0)
            f = P.bl * P.F[P.p0 * P.hs + i];
    }
    // the right wall, from the mirrored index
    const long long im = P.n - 1 - i;
    const int pm = (int)(im & 1);
    const long long ir = im - pm;
    if (ir <= R) {
        const E *h = STAGED ? taps + 2 * R + 1 + (2 + pm) * (R + 1) + ir : nullptr;
        const double *g = P.h + (P.pr * 2 + pm) * P.hs + ir;
        const long long m = R - ir < P.n - 1 - jl ? R - ir : P.n - 1 - jl;
        add((int)(P.n - 1 - jh), (int)m + 1, [&](int x) { return get(h, g, x); }, s_w + (P.n - 1 - wlo), -1);
        if (x0 == 0 && P.br != 0.0)
            f = fma(P.br, P.F[P.pr * P.hs + im], f);
    }
    return s[0].value() + s[1].value() + f;
}

// Rows [r0, rend) by NT threads (all of named barrier 1), up to ROWS of them,
// a row by PARTS warps; s_w holds kDotWin doubles, and 32 PARTS (ROWS + 2)
// more where PARTS > 1.
// taps: the operator's arrays in shared memory (STAGED: dot_stage's, as pairs
// for FP32 states), else NULL.
template <typename T, int NT, int ROWS, int PARTS = 1, bool STAGED = false>
__device__ __forceinline__ void dot_rows(const PropRun &P, DotShared<ROWS> &sh, double *s_w, const double *taps,
                                         long long r0, long long rend)
{
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int pe = (P.p0 + P.k) & 1, R = P.R;
    auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };
    // an exit also needs the partners of the outer rows
    const long long lo = P.exit && r0 > 0 && ((r0 + pe) & 1) ? r0 - 1 : r0;
    const long long hi = P.exit && rend < P.n && !((rend - 1 + pe) & 1) ? rend + 1 : rend;
    const long long wlo = lo - R > 0 ? lo - R : 0;
    const long long whi = hi + R < P.n ? hi + R : P.n;
    if (t < ROWS + 2)
        sh.bad[t] = 0;
    constexpr bool FP32 = sizeof(T) == 4 && STAGED;
    float2 *w32 = reinterpret_cast<float2 *>(s_w);
    const int win = (int)(whi - wlo);
    bool fp32 = FP32;
    if (FP32) {
        int code = 0;
        if (t == 0)
            sh.code = 0;
        sync();
        for (int x0 = t; x0 < win; x0 += 4 * NT) {
            float2 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                v[u] = x0 + u * NT < win ? load_w32(P, wlo + x0 + u * NT, code) : make_float2(0.0f, 0.0f);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (x0 + u * NT < win)
                    w32[x0 + u * NT] = v[u];
        }
        code = __reduce_max_sync(0xffffffffu, code);
        if (lane == 0)
            atomicMax(&sh.code, code);
        sync();
        // a product of a value below 2^-70 with a tap may be subnormal; w
        // reaches 2^21 times a value (r <= 1e6).  (All zeros are fine.)
        fp32 = sh.code == 0 || (sh.code >= 127 - 70 && sh.code < 127 + 90);
        if (sh.code == 0)
            fp32 = P.bl == 0.0 && P.br == 0.0;
    }
    if (!fp32) {
        for (int x0 = t; x0 < win; x0 += 4 * NT) {
            double v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                v[u] = x0 + u * NT < win ? load_w<T>(P, wlo + x0 + u * NT) : 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (x0 + u * NT < win)
                    s_w[x0 + u * NT] = v[u];
        }
        sync();
    }
    // a value that is not finite spoils every row it reaches in k steps, also
    // beyond the taps that are kept
    if (R < P.k) {
        const long long clo = lo - P.k > 0 ? lo - P.k : 0, chi = hi + P.k < P.n ? hi + P.k : P.n;
        // (a value spoils its own and its partner's right-hand side)
        const T *in = static_cast<const T *>(P.in);
        const long long slo = clo > 0 ? clo - 1 : 0, shi = chi < P.n ? chi + 1 : P.n;
        auto mark = [&](long long v) {
            if (isfinite(load_w<T>(P, v)))
                return;
            for (int q = 0; q < (int)(hi - lo); ++q) {
                const long long d = v - (lo + q);
                const int right = reach_right(P, lo + q);
                if (d <= right && -d <= 2 * P.k - 1 - right)
                    sh.bad[q] = 1;
            }
        };
        bool any = false;
        for (long long j = slo + t; j < shi; j += 8 * NT)
#pragma unroll
            for (int u = 0; u < 8; ++u)
                any |= may_spoil(j + u * NT < shi ? in[j + u * NT] : (T)0);
        if (t == 0 && clo == 0)  // the wall terms
            mark(0);
        if (t == 32 && chi == P.n)
            mark(P.n - 1);
        if (any)
            for (long long j = slo + t; j < shi; j += NT)
                if (may_spoil(in[j]))
                    for (long long v = j - 1 > clo ? j - 1 : clo; v <= j + 1 && v < chi; ++v)
                        mark(v);
        sync();
    }
    for (int z = warp; z < (int)(hi - lo) * PARTS; z += NT / 32) {
        const int q = z / PARTS, x0 = z % PARTS * 32 + lane;  // this lane's taps: x0, x0 + 32 PARTS, ...
        double s;
        if (FP32 && fp32)
            s = row_part<float2, PARTS, true>(P, w32, wlo, reinterpret_cast<const float2 *>(taps), lo + q, x0);
        else
            s = row_part<double, PARTS, STAGED && !FP32>(P, s_w, wlo, taps, lo + q, x0);
        if (PARTS > 1) {
            s_w[kDotWin + z * 32 + lane] = s;
            continue;
        }
        s = warp_sum_rounded_once<1>({s});
        if (lane == 0)
            sh.row[q] = sh.bad[q] ? s + __longlong_as_double(0x7ff8000000000000ll) : s;
    }
    sync();
    if (PARTS > 1) {
        for (int q = warp; q < (int)(hi - lo); q += NT / 32) {
            double v[PARTS];
#pragma unroll
            for (int p = 0; p < PARTS; ++p)
                v[p] = s_w[kDotWin + (q * PARTS + p) * 32 + lane];
            const double s = warp_sum_rounded_once(v);
            if (lane == 0)
                sh.row[q] = sh.bad[q] ? s + __longlong_as_double(0x7ff8000000000000ll) : s;
        }
        sync();
    }
    if (t < (int)(rend - r0)) {
        const long long i = r0 + t;
        double v = sh.row[i - lo];
        if (P.exit) {
            const long long m = ((i + pe) & 1) ? i - 1 : i + 1;
            // (x1 + x2 = 1)
            v = (m >= 0 && m < P.n) ? fma(P.x2, sh.row[m - lo] - v, v) : P.xs * v;
        }
        static_cast<T *>(P.out)[i] = (T)v;
    }
    sync();
}

// The blocks the tiles listed, `listed` of them: item `it` is eight rows.
template <typename T, int NT, bool STAGED = false>
__device__ __forceinline__ void dot_listed(const PropRun &P, DotShared<kDotRows> &sh, double *s_w, const double *taps,
                                           long long it)
{
    const long long r0 = (long long)P.list[it / (kPropBlk / kDotRows)] * kPropBlk + it % (kPropBlk / kDotRows) * kDotRows;
    dot_rows<T, NT, kDotRows, 1, STAGED>(P, sh, s_w, taps, r0, r0 + kDotRows < P.n ? r0 + kDotRows : P.n);
}

}  // namespace
}  // namespace ge

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

// ---- reading the state ---------------------------------------------------

// Point j's right-hand side w = (1 - r) u + r u_partner (+ the wall terms),
// the groups those of parity 1 - p0 -- or the value itself after the first
// operator, when the buffer holds w.
template <typename T>
__device__ __forceinline__ double load_w(const PropRun &P, long long j)
{
    const T *in = static_cast<const T *>(P.in);
    const double u = (double)in[j];
    if (!P.entry)
        return u;
    const long long m = ((j + 1 - P.p0) & 1) ? j - 1 : j + 1;
    double w = P.omr * u;
    if (m >= 0 && m < P.n)
        w = fma(P.r, (double)in[m], w);
    if (j == 0)
        w += P.fl;
    if (j == P.n - 1)
        w += P.fr;
    return w;
}

// ---- dot products --------------------------------------------------------

// A few rows of a CTA: the rows near the walls (or all rows of a small grid),
// and the blocks a tile left out.  The window of right-hand sides is staged
// in shared memory as doubles; one warp takes one row's sum.  Bound by the
// FP64 unit (two taps' widths of multiply-adds a row).
constexpr int kDotRows = 8, kEdgeRows = 16;

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
};

// Rows [r0, rend) by NT threads (all of named barrier 1), up to ROWS of them;
// s_w holds kDotWin doubles.
template <typename T, int NT, int ROWS>
__device__ __forceinline__ void dot_rows(const PropRun &P, DotShared<ROWS> &sh, double *s_w, long long r0, long long rend)
{
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int pe = (P.p0 + P.k) & 1, R = P.R;
    auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };
    // with the exit at parity 1 the outer rows' partners lie outside the item
    const int ext = P.exit && pe;
    const long long lo = r0 - ext > 0 ? r0 - ext : 0;
    const long long hi = rend + ext < P.n ? rend + ext : P.n;
    const long long wlo = lo - R > 0 ? lo - R : 0;
    const long long whi = hi + R < P.n ? hi + R : P.n;
    if (t < ROWS + 2)
        sh.bad[t] = 0;
#pragma unroll 4
    for (long long j = wlo + t; j < whi; j += NT)
        s_w[j - wlo] = load_w<T>(P, j);
    sync();
    // a value that is not finite spoils every row it reaches in k steps, also
    // beyond the taps that are kept
    if (R < P.k) {
        const long long clo = lo - P.k > 0 ? lo - P.k : 0, chi = hi + P.k < P.n ? hi + P.k : P.n;
#pragma unroll 4
        for (long long j = clo + t; j < chi; j += NT) {
            if (!isfinite(j >= wlo && j < whi ? s_w[j - wlo] : load_w<T>(P, j))) {
                for (int q = 0; q < (int)(hi - lo); ++q) {
                    const long long d = j - (lo + q);
                    const int right = reach_right(P, lo + q);
                    if (d <= right && -d <= 2 * P.k - 1 - right)
                        sh.bad[q] = 1;
                }
            }
        }
        sync();
    }
    for (int q = warp; q < (int)(hi - lo); q += NT / 32) {
        const long long i = lo + q;
        const int ph = (int)(i & 1), rev = (P.p0 ^ ph) & 1;
        const int right = reach_right(P, i), left = 2 * P.k - 1 - right;
        const long long jl = i - (left < R ? left : R) > 0 ? i - (left < R ? left : R) : 0;
        const long long jh = i + (right < R ? right : R) < P.n - 1 ? i + (right < R ? right : R) : P.n - 1;
        double s = 0.0;
        {
            const double *w = s_w + (jl - wlo);
            const int m = (int)(jh - jl) + 1;
            const double *e = rev ? P.e + (i - jl) : P.e - (i - jl);
            const int se = rev ? -1 : 1;
#pragma unroll 8
            for (int x = lane; x < m; x += 32)
                s = fma(__ldg(e + se * x), w[x], s);
        }
        // the left wall: h_{i&1}(j + i - (i & 1)) for j >= 0
        const long long il = i - ph;
        if (il <= R) {
            const double *h = P.h + (P.p0 * 2 + ph) * P.hs + il;
            const long long m = R - il < jh ? R - il : jh;
#pragma unroll 8
            for (int x = (int)jl + lane; x <= (int)m; x += 32)
                s = fma(__ldg(h + x), s_w[x - wlo], s);
            if (lane == 0 && P.bl != 0.0)
                s = fma(P.bl, P.F[P.p0 * P.hs + i], s);
        }
        // the right wall, from the mirrored index
        const long long im = P.n - 1 - i;
        const int pm = (int)(im & 1);
        const long long ir = im - pm;
        if (ir <= R) {
            const double *h = P.h + (P.pr * 2 + pm) * P.hs + ir;
            const long long m = R - ir < P.n - 1 - jl ? R - ir : P.n - 1 - jl;
            const double *w = s_w + (P.n - 1 - wlo);
#pragma unroll 8
            for (int x = (int)(P.n - 1 - jh) + lane; x <= (int)m; x += 32)
                s = fma(__ldg(h + x), w[-x], s);
            if (lane == 0 && P.br != 0.0)
                s = fma(P.br, P.F[P.pr * P.hs + im], s);
        }
        s = warp_sum(s);
        if (lane == 0)
            sh.row[q] = sh.bad[q] ? s + __longlong_as_double(0x7ff8000000000000ll) : s;
    }
    sync();
    if (t < (int)(rend - r0)) {
        const long long i = r0 + t;
        double v = sh.row[i - lo];
        if (P.exit) {
            const long long m = ((i + pe) & 1) ? i - 1 : i + 1;
            v = (m >= 0 && m < P.n) ? fma(P.x2, sh.row[m - lo], P.x1 * v) : P.xs * v;
        }
        static_cast<T *>(P.out)[i] = (T)v;
    }
    sync();
}

// The blocks the tiles listed, `listed` of them: item `it` is eight rows.
template <typename T, int NT>
__device__ __forceinline__ void dot_listed(const PropRun &P, DotShared<kDotRows> &sh, double *s_w, long long it)
{
    const long long r0 = (long long)P.list[it / (kPropBlk / kDotRows)] * kPropBlk + it % (kPropBlk / kDotRows) * kDotRows;
    dot_rows<T, NT, kDotRows>(P, sh, s_w, r0, r0 + kDotRows < P.n ? r0 + kDotRows : P.n);
}

}  // namespace
}  // namespace ge

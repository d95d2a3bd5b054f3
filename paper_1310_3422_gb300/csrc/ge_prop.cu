// ge_prop.cu -- the kernels of composed steps (ge_prop.h): building an
// operator's taps by binary powering, cutting the taps into digits, applying
// an operator on the tensor cores away from the walls (tiles) and as FP64 dot
// products near them (dots).
//
// Tiles.  A value and a tap are fixed-point numbers: integers of base-256
// digits, the value relative to the largest magnitude of its tile, the tap
// relative to the largest tap.  Digits are small integers, exact in FP16;
// their products sum in the FP32 accumulators of tcgen05.mma without rounding
// while a sum stays below 2^24, and the accumulators of equal weight i + j
// (value digit j, tap digit i) join as 64-bit integers.  So a tile's result
// is the exact fixed-point sum, rounded once.
//   FP64: values to 2^-62 of the tile's largest, 8 digits; taps to about
//     2^-62, 7 digits; the 35 products with i + j <= 7 (the rest is below
//     2^-64 of the largest value).
//   FP32: values to 2^-30, taps to about 2^-39, 4 digits each, 10 products.
// (FP64 values in seven digits, 2^-54, were 14 % faster on large grids: 2^24
// points, r = 2, 2000 steps, 2.09 ms, now 2.42.  But a stretch of rough data
// 2^-8 of its neighbours erred 146 times as much as step by step, 24 steps at
// r = 1; now 0.7 times.)
// Step by step the same k steps cost k multiply-adds a point on the FP64 (or
// FP32) pipes; composed they cost the taps' width times the products on the
// tensor cores, and the width grows with sqrt(k) only.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "ge_internal.h"
#include "ge_prop.h"
#include "ge_prop_dev.cuh"
#include "ge_tc.cuh"

namespace ge {
namespace {

// ---- building an operator ------------------------------------------------

// A tap of a row of parity `phase` of the chain starting at parity q: the
// even rows' taps of the chain starting at parity 0, reversed when exactly
// one of the two differs.
__device__ __forceinline__ double tap(const double *e, int R, int q_phase, int d)
{
    d = (q_phase & 1) ? -d : d;
    return (d >= -R && d <= R) ? e[d] : 0.0;
}
// The direction of those taps.
__device__ __forceinline__ int dir(int q_phase) { return (q_phase & 1) ? -1 : 1; }

// An unevaluated sum of two doubles.
struct Dd {
    double hi, lo;
};
__device__ __forceinline__ Dd two_sum(double a, double b)
{
    const double s = a + b, t = s - a;
    return {s, (a - (s - t)) + (b - t)};
}
__device__ __forceinline__ Dd dd_add(Dd a, Dd b)
{
    const Dd s = two_sum(a.hi, b.hi);
    return two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__device__ __forceinline__ Dd dd_mul(Dd a, Dd b)
{
    const double p = a.hi * b.hi;
    return two_sum(p, fma(a.hi, b.hi, -p) + fma(a.hi, b.lo, a.lo * b.hi));
}

// ---- the short chain: 128-bit fixed point

// Signed fixed-point number of 126 fraction bits.
struct Fix {
    unsigned long long lo;
    long long hi;
};
__device__ __forceinline__ Fix fix_sub(Fix a, Fix b)
{
    return {a.lo - b.lo, (long long)((unsigned long long)a.hi - (unsigned long long)b.hi - (a.lo < b.lo))};
}
__device__ __forceinline__ Fix fix_add(Fix a, Fix b)
{
    const unsigned long long lo = a.lo + b.lo;
    return {lo, (long long)((unsigned long long)a.hi + (unsigned long long)b.hi + (lo < a.lo))};
}
// x times a fraction f 2^-64, rounded down in magnitude.
__device__ __forceinline__ Fix fix_mul(Fix x, unsigned long long f)
{
    const bool neg = x.hi < 0;
    if (neg)
        x = fix_sub(Fix{0, 0}, x);
    const unsigned long long xh = (unsigned long long)x.hi, l = xh * f, m = __umul64hi(x.lo, f);
    const Fix r{l + m, (long long)(__umul64hi(xh, f) + (l + m < l))};
    return neg ? fix_sub(Fix{0, 0}, r) : r;
}
// As a double-double.
__device__ __forceinline__ Dd fix_dd(Fix x)
{
    const bool neg = x.hi < 0;
    if (neg)
        x = fix_sub(Fix{0, 0}, x);
    const unsigned long long h = (unsigned long long)x.hi;
    const double a = (double)(unsigned)(h >> 32) * 0x1p-30, b = (double)(unsigned)h * 0x1p-62;
    const double c = (double)(unsigned)(x.lo >> 32) * 0x1p-94, d = (double)(unsigned)x.lo * 0x1p-126;
    const Dd ab = two_sum(a, b), cd = two_sum(c, d);
    const Dd r = two_sum(ab.hi, ab.lo + cd.hi);
    const double e = ((ab.lo + cd.hi) - ab.lo);
    const Dd v = two_sum(r.hi, r.lo + ((cd.hi - e) + cd.lo));
    return neg ? Dd{-v.hi, -v.lo} : v;
}

// The chain of k <= kPropShort steps, step by step: rows of the operator as
// vectors, the steps applied from the last back (a step is symmetric): the
// even row of the infinite grid from parity 0, and rows 0 and 1 of the half
// grid from both parities.  An element per thread, in 128-bit fixed point:
// FP64 pairs would take ten operations an update on the SM's one FP64 unit
// (19 cycles each a warp) where the integer pipes take a few cycles.
constexpr int kShortThreads = (2 * kPropShort + 3 + 4 * (kPropShort + 3) + 31) / 32 * 32;

__global__ void __launch_bounds__(kShortThreads) prop_short_kernel(double *e, double *el, double *h, double *hl, int hs, int k,
                                                         PropCoef c)
{
    constexpr int kE = 2 * kPropShort + 3, kW = kPropShort + 3;  // elements of the infinite row, of a wall row
    __shared__ Fix s_x[2][kE + 4 * kW + 2];
    const int t = threadIdx.x;
    const bool inf = t < kE, used = t < kE + 4 * kW;
    const int w = (t - kE) / kW, pos = inf ? t - (kPropShort + 1) : (t - kE) % kW;  // lattice position
    const int p = inf ? 0 : w >> 1, b = inf ? 0 : w & 1;
    const int first = inf ? -(kPropShort + 1) : 0, last = kPropShort + (inf ? 1 : 2);
    Fix x{0, used && pos == b ? (1ll << 62) : 0};
    for (int s = k - 1; s >= 0; --s) {
        const int par = (p + s) & 1, q = s & 1;
        if (used)
            s_x[q][t] = x;
        __syncthreads();
        if (used) {
            const int m = ((pos + par) & 1) ? -1 : 1;  // the pair of parity par
            if (pos + m >= first && pos + m <= last) {
                x = fix_add(x, fix_mul(fix_sub(s_x[q][t + m], x), c.be_frac));
            } else if (!inf && pos + m < 0) {
                x = fix_mul(x, c.ka_frac);
                if (c.ka[0] < 0.0)
                    x = fix_sub(Fix{0, 0}, x);
            }
        }
    }
    __syncthreads();
    if (used)
        s_x[0][t] = x;
    __syncthreads();
    const int R = k + 1;
    if (inf && pos >= -R && pos <= R) {
        const Dd v = fix_dd(x);
        e[pos] = v.hi;
        el[pos] = v.lo;
    } else if (used && !inf && pos <= R) {
        // less the infinite grid's tap at distance pos - b
        const int d = dir(p ^ b) * (pos - b);
        const Dd v = fix_dd(fix_sub(x, s_x[0][d + kPropShort + 1]));
        h[w * hs + pos] = v.hi;
        hl[w * hs + pos] = v.lo;
    }
}

// ---- doubling the chain

// Chain of 2 k1 + delta steps from the chain of k1: Q_{2k+1} = Q_k Q_k C, the
// extra first step mixing the columns of a pair.  A block takes 32 columns
// (30 with delta: the outer two only lend their sums) of one row, a column
// per thread, and its four warps a quarter of the terms each: a term costs
// one multiply-add on the FP64 unit, which bounds the kernel, a broadcast and
// a conflict-free read.  (A warp per entry, its lanes sharing the terms: 70 us
// for the last level of k = 1999, r = 0.7; columns per thread: 38 us.)
// Rounding leaves the whole operator a common factor near 1, which the finish
// takes out.  `par`: the start parities whose wall arrays are needed (bit p).
constexpr int kLevelPad = 36;  // zeros around the staged arrays: a block's columns overreach by at most 33

__global__ void __launch_bounds__(128) prop_level_kernel(const PropLevel P)
{
    extern __shared__ double st[];
    __shared__ double s_part[4][32], s_edge[2][4];
    const int t = threadIdx.x, lane = t & 31, seg = t >> 5, R = P.R1, dl = P.delta;
    const int ne = 2 * R + 1 + 2 * kLevelPad, nh = R + 1 + 2 * kLevelPad;
    double *e = st + R + kLevelPad, *h = st + ne + kLevelPad;  // h: row class x at h + x nh
    for (int i = t; i < ne; i += 128) {
        const int d = i - R - kLevelPad;
        st[i] = d >= -R && d <= R ? P.e0[d] : 0.0;
    }
#pragma unroll 1
    for (int x = 0; x < 4; ++x)
        for (int i = t; i < nh; i += 128) {
            const int d = i - kLevelPad;
            st[ne + x * nh + i] = d >= 0 && d <= R ? P.h0[x * P.hs + d] : 0.0;
        }
    __syncthreads();
    const int per = dl ? 30 : 32;
    const int b_int = (2 * P.R2 + 1 + per - 1) / per, b_wall = (P.R2 + 1 + per - 1) / per;
    const int rows = P.par == 3 ? 4 : 2;
    const bool wall = (int)blockIdx.x >= b_int;
    const int wb = wall ? ((int)blockIdx.x - b_int) / b_wall : 0;
    if (wb >= rows)
        return;
    const int pb = wb + (P.par == 2 ? 2 : 0), p = wall ? pb >> 1 : 0, b = wall ? pb & 1 : 0;
    const int first = wall ? 0 : -P.R2;                        // first column of the row
    const int blk = wall ? ((int)blockIdx.x - b_int) % b_wall : (int)blockIdx.x;
    const int j0 = first + blk * per - dl, j = j0 + lane;      // this block's columns j0 .. j0 + 31
    const int qs = (p + P.k1 + dl) & 1, qf = (p + dl) & 1;
    const int s2 = dir(qs ^ b), s1e = dir(qf), s1o = -s1e;     // directions: the later chain's row, the earlier one's columns
    double *g2 = st + ne + 4 * nh;  // the later chain's row b in full, a2 + h2
    if (wall) {
        const double *h2 = h + (qs * 2 + b) * nh;
        for (int l = t; l < R + kLevelPad; l += 128)
            g2[l] = (l - b <= R ? e[s2 * (l - b)] : 0.0) + h2[l];
        __syncthreads();
    }
    // terms c[l] a1[j - l], l in [lo, hi] by this warp, a pair of columns l at a time
    auto conv = [&](const double *c, int sc, int lo, int hi) {
        if (hi < lo)
            return 0.0;
        const int n = hi - lo + 1, q = (n + 3) / 4;
        int l = lo + seg * q;
        const int end = l + q - 1 < hi ? l + q - 1 : hi;
        // eight sums: rounding grows with the length of each
        double x0[4] = {}, x1[4] = {};
        if (l <= end && (l & 1)) {
            x1[0] = c[sc * l] * e[s1o * (j - l)];
            ++l;
        }
        for (; l + 7 <= end; l += 8) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                x0[u] = fma(c[sc * (l + 2 * u)], e[s1e * (j - l - 2 * u)], x0[u]);
                x1[u] = fma(c[sc * (l + 2 * u + 1)], e[s1o * (j - l - 2 * u - 1)], x1[u]);
            }
        }
        for (; l + 1 <= end; l += 2) {
            x0[0] = fma(c[sc * l], e[s1e * (j - l)], x0[0]);
            x1[0] = fma(c[sc * (l + 1)], e[s1o * (j - l - 1)], x1[0]);
        }
        if (l <= end)
            x0[0] = fma(c[sc * l], e[s1e * (j - l)], x0[0]);
        return ((x0[0] + x0[1]) + (x0[2] + x0[3])) + ((x1[0] + x1[1]) + (x1[2] + x1[3]));
    };
    // the columns' overreach: |j - l| <= R + 33 stays inside the padding
    const int cl = j0 - R > b - R ? j0 - R : b - R, ch = j0 + 31 + R < b + R ? j0 + 31 + R : b + R;
    double v;
    if (!wall) {
        v = conv(e - s2 * b, s2, cl, ch);
    } else {
        // sum over l >= 0 of h2 a1 + (a2 + h2) h1, less the infinite product's part from l < 0
        const double *h2 = h + (qs * 2 + b) * nh;
        v = conv(h2, 1, j0 - R > 0 ? j0 - R : 0, R) - conv(e - s2 * b, s2, cl, ch < -1 ? ch : -1);
        const double *h1e = h + qf * 2 * nh, *h1o = h1e + nh;
        const int hi = R - j0 + 1 < R + 1 ? R - j0 + 1 : R + 1;
        if (hi >= 0) {
            const int q = ((hi + 1 + 3) / 4 + 1) & ~1;
            const int l0 = seg * q, end = l0 + q - 1 < hi ? l0 + q - 1 : hi;
            const int jj = j > 0 ? j : 0;  // column -1 takes no part
            double x0[4] = {}, x1[4] = {};
            int l = l0;
            for (; l + 6 <= end; l += 8) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    x0[u] = fma(g2[l + 2 * u], h1e[jj + l + 2 * u], x0[u]);
                    x1[u] = fma(g2[l + 2 * u + 1], h1o[jj + l + 2 * u], x1[u]);
                }
            }
            for (; l <= end; l += 2) {
                x0[0] = fma(g2[l], h1e[jj + l], x0[0]);
                x1[0] = fma(g2[l + 1], h1o[jj + l], x1[0]);
            }
            v += ((x0[0] + x0[1]) + (x0[2] + x0[3])) + ((x1[0] + x1[1]) + (x1[2] + x1[3]));
        }
    }
    s_part[seg][lane] = v;
    if (wall && dl && p == 1 && j0 < 0) {
        // a singleton's column has no partner: the infinite product's own
        // entries at columns 0 and -1, terms spread over the block
        double a0 = 0.0, am = 0.0;
        for (int d = -R + t; d <= R; d += 128) {
            const double a2 = e[s2 * d];
            const int l = b + d, s1 = dir(qf ^ l);
            if (l <= R && l >= -R)
                a0 = fma(a2, e[s1 * -l], a0);
            if (-1 - l <= R && -1 - l >= -R)
                am = fma(a2, e[s1 * (-1 - l)], am);
        }
        a0 = warp_sum(a0);
        am = warp_sum(am);
        if (lane == 0) {
            s_edge[0][seg] = a0;
            s_edge[1][seg] = am;
        }
    }
    __syncthreads();
    if (seg != 0)
        return;
    v = (s_part[0][lane] + s_part[1][lane]) + (s_part[2][lane] + s_part[3][lane]);
    if (dl) {
        const double up = __shfl_down_sync(0xffffffffu, v, 1), dn = __shfl_up_sync(0xffffffffu, v, 1);
        double x = fma(P.c.al[0], v, P.c.be[0] * (((j + p) & 1) ? dn : up));
        if (wall && p == 1 && j == 0) {
            const double a0 = (s_edge[0][0] + s_edge[0][1]) + (s_edge[0][2] + s_edge[0][3]);
            const double am = (s_edge[1][0] + s_edge[1][1]) + (s_edge[1][2] + s_edge[1][3]);
            x = P.c.ka[0] * (a0 + v) - P.c.al[0] * a0 - P.c.be[0] * am;
        }
        v = x;
    }
    if (j < first || j > P.R2 || (dl && (lane == 0 || lane == 31)))
        return;
    if (wall) {
        P.h1[pb * P.hs + j] = v;
    } else {
        P.e1[j] = v;
    }
}

// round(x 2^E), at most 2^62 in magnitude.
__device__ __forceinline__ long long fixed_of(double x, int E)
{
    const long long u = __double_as_longlong(x);
    const int e = (int)(u >> 52) & 0x7ff;
    unsigned long long m = (unsigned long long)u & 0x000fffffffffffffull;
    if (e)
        m |= 0x0010000000000000ull;
    const int sh = (e ? e : 1) - 1075 + E;
    if (sh >= 0) {
        m <<= sh;
    } else {
        const int n = -sh < 60 ? -sh : 60;
        m = (m + (1ull << (n - 1))) >> n;
    }
    return u < 0 ? -(long long)m : (long long)m;
}

// ---- the finished operator

// The finished operator from the last level's arrays (small blocks, to spread
// the double-doubles over the SMs' FP64 units):
// taps and wall arrays divided by the taps' sum, the wall values' part, and
// the rows of the tensor cores' operator as double-doubles, with their largest
// magnitude: the exit folded into the last operator of a call (u = x1 w + x2
// w_partner, pairs of the last step's parity) and the entry into the first
// one (w = u + r (u_partner - u): a combination of columns), so that tiles
// read and write the state as it is.
//   F: with both walls 1 the constant state is steady, so F_i is what row i
// misses of it: 1 - sum_j Q(i, j), plus the first point's own wall term,
// which its right-hand side holds at parity 1.
constexpr int kFinishThreads = 64;

__global__ void __launch_bounds__(kFinishThreads) prop_finish_kernel(const PropLevel P, const PropFinish Q)
{
    auto e_low = [&](int d) { return P.el0 ? P.el0[d] : 0.0; };
    __shared__ long long part[kFinishThreads / 32];
    __shared__ double s_miss;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, R = P.R1;
    {
        // (as integers: rounded sums would leave every row a common error of
        // 2^-53, which adds up over the operators of a call)
        long long s = 0;
        for (int i = -R + t; i <= R; i += kFinishThreads)
            s += fixed_of(P.e0[i], 62) + fixed_of(e_low(i), 62);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0)
            part[warp] = s;
    }
    __syncthreads();
    if (t == 0) {
        long long s = 1ll << 62;
        for (int i = 0; i < kFinishThreads / 32; ++i)
            s -= part[i];
        s_miss = (double)s * 0x1p-62;
    }
    __syncthreads();
    const double miss = s_miss;
    const int gid = blockIdx.x * kFinishThreads + t, n_int = 2 * R + 1, n_h = 4 * (R + 1), RX = R + 4, n_x = 2 * (2 * RX + 1);
    if (gid < n_int) {
        P.e1[gid - R] = P.e0[gid - R] + fma(miss, P.e0[gid - R], e_low(gid - R));
    } else if (gid < n_int + n_h) {
        const int w = gid - n_int, i = w / (R + 1) * P.hs + w % (R + 1);
        P.h1[i] = P.h0[i] + fma(miss, P.h0[i], P.hl0 ? P.hl0[i] : 0.0);
    } else if (Q.x && gid < n_int + n_h + n_x) {
        const int i = gid - n_int - n_h, phase = i & 1, d = (i >> 1) - RX;
        const int s = ((phase ^ Q.p0 ^ Q.k) & 1) ? -1 : 1, a = Q.p0 ^ phase;
        // the row with the exit, at column phase + d
        auto row = [&](int d) {
            auto low = [&](int q_phase, int x) { return P.el0 ? tap(P.el0, R, q_phase, x) : 0.0; };
            Dd v{tap(P.e0, R, a, d), low(a, d)};
            if (Q.exit)
                v = dd_add(dd_mul(Dd{Q.x1, 0.0}, v),
                           dd_mul(Dd{Q.x2, 0.0}, Dd{tap(P.e0, R, a ^ 1, d - s), low(a ^ 1, d - s)}));
            return v;
        };
        Dd v = row(d);
        if (Q.entry) {
            // v_j + r (v_partner - v_j), the pairs of parity 1 - p0
            const Dd w = row(((phase + d + 1 - Q.p0) & 1) ? d - 1 : d + 1);
            v = dd_add(v, dd_mul(Dd{Q.r, 0.0}, dd_add(w, Dd{-v.hi, -v.lo})));
        }
        Q.x[2 * i] = v.hi;
        Q.x[2 * i + 1] = v.lo;
        atomicMax(Q.x_max, (unsigned long long)__double_as_longlong(fabs(v.hi)));
    }
    const int o = blockIdx.x * (kFinishThreads / 32) + warp;
    if (!Q.F || o >= 2 * (R + 2))
        return;
    const int p = o / (R + 2), i = o % (R + 2), b = i & 1;
    if (!((P.par >> p) & 1))
        return;
    double s = 0.0;
#pragma unroll 4
    for (int d = -R + lane; d < -i; d += 32)
        s += tap(P.e0, R, p ^ b, d);
#pragma unroll 4
    for (int x = i - b + lane; x <= R; x += 32)
        s -= P.h0[(p * 2 + b) * P.hs + x];
    s = warp_sum(s);
    if (lane == 0) {
        if (p == 1)
            s -= Q.r * (tap(P.e0, R, p ^ b, -i) + (i - b <= R ? P.h0[(p * 2 + b) * P.hs + i - b] : 0.0));
        s = fma(miss, s, s);
        if (i == 0 && ((p + Q.k) & 1))
            s += Q.r;
        Q.F[p * P.hs + i] = s;
    }
}

// Digit tables for the tensor cores.  The operand of a block of 64 outputs n
// and window position k (64 + 2 W of them, from -W on) is the tap k - n - W;
// eight consecutive k of a row are one 16-byte piece, and a piece depends on
// n - k only (and on the parity of n): row rho of digit i's table holds
// d = 56 + W_i - rho + t, t = 0..7, and the operand's piece (n, k = 8c) is
// row n - 8c + 56 + 2 W_i.
constexpr int kPropQ = 2 * kPropRMax + 13;

__global__ void __launch_bounds__(1024) prop_digits_kernel(const double *x, const unsigned long long *x_max, int R,
                                                           int nd, int comp, int hb_max, int tab_cap, unsigned char *tab,
                                                           PropHeader *hdr)
{
    extern __shared__ long long q[];  // [2][kPropQ]
    constexpr int kQ = kPropQ, kMid = kPropRMax + 6;
    __shared__ long long s_sum[2];
    __shared__ float s_abs[32][2];
    __shared__ int s_W[8], s_row0[8];
    __shared__ int s_ok;
    const int t = threadIdx.x, RX = R + 4;
    if (t < 8)
        s_W[t] = 0;
    if (t < 2)
        s_sum[t] = 0;
    // largest scale that keeps the top digit below 127 and a row's sum of
    // magnitudes (1, more where the entry is folded in) below 2^62
    const int count = 2 * (2 * RX + 1);
    {
        // (FP32 and integers throughout: one SM's FP64 unit would take longer)
        float m = 0.0f;
        for (int i = t; i < count; i += 1024)
            m += fabsf((float)x[2 * i]);
        // the phases alternate over the threads
#pragma unroll
        for (int o = 16; o > 1; o >>= 1)
            m += __shfl_xor_sync(0xffffffffu, m, o);
        if ((t & 31) < 2)
            s_abs[t >> 5][t & 1] = m;
    }
    __syncthreads();
    float row_abs[2];  // sums of magnitudes of the two phases' rows
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        row_abs[p] = s_abs[t & 31][p];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            row_abs[p] += __shfl_xor_sync(0xffffffffu, row_abs[p], o);
    }
    const float abs_sum = row_abs[0] + row_abs[1];  // twice a row's
    // 126 / max in [2^(ex - 1), 2^ex): the quotient's exponent, one less to be safe of its rounding
    int ex, es;
    frexpf(125.99f / (float)__longlong_as_double((long long)*x_max), &ex);
    frexpf(0.499f * abs_sum, &es);
    const int e0 = ex - 1 + 8 * (nd - 1), e1 = 62 - es, E = e0 < e1 ? e0 : e1;
    auto add_sum = [&](int phase, long long v) {
        // two phases alternate over the lanes: sum the even and the odd lanes
        long long s = v;
        for (int o = 16; o > 1; o >>= 1)
            s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 31) < 2)
            atomicAdd(reinterpret_cast<unsigned long long *>(&s_sum[phase]), (unsigned long long)s);
    };
    for (int i0 = 0; i0 < count; i0 += 1024) {
        const int i = i0 + t, phase = i & 1, d = (i >> 1) - RX;
        long long v = 0;
        if (i < count) {
            v = fixed_of(x[2 * i], E) + fixed_of(x[2 * i + 1], E);
            q[phase * kQ + kMid + d] = v;
        }
        add_sum(phase, v);
    }
    __syncthreads();
    // the rows' sum is exactly 1, so a constant stays what it is: the taps
    // share what rounding left in proportion to their magnitudes (put on one
    // tap it would be white noise next to the smoothed field; in proportion
    // to the taps themselves, which at large r are of both signs and sum to
    // far less than their magnitudes, it changed each by up to r 2^-53 of
    // itself), the middle one takes the rest
    const float unit = __int_as_float((127 - E) << 23);
    const float miss[2] = {(float)((1LL << E) - s_sum[0]) * unit / row_abs[0],
                           (float)((1LL << E) - s_sum[1]) * unit / row_abs[1]};
    __syncthreads();
    if (t < 2)
        s_sum[t] = 0;
    __syncthreads();
    for (int i0 = 0; i0 < count; i0 += 1024) {
        const int i = i0 + t, phase = i & 1, d = (i >> 1) - RX;
        long long v = 0;
        if (i < count) {
            v = q[phase * kQ + kMid + d];
            v += __float2ll_rn(fabsf((float)v) * miss[phase]);
            q[phase * kQ + kMid + d] = v;
        }
        add_sum(phase, v);
    }
    __syncthreads();
    if (t < 2)
        q[t * kQ + kMid] += (1LL << E) - s_sum[t];
    __syncthreads();
    const unsigned long long bias = nd == kPropNd64 ? 0x0080808080808080ull : 0x80808080ull;
    int w[kPropNd64] = {};
    for (int i = t; i < count; i += 1024) {
        const int phase = i & 1, d = (i >> 1) - RX;
        const unsigned long long y = (unsigned long long)q[phase * kQ + kMid + d] + bias;
#pragma unroll
        for (int j = 0; j < kPropNd64; ++j)
            if (j < nd && ((y >> (8 * (nd - 1 - j))) & 255) != 128)
                w[j] = max(w[j], d < 0 ? -d : d);
    }
#pragma unroll
    for (int j = 0; j < kPropNd64; ++j) {
        const int m = __reduce_max_sync(0xffffffffu, w[j]);
        if ((t & 31) == 0)
            atomicMax(&s_W[j], m);
    }
    __syncthreads();
    if (t == 0) {
        int rows = 0, ok = 1;
        for (int j = 0; j < nd; ++j) {
            int W = (s_W[j] + 15) / 16 * 16;
            if (W > hb_max * kPropBlk) {
                W = hb_max * kPropBlk;
                ok = 0;
            }
            s_W[j] = W;
            s_row0[j] = rows;
            rows += 120 + 2 * W;
        }
        if (rows * 16 > tab_cap) {
            ok = 0;
            rows = 0;
        }
        s_ok = ok;
        hdr->E = E;
        // What the digits drop (products of the next weight, of N taps) has a
        // root mean square of 2^-10 sqrt(N) units of the sums, FP32 2^-1.3
        // sqrt(N).  FP64: N grows with the taps' scale, and a block's results
        // are kept to 2^-54 of their largest.  FP32: to 2^-22 (the compensated
        // kernel's 2^-23; wide taps smooth out more of its early roundings),
        // where the steps one by one err as much.  Rows of far larger
        // magnitudes than their sum (large r) cancel, also step by step.
        hdr->keep = es >= 2 ? 0 : nd == kPropNd64 ? (E + 38) >> 1 : comp && E < 38 ? 34 : 33;
        hdr->ok = ok;
        hdr->rows = rows;
        for (int j = 0; j < nd; ++j) {
            hdr->W[j] = s_W[j];
            hdr->row0[j] = s_row0[j];
        }
    }
    __syncthreads();
    if (!s_ok)
        return;
    for (int j = 0; j < nd; ++j) {
        const int W = s_W[j], sh = 8 * (nd - 1 - j);
        for (int rho = t; rho < 120 + 2 * W; rho += 1024) {
            __align__(16) __half v[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int d = 56 + W - rho + c;
                unsigned long long y = bias;
                if (d >= -RX && d <= RX)
                    y += (unsigned long long)q[(rho & 1) * kQ + kMid + d];
                v[c] = __int2half_rn((int)((y >> sh) & 255) - 128);
            }
            *reinterpret_cast<uint4 *>(tab + (size_t)(s_row0[j] + rho) * 16) = *reinterpret_cast<const uint4 *>(v);
        }
    }
}

// ---- dot products --------------------------------------------------------

// All rows of a grid too small for tiles, or the blocks the tiles listed.
template <typename T>
__global__ void __launch_bounds__(256) prop_dot_kernel(const __grid_constant__ PropRun P)
{
    extern __shared__ double s_w[];
    double *taps = s_w + kDotWin;
    __shared__ DotShared<kDotRows> sh;
    if (P.tiles > 0) {
        const long long items = (long long)*reinterpret_cast<const volatile int *>(P.count) * (kPropBlk / kDotRows);
        if (blockIdx.x == 0 && threadIdx.x == 0)
            *P.count_next = 0;
        if (blockIdx.x < items)
            dot_stage<256>(P, reinterpret_cast<typename PairOf<T>::E *>(taps));
        for (long long it = blockIdx.x; it < items; it += gridDim.x)
            dot_listed<T, 256, true>(P, sh, s_w, taps, it);
    } else {
        dot_stage<256>(P, reinterpret_cast<typename PairOf<T>::E *>(taps));
        const int shift = item_shift(P);
        for (long long r0 = blockIdx.x * (long long)kDotRows - shift; r0 < P.n; r0 += gridDim.x * (long long)kDotRows) {
            const long long r1 = r0 + kDotRows;
            dot_rows<T, 256, kDotRows, 1, true>(P, sh, s_w, taps, r0 > 0 ? r0 : 0, r1 < P.n ? r1 : P.n);
        }
    }
}

// ---- tiles on the tensor cores -------------------------------------------

// Blocks whose values all lie below 2^-P.range of the largest value of the
// window go to the dot products: the fixed-point sum would leave them too few
// digits of their own.  So do those below 2^-kFar of the largest value that
// reaches them at all: what lies beyond the window counts with taps that the
// digits leave out, 2^-64 (FP32: 2^-39) of the sum in all.
template <typename T>
struct TileShape;
template <>
struct TileShape<double> {
    static constexpr int ND = kPropNd64, NV = kPropNv64, kHb = kPropHb64, kTab = kPropTab64, kFar = 10;
    static constexpr int kGroups = 9, kCols = 512;
};
template <>
struct TileShape<float> {
    static constexpr int ND = kPropNd32, NV = kPropNv32, kHb = kPropHb32, kTab = kPropTab32, kFar = 10;
    static constexpr int kGroups = 4, kCols = 256;
};

// A value digit's plane: a 128-byte row of 64 FP16 digits per block of the
// tile and its halo, the row's eight 16-byte pieces in descending order and
// swizzled (piece position ^ row mod 8) as the tensor cores' 128-byte swizzle
// reads them: a window that starts blocks further on is the same plane rows
// further on, and every eight rows of a piece cover all banks.  (The same
// plane unswizzled, rows of 16 bytes, took 85 to 90 cycles an MMA.)
template <typename T>
constexpr int kPlaneRows = sizeof(T) == 8 ? kPropRows64 : kPropTileBlks + 2 * TileShape<T>::kHb;
// (the MMA reads 128 rows from wherever a window starts: past the last plane's
// end in a tile of fewer blocks)
template <typename T>
constexpr int kTileSmem = TileShape<T>::kTab + (TileShape<T>::NV * kPlaneRows<T> + kPropTileBlks + 2 * TileShape<T>::kHb - kPlaneRows<T>) * 128 + 1024;
// The finished rows leave through the planes' space, padded so that the lanes
// (a row each) write different banks.
template <typename T>
constexpr int kStageRow = kPropBlk * (int)sizeof(T) + 16;

static_assert(kTileSmem<double> <= 232448 - 2560 && kTileSmem<float> <= 232448 - 2560, "tile exceeds shared memory");

// Digit products of each accumulator, in issue order: sum g holds the products
// of weight(g) whose tap digit lies in [lo(g), hi(g)], the value digit being
// weight(g) less that.  FP64's weight 4 takes
// two sums so that each stays exact; its first and last sum share one
// accumulator (512 columns hold eight).
struct Groups64 {
    __host__ __device__ static constexpr int weight(int g) { return g <= 3 ? 7 - g : 8 - g; }
    __host__ __device__ static constexpr int lo(int g) { return g == 4 ? 3 : 0; }
    __host__ __device__ static constexpr int hi(int g) { return g == 0 ? 6 : g == 3 ? 2 : weight(g); }
};
struct Groups32 {
    __host__ __device__ static constexpr int weight(int g) { return 3 - g; }
    __host__ __device__ static constexpr int lo(int) { return 0; }
    __host__ __device__ static constexpr int hi(int g) { return weight(g); }
};
template <typename T>
struct GroupsOf;
template <>
struct GroupsOf<double> {
    using G = Groups64;
};
template <>
struct GroupsOf<float> {
    using G = Groups32;
};

// Exponent code of a value: 0 for zero, else its biased exponent (1 for
// subnormals; all ones for infinities and NaN).
__device__ __forceinline__ int code_of(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu;
    const int e = (int)(hi >> 20);
    return e ? e : ((hi | (unsigned)__double2loint(x)) ? 1 : 0);
}
__device__ __forceinline__ int code_of(float x)
{
    const unsigned u = __float_as_uint(x) & 0x7fffffffu;
    const int e = (int)(u >> 23);
    return e ? e : (u ? 1 : 0);
}
template <typename T>
constexpr int kCodeInf = sizeof(T) == 8 ? 2047 : 255;

// Whether a tile leaves a block to dot products for its values: the code of
// its largest, of the window's and of the cone's.  (Where the results will be
// looked at, they decide, and the values only spare the tile a lost cause:
// where a smooth field crosses zero they may be small.)
template <typename T>
__device__ __forceinline__ bool values_too_small(const PropRun &P, int keep, int q, int ref, int cone)
{
    return cone == kCodeInf<T> || q == 0 || q < ref - P.range - (keep > 0 ? 4 : 0) || q < cone - TileShape<T>::kFar;
}

// Whether it does for its results: bits[0] those of block `row`'s largest sum.
__device__ __forceinline__ bool results_too_small(const PropRun &P, const int *bits, int row, int rows, int keep)
{
    int b = bits[row];
    if (P.near)
        b = max(b, max(row > 0 ? bits[row - 1] : 0, row + 1 < rows ? bits[row + 1] : 0));
    return b < keep;
}

// round(x 2^(62 - e)), FP32 round(x 2^(30 - e)), for |x| < 2^e, e = code -
// bias + 1 of the tile's largest value; `ref` is that largest code.
__device__ __forceinline__ long long to_fixed(double x, int ref)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(u >> 52) & 0x7ff;
    unsigned long long m = u & 0x000fffffffffffffull;
    if (e)
        m |= 0x0010000000000000ull;
    // x = m 2^(ec - 1075), 2^e_tile = 2^(ref - 1022): shift by ec - ref + 9
    const int sh = (e ? e : 1) - ref + 9;
    if (sh >= 0) {
        m <<= sh;
    } else {
        const int n = -sh < 60 ? -sh : 60;
        m = (m + (1ull << (n - 1))) >> n;
    }
    return (long long)u < 0 ? -(long long)m : (long long)m;
}
__device__ __forceinline__ int to_fixed(float x, int ref)
{
    const unsigned u = __float_as_uint(x);
    const int e = (int)(u >> 23) & 0xff;
    unsigned m = u & 0x007fffffu;
    if (e)
        m |= 0x00800000u;
    // x = m 2^(ec - 150), 2^e_tile = 2^(ref - 126): shift by ec - ref + 6
    const int sh = (e ? e : 1) - ref + 6;
    if (sh >= 0) {
        m <<= sh;
    } else {
        const int n = -sh < 30 ? -sh : 30;
        m = (m + (1u << (n - 1))) >> n;
    }
    return (int)u < 0 ? -(int)m : (int)m;
}

// x 2^e for a normal x whose product is normal too; and 2^e.
__device__ __forceinline__ float add_exponent(float x, int e) { return __int_as_float(__float_as_int(x) + (e << 23)); }
template <typename T>
__device__ __forceinline__ T pow2(int e);
template <>
__device__ __forceinline__ double pow2<double>(int e)
{
    return __hiloint2double((e + 1023) << 20, 0);
}
template <>
__device__ __forceinline__ float pow2<float>(int e)
{
    return __int_as_float((e + 127) << 23);
}

// z 2^e rounded to nearest even, for a normal result.
template <typename T>
__device__ __forceinline__ T from_fixed(long long z, int e);
template <>
__device__ __forceinline__ double from_fixed<double>(long long z, int e)
{
    return fixed_to_double(z, e);
}
template <>
__device__ __forceinline__ float from_fixed<float>(long long z, int e)
{
    return z ? add_exponent((float)z, e) : 0.0f;
}

// Whether from_fixed takes every 64-bit integer times 2^e.
template <typename T>
__device__ __forceinline__ bool plain_exponent(int e)
{
    return sizeof(T) == 8 ? e >= -1021 && e <= 959 : e >= -125 && e <= 63;
}

// Two digits as FP16: bytes b of two biased values to (b - 128).
__device__ __forceinline__ uint32_t half_pair(uint32_t a, uint32_t b, uint32_t sel)
{
    const uint32_t v = (__byte_perm(a, b, sel) & 0x00ff00ffu) | 0x64006400u;  // 1024 + byte
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&v), __float2half2_rn(1152.0f));
    return *reinterpret_cast<const uint32_t *>(&h);
}

// K-major operand with 128-byte rows and the 128-byte swizzle: groups of eight
// rows 1024 bytes apart (the leading offset is unused).
__device__ __forceinline__ uint64_t swizzled_desc(uint32_t addr)
{
    return ((addr & 0x3FFFF) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes
// (contiguous, 128 bytes), `lead` bytes apart along K and 128 along the rows.
__device__ __forceinline__ uint64_t plain_desc(uint32_t addr, uint32_t lead)
{
    return ((addr & 0x3FFFF) >> 4) | ((uint64_t)(lead >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}

// kind::f16 with FP16 operands and FP32 accumulators, M = 128, N = 64.
constexpr uint32_t kIdescF16 = (1u << 4) | ((uint32_t)(kPropBlk >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

// Eight values as digits, one 16-byte piece of each plane.
template <typename T>
__device__ __forceinline__ void convert8(const T (&x)[8], int ref, unsigned char *dst, size_t plane)
{
    constexpr int NV = TileShape<T>::NV;
    uint32_t lo[8], hi[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        if (NV == kPropNv64) {
            const unsigned long long y = (unsigned long long)to_fixed((double)x[v], ref) + 0x8080808080808080ull;
            lo[v] = (uint32_t)y;
            hi[v] = (uint32_t)(y >> 32);
        } else {
            lo[v] = (uint32_t)to_fixed((float)x[v], ref) + 0x80808080u;
        }
    }
#pragma unroll
    for (int d = 0; d < NV; ++d) {
        const int byte = NV - 1 - d;
        const uint32_t sel = byte < 4 ? (uint32_t)(byte | (byte << 4) | ((byte + 4) << 8) | ((byte + 4) << 12))
                                      : (uint32_t)((byte - 4) | ((byte - 4) << 4) | (byte << 8) | (byte << 12));
        uint4 q;
        q.x = byte < 4 ? half_pair(lo[0], lo[1], sel) : half_pair(hi[0], hi[1], sel);
        q.y = byte < 4 ? half_pair(lo[2], lo[3], sel) : half_pair(hi[2], hi[3], sel);
        q.z = byte < 4 ? half_pair(lo[4], lo[5], sel) : half_pair(hi[4], hi[5], sel);
        q.w = byte < 4 ? half_pair(lo[6], lo[7], sel) : half_pair(hi[6], hi[7], sel);
        *reinterpret_cast<uint4 *>(dst + (size_t)d * plane) = q;
    }
}

// The accumulators of a row's points: 64-bit sums in units of weight 5 (FP32:
// weight 3), and for FP64 the next 16 bits of each (weights 6 and 7), two to a
// register.
template <typename T, int N>
struct Sums {
    long long hi[N] = {};
    uint32_t low[sizeof(T) == 8 ? N / 2 : 1] = {};
    // one digit sum of weight w (FP64: 7 first, then 6)
    __device__ __forceinline__ void fold(int v, int w, int z)
    {
        if (sizeof(T) == 4) {
            hi[v] += (long long)z << (8 * (3 - (w < 4 ? w : 3)));
        } else if (w >= 6) {
            const long long s = w == 7 ? (long long)z : hi[v] + ((long long)z << 8);
            if (w == 6) {
                low[v / 2] |= ((uint32_t)s & 0xffff) << (v & 1) * 16;
                hi[v] = s >> 16;
            } else {
                hi[v] = s;
            }
        } else {
            hi[v] += (long long)z << (8 * (5 - w));
        }
    }
    __device__ __forceinline__ int last(int v) const { return (int)(low[v / 2] >> (v & 1) * 16) & 0xffff; }
    // bits of the largest
    __device__ __forceinline__ int bits() const
    {
        unsigned long long m = 0;
#pragma unroll
        for (int v = 0; v < N; ++v)
            m |= (unsigned long long)(hi[v] ^ (hi[v] >> 63));
        return 64 - __clzll((long long)m);
    }
};

// A sum and its 16 low bits, the sum of `bits` bits or fewer, as one integer
// times 2^-shift.
__device__ __forceinline__ int join_shift(int bits) { return bits < 46 ? 16 : 62 - bits; }
__device__ __forceinline__ long long join(long long hi, int low, int shift)
{
    return (long long)((unsigned long long)hi << shift) + (low >> (16 - shift));
}

// out = (hi + low 2^-16) 2^ex, rounded once (FP32: no low part).
template <typename T>
__device__ __forceinline__ T finish_point(long long hi, int low, int ex, bool plain)
{
    long long z = hi;
    if (sizeof(T) == 8) {
        const int shift = join_shift(64 - __clzll(hi ^ (hi >> 63)));
        z = join(hi, low, shift);
        if (plain)
            return from_fixed<T>(z, ex - shift);
        // near the ends of the exponent range
        return (T)z * pow2<T>(ex / 2) * pow2<T>(ex - ex / 2 - shift);
    }
    return plain ? from_fixed<T>(z, ex) : (T)z * pow2<T>(ex / 2) * pow2<T>(ex - ex / 2);
}
// The exponent of a tile's sums, and whether finish_point's results are normal
// whatever the sum: FP64 2^ex = 2^(e + 2 - E), FP32 2^(e - 6 - E), 2^e above
// the tile's largest value (code `ref`).
template <typename T>
__device__ __forceinline__ int sum_exponent(int ref, int E) { return sizeof(T) == 8 ? ref - 1022 + 2 - E : ref - 126 - 6 - E; }
template <typename T>
__device__ __forceinline__ bool plain_sums(int ex)
{
    return plain_exponent<T>(ex) && (sizeof(T) == 4 || plain_exponent<T>(ex - 16));
}

// N finished points of a row to the staging buffer: out = acc 2^ex.
template <typename T, int N>
__device__ __forceinline__ void finish_row(const long long (&acc)[N], int ex, unsigned char *o)
{
    if (plain_exponent<T>(ex)) {
#pragma unroll
        for (int v = 0; v < N; v += 16 / sizeof(T)) {
            T y[16 / sizeof(T)];
#pragma unroll
            for (int z = 0; z < (int)(16 / sizeof(T)); ++z)
                y[z] = from_fixed<T>(acc[v + z], ex);
            *reinterpret_cast<uint4 *>(o + v * sizeof(T)) = *reinterpret_cast<const uint4 *>(y);
        }
    } else {  // near the ends of the exponent range
        const T s1 = pow2<T>(ex / 2), s2 = pow2<T>(ex - ex / 2);
#pragma unroll
        for (int v = 0; v < N; ++v)
            reinterpret_cast<volatile T *>(o)[v] = (T)acc[v] * s1 * s2;
    }
}

// The four MMAs of 64 points of a window, `end` steps of 16 in all: ad, bd at
// the first step, q the window's first piece of its row.
__device__ __forceinline__ void issue_product(bool leader, uint32_t dcol, uint64_t ad, uint64_t bd, int q, int end,
                                              uint32_t &acc)
{
    const uint64_t a0 = (uint64_t)(6 - q), a1 = (uint64_t)(6 - ((q + 2) & 7) + ((q + 2) & 8)),
                   a2 = (uint64_t)(6 - ((q + 4) & 7) + ((q + 4) & 8)), a3 = (uint64_t)(6 - ((q + 6) & 7) + ((q + 6) & 8));
    int s = 0;
#pragma unroll 1
    for (; s + 4 <= end; s += 4) {
        tc_mma_if(leader, dcol, ad + a0, bd, kIdescF16, acc);
        tc_mma_if(leader, dcol, ad + a1, bd - 16, kIdescF16, 1);
        tc_mma_if(leader, dcol, ad + a2, bd - 32, kIdescF16, 1);
        tc_mma_if(leader, dcol, ad + a3, bd - 48, kIdescF16, 1);
        acc = 1;
        ad += 8;
        bd -= 64;
    }
    if (s < end) {
        tc_mma_if(leader, dcol, ad + a0, bd, kIdescF16, acc);
        if (s + 1 < end)
            tc_mma_if(leader, dcol, ad + a1, bd - 16, kIdescF16, 1);
        if (s + 2 < end)
            tc_mma_if(leader, dcol, ad + a2, bd - 32, kIdescF16, 1);
        acc = 1;
    }
}

// 16 warps that convert and drain: chains of integer instructions with little
// else to hide their latency.  2 that issue the MMAs, every other sum each:
// one warp issues one in 54 cycles, and spends 200 to 300 between two digit
// products, where the tensor cores take 48.
constexpr int kTileWarps = 16, kMmaWarps = 2;
constexpr int kTileConv = 32 * kTileWarps, kTileThreads = kTileConv + 32 * kMmaWarps;
constexpr int kEdgeParts = kTileWarps / kEdgeRows, kEdgeScratch = 32 * kEdgeParts * (kEdgeRows + 2);
constexpr int kTileCols = kPropBlk / (kTileWarps / 4);  // points of a block a thread drains
static_assert((kDotWin + kEdgeScratch + dot_taps(kPropR64Max)) * 8 <= kTileSmem<double> - 1024 &&
                  (kDotWin + kEdgeScratch + dot_taps(kPropRMax)) * 8 <= kTileSmem<float> - 1024,
              "the rows near a wall fit");

// SPLIT: a cluster of 2, 4 or 8 CTAs per tile, for grids with fewer tiles than
// SMs.  Each CTA issues its share of every digit product's MMAs, in units of
// four; the sums are integers, so the shares add up to what one CTA's sum
// would have been, bit for bit.  They meet in shared memory as 64-bit
// integers, and each CTA finishes its share of the points of every block.
// The conversion is not shared: a digit product's window is its own, and
// their union is nearly the whole one.  The launcher weighs the tile's time
// against that of the wall rows, which need the CTAs without a tile: n =
// 100,003, k = 1999, FP64 takes 4 CTAs a tile, 68 -> 42 us a call (8: 57, 2:
// 59); n = 500,000 takes 2, 82 -> 67 us; n = 300,001, FP32, two operators:
// 100 -> 82 us.
template <typename T>
constexpr int kPartHigh = kPropTileBlks * kPropBlk * 8;  // bytes of a CTA's sums [64 points][128 blocks]; FP64: 16 last bits follow
static_assert(kPartHigh<double> / 8 * 10 <= kPropTab64 && kPartHigh<float> <= kPropTab32, "the sums fit the tables' space");
// One partial sum from each CTA of the cluster, and for FP64 its last bits.
template <typename T, int C>
__device__ __forceinline__ void add_parts(uint32_t addr, uint32_t addr_low, long long &hi, int &low)
{
    long long h[C];
    unsigned short l[C];
#pragma unroll
    for (int p = 0; p < C; ++p) {
        uint32_t a, b;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(p));
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(addr_low), "r"(p));
        asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(h[p]) : "r"(a) : "memory");
        if (sizeof(T) == 8)
            asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(l[p]) : "r"(b) : "memory");
    }
    hi = low = 0;
#pragma unroll
    for (int p = 0; p < C; ++p) {
        hi += h[p];
        if (sizeof(T) == 8)
            low += l[p];
    }
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename T, bool SPLIT>
__global__ void __launch_bounds__(kTileThreads, 1) prop_tile_kernel(const __grid_constant__ PropRun P)
{
    using S = TileShape<T>;
    using G = typename GroupsOf<T>::G;
    constexpr int ND = S::ND, C = kPlaneRows<T>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                          ~static_cast<uintptr_t>(1023));
    unsigned char *xp = sm + S::kTab;  // value digits: [digit][C rows][128 bytes], then the finished rows
    __shared__ __align__(8) uint64_t tab_full, done[S::kGroups], reuse;
    __shared__ uint32_t tmem_sh;
    __shared__ volatile int s_abort;
    __shared__ int s_code[C + 8];
    __shared__ int s_max[2];  // largest code: the window, the whole cone
    __shared__ int s_keep;    // blocks the tile itself answers
    __shared__ int s_bits[kPropTileBlks];  // bits of each block's largest sum
    __shared__ int s_left;
    __shared__ PropHeader s_hdr;
    __shared__ DotShared<kEdgeRows> s_dot;
    __shared__ int4 s_prod[S::kGroups * ND];  // see below
    __shared__ int s_used;                    // split: sums this CTA has products of

    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t < (int)(sizeof(PropHeader) / 4))
        reinterpret_cast<int *>(&s_hdr)[t] = reinterpret_cast<const int *>(P.hdr)[t];
    if (t == 0) {
        bar_init(&tab_full, 1);
        for (int g = 0; g < S::kGroups; ++g)
            bar_init(&done[g], 1);
        bar_init(&reuse, kTileWarps);
        s_used = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    if (warp == kTileWarps) {
        tmem_alloc(&tmem_sh, S::kCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = tmem_sh;
    if (blockIdx.x == 0 && t < 3 && P.zero[t])
        *P.zero[t] = 0;
    const int ctas = SPLIT ? P.split : 1, lg = SPLIT ? 31 - __clz(ctas) : 0, rank = SPLIT ? (int)blockIdx.x & (ctas - 1) : 0;
    // Tiles (split: one per cluster), then the rows near a wall: the CTAs with
    // a tile less (split: without one) take edge_rounds items each, and what
    // is left is everyone's.
    const int busy = SPLIT ? (int)P.tiles * ctas : (int)(P.tiles % gridDim.x);  // CTAs with a tile more
    const int spare = busy ? (int)gridDim.x - busy : 0, me = (int)blockIdx.x - busy;
    const int shift = item_shift(P);
    const long long edge_l = item_count(P.rows_l, kEdgeRows, shift);
    const long long edges = edge_l + item_count(P.n - P.row_r, kEdgeRows, shift);
    const long long early = (long long)spare * P.edge_rounds < edges ? (long long)spare * P.edge_rounds : edges;
    const long long first_edge = spare > 0 && me >= 0 && me < early ? P.tiles + me : P.tiles + early + blockIdx.x;
    const long long first = SPLIT ? (me < 0 ? (long long)blockIdx.x >> lg : first_edge)
                                  : ((long long)blockIdx.x < P.tiles ? (long long)blockIdx.x : first_edge);
    auto after = [&](long long x) {
        if (x < P.tiles)
            return !SPLIT && x + gridDim.x < P.tiles ? x + (long long)gridDim.x : first_edge;
        if (x < P.tiles + early)
            return x + spare < P.tiles + early ? x + spare : P.tiles + early + (long long)blockIdx.x;
        return x + (long long)gridDim.x;
    };
    const int hb = P.hb, per = P.per, ok_tab = s_hdr.ok && s_hdr.rows * 16 <= S::kTab;
    const bool has_tab = ok_tab && first < P.tiles;
    if (t == 0 && has_tab) {
        bar_expect_tx(&tab_full, (uint32_t)s_hdr.rows * 16);
        bulk_load(sm, P.tab, (uint32_t)s_hdr.rows * 16, &tab_full);
    }
    // the digit products' first descriptors and steps, in issue order
    for (int z = t; z < S::kGroups * ND; z += kTileThreads) {
        const int g = z / ND, i = z % ND;
        if (i < G::lo(g) || i > G::hi(g))
            continue;
        const int W = s_hdr.W[i], steps = (kPropBlk + 2 * W) / 16, units = (steps + 3) / 4;
        int u0 = 0, u1 = units;
        if (SPLIT) {
            const int turn = (g + 3 * i) & (ctas - 1);
            u0 = (units * rank + turn) >> lg;
            u1 = (units * (rank + 1) + turn) >> lg;
            if (u1 > u0)
                atomicOr(&s_used, 1 << g);
        }
        // window position -W: block -W >> 6, piece q of its row (descending, as the
        // table's rows run); four steps go 64 points on, to the next row
        int4 p;
        p.x = (int)((uint32_t)(((G::weight(g) - i) * C + hb + (-W >> 6)) * 128) >> 4) + 8 * u0;
        p.y = s_hdr.row0[i] + 48 + 2 * W - 64 * u0;
        p.z = (-W & 63) >> 3;
        p.w = (4 * u1 < steps ? 4 * u1 : steps) - 4 * u0;
        s_prod[z] = p;
    }
    bool tab_waited = false, staged = false;
    uint32_t phase = 0;
    const T *in = static_cast<const T *>(P.in);
    T *out = static_cast<T *>(P.out);

    for (long long tile = first; tile < P.tiles + edges; tile = after(tile)) {
        if (tile >= P.tiles) {
            // rows near a wall, after the tiles: they fill the last wave
            double *s_w = reinterpret_cast<double *>(sm), *taps = s_w + kDotWin + kEdgeScratch;
            if (warp < kTileWarps) {
                if (!staged) {
                    // the tables' and planes' space: nothing still writes or reads it
                    bulk_wait_read0();
                    if (has_tab)
                        bar_drain(&tab_full, 0, kWaitLimitCycles);
                    asm volatile("bar.sync 1, %0;" ::"n"(kTileConv) : "memory");
                    dot_stage<kTileConv>(P, reinterpret_cast<typename PairOf<T>::E *>(taps));
                    staged = true;
                }
                const long long x = tile - P.tiles;
                const long long a = x < edge_l ? 0 : P.row_r, b = x < edge_l ? P.rows_l : P.n;
                const long long r0 = a + (x < edge_l ? x : x - edge_l) * kEdgeRows - shift, r1 = r0 + kEdgeRows;
                dot_rows<T, kTileConv, kEdgeRows, kEdgeParts, true>(P, s_dot, s_w, taps, r0 > a ? r0 : a, r1 < b ? r1 : b);
            }
            continue;
        }
        const long long b0 = P.blk0 + tile * per;                 // first output block
        const int nb = (int)(P.blk1 - b0 < per ? P.blk1 - b0 : per);
        const long long base = (b0 - hb) * kPropBlk;              // first point of the window
        const int chunks = (per + 2 * hb) * 8;                    // 8 points each
        constexpr int kIter = (C * 8 + kTileConv - 1) / kTileConv;
        if (t < 2)
            s_max[t] = 0;
        if (t == 2)
            s_keep = 0;
        if (t == 3)  // the step-by-step form is going to answer for the whole grid
            s_left = *reinterpret_cast<const volatile int *>(P.count) > P.gate_min;
        __syncthreads();
        // the window in registers, a chunk of 8 points per turn; the largest
        // exponent of every block and of the window
        T x[kIter][8];
        if (warp < kTileWarps) {
            int wmax = 0;
            constexpr int kV = 16 / sizeof(T);
#pragma unroll
            for (int c = 0; c < kIter; ++c) {
                const int u = c * kTileConv + t;
                const long long j = base + (long long)u * 8;
                // whole chunks only: the few points past the last one lie
                // beyond every window that is used
                const bool in_range = u < chunks && j + 8 <= P.n;
#pragma unroll
                for (int v = 0; v < 8 / kV; ++v) {
                    uint4 q = make_uint4(0, 0, 0, 0);
                    if (in_range)
                        q = *reinterpret_cast<const uint4 *>(in + j + v * kV);
                    *reinterpret_cast<uint4 *>(&x[c][v * kV]) = q;
                }
            }
            // the next tile's window on its way to L2
            if (!SPLIT && tile + gridDim.x < P.tiles) {
                const long long nx = base + (long long)gridDim.x * per * kPropBlk + (long long)t * 128 / sizeof(T);
                for (long long z = nx; z < nx - (long long)t * 128 / sizeof(T) + (long long)chunks * 8 && z < P.n;
                     z += (long long)kTileConv * 128 / sizeof(T))
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(in + z));
            }
#pragma unroll
            for (int c = 0; c < kIter; ++c) {
                const int u = c * kTileConv + t;
                int m = 0;
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    const int q = code_of(x[c][v]);
                    m = q > m ? q : m;
                }
                wmax = m > wmax ? m : wmax;
                // eight lanes hold a block
                for (int z = 1; z < 8; z <<= 1) {
                    const int y = __shfl_xor_sync(0xffffffffu, m, z);
                    m = y > m ? y : m;
                }
                if ((t & 7) == 0 && u < chunks)
                    s_code[u >> 3] = m;
            }
            // the rest of the cone: everything that reaches the tile's blocks in
            // k steps, the walls included (tiles leave out what a wall adds
            // beyond the rows near it, so it counts against their own values)
            int cmax = wmax;
            const long long clo = b0 * kPropBlk - P.k - 2, chi = (b0 + nb) * kPropBlk + P.k + 2;
            cmax = max(cmax, max(clo <= 0 ? P.wall_l : 0, chi >= P.n ? P.wall_r : 0));
            auto scan = [&](long long a, long long b) {
                for (long long j = a + t; j < b; j += 4 * kTileConv)
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        cmax = max(cmax, code_of(j + u * kTileConv < b ? in[j + u * kTileConv] : (T)0));
            };
            scan(clo > 0 ? clo : 0, base);
            scan(base + (long long)chunks * 8, chi < P.n ? chi : P.n);
            for (long long j = (P.n & ~7LL) + t; j < P.n && j < chi; j += kTileConv)  // the ragged end
                cmax = max(cmax, code_of(in[j]));
            bulk_wait_read0();  // the last tile's rows have left the planes
            wmax = __reduce_max_sync(0xffffffffu, wmax);
            cmax = __reduce_max_sync(0xffffffffu, cmax);
            if (lane == 0) {
                atomicMax(&s_max[0], wmax);
                atomicMax(&s_max[1], cmax);
            }
        }
        __syncthreads();
        // (a cluster's CTAs must agree, and have one tile only)
        if (!SPLIT && s_left)
            break;
        const int ref = s_max[0], cone = s_max[1];
        bool listed = false;  // block t
        if (t < nb) {
            s_bits[t] = 0;
            listed = cone > 0 && (!ok_tab || values_too_small<T>(P, s_hdr.keep, s_code[hb + t], ref, cone));
            if (listed && rank == 0)
                P.list[atomicAdd(P.count, 1)] = (int)(b0 + t);
            else if (!listed && cone > 0)
                s_keep = 1;
        }
        if (warp < kTileWarps && cone != kCodeInf<T>) {
#pragma unroll
            for (int c = 0; c < kIter; ++c) {
                const int u = c * kTileConv + t;
                if (u < chunks) {
                    // biased fixed-point values: every byte is a digit + 128
                    unsigned char *dst = xp + (u >> 3) * 128 + ((7 - (u & 7)) ^ ((u >> 3) & 7)) * 16;
                    convert8(x[c], ref, dst, (size_t)C * 128);
                }
            }
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const bool keep = s_keep != 0;
        if (warp >= kTileWarps) {
            if (keep) {
                // the whole warp runs the loop, so descriptors stay in uniform
                // registers; one lane issues
                const bool leader = elect_one();
                bool ok = true;
                if (!tab_waited) {
                    ok = bar_wait(&tab_full, 0, kWaitLimitCycles, &s_abort);
                    tab_waited = true;
                }
                const uint64_t ad0 = swizzled_desc(saddr(xp)), bd0 = plain_desc(saddr(sm), 128);
#pragma unroll 1
                for (int g = warp - kTileWarps; ok && g < S::kGroups; g += kMmaWarps) {
                    const int lo = G::lo(g), hi = G::hi(g);
                    uint32_t acc = 0;
                    if (g * kPropBlk >= S::kCols) {
                        // sum 0's accumulator again, once the warps have read it
                        ok = bar_wait(&reuse, phase, kWaitLimitCycles, &s_abort);
                        tc_fence_after();
                        if (!ok)
                            break;
                    }
                    const uint32_t dcol = tbase + (uint32_t)(g * kPropBlk % S::kCols);
#pragma unroll 1
                    for (int i = lo; i <= hi; ++i) {
                        const int4 p = s_prod[g * ND + i];
                        issue_product(leader, dcol, ad0 + (uint32_t)__shfl_sync(0xffffffffu, p.x, 0),
                                      bd0 + (uint32_t)__shfl_sync(0xffffffffu, p.y, 0), __shfl_sync(0xffffffffu, p.z, 0),
                                      __shfl_sync(0xffffffffu, p.w, 0), acc);
                    }
                    tc_commit_if(leader, &done[g]);
                    __syncwarp();
                }
                if (!ok && lane == 0) {
                    atomicExch(P.err, kDevTimeout);
                    s_abort = 1;
                }
            }
            __syncwarp();
        } else if (keep) {
            // drain: kTileCols columns (points of a block) of the lane's block
            const int row = (warp & 3) * 32 + lane, col = (warp >> 2) * kTileCols;
            Sums<T, kTileCols> acc;
            bool ok = true;
#pragma unroll
            for (int g = 0; g < S::kGroups; ++g) {
                ok = ok && bar_wait(&done[g], phase, kWaitLimitCycles, &s_abort);
                if (!__any_sync(0xffffffffu, !ok)) {
                    tc_fence_after();
                    uint32_t v[kTileCols];
                    tmem_ld16(tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(g * kPropBlk % S::kCols + col), v);
                    tmem_wait_ld();
                    if (g == 0 && S::kGroups * kPropBlk > S::kCols) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0)
                            bar_arrive(&reuse);
                    }
                    const int w = G::weight(g);
                    const bool mine = !SPLIT || ((s_used >> g) & 1);
#pragma unroll
                    for (int q = 0; q < kTileCols; ++q) {
                        const int z = mine ? __float2int_rn(__uint_as_float(v[q])) : 0;
                        acc.fold(q, w, z);
                    }
                }
            }
            if (__any_sync(0xffffffffu, !ok)) {
                if (lane == 0) {
                    atomicExch(P.err, kDevTimeout);
                    s_abort = 1;
                }
            } else if (SPLIT) {
#pragma unroll
                for (int v = 0; v < kTileCols; ++v) {
                    const int at = (col + v) * kPropTileBlks + row;
                    if (sizeof(T) == 8)
                        reinterpret_cast<unsigned short *>(sm + kPartHigh<T>)[at] = (unsigned short)acc.last(v);
                    reinterpret_cast<long long *>(sm)[at] = acc.hi[v];
                }
            } else if (!SPLIT && row < nb) {
                const int ex = sum_exponent<T>(ref, s_hdr.E);
                const bool plain = plain_sums<T>(ex);
                unsigned char *o = xp + row * kStageRow<T> + col * (int)sizeof(T);
                atomicMax(&s_bits[row], acc.bits());
#pragma unroll
                for (int v = 0; v < kTileCols; v += 16 / sizeof(T)) {
                    T y[16 / sizeof(T)];
#pragma unroll
                    for (int z = 0; z < (int)(16 / sizeof(T)); ++z)
                        y[z] = finish_point<T>(acc.hi[v + z], sizeof(T) == 8 ? acc.last(v + z) : 0, ex, plain);
                    *reinterpret_cast<uint4 *>(o + v * sizeof(T)) = *reinterpret_cast<const uint4 *>(y);
                }
            }
            if (!SPLIT) {
                // every row by one bulk copy (a row per thread storing 16-byte
                // pieces: 15000 cycles a tile)
                fence_async_smem();
                asm volatile("bar.sync 1, %0;" ::"n"(kTileConv) : "memory");
                if (t < nb && !s_abort) {
                    bulk_store(out + (b0 + t) * kPropBlk, xp + t * kStageRow<T>, kPropBlk * (uint32_t)sizeof(T));
                    bulk_commit();
                    if (!listed && results_too_small(P, s_bits, t, nb, s_hdr.keep))
                        P.list[atomicAdd(P.count, 1)] = (int)(b0 + t);
                }
            }
        } else if (cone == 0 && rank == 0) {
            const int row = (warp & 3) * 32 + lane, col = (warp >> 2) * kTileCols;
            if (row < nb) {
                T *o = out + (b0 + row) * kPropBlk + col;
                for (int v = 0; v < kTileCols; ++v)
                    o[v] = (T)0;
            }
        }
        if (SPLIT) {
            __syncwarp();
            cluster_sync();
            if (keep && warp < kTileWarps) {
                const int share = kPropBlk / ctas, ex = sum_exponent<T>(ref, s_hdr.E);
                const bool plain = plain_sums<T>(ex);
                // a warp reads 32 blocks' sums of one point (contiguous: reads
                // from another CTA's memory cost by the piece)
#pragma unroll 2
                for (int u = t; u < share * kPropTileBlks; u += kTileConv) {
                    const int row = u % kPropTileBlks, col = rank * share + u / kPropTileBlks;
                    if (row >= nb)
                        continue;
                    const uint32_t cell = (uint32_t)(col * kPropTileBlks + row), at = saddr(sm) + cell * 8,
                                   at_low = saddr(sm) + kPartHigh<T> + cell * 2;
                    long long z;
                    int low;
                    if (ctas == 2)
                        add_parts<T, 2>(at, at_low, z, low);
                    else if (ctas == 4)
                        add_parts<T, 4>(at, at_low, z, low);
                    else
                        add_parts<T, 8>(at, at_low, z, low);
                    z += low >> 16;
                    atomicMax(&s_bits[row], 64 - __clzll(z ^ (z >> 63)));
                    out[(b0 + row) * kPropBlk + col] = finish_point<T>(z, low & 0xffff, ex, plain);
                }
                // the blocks' largest sums, of every CTA's points, to the first
                asm volatile("bar.sync 1, %0;" ::"n"(kTileConv) : "memory");
                if (t < nb && rank != 0) {
                    uint32_t at;
                    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(saddr(&s_bits[t])), "r"(0));
                    asm volatile("red.relaxed.cluster.shared::cluster.max.s32 [%0], %1;" ::"r"(at), "r"(s_bits[t]) : "memory");
                }
            }
            __syncwarp();
            cluster_sync();
            if (keep && rank == 0 && t < nb && !listed && !s_abort && results_too_small(P, s_bits, t, nb, s_hdr.keep))
                P.list[atomicAdd(P.count, 1)] = (int)(b0 + t);
        }
        if (keep)
            phase ^= 1;
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (s_abort)
            break;
    }
    bulk_wait0();
    // the table's copy and MMAs in flight end before the CTA does
    if (t == 0 && has_tab)
        bar_drain(&tab_full, 0, kWaitLimitCycles);
    if (s_abort && t < kMmaWarps)
        bar_drain(&done[S::kGroups - 1 - t], phase ^ 1, kWaitLimitCycles);
    __syncthreads();
    if (warp == kTileWarps)
        tmem_dealloc(tbase, S::kCols);
}

// ---- two teams -------------------------------------------------------------

// Large FP32 grids whose taps reach a few blocks only: the table and the planes
// of two tiles fit shared memory, and two teams of eight warps and an issuing
// warp each take a tile of their own, so that one team's MMAs run under the
// other's loads, conversion and drain (in prop_tile_kernel, where a tile's
// planes fill shared memory, these take 18,000 cycles a tile during which the
// tensor cores idle).  The teams issue in turn.  A team has 256 of the 512
// columns: four accumulators, a ring that its sums go round.  Tiles of as many
// blocks as fit, up to 128 (of the MMA's 128 rows the others are not used).
// 2^24 points, 2000 steps: 387 -> 312 us a call.  (FP64: the eight planes of
// two tiles leave each 94 blocks where prop_tile_kernel's have 126: 2^22
// points, 24 steps, 138 us, 114 there.)
constexpr int kTeamWarps = 8, kTeam = 32 * kTeamWarps, kRing = 4;
constexpr int kDuoHb = 11;               // widest halo
constexpr int kDuoSmem = 232448 - 4096;  // static shared memory: below 4 KB
constexpr int kTeamCols = kPropBlk / (kTeamWarps / 4);
// Rows of a plane, and blocks of a tile, with `tab` bytes of tables: the MMA
// reads 128 rows whatever the tile, also past the last plane's end.
__host__ __device__ __forceinline__ int duo_rows(int tab, int hb)
{
    constexpr int NV = kPropNv32;
    const int need = 128 + 2 * hb, left = kDuoSmem - 1024 - ((tab + 1023) & ~1023);
    // (in eights, both the rows there are and the rows there could be use of:
    // a swizzled plane starts on 1024 bytes)
    const int rows = (left - (need + 7) * 128) / ((2 * NV - 1) * 128) & ~7,
              most = (need + 7) & ~7;
    return rows < most ? rows : most;
}

__global__ void __launch_bounds__(kTileThreads, 1) prop_duo_kernel(const __grid_constant__ PropRun P)
{
    using T = float;
    using S = TileShape<T>;
    using G = typename GroupsOf<T>::G;
    constexpr int ND = S::ND, NV = S::NV, NG = S::kGroups;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                          ~static_cast<uintptr_t>(1023));
    __shared__ __align__(8) uint64_t tab_full, full[2], done[2][NG], reuse[2][kRing];
    __shared__ uint32_t tmem_sh;
    __shared__ volatile int s_abort, s_stop[2];
    __shared__ int s_code[2][kPropTileBlks + 2 * S::kHb + 8];
    __shared__ int s_max[2][2], s_keep[2], s_left[2], s_turn;
    __shared__ int s_bits[2][kPropTileBlks];
    __shared__ PropHeader s_hdr;
    __shared__ DotShared<kEdgeRows> s_dot;
    __shared__ int4 s_prod[NG * ND];

    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t < (int)(sizeof(PropHeader) / 4))
        reinterpret_cast<int *>(&s_hdr)[t] = reinterpret_cast<const int *>(P.hdr)[t];
    if (t == 0) {
        bar_init(&tab_full, 1);
        for (int m = 0; m < 2; ++m) {
            bar_init(&full[m], kTeamWarps);
            for (int g = 0; g < NG; ++g)
                bar_init(&done[m][g], 1);
            for (int g = 0; g < kRing; ++g)
                bar_init(&reuse[m][g], kTeamWarps);
            s_stop[m] = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
        s_turn = 0;
    }
    if (warp == kTileWarps) {
        tmem_alloc(&tmem_sh, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = tmem_sh;
    if (blockIdx.x == 0 && t < 3 && P.zero[t])
        *P.zero[t] = 0;
    const int hb = P.hb, tab_bytes = s_hdr.rows * 16;
    // (a table the tiles cannot hold: by the plan's rule there is none, and
    // every block would take dot products)
    const bool ok_tab = s_hdr.ok && tab_bytes <= S::kTab && duo_rows(tab_bytes, hb) > 2 * hb;
    const int C = ok_tab ? duo_rows(tab_bytes, hb) : 64 + 2 * hb;
    const int per = C - 2 * hb < kPropTileBlks ? C - 2 * hb : kPropTileBlks;  // blocks of a tile
    const long long tiles = (P.blk1 - P.blk0 + per - 1) / per;
    if (t == 0 && ok_tab) {
        bar_expect_tx(&tab_full, (uint32_t)tab_bytes);
        bulk_load(sm, P.tab, (uint32_t)tab_bytes, &tab_full);
    }
    // the digit products' first descriptors and steps, in issue order
    for (int z = t; z < NG * ND; z += kTileThreads) {
        const int g = z / ND, i = z % ND;
        if (i < G::lo(g) || i > G::hi(g))
            continue;
        const int W = s_hdr.W[i];
        int4 p;
        p.x = (((G::weight(g) - i) * C + hb + (-W >> 6)) * 128) >> 4;
        p.y = s_hdr.row0[i] + 48 + 2 * W;
        p.z = (-W & 63) >> 3;
        p.w = (kPropBlk + 2 * W) / 16;
        s_prod[z] = p;
    }
    __syncthreads();
    unsigned char *planes = sm + ((tab_bytes + 1023) & ~1023);
    const T *in = static_cast<const T *>(P.in);
    T *out = static_cast<T *>(P.out);

    if (warp >= kTileWarps) {
        // ---- issuing warp of team m ------------------------------------------
        const int m = warp - kTileWarps;
        const bool leader = elect_one();
        bool ok = true, tab_waited = false;
        const uint64_t ad0 = swizzled_desc(saddr(planes + (size_t)m * NV * C * 128)), bd0 = plain_desc(saddr(sm), 128);
        int committed = -1;
        for (uint32_t n = 0; ok; ++n) {  // n: the team's tiles so far
            ok = __all_sync(0xffffffffu, bar_wait(&full[m], n & 1, kWaitLimitCycles, &s_abort));
            if (!ok || s_stop[m])
                break;
            // one team's MMAs at a time: side by side, both would take twice as
            // long, and then convert and drain side by side too
            if (lane == 0) {
                const long long t0 = clock64();
                while (atomicCAS(&s_turn, 0, 1) != 0 && !s_abort && clock64() - t0 < kWaitLimitCycles)
                    __nanosleep(40);
            }
            __syncwarp();
            tc_fence_after();
            if (!tab_waited) {
                ok = __all_sync(0xffffffffu, bar_wait(&tab_full, 0, kWaitLimitCycles, &s_abort));
                tab_waited = true;
            }
#pragma unroll 1
            for (int g = 0; ok && g < NG; ++g) {
                const int slot = g % kRing;
                // uses of the slot before this one: each must have been read
                const uint32_t uses = n * ((NG - slot + kRing - 1) / kRing) + g / kRing;
                if (uses > 0) {
                    ok = __all_sync(0xffffffffu, bar_wait(&reuse[m][slot], (uses - 1) & 1, kWaitLimitCycles, &s_abort));
                    tc_fence_after();
                    if (!ok)
                        break;
                }
                const int lo = G::lo(g), hi = G::hi(g);
                uint32_t acc = 0;
                const uint32_t dcol = tbase + (uint32_t)(m * 256 + slot * kPropBlk);
#pragma unroll 1
                for (int i = lo; i <= hi; ++i) {
                    const int4 p = s_prod[g * ND + i];
                    issue_product(leader, dcol, ad0 + (uint32_t)__shfl_sync(0xffffffffu, p.x, 0),
                                  bd0 + (uint32_t)__shfl_sync(0xffffffffu, p.y, 0), __shfl_sync(0xffffffffu, p.z, 0),
                                  __shfl_sync(0xffffffffu, p.w, 0), acc);
                }
                tc_commit_if(leader, &done[m][g]);
                __syncwarp();
                committed = (int)((n & 1) << 8) | g;
            }
            if (lane == 0)
                atomicExch(&s_turn, 0);
        }
        if (!ok && lane == 0) {
            atomicExch(P.err, kDevTimeout);
            s_abort = 1;
        }
        // MMAs in flight end before the CTA does
        if (s_abort && committed >= 0)
            bar_drain(&done[m][committed & 255], (uint32_t)(committed >> 8), kWaitLimitCycles);
        __syncwarp();
    } else {
        // ---- a team: load, convert, drain -------------------------------------
        const int m = warp / kTeamWarps, tw = warp % kTeamWarps, tt = t % kTeam;
        auto sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(2 + m), "n"(kTeam) : "memory"); };
        unsigned char *xp = planes + (size_t)m * NV * C * 128;
        uint32_t phase = 0;
        for (long long tile = (long long)blockIdx.x * 2 + m; tile < tiles; tile += 2LL * gridDim.x) {
            const long long b0 = P.blk0 + tile * per;
            const int nb = (int)(P.blk1 - b0 < per ? P.blk1 - b0 : per);
            const long long base = (b0 - hb) * kPropBlk;
            const int chunks = (per + 2 * hb) * 8;
            constexpr int kIter = ((kPropTileBlks + 2 * kDuoHb) * 8 + kTeam - 1) / kTeam;
            if (tt < 2)
                s_max[m][tt] = 0;
            if (tt == 2)
                s_keep[m] = 0;
            if (tt == 3)
                s_left[m] = *reinterpret_cast<const volatile int *>(P.count) > P.gate_min;
            sync();
            T x[kIter][8];
            int wmax = 0;
            constexpr int kV = 16 / sizeof(T);
#pragma unroll
            for (int c = 0; c < kIter; ++c) {
                const int u = c * kTeam + tt;
                const long long j = base + (long long)u * 8;
                const bool in_range = u < chunks && j + 8 <= P.n;
#pragma unroll
                for (int v = 0; v < 8 / kV; ++v) {
                    uint4 q = make_uint4(0, 0, 0, 0);
                    if (in_range)
                        q = *reinterpret_cast<const uint4 *>(in + j + v * kV);
                    *reinterpret_cast<uint4 *>(&x[c][v * kV]) = q;
                }
            }
            // the next tile's window on its way to L2
            if (tile + 2LL * gridDim.x < tiles) {
                const long long nx = base + 2LL * gridDim.x * per * kPropBlk;
                for (long long z = nx + (long long)tt * 128 / (long long)sizeof(T); z < nx + (long long)chunks * 8 && z < P.n;
                     z += (long long)kTeam * 128 / (long long)sizeof(T))
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(in + z));
            }
#pragma unroll
            for (int c = 0; c < kIter; ++c) {
                const int u = c * kTeam + tt;
                int q = 0;
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    const int y = code_of(x[c][v]);
                    q = y > q ? y : q;
                }
                wmax = q > wmax ? q : wmax;
                for (int z = 1; z < 8; z <<= 1) {
                    const int y = __shfl_xor_sync(0xffffffffu, q, z);
                    q = y > q ? y : q;
                }
                if ((tt & 7) == 0 && u < chunks)
                    s_code[m][u >> 3] = q;
            }
            // the rest of the cone, the walls included
            int cmax = wmax;
            const long long clo = b0 * kPropBlk - P.k - 2, chi = (b0 + nb) * kPropBlk + P.k + 2;
            cmax = max(cmax, max(clo <= 0 ? P.wall_l : 0, chi >= P.n ? P.wall_r : 0));
            auto scan = [&](long long a, long long b) {
                for (long long j = a + tt; j < b; j += 4 * kTeam)
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        cmax = max(cmax, code_of(j + u * kTeam < b ? in[j + u * kTeam] : (T)0));
            };
            scan(clo > 0 ? clo : 0, base);
            scan(base + (long long)chunks * 8, chi < P.n ? chi : P.n);
            for (long long j = (P.n & ~7LL) + tt; j < P.n && j < chi; j += kTeam)
                cmax = max(cmax, code_of(in[j]));
            bulk_wait_read0();  // the last tile's rows have left the planes
            wmax = __reduce_max_sync(0xffffffffu, wmax);
            cmax = __reduce_max_sync(0xffffffffu, cmax);
            if (lane == 0) {
                atomicMax(&s_max[m][0], wmax);
                atomicMax(&s_max[m][1], cmax);
            }
            sync();
            if (s_left[m])
                break;
            const int ref = s_max[m][0], cone = s_max[m][1];
            bool listed = false;  // block tt
            if (tt < nb) {
                s_bits[m][tt] = 0;
                listed = cone > 0 && (!ok_tab || values_too_small<T>(P, s_hdr.keep, s_code[m][hb + tt], ref, cone));
                if (listed)
                    P.list[atomicAdd(P.count, 1)] = (int)(b0 + tt);
                else if (cone > 0)
                    s_keep[m] = 1;
            }
            if (ok_tab && cone != kCodeInf<T>) {
#pragma unroll
                for (int c = 0; c < kIter; ++c) {
                    const int u = c * kTeam + tt;
                    if (u < chunks)
                        convert8(x[c], ref, xp + (u >> 3) * 128 + ((7 - (u & 7)) ^ ((u >> 3) & 7)) * 16, (size_t)C * 128);
                }
            }
            fence_async_smem();
            tc_fence_before();
            sync();
            if (!s_keep[m]) {
                if (cone == 0 && tt < nb * 2) {
                    T *o = out + b0 * kPropBlk + tt * 32;
                    for (int v = 0; v < 32; ++v)
                        o[v] = (T)0;
                }
                continue;
            }
            if (lane == 0)
                bar_arrive(&full[m]);
            // drain: kTeamCols points of the lane's block
            const int row = (warp & 3) * 32 + lane, col = (tw >> 2) * kTeamCols;
            Sums<T, kTeamCols> acc;
            bool ok = true;
#pragma unroll 1
            for (int g = 0; g < NG; ++g) {
                ok = ok && bar_wait(&done[m][g], phase, kWaitLimitCycles, &s_abort);
                if (!__any_sync(0xffffffffu, !ok)) {
                    tc_fence_after();
#pragma unroll
                    for (int h = 0; h < kTeamCols; h += 16) {
                        uint32_t v[16];
                        tmem_ld16(tbase + ((uint32_t)((warp & 3) * 32) << 16) +
                                      (uint32_t)(m * 256 + g % kRing * kPropBlk + col + h), v);
                        tmem_wait_ld();
                        if (h + 16 == kTeamCols) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0)
                                bar_arrive(&reuse[m][g % kRing]);
                        }
#pragma unroll
                        for (int q = 0; q < 16; ++q)
                            acc.fold(h + q, G::weight(g), __float2int_rn(__uint_as_float(v[q])));
                    }
                }
            }
            if (__any_sync(0xffffffffu, !ok)) {
                if (lane == 0) {
                    atomicExch(P.err, kDevTimeout);
                    s_abort = 1;
                }
            } else if (row < nb) {
                atomicMax(&s_bits[m][row], acc.bits());
                finish_row<T>(acc.hi, sum_exponent<T>(ref, s_hdr.E), xp + row * kStageRow<T> + col * (int)sizeof(T));
            }
            fence_async_smem();
            sync();
            if (tt < nb && !s_abort) {
                bulk_store(out + (b0 + tt) * kPropBlk, xp + tt * kStageRow<T>, kPropBlk * (uint32_t)sizeof(T));
                bulk_commit();
                if (!listed && results_too_small(P, s_bits[m], tt, nb, s_hdr.keep))
                    P.list[atomicAdd(P.count, 1)] = (int)(b0 + tt);
            }
            phase ^= 1;
            if (s_abort)
                break;
        }
        if (tt == 0)
            s_stop[m] = 1;
        sync();
        if (lane == 0)
            bar_arrive(&full[m]);
        bulk_wait0();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (t == 0 && ok_tab)
        bar_drain(&tab_full, 0, kWaitLimitCycles);
    __syncthreads();
    if (warp == kTileWarps)
        tmem_dealloc(tbase, 512);
    if (s_abort || warp >= kTileWarps)
        return;
    // rows near a wall: they fill the last wave, the CTAs with fewer tiles first
    const int shift = item_shift(P);
    const long long edge_l = item_count(P.rows_l, kEdgeRows, shift);
    const long long edges = edge_l + item_count(P.n - P.row_r, kEdgeRows, shift);
    // (a CTA's pair of tiles takes as long as about four items)
    const int busy = (int)((tiles + 1) / 2 % gridDim.x), spare = busy ? (int)gridDim.x - busy : 0;
    const bool few = spare > 0 && edges <= 4LL * spare;
    const int me = (int)blockIdx.x - busy;
    double *s_w = reinterpret_cast<double *>(sm), *taps = s_w + kDotWin + kEdgeScratch;
    bool staged = false;
    for (long long x = few && me < 0 ? edges : me < 0 ? me + (long long)gridDim.x : me; x < edges;
         x += few ? spare : (int)gridDim.x) {
        if (!staged)
            dot_stage<kTileConv>(P, reinterpret_cast<typename PairOf<T>::E *>(taps));
        staged = true;
        const long long a = x < edge_l ? 0 : P.row_r, b = x < edge_l ? P.rows_l : P.n;
        const long long r0 = a + (x < edge_l ? x : x - edge_l) * kEdgeRows - shift, r1 = r0 + kEdgeRows;
        dot_rows<T, kTileConv, kEdgeRows, kEdgeParts, true>(P, s_dot, s_w, taps, r0 > a ? r0 : a, r1 < b ? r1 : b);
    }
}

}  // namespace

cudaError_t prop_prepare()
{
    // once per device: the attributes, and every kernel loaded before a stream
    // capture may need it
    static std::mutex lock;
    static unsigned long long ready[4];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    std::lock_guard<std::mutex> hold(lock);
    if (dev < 256 && (ready[dev >> 6] >> (dev & 63)) & 1)
        return cudaSuccess;
    cudaFuncAttributes fa;
    auto smem = [&](auto *f, int bytes) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    smem(prop_tile_kernel<double, false>, kTileSmem<double>);
    smem(prop_tile_kernel<double, true>, kTileSmem<double>);
    smem(prop_tile_kernel<float, false>, kTileSmem<float>);
    smem(prop_tile_kernel<float, true>, kTileSmem<float>);
    smem(prop_duo_kernel, kDuoSmem);
    smem(prop_dot_kernel<double>, (kDotWin + dot_taps(kPropRMax)) * 8);
    smem(prop_dot_kernel<float>, (kDotWin + dot_taps(kPropRMax)) * 8);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(prop_digits_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 2 * kPropQ * 8);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(prop_level_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (7 * kPropRMax + 11 * kLevelPad + 8) * 8);
    const void *rest[] = {(const void *)prop_short_kernel, (const void *)prop_finish_kernel};
    for (const void *f : rest)
        if (e == cudaSuccess)
            e = cudaFuncGetAttributes(&fa, f);
    if (e == cudaSuccess && dev < 256)
        ready[dev >> 6] |= 1ull << (dev & 63);
    return e;
}

cudaError_t prop_launch_short(double *e, double *el, double *h, double *hl, int hs, int k, const PropCoef &c,
                              cudaStream_t s)
{
    prop_short_kernel<<<1, kShortThreads, 0, s>>>(e, el, h, hl, hs, k, c);
    return cudaGetLastError();
}

cudaError_t prop_launch_level(const PropLevel &a, cudaStream_t s)
{
    const int per = a.delta ? 30 : 32;
    const int grid = (2 * a.R2 + 1 + per - 1) / per + (a.par == 3 ? 4 : 2) * ((a.R2 + 1 + per - 1) / per);
    const size_t bytes = (size_t)(2 * a.R1 + 1 + 2 * kLevelPad + 4 * (a.R1 + 1 + 2 * kLevelPad) + a.R1 + kLevelPad) * 8;
    prop_level_kernel<<<grid, 128, bytes, s>>>(a);
    return cudaGetLastError();
}

cudaError_t prop_launch_finish(const PropLevel &a, const PropFinish &f, cudaStream_t s)
{
    const int R = a.R1, threads = 2 * R + 1 + 4 * (R + 1) + (f.x ? 2 * (2 * R + 9) : 0);
    const int warps = f.F ? 2 * (R + 2) : 0;
    const int bw = (warps * 32 + kFinishThreads - 1) / kFinishThreads, bt = (threads + kFinishThreads - 1) / kFinishThreads;
    prop_finish_kernel<<<bw > bt ? bw : bt, kFinishThreads, 0, s>>>(a, f);
    return cudaGetLastError();
}

cudaError_t prop_launch_digits(const PropSet &set, const PropFinish &f, int R, int prec, int hb_max, cudaStream_t s)
{
    prop_digits_kernel<<<1, 1024, 2 * kPropQ * 8, s>>>(f.x, f.x_max, R, prec == 0 ? kPropNd64 : kPropNd32,
                                                                    prec == 2, hb_max,
                                                                    prec == 0 ? kPropTab64 : kPropTab32, set.tab, set.hdr);
    return cudaGetLastError();
}

// Clusters of 2, 4 and 8 CTAs the device holds at once (a cluster lies within
// one group of SMs), asked once per device.
static cudaError_t split_clusters(int f64, int ctas, int *clusters)
{
    static std::mutex lock;
    static int known[64][2][9];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    std::lock_guard<std::mutex> hold(lock);
    int *k = dev < 64 ? &known[dev][f64 ? 1 : 0][ctas] : nullptr;
    if (k && *k) {
        *clusters = *k - 1;
        return cudaSuccess;
    }
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)ctas);
    c.blockDim = dim3(kTileThreads);
    c.dynamicSmemBytes = (size_t)(f64 ? kTileSmem<double> : kTileSmem<float>);
    c.attrs = &at;
    c.numAttrs = 1;
    e = f64 ? cudaOccupancyMaxActiveClusters(clusters, prop_tile_kernel<double, true>, &c)
            : cudaOccupancyMaxActiveClusters(clusters, prop_tile_kernel<float, true>, &c);
    if (e == cudaSuccess && k)
        *k = *clusters + 1;
    return e;
}

cudaError_t prop_launch_tiles(PropRun a, int f64, int num_sms, cudaStream_t s)
{
    const int shift = item_shift(a);
    const long long edges = item_count(a.rows_l, kEdgeRows, shift) + item_count(a.n - a.row_r, kEdgeRows, shift);
    // Fewer tiles than SMs: the cluster size, and the rounds of wall rows for
    // the CTAs without a tile, that should be done first, in cycles (measured
    // on this device: loading and converting a tile, an MMA, finishing it, an
    // item of wall rows; a digit's reach is on average 0.62 of the halo).
    int best = 1, split_grid = 0;
    const double mmas = (f64 ? 35.0 : 10.0) * (4 + 5 * a.hb), start = f64 ? 15500 : 11000;
    const double item = f64 ? 7000 + 16.0 * a.R : 6500 + 6.0 * a.R;
    if (a.tiles < num_sms) {
        const double rounds = std::ceil((double)edges / (double)(num_sms - a.tiles));
        double least = std::max(start + 50 * mmas + 6000, 4000 + rounds * item);
        for (int ctas = 2; ctas <= 8 && a.tiles * ctas <= num_sms; ctas *= 2) {
            int clusters = 0;
            cudaError_t e = split_clusters(f64, ctas, &clusters);
            if (e != cudaSuccess)
                return e;
            if (a.tiles > clusters)
                break;
            const int grid = (int)std::min<long long>(clusters, a.tiles + (edges + ctas - 1) / ctas) * ctas;
            const int spare = grid - (int)a.tiles * ctas;
            const double tile = start + 60 * mmas / ctas + 11000;
            const int all = spare > 0 ? (int)((edges + spare - 1) / spare) : 0;
            const int under = spare > 0 ? std::min(all, (int)((tile - 4000) / item)) : 0;
            for (int r : {under, all}) {
                const long long left = std::max(0LL, edges - (long long)r * spare);
                const double total = std::max(tile, 4000 + r * item) + (double)((left + grid - 1) / grid) * (item + 4000);
                if (total < least) {
                    least = total;
                    best = ctas;
                    a.edge_rounds = r;
                    a.split = ctas;
                    split_grid = grid;
                }
            }
        }
    }
    if (best > 1) {
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)best;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cudaLaunchConfig_t c{};
        c.gridDim = dim3((unsigned)split_grid);
        c.blockDim = dim3(kTileThreads);
        c.dynamicSmemBytes = (size_t)(f64 ? kTileSmem<double> : kTileSmem<float>);
        c.stream = s;
        c.attrs = &at;
        c.numAttrs = 1;
        return f64 ? cudaLaunchKernelEx(&c, prop_tile_kernel<double, true>, a)
                   : cudaLaunchKernelEx(&c, prop_tile_kernel<float, true>, a);
    }
    if (!f64 && a.tiles >= 2 * num_sms && a.hb <= kDuoHb) {
        prop_duo_kernel<<<num_sms, kTileThreads, kDuoSmem, s>>>(a);
        return cudaGetLastError();
    }
    const int grid = (int)(a.tiles + edges < num_sms ? a.tiles + edges : num_sms);
    a.edge_rounds = (int)std::min((double)edges, std::max(1.0, (start + 50 * mmas - 4000) / item));
    if (f64)
        prop_tile_kernel<double, false><<<grid, kTileThreads, kTileSmem<double>, s>>>(a);
    else
        prop_tile_kernel<float, false><<<grid, kTileThreads, kTileSmem<float>, s>>>(a);
    return cudaGetLastError();
}

cudaError_t prop_launch_dots(const PropRun &a, int f64, int grid, cudaStream_t s)
{
    const size_t bytes = (size_t)(kDotWin + dot_taps(a.R)) * 8;
    if (f64)
        prop_dot_kernel<double><<<grid, 256, bytes, s>>>(a);
    else
        prop_dot_kernel<float><<<grid, 256, bytes, s>>>(a);
    return cudaGetLastError();
}

}  // namespace ge

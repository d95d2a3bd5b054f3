// ge_prop.h -- composed steps: k block steps of the group explicit scheme as
// one banded operator, built once per (k, parity) and applied to the whole
// grid in one pass (ge_prop.cu, ge_prop_plan.cpp).
//
// With w = (I - r G_{1-p}) u + f the right-hand side of a step's group
// systems, one step is w <- C_p w + f, C_p = (I - r G_p)(I + r G_p)^{-1} =
// [[1, 2r], [2r, 1]] / (1 + 2r) on every group: a convex combination, the
// same at every group of the grid.  So k steps are w <- Q w + F with
//   Q(i, j) = A_{i&1}(j - i) + h_{i&1}(j + i - (i & 1)) (left wall)
//             + its mirror image (right wall),
// A the taps far from the walls (positive, sum 1; the odd rows' taps are the
// even rows' reversed, and starting at parity 1 swaps the two), h what a wall
// adds (a reflection depends on the distance travelled to the wall and back,
// j + i, only) and F the wall values' part.  For k <= n - 2 no point is
// reached by a reflection off both walls.
#pragma once

#include <atomic>
#include <cstdint>
#include <cuda_runtime_api.h>

#include "ge_internal.h"

namespace ge {

// Most taps kept per side (FP32; an FP64 context keeps up to kPropR64Max).
constexpr int kPropRMax = 1536, kPropR64Max = 704;
// Points of one block (columns of the accumulator) and blocks of a tile (its
// rows, the 128 lanes of tensor memory).  FP64: with its halo a tile has 128,
// the rows of a plane of digits that leave room for eight of them, and that
// 512 threads load in two turns.
constexpr int kPropBlk = 64;
constexpr int kPropTileBlks = 128, kPropRows64 = 128;
// Digits (base 256) of a tap and of a value: FP64 and FP32 storage.
constexpr int kPropNd64 = 7, kPropNd32 = 4;
constexpr int kPropNv64 = 8, kPropNv32 = 4;
// Bytes of the tap tables in shared memory (FP64: at most 93,824 by the plan's rule).
constexpr int kPropTab64 = 93 * 1024, kPropTab32 = 136 * 1024;
// Halo blocks a tile may have on each side.
constexpr int kPropHb64 = 8, kPropHb32 = 16;

// Device-written description of one operator's digit tables.
struct PropHeader {
    int E;         // a tap is its integer times 2^-E
    int ok;        // 0: the tables do not fit (never, by the plan's rule): every block takes the dot products
    int rows;      // 16-byte rows in all tables
    int keep;      // bits the largest sum of a block needs to be the tile's answer
    int W[8];      // reach of digit i's table: its taps beyond |d| = W are zero
    int row0[8];   // first row of digit i's table
};

// One operator's device arrays.
struct PropSet {
    double *e;          // taps of the even rows, chain starting at parity 0: e[-R..R] around the pointer
    double *h;          // wall arrays h[(parity * 2 + row) * hs + t]
    double *F;          // wall-value parts F[parity * hs + i]
    unsigned char *tab; // digit tables
    PropHeader *hdr;
    // host-side key and state
    int k, p0, entry, exit;
    int valid;          // arrays are written by work already on the stream
    long long used;
};

constexpr int kPropSets = 6;

// Which operators captured graphs read: a count each, held by the graphs (and
// whatever is instantiated from them) as user objects, which CUDA gives back
// when the last of them is gone.  That may be after the context is, so the
// counts have an owner count of their own.
struct PropPins {
    struct Slot {
        std::atomic<int> graphs{0};
        PropPins *owner = nullptr;
    } slot[kPropSets];
    std::atomic<int> owners{1};
    static PropPins *make();  // NULL: out of memory
    void drop();              // one owner less
    // The graph that `stream` is being captured into reads operator i.
    void pin(int i, cudaStream_t stream);
    bool pinned(int i) const { return slot[i].graphs.load(std::memory_order_acquire) > 0; }
};

// Per-context state.
struct PropState {
    void *mem = nullptr;          // one allocation for everything below
    PropSet set[kPropSets];
    PropPins *pins = nullptr;
    double *scratch[2];           // the chain's ping-pong arrays (e, h)
    double *x = nullptr;          // rows for the digits, and the word of their largest
    int *list = nullptr;          // blocks that need dot products
    int *count = nullptr;         // two words: the current launch's and the next one's
    long long clock = 0;
    TbRounds rounds;              // scratch of the launch being planned
    int rcap = 0, hs = 0;         // taps the arrays hold per side, stride of the wall arrays
};

struct PropTarget {
    void *buf[2];
    long long n;
    double r, beta_l, beta_r;
    int f64;             // element type of the state
    int num_sms;
    int *err;
    // the step-by-step form of an operator (tb_rounds_kernel), for data that
    // would need dot products nearly everywhere
    TbTarget tiled;
    const TbParams *base;
    double growth_lo;
    int prec, depth, rounds_grid;
};

// Arguments of the kernels that advance the state.
struct PropRun {
    const void *in;
    void *out;
    long long n;
    double r, x2, xs;           // entry and exit coefficients
    double fl, fr;              // r beta_l, r beta_r
    double bl, br;
    int wall_l, wall_r;         // exponent codes of what the walls add (tiles: see code_of)
    int k, p0, pr;              // block steps, start parity, start parity seen from the right wall
    int entry, exit;
    int R;                      // reach of the FP64 taps
    int hs;                     // stride of the wall arrays
    const double *e, *h, *F;
    const unsigned char *tab;
    const PropHeader *hdr;
    int *err;
    // tiles: blocks [blk0, blk1) in tiles of `per`, hb halo blocks per side
    long long blk0, blk1, tiles;
    int per, hb;
    // a block is left to dot products when its values lie below 2^-range
    // (2^-(range + 4) with a PropHeader::keep) of the largest of the tile's
    // window, or its results and those of `near` blocks a side have fewer bits
    // than PropHeader::keep
    int range, near;
    // dot products: rows [0, rows_l) and [row_r, n), and the listed blocks
    long long rows_l, row_r;
    int *list, *count, *count_next;
    int gate_min;      // more listed blocks than this: left to the step-by-step form
    int split;         // CTAs per tile, and items of wall rows for each CTA without one (set by the launcher)
    int edge_rounds;
    int *zero[3];      // words the tiles clear for it: barrier, two tile queues
};

// Pair and singleton coefficients of one step, (high, low) parts.
struct PropCoef {
    double al[2], be[2], ka[2];
    unsigned long long be_frac, ka_frac;  // be and |ka| times 2^64
};

// One doubling of the chain (k1 -> 2 k1 + delta), or its end.
struct PropLevel {
    const double *e0, *el0, *h0, *hl0;  // el0, hl0: the low parts, or NULL
    double *e1, *h1;
    int k1, R1, R2, delta, hs;
    int par;  // start parities whose wall arrays are needed (bit p)
    PropCoef c;
};
// What the finish makes of the last level's arrays (see prop_finish_kernel).
struct PropFinish {
    int k, p0, entry, exit;
    double r, x1, x2;
    double *F;                    // NULL: both walls 0
    double *x;                    // rows of the tensor cores' operator, or NULL
    unsigned long long *x_max;    // their largest magnitude's bits (zeroed)
};
// Longest chain built step by step.
constexpr int kPropShort = 31;

// Kernel launchers (ge_prop.cu).
cudaError_t prop_launch_short(double *e, double *el, double *h, double *hl, int hs, int k, const PropCoef &c,
                              cudaStream_t s);
cudaError_t prop_launch_level(const PropLevel &a, cudaStream_t s);
cudaError_t prop_launch_finish(const PropLevel &a, const PropFinish &f, cudaStream_t s);
cudaError_t prop_launch_digits(const PropSet &set, const PropFinish &f, int R, int prec, int hb_max, cudaStream_t s);
cudaError_t prop_launch_tiles(PropRun a, int f64, int num_sms, cudaStream_t s);
cudaError_t prop_launch_dots(const PropRun &a, int f64, int grid, cudaStream_t s);
cudaError_t prop_prepare();  // per-device kernel attributes

// Grids below this take dot products for every row.
constexpr long long kPropTileMin = 8192;

// Planning (ge_prop_plan.cpp).
size_t prop_bytes(long long n, int f64);
void prop_carve(PropState *st, void *mem, long long n, int f64);
// Whether a call of `steps` steps on n points takes this path.
// (prec as in tb_run).
bool prop_takes(long long n, double r, long long steps, int prec);
// Advance `steps` steps; *cur as in tb_run.  *taken = 0: nothing done (every
// operator slot belongs to a captured graph).  build_only: put the operators
// on the stream, and nothing else.
cudaError_t prop_run(PropState *st, const PropTarget &t, int *cur, long long step0, long long steps, int *taken,
                     cudaStream_t s, bool build_only = false);

}  // namespace ge

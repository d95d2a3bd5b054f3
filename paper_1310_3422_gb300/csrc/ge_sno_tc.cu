// ge_sno_tc.cu -- the surrogate's inference GEMMs, and the weight gradients of
// its training, on the fifth-generation
// tensor cores: tcgen05.mma with the accumulator in tensor memory (TMEM),
// operands staged in shared memory by 2D TMA copies, and the epilogue fused.
// The paper has no counterpart (the surrogate is a deployment variant of the
// GE solve; see ge_sno.h for the model).
//
// Three kernels: two of one template, each over 128-row tiles of the activation
// rows (all problems' grid points, [rows][64] BF16, channel last):
//   layer (MODE 0):  pre = G y + v W + b, then GELU (not after the last
//       layer), written as the next BF16 activation.  G [n][2M] is the
//       inverse truncated DFT, y [2M][C] the mode-mixed spectrum of the
//       tile's problem, v the tile's activations, W [C][C] the pointwise
//       weights.  Two products accumulate into one TMEM tile: K = 2M = 32
//       (G y) and K = C = 64 (v W).
//   projection (MODE 1): out = u0 + q2 + sum_h GELU(v Q1 + q1)_h Q2_h, one
//       FP32 value per row; the hidden layer (N = H = 128) lives in TMEM
//       only, and each thread sums its row in a fixed order;
// and the truncated DFT vh[b] = F v[b] of a layer's input (sno_tc_dft_kernel,
// described where it is defined).
//
// A operands are K-major with 128-byte (C = 64 BF16) or 64-byte (2M = 32
// BF16) rows, TMA-swizzled (SWIZZLE_128B / SWIZZLE_64B) as the tensor cores
// read them.  B operands: the spectrum y [2M][C] and the activations v (in
// the DFT) are read as stored, MN-major (N = 64 channels contiguous, one
// 128-byte swizzle atom wide); W and Q1 go through transposed copies W^T
// [C][C] and Q1^T [H][C] (K-major; sno_prepare writes them when the
// parameters change).  One MMA instruction covers 128 rows x N columns
// x 16 of K.
//
// Warp roles (160 threads): warp 4 lane 0 is the producer: it issues the TMA
// loads of a stage (two stages) and, once they land, the MMAs of the tile
// into a TMEM accumulator (two in the layer, one in the projection), then
// commits them to an mbarrier.
// Warps 0-3 drain the accumulator of a finished tile (warp w reads TMEM
// lanes 32w .. 32w + 31, i.e. tile rows) with tcgen05.ld, hand it back, and
// run the epilogue.  So the loads of tile i+1 (and, in the layer, its MMAs)
// run under the epilogue of tile i.  The layer's output leaves through a
// small per-warp staging buffer and TMA stores (whole 128-byte lines).
//
// Every wait is bounded: on expiry the kernel records GE_ETIMEOUT in the
// device error word, stops every role at its next wait, lets its own copies
// and MMAs in flight finish (each wait bounded again), frees its TMEM and
// returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "ge_f32x2.cuh"
#include "ge_internal.h"
#include "ge_sno_internal.h"
#include "ge_tc.cuh"

namespace ge {
namespace {

// Shared-memory matrix descriptor of a K-major operand tile whose rows of
// `row_bytes` (128 or 64) are TMA-swizzled with the same width: groups of 8
// rows lie 8 * row_bytes apart (stride byte offset), the leading byte offset
// is unused for a swizzled K-major tile, bits 46-47 hold the descriptor
// version (1), bits 61-63 the swizzle (2: 128-byte, 4: 64-byte).  The tile
// starts on a 1024-byte boundary; a K step of 16 BF16 (32 bytes) inside the
// swizzle row advances the start address.
__device__ __forceinline__ uint64_t smem_desc(const void *tile, uint32_t row_bytes)
{
    const uint64_t addr = saddr(tile);
    const uint64_t layout = row_bytes == 128 ? 2 : 4;
    return ((addr & 0x3FFFF) >> 4) | (1ull << 16) | ((uint64_t)((8 * row_bytes) >> 4) << 32) | (1ull << 46) |
           (layout << 61);
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
// (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits
// 17-22, M >> 4 at bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// B operand descriptor, MN-major with a 128-byte swizzle, for a tile of K
// rows of 64 BF16 N values (one swizzle atom wide, as TMA stores a box 128
// bytes wide): 8-row K groups 1024 bytes apart.  The instruction descriptor
// marks A MN-major with bit 15, B with bit 16.
constexpr uint32_t kIdescBMn = 1u << 16;
__device__ __forceinline__ uint64_t smem_desc_mn128(const void *tile, uint32_t atom_stride = 1024)
{
    // atom_stride: bytes from one 64-wide atom across M or N to the next
    // (the leading byte offset), for operands of two atoms
    const uint64_t addr = saddr(tile);
    return ((addr & 0x3FFFF) >> 4) | ((uint64_t)(atom_stride >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}
constexpr uint32_t kIdescAMn = 1u << 15;

// GELU, tanh form: GELU(x) = x (1 + tanh(k0 (x + k1 x^3))) / 2
constexpr float kGeluK0 = 0.7978845608028654f, kGeluK0K1 = 0.7978845608028654f * 0.044715f;

__device__ __forceinline__ float gelu_hw(float x)
{
    const float k0 = 0.7978845608028654f, k1 = 0.044715f;
    float t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(k0 * (x + k1 * x * x * x)));
    return 0.5f * x * (1.0f + t);
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);  // .x = a (low half), .y = b
    return *reinterpret_cast<const uint32_t *>(&h);
}

// A lane's row of 32 BF16 into a warp's staging buffer of 32 such rows: the
// 16-byte chunk q of row `lane` sits at chunk q ^ ((lane >> 1) & 3), the
// 64-byte swizzle the store's tensor map reads.
__device__ __forceinline__ void stage_rows(unsigned char *stg, int lane, const uint32_t (&w)[16])
{
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4 *>(stg + lane * 64 + ((q ^ ((lane >> 1) & 3)) << 4)) =
            make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
}

// The kernels of this file start before the one launched before them has
// finished, and set up (barriers, tensor memory) under its end: nothing
// before this call may read or write what that kernel does.  It comes after
// the CTA's tensor memory is allocated, so that the next kernel's CTAs, which
// it lets in, cannot take it first.
__device__ __forceinline__ void after_previous()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

constexpr int kTcThreads = 160;
constexpr int kTileM = 128;

template <int MODE>
struct TcShape {
    static constexpr int N = MODE == 0 ? 64 : 128;                  // output columns (TMEM columns per stage)
    static constexpr uint32_t kA2 = kTileM * 128;                    // v tile: 128 rows x 64 BF16
    static constexpr uint32_t kA1 = MODE == 0 ? kTileM * 64 : 0;     // G tile: 128 rows x 32 BF16
    static constexpr uint32_t kB1 = MODE == 0 ? 32 * 128 : 0;        // y: 32 rows x 64 BF16
    static constexpr uint32_t kStage = kA2 + kA1 + kB1;              // bytes of one stage (x1024)
    static constexpr uint32_t kB2 = N * 128;                         // W^T (64 rows) or Q1^T (128 rows)
    // TMEM accumulators: the layer keeps two (the next tile's MMAs run under
    // this tile's epilogue); the projection one, so that four CTAs fit an SM
    // (4 x 128 of the 512 columns) and their 16 epilogue warps hide the
    // latency of its GELU arithmetic
    static constexpr int kAccs = MODE == 0 ? 2 : 1;
    static constexpr uint32_t kTmemCols = kAccs * N;
    // layer: per epilogue warp a 2 KB staging buffer of its 32 output rows x
    // 32 columns (64-byte swizzle), written to global memory by a TMA store
    static constexpr uint32_t kOut = MODE == 0 ? 4 * 2048 : 0;
    static constexpr int kSmem = (int)(2 * kStage + kB2 + kOut + 1024);
};

template <int MODE>
__global__ void __launch_bounds__(kTcThreads) sno_tc_kernel(const __grid_constant__ CUtensorMap tmA1,
                                                            const __grid_constant__ CUtensorMap tmB1,
                                                            const __grid_constant__ CUtensorMap tmA2,
                                                            const __grid_constant__ CUtensorMap tmB2,
                                                            const __grid_constant__ CUtensorMap tmOut,
                                                            const __grid_constant__ SnoTcArgs P)
{
    using S = TcShape<MODE>;
    constexpr int N = S::N;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    unsigned char *b2 = sm + 2 * S::kStage;
    __shared__ __align__(8) uint64_t full[2], mma_done[2], acc_empty[2], b2_full;
    __shared__ uint32_t tmem_base_sh;
    __shared__ __align__(16) float s_bias[N];
    __shared__ __align__(16) float s_q2[N];
    __shared__ volatile int s_abort;

    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        for (int s = 0; s < 2; ++s) {
            bar_init(&full[s], 1);
            bar_init(&mma_done[s], 1);
            bar_init(&acc_empty[s], 4);
        }
        bar_init(&b2_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    if (warp == 0) {
        tmem_alloc(&tmem_base_sh, S::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    after_previous();
    for (int i = t; i < N; i += kTcThreads) {
        s_bias[i] = P.bias[i];
        // the projection keeps Q2 / 2 (exact): GELU's factor 1/2 moves onto it
        s_q2[i] = MODE == 1 ? 0.5f * P.q2w[i] : 0.0f;
    }
    __syncthreads();
    const uint32_t tbase = tmem_base_sh;
    const long long my_tiles =
        P.n_tiles > (long long)blockIdx.x ? (P.n_tiles - 1 - (long long)blockIdx.x) / gridDim.x + 1 : 0;

    if (warp == 4) {
        if (lane == 0 && my_tiles > 0) {
            // ---- producer: TMA loads and MMA issue ----------------------
            constexpr uint32_t idesc = idesc_bf16(kTileM, N);
            auto load_stage = [&](int s, long long i) {
                const long long g = (long long)blockIdx.x + i * gridDim.x;
                unsigned char *st = sm + s * S::kStage;
                bar_expect_tx(&full[s], S::kStage);
                tma_2d(st, &tmA2, 0, (int)(g * kTileM), &full[s]);
                if (MODE == 0) {
                    const long long b = g / P.tiles_per_problem, tt = g % P.tiles_per_problem;
                    tma_2d(st + S::kA2, &tmA1, 0, (int)(tt * kTileM), &full[s]);
                    tma_2d(st + S::kA2 + S::kA1, &tmB1, 0, (int)(b * 32), &full[s]);
                }
            };
            bar_expect_tx(&b2_full, S::kB2);
            tma_2d(b2, &tmB2, 0, P.b2_row, &b2_full);
            load_stage(0, 0);
            long long issued = 0, committed = 0;  // stages loaded, tiles committed
            bool ok = bar_wait(&b2_full, 0, P.limit, &s_abort);
            for (long long i = 0; ok && i < my_tiles; ++i) {
                const int s = (int)(i & 1);
                if (i + 1 < my_tiles) {
                    const int s1 = (int)((i + 1) & 1);
                    // stage s1 is free once the MMAs of tile i - 1 (which read it) are done
                    if (i >= 1 && !(ok = bar_wait(&mma_done[s1], (uint32_t)(((i - 1) >> 1) & 1), P.limit, &s_abort)))
                        break;
                    load_stage(s1, i + 1);
                    issued = i + 1;
                }
                if (!(ok = bar_wait(&full[s], (uint32_t)((i >> 1) & 1), P.limit, &s_abort)))
                    break;
                // accumulator i % kAccs is free once the epilogue of tile
                // i - kAccs has read it
                const int ac = (int)(i % S::kAccs);
                if (i >= S::kAccs && !(ok = bar_wait(&acc_empty[ac], (uint32_t)(((i - S::kAccs) / S::kAccs) & 1),
                                                      P.limit, &s_abort)))
                    break;
                tc_fence_after();
                const uint32_t acc = tbase + (uint32_t)(ac * N);
                unsigned char *st = sm + s * S::kStage;
                const uint64_t a2 = smem_desc(st, 128), bw = smem_desc(b2, 128);
                if (MODE == 0) {
                    // G y: the spectrum y[b] [2M][C] is read as stored (channels
                    // contiguous: an MN-major B operand, K steps of 16 rows =
                    // 2048 bytes); G's K step is 32 bytes inside its swizzle row
                    const uint64_t a1 = smem_desc(st + S::kA2, 64), b1 = smem_desc_mn128(st + S::kA2 + S::kA1);
                    tc_mma(acc, a1, b1, idesc | kIdescBMn, 0);
                    tc_mma(acc, a1 + 2, b1 + (2048 >> 4), idesc | kIdescBMn, 1);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    tc_mma(acc, a2 + 2 * k, bw + 2 * k, idesc, (MODE == 0 || k > 0) ? 1u : 0u);
                tc_commit(&mma_done[s]);
                committed = i + 1;
            }
            if (!ok) {
                atomicExch(P.err, kDevTimeout);
                s_abort = 1;
                // this CTA's own work in flight: the loads it issued and the
                // MMAs it committed
                bar_drain(&b2_full, 0, kWaitLimitCycles);
                for (long long j = committed; j <= issued; ++j)
                    bar_drain(&full[j & 1], (uint32_t)((j >> 1) & 1), kWaitLimitCycles);
                if (committed > 0)
                    bar_drain(&mma_done[(committed - 1) & 1], (uint32_t)(((committed - 1) >> 1) & 1),
                              kWaitLimitCycles);
            }
        }
        __syncwarp();
    } else {
        // ---- epilogue warps 0-3: TMEM lanes 32 warp .. 32 warp + 31 ------
        for (long long i = 0; i < my_tiles; ++i) {
            const int s = (int)(i & 1);
            const long long g = (long long)blockIdx.x + i * gridDim.x;
            const long long row = g * kTileM + warp * 32 + lane;
            const bool ok = bar_wait(&mma_done[s], (uint32_t)((i >> 1) & 1), P.limit, &s_abort);
            if (__any_sync(0xffffffffu, !ok)) {
                if (lane == 0 && !s_abort) {
                    atomicExch(P.err, kDevTimeout);
                    s_abort = 1;
                }
                break;
            }
            tc_fence_after();
            const int ac = (int)(i % S::kAccs);
            const uint32_t taddr = tbase + ((uint32_t)(warp * 32) << 16) + (uint32_t)(ac * N);
            if (MODE == 0) {
                uint32_t r0[32], r1[32];
                tmem_ld32(taddr, r0);
                tmem_ld32(taddr + 32, r1);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    bar_arrive(&acc_empty[ac]);
                // the warp's 32 rows leave through its staging buffer, 32
                // columns (64 bytes a row) at a time
                unsigned char *stg = sm + 2 * S::kStage + S::kB2 + warp * 2048;
                const long long row0 = g * kTileM + warp * 32;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t *r = h ? r1 : r0;
                    uint32_t w[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        float a = __uint_as_float(r[2 * c]) + s_bias[32 * h + 2 * c];
                        float b = __uint_as_float(r[2 * c + 1]) + s_bias[32 * h + 2 * c + 1];
                        if (P.gelu) {
                            a = gelu_hw(a);
                            b = gelu_hw(b);
                        }
                        w[c] = pack_bf16(a, b);
                    }
                    // the buffer is free once the previous store has read it
                    if (lane == 0)
                        bulk_wait_read0();
                    __syncwarp();
                    stage_rows(stg, lane, w);
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&tmOut, stg, 32 * h, (int)row0);
                        bulk_commit();
                    }
                }
            } else {
                // sum_h GELU(x_h) Q2_h with x_h = acc_h + q1_h, on column pairs
                // in packed FP32: GELU(x) Q2 = (x + x tanh(a)) (Q2 / 2) with
                // a = x (k0 + k0 k1 x^2).  Pair p of the row goes to partial
                // sum p % 4 (four short dependency chains); the partial sums
                // and their two lanes are added at the end in a fixed order.
                // TMEM is read 64 columns at a time (two loads, one wait).
                const uint64_t c_lo = f2(kGeluK0, kGeluK0), c_hi = f2(kGeluK0K1, kGeluK0K1);
                uint64_t part[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    part[k] = f2(0.0f, 0.0f);
#pragma unroll
                for (int h = 0; h < N / 64; ++h) {
                    uint32_t r[2][32];
                    tmem_ld32(taddr + 64 * h, r[0]);
                    tmem_ld32(taddr + 64 * h + 32, r[1]);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 64; c += 2) {
                        const int col = 64 * h + c;
                        const float2 bq = *reinterpret_cast<const float2 *>(&s_bias[col]);
                        const float2 wq = *reinterpret_cast<const float2 *>(&s_q2[col]);
                        const uint32_t *rr = r[c >> 5];
                        const uint64_t x =
                            f2_add(f2(__uint_as_float(rr[c & 31]), __uint_as_float(rr[(c & 31) + 1])), f2(bq.x, bq.y));
                        const uint64_t a = f2_mul(x, f2_fma(f2_mul(x, x), c_hi, c_lo));
                        const float2 af = f2_split(a);
                        float t0, t1;
                        asm("tanh.approx.f32 %0, %1;" : "=f"(t0) : "f"(af.x));
                        asm("tanh.approx.f32 %0, %1;" : "=f"(t1) : "f"(af.y));
                        part[(c >> 1) & 3] = f2_fma(f2_fma(x, f2(t0, t1), x), f2(wq.x, wq.y), part[(c >> 1) & 3]);
                    }
                }
                const float2 accf = f2_split(f2_add(f2_add(part[0], part[1]), f2_add(part[2], part[3])));
                const float sum = accf.x + accf.y;
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    bar_arrive(&acc_empty[ac]);
                float *out = static_cast<float *>(P.out);
                out[row] = P.u0[row] + P.q2b[0] + sum;
            }
        }
    }
    // the layer's output stores have landed before the CTA exits
    if (MODE == 0 && warp < 4 && lane == 0)
        bulk_wait0();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        tmem_dealloc(tbase, S::kTmemCols);
}

// ---- truncated DFT on the tensor cores ------------------------------------
//
// vh[b] = F v[b]: F [2M][n] (the truncated transform, 2M = 32 rows), v[b]
// [n][C] the problem's activations (C = 64).  One MMA takes M = 128 rows of
// A: A is F's 32 rows of a 128-point chunk of the grid (K-major, 128-byte
// swizzle); its rows 32 .. 127 are whatever shared memory of the same stage
// follows them, and the accumulator rows they produce are never read.  B is the activation
// tile exactly as the layer kernel loads it ([128 points][64 channels]): the
// channels (N) are contiguous, so B is MN-major, with 8-point groups 1024
// bytes apart and 16 points (one K step) 2048 bytes on.  A CTA takes whole
// problems: the n / 128 chunks (8 MMAs each) accumulate into one TMEM tile,
// then warp 0 (TMEM lanes 0 .. 31 = the 2M transform rows) writes vh[b] as
// BF16 [2M][C].  Warp 1's lane 0 is the producer (ST stages of TMA loads,
// the MMAs, commits); two accumulators, so the next problem's MMAs run
// under the previous one's write-out.  Bounded waits as in sno_tc_kernel.
// Two stages let four CTAs share an SM, the choice for many problems; with at
// most one problem per SM a CTA is alone and the latency
// of its loads counts, so all 8 chunks of 1024 points are in flight (64 problems: 10.9 -> 9.8 us).
constexpr int kDftThreads = 64;
constexpr uint32_t kDftAtom = 32 * 128;              // F rows of one 64-point half of a chunk
constexpr uint32_t kDftV = 128 * 128;                // the activation tile
constexpr uint32_t kDftStage = 2 * kDftAtom + kDftV;  // 24 KB: F halves first, so A's unused rows stay inside
constexpr int dft_smem(int stages) { return stages * (int)kDftStage + 1024; }

template <int ST>
__global__ void __launch_bounds__(kDftThreads) sno_tc_dft_kernel(const __grid_constant__ CUtensorMap tmF,
                                                                 const __grid_constant__ CUtensorMap tmV,
                                                                 const __grid_constant__ SnoTcArgs P)
{
    const int kChunks = P.tiles_per_problem;  // 128-point chunks of a problem
    constexpr uint32_t idesc = idesc_bf16(128, 64) | kIdescBMn;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    __shared__ __align__(8) uint64_t full[ST], freed[ST], done[2], acc_empty[2];
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int s_abort;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        for (int s = 0; s < ST; ++s) {
            bar_init(&full[s], 1);
            bar_init(&freed[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            bar_init(&done[s], 1);
            bar_init(&acc_empty[s], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    if (warp == 0) {
        tmem_alloc(&tmem_base_sh, 128);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    after_previous();
    const uint32_t tbase = tmem_base_sh;
    const long long problems = P.n_tiles / P.tiles_per_problem;
    const long long mine = problems > (long long)blockIdx.x ? (problems - 1 - (long long)blockIdx.x) / gridDim.x + 1 : 0;

    if (warp == 1) {
        if (lane == 0 && mine > 0) {
            // ---- producer: loads and MMAs, item = (problem, chunk) ----------
            const long long items = mine * kChunks;
            auto load = [&](long long it) {
                const int s = (int)(it % ST);
                const long long b = (long long)blockIdx.x + (it / kChunks) * gridDim.x;
                const int ch = (int)(it % kChunks);
                unsigned char *st = sm + s * kDftStage;
                bar_expect_tx(&full[s], 2 * kDftAtom + kDftV);
                tma_2d(st, &tmF, ch * 128, 0, &full[s]);
                tma_2d(st + kDftAtom, &tmF, ch * 128 + 64, 0, &full[s]);
                tma_2d(st + 2 * kDftAtom, &tmV, 0, (int)((b * kChunks + ch) * 128), &full[s]);
            };
            long long issued = 0, committed = 0;
            bool ok = true;
            for (; issued < ST - 1 && issued < items; ++issued)
                load(issued);
            for (long long it = 0; ok && it < items; ++it) {
                const int s = (int)(it % ST);
                const long long prob = it / kChunks;
                const int ch = (int)(it % kChunks);
                if (it + ST - 1 < items) {
                    // its stage is free once the MMAs of item it - 1 are done
                    if (it >= 1 && !(ok = bar_wait(&freed[(it - 1) % ST], (uint32_t)(((it - 1) / ST) & 1), P.limit,
                                                   &s_abort)))
                        break;
                    load(it + ST - 1);
                    issued = it + ST;
                }
                if (!(ok = bar_wait(&full[s], (uint32_t)((it / ST) & 1), P.limit, &s_abort)))
                    break;
                const int a = (int)(prob & 1);  // accumulator of this problem
                if (ch == 0 && prob >= 2 &&
                    !(ok = bar_wait(&acc_empty[a], (uint32_t)(((prob - 2) >> 1) & 1), P.limit, &s_abort)))
                    break;
                tc_fence_after();
                unsigned char *st = sm + s * kDftStage;
                const uint32_t acc = tbase + (uint32_t)(a * 64);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    // K step k: points 16k .. 16k + 15 of the chunk
                    const uint64_t ad = smem_desc(st + (k >> 2) * kDftAtom, 128) + (uint64_t)(2 * (k & 3));
                    const uint64_t bd = smem_desc_mn128(st + 2 * kDftAtom) + (uint64_t)(k * (2048 >> 4));
                    tc_mma(acc, ad, bd, idesc, (ch > 0 || k > 0) ? 1u : 0u);
                }
                tc_commit(&freed[s]);
                if (ch == kChunks - 1)
                    tc_commit(&done[a]);
                committed = it + 1;
            }
            if (!ok) {
                atomicExch(P.err, kDevTimeout);
                s_abort = 1;
                for (long long j = committed; j < issued; ++j)
                    bar_drain(&full[j % ST], (uint32_t)((j / ST) & 1), kWaitLimitCycles);
                if (committed > 0)
                    bar_drain(&freed[(committed - 1) % ST], (uint32_t)(((committed - 1) / ST) & 1), kWaitLimitCycles);
            }
        }
        __syncwarp();
    } else {
        // ---- warp 0: TMEM lanes 0 .. 31 (transform rows) -> vh[b] ----------
        for (long long prob = 0; prob < mine; ++prob) {
            const int a = (int)(prob & 1);
            const bool ok = bar_wait(&done[a], (uint32_t)((prob >> 1) & 1), P.limit, &s_abort);
            if (__any_sync(0xffffffffu, !ok)) {
                if (lane == 0 && !s_abort) {
                    atomicExch(P.err, kDevTimeout);
                    s_abort = 1;
                }
                break;
            }
            tc_fence_after();
            uint32_t r0[32], r1[32];
            const uint32_t taddr = tbase + (uint32_t)(a * 64);
            tmem_ld32(taddr, r0);
            tmem_ld32(taddr + 32, r1);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                bar_arrive(&acc_empty[a]);
            const long long b = (long long)blockIdx.x + prob * gridDim.x;
            uint4 *dst = reinterpret_cast<uint4 *>(static_cast<unsigned char *>(P.out) + (b * 32 + lane) * 128);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t *r = h ? r1 : r0;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    dst[4 * h + q] = make_uint4(pack_bf16(__uint_as_float(r[8 * q]), __uint_as_float(r[8 * q + 1])),
                                                pack_bf16(__uint_as_float(r[8 * q + 2]), __uint_as_float(r[8 * q + 3])),
                                                pack_bf16(__uint_as_float(r[8 * q + 4]), __uint_as_float(r[8 * q + 5])),
                                                pack_bf16(__uint_as_float(r[8 * q + 6]), __uint_as_float(r[8 * q + 7])));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        tmem_dealloc(tbase, 128);
}

// ---- per-mode complex mixing on the tensor cores ---------------------------
//
// y[b, m] = vh[b, m] Wspec_m for every mode m: vh[b, m] is the 2C = 128 values
// (real and imaginary parts of the C channels) of mode m of problem b, Wspec_m
// the [2C][2C] real form of the complex mode weights.  A CTA takes 128
// problems of one mode: A = those problems' vh[., m] rows (K-major, two
// 64-wide 128-byte-swizzled boxes), B = Wspec_m^T [N][K] (K-major, written so
// by sno_prepare), one 128 x 128 FP32
// accumulator in TMEM after 8 MMAs of K = 16.  Thread 0 issues the four loads
// and the MMAs; the four warps then read back their 32 rows each and write
// y[b, m] as BF16 (rows past the batch are not written).
constexpr int kMixThreads = 128;
constexpr uint32_t kMixHalf = 128 * 128;  // one 64-wide box of 128 rows
constexpr int kMixSmem = (int)(4 * kMixHalf) + 1024;

__global__ void __launch_bounds__(kMixThreads) sno_tc_mix_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                 const __grid_constant__ CUtensorMap tmB,
                                                                 const __grid_constant__ SnoTcMixArgs P)
{
    constexpr uint32_t idesc = idesc_bf16(128, 128);
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    unsigned char *sa = sm, *sb = sm + 2 * kMixHalf;
    __shared__ __align__(8) uint64_t full, done;
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int s_abort;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int m = blockIdx.y;
    const int row0 = blockIdx.x * 128;
    if (t == 0) {
        bar_init(&full, 1);
        bar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    if (warp == 0) {
        tmem_alloc(&tmem_base_sh, 128);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    after_previous();
    const uint32_t tbase = tmem_base_sh;
    if (t == 0) {
        bar_expect_tx(&full, 4 * kMixHalf);
        tma_2d(sa, &tmA, m * 128, row0, &full);
        tma_2d(sa + kMixHalf, &tmA, m * 128 + 64, row0, &full);
        tma_2d(sb, &tmB, 0, P.b_row0 + m * 128, &full);
        tma_2d(sb + kMixHalf, &tmB, 64, P.b_row0 + m * 128, &full);
        if (bar_wait(&full, 0, P.limit, &s_abort)) {
            tc_fence_after();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint64_t ad = smem_desc(sa + h * kMixHalf, 128), bd = smem_desc(sb + h * kMixHalf, 128);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    tc_mma(tbase, ad + 2 * k, bd + 2 * k, idesc, (h > 0 || k > 0) ? 1u : 0u);
            }
            tc_commit(&done);
        } else {
            atomicExch(P.err, kDevTimeout);
            s_abort = 1;
            bar_drain(&full, 0, kWaitLimitCycles);  // the loads in flight land before the CTA exits
        }
    }
    const bool ok = bar_wait(&done, 0, P.limit, &s_abort);
    if (__any_sync(0xffffffffu, !ok)) {
        if (lane == 0 && !s_abort) {
            atomicExch(P.err, kDevTimeout);
            s_abort = 1;
        }
        if (t == 0)
            bar_drain(&done, 0, kWaitLimitCycles);  // MMAs it issued finish before TMEM is freed
    } else {
        tc_fence_after();
        const int b = row0 + warp * 32 + lane;
        uint4 *dst = reinterpret_cast<uint4 *>(static_cast<unsigned char *>(P.y) +
                                               ((long long)b * P.row_elems + (long long)m * 128) * 2);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            uint32_t r[32];
            tmem_ld32(tbase + ((uint32_t)(warp * 32) << 16) + (uint32_t)(32 * h), r);
            tmem_wait_ld();
            if (b < P.batch) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    dst[4 * h + q] = make_uint4(pack_bf16(__uint_as_float(r[8 * q]), __uint_as_float(r[8 * q + 1])),
                                                pack_bf16(__uint_as_float(r[8 * q + 2]), __uint_as_float(r[8 * q + 3])),
                                                pack_bf16(__uint_as_float(r[8 * q + 4]), __uint_as_float(r[8 * q + 5])),
                                                pack_bf16(__uint_as_float(r[8 * q + 6]), __uint_as_float(r[8 * q + 7])));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        tmem_dealloc(tbase, 128);
}

// ---- weight gradients on the tensor cores -----------------------------------
//
// dW = X^T dY, the sum over all grid points (rows) of products of two
// activations [rows][64 or 128] as they lie in memory: the rows are the K
// dimension, both operands are MN-major.  A CTA takes every gridDim.x-th
// chunk of 128 rows: up to four stages of TMA loads in flight, 8 MMAs of K =
// 16 a chunk into one FP32 accumulator in TMEM, then the result is added to
// global memory.
//   KIND 0 / 1: X [rows][64], dY [rows][64 / 128].  The instruction has 128
//       rows of A and X gives 64: the others come from a constant tile whose
//       first column is 1 (the second atom of A, at its own stride), so that
//       accumulator row 64 is the column sum of dY, the bias gradient.  Each
//       CTA stores its own; they are added in a fixed order, so that it is the
//       same from run to run, by the next KIND 2 launch.  (By the last CTA to
//       finish: 3 to 6 us a launch.)
//   KIND 2: one CTA per mode, X and dY [rows = problems][128]; D = X^T dY is
//       folded to the complex weights' gradients before it is stored.  A
//       few more CTAs add the bias parts meanwhile.
// Bound by the latency of the loads and of the adds (16 MB in KIND 0: 2.4 us
// at the copy rate).  65,536 rows, cold caches: KIND 0 takes 11.1 us, KIND 1
// 12.5 us; as mma.sync tiles with split K, a column-sum pass and a memset
// they took 38 and 40 us.  KIND 2, 64 problems: 7.5 us, before 19.4 us with
// the folding as a pass of its own.
template <int KIND>
struct GradShape {
    static constexpr int AT = KIND == 2 ? 2 : 1, NB = KIND == 0 ? 1 : 2;  // 64-wide atoms of X and dY
    static constexpr uint32_t kAtom = 128 * 128;
    static constexpr uint32_t kStage = (AT + NB) * kAtom;
    static constexpr int ST = KIND == 2 ? 2 : 4;
    static constexpr uint32_t kOnes = KIND == 2 ? 0 : 16 * 128;
    static constexpr int kSmem = (int)(ST * kStage + kOnes) + 1024;
};
constexpr int kGradThreads = 160;

__device__ __forceinline__ void red_add4(float *p, float a, float b, float c, float d)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// Columns 16 c .. 16 c + 15 of the parts [ctas][cols] of a bias gradient, added
// in a fixed order by 128 threads: thread (k, j) takes CTAs k, k + 32, ..., so
// that all loads are in flight at once.
__device__ __forceinline__ void add_bias_parts(const SnoBiasParts &b, int c, float4 (&sh)[128])
{
    const int t = threadIdx.x, at = 4 * c + t % 4;
    const float4 *part = reinterpret_cast<const float4 *>(b.part);
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 5
    for (int i = t / 4; i < b.ctas; i += 32) {
        const float4 x = __ldcg(part + i * (b.cols / 4) + at);
        v.x += x.x, v.y += x.y, v.z += x.z, v.w += x.w;
    }
    sh[t] = v;
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (t < 4) {
#pragma unroll 8
        for (int k = 1; k < 32; ++k) {
            const float4 x = sh[4 * k + t];
            v.x += x.x, v.y += x.y, v.z += x.z, v.w += x.w;
        }
        reinterpret_cast<float4 *>(b.out)[at] = v;
    }
}

template <int KIND>
__global__ void __launch_bounds__(kGradThreads) sno_tc_grad_kernel(const __grid_constant__ CUtensorMap tmX,
                                                                   const __grid_constant__ CUtensorMap tmY,
                                                                   const __grid_constant__ SnoTcGradArgs P)
{
    using S = GradShape<KIND>;
    constexpr int N = 64 * S::NB, ST = S::ST;
    constexpr uint32_t idesc = idesc_bf16(128, N) | kIdescAMn | kIdescBMn;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    unsigned char *ones = sm + ST * S::kStage;
    __shared__ __align__(8) uint64_t full[ST], freed[ST], done;
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int s_abort;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if constexpr (KIND == 2) {
        if ((int)blockIdx.y >= P.modes) {
            __shared__ float4 sh[128];
            const int c = (int)blockIdx.y - P.modes, first = P.bias[0].cols / 16;
            after_previous();
            if (t < 128)
                add_bias_parts(P.bias[c < first ? 0 : 1], c < first ? c : c - first, sh);
            return;
        }
    }
    if (t == 0) {
        for (int s = 0; s < ST; ++s) {
            bar_init(&full[s], 1);
            bar_init(&freed[s], 1);
        }
        bar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    if (warp == 0) {
        tmem_alloc(&tmem_base_sh, N);
        tmem_relinquish();
    }
    // 16 K rows of 64 values, value 0 = 1: in row k the 16-byte chunk 0 lies
    // at chunk k & 7 (128-byte swizzle)
    for (int i = t; i < (int)S::kOnes / 16; i += kGradThreads)
        reinterpret_cast<uint4 *>(ones)[i] = make_uint4((i & 7) == ((i >> 3) & 7) ? 0x3F80u : 0u, 0u, 0u, 0u);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    after_previous();
    const uint32_t tbase = tmem_base_sh;
    const long long chunks = (P.rows + 127) / 128;
    const long long mine = chunks > (long long)blockIdx.x ? (chunks - 1 - (long long)blockIdx.x) / gridDim.x + 1 : 0;
    const int x0 = KIND == 2 ? (int)blockIdx.y * 128 : 0;

    if (warp == 4) {
        auto load = [&](long long it) {
            if (lane == 0) {
                const int s = (int)(it % ST);
                const int row = (int)(((long long)blockIdx.x + it * gridDim.x) * 128);
                unsigned char *st = sm + s * S::kStage;
                bar_expect_tx(&full[s], S::kStage);
                for (int q = 0; q < S::AT; ++q)
                    tma_2d(st + q * S::kAtom, &tmX, x0 + 64 * q, row, &full[s]);
                for (int q = 0; q < S::NB; ++q)
                    tma_2d(st + (S::AT + q) * S::kAtom, &tmY, x0 + 64 * q, row, &full[s]);
            }
        };
        long long issued = 0, committed = 0;
        bool ok = true;
        for (; issued < ST && issued < mine; ++issued)
            load(issued);
        for (long long it = 0; it < mine; ++it) {
            const int s = (int)(it % ST);
            if (!(ok = __all_sync(0xffffffffu, bar_wait(&full[s], (uint32_t)((it / ST) & 1), P.limit, &s_abort))))
                break;
            unsigned char *st = sm + s * S::kStage;
            const long long left = P.rows - ((long long)blockIdx.x + it * gridDim.x) * 128;
            const int valid = left < 128 ? (int)left : 128, steps = (valid + 15) / 16;
            if (valid < 16 * steps) {
                // rows past the end (another batch's): zero in both operands
                for (int i = lane; i < (16 * steps - valid) * 8; i += 32)
                    for (int q = 0; q < S::AT + S::NB; ++q)
                        *reinterpret_cast<uint4 *>(st + q * S::kAtom + valid * 128 + i * 16) = make_uint4(0, 0, 0, 0);
                fence_async_smem();
            }
            __syncwarp();
            if (lane == 0) {
                tc_fence_after();
                unsigned char *b = st + S::AT * S::kAtom;
                for (int k = 0; k < steps; ++k) {
                    unsigned char *a = st + k * 2048;
                    const uint32_t second = KIND == 2 ? S::kAtom : (uint32_t)(ones - a);
                    tc_mma(tbase, smem_desc_mn128(a, second), smem_desc_mn128(b + k * 2048, S::kAtom), idesc,
                           (it > 0 || k > 0) ? 1u : 0u);
                }
                tc_commit(&freed[s]);
                if (it == mine - 1)
                    tc_commit(&done);
            }
            committed = it + 1;
            // refill the stage of the item before
            if (it >= 1 && it - 1 + ST < mine) {
                const long long q = it - 1;
                if (!(ok = __all_sync(0xffffffffu, bar_wait(&freed[q % ST], (uint32_t)((q / ST) & 1), P.limit,
                                                            &s_abort))))
                    break;
                load(q + ST);
                issued = q + ST + 1;
            }
        }
        if (!ok && lane == 0) {
            atomicExch(P.err, kDevTimeout);
            s_abort = 1;
            for (long long j = committed; j < issued; ++j)
                bar_drain(&full[j % ST], (uint32_t)((j / ST) & 1), kWaitLimitCycles);
            if (committed > 0)
                bar_drain(&freed[(committed - 1) % ST], (uint32_t)(((committed - 1) / ST) & 1), kWaitLimitCycles);
        }
        __syncwarp();
    } else if (mine > 0) {
        const bool ok = __all_sync(0xffffffffu, bar_wait(&done, 0, P.limit, &s_abort));
        if (!ok && lane == 0 && !s_abort) {
            atomicExch(P.err, kDevTimeout);
            s_abort = 1;
        }
        tc_fence_after();
        const uint32_t taddr = tbase + ((uint32_t)(warp * 32) << 16);
        const int row = warp * 32 + lane;
        if (KIND == 2) {
            // thread i holds row i of D; with R_im the rows 64 .. 127,
            //   dRr[o][i] = D[i][o] + D[64 + i][64 + o]
            //   dRi[o][i] = D[i][64 + o] - D[64 + i][o]
            float *other = reinterpret_cast<float *>(sm);  // the stages are read: [128 columns][64 rows]
            if (ok && warp >= 2)
                for (int h = 0; h < 4; ++h) {
                    uint32_t r[32];
                    tmem_ld32(taddr + 32 * h, r);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 32; ++c)
                        other[(32 * h + c) * 64 + row - 64] = __uint_as_float(r[c]);
                }
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (ok && warp < 2)
                for (int h = 0; h < 4; ++h) {
                    uint32_t r[32];
                    tmem_ld32(taddr + 32 * h, r);
                    tmem_wait_ld();
                    float *dst = (h < 2 ? P.drr : P.dri) + (long long)blockIdx.y * 64 * 64;
#pragma unroll
                    for (int c = 0; c < 32; ++c) {
                        const int o = 32 * (h & 1) + c;
                        const float v = __uint_as_float(r[c]), w = other[(h < 2 ? 64 + o : o) * 64 + row];
                        dst[o * 64 + row] = h < 2 ? v + w : v - w;
                    }
                }
        } else {
            if (ok && warp < 3)
                for (int h = 0; h < N / 32; ++h) {
                    uint32_t r[32];
                    tmem_ld32(taddr + 32 * h, r);
                    tmem_wait_ld();
                    float *dst = (row < 64 ? P.dw + row * N : P.part + (long long)blockIdx.x * N) + 32 * h;
#pragma unroll
                    for (int c = 0; c < 32; c += 4) {
                        const float4 v = make_float4(__uint_as_float(r[c]), __uint_as_float(r[c + 1]),
                                                     __uint_as_float(r[c + 2]), __uint_as_float(r[c + 3]));
                        if (row < 64)
                            red_add4(dst + c, v.x, v.y, v.z, v.w);
                        else if (row == 64)
                            *reinterpret_cast<float4 *>(dst + c) = v;
                    }
                }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        tmem_dealloc(tbase, N);
}

template <typename... Params, typename... Args>
cudaError_t launch_early(void (*kernel)(Params...), dim3 grid, int threads, int smem, cudaStream_t s, int early,
                         const Args &...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = (size_t)smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, args...);
}

// Dynamic shared memory a kernel may take, on the current device, and (where
// per_sm is given) its co-resident CTAs per SM: what shared memory holds at
// the largest carve-out (the kernel's static and dynamic bytes plus the
// driver's reserve per CTA), what the registers hold, and at most `most`, so
// that their TMEM columns (512 per SM) all fit.
template <typename... Params>
cudaError_t prepare_kernel(void (*kernel)(Params...), int threads, int smem, int most, int *per_sm)
{
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess || !per_sm)
        return e;
    cudaFuncAttributes fa{};
    int dev = 0, sm_bytes = 0, reserve = 0;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
        e = cudaFuncGetAttributes(&fa, kernel);
    if (e == cudaSuccess)
        e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&reserve, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e != cudaSuccess)
        return e;
    const int fit = sm_bytes / (smem + (int)fa.sharedSizeBytes + reserve),
              regs = 65536 / ((fa.numRegs + 7) / 8 * 8 * threads);
    *per_sm = fit < regs ? fit : regs;
    *per_sm = *per_sm < most ? *per_sm : most;
    return *per_sm < 1 ? cudaErrorInvalidConfiguration : cudaSuccess;
}

template <int MODE>
cudaError_t launch_tc(const SnoTcMaps &m, const SnoTcArgs &a, int ctas, cudaStream_t s)
{
    using S = TcShape<MODE>;
    long long grid = ctas;
    if (grid > a.n_tiles)
        grid = a.n_tiles;
    if (grid < 1)
        return cudaSuccess;
    if (!m.a2 || !m.b2 || (MODE == 0 && (!m.a1 || !m.b1 || !m.out)))
        return cudaErrorInvalidValue;
    // the projection has no first product and no output map: those
    // parameters repeat a2
    const CUtensorMap *a1 = static_cast<const CUtensorMap *>(MODE == 0 ? m.a1 : m.a2);
    const CUtensorMap *b1 = static_cast<const CUtensorMap *>(MODE == 0 ? m.b1 : m.a2);
    const CUtensorMap *o = static_cast<const CUtensorMap *>(MODE == 0 ? m.out : m.a2);
    return launch_early(sno_tc_kernel<MODE>, dim3((unsigned)grid), kTcThreads, S::kSmem, s, a.early, *a1, *b1,
                        *static_cast<const CUtensorMap *>(m.a2), *static_cast<const CUtensorMap *>(m.b2), *o, a);
}

template <int ST>
cudaError_t launch_dft(const CUtensorMap &f, const CUtensorMap &v, const SnoTcArgs &a, int ctas, cudaStream_t s)
{
    const long long problems = a.n_tiles / a.tiles_per_problem;
    long long grid = ctas;
    if (grid > problems)
        grid = problems;
    if (grid < 1)
        return cudaSuccess;
    return launch_early(sno_tc_dft_kernel<ST>, dim3((unsigned)grid), kDftThreads, dft_smem(ST), s, a.early, f, v, a);
}

template <int KIND>
cudaError_t launch_grad(const void *map_x, const void *map_y, const SnoTcGradArgs &a, dim3 grid, cudaStream_t s)
{
    using S = GradShape<KIND>;
    if (!map_x || !map_y || a.rows < 0 || a.rows > 0x7FFFFF00LL)
        return cudaErrorInvalidValue;
    if (a.rows == 0 || grid.x == 0 || grid.y == 0)
        return cudaSuccess;
    return launch_early(sno_tc_grad_kernel<KIND>, grid, kGradThreads, S::kSmem, s, a.early, *static_cast<const CUtensorMap *>(map_x),
                        *static_cast<const CUtensorMap *>(map_y), a);
}

}  // namespace

cudaError_t sno_tc_prepare(SnoTcGrid *g, int sms)
{
    int layer = 0, projection = 0, dft2 = 0, dft8 = 0;
    auto tmem = [](uint32_t cols) { return 512 / (int)cols; };
    cudaError_t e = prepare_kernel(sno_tc_kernel<0>, kTcThreads, TcShape<0>::kSmem, tmem(TcShape<0>::kTmemCols), &layer);
    if (e == cudaSuccess)
        e = prepare_kernel(sno_tc_kernel<1>, kTcThreads, TcShape<1>::kSmem, tmem(TcShape<1>::kTmemCols), &projection);
    if (e == cudaSuccess)
        e = prepare_kernel(sno_tc_dft_kernel<2>, kDftThreads, dft_smem(2), tmem(128), &dft2);
    if (e == cudaSuccess)
        e = prepare_kernel(sno_tc_dft_kernel<8>, kDftThreads, dft_smem(8), tmem(128), &dft8);
    if (e == cudaSuccess)
        e = prepare_kernel(sno_tc_mix_kernel, kMixThreads, kMixSmem, 0, nullptr);
    if (e == cudaSuccess)
        e = prepare_kernel(sno_tc_grad_kernel<0>, kGradThreads, GradShape<0>::kSmem, 0, nullptr);
    if (e == cudaSuccess)
        e = prepare_kernel(sno_tc_grad_kernel<1>, kGradThreads, GradShape<1>::kSmem, 0, nullptr);
    if (e == cudaSuccess)
        e = prepare_kernel(sno_tc_grad_kernel<2>, kGradThreads, GradShape<2>::kSmem, 0, nullptr);
    *g = {sms, sms * layer, sms * projection, sms * dft2, sms * dft8};
    return e;
}

cudaError_t sno_tc_layer(const SnoTcMaps &m, const SnoTcArgs &a, const SnoTcGrid &g, cudaStream_t s)
{
    return launch_tc<0>(m, a, g.layer, s);
}

cudaError_t sno_tc_projection(const SnoTcMaps &m, const SnoTcArgs &a, const SnoTcGrid &g, cudaStream_t s)
{
    return launch_tc<1>(m, a, g.projection, s);
}

cudaError_t sno_tc_dft(const void *map_f, const void *map_v, const SnoTcArgs &a, const SnoTcGrid &g, cudaStream_t s)
{
    if (!map_f || !map_v || a.tiles_per_problem < 1)
        return cudaErrorInvalidValue;
    const CUtensorMap &f = *static_cast<const CUtensorMap *>(map_f), &v = *static_cast<const CUtensorMap *>(map_v);
    return a.n_tiles / a.tiles_per_problem <= g.sms ? launch_dft<8>(f, v, a, g.dft8, s) : launch_dft<2>(f, v, a, g.dft2, s);
}

cudaError_t sno_tc_mix(const void *map_vh, const void *map_wst, const SnoTcMixArgs &a, int modes, cudaStream_t s)
{
    if (!map_vh || !map_wst || modes < 1 || a.batch < 0)
        return cudaErrorInvalidValue;
    if (a.batch == 0)
        return cudaSuccess;
    const dim3 grid((unsigned)((a.batch + 127) / 128), (unsigned)modes);
    return launch_early(sno_tc_mix_kernel, grid, kMixThreads, kMixSmem, s, a.early, *static_cast<const CUtensorMap *>(map_vh),
                        *static_cast<const CUtensorMap *>(map_wst), a);
}

int sno_tc_grad_ctas(long long rows, int sms)
{
    const long long chunks = (rows + 127) / 128, per = (chunks + sms - 1) / sms;
    return (int)(per > 0 ? (chunks + per - 1) / per : 0);
}

cudaError_t sno_tc_grad(const void *map_x, const void *map_y, const SnoTcGradArgs &a, int cols, int sms, cudaStream_t s)
{
    if (cols != 64 && cols != 128)
        return cudaErrorInvalidValue;
    const dim3 grid((unsigned)sno_tc_grad_ctas(a.rows, sms), 1);
    return cols == 64 ? launch_grad<0>(map_x, map_y, a, grid, s) : launch_grad<1>(map_x, map_y, a, grid, s);
}

cudaError_t sno_tc_grad_spec(const void *map_vh, const void *map_dy, const SnoTcGradArgs &a, int modes, cudaStream_t s)
{
    SnoTcGradArgs b = a;
    b.modes = modes;
    const unsigned extra = (unsigned)(a.bias[0].cols + a.bias[1].cols) / 16;
    return launch_grad<2>(map_vh, map_dy, b, dim3(1, (unsigned)modes + extra), s);
}

}  // namespace ge

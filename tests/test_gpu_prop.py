"""Composed steps (GE_KERNEL_AUTO): k steps as one banded operator, on the
tensor cores away from the walls and as FP64 dot products near them, against
the oracle and the tiled kernel.

Tolerances: FP64 1e-12 relative max-norm (tests/tolerances.py), FP32 1e-5, as
for every other path.  Where the data's magnitude changes from block to block
(64 points) each block is held to its own largest value: the operator takes
dot products for blocks below 2^-16 of what reaches them, and the others keep
at least 54 - 16 - 1 bits, so 2^-37 a pass and at most a few passes: 1e-10.
"""
import numpy as np
import pytest
import torch

import oracle
from tolerances import tol64
from paper_1310_3422_gb300 import binding as B
from paper_1310_3422_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def auto_run(u0, r, bl, br, steps, prec=B.GE_F64, step0=0):
    x = torch.as_tensor(np.asarray(u0), dtype=B.dtype_of(prec), device=DEV).contiguous()
    ctx = B.ge_create(len(u0), r, bl, br, prec, x)
    B.ge_write_state(ctx, x, step0)
    B.ge_step_n(ctx, steps)
    out = torch.empty_like(x)
    B.ge_read_state(ctx, out)
    B.ge_sync(ctx)
    assert B.ge_get_step(ctx) == step0 + steps
    B.ge_destroy(ctx)
    return out.double().cpu().numpy()


def rel_max(got, want):
    return float(np.max(np.abs(got - want)) / np.max(np.abs(want)))


# all dot products below 8192 points; above, tiles of 128 blocks of 64 points
# between the two wall ranges: one block, one tile more or less, odd ends
@pytest.mark.parametrize("n", [16, 17, 65, 1000, 8191, 8192, 9281, 17407, 17473, 40001])
@pytest.mark.parametrize("steps", [20, 21, 200, 777])
@pytest.mark.parametrize("r", [0.01, 0.7, 2.0, 6.0])
def test_matches_the_oracle(n, steps, r):
    step0 = steps & 1
    u0 = inputs.random_state(n, seed=n + steps)
    want = oracle.run(u0, r, 0.3, -0.8, steps, step0)
    assert rel_max(auto_run(u0, r, 0.3, -0.8, steps, step0=step0), want) <= tol64(r)
    f0 = u0.astype(np.float32).astype(np.float64)
    want = oracle.run(f0, r, 0.3, -0.8, steps, step0)
    for prec in (B.GE_F32, B.GE_F32_COMP):
        assert rel_max(auto_run(f0, r, 0.3, -0.8, steps, prec, step0), want) <= 1e-5


@pytest.mark.parametrize("prec,tol", [(B.GE_F64, 1e-10), (B.GE_F32, 1e-3)])
def test_each_block_keeps_its_own_digits(prec, tol):
    """A pulse on a zero ground, steps between magnitudes, and a ramp over 30 decades."""
    n, r, steps = 50000, 1.5, 140
    u0 = np.zeros(n)
    u0[9000:9400] = 1.0
    u0[20000:30000] = 1e-20 * inputs.random_state(10000, seed=3)
    u0[25000:25064] += 1.0
    u0[35000:45000] = 10.0 ** np.linspace(-20, 0, 10000)
    u0 = u0.astype(np.float32).astype(np.float64)
    want = oracle.run(u0, r, 0.0, 0.0, steps)
    got = auto_run(u0, r, 0.0, 0.0, steps, prec)
    floor = 1e-30 if prec == B.GE_F64 else 1e-25
    for a in range(0, n, 64):
        big = np.max(np.abs(want[a:a + 64]))
        if big > floor:
            assert np.max(np.abs(got[a:a + 64] - want[a:a + 64])) <= tol * big, a
    assert not got[np.flatnonzero(want == 0.0)].any()


@pytest.mark.parametrize("r,steps", [(0.05, 300), (2.0, 100)])
def test_values_that_are_not_finite_reach_as_far_as_step_by_step(r, steps):
    n = 30000
    u0 = inputs.random_state(n, seed=9)
    u0[12000], u0[25001] = np.nan, np.nan
    want = oracle.run(u0, r, 0.1, 0.2, steps)
    got = auto_run(u0, r, 0.1, 0.2, steps)
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    ok = np.isfinite(want)
    assert rel_max(got[ok], want[ok]) <= tol64(r)


@pytest.mark.parametrize("prec,n,r,steps", [
    (B.GE_F64, 1 << 20, 1.0, 60), (B.GE_F64, (1 << 19) + 7, 4.0, 801), (B.GE_F32, (1 << 18) + 1, 4.0, 2001),
    (B.GE_F32_COMP, 1 << 18, 4.0, 2000)])
def test_grids_of_spikes_go_step_by_step(prec, n, r, steps):
    """Most blocks far below their neighbours: the whole grid takes the steps
    themselves, as rounds of one launch (the longer runs: several operators,
    the middle ones between right-hand sides, the scale taken out)."""
    u0 = np.zeros(n)
    u0[::4999] = 1.0
    want = oracle.run(u0, r, 0.2, -0.1, steps)
    got = auto_run(u0, r, 0.2, -0.1, steps, prec)
    assert rel_max(got, want) <= (tol64(r) if prec == B.GE_F64 else 1e-5)
    if prec == B.GE_F64:  # blocks between the spikes keep their own digits
        for a in range(64 * 20, n - 64 * 20, 64 * 37):
            big = np.max(np.abs(want[a:a + 64]))
            assert np.max(np.abs(got[a:a + 64] - want[a:a + 64])) <= 1e-10 * big, a


def test_magnitudes_near_the_ends_of_the_exponent_range():
    n, r, steps = 20000, 2.0, 200
    u0 = inputs.random_state(n, seed=4)
    want = oracle.run(u0, r, 0.0, 0.0, steps)
    for e in (-1000, 1000):
        got = auto_run(np.ldexp(u0, e), r, 0.0, 0.0, steps)
        assert rel_max(np.ldexp(got, -e), want) <= tol64(r)


def test_captured_graph_and_later_direct_calls():
    """A call captured from a fresh context builds its operator in the graph;
    replays and direct calls (the same steps, others, and more kinds than the
    context keeps) give the same results."""
    n, r = 20001, 1.2
    u0 = inputs.random_state(n, seed=12)
    x = torch.tensor(u0, device=DEV)
    out = torch.empty_like(x)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = B.ge_create(n, r, 0.2, -0.1, B.GE_F64, x, stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            B.ge_write_state(ctx, x, 0)
            B.ge_step_n(ctx, 300)
            B.ge_read_state(ctx, out)
        for steps in ("replay", 300, 40, 41, 60, "replay", 80, 100, 300, "replay"):
            out.zero_()
            if steps == "replay":
                graph.replay()
            else:
                B.ge_write_state(ctx, x, 0)
                B.ge_step_n(ctx, steps)
                B.ge_read_state(ctx, out)
            B.ge_sync(ctx)
            want = oracle.run(u0, r, 0.2, -0.1, 300 if steps == "replay" else steps)
            assert rel_max(out.cpu().numpy(), want) <= tol64(r), steps
        del graph
    torch.cuda.synchronize()


# 2, 11, 30, 70 and 75 tiles: clusters of 8, 8, 4, 2 and 2 CTAs a tile, where
# the device holds that many; 97 tiles in the larger grid: one CTA each
@pytest.mark.parametrize("n", [20000, 93001, 249990, 580003, 619000])
@pytest.mark.parametrize("r,steps", [(0.01, 21), (0.7, 300), (0.7, 2000)])
@pytest.mark.parametrize("prec", [B.GE_F64, B.GE_F32, B.GE_F32_COMP])
def test_split_tiles_give_the_same_bits(n, r, steps, prec):
    """Integer sums split over a cluster are the unsplit ones: the start of a
    larger grid, whose tiles are not split, gives the same bits away from the
    smaller grid's right wall (a tile and its halo, at most 16 blocks)."""
    if prec != B.GE_F64:
        steps = max(steps, 150)  # fewer go step by step, from 128 + n 192 / 2^24
    u0 = inputs.random_state(800000, seed=3)
    want = auto_run(u0, r, 0.3, -0.8, steps, prec)
    got = auto_run(u0[:n], r, 0.3, -0.8, steps, prec)
    m = n - 8192 - 17 * 64
    assert np.array_equal(got[:m], want[:m])
    assert np.all(np.isfinite(got))


# an FP32 row's sum runs in FP32 between 2^-70 and 2^90, else in FP64; above
# 8192 points these are the rows near a wall
@pytest.mark.parametrize("n", [1000, 9281])
@pytest.mark.parametrize("exp", [-100, -71, -69, 88, 91, 100])
def test_fp32_rows_at_any_magnitude(n, exp):
    """The scheme is linear: data and walls times 2^exp give the result times
    2^exp, within the FP32 tolerance."""
    r, steps = 0.7, 300
    u0 = inputs.random_state(n, seed=exp + 200).astype(np.float32).astype(np.float64)
    want = oracle.run(u0, r, 0.25, -0.75, steps, 0)
    s = 2.0 ** exp
    got = auto_run(u0 * s, r, 0.25 * s, -0.75 * s, steps, B.GE_F32)
    assert rel_max(got / s, want) <= 1e-5


def tiled_run(u0, r, bl, br, steps, prec):
    x = torch.as_tensor(np.asarray(u0), dtype=B.dtype_of(prec), device=DEV).contiguous()
    ctx = B.ge_create(len(u0), r, bl, br, prec, x)
    B.ge_set_kernel(ctx, B.GE_KERNEL_TEMPORAL, 0)
    B.ge_step_n(ctx, steps)
    out = torch.empty_like(x)
    B.ge_read_state(ctx, out)
    B.ge_sync(ctx)
    B.ge_destroy(ctx)
    return out.double().cpu().numpy()


# large enough for two teams a CTA on 152 SMs (304 tiles of 128 blocks), with
# the narrowest and the widest halos they take, whole and ragged last tiles
@pytest.mark.parametrize("n", [304 * 8192 + 64 * 22 * 2 + 1, 2700003])
@pytest.mark.parametrize("prec,r,steps", [(B.GE_F64, 0.01, 24), (B.GE_F64, 0.5, 24), (B.GE_F64, 2.0, 41),
                                          (B.GE_F32, 0.05, 200), (B.GE_F32, 2.0, 400), (B.GE_F32, 2.0, 2000)])
def test_two_teams_match_the_tiled_kernel(n, prec, r, steps):
    """Each path is within its tolerance of the exact steps: twice that apart.
    Random data, and the same with a stretch of zeros, a far smaller one and
    (last) an infinity, whose reach both paths agree on."""
    tol = 2 * tol64(r) if prec == B.GE_F64 else 2e-5
    u0 = inputs.random_state(n, seed=n % 97)
    if prec != B.GE_F64:
        u0 = u0.astype(np.float32).astype(np.float64)
    assert rel_max(auto_run(u0, r, 0.3, -0.8, steps, prec), tiled_run(u0, r, 0.3, -0.8, steps, prec)) <= tol
    u0[n // 3:n // 3 + 100000] = 0.0
    u0[n // 2:n // 2 + 30000] *= 2.0 ** -40
    got, want = auto_run(u0, r, 0.3, -0.8, steps, prec), tiled_run(u0, r, 0.3, -0.8, steps, prec)
    assert rel_max(got, want) <= tol
    inner = slice(n // 2 + 2 * steps + 64, n // 2 + 30000 - 2 * steps - 64)
    assert rel_max(got[inner], want[inner]) <= (1e-10 if prec == B.GE_F64 else 1e-3)
    u0[n // 4] = np.inf
    got, want = auto_run(u0, r, 0.3, -0.8, steps, prec), tiled_run(u0, r, 0.3, -0.8, steps, prec)
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    ok = np.isfinite(want)
    assert rel_max(got[ok], want[ok]) <= tol


# dot products only; split tiles; whole tiles; and, FP32, two teams a CTA
@pytest.mark.parametrize("n", [5000, 40001, 1300001])
@pytest.mark.parametrize("prec,r,steps", [(B.GE_F64, 2.0, 700), (B.GE_F64, 0.7, 2001), (B.GE_F32, 2.0, 2000),
                                          (B.GE_F32, 4.0, 1800), (B.GE_F32_COMP, 2.0, 2001)])
def test_a_hot_wall_beside_a_quiet_field(n, prec, r, steps):
    """What a wall sends into a field of zeros, and into one far below it,
    arrives block by block down to 2^-86 of the wall value (ge.h: 2^-100; the
    last standard deviation is cut off with the taps): within the FP64 (1e-10,
    as above) and FP32 tolerances of each block's largest value."""
    tol, far = (1e-10, 2.0 ** -86) if prec == B.GE_F64 else (1e-5, 2.0 ** -86)
    for ground in (0.0, 2.0 ** -60):
        for left, right in ((1.0, 0.0), (0.0, -1.0)):
            u0 = ground * np.sin(np.arange(n) * 0.01)
            u0 = u0.astype(np.float32).astype(np.float64)
            want = oracle.run(u0, r, left, right, steps)
            got = auto_run(u0, r, left, right, steps, prec)
            rows = min(n, 64 * 64)
            for a in range(0, rows, 64):
                part = slice(a, a + 64) if left else slice(n - 64 - a, n - a)
                big = np.max(np.abs(want[part]))
                if big > far:
                    assert np.max(np.abs(got[part] - want[part])) <= tol * big, (ground, left, a)


@pytest.mark.parametrize("r,steps", [(7.5, 670), (12.0, 640), (16.0, 690)])
def test_two_teams_with_the_largest_tables(r, steps):
    """The widest halo of two FP32 teams with taps that reach as far as the
    steps do: the tables leave the planes the least room."""
    n = 304 * 8192 + 64 * 22 * 2 + 1
    u0 = inputs.random_state(n, seed=7).astype(np.float32).astype(np.float64)
    assert rel_max(auto_run(u0, r, 0.3, -0.8, steps, B.GE_F32), tiled_run(u0, r, 0.3, -0.8, steps, B.GE_F32)) <= 2e-5


@pytest.mark.parametrize("prec,n,r,steps", [(B.GE_F64, 327663, 7.0, 36), (B.GE_F32, 1942719, 3e-5, 803)])
def test_spikes_cost_no_multiple_of_the_tiled_kernel(prec, n, r, steps):
    """Taps of a few points, nearly every block left to dot products: their
    set-up counts, and the steps themselves are sooner done.  (The pass of the
    tiles that finds out costs up to a third of a call here: twice is allowed.)"""
    x = torch.zeros(n, dtype=B.dtype_of(prec), device=DEV)
    x[::4999] = 1.0
    ms = {}
    for kernel in (B.GE_KERNEL_AUTO, B.GE_KERNEL_TEMPORAL):
        ctx = B.ge_create(n, r, 0.5, 0.0, prec, x)
        B.ge_set_kernel(ctx, kernel, 0)
        times = []
        for _ in range(6):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            B.ge_write_state(ctx, x, 0)
            start.record()
            B.ge_step_n(ctx, steps)
            end.record()
            B.ge_sync(ctx)
            torch.cuda.synchronize()
            times.append(start.elapsed_time(end))
        ms[kernel] = min(times)
        B.ge_destroy(ctx)
    assert ms[B.GE_KERNEL_AUTO] <= 2.0 * ms[B.GE_KERNEL_TEMPORAL], ms

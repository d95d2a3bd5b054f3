"""The launch shapes chosen by size give the results of any other shape."""
import numpy as np
import pytest
import torch

import oracle
from tolerances import tol64
from paper_1310_3422_gb300 import binding as B
from paper_1310_3422_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


# n on both sides of the lines between depths 48, 32, 24, 16, 12 and 8 (one
# tile an SM on 152 SMs), and 8 forced: the same arithmetic at every depth
@pytest.mark.parametrize("prec", [B.GE_F64, B.GE_F32])
@pytest.mark.parametrize("k", [2, 7, 16, 64])
@pytest.mark.parametrize("n", [300, 90001, 160000, 1 << 20, 1300007])
def test_width_depth_by_size(prec, k, n):
    steps = 53
    x = torch.as_tensor(inputs.random_state(n, seed=n % 89), dtype=B.dtype_of(prec), device=DEV)

    def run(depth):
        ctx = B.ge_create(n, 1.3, 0.2, -0.5, prec, x)
        if depth:
            B.ge_set_kernel(ctx, B.GE_KERNEL_AUTO, depth)
        B.ge_set_subdomain_width(ctx, k)
        B.ge_step_n(ctx, steps)
        out = torch.empty_like(x)
        B.ge_read_state(ctx, out)
        B.ge_sync(ctx)
        B.ge_destroy(ctx)
        return out

    assert torch.equal(run(0), run(8))


# few tiles, many tiles of long problems, many of problems shorter than a tile
@pytest.mark.parametrize("prec", [B.GE_F64, B.GE_F32, B.GE_F32_COMP])
@pytest.mark.parametrize("sizes", [[256, 3000, 17, 900], [40000] * 40, [700, 1500, 2900] * 500])
def test_batch_shape_by_size(prec, sizes):
    rng = np.random.default_rng(len(sizes))
    n = np.asarray(sizes, np.int64)
    per = 32
    off = np.concatenate([[0], np.cumsum((n + per - 1) // per * per)[:-1]]).astype(np.int64)
    total = int(off[-1] + (n[-1] + per - 1) // per * per)
    r = rng.uniform(0.25, 4.0, len(n))
    u = rng.uniform(-1.0, 1.0, total).astype(np.float32).astype(np.float64)
    zero = np.zeros(len(n))
    plan = B.ge_batch_create(n, r, zero, zero, off, total, prec)
    x = torch.as_tensor(u, dtype=B.dtype_of(prec), device=DEV)
    B.ge_batch_run(plan, x, 230)
    B.ge_batch_sync(plan)
    got = x.double().cpu().numpy()
    for i in list(range(min(4, len(n)))) + [len(n) - 1]:
        want = oracle.run(u[off[i]:off[i] + n[i]], r[i], 0.0, 0.0, 230)
        tol = tol64(r[i]) if prec == B.GE_F64 else 1e-5
        assert np.max(np.abs(got[off[i]:off[i] + n[i]] - want)) <= tol * np.max(np.abs(want)), i
    B.ge_batch_destroy(plan)


@pytest.mark.parametrize("problems", [4, 600])
def test_a_plans_own_choice_follows_its_kernel(problems):
    """Depth 0 is the plan's own choice, for the kernel it runs at the time; a
    chosen depth or geometry stays."""
    n = np.full(problems, 4096, np.int64)
    off = np.arange(problems, dtype=np.int64) * 4096
    r, zero = np.full(problems, 1.0), np.zeros(problems)

    def shape(*calls):
        plan = B.ge_batch_create(n, r, zero, zero, off, problems * 4096, B.GE_F64)
        for f, *args in calls:
            f(plan, *args)
        got = B.ge_batch_get_depth(plan), B.ge_batch_get_geometry(plan)[0]
        B.ge_batch_destroy(plan)
        return got

    df, auto = (B.ge_batch_set_kernel, B.GE_KERNEL_TEMPORAL_DF), (B.ge_batch_set_kernel, B.GE_KERNEL_AUTO)
    own, own_df = shape(), shape(df)
    assert own_df == (48, 256) and own != own_df
    assert shape((B.ge_batch_set_depth, 0)) == own and shape((B.ge_batch_set_depth, 0), df) == own_df
    assert shape((B.ge_batch_set_depth, 96), (B.ge_batch_set_depth, 0), df) == own_df
    assert shape((B.ge_batch_set_depth, 0), df, auto) == own
    assert shape((B.ge_batch_set_depth, 96), df) == (96, 256)
    assert shape((B.ge_batch_set_geometry, 256, 0), df, auto) == (own[0], 256)

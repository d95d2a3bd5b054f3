"""Errors of composed steps (GE_KERNEL_AUTO) against the steps evaluated in
extended precision (numpy.longdouble: 64 or 113 bits), beside those of the
tiled kernel, which takes the same steps one by one."""
import numpy as np
import pytest
import torch

from paper_1310_3422_gb300 import binding as B

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
LD = np.longdouble
SLACK = 1.25


def exact(u0, r, bl, br, steps):
    """Steps of parity 0, 1, 0, ... of the rows of u0: (I + r G_p) u' = (I - r G_1-p) u + r walls."""
    u, r = np.array(u0, dtype=LD), LD(r)
    n = u.shape[-1]
    for s in range(steps):
        p = s & 1
        w = (1 - r) * u
        a, b = slice(1 - p, n - ((n - 1 + p) & 1), 2), slice(2 - p, n - ((n - 1 + p) & 1), 2)
        w[..., a] += r * u[..., b]
        w[..., b] += r * u[..., a]
        w[..., 0] += r * LD(bl)
        w[..., -1] += r * LD(br)
        u = w / (1 + r)
        a, b = slice(p, n - ((n - p) & 1), 2), slice(p + 1, n - ((n - p) & 1), 2)
        u[..., a] = ((1 + r) * w[..., a] + r * w[..., b]) / (1 + 2 * r)
        u[..., b] = ((1 + r) * w[..., b] + r * w[..., a]) / (1 + 2 * r)
    return u


def run(u0, r, bl, br, steps, kernel, prec=B.GE_F64):
    x = torch.as_tensor(np.asarray(u0), dtype=B.dtype_of(prec), device=DEV).contiguous()
    ctx = B.ge_create(len(u0), r, bl, br, prec, x)
    B.ge_set_kernel(ctx, kernel, 0)
    B.ge_step_n(ctx, steps)
    out = torch.empty_like(x)
    B.ge_read_state(ctx, out)
    B.ge_sync(ctx)
    B.ge_destroy(ctx)
    return out.cpu().numpy()


def rms_errors(u0, r, bl, br, steps, prec, parts=None):
    """RMS error of both kernels over the rows of u0, divided by the exact
    field's RMS there (over `parts` of a row)."""
    want = exact(u0, r, bl, br, steps)
    parts = slice(None) if parts is None else parts
    norm = np.sqrt(np.mean(want[:, parts] ** 2))
    return [float(np.sqrt(np.mean([np.mean((run(u, r, bl, br, steps, kernel, prec)[parts] - w[parts]) ** 2)
                                   for u, w in zip(u0, want)])) / norm)
            for kernel in (B.GE_KERNEL_AUTO, B.GE_KERNEL_TEMPORAL)]


def rough(seeds, n, dtype=np.float64):
    return np.stack([np.random.default_rng(s).standard_normal(n) for s in range(seeds)]).astype(dtype).astype(np.float64)


# r far above any the other tests take: taps of both signs, up to r / 2; dot
# products only, and tiles
@pytest.mark.parametrize("n", [1024, 12000])
@pytest.mark.parametrize("r", [30.0, 1000.0, 1e6])
@pytest.mark.parametrize("prec,steps", [(B.GE_F64, 24), (B.GE_F64, 150), (B.GE_F32, 150), (B.GE_F32_COMP, 150)])
def test_large_mesh_ratios(n, r, prec, steps):
    """Composed steps err no more than steps one by one, up to the scatter of
    one rough field's error (a few hundred independent samples: 1.25)."""
    u0 = rough(1, n, np.float64 if prec == B.GE_F64 else np.float32)
    auto, tiled = rms_errors(u0, r, 0.3, -0.8, steps, prec)
    assert auto <= SLACK * tiled, (auto, tiled)


# dot products only (n < 8192): few and many steps, each row's sum a few or a
# few hundred terms; the r of the tests' accuracy runs
@pytest.mark.parametrize("r,steps", [(0.05, 8), (0.5, 24), (0.5, 100), (1.0, 8), (1.0, 24), (1.0, 400), (2.0, 24),
                                     (4.0, 100)])
def test_short_rows_of_rough_data(r, steps):
    """Composed steps err no more than steps one by one.  Sixteen fields of
    1024 points, whose errors are correlated over the reach of the steps (r =
    1, 400 steps: 28 points): some 500 independent samples of a mean square,
    6 % in its root for either kernel, 1.1."""
    auto, tiled = rms_errors(rough(16, 1024), r, 0.3, -0.8, steps, B.GE_F64)
    assert auto <= 1.1 * tiled, (auto, tiled)


# either side of where blocks go to dot products instead: by their values
# (2^-8 to 2^-12 of their neighbours', FP32 2^-5 to 2^-9), by their results
@pytest.mark.parametrize("level", [2, 4, 5, 6, 7, 8, 9, 10, 12, 16, 24])
@pytest.mark.parametrize("prec,r,steps", [(B.GE_F64, 1.0, 24), (B.GE_F64, 0.5, 100), (B.GE_F64, 2.0, 300),
                                          (B.GE_F32, 1.0, 150), (B.GE_F32, 4.0, 400), (B.GE_F32_COMP, 1.0, 150),
                                          (B.GE_F32_COMP, 4.0, 400)])
def test_quiet_stretches_keep_their_precision(prec, r, steps, level):
    """Stretches of rough data 2^-level of the data around them: within them
    (14 standard deviations of the taps from their ends) composed steps err no
    more than steps one by one, relative to the stretch's own field."""
    u0 = rough(1, 20000, np.float64 if prec == B.GE_F64 else np.float32)
    inner = np.zeros(20000, bool)
    margin = int(14 * np.sqrt(2 * r * steps)) + 10
    for a in (6000, 13000):
        u0[:, a:a + 3000] *= 2.0 ** -level
        inner[a + margin:a + 3000 - margin] = True
    auto, tiled = rms_errors(u0, r, 0.3, -0.8, steps, prec, inner)
    assert auto <= SLACK * tiled, (auto, tiled)


# shorter than a launch of the compensated kernel, as long, and longer
@pytest.mark.parametrize("n", [19, 41, 129, 130, 400])
def test_short_compensated_grids(n):
    """A state rounded to FP32 at the end of every operator errs no more than
    one rounded at the end of every launch of the tiled kernel."""
    auto, tiled = rms_errors(rough(16, n, np.float32), 1e-4, 0.25, -0.75, 958, B.GE_F32_COMP)
    assert auto <= SLACK * tiled, (auto, tiled)


@pytest.mark.parametrize("prec", [B.GE_F64, B.GE_F32])
@pytest.mark.parametrize("r", [1.4e-6, 1e-7, 1e-12, 1e-300])
def test_steps_that_hardly_move(prec, r):
    """The tiled kernel at mesh ratios where its scale never needs taking down,
    and the default path, whichever it takes."""
    u0 = rough(1, 3000, np.float64 if prec == B.GE_F64 else np.float32)
    want = exact(u0, r, 0.3, -0.8, 60)[0]
    for kernel in (B.GE_KERNEL_TEMPORAL, B.GE_KERNEL_AUTO):
        got = run(u0[0], r, 0.3, -0.8, 60, kernel, prec)
        assert np.max(np.abs(got - want)) <= (1e-12 if prec == B.GE_F64 else 1e-5) * np.max(np.abs(want))


@pytest.mark.parametrize("n,r,steps", [(24, 0.003, 2000), (100, 1.0, 4000), (300, 1.0, 6000), (1000, 4.0, 5000)])
def test_many_operators_one_after_the_other(n, r, steps):
    """Twenty and more operators: what each has wrong in common with the last
    adds up, and stays below what the steps one by one add up."""
    x = np.arange(1, n + 1) / (n + 1)
    for u0 in (rough(2, n), np.stack([np.sin(3 * np.pi * x) + 0.2 * np.sin(40 * np.pi * x)])):
        auto, tiled = rms_errors(u0, r, 0.3, -0.8, steps, B.GE_F64)
        assert auto <= SLACK * tiled, (auto, tiled)

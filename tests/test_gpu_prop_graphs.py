"""Composed steps (GE_KERNEL_AUTO) captured in CUDA graphs: the operators a
graph reads belong to it while it lives, and only then."""
import time

import numpy as np
import pytest
import torch

import oracle
from tolerances import tol64
from paper_1310_3422_gb300 import binding as B
from paper_1310_3422_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
N, R = 20001, 1.2


def fresh(x, steps, kernel=B.GE_KERNEL_AUTO, r=R, bl=0.2, br=-0.1, prec=B.GE_F64):
    ctx = B.ge_create(x.numel(), r, bl, br, prec, x)
    B.ge_set_kernel(ctx, kernel, 0)
    out = direct(ctx, x, steps)
    B.ge_destroy(ctx)
    return out


def direct(ctx, x, steps):
    out = torch.empty_like(x)
    B.ge_write_state(ctx, x, 0)
    B.ge_step_n(ctx, steps)
    B.ge_read_state(ctx, out)
    B.ge_sync(ctx)
    return out.cpu().numpy()


def capture(ctx, x, out, steps, stream):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        B.ge_write_state(ctx, x, 0)
        B.ge_step_n(ctx, steps)
        B.ge_read_state(ctx, out)
    return graph


def test_operators_come_back_when_a_graph_is_gone():
    """Nine graphs, one after the other, of a context that keeps six operators:
    a call of yet another kind afterwards still takes composed steps (the bits
    of a fresh context's, which are not the tiled kernel's)."""
    x = torch.tensor(inputs.random_state(N, seed=12), device=DEV)
    want, tiled = fresh(x, 500), fresh(x, 500, B.GE_KERNEL_TEMPORAL)
    assert not np.array_equal(want, tiled)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = B.ge_create(N, R, 0.2, -0.1, B.GE_F64, x, stream)
        out = torch.empty_like(x)
        for i in range(9):
            graph = capture(ctx, x, out, 40 + 20 * i, stream)
            graph.replay()
            B.ge_sync(ctx)
            del graph
        deadline = time.monotonic() + 10.0  # CUDA gives them back in its own time
        while True:
            got = direct(ctx, x, 500)
            if np.array_equal(got, want) or time.monotonic() > deadline:
                break
            time.sleep(0.05)
        assert np.array_equal(got, want)
        B.ge_destroy(ctx)


def test_live_graphs_keep_their_operators():
    """Three graphs of three operators each would need nine: whatever each got,
    their replays and direct calls in between give the same results, also after
    the context's other graphs are gone; a graph may outlive its context."""
    u0 = inputs.random_state(N, seed=13)
    x = torch.tensor(u0, device=DEV)
    steps = (4000, 4400, 4800)  # r k at most 1512 an operator: a first, middle ones, a last
    want = {s: oracle.run(u0, R, 0.2, -0.1, s) for s in steps + (300,)}
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = B.ge_create(N, R, 0.2, -0.1, B.GE_F64, x, stream)
        outs = [torch.empty_like(x) for _ in steps]
        graphs = [capture(ctx, x, o, s, stream) for s, o in zip(steps, outs)]

        def check(i):
            outs[i].zero_()
            graphs[i].replay()
            B.ge_sync(ctx)
            assert np.max(np.abs(outs[i].cpu().numpy() - want[steps[i]])) <= tol64(R) * np.max(np.abs(want[steps[i]]))

        for i in (0, 1, 2, 0):
            check(i)
            for s in (300, steps[(i + 1) % 3]):
                got = direct(ctx, x, s)
                assert np.max(np.abs(got - want[s])) <= tol64(R) * np.max(np.abs(want[s]))
        graphs[1] = None
        torch.cuda.synchronize()
        time.sleep(0.2)
        for s in (300, 700, 900, 1100):
            direct(ctx, x, s)
        check(0)
        check(2)
        B.ge_destroy(ctx)
        del graphs
    torch.cuda.synchronize()


@pytest.mark.parametrize("prec,n,r,steps", [(B.GE_F64, 1 << 20, 1.0, 60), (B.GE_F32, (1 << 18) + 1, 4.0, 2001)])
def test_the_step_by_step_rounds_in_a_graph(prec, n, r, steps):
    """Spikes on zeros, where most blocks are left to the cooperative launch
    that takes the steps themselves: captured, replayed, and direct."""
    u0 = np.zeros(n)
    u0[::4999] = 1.0
    want = oracle.run(u0, r, 0.2, -0.1, steps)
    tol = (tol64(r) if prec == B.GE_F64 else 1e-5) * np.max(np.abs(want))
    x = torch.tensor(u0, dtype=B.dtype_of(prec), device=DEV)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = B.ge_create(n, r, 0.2, -0.1, prec, x, stream)
        out = torch.empty_like(x)
        graph = capture(ctx, x, out, steps, stream)
        for _ in range(2):
            out.zero_()
            graph.replay()
            B.ge_sync(ctx)
            assert np.max(np.abs(out.double().cpu().numpy() - want)) <= tol
            assert np.max(np.abs(direct(ctx, x, steps).astype(np.float64) - want)) <= tol
        del graph
        B.ge_destroy(ctx)

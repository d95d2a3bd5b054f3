"""One-shot solves from host memory: contexts from the memory pool, and the
copy beside the operators' kernels, in several threads at once."""
import ctypes
import os
import threading

import numpy as np
import pytest
import torch

from paper_1310_3422_gb300 import binding as B
from paper_1310_3422_gb300 import inputs
from paper_1310_3422_gb300.build import CUDA_HOME

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def on_device(u0, r, steps, prec):
    x = torch.as_tensor(u0, device=DEV)
    ctx = B.ge_create(len(u0), r, 0.2, -0.4, prec, x)
    B.ge_step_n(ctx, steps)
    out = torch.empty_like(x)
    B.ge_read_state(ctx, out)
    B.ge_sync(ctx)
    B.ge_destroy(ctx)
    return out.cpu().numpy()


# too few steps to compose; dot products only; tiles; the largest pooled
# context and one past the pool's 64 MB
@pytest.mark.parametrize("n,steps", [(64, 5), (5000, 300), (100003, 300), (3500000, 40), (4500000, 40)])
@pytest.mark.parametrize("prec", [B.GE_F64, B.GE_F32])
def test_threads_get_their_own_result(n, steps, prec):
    """Four threads, three solves each, different data and r: bit for bit the
    result of a context on the device."""
    dt = np.float64 if prec == B.GE_F64 else np.float32
    data = [inputs.random_state(n, seed=40 + i).astype(dt) for i in range(4)]
    rs = [0.3, 0.7, 1.1, 1.6]
    want = [on_device(u, r, steps, prec) for u, r in zip(data, rs)]
    got = [[], [], [], []]

    def work(i):
        for _ in range(3):
            out = np.empty(n, dt)
            B.ge_solve(n, rs[i], 0.2, -0.4, prec, B.GE_KERNEL_AUTO, 0, steps, data[i], out)
            got[i].append(out)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(4):
        assert len(got[i]) == 3
        for out in got[i]:
            assert np.array_equal(out, want[i])


def test_destroy_waits_for_a_graph_on_another_stream():
    """The next context may get a released one's memory: nothing of the old
    one may still be running, also where its own stream is idle."""
    n = 1 << 20
    x = torch.as_tensor(inputs.random_state(n, seed=3), device=DEV)
    own, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(own):
        ctx = B.ge_create(n, 1.0, 0.0, 0.0, B.GE_F64, x, own)
        B.ge_set_kernel(ctx, B.GE_KERNEL_TEMPORAL, 0)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=own):
            B.ge_step_n(ctx, 20000)  # some 30 ms
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        graph.replay()
        done = torch.cuda.Event()
        done.record(other)
    assert not done.query()
    B.ge_destroy(ctx)
    assert done.query()
    del graph


def test_destroy_does_not_need_the_stream():
    """A context outlives its stream: the work it left there ends before the
    memory goes, and the next context's result is its own."""
    rt = ctypes.CDLL(os.path.join(CUDA_HOME, "lib64", "libcudart.so.13"))
    n = 100003
    u = [inputs.random_state(n, seed=s) for s in (5, 6)]
    want = on_device(u[1], 0.7, 300, B.GE_F64)
    for _ in range(3):
        handle = ctypes.c_void_p()
        assert rt.cudaStreamCreateWithFlags(ctypes.byref(handle), 1) == 0
        ctx = B.ge_create(n, 0.7, 0.2, -0.4, B.GE_F64, torch.as_tensor(u[0], device=DEV), handle.value)
        B.ge_step_n(ctx, 3000)
        assert rt.cudaStreamDestroy(handle) == 0
        B.ge_destroy(ctx)
        assert np.array_equal(on_device(u[1], 0.7, 300, B.GE_F64), want)

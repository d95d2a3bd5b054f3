"""Weight gradients of the surrogate on tcgen05 (plain mode): the activations
and their gradients are the same bits as on the mma.sync path, so what is left
is the order of FP32 sums."""
import numpy as np
import pytest
import torch

from paper_1310_3422_gb300 import binding as B
from test_gpu_sno import FULL, make_model, test_tensor_core_path_matches_the_mma_path as inference_matches
from test_gpu_sno_train import loss_grad

pytestmark = pytest.mark.gpu


# 19 problems: a whole 16-row step and a rest for a mode's gradient; 64: the
# training batch; 130, 300: more chunks than SMs, and a rest
@pytest.mark.parametrize("batch,first", [(1, 0), (3, 40), (19, 0), (64, 0), (130, 200), (300, 0)])
def test_gradients_differ_by_the_order_of_sums_only(batch, first):
    """Losses bit for bit.  A gradient is summed in chains of at most 128
    roundings to 2^-23 (16 rows each, over the CTAs of 152 SMs) and as many
    additions of the parts, on either path: below 5e-5 of a block's norm."""
    m = make_model(FULL, max(batch, first), seed=3, split=0)
    if first:
        loss_grad(m, first, 5)
    loss_tc, tc = loss_grad(m, batch, 12)
    B.ge_sno_set_tensor_cores(m, 0)
    loss_mma, mma = loss_grad(m, batch, 12)
    assert np.array_equal(loss_tc, loss_mma)
    for k in mma:
        den = max(np.linalg.norm(mma[k]), 1e-12)
        assert np.linalg.norm(tc[k] - mma[k]) <= 5e-5 * den, (k, np.linalg.norm(tc[k] - mma[k]) / den)
    B.ge_sno_destroy(m)


@pytest.mark.parametrize("batch", [3, 64, 300])
def test_all_but_the_matrices_are_the_same_from_run_to_run(batch):
    """Bias gradients, spectral gradients and the last projection's are summed
    in a fixed order (the matrices' parts are added as they come)."""
    m = make_model(FULL, batch, seed=3, split=0)
    _, want = loss_grad(m, batch, 12)
    for _ in range(6):
        _, got = loss_grad(m, batch, 12)
        for k in want:
            if k[0] != "W" and k != "Q1":
                assert np.array_equal(got[k], want[k]), k
    B.ge_sno_destroy(m)


@pytest.mark.parametrize("batch", [152, 153])
def test_inference_on_either_side_of_the_transform_kernels_line(batch):
    """One problem per SM has all eight chunks of its transform in flight, more
    problems two: the last batch of the one kernel on 152 SMs, the first of the other."""
    inference_matches(batch)

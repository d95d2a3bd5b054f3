"""Training with the weight gradients on tcgen05 against the mma.sync path.

Both round the same values to BF16 and accumulate in FP32, so the gradients
differ by the order of the sums and by BF16 roundings that fall the other way
(2^-8 relative each, at about ten points between a weight and the loss):
sqrt(10) 2^-8 = 1.2e-2 relative L2 if every one did, per parameter block."""
import numpy as np
import pytest
import torch

from paper_1310_3422_gb300 import binding as B
from test_gpu_sno import DEV, FULL, blocks, dev, make_model, problem_batch

pytestmark = pytest.mark.gpu
TOL = 1.2e-2


def loss_grad(m, batch, seed):
    u0, r, bl, br = problem_batch(FULL, batch, seed)
    target = (u0 + 0.1 * np.random.default_rng(seed).standard_normal(u0.shape)).astype(np.float32)
    loss = torch.empty(batch, dtype=torch.float32, device=DEV)
    grads = torch.empty(B.ge_sno_num_params(m), dtype=torch.float32, device=DEV)
    B.ge_sno_loss_grad(m, batch, *dev(u0, r, bl, br, target), loss, grads)
    B.ge_sno_sync(m)
    return loss.cpu().numpy(), blocks(FULL, grads.cpu().numpy().astype(np.float64))


# 1 and 3: a mode's weight gradient sums fewer rows than one 16-row step;
# 19: a step and a remainder; 152, 153: the last batch whose DFT keeps 8
# stages, the first that keeps 2; 130, 300: a whole chunk of 128 and a rest.
# `first`: a larger batch run before leaves its rows in the buffers.
@pytest.mark.parametrize("batch,first", [(1, 0), (3, 40), (19, 0), (130, 200), (152, 0), (153, 0), (300, 0)])
def test_gradients_match_the_mma_path(batch, first):
    m = make_model(FULL, max(batch, first), seed=3, split=0)
    assert B.ge_sno_get_tensor_cores(m) == 1
    if first:
        loss_grad(m, first, 5)
    loss_tc, tc = loss_grad(m, batch, 12)
    B.ge_sno_set_tensor_cores(m, 0)
    loss_mma, mma = loss_grad(m, batch, 12)
    np.testing.assert_allclose(loss_tc, loss_mma, rtol=TOL)
    for k in mma:
        den = max(np.linalg.norm(mma[k]), 1e-12)
        assert np.linalg.norm(tc[k] - mma[k]) <= TOL * den, (k, np.linalg.norm(tc[k] - mma[k]) / den)
    B.ge_sno_destroy(m)

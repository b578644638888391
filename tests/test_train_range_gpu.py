"""The training loss at the upper end of FP32: a mean of squares that FP32 holds is
finite however many rows it is the mean of."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 31, 256, 300, 20000])
def test_loss_of_large_residuals(rows):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2311_10201_gb300 as fbpt
    fbpt.build()
    p = np.zeros(fbpt.lib().fbpt_policy_param_count(), np.float32)
    p[6:12] = 1  # all weights zero: every output is 0
    y = np.full(rows, 3e18, np.float32)
    loss, grad = fbpt.policy_loss_grad(p, np.zeros((rows, 6), np.float32), np.zeros(rows, np.uint32), y)
    # a thread's squares are summed in FP32 (one of 20,000 rows here), rounded once each
    assert loss == pytest.approx(float(y[0]) ** 2, rel=1e-6)
    # the gradient of the taken output's bias is the mean of 2 * (0 - y): a few hundred FP32 additions
    assert grad[-8] == pytest.approx(-2 * float(y[0]), rel=256 * 2.0**-24)
    assert np.all(grad[-7:] == 0)

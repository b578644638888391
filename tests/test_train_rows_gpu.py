"""The training kernel at the row counts where its tiling can go wrong (warps of
32 rows, CTAs of 256, two CTAs an SM), with actions over all eight outputs, and
with non-finite rows; the update fused into the last CTA against separate
gradient and Adam calls."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fbpt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2311_10201_gb300 as f
    f.build()
    return f


def problem(seed, rows):
    rng = np.random.default_rng(seed)
    p = rng.normal(0, 0.4, mlp.N_PARAMS)
    P = mlp.unpack(p)
    P["mu"][:] = rng.normal(0, 1, mlp.N_IN)
    P["sd"][:] = rng.uniform(0.5, 2, mlp.N_IN)
    X = rng.normal(0, 2, (rows, mlp.N_IN)).astype(np.float32)
    return p.astype(np.float32), X, rng.integers(0, mlp.N_OUT, rows), rng.normal(0, 1, rows).astype(np.float32)


# 152 SMs x 2 CTAs x 256 rows = 77,824: one round of the grid, and one row more
@pytest.mark.parametrize("rows", [1, 31, 32, 33, 255, 257, 1000, 77824, 77825, 100003])
def test_gradient_at_the_tiling_edges(fbpt, rows):
    p, X, a, y = problem(rows, rows)
    L_ref, g_ref = mlp.loss_grad(p.astype(np.float64), X.astype(np.float64), a, y.astype(np.float64))
    L, g = fbpt.policy_loss_grad(p, X, a, y)
    # FP32 sums of at most ~100 terms per accumulator: the bounds of the 600-row test
    assert abs(L - L_ref) <= 1e-5 * max(1.0, abs(L_ref))
    assert np.max(np.abs(g - g_ref)) <= 2e-5 * np.max(np.abs(g_ref)) + 1e-7


def test_fused_update_equals_separate_calls(fbpt):
    """Three training steps against loss_grad + adam_step calls: the same
    kernel arithmetic up to the order of the FP32 gradient sums (relative
    2e-5), which Adam's step can turn into at most lr per weight and step where
    a gradient is rounding noise; all others agree to 2e-5 of lr per step
    times the conditioning 1/sqrt(v) (bounded by 100 here)."""
    p, X, a, y = problem(5, 4097)
    lr = 3e-3
    pol, L = fbpt.policy_train(X, a, y, steps=3, lr=lr, init=p)
    P, m, v = p, np.zeros_like(p), np.zeros_like(p)
    gs = []
    for t in (1, 2, 3):
        _, g = fbpt.policy_loss_grad(P, X, a, y)
        gs.append(np.abs(g))
        P, m, v = fbpt.policy_adam_step(P, g, m, v, t, lr)
    L2, _ = fbpt.policy_loss_grad(P, X, a, y)
    d = np.abs(pol.params() - P)
    strong = np.min(gs, axis=0) > 1e-3 * np.max(gs)
    assert np.all(d[strong] <= 3 * lr * 2e-5 * 1000 + 4 * np.finfo(np.float32).eps * np.abs(P[strong]))
    assert np.all(d <= 3 * 2 * lr)
    assert np.array_equal(pol.params()[:12], p[:12])
    assert abs(L - L2) <= 1e-3 * max(1.0, L2)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_a_non_finite_row_reaches_only_the_weights_it_touches(fbpt, bad):
    """A target that is not finite makes its row's error so: the gradient is
    non-finite exactly at the weights of units that are on for that row
    (a zero activation or error adds nothing), as the FP64 rule applied row by
    row says."""
    p, X, a, y = problem(11, 70)
    y[40] = bad
    out, (Xn, a1, h1, a2, h2) = mlp.forward(p.astype(np.float64), X.astype(np.float64))
    on1, on2 = h1[40] > 0, h2[40] > 0
    _, g = fbpt.policy_loss_grad(p, X, a, y)
    G = mlp.unpack(g)
    assert np.array_equal(~np.isfinite(G["b2"]), on2)
    assert np.array_equal(~np.isfinite(G["W2"]), on2[:, None] & on1[None, :])
    assert np.array_equal(~np.isfinite(G["b1"]), on1)

"""The update's prepared epochs (permuted rows and advantage statistics of all
minibatches at once, gathers by 32-byte pieces of the sample-major rows)
against the per-minibatch calls, which draw the permutation and the
statistics inside the step; and the bf16 engine's weight gradients in grouped
launches against the GEMM path at minibatches of a few rows."""
import numpy as np
import pytest

from test_gpu_learner import COHERENT, GRAD_TOL, HP, _dev, _learner, _on_rollout_policy, _traj, _weights
from parity_util import need_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,D,A,H,T,N,B,mb,value_only", [
    ("fp32", 5, 8, 32, 3, 7, 2, 3, False),          # the smallest minibatch, rows of 16 floats
    ("fp32", 7, 3, 32, 5, 1237, 2049, 2, False),    # one past a block of advantages; part of the batch
    ("fp32", 64, 8, 64, 2, 4099, 4096, 2, False),   # the widest row
    ("tf32", 18, 8, 64, 9, 911, 2733, 3, False),    # every row used
    ("bf16", 1, 1, 32, 4, 515, 257, 8, False),      # the narrowest row
    ("bf16", 18, 8, 256, 4, 1025, 2047, 2, False),  # engine path
    ("bf16", 12, 6, 256, 4, 700, 1399, 2, True),
    # epochs of four minibatches and more, the prepared ones: the same edges
    ("fp32", 5, 8, 32, 3, 7, 2, 9, False),
    ("fp32", 7, 3, 32, 8, 1237, 2049, 4, False),
    ("fp32", 64, 8, 64, 4, 4099, 4096, 4, False),
    ("tf32", 18, 8, 64, 9, 1012, 2277, 4, False),
    ("bf16", 18, 8, 256, 8, 1025, 2047, 4, False),
    ("bf16", 12, 6, 256, 8, 700, 1399, 4, True),
])
def test_update_equals_minibatch_calls(precision, D, A, H, T, N, B, mb, value_only):
    torch = need_gpu()
    pw, vw = _weights(D, H, A, seed=5)
    traj = _dev(torch, _on_rollout_policy(_traj(6, T, N, D, A), pw, D, H, A))
    if value_only:
        traj = {k: traj[k] for k in ("obs", "ret")}
    a, b = (_learner(D, A, H, B, precision, value_only=value_only) for _ in range(2))
    for q in (a, b):
        q.set_weights(pw, vw)
    a.update(traj, 2, mb)
    for e in range(2):
        for j in range(mb):
            b.grads(traj, e, j)
            b.apply()
    # The same samples give the same gradient up to the order of the
    # advantages' fp64 sums; Adam's steps are lr in size whatever the
    # gradient's, so other samples would move most weights by about lr.
    for x, y, w0 in zip(a.get_weights(), b.get_weights(), (pw, vw)):
        assert value_only or np.abs(y - w0).mean() >= 0.1 * HP["lr"]
        assert np.abs(x - y).mean() <= 1e-2 * HP["lr"]
    assert a.status().code == 0


@pytest.mark.parametrize("D,A,B,value_only", [
    (18, 8, 2, True), (12, 6, 63, True), (7, 3, 5000, True),
    (12, 6, 63, False), (18, 8, 257, False), (7, 3, 5000, False)])
def test_grouped_weight_gradients(D, A, B, value_only):
    """The clip is off and every advantage near 1, since a log-prob rounded
    across the clip's edge takes a sample's whole gradient with it (that is
    the forward's rounding, not the products').  Each path then stays within
    twice GRAD_TOL of the oracle, so they differ by at most four times that;
    a product left out or misplaced is off by order one."""
    torch = need_gpu()
    H, T, N = 256, 4, 2048
    pw, vw = _weights(D, H, A, seed=3)
    traj = _on_rollout_policy(_traj(8, T, N, D, A), pw, D, H, A)
    traj["adv"] = (1.0 + 0.1 * np.random.default_rng(6).normal(size=(T, N))).astype(np.float32)
    traj = _dev(torch, traj)
    if value_only:
        traj = {k: traj[k] for k in ("obs", "ret")}
    g = []
    for gemm in (False, True):
        L = _learner(D, A, H, B, "bf16", gemm_path=gemm, value_only=value_only, **COHERENT)
        L.set_weights(pw, vw)
        grad = torch.empty(L.n_policy + L.n_value, device="cuda")
        L.grads(traj, 0, 0, grad=grad)
        assert L.status().code == 0
        g.append(to_np(grad))
    for sl in (slice(0, L.n_policy), slice(L.n_policy, None)):
        scale = np.abs(g[1][sl]).max()
        if value_only and sl.start == 0:
            assert scale == 0.0 and not g[0][sl].any()
            continue
        err = np.abs(g[0][sl] - g[1][sl]).max() / scale
        print(f"[grouped D={D} B={B}] {err:.2e}")
        assert err <= 4 * GRAD_TOL["bf16"]


@pytest.mark.parametrize("D,A,B", [(18, 8, 2), (12, 6, 255), (18, 8, 257), (7, 3, 5000), (18, 8, 30011)])
def test_a_gradient_does_not_depend_on_its_launch(D, A, B):
    """The K ranges of a weight gradient are its own product's: the value network's gradient has the same bits alone
    and in one launch with the policy's."""
    torch = need_gpu()
    H, T, N = 256, 16, 2048
    pw, vw = _weights(D, H, A, seed=3)
    traj = _dev(torch, _traj(8, T, N, D, A))
    g = []
    for value_only in (False, True):
        L = _learner(D, A, H, B, "bf16", value_only=value_only)
        L.set_weights(pw, vw)
        grad = torch.empty(L.n_policy + L.n_value, device="cuda")
        L.grads({k: traj[k] for k in ("obs", "ret")} if value_only else traj, 0, 0, grad=grad)
        assert L.status().code == 0
        g.append(to_np(grad)[L.n_policy:])
    assert np.abs(g[0]).max() > 0 and np.array_equal(g[0], g[1])


@pytest.mark.parametrize("precision,H,B,mb", [
    ("fp32", 32, 255, 4), ("fp32", 32, 257, 6), ("tf32", 64, 2049, 4), ("bf16", 256, 4097, 4), ("bf16", 256, 700, 5)])
def test_prepared_advantage_sums_are_the_minibatch_calls(precision, H, B, mb):
    """Advantages far from zero: the variance is what is left of sums 10^10 times as large, so that it shows any other
    order of the fp64 additions.  The weights are the same bits as after the per-minibatch calls."""
    torch = need_gpu()
    D, A, T, N = 18, 8, 8, 2053
    pw, vw = _weights(D, H, A, seed=5)
    traj = _on_rollout_policy(_traj(6, T, N, D, A), pw, D, H, A)
    traj["adv"] = (1000.0 + 0.01 * traj["adv"]).astype(np.float32)
    traj = _dev(torch, traj)
    a, b = (_learner(D, A, H, B, precision) for _ in range(2))
    for q in (a, b):
        q.set_weights(pw, vw)
    a.update(traj, 2, mb)
    for e in range(2):
        for j in range(mb):
            b.grads(traj, e, j)
            b.apply()
    for x, y in zip(a.get_weights(), b.get_weights()):
        assert np.array_equal(x, y)

"""The exact-fp32 network kernels (csrc/k_fp32.cu) at the edges of their tiles.

A rollout's tile holds 8, 16 or 32 envs depending on the batch (8, 16 and 32
rows per SM are the lines), with sums in one order whatever the tile: envs of a
small batch must equal the same envs of a large one bit for bit, and the
oracle's trajectory within the fp32 tolerance of the other rollout tests
(1e-5 relative of max(|x|, 1): 32-bit rounding over a few steps).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEYS = ("obs", "act", "logp", "value", "rew", "done")


def make(auvenv, W, model, hidden, n, heads):
    w = W.workload("tiny_64" if model == "fossen" else "paper_tiny", n_envs=n, hidden=hidden, has_value=1,
                   policy_out=heads, substeps=2, episode_len=3, dr_enable=1, current_range=0.2)
    pw, vw = W.policy_weights(w, 0.1), W.value_weights(w, 0.1)
    env = auvenv.Env(w)
    env.set_weights(pw, vw)
    env.reset()
    return w, pw, vw, env


@pytest.mark.parametrize("model,heads", [("fossen", 8), ("fossen", 16), ("paper", 6), ("paper", 12)])
@pytest.mark.parametrize("hidden", [64, 256])
def test_rollout_tiles(model, heads, hidden):
    from oracle import oracle as O
    from paper_2512_13359_gb300 import auvenv
    from paper_2512_13359_gb300 import workloads as W
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    T, ref = 4, None
    for n in (1, 9, 8 * sms + 1, 16 * sms + 1, 32 * sms + 1):   # one lane; ragged 8-, 16- and 32-tiles, one and two CTAs an SM
        w, pw, vw, env = make(auvenv, W, model, hidden, n, heads)
        traj = env.alloc_traj(T)
        env.rollout(T, traj)
        assert env.status().code == 0
        got = {k: traj[k].cpu().numpy() for k in KEYS}
        got["state"] = env.state.cpu().numpy()
        ids = np.unique([0, n // 2, n - 1])
        m = O.paper_model(w) if model == "paper" else O.model(w)
        b = (O.PaperBatch if model == "paper" else O.Batch)(ids)
        (O.paper_reset if model == "paper" else O.reset)(m, b)
        out = (O.paper_rollout if model == "paper" else O.rollout)(m, b, pw, vw, 0, T)
        assert np.array_equal(got["done"][:, ids], out["done"])
        for k in ("obs", "act", "logp", "value", "rew"):
            err = np.abs(got[k][..., ids] - out[k]) / np.maximum(np.abs(out[k]), 1.0)
            assert err.max() <= 1e-5, (n, k, err.max())
        if ref is not None:
            for k, v in ref.items():
                assert np.array_equal(v, got[k][..., :v.shape[-1]]), (n, k)
        ref = got


@pytest.mark.parametrize("model,heads", [("fossen", 16), ("paper", 6)])
@pytest.mark.parametrize("hidden", [64, 256])
def test_rows_tiles(model, heads, hidden):
    """env_policy_forward and env_value, 1 row to several tiles per CTA, against float64 (1e-5 of the
    output's scale: 32-bit sums of 256 products)."""
    from paper_2512_13359_gb300 import auvenv
    from paper_2512_13359_gb300 import workloads as W
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    D = W.OBS_DIM if model == "fossen" else W.PAPER_OBS_DIM

    def net(flat, out, x):
        H, p, o = hidden, [], 0
        for s in ((H, D), (H,), (H, H), (H,), (out, H), (out,)):
            p.append(flat[o:o + int(np.prod(s))].astype(np.float64).reshape(s))
            o += int(np.prod(s))
        h = np.tanh(np.tanh(x @ p[0].T + p[1]) @ p[2].T + p[3])
        return h @ p[4].T + p[5]

    for n in (1, 8 * sms, 8 * sms + 1, 64 * sms + 33):
        w, pw, vw, env = make(auvenv, W, model, hidden, n, heads)
        x = W.random_observations(n, n, D)
        xd = torch.from_numpy(x).cuda()
        head, value = torch.empty(n, heads, device="cuda"), torch.empty(n, device="cuda")
        env.policy_forward(xd, head, value)
        only = torch.empty(n, heads, device="cuda")
        env.policy_forward(xd, only)
        v2 = torch.empty(2, n, device="cuda")
        env.value(torch.stack([xd.T.contiguous(), xd.T.contiguous()]), v2)
        assert env.status().code == 0
        assert torch.equal(head, only) and torch.equal(v2[0], value) and torch.equal(v2[1], value)
        for got, want in ((head, net(pw, heads, x)), (value[:, None], net(vw, 1, x))):
            assert np.abs(got.cpu().numpy() - want).max() <= 1e-5 * max(1.0, np.abs(want).max())

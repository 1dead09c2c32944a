"""The replay buffer's insert kernel (csrc/rbuf.cu) at its tile edges: inserts of more steps than a block takes (8), env
counts around its 64 (32 for wide observations) and spans that wrap inside a tile.  Copies: bit-exact against the
oracle's ring."""
import numpy as np
import pytest

from parity_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,A", [(18, 8), (12, 6), (37, 5), (1, 4), (130, 3), (256, 64)])
@pytest.mark.parametrize("N", [1, 31, 33, 64, 65, 130])
def test_insert_and_sample(D, A, N):
    torch = need_gpu()
    from oracle import offpolicy_oracle as F
    from paper_2512_13359_gb300 import auvenv
    C = 19 * N + 3
    rb, ref = auvenv.ReplayBuffer(D, A, C), F.ReplayBuffer(D, A, C)
    rng = np.random.default_rng(N * 100 + D)
    for T in (1, 8, 9, 17):   # one step, a whole block, one more, three blocks (wrapping the ring)
        x = (rng.normal(size=(T, D, N)), rng.normal(size=(T, A, N)), rng.normal(size=(T, N)),
             rng.random((T, N)) < 0.2, rng.normal(size=(D, N)))
        x = [v.astype(np.uint8 if v.dtype == bool else np.float32) for v in x]
        rb.insert(*(torch.from_numpy(v).cuda() for v in x))
        ref.insert(*x)
        assert rb.size == (ref.size, ref.head)
    B = 4 * C   # every slot is drawn (but for chance)
    out, want = rb.sample(B, seed=5, draw=1, with_idx=True), ref.sample(5, 1, B)
    assert np.array_equal(out["idx"].cpu().numpy(), want["idx"].astype(np.int32))
    for k in ("obs", "act", "rew", "next_obs", "done"):
        assert np.array_equal(out[k].cpu().numpy(), want[k]), k


@pytest.mark.parametrize("D,A", [(18, 8), (130, 3)])
@pytest.mark.parametrize("N,T,C", [
    (65, 3, 64), (130, 1, 129), (1, 40, 7),      # C one below a multiple of N; a tile of one env
    (200, 2, 5), (33, 17, 1),                    # C far below a tile
    (100, 9, 450), (64, 24, 64 * 16 + 10),       # the first stored env in mid-step; whole blocks of steps dropped
])
def test_insert_more_than_the_ring_holds(D, A, N, T, C):
    """Several transitions of one insert share a slot: the newest of them stays, whole."""
    torch = need_gpu()
    from oracle import offpolicy_oracle as F
    from paper_2512_13359_gb300 import auvenv
    rb, ref = auvenv.ReplayBuffer(D, A, C), F.ReplayBuffer(D, A, C)
    rng = np.random.default_rng(N + T)
    for steps in (1, T, T):   # the first moves head off slot 0
        x = (rng.normal(size=(steps, D, N)), rng.normal(size=(steps, A, N)), rng.normal(size=(steps, N)),
             rng.random((steps, N)) < 0.2, rng.normal(size=(D, N)))
        x = [v.astype(np.uint8 if v.dtype == bool else np.float32) for v in x]
        rb.insert(*(torch.from_numpy(v).cuda() for v in x))
        ref.insert(*x)
        assert rb.size == (ref.size, ref.head)
        B = 8 * C + 64   # every slot is drawn (but for chance)
        out, want = rb.sample(B, seed=7, draw=steps, with_idx=True), ref.sample(7, steps, B)
        for k in ("obs", "act", "rew", "next_obs", "done"):
            assert np.array_equal(out[k].cpu().numpy(), want[k]), k


@pytest.mark.parametrize("N,T", [(40000, 17), (20001, 9), (20001, 8), (10001, 17), (5000, 17), (2500, 17)])
@pytest.mark.parametrize("over", [False, True])
def test_steps_per_block(N, T, over):
    """Eight, four, two or one steps to a block by the size of the grid, a last block of fewer; a ring that wraps, and one
    that holds less than the insert.  Whole arrays against the definition."""
    torch = need_gpu()
    from paper_2512_13359_gb300 import auvenv
    D, A, rows = 18, 8, T * N
    C = rows - N // 2 - 3 if over else rows + N // 3 + 1
    rb = auvenv.ReplayBuffer(D, A, C)
    rng = np.random.default_rng(N + T)
    ref = {}
    head = 0
    for steps in (1, T):
        x = (rng.random((steps, D, N)), rng.random((steps, A, N)), rng.random((steps, N)), rng.random((steps, N)) < 0.2,
             rng.random((D, N)))
        x = [v.astype(np.uint8 if v.dtype == bool else np.float32) for v in x]
        rb.insert(*(torch.from_numpy(v).cuda() for v in x))
        slots = (head + np.arange(steps * N)) % C
        flat = dict(obs=x[0].transpose(0, 2, 1).reshape(-1, D), act=x[1].transpose(0, 2, 1).reshape(-1, A), rew=x[2].ravel(),
                    next_obs=np.concatenate([x[0][1:], x[4][None]]).transpose(0, 2, 1).reshape(-1, D), done=x[3].ravel())
        for k, v in flat.items():
            ref.setdefault(k, np.zeros((C,) + v.shape[1:], v.dtype))
            ref[k][slots[-C:]] = v[-C:]
        head = (head + steps * N) % C
    out = rb.sample(4 * C, seed=3, draw=1, with_idx=True)
    idx = out["idx"].cpu().numpy().view(np.uint32)
    assert np.unique(idx).size > 0.97 * C   # (but for chance, 1 - e^-4 of the slots are drawn)
    for k, v in ref.items():
        assert np.array_equal(out[k].cpu().numpy(), v[idx]), k

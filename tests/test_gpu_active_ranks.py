"""Active lists with cell grouping: the set, its groups and its interactions at the edges of the mask words (32
particles) and of the compaction's tiles (8192), twice in a row (the masks are left clear for the next list)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_07279_gb300 import build
    from paper_1610_07279_gb300 import gothic as g
    build.build()
    g.load()
    return torch, g


@pytest.mark.parametrize("n", [1, 31, 32, 33, 8193, 32767, 32768, 32769, 70001])
def test_lists_match_the_oracle(env, n):
    torch, g = env
    import oracle as O
    rng = np.random.default_rng(n)
    pos = (rng.standard_normal((n, 3)) * rng.uniform(0.05, 2.0, (n, 1))).astype(np.float32)
    mass = rng.uniform(0.5, 1.5, n).astype(np.float32) / n
    prm = g.gt_default_params()
    prm.mac, prm.theta, prm.group_max, prm.group_mode = g.GT_MAC_OPENING_ANGLE, 1.0, 7, g.GT_GROUP_CELLS
    s = g.System(n, prm)
    s.set_state(pos.astype(np.float64), np.zeros((n, 3)), mass)
    s.build_tree()
    p4 = np.concatenate([pos, mass[:, None]], axis=1)
    key = O.keys(p4, prm.key_curve)[0]
    skey = O.sort(key)[1]
    tree = O.build_tree(skey, prm.leaf_max)

    def check(d_act, want):
        acc = torch.zeros((want.size, 4), device="cuda")
        s.accel_active(d_act, None, acc, n_active=None if d_act is None else d_act.numel())
        s.sync()
        assert np.array_equal(s.get_active(), want)
        st = s.stats()
        assert st["n_active"] == want.size
        assert st["n_groups"] == len(O.group_starts(tree, n, want, prm.group_max, prm.group_mode)) - 1
        return acc.cpu().numpy()

    every = np.arange(n, dtype=np.uint32)
    whole = check(None, every)
    if n > 2:
        some = [np.unique(np.r_[0, n - 1, rng.integers(0, n, max(n // 50, 1))]), every[: n - 1], every[-1:], every]
    else:
        some = [every]
    for want in some + [some[0]]:
        want = want.astype(np.uint32)
        got = check(torch.from_numpy(want.astype(np.int32)).cuda(), want)
        assert np.all(np.isfinite(got)) and np.all(got[:, :3].any(axis=1) | (n == 1))
        if want.size == n:  # the same groups as without a list
            assert np.array_equal(got, whole)
    s.close()

"""Which groups gt_start walks a second time: those with a force near a level's threshold get other roundings than
gt_accel_active gives them, all others the same bits."""
import numpy as np
import pytest

from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu


def _distance(a, c):
    """|a|^2 / c^2 relative to the nearest power of 16, less 1."""
    x = (a.astype(np.float64) ** 2).sum(axis=1) / c ** 2
    return np.abs(x / 16.0 ** np.round(np.log2(x) / 4.0) - 1.0)


@pytest.mark.parametrize("n,gmax,leaf", [(9000, 48, 16), (3 * 3648 * 8, 8, 16)])  # teams of warps; single ones
@pytest.mark.parametrize("side", [-0.75, 0.5])  # of the window, below (the further half of it) and above the threshold
def test_groups_near_a_threshold_are_walked_again(env, n, gmax, leaf, side):  # noqa: F811
    torch, g, O = env
    rng = np.random.default_rng(n)
    pos = (rng.standard_normal((n, 3)) * rng.uniform(0.05, 2.0, (n, 1))).astype(np.float32).astype(np.float64)
    mass = rng.uniform(0.5, 1.5, n).astype(np.float32) / n
    aold = np.full(n, 1.0, np.float32)
    prm = g.gt_default_params()
    prm.eps, prm.group_max, prm.leaf_max, prm.group_mode = 0.02, gmax, leaf, g.GT_GROUP_RUNS
    eps = float(np.float32(0.02))

    s = g.System(n, prm)
    s.set_state(pos, np.zeros_like(pos), mass)
    s.build_tree()
    out = torch.zeros((n, 4), device="cuda")
    s.accel_active(None, torch.from_numpy(aold).cuda(), out)
    s.sync()
    s.close()
    ref = out.cpu().numpy()
    again = 0
    for i in rng.choice(n, 3, replace=False):
        x = 1.0 + side * 2.0 ** -17  # of particle i
        c = np.linalg.norm(ref[i, :3].astype(np.float64)) / np.sqrt(x)
        prm.eta = c / (2.0 * eps)
        s = g.System(n, prm)
        s.set_state(pos, np.zeros_like(pos), mass)
        s.start(aold)
        got = s.get_state()["acc"]
        s.close()
        differ = (got.view(np.uint32) != ref.view(np.uint32)).any(axis=1)
        d = _distance(ref[:, :3], c) * 2.0 ** 17
        group = np.arange(n) // gmax
        near, unsure = np.unique(group[d < 0.9]), np.unique(group[(d >= 0.9) & (d < 1.1)])
        assert group[i] in near
        assert set(np.unique(group[differ])) <= set(near) | set(unsure)
        again += differ[group == group[i]].sum()
    assert again > 0  # (sums of hundreds of terms in another order: equal in all bits for hardly any member)

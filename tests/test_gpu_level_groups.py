"""Groups whose forces lie at a block-step level's threshold are walked a second time, in a fixed order of
summation: the same interactions, the same forces up to the rounding of FP32 sums."""
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


# Two sums of at most n FP32 terms in different orders: each is within ~ sqrt(n) 2^-24 of the exact one (random
# roundings; n = 12000 terms at most here, and the packed halves and lanes split them), taken four times for the
# worst of a few thousand particles, against the sum of the terms' magnitudes, here a few |a| at most.
TOL = 4 * 2 * np.sqrt(12000) * 2.0 ** -24


@pytest.mark.parametrize("n,leaf,gmax,queue,mac,S", [(9000, 16, 64, 16384, 1, 0), (9000, 1, 33, 16384, 1, 0),
                                                     (9000, 40, 20, 16384, 0, 0), (12000, 300, 64, 16384, 1, 0),
                                                     (9000, 16, 64, 4096, 2, 1), (700, 5000, 7, 8192, 0, 4)])
def test_groups_at_a_threshold(env, n, leaf, gmax, queue, mac, S):
    torch, g = env
    rng = np.random.default_rng(n + leaf)
    pos = (rng.standard_normal((n, 3)) * rng.uniform(0.05, 2.0, (n, 1))).astype(np.float32).astype(np.float64)
    if leaf == 5000:
        pos[:600] = pos[0]  # one leaf of coincident particles
    mass = rng.uniform(0.5, 1.5, n).astype(np.float32) / n
    aold = np.full(n, 1.0, np.float32)
    prm = g.gt_default_params()
    prm.eps, prm.mac, prm.group_max, prm.leaf_max, prm.walk_queue, prm.ij_share = 0.02, mac, gmax, leaf, queue, S
    prm.group_mode = g.GT_GROUP_CELLS

    def system(eta):
        prm.eta = eta
        s = g.System(n, prm)
        s.set_state(pos, np.zeros_like(pos), mass)
        return s

    s = system(0.025)
    s.build_tree()
    acc = torch.zeros((n, 4), device="cuda")
    before = s.stats()["interactions"]
    s.accel_active(None, torch.from_numpy(aold).cuda(), acc)
    s.sync()
    inter = s.stats()["interactions"] - before
    s.close()
    ref = acc.cpu().numpy().astype(np.float64)
    a = np.linalg.norm(ref[:, :3], axis=1)
    for i in rng.choice(n, 4, replace=False):  # eta for which particle i's |a| is c = 2 eta eps
        s = system(float(a[i]) / (2.0 * 0.02))
        s.start(aold)
        st = s.get_state()
        assert s.stats()["interactions"] == inter
        s.close()
        got = st["acc"].astype(np.float64)
        assert np.all(np.linalg.norm(got[:, :3] - ref[:, :3], axis=1) <= TOL * np.abs(ref[:, 3]).max() + TOL * a)
        assert np.all(np.abs(got[:, 3] - ref[:, 3]) <= TOL * np.abs(ref[:, 3]))

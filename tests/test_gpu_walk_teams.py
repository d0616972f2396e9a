"""A walk of few groups takes teams of warps, a walk of many one warp per group: the same forces bit for bit,
the same interactions and the same MAC tests."""
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


# Group sizes on both sides of 32 and of powers of two; leaves of one particle, of more than a warp, and larger
# than the list of a warp (256 entries) and of a team; the smallest queue with a breadth-first part, at which a
# team hands groups back to one warp, and one without.
@pytest.mark.parametrize("gmax,leaf,queue,mac", [(1, 16, 16384, 1), (8, 1, 16384, 1), (33, 16, 16384, 1),
                                                 (34, 8, 8192, 0), (49, 40, 16384, 2), (64, 300, 16384, 1),
                                                 (7, 5000, 8192, 0), (20, 4, 4096, 1)])
def test_teams_match_single_warps(env, gmax, leaf, queue, mac):
    torch, g = env
    parts = (300, 2000, 5000, 1, 99)  # groups per call: teams of 8, 4, 2, 8, 8
    n = sum(parts) * gmax             # all of them: single warps (more than twice the 152 x 3 x 8 warps)
    rng = np.random.default_rng(11)
    pos = (rng.standard_normal((n, 3)) * rng.uniform(0.05, 2.0, (n, 1))).astype(np.float32).astype(np.float64)
    prm = g.gt_default_params()
    prm.eps, prm.mac, prm.group_max, prm.leaf_max, prm.walk_queue = 0.02, mac, gmax, leaf, queue
    prm.group_mode = g.GT_GROUP_RUNS  # the groups of a list are the runs of its entries
    s = g.System(n, prm)
    s.set_state(pos, np.zeros_like(pos), rng.uniform(0.5, 1.5, n).astype(np.float32) / n)
    s.build_tree()
    aold = torch.rand(n, generator=torch.Generator("cuda").manual_seed(5), device="cuda") + 0.1
    whole = torch.arange(n, dtype=torch.int32, device="cuda")

    def walk(a, b):
        acc = torch.zeros((b - a, 4), device="cuda")
        before = s.stats()
        s.accel_active(whole[a:b].clone(), aold, acc)
        s.sync()
        after = s.stats()
        return acc, after["interactions"] - before["interactions"], after["mac_tests"] - before["mac_tests"]

    one, inter, tests = walk(0, n)
    got, at = [], 0
    for p in parts:
        got.append(walk(at, at + p * gmax))
        at += p * gmax
    s.close()
    assert torch.equal(torch.cat([x[0] for x in got]), one)
    assert sum(x[1] for x in got) == inter and sum(x[2] for x in got) == tests

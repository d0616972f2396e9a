"""Keys that agree in the bits that the tree sort's passes cover, in long runs: the order and tree of the oracle, bit
for bit, with the runs' lengths checked here, and times that stay near those of keys without such runs."""
import numpy as np
import pytest

from test_gpu_parity import _check_tree, _oracle_tree, _params, env  # noqa: F401

pytestmark = pytest.mark.gpu


def _build_times(torch, g, pos, fresh):
    """Median microseconds of a build, of the state as given or (not fresh) from its own key order."""
    n = len(pos)
    s = g.System(n, _params(g, 0.01, leaf_max=16, node_factor=4))
    state = (torch.from_numpy(pos).cuda(), torch.zeros((n, 3), dtype=torch.float64, device="cuda"),
             torch.full((n,), 1.0 / n, device="cuda"))
    s.set_state(*state)
    t = []
    for _ in range(13):
        if fresh:
            s.set_state(*state)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        e[0].record()
        s.build_tree()
        e[1].record()
        torch.cuda.synchronize()
        t.append(1e3 * e[0].elapsed_time(e[1]))
    s.sync()
    s.close()
    return sorted(t[3:])[5]


def _plummer(n, far, seed=3):
    rng = np.random.default_rng(seed)
    r = np.minimum((rng.uniform(1e-10, 1.0 - 1e-10, n) ** (-2.0 / 3.0) - 1.0) ** -0.5, 100.0)
    d = rng.standard_normal((n, 3))
    pos = r[:, None] * d / np.linalg.norm(d, axis=1)[:, None]
    if far:
        pos[5] = (far, 0.0, 0.0)
    return pos.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("far", [1e5, 1e6])
def test_time_of_one_blocks_sort_with_a_long_run_in_order(env, far):  # noqa: F811
    """One particle far off: nearly all keys agree in their highest 40 bits and are in order already.  A thread that
    looked along the whole run took 800 us; the rest of such a build (deep chains) 150 more than without it."""
    torch, g, O = env
    assert _build_times(torch, g, _plummer(8192, far), False) < _build_times(torch, g, _plummer(8192, 0.0), False) + 400.0

"""Keys that agree in the bits that the tree sort's passes cover: runs of every length, put in order by a thread, by
a block in shared memory and by a block through memory, in order already, and crowded into a corner of the cube (the
low passes run); keys, order and tree against the oracle, bit for bit."""
import numpy as np
import pytest

from test_gpu_parity import _check_tree, _oracle_tree, _params, env  # noqa: F401

pytestmark = pytest.mark.gpu


def _clumps(sizes, n_field, radius, seed, far=None):
    """A uniform field of n_field particles in the unit cube and clumps of the given sizes and radius in it."""
    rng = np.random.default_rng(seed)
    parts = [rng.uniform(0.0, 1.0, (n_field, 3))]
    for m in sizes:
        parts.append(rng.uniform(0.2, 0.8, 3) + radius * rng.uniform(-1.0, 1.0, (m, 3)))
    pos = np.concatenate(parts)
    if far is not None:
        pos[0] = far
    pos = pos[rng.permutation(len(pos))].astype(np.float32).astype(np.float64)
    return pos


# cells of level 16 have side 1.5e-5: clumps of radius 4e-6 lie in one or a few of them (FP32 positions near 0.5 are
# 6e-8 apart, so their particles differ below level 16)
@pytest.mark.parametrize("sizes,n_field,radius,far", [
    ((2, 3, 15, 16, 17, 18, 31, 33, 64), 500, 4e-6, None),      # around the one-thread limit of 16
    ((400, 4095, 4096, 4097), 60000, 2e-6, None),               # around a tile in shared memory
    ((20000,), 300000, 4e-6, None),                             # tile after tile through memory
    ((9000,), 200000, 1e-9, None),                              # a long run of equal keys
    ((), 30000, 0.0, (40000.0, 0.0, 0.0)),                      # all but one in a corner: crowded
    ((64,), 5000, 4e-6, (0.5, 3000.0, 0.5)),                    # near the crowding threshold
    ((), 1, 0.0, None), ((2,), 1, 0.0, None),
    # one block's sort (at most 8192 particles): runs around its limit of 32, a run that takes all passes
    ((2, 5, 31, 32, 33, 34), 8000, 4e-6, None), ((33,), 8160, 4e-6, None), ((3000,), 5192, 1e-5, None),
    ((5000,), 300, 1e-9, None), ((), 8192, 0.0, (40000.0, 0.0, 0.0)), ((), 8193, 0.0, None), ((), 255, 0.0, None),
])
def test_runs_of_equal_sorted_bits(env, sizes, n_field, radius, far):  # noqa: F811
    torch, g, O = env
    pos = _clumps(sizes, n_field, radius, 7, far)
    n = len(pos)
    mass = np.full(n, np.float32(1.0 / n))
    s = g.System(n, _params(g, 0.01, leaf_max=16, node_factor=4))
    s.set_state(pos, np.zeros_like(pos), mass)
    s.build_tree()
    t = s.get_tree()
    s.sync()
    ref = _oracle_tree(O, pos, mass, 16, cap=4 * n + 2048)
    _check_tree(t, ref)
    s.build_tree()  # from its own order
    t2 = s.get_tree()
    s.sync()
    assert np.array_equal(t2["keys"], t["keys"]) and t2["n_nodes"] == t["n_nodes"]
    s.close()

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


def _clumps(n_field, sizes, radius, seed=7):
    """A uniform field in the unit cube (both corners held) and clumps of the given sizes inside a cell of level 16."""
    rng = np.random.default_rng(seed)
    cells = rng.choice(52000 ** 2, len(sizes), replace=False)  # different ones
    parts = [rng.uniform(0.0, 1.0, (n_field, 3))]
    for m, c in zip(sizes, cells):
        centre = (np.array([c // 52000, c % 52000, rng.integers(52000)]) + 6000.5) / 65536.0
        parts.append(centre + radius * rng.uniform(-1.0, 1.0, (m, 3)))
    pos = np.concatenate(parts)
    pos[0], pos[1] = 0.0, 1.0
    return pos[rng.permutation(len(pos))].astype(np.float32).astype(np.float64)


def _runs(keys):
    return np.unique(keys >> np.uint64(15), return_counts=True)[1]


def _whole(keys):
    """Whether the low passes run: the library's rule."""
    n, longest, run = len(keys), len(keys), float(len(keys))
    for p in range(2, 8):
        c = np.bincount(((keys >> np.uint64(8 * p - 1)) & np.uint64(255)).astype(np.int64), minlength=256)
        longest, run = min(longest, c.max()), run * ((c / n) ** 2).sum()
    return longest / n >= 0.01 or run >= 2.0


# (cells of level 16 have side 1.5e-5; FP32 positions near 0.5 are 6e-8 apart, so a clump's particles differ below level
# 16; one of radius 0 is a run of equal keys)
CASES = [
    (9000, (2, 3, 15, 16, 17, 18, 31, 33, 64), 4e-6),       # around the limit of one thread
    (60000, (17,) * 2000, 4e-6),                             # more than 256 runs to a block
    (4000, (17, 40, 3) * 300, 4e-6), (500, (20,) * 3000, 4e-6),
    (900000, (2047, 2048, 2049, 4000), 4e-6),                # around a tile of beginnings
    (2600000, (4095, 4096, 4097, 9000, 12000), 4e-6),       # around a block's shared memory, and through memory
    (1900000, (4095, 4096, 4097, 9000), 0.0), (60000, (300, 17), 0.0),
    (1900000, (5000, 18, 5000, 30, 9000) * 3, 5e-7),         # long runs among short ones, many keys equal
]


@pytest.mark.parametrize("n_field,sizes,radius", CASES)
def test_runs_that_the_passes_leave(env, n_field, sizes, radius):  # noqa: F811
    torch, g, O = env
    pos = _clumps(n_field, sizes, radius)
    n = len(pos)
    mass = np.full(n, np.float32(1.0 / n))
    s = g.System(n, _params(g, 0.01, leaf_max=16, node_factor=4))
    s.set_state(pos, np.zeros_like(pos), mass)
    s.build_tree()
    t = s.get_tree()
    s.sync()
    ref = _oracle_tree(O, pos, mass, 16, cap=4 * n + 2048)
    got = np.sort(_runs(ref["skey"]))[::-1]
    assert n > 8192 and not _whole(ref["skey"])
    assert np.all(got[: len(sizes)] >= np.sort(sizes)[::-1])  # every clump is a run
    assert got[0] <= max(sizes) + 3                           # (and a particle of the field may lie in its cell)
    _check_tree(t, ref)
    s.build_tree()  # from its own order: all runs are in order already
    t2 = s.get_tree()
    s.sync()
    assert np.array_equal(t2["keys"], t["keys"]) and t2["n_nodes"] == t["n_nodes"]
    s.close()


@pytest.mark.parametrize("n,far,whole", [(1 << 17, 5000.0, False), (1 << 17, 10000.0, True), (20000, 11000.0, False),
                                         (20000, 40000.0, True)])
def test_crowded_by_one_particle_far_off(env, n, far, whole):  # noqa: F811
    torch, g, O = env
    pos = _plummer(n, far)
    mass = np.full(n, np.float32(1.0 / n))
    s = g.System(n, _params(g, 0.01, leaf_max=16, node_factor=4))
    s.set_state(pos, np.zeros_like(pos), mass)
    s.build_tree()
    t = s.get_tree()
    s.sync()
    s.close()
    ref = _oracle_tree(O, pos, mass, 16, cap=4 * n + 2048)
    assert _whole(ref["skey"]) == whole and _runs(ref["skey"]).max() > 16
    _check_tree(t, ref)


def test_members_of_a_batch(env):  # noqa: F811
    torch, g, O = env
    cases = [(9000, (17,) * 300, 4e-6), (200000, (900, 20, 800), 4e-6), (9000, (40, 16, 15), 0.0)] * 3
    state = [_clumps(*c, seed=k) for k, c in enumerate(cases)]
    prm = _params(g, 0.01, leaf_max=16, node_factor=4)
    b = g.Batch([len(p) for p in state], [prm] * len(state))
    for m, p in zip(b.systems, state):
        m.set_state(p, np.zeros_like(p), np.full(len(p), 1.0 / len(p), np.float32))
    b.accel()
    b.sync()
    for m, p in zip(b.systems, state):
        ref = _oracle_tree(O, p, np.full(len(p), np.float32(1.0 / len(p))), 16, cap=4 * len(p) + 2048)
        assert not _whole(ref["skey"])
        t = m.get_tree()
        assert np.array_equal(t["keys"], ref["skey"]) and np.array_equal(t["order"], ref["order"])
    b.close()


@pytest.mark.parametrize("far", [2500.0, 5000.0])
def test_time_with_one_particle_far_off(env, far):  # noqa: F811
    """2^22 particles: 1.03 of the time without it; with a block for every run of more than 16 keys it was 2.7."""
    torch, g, O = env
    n = 1 << 22
    assert _build_times(torch, g, _plummer(n, far), True) < 1.5 * _build_times(torch, g, _plummer(n, 0.0), True)


def test_time_with_a_tight_clump(env):  # noqa: F811
    """5 % of 2^22 particles in one cell of level 16: they were sorted by one block, 1.7 of the time without them."""
    torch, g, O = env
    n = 1 << 22
    assert (_build_times(torch, g, _clumps(n - n // 20, (n // 20,), 4e-6), True)
            < 1.3 * _build_times(torch, g, _clumps(n, (), 0.0), True))

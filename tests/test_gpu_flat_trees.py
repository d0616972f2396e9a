"""Systems whose cells have few children (sheets, lines, clumps on a line): single warps pack their batches, teams
don't; the same forces bit for bit, the oracle's interactions, alone and among solid members of a batch, and no
slower than a solid body."""
import numpy as np
import pytest

from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu


def _positions(kind, n, seed):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, 1.0, (n, 3))
    if kind == "sheet":
        pos[:, 2] = 0.5
    elif kind == "line":
        pos[:, 1:] = 0.5
    elif kind == "chains":  # pairs so close that their cells are chains of one child each
        pos[:, 1:] = 0.5
        pos[1::2] = pos[: 2 * (n // 2) : 2] + 1e-6
    return pos.astype(np.float32).astype(np.float64)


def _params(g, **kw):
    prm = g.gt_default_params()
    prm.eps, prm.node_factor, prm.walk_queue = 0.01, 16, 16384
    for k, v in kw.items():
        setattr(prm, k, v)
    return prm


@pytest.mark.parametrize("kind", ["sheet", "line", "chains", "solid"])
@pytest.mark.parametrize("gmax,leaf,mac", [(8, 1, 1), (33, 16, 1), (5, 3, 0), (16, 300, 2)])
def test_packed_batches_match_teams(env, kind, gmax, leaf, mac):  # noqa: F811
    torch, g, O = env
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    warps = 24 * nsm
    parts = (warps // 8 - 3, warps // 3 - 5, 1, 99)  # groups per call: teams of 8, 4, 8, 8
    whole_groups = max(sum(parts), 2 * warps + 7)     # single warps, of a solid body too
    n = whole_groups * gmax
    pos = _positions(kind, n, gmax)
    s = g.System(n, _params(g, group_mode=g.GT_GROUP_RUNS, group_max=gmax, leaf_max=leaf, mac=mac))
    s.set_state(pos, np.zeros_like(pos), np.random.default_rng(1).uniform(0.5, 1.5, n).astype(np.float32) / n)
    s.build_tree()
    aold = torch.rand(n, generator=torch.Generator("cuda").manual_seed(5), device="cuda") + 0.1
    every = torch.arange(n, dtype=torch.int32, device="cuda")

    def walk(a, b):
        acc = torch.zeros((b - a, 4), device="cuda")
        before = s.stats()
        s.accel_active(every[a:b].clone(), aold, acc)
        s.sync()
        after = s.stats()
        return acc, after["interactions"] - before["interactions"], after["mac_tests"] - before["mac_tests"]

    one = walk(0, n)
    at = [0]
    got = []
    for p in parts + (whole_groups - sum(parts),):
        got.append(walk(at[-1], at[-1] + p * gmax))
        at.append(at[-1] + p * gmax)
    s.close()
    assert torch.equal(torch.cat([x[0] for x in got]), one[0])
    assert sum(x[1] for x in got) == one[1] and sum(x[2] for x in got) == one[2]


@pytest.mark.parametrize("kind,n,leaf", [("sheet", 20000, 16), ("line", 9000, 4), ("chains", 3000, 2)])
def test_forces_against_the_oracle(env, kind, n, leaf):  # noqa: F811
    torch, g, O = env
    pos = _positions(kind, n, 3)
    mass = np.full(n, np.float32(1.0 / n))
    prm = _params(g, group_mode=g.GT_GROUP_CELLS, leaf_max=leaf)
    s = g.System(n, prm)
    s.set_state(pos, np.zeros_like(pos), mass)
    s.build_tree()
    p4 = np.concatenate([pos, mass[:, None]], axis=1).astype(np.float32)
    oprm = O.Params(eps=O.f32(prm.eps), leaf_max=leaf, group_max=prm.group_max)
    aold = O.bootstrap_aold(p4, oprm)
    ref = O.tree_force(p4, oprm, aold=aold)
    acc = torch.zeros((n, 4), device="cuda")
    s.accel_active(None, torch.from_numpy(aold[ref["order"]]).cuda(), acc)
    s.sync()
    assert s.stats()["interactions"] == int(ref["inter"].sum())
    s.close()
    a, r = acc.cpu().numpy().astype(np.float64), ref["acc"]
    # FP32 sums of up to N terms: ~ sqrt(N) 2^-24 of the terms' magnitudes (random roundings), times 4 for the worst of
    # many and 2 for the packed halves; a term is at most |its potential| / (2 eps)
    tol = 8.0 * np.sqrt(ref["inter"].max()) * 2.0 ** -24
    assert np.all(np.linalg.norm(a[:, :3] - r[:, :3], axis=1) <= tol * np.abs(r[:, 3]) / (2.0 * prm.eps))
    assert np.all(np.abs(a[:, 3] - r[:, 3]) <= tol * np.abs(r[:, 3]))


def test_members_of_a_batch(env):  # noqa: F811
    torch, g, O = env
    kinds = ["sheet", "solid", "line", "solid", "chains", "sheet", "line", "solid"] * 2
    ns = [1500 + 701 * k for k in range(len(kinds))]
    prm = _params(g, leaf_max=8, group_mode=g.GT_GROUP_CELLS)
    b = g.Batch(ns, [prm] * len(ns))
    state = [(_positions(k, n, n), np.zeros((n, 3)), np.full(n, 1.0 / n, np.float32)) for k, n in zip(kinds, ns)]
    for m, st in zip(b.systems, state):
        m.set_state(*st)
    b.accel(bootstrap=True)
    b.sync()
    for k, n in enumerate(ns):
        acc, ids = b.get_acc(k)
        one = g.System(n, prm)
        one.set_state(*state[k])
        one.build_tree()
        out = torch.zeros((n, 4), device="cuda")
        one.accel_active(None, torch.from_numpy(b.systems[k].get_state()["aold"]).cuda(), out)
        one.sync()
        assert np.array_equal(acc[:n].view(np.uint32), out.cpu().numpy().view(np.uint32)), (k, kinds[k])
        one.close()
    b.close()


def test_a_line_is_walked_faster_than_a_solid_body(env):  # noqa: F811
    """2^18 particles, leaves of 4: a line 0.51 of a cube's time with packed batches, 0.87 without."""
    torch, g, O = env
    n = 1 << 18
    times = {}
    for kind in ("line", "solid"):
        pos = _positions(kind, n, 1)
        s = g.System(n, _params(g, leaf_max=4, group_mode=g.GT_GROUP_CELLS))
        s.set_state(pos, np.zeros_like(pos), np.full(n, 1.0 / n, np.float32))
        s.build_tree()
        acc, aold, t = torch.zeros((n, 4), device="cuda"), torch.ones(n, device="cuda"), []
        for _ in range(12):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            s.accel_active(None, aold, acc)
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]))
        times[kind] = sorted(t[2:])[5]
        s.sync()
        s.close()
    assert times["line"] < 0.7 * times["solid"], times

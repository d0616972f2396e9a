"""Members of a batch and requests of a server share their launches: the same results, bit for bit, as systems of
their own, for sizes on both sides of the one-block sort (8192), one particle, mixed leaf sizes, key curves and
groupings, and a member that has launches of its own (leaves above 64)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = (1, 33, 8192, 8193, 20011)


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


def _system(g, n, seed, crowded=False, **kw):
    rng = np.random.default_rng(seed)
    pos = rng.standard_normal((n, 3)) * rng.uniform(0.05, 2.0, (n, 1))
    if crowded:  # keys that share their highest digits: every digit is sorted
        pos[: n - 1] = 100.0 + 1e-4 * pos[: n - 1]
    prm = g.gt_default_params()
    prm.eps, prm.levels, prm.rebuild_every, prm.walk_queue = 0.02, 5, 2, 8192
    for k, v in kw.items():
        setattr(prm, k, v)
    return dict(n=n, pos=pos, vel=0.1 * rng.standard_normal((n, 3)), prm=prm,
                mass=rng.uniform(0.5, 1.5, n).astype(np.float32) / n)


def _mix(g):
    cells, runs = g.GT_GROUP_CELLS, g.GT_GROUP_RUNS
    kw = [dict(leaf_max=16, group_mode=cells), dict(leaf_max=16, group_mode=runs), dict(leaf_max=7, group_mode=cells),
          dict(leaf_max=32, group_mode=runs, key_curve=g.GT_KEY_HILBERT), dict(leaf_max=16, group_mode=cells, group_max=50)]
    out = [_system(g, n, 3 + n, **k) for n, k in zip(SIZES, kw)]
    out.append(_system(g, 9001, 5, leaf_max=100, group_mode=cells))
    out.append(_system(g, 9000, 6, crowded=True, group_mode=cells))
    return out


# the small ones alone: one block sorts each; with the others: their sort passes
@pytest.mark.parametrize("which", [(0, 1, 2), (0, 1, 2, 3, 4, 5, 6), (4,), (5,)])
def test_batch_members(env, which):
    torch, g = env
    sys = [_mix(g)[k] for k in which] * -(-8 // len(which))  # eight at least share launches
    b = g.Batch([s["n"] for s in sys], [s["prm"] for s in sys])
    for m, s in zip(b.systems, sys):
        m.set_state(s["pos"], s["vel"], s["mass"])

    def check():
        b.sync()
        for k, s in enumerate(sys):
            acc, ids = b.get_acc(k)
            one = g.System(s["n"], s["prm"])
            one.set_state(s["pos"], s["vel"], s["mass"])
            one.build_tree()
            out = torch.zeros((s["n"], 4), device="cuda")
            one.accel_active(None, torch.from_numpy(b.systems[k].get_state()["aold"]).cuda(), out)
            one.sync()
            assert np.array_equal(ids[: s["n"]], one.get_state()["id"]), k
            assert np.array_equal(acc[: s["n"]].view(np.uint32), out.cpu().numpy().view(np.uint32)), k
            one.close()

    b.accel(bootstrap=True)
    check()
    b.capture()
    b.launch()
    b.launch()
    check()
    b.set_knobs(8, 20, 0)  # other trees and groups: a new table
    for s in sys:
        s["prm"].leaf_max, s["prm"].group_max = 8, 20
    b.accel()
    check()
    b.close()


def test_server_requests(env):
    torch, g = env
    sys, nsteps = _mix(g), 5
    srv = g.Server(64 << 30, max_slots=len(sys), walk_queue=8192)
    todo = {srv.submit(s["pos"], s["vel"], s["mass"], s["prm"], nsteps): s for s in sys}
    while todo:
        for t in list(todo):
            s = todo[t]
            pos, vel = np.zeros((s["n"], 3)), np.zeros((s["n"], 3))
            if not srv.poll(t, pos, vel):
                continue
            del todo[t]
            one = g.System(s["n"], s["prm"])
            one.set_state(s["pos"], s["vel"], s["mass"])
            one.start()
            for _ in range(nsteps):
                one.block_step()
            ref = one.get_state()
            one.close()
            order = ref["id"].astype(np.int64)
            assert np.array_equal(pos[order], ref["pos"]) and np.array_equal(vel[order], ref["vel"]), s["n"]
    srv.close()

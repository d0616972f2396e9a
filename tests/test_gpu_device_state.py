"""State loaded from and read into device arrays (in place), host arrays and unaligned device arrays (through the
system's scratch) is the same bit for bit."""
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


@pytest.mark.parametrize("n", [1, 2, 255, 256, 1001])
def test_device_host_and_unaligned_arrays_agree(env, n):
    torch, g = env
    rng = np.random.default_rng(n)
    pos, vel = rng.standard_normal((n, 3)), rng.standard_normal((n, 3))
    arrays = {"pos": pos, "vel": vel, "mass": rng.uniform(0.1, 1.0, n).astype(np.float32),
              "level": rng.integers(0, 8, n).astype(np.uint8), "t0": np.zeros(n, np.int64),
              "aold": rng.uniform(0.1, 1.0, n).astype(np.float32), "acc": rng.standard_normal((n, 4)).astype(np.float32)}
    out_like = {**arrays, "id": np.zeros(n, np.uint32)}

    def place(a, how):
        if how == "host":
            return a.copy()
        raw = np.frombuffer(a.tobytes(), np.uint8)
        t = torch.zeros(raw.size + 16, dtype=torch.uint8, device="cuda")
        off = 0 if how == "device" else 1 if a.dtype == np.uint8 else a.dtype.itemsize // 2
        t = t[off:off + raw.size]
        t.copy_(torch.from_numpy(raw.copy()).cuda())
        return t

    got = []
    for how in ("host", "device", "unaligned"):
        prm = g.gt_default_params()
        prm.rebuild_every = 2
        s = g.System(n, prm)
        a = {k: place(v, how) for k, v in arrays.items()}
        s.set_state(a["pos"], a["vel"], a["mass"])
        s.set_integrator_state(a["level"], a["t0"], a["aold"], a["acc"], 0.25, 0)
        s.build_tree()
        out = s.get_state({k: place(np.zeros_like(v), how) for k, v in out_like.items()})
        got.append({k: v.tobytes() if how == "host" else v.cpu().numpy().tobytes() for k, v in out.items()})
        s.close()
    assert got[0] == got[1] == got[2]

"""Kernels that are set up while the one before them still runs see all that it wrote: builds, sorts and walks back to
back on one stream equal those with a wait after each."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7, 8192, 8193, 300001])
def test_back_to_back(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_07279_gb300 import build
    from paper_1610_07279_gb300 import gothic as g
    build.build()
    g.load()
    rng = np.random.default_rng(n)
    sets = [(rng.standard_normal((n, 3)) * rng.uniform(0.05, 2.0, (n, 1))) for _ in range(3)]
    mass = np.full(n, 1.0 / n, np.float32)
    dev = [(torch.from_numpy(p).cuda(), torch.zeros((n, 3), dtype=torch.float64, device="cuda"),
            torch.from_numpy(mass).cuda()) for p in sets]
    aold = torch.ones(n, device="cuda")
    prm = g.gt_default_params()
    prm.eps = 0.02
    s = g.System(n, prm)
    out = [torch.zeros((n, 4), device="cuda") for _ in sets]

    def force(k, wait):
        s.set_state(*dev[k])
        s.build_tree()
        if wait:
            torch.cuda.synchronize()
        s.accel_active(None, aold, out[k])
        if wait:
            torch.cuda.synchronize()

    ref = []
    for k in range(3):
        force(k, True)
        ref.append(out[k].clone())
    for _ in range(5):
        for o in out:
            o.zero_()
        for k in range(3):
            force(k, False)
        s.sync()
        for k in range(3):
            assert torch.equal(out[k], ref[k]), k
    s.close()

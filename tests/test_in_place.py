"""Arrays that a kernel takes in place lie inside their allocation: the rule (csrc/in_place.h) on the host, and on the
GPU that arrays which end where their allocation ends are taken in place (fewer launches), with the same results."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1610_07279_gb300", "csrc")


def test_ranges(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "in_place_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, os.path.join(HERE, "in_place_check.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.gpu
def test_arrays_at_the_end_of_their_allocation():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_07279_gb300 import build
    from paper_1610_07279_gb300 import gothic as g
    build.build()
    g.load()
    n = 1 << 20  # 24 MiB: an allocation of its own, a whole number of the allocator's 2 MiB
    rng = np.random.default_rng(2)
    host = (rng.standard_normal((n, 3)), rng.standard_normal((n, 3)), rng.uniform(0.5, 1.5, n).astype(np.float32))
    torch.cuda.empty_cache()
    dev = [torch.from_numpy(a).cuda() for a in host]
    prm = g.gt_default_params()
    prm.eps = 0.02
    out = []
    for state in (host, dev):
        s = g.System(n, prm)
        before = g.gt_kernel_launches()
        s.set_state(*state)
        launches = g.gt_kernel_launches() - before
        s.sync()
        out.append((launches, s.get_state()))
        s.close()
    assert out[1][0] == 1 < out[0][0]
    for f in ("pos", "vel", "mass"):
        assert np.array_equal(out[0][1][f], out[1][1][f]), f

"""The bit masks behind active sets and groups after an error was reported: a call that latched one may have left bits
in them.  Bits are set here in the system's workspace, found by the rank words that lie behind the masks."""
import numpy as np
import pytest

from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5000, 200003])
def test_reporting_an_error_clears_the_masks(env, n):  # noqa: F811
    torch, g, O = env
    rng = np.random.default_rng(n)
    prm = g.gt_default_params()
    prm.eps, prm.group_mode = 0.02, g.GT_GROUP_CELLS
    s = g.System(n, prm)
    s.set_state(rng.standard_normal((n, 3)), np.zeros((n, 3)), np.full(n, 1.0 / n, np.float32))
    s.build_tree()
    aold, ref, acc = torch.ones(n, device="cuda"), torch.zeros((n, 4), device="cuda"), torch.zeros((n, 4), device="cuda")
    s.accel_active(None, aold, ref)
    evens = torch.arange(0, n, 2, dtype=torch.int32, device="cuda")
    s.accel_active(evens, aold, torch.zeros((len(evens), 4), device="cuda"))
    s.sync()
    # every other particle active: the rank words are (0x55555555, 16 k); the masks of n / 32 + 1 words are before them,
    # every array 256-byte aligned
    words = s.ws[: s.ws.numel() // 256 * 256].view(torch.int32)
    head = words.view(-1, 64)[:, :4].cpu().numpy()
    at = np.flatnonzero((head == np.array([0x55555555, 0, 0x55555555, 16])).all(axis=1))
    assert len(at) == 1
    marks = (int(at[0]) - (4 * (n // 32 + 1) + 255) // 256) * 64
    assert not words[marks: marks + n // 32 + 1].any()
    words[marks: marks + n // 32] = -1  # a group for every particle
    torch.cuda.synchronize()
    assert s.probe_bounded_wait(1) == g.GT_ETIMEOUT  # an error is latched, reported and cleared
    s.accel_active(None, aold, acc)
    s.sync()
    s.close()
    assert torch.equal(acc, ref)

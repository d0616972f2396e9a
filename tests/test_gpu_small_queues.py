"""Walk queues that are depth-first from the start: no teams, which would hand every group back to one of their warps;
the same forces in a batch as alone, and in a time near that with a larger queue."""
import numpy as np
import pytest

from paper_1610_07279_gb300 import ics
from test_gpu_parity import env  # noqa: F401
from test_gpu_sort_long_runs import _plummer

pytestmark = pytest.mark.gpu


def test_time_of_few_groups_with_a_small_queue(env):  # noqa: F811
    """A Plummer sphere of 2^16 (3618 groups): 162 us with a queue of 4096 and teams, 115 without them, 119 with a queue of
    16384, which teams of four can use."""
    torch, g, O = env
    n = 1 << 16
    pos = _plummer(n, 0.0)
    times = {}
    for queue in (4096, 16384):
        prm = g.gt_default_params()
        prm.eps, prm.leaf_max, prm.walk_queue, prm.group_mode = 0.01, 16, queue, g.GT_GROUP_CELLS
        s = g.System(n, prm)
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
        times[queue] = sorted(t[2:])[5]
        s.sync()
        s.close()
    assert times[4096] < 1.2 * times[16384], times


@pytest.mark.parametrize("queues", [(4096,), (1024, 16384), (8192, 2048, 16384)])
def test_members_with_small_queues(env, queues):  # noqa: F811
    torch, g, O = env
    prms, states = [], []
    for k in range(9):
        prm = g.gt_default_params()
        prm.eps, prm.walk_queue, prm.group_mode = 0.01, queues[k % len(queues)], g.GT_GROUP_CELLS
        prms.append(prm)
        states.append(ics.plummer(900 + 411 * k, seed=k)[:3])
    b = g.Batch([len(s[2]) for s in states], prms)
    for m, s in zip(b.systems, states):
        m.set_state(*s)
    b.accel(bootstrap=True)
    b.sync()
    for k, s in enumerate(states):
        n = len(s[2])
        one = g.System(n, prms[k])
        one.set_state(*s)
        one.build_tree()
        out = torch.zeros((n, 4), device="cuda")
        one.accel_active(None, torch.from_numpy(b.systems[k].get_state()["aold"]).cuda(), out)
        one.sync()
        assert np.array_equal(b.get_acc(k)[0][:n].view(np.uint32), out.cpu().numpy().view(np.uint32)), k
        one.close()
    b.close()

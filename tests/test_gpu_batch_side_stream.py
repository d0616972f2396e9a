"""A batch's first evaluation on its own stream, which doesn't wait for the default stream: its tables have arrived,
the forces are those of a batch on the default stream, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsys", [3, 8, 64])
def test_first_evaluation_on_a_side_stream(nsys):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_07279_gb300 import build
    from paper_1610_07279_gb300 import gothic as g
    build.build()
    g.load()
    rng = np.random.default_rng(nsys)
    n = 700
    prm = g.gt_default_params()
    prm.eps, prm.walk_queue = 0.02, 8192
    state = [(rng.standard_normal((n, 3)), np.zeros((n, 3)), np.full(n, 1.0 / n, np.float32)) for _ in range(nsys)]
    out = []
    for stream in (None, 0):  # a stream of the batch's own, the default stream
        for _ in range(4):    # a new batch: its tables are written and read at once
            b = g.Batch([n] * nsys, [prm] * nsys, stream)
            for m, s in zip(b.systems, state):
                m.set_state(*s)
            torch.cuda.synchronize()
            b.accel(bootstrap=True)
            b.sync()
            out.append(np.stack([b.get_acc(k)[0][:n].view(np.uint32) for k in range(nsys)]))
            b.close()
    assert all(np.array_equal(o, out[0]) for o in out[1:])

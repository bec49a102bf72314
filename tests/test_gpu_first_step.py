"""ehd_step enqueues work on the run's stream and nothing else, the first step
of a run included (it decides whether the run steps on chip): it does not wait
for work on the default stream, and it may be called while a capture in the
strictest mode is going on in the same thread, after which the run has the same
form (and bits) as any other."""
import numpy as np
import pytest

import workloads as wl

from captured_graph import captured

gpu = pytest.mark.gpu
SIZES = [(64, 52, {}), (128, 104, {}), (256, 205, {}), (64, 52, dict(storage="f64"))]


def _run(nx, ny, kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    a, ph = wl.roll(93, 0.1)
    return torch, ehd.Run(nx, ny, 190.0, 10, 10, 4000, 0.25, u_ion=5e-3, amp=a, phase=ph, **kw)


@gpu
@pytest.mark.parametrize("nx,ny,kw", SIZES)
def test_first_step_does_not_wait_for_the_default_stream(nx, ny, kw):
    _run(nx, ny, kw)[1].step(1).sync()  # kernels loaded
    torch, r = _run(nx, ny, kw)
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)  # about 0.2 s of the legacy default stream
    e = torch.cuda.Event()
    e.record()
    r.step(1)
    assert not e.query(), "ehd_step waited for the default stream"
    torch.cuda.synchronize()
    r.close()


@gpu
@pytest.mark.parametrize("nx,ny,kw", SIZES)
def test_first_step_during_a_capture_of_another_stream(nx, ny, kw):
    torch, r = _run(nx, ny, kw)
    _, ref = _run(nx, ny, kw)
    x = torch.zeros(1000, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):  # capture_error_mode "global"
        x += 1
        r.step(3)
    g.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 1000.0
    ref.step(3)
    (fa, ga), (fb, gb) = r.save(), ref.save()
    assert np.array_equal(fa, fb) and np.array_equal(ga, gb)
    from paper_1812_05711_gb300 import ehd_stream
    forms = [captured(ehd_stream(v.handle), lambda: v.step(1))[0] for v in (r, ref)]
    assert forms[0] == forms[1]
    assert ("k_resident" in forms[0][0]) == (nx * ny <= 128 * 104 and not kw)
    r.close()
    ref.close()

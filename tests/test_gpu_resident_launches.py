"""On-chip runs of more steps than one launch takes: the launches follow each
other with the same bits as a kernel per phase, and none holds the GPU's SMs
for long (looked at in a captured graph)."""
import numpy as np
import pytest

import workloads as wl

from captured_graph import captured

gpu = pytest.mark.gpu


def _runs(n, nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    a, ph = wl.roll(95, 0.1)
    return ehd, [ehd.Run(nx, ny, 190.0, 10, 10, 4000, 0.25, u_ion=5e-3, amp=a, phase=ph) for _ in range(n)]


@gpu
@pytest.mark.parametrize("nx,ny,steps", [(64, 52, 256), (64, 52, 257), (128, 104, 515)])
def test_many_launches_same_bits(nx, ny, steps):
    ehd, (r1, r2) = _runs(2, nx, ny)
    r1.step(steps)
    for _ in range(steps // 103):
        ehd.ehd_step_profile(r2.handle, 103)
    ehd.ehd_step_profile(r2.handle, steps % 103)
    (fa, ga), (fb, gb) = r1.save(), r2.save()
    assert np.array_equal(fa, fb) and np.array_equal(ga, gb)
    assert r1.diagnostics() == r2.diagnostics()


@gpu
def test_other_streams_get_their_turn():
    ehd, (r,) = _runs(1, 128, 104)
    r.step(1)
    r.sync()
    names, edges = captured(ehd.ehd_stream(r.handle), lambda: ehd.ehd_step(r.handle, 4096))
    assert all("k_resident" in n for n in names)
    assert len(names) >= 8, "one launch holds 16 SMs for more than 3 ms"
    assert not any(prog for _, _, prog in edges)

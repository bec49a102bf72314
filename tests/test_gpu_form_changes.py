"""A run that leaves the on-chip form (a launch shape was asked for, or the
instrumented step): k_resident is then the populations' last writer with no
Poisson solve behind it, and the step kernel, which reads the populations
before it waits for its predecessor, must follow it in plain stream order.
The launches are looked at without being run (captured into a graph); the
results are compared bit for bit."""
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
    a, ph = wl.roll(91, 0.1)
    return ehd, [ehd.Run(nx, ny, 190.0, 10, 10, 4000, 0.25, u_ion=5e-3, amp=a, phase=ph) for _ in range(n)]


@gpu
@pytest.mark.parametrize("param,value", [("pdl", 15), ("slab_rows", 8), ("ring_depth", 2)])
def test_step_kernel_after_on_chip_waits_for_all_of_it(param, value):
    ehd, (r,) = _runs(1, 64, 52)
    r.step(1)  # (the run's form is decided by its first step)
    r.sync()

    def calls():
        ehd.ehd_step(r.handle, 3)
        ehd.ehd_tune(r.handle, param, value)
        ehd.ehd_step(r.handle, 2)

    names, edges = captured(ehd.ehd_stream(r.handle), calls)
    assert sum("k_resident" in n for n in names) == 1, names
    behind = [(b, prog) for a, b, prog in edges if a and "k_resident" in a]
    assert len(behind) == 1 and "k_march2" in behind[0][0] and not behind[0][1], behind
    # the second step's kernel is again launched programmatically behind the solve
    again = [prog for a, b, prog in edges if b and "k_march2" in b and a and "k_irfft" in a]
    assert again == [True], edges


@gpu
@pytest.mark.parametrize("nx,ny", [(64, 52), (128, 104), (256, 40)])
@pytest.mark.parametrize("more", [1, 3, 19])
def test_on_chip_then_tuned_same_bits(nx, ny, more):
    ehd, (r1, r2) = _runs(2, nx, ny)
    r1.step(5)
    ehd.ehd_tune(r1.handle, "pdl", 15)
    r1.step(more)
    ehd.ehd_step_profile(r2.handle, 5 + more)
    (fa, ga), (fb, gb) = r1.save(), r2.save()
    assert np.array_equal(fa, fb) and np.array_equal(ga, gb)
    A, B = r1.fields(), r2.fields()
    for k in A:
        assert np.array_equal(A[k], B[k]), k
    assert r1.diagnostics() == r2.diagnostics()

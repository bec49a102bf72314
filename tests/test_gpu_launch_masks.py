"""Launch masks: a run's default follows its y solve unless a mask was asked
for, and the bits do not depend on the mask -- beside the lines where the
default changes (1140 rows of 1024, 9 2^16 nodes, rows of 2048), with the mean
mode on its own stream and not, both y solves."""
import numpy as np
import pytest

gpu = pytest.mark.gpu


def _run(nx, ny, mask, y_solver, **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    r = ehd.Run(nx, ny, 190.0, 10, 10, 4000, 0.25, u_ion=5e-3, amp=[0.1], phase=[0.3], **kw)
    ehd.ehd_tune(r.handle, "y_solver", y_solver)
    if mask is not None:
        ehd.ehd_tune(r.handle, "pdl", mask)
    return ehd, r


@gpu
@pytest.mark.parametrize("nx,ny,y_solver,kw", [(1024, 1025, 0, {}), (1024, 1139, 0, {}), (1024, 1140, 0, {}),
                                               (1024, 1140, 0, dict(storage="bf16")),
                                               (1024, 1140, 0, dict(ex_spectral=1)), (512, 1152, 0, {}), (512, 1153, 0, {}),
                                               (512, 1056, 1, {}), (2048, 300, 1, {}), (1024, 1040, 1, {})])
def test_same_bits_with_every_mask(nx, ny, y_solver, kw):
    _, r = _run(nx, ny, None, y_solver, **kw)
    r.step(19)
    f, g = r.save()
    F = r.fields(["phi", "Ey"])
    r.close()
    for mask in (0, 15):
        _, r = _run(nx, ny, mask, y_solver, **kw)
        r.step(19)
        f2, g2 = r.save()
        G = r.fields(["phi", "Ey"])
        r.close()
        assert np.array_equal(f, f2) and np.array_equal(g, g2)
        assert all(np.array_equal(F[k], G[k]) for k in F)


@gpu
def test_default_mask_follows_the_y_solve():
    ehd, r = _run(2048, 400, None, 0)
    tri = ehd.ehd_tune_get(r.handle, "pdl")
    ehd.ehd_tune(r.handle, "y_solver", 1)
    odd = ehd.ehd_tune_get(r.handle, "pdl")
    assert odd & 2 and odd != tri  # the solve, by far the longest of the Poisson kernels, is launched ahead
    ehd.ehd_tune(r.handle, "y_solver", 0)
    assert ehd.ehd_tune_get(r.handle, "pdl") == tri
    ehd.ehd_tune(r.handle, "pdl", 3)
    ehd.ehd_tune(r.handle, "y_solver", 1)
    assert ehd.ehd_tune_get(r.handle, "pdl") == 3

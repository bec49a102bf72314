"""Small FP32-compute runs step with their whole state on chip (ehd_step); the
instrumented step (ehd_step_profile) runs the same steps one kernel per phase.
Both give the same bits -- populations, potential, wall fluxes -- for every
row length and storage type that fits, at the smallest and largest row counts,
where bands of rows are uneven, where a chunk of the wavenumber solve holds
one to four rows and the last chunk fewer, for both wall placements, and when
the two forms take turns on one run."""
import numpy as np
import pytest

import workloads as wl

gpu = pytest.mark.gpu


def _pair(nx, ny, storage="f32", **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    a, ph = wl.roll(71, 0.1)
    return ehd, [ehd.Run(nx, ny, 190.0, 10, 10, 4000, 0.25, storage=storage, u_ion=5e-3, amp=a, phase=ph, **kw)
                 for _ in range(2)]


def _same(r1, r2):
    (fa, ga), (fb, gb) = r1.save(), r2.save()
    assert np.array_equal(fa, fb) and np.array_equal(ga, gb)
    A, B = r1.fields(), r2.fields()
    for k in A:
        assert np.array_equal(A[k], B[k]), k
    assert r1.diagnostics() == r2.diagnostics()


@gpu
@pytest.mark.parametrize("nx,ny", [(64, 15), (64, 16), (64, 17), (64, 33), (64, 95), (64, 97), (64, 128), (64, 129),
                                   (128, 31), (128, 66), (128, 104), (128, 128), (256, 16), (256, 41), (256, 80),
                                   (256, 81)])
def test_on_chip_steps_same_bits(nx, ny):
    """(15, 129 and 81 rows: one beyond what fits, both forms are the same.)"""
    ehd, (r1, r2) = _pair(nx, ny)
    r1.step(21)
    ehd.ehd_step_profile(r2.handle, 21)
    _same(r1, r2)


@gpu
@pytest.mark.parametrize("storage", ["bf16", "f16", "f64"])
@pytest.mark.parametrize("nx,ny", [(64, 52), (128, 101), (256, 37)])
def test_on_chip_steps_storage_types(storage, nx, ny):
    ehd, (r1, r2) = _pair(nx, ny, storage, compute="f32")
    r1.step(21)
    ehd.ehd_step_profile(r2.handle, 21)
    _same(r1, r2)


@gpu
@pytest.mark.parametrize("kw", [dict(wall_mode=1), dict(x_symbol=1), dict(dc_printed=1), dict(perturbation=1),
                                dict(ex_spectral=1), dict(step_kernel=1)])
def test_on_chip_steps_options(kw):
    ehd, (r1, r2) = _pair(64, 52, **kw)
    r1.step(21)
    ehd.ehd_step_profile(r2.handle, 21)
    _same(r1, r2)


@gpu
def test_on_chip_and_kernel_per_phase_take_turns():
    ehd, (r1, r2) = _pair(128, 45)
    for n in (1, 2, 17, 4):
        r1.step(n)
        ehd.ehd_step_profile(r1.handle, 3)
    ehd.ehd_step_profile(r2.handle, 36)
    _same(r1, r2)


@gpu
def test_on_chip_non_finite_state_is_reported():
    ehd, (r1, r2) = _pair(64, 40)
    f, g = r1.save()
    g[3, 20, 33] = np.inf
    r1.load(f, g)
    r1.step(2)
    with pytest.raises(ehd.EhdError) as ei:
        r1.sync()
    assert ei.value.status == -4

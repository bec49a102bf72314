"""Runs that step one node per thread against the march form of the same run
(asking for a launch shape selects it): the same bits -- populations, fields,
wall fluxes -- for every row length and storage type, row counts that end a
slab anywhere (first row, last row, one row), at the smallest and near the
largest sizes, both wall placements, through graph replays and single steps,
and when the two forms take turns."""
import numpy as np
import pytest

import workloads as wl

gpu = pytest.mark.gpu


def _runs(nx, ny, storage="f32", **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    a, ph = wl.roll(81, 0.1)
    push, march = (ehd.Run(nx, ny, 190.0, 10, 10, 4000, 0.25, storage=storage, compute="f32", u_ion=5e-3, amp=a,
                           phase=ph, **kw) for _ in range(2))
    ehd.ehd_tune(march.handle, "pdl", 7)
    return ehd, push, march


def _same(r1, r2):
    (fa, ga), (fb, gb) = r1.save(), r2.save()
    assert np.array_equal(fa, fb) and np.array_equal(ga, gb)
    A, B = r1.fields(), r2.fields()
    for k in A:
        assert np.array_equal(A[k], B[k]), k
    assert r1.diagnostics() == r2.diagnostics()


@gpu
@pytest.mark.parametrize("nx,ny", [(64, 129), (64, 1024), (128, 130), (256, 81), (256, 205), (512, 15), (512, 16),
                                   (512, 37), (512, 416), (512, 1024), (1024, 17), (1024, 300), (1024, 512)])
def test_one_node_per_thread_same_bits(nx, ny):
    """(512 x 15 and, at their largest, 2^19 nodes: where the form ends.)"""
    ehd, push, march = _runs(nx, ny)
    push.step(21)
    march.step(21)
    _same(push, march)
    push.close()
    march.close()


@gpu
@pytest.mark.parametrize("storage", ["f64", "bf16", "f16"])
@pytest.mark.parametrize("nx,ny", [(64, 131), (512, 53), (1024, 40)])
def test_one_node_per_thread_storage_types(storage, nx, ny):
    ehd, push, march = _runs(nx, ny, storage)
    push.step(21)
    march.step(21)
    _same(push, march)


@gpu
@pytest.mark.parametrize("kw", [dict(wall_mode=1), dict(x_symbol=1), dict(dc_printed=1)])
def test_one_node_per_thread_options(kw):
    ehd, push, march = _runs(256, 90, **kw)
    push.step(21)
    march.step(21)
    _same(push, march)


@gpu
def test_one_node_per_thread_takes_turns_with_the_march():
    """One run, 7 steps one node per thread and then, its launch shape set, the
    march form; against the march form throughout."""
    ehd, push, march = _runs(512, 99)
    push.step(1)
    ehd.ehd_step_profile(push.handle, 3)
    push.step(3)
    ehd.ehd_tune(push.handle, "pdl", 7)
    push.step(20)
    march.step(27)
    _same(push, march)


@gpu
def test_one_node_per_thread_non_finite_state_is_reported():
    ehd, push, _ = _runs(256, 120)
    f, g = push.save()
    f[5, 60, 200] = np.nan
    push.load(f, g)
    push.step(2)
    with pytest.raises(ehd.EhdError) as ei:
        push.sync()
    assert ei.value.status == -4

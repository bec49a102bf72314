"""Row transforms of rows of 64 to 512 with every lane of a warp at work: a
single run (one row per warp) has bit for bit the state it reaches as a batch
member, whose transforms take the other form (several rows per warp, 32-point
transforms in registers) -- row counts that leave a CTA's warps without a row,
channels of two rows, charge far from uniform."""
import numpy as np
import pytest

import workloads as wl

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("nx,ny", [(64, 2), (64, 29), (128, 33), (256, 41), (512, 37)])
def test_single_run_equals_batch_member(nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    w9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]

    def mk():
        r = ehd.Run(nx, ny, 190.0, 10, 10, 4000, 0.25, storage="f32", u_ion=5e-3)
        rho0 = r.params()["rho0"]
        r.load(wl.random_populations(nx, ny, 61, 1.0, 0.01) * w9, wl.random_populations(nx, ny, 62, rho0, 0.3) * w9)
        return r

    alone, member = mk(), mk()
    batch = ehd.Batch(1, max_nx=512, max_ny=64)
    batch.add(member, 12)
    batch.tick(12)
    batch.sync()
    alone.step(12)
    (fa, ga), (fb, gb) = alone.save(), member.save()
    assert np.array_equal(fa, fb) and np.array_equal(ga, gb)
    assert np.array_equal(alone.fields()["phi"], member.fields()["phi"])
    batch.close()


@gpu
@pytest.mark.parametrize("max_ny", [1024, 1100])
def test_uneven_members_equal_single_runs(max_ny):
    """Members of every row length beside each other, budgets that end inside a
    tick, one tick after the other: with the mean modes among the wavenumber
    items (batches of up to 1024 rows) and on the second stream (above)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    sizes = [(64, max_ny - 3, 9), (128, 45, 14), (256, 21, 3), (512, 30, 14), (1024, 17, 6), (2048, 9, 14)]

    def mk(k, nx, ny):
        a, ph = wl.roll(90 + k, 0.1)
        return ehd.Run(nx, ny, 150.0 + 15 * k, 10, 10, 4000, 0.25, storage="f32", u_ion=2e-3, amp=a, phase=ph)

    batch = ehd.Batch(len(sizes), max_nx=2048, max_ny=max_ny)
    members = []
    for k, (nx, ny, n) in enumerate(sizes):
        r = mk(k, nx, ny)
        batch.add(r, n)
        members.append(r)
    for _ in range(3):
        batch.tick(6)
    batch.sync()
    for k, (nx, ny, n) in enumerate(sizes):
        alone = mk(k, nx, ny)
        ehd.ehd_tune(alone.handle, "slab_rows", 4)  # the batch's slab height at this size
        ehd.ehd_tune(alone.handle, "fft_cta", 0)    # and its warp transforms for rows of 2048
        alone.step(n)
        (fa, ga), (fb, gb) = alone.save(), members[k].save()
        assert np.array_equal(fa, fb) and np.array_equal(ga, gb), (nx, ny)
        assert np.array_equal(alone.fields()["phi"], members[k].fields()["phi"]), (nx, ny)
        da, db = alone.diagnostics(), members[k].diagnostics()
        assert da == db, (nx, ny)
        alone.close()
    batch.close()

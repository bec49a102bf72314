"""The plain FP64 step against the oracle at the edges of its kernels: rows of
every transform length (odd and even radix counts, several rows per warp, one
row per CTA), row counts that leave a warp or CTA part empty, one and two
wavenumbers per CTA, chunks of fewer rows than lanes and the tallest channel
one warp per wavenumber can hold, from loaded far-from-equilibrium
populations as well as from the initial state.

The bound is the 1e-12 (scaled max norm) of the path's parity tests plus, for
the tall channel, the oracle's own rounding of the mean mode's elimination,
which grows with the square of the rows (2.1e-12 at 840 of them)."""
import numpy as np
import pytest

import workloads as wl

gpu = pytest.mark.gpu


def _errors(Nx, Ny, steps, random_state=False, u_ion=5e-3, **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as o
    import paper_1812_05711_gb300 as ehd
    a, ph = wl.roll(41, 1e-2)
    p = o.setup(Nx, Ny, 180.0, 10.0, 10.0, 4000.0, 0.25, u_ion=u_ion, **kw)
    run = ehd.Run(Nx, Ny, 180.0, 10.0, 10.0, 4000.0, 0.25, storage="f64", u_ion=u_ion, amp=a, phase=ph, **kw)
    if random_state:
        _, _, w, _ = o.lattice()
        f = wl.random_populations(Nx, Ny, 51, 1.0, 0.05) * w[:, None, None]
        g = wl.random_populations(Nx, Ny, 52, p.rho0, 0.3) * w[:, None, None]
        s = o.state_from(p, f, g)
        run.load(f, g)
    else:
        s = o.init_state(p, a, ph)
    run.step(steps)
    o.step(s, steps)
    sc = {"rho": 1.0, "ux": p.u_ion, "uy": p.u_ion, "rho_c": p.rho0, "phi": 1.0, "Ex": 1 / p.H, "Ey": 1 / p.H}
    A, B, d = run.fields(), o.fields(s), run.diagnostics()
    run.close()
    assert d["charge"] == pytest.approx(B["rho_c"].sum(), rel=1e-13)
    return {k: float(np.abs(A[k] - B[k]).max() / sc[k]) for k in A}


@gpu
@pytest.mark.parametrize("Nx,Ny", [(16, 17), (32, 31), (64, 33), (128, 2), (256, 7), (512, 37), (1024, 9), (2048, 33)])
@pytest.mark.parametrize("random_state", [False, True])
def test_fp64_rows_of_every_length(Nx, Ny, random_state):
    e = _errors(Nx, Ny, 20, random_state)
    assert max(e.values()) <= 1e-12, e


@gpu
@pytest.mark.parametrize("kw", [dict(wall_mode=1), dict(x_symbol=1)])
def test_fp64_variants(kw):
    e = _errors(64, 52, 40, **kw)
    assert max(e.values()) <= 1e-12, e


@gpu
def test_fp64_tall_channel():
    """8192 rows: the largest tile of one wavenumber in shared memory (200 KB
    with its scratch).  One solve of the charge of a loaded state; the bound
    for E_y and phi scales the oracle's 2.1e-12 at 840 rows by (8192 / 840)^2."""
    e = _errors(16, 8192, 1, u_ion=2e-3)
    assert max(e["phi"], e["Ex"], e["Ey"]) <= 2.1e-12 * (8192 / 840) ** 2, e
    assert max(e["rho"], e["rho_c"]) <= 1e-12, e

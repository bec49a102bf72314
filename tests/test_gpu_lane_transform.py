"""The row transforms of runs (LaneFft for rows of 64 to 512, the wide form for
rows of 1024, the CTA form for 2048) against FP64: the potential's fluctuation of
a Poisson solve of a charge far from uniform.  A single run and a batch member of
up to 512 columns share LaneFft, so that comparing the two says nothing of it.

Tolerance (rms over the channel, of the fluctuation's rms F): the two transforms
round each of log2(Nx) stages, and the solve each of its two sweeps, 2^-24 of the
value at most, so 2 log2(Nx) + 2 roundings; the charge is summed from nine
populations, 9 roundings of the charge, whose rms is R times its fluctuation's;
each rounding's rms is at most 2^-24, and four times their sum is allowed."""
import math

import numpy as np
import pytest

import workloads as wl
from test_gpu_noalloc_limits import _exact

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("nx,ny", [(64, 29), (128, 33), (256, 41), (512, 37), (1024, 23), (2048, 21)])
def test_row_transforms_against_fp64(nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    w9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    r = ehd.Run(nx, ny, 190.0, 10, 10, 4000, 0.25, u_ion=5e-3)
    p = r.params()
    r.load(wl.random_populations(nx, ny, 61, 1.0, 0.01) * w9, wl.random_populations(nx, ny, 62, p["rho0"], 0.5) * w9)
    rc = r.save()[1].sum(0)
    phi = r.fields(["phi"])["phi"]
    r.close()
    want = _exact(rc, p["eps"], 1.0, 0)

    def fluct(a):
        return a - a.mean(axis=1, keepdims=True)

    def rms(a):
        return math.sqrt(float((a * a).mean()))

    F, R = rms(fluct(want)), rms(rc) / rms(fluct(rc))
    tol = 4 * 2.0 ** -24 * (2 * math.log2(nx) + 2 + 9 * R) * F
    err = rms(fluct(phi) - fluct(want))
    print(nx, "error", err / F, "allowed", tol / F)
    assert err <= tol

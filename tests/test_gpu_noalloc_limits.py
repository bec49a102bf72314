"""The one-launch form of ehd_poisson_noalloc where its rule ends (16 rows, 2^18
nodes) and where its chunks of rows are 1, 2, 16 and 128 rows long, one size
beyond each line; which form ran is read from the call captured into a graph.
The one-launch solves are compared with a plain 64-bit one, with the tolerance
of test_gpu_noalloc_cluster.py (the three-kernel form's, which grows with the
rows, is test_zz_no_alloc.py's)."""
import math

import numpy as np
import pytest

from captured_graph import captured

gpu = pytest.mark.gpu


def _exact(rc, eps, phi0, wall_mode):
    linalg = pytest.importorskip("scipy.linalg")
    ny, nx = rc.shape
    S = np.fft.rfft(-rc.astype(np.float64) / eps, axis=1)
    ab = np.ones((3, ny))
    for m in range(S.shape[1]):
        k = 2 * math.pi * m / nx
        ab[1] = -(2.0 + k * k)
        if wall_mode == 0:
            ab[1, 0] -= 1
            ab[1, -1] -= 1
        b = S[:, m].copy()
        if m == 0:
            b[0] -= (2 if wall_mode == 0 else 1) * nx * phi0
        S[:, m] = linalg.solve_banded((1, 1), ab, b)
    return np.fft.irfft(S, n=nx, axis=1)


@gpu
@pytest.mark.parametrize("nx,ny,wall_mode,one_launch", [
    (64, 16, 1, True), (64, 4096, 0, True), (64, 4095, 1, True), (64, 50, 0, True), (128, 2048, 0, True),
    (128, 15, 0, False), (128, 2049, 0, False), (256, 1024, 1, True), (256, 1025, 0, False), (512, 31, 0, True),
    (512, 500, 0, True), (512, 512, 0, True), (512, 513, 0, False), (1024, 40, 0, False), (32, 40, 1, False)])
def test_limits_of_the_one_launch_form(nx, ny, wall_mode, one_launch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    rng = np.random.default_rng(nx + ny)
    y = (np.arange(ny) + 0.5) / ny
    rc = (1 / np.sqrt(y + 0.05)[:, None] + 0.3 * rng.standard_normal((ny, nx))).astype(np.float32) * np.float32(1e-3)
    eps = 2e-4 * ny * ny
    src = torch.from_numpy(rc).cuda()
    phi = torch.zeros_like(src)
    s = torch.cuda.Stream()

    def call():
        ehd.ehd_poisson_noalloc(nx, ny, eps, 0.7, wall_mode, src.data_ptr(), phi.data_ptr(), s.cuda_stream)

    torch.cuda.synchronize()
    names = captured(s.cuda_stream, call)[0]
    solve = [n for n in names if "k_na_tables" not in n]
    assert len(solve) == (1 if one_launch else 3), names
    assert any("k_solve" in n for n in solve) == one_launch, names
    if not one_launch:
        return
    call()
    torch.cuda.synchronize()
    want = _exact(rc, eps, 0.7, wall_mode)
    fluct = np.abs(want - want.mean(axis=1, keepdims=True)).max()
    tol = 2.0 ** -24 * (np.abs(want).max() + 8 * math.log2(nx) * fluct)
    err = np.abs(phi.cpu().numpy() - want).max()
    assert err <= tol, (err, tol)

"""The one-launch form of ehd_poisson_noalloc (64 to 512 columns, up to 2^18
nodes) against a plain 64-bit solve, over row lengths, row counts that leave
bands uneven and chunks short, both wall placements, one row count below the
form's smallest, a pointer that is not aligned to a pair (which takes the
kernel-per-phase form) and a solve in place.

The tolerance is FP32's for this solve: the output's rounding (6e-8 of phi's
scale 1) plus the transform's, 2^-24 log2(Nx) of the fluctuation's scale."""
import math

import numpy as np
import pytest

gpu = pytest.mark.gpu


def _exact(rc, eps, phi0, wall_mode):
    ny, nx = rc.shape
    s = -rc.astype(np.float64) / eps
    S = np.fft.rfft(s, axis=1)
    out = np.empty_like(S)
    for m in range(S.shape[1]):
        k = 2 * math.pi * m / nx
        A = np.diag(np.full(ny, -(2.0 + k * k))) + np.diag(np.ones(ny - 1), 1) + np.diag(np.ones(ny - 1), -1)
        if wall_mode == 0:
            A[0, 0] -= 1
            A[-1, -1] -= 1
        b = S[:, m].copy()
        if m == 0:
            b[0] -= (2 if wall_mode == 0 else 1) * nx * phi0
        out[:, m] = np.linalg.solve(A, b)
    return np.fft.irfft(out, n=nx, axis=1)


@gpu
@pytest.mark.parametrize("nx,ny,wall_mode", [(64, 15, 0), (64, 16, 0), (64, 33, 1), (128, 101, 0), (256, 17, 1),
                                             (256, 208, 0), (512, 64, 0), (512, 131, 1)])
@pytest.mark.parametrize("how", ["plain", "odd pointer", "in place"])
def test_one_launch_solve(nx, ny, wall_mode, how):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    rng = np.random.default_rng(nx + ny)
    y = (np.arange(ny) + 0.5) / ny
    rc = (1 / np.sqrt(y + 0.05)[:, None] + 0.3 * rng.standard_normal((ny, nx))).astype(np.float32) * np.float32(1e-3)
    eps = 2e-4 * ny * ny
    buf = torch.zeros(nx * ny + 2, device="cuda")
    off = 1 if how == "odd pointer" else 0
    src = buf[off:off + nx * ny].view(ny, nx)
    src.copy_(torch.from_numpy(rc))
    phi = src if how == "in place" else torch.zeros_like(src)
    s = torch.cuda.current_stream().cuda_stream
    for _ in range(1 if how == "in place" else 2):
        ehd.ehd_poisson_noalloc(nx, ny, eps, 0.7, wall_mode, src.data_ptr(), phi.data_ptr(), s)
    want = _exact(rc, eps, 0.7, wall_mode)
    got = phi.cpu().numpy()
    fluct = np.abs(want - want.mean(axis=1, keepdims=True)).max()
    tol = 2.0 ** -24 * (np.abs(want).max() + 8 * math.log2(nx) * fluct)
    assert np.abs(got - want).max() <= tol, (np.abs(got - want).max(), tol)

"""The one-launch Poisson solve at the ends of FP32's range: charge whose row
sums exceed the largest FP32 number although every value and the potential are
finite, and charge near the smallest normal number; rows of one sign, of
alternating sign and cancelling ones.  Against the plain 64-bit solve in scaled
numbers (the solve is linear), with the tolerance of FP32 for it: the output's
rounding and the transform's, 2^-24 each of the largest value per stage."""
import math

import numpy as np
import pytest

from test_gpu_noalloc_limits import _exact

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("nx,ny", [(64, 16), (256, 17), (512, 16)])
@pytest.mark.parametrize("scale", [4e36, 1e30, 1e-30])
@pytest.mark.parametrize("rows", ["alike", "alternating", "cancelling"])
def test_range(nx, ny, scale, rows):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    unit = np.ones((ny, nx), dtype=np.float32)
    if rows == "alternating":
        unit[::2] = -1
    elif rows == "cancelling":
        unit[:, ::2] = -1
        scale = min(scale, 1e35)  # (the row's highest wavenumber is Nx times as large)
    rc = unit * np.float32(scale)
    src = torch.from_numpy(rc).cuda()
    phi = torch.zeros_like(src)
    s = torch.cuda.current_stream().cuda_stream
    ehd.ehd_poisson_noalloc(nx, ny, 1.0, 0.0, 0, src.data_ptr(), phi.data_ptr(), s)
    got = phi.cpu().numpy().astype(np.float64) / float(np.float32(scale))
    want = _exact(unit, 1.0, 0.0, 0)
    tol = 2.0 ** -24 * (np.abs(want).max() + 8 * math.log2(nx))
    assert np.isfinite(got).all()
    assert np.abs(got - want).max() <= tol, (np.abs(got - want).max(), tol)

"""Which form a run steps in, read from a step captured into a graph: the forms
that share their bits with another one would pass every comparison if they never
ran.  The sizes of the comparisons (test_gpu_resident.py, test_gpu_push.py) and
one beyond each line."""
import pytest

from captured_graph import captured

gpu = pytest.mark.gpu
CHIP, PUSH, MARCH, STEP, STEP64 = "k_resident", "k_push", "k_march2", "k_step", "k_step64"


def _names(nx, ny, tune=(), **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    r = ehd.Run(nx, ny, 190.0, 10, 10, 4000, 0.25, u_ion=5e-3, amp=[0.1], phase=[0.2], **kw)
    for k, v in tune:
        ehd.ehd_tune(r.handle, k, v)
    r.step(1)
    r.sync()
    names = captured(ehd.ehd_stream(r.handle), lambda: r.step(1))[0]
    r.close()
    return names


def _form(names):
    if any(CHIP in n for n in names):
        assert len(names) == 1
        return CHIP
    found = [f for f in (PUSH, MARCH, STEP64, STEP) if any(f in n and "rfft" not in n for n in names)]
    return found[0] if found else names


@gpu
@pytest.mark.parametrize("nx,ny,form", [
    (64, 15, MARCH), (64, 16, CHIP), (64, 17, CHIP), (64, 97, CHIP), (64, 128, CHIP), (64, 129, PUSH),
    (128, 31, CHIP), (128, 104, CHIP), (128, 128, CHIP), (128, 130, PUSH), (256, 16, CHIP), (256, 80, CHIP),
    (256, 81, PUSH), (256, 205, PUSH), (512, 15, MARCH), (512, 16, PUSH), (512, 416, PUSH), (512, 1024, PUSH),
    (64, 1024, PUSH), (64, 1025, MARCH), (1024, 17, PUSH), (1024, 512, PUSH), (1024, 513, MARCH), (2048, 64, MARCH),
    (32, 40, MARCH)])
def test_form_by_size(nx, ny, form):
    names = _names(nx, ny)
    assert _form(names) == form, names
    assert any("k_rfft_push" in n for n in names) == (form == PUSH), names


@gpu
@pytest.mark.parametrize("nx,ny,kw,tune,form", [
    (64, 52, dict(storage="bf16"), (), CHIP), (64, 52, dict(storage="f16"), (), CHIP),
    (128, 101, dict(storage="bf16"), (), CHIP), (256, 37, dict(storage="f16"), (), CHIP),
    (64, 52, dict(wall_mode=1), (), CHIP), (64, 52, dict(storage="f64", compute="f32"), (), PUSH),
    (512, 53, dict(storage="f64", compute="f32"), (), PUSH), (1024, 40, dict(storage="bf16"), (), PUSH),
    (64, 52, dict(perturbation=1), (), MARCH), (64, 52, dict(ex_spectral=1), (), MARCH),
    (64, 52, dict(step_kernel=1), (), STEP), (64, 52, dict(storage="f64"), (), STEP64),
    (64, 52, {}, (("pdl", 7),), MARCH), (512, 99, {}, (("pdl", 7),), MARCH)])
def test_form_by_kind(nx, ny, kw, tune, form):
    names = _names(nx, ny, tune, **kw)
    assert _form(names) == form, names

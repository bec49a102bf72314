"""ehd_footprint bounds what a run in the perturbation form holds, its base
state's arrays included: short and tall channels of every row length's kind."""
import pytest

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("nx,ny", [(64, 24), (128, 104), (64, 2000), (512, 416), (2048, 61)])
def test_footprint_bounds_a_perturbation_run(nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1812_05711_gb300 as ehd
    ehd.use_torch_allocator(True)
    try:
        torch.cuda.synchronize()
        before = torch.cuda.memory_allocated()
        run = ehd.Run(nx, ny, 200.0, 10, 10, 4000, 0.25, amp=[1e-3], phase=[0.0], perturbation=1)
        run.step(4)
        run.sync()
        held = torch.cuda.memory_allocated() - before
        run.close()
        assert held <= ehd.ehd_footprint(nx, ny, ehd.STORAGE["f32"])
    finally:
        ehd.use_torch_allocator(False)

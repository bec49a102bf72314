"""The bench's DRAM traffic of the step kernel is void once any source of the
kernel has changed: the kernel's file and every header that it includes."""
import shutil

import pytest

import bench


def test_sources_hold_the_collision():
    assert {"k_march.cu", "march_dev.cuh", "ehd_dev.cuh"} <= set(bench._kernel_sources())


@pytest.mark.parametrize("name", bench._kernel_sources())
def test_hash_follows_every_source(tmp_path, name):
    shutil.copytree(bench.CSRC, tmp_path / "csrc")
    before = bench._kernel_hash(str(tmp_path / "csrc"))
    assert before == bench._kernel_hash()
    with open(tmp_path / "csrc" / name, "a") as fh:
        fh.write("// changed\n")
    assert bench._kernel_hash(str(tmp_path / "csrc")) != before


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("pert", [0, 1])
def test_launches_per_step(storage, pert):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if pert and storage == "f64":
        pytest.skip("the perturbation form computes in FP32")
    import paper_1812_05711_gb300 as ehd
    from captured_graph import captured
    r = ehd.Run(2048, 1680, 190.0, 10, 10, 4000, 0.25, storage=storage, amp=[0.1], phase=[0.2], perturbation=pert)
    r.step(1)
    r.sync()
    names = captured(ehd.ehd_stream(r.handle), lambda: r.step(1))[0]
    r.close()
    assert len(names) == bench.LAUNCHES_PER_STEP[storage] + 2 * pert, names

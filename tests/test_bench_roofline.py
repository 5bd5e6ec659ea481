"""What the benchmark's roofline says of the step kernel, without a GPU: a
stored traffic capture counts only for launches that advance as many steps as
the captured one, and the kernel is named by its launches."""
import json

import pytest

import bench
from paper_1608_04118_gb300 import build as B


@pytest.fixture
def capture(tmp_path, monkeypatch):
    """A capture of the current source: a two-step launch at 4096 x 4096."""
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "step_traffic.json").write_text(json.dumps({
        "source_hash": B.kernel_source_hash(),
        "entries": {"f32/npt2/steps2/4096": {"nodes": 4096 * 4096,
                                             "dram_bytes_per_launch": 2.5e9}}}))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))


@pytest.mark.parametrize("n,npt,steps,launches,expect", [
    (4096, 2, 20, 10, 2.5e9), (8192, 2, 20, 10, 1e10),
    (1024, 2, 20, 20, None),  # the one-step kernel of the same schedule
    (4096, 2, 1, 1, None), (4096, 2, 5, 3, None), (1024, 1, 20, 10, None)])
def test_traffic_is_of_launches_of_the_captured_form(capture, n, npt, steps, launches, expect):
    assert bench.kernel_traffic("f32", n, npt, steps, launches)[0] == expect


def test_the_committed_capture_names_its_steps_per_launch():
    with open(bench.os.path.join(bench.ROOT, "profiles", "step_traffic.json")) as fh:
        assert all("/steps" in k for k in json.load(fh)["entries"])


@pytest.mark.parametrize("storage,schedule,staged,n,steps,launches,expect", [
    ("f32", (128, 1, 2), 0, 4096, 20, 10, "k_step2_pair"),
    ("f32", (128, 1, 2), 0, 4096, 1, 1, "k_step_pair"),
    ("f16", (32, 4, 2), 0, 2048, 20, 20, "k_step_pair"),
    ("f32", (64, 2, 1), 0, 1024, 20, 10, "k_step2_node"),
    ("f32", (64, 2, 1), 0, 128, 20, 5, "k_step_tile"),
    ("bf16", (64, 2, 1), 0, 200, 3, 1, "k_step_tile"),
    ("f32", (64, 2, 1), 0, 512, 20, 20, "k_step"),
    ("f32", (32, 4, 2), 1, 4096, 20, 20, "k_step_tma"),
    ("f64", (64, 2, 1), 0, 1024, 20, 20, "k_step_list"),
    ("f64", (128, 2, 1), 0, 1024, 20, 20, "k_step")])
def test_the_kernel_is_named_by_its_launches(storage, schedule, staged, n, steps, launches, expect):
    assert bench.step_kernel(storage, schedule, staged, n, steps, launches) == expect

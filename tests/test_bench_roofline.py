"""What the benchmark's roofline says of the step kernel, without a GPU: a
stored traffic capture counts only for launches that advance as many steps as
the captured one."""
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

"""Two time steps per launch (k_step2_pair, k_step2_node) against one step at
a time.

Large cavities with two nodes per thread advance two steps in one pass; the
fields, the populations and the observables have to be the bits of single
steps, which take the one-step kernels that the oracle tests cover.  Widths
around one and two strips of 30 pairs (the first also owns pair 0, the last
the pair at its end), odd widths (a lone wall node in the last pair), four and
five rows (no row that is not next to a wall) and rows that leave a ragged
last segment; an odd number of steps and one beyond the captured graph.
"""
import numpy as np
import pytest

from paper_1608_04118_gb300 import workloads as W
from tests.helpers import cavity_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

NODES = {"f32": 1 << 22, "f16": 1 << 24, "bf16": 1 << 24}


def _run(cfg, storage, phi, fields, chunks, schedule=(32, 4, 2)):
    c = cavity_for(cfg, storage=storage, phi=phi).set_schedule(*schedule)
    c.set_fields(porosity=phi, **fields)
    for n in chunks:
        c.step(n)
    out = (c.fields(), c.get_state()[64:], c.observables(), c.launches, c.kernel_launches)
    c.close()
    return out


@pytest.mark.parametrize("storage,nx,ny,steps,field,correction", [
    ("f32", 33, 130_000, 5, True, 0), ("f32", 60, 70_001, 4, False, 0),
    ("f32", 62, 67_651, 5, True, 1), ("f32", 63, 66_600, 5, True, 0),
    ("f32", 64, 65_537, 4, False, 0), ("f32", 65, 64_600, 5, True, 0),
    ("f32", 66, 63_600, 3, True, 0), ("f32", 123, 34_200, 4, True, 0),
    ("f32", 124, 33_900, 5, False, 0), ("f32", 126, 33_300, 4, True, 0),
    ("f32", 1_048_576, 4, 5, True, 0), ("f32", 838_861, 5, 4, True, 0),
    ("f32", 2049, 2053, 75, True, 0), ("f32", 2048, 2048, 70, True, 1),
    ("f16", 129, 130_100, 5, True, 0), ("bf16", 130, 129_100, 4, False, 0),
    ("f16", 4096, 4096, 36, True, 0), ("bf16", 4099, 4101, 5, True, 0),
    ("bf16", 3_400_001, 5, 5, True, 0)])
def test_two_steps_per_launch_give_the_bits_of_single_steps(storage, nx, ny, steps, field,
                                                            correction):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    assert nx * ny >= NODES[storage]
    cfg = dict(W.random_params(301, nx, ny), thermal_correction=correction, ergun=bool(field))
    fields = W.random_fields(nx, ny, 302)
    phi = W.porosity_field(nx, ny, 0.4, 0.9, seed=303).reshape(-1) if field else None
    _same(_run(cfg, storage, phi, fields, [steps]), _run(cfg, storage, phi, fields, [1] * steps),
          steps)


@pytest.mark.parametrize("nx,ny,steps,field,correction", [
    (31, 34_000, 5, True, 0), (32, 33_000, 4, False, 0), (33, 32_000, 5, True, 1),
    (60, 17_600, 4, True, 0), (61, 17_300, 5, False, 0), (62, 17_001, 4, True, 0),
    (63, 16_900, 3, True, 0), (262_144, 4, 5, True, 0), (209_716, 5, 4, True, 0),
    (1027, 1025, 75, True, 0)])
def test_two_steps_with_one_node_per_thread(nx, ny, steps, field, correction):
    """The one-node walk: widths around one and two strips of 30 nodes."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    assert nx * ny >= 1 << 20
    cfg = dict(W.random_params(311, nx, ny), thermal_correction=correction, ergun=bool(field))
    fields = W.random_fields(nx, ny, 312)
    phi = W.porosity_field(nx, ny, 0.4, 0.9, seed=313).reshape(-1) if field else None
    _same(_run(cfg, "f32", phi, fields, [steps], (64, 2, 1)),
          _run(cfg, "f32", phi, fields, [1] * steps, (64, 2, 1)), steps)


def _same(a, b, steps):
    for k in a[0]:
        assert np.array_equal(a[0][k], b[0][k]), k
    assert a[1] == b[1]
    for k in a[2]:
        assert a[2][k] == b[2][k] or np.isnan(a[2][k]), k
    assert a[3] == b[3] == steps
    assert a[4] == (steps + 1) // 2 and b[4] == steps

"""Several time steps per launch on small cavities (k_step_tile) against one
step at a time.

Small cavities with one node per thread advance up to four steps per launch
from tiles in shared memory; the fields, the populations and the observables
have to be the bits of single steps, which take the one-step kernel that the
oracle tests cover.  Sizes from one tile of two nodes upwards (every node next
to a wall), tiles cut unevenly, thin lattices, the largest size that takes the
tiles and one that does not; remainders of one, two and three steps and a call
that replays the captured graph; per-node porosity, local h_v (its |u| passes
between the steps too) and the correction term.
"""
import numpy as np
import pytest

from paper_1608_04118_gb300 import workloads as W
from tests.helpers import cavity_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _run(cfg, storage, phi, fields, chunks):
    c = cavity_for(cfg, storage=storage, phi=phi).set_schedule(64, 2, 1)
    c.set_fields(porosity=phi, **fields)
    for n in chunks:
        c.step(n)
    out = (c.fields(), c.get_state()[64:], c.observables(), c.launches, c.kernel_launches)
    c.close()
    return out


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny,steps,field,local", [
    (4, 4, 3, True, 0), (5, 4, 9, False, 1), (7, 9, 6, True, 0), (8, 300, 5, True, 1),
    (300, 5, 7, False, 0), (64, 64, 41, False, 0), (65, 63, 40, True, 1), (131, 97, 10, True, 0),
    (200, 180, 6, True, 1), (200, 190, 35, True, 0)])
def test_steps_per_launch_change_no_bit(storage, nx, ny, steps, field, local):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = dict(W.random_params(401, nx, ny), thermal_correction=local, hv_local=local,
               Dp_over_L=0.0135, ergun=bool(field))
    fields = W.random_fields(nx, ny, 402)
    phi = W.porosity_field(nx, ny, 0.4, 0.9, seed=403).reshape(-1) if field else None
    a = _run(cfg, storage, phi, fields, [steps])
    b = _run(cfg, storage, phi, fields, [1] * steps)
    for k in a[0]:
        assert np.array_equal(a[0][k], b[0][k]), k
    assert a[1] == b[1]
    for k in a[2]:
        assert a[2][k] == b[2][k] or np.isnan(a[2][k]), k
    assert a[3] == b[3] == steps
    assert a[4] == (steps + 3) // 4 and b[4] == steps


def test_larger_lattices_take_one_step_per_launch():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cavity_for(W.random_params(404, 256, 256)).set_fields().step(40)
    assert c.kernel_launches == c.launches == 40

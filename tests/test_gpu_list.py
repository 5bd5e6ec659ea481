"""The FP64 step from a list of nodes (the default schedule) against the
block kernel of an explicit schedule: the same bits, at sizes where the list
can go wrong -- every node a wall or next to one, interiors that fill whole
warps exactly, by one more or one less, thin lattices, several blocks."""
import numpy as np
import pytest

from paper_1608_04118_gb300 import workloads as W
from tests.helpers import cavity_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,field,local", [
    (4, 4, True, 0), (5, 7, False, 1), (34, 34, True, 1), (35, 33, True, 0), (33, 35, False, 0),
    (300, 5, True, 0), (4, 200, False, 0), (131, 97, True, 1)])
def test_node_list_gives_the_bits_of_the_block_kernel(nx, ny, field, local):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = dict(W.random_params(601, nx, ny), thermal_correction=local, hv_local=local,
               Dp_over_L=0.0135, ergun=bool(field))
    fields = W.random_fields(nx, ny, 602)
    phi = W.porosity_field(nx, ny, 0.4, 0.9, seed=603).reshape(-1) if field else None
    out = []
    for schedule in ((64, 2, 1), (128, 2, 1)):
        c = cavity_for(cfg, storage="f64", phi=phi).set_schedule(*schedule)
        c.set_fields(porosity=phi, **fields).step(41)
        out.append((c.fields(), c.get_state()[64:]))
        c.close()
    for k in out[0][0]:
        assert np.array_equal(out[0][0][k], out[1][0][k]), k
    assert out[0][1] == out[1][1]

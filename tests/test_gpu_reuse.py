"""One handle used for several runs: the captured step graphs outlive
set_fields while the lattice constants stay the same, and only then."""
import numpy as np
import pytest

from paper_1608_04118_gb300 import workloads as W
from tests.helpers import cavity_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage,nx,ny", [("f32", 60, 44), ("f64", 40, 33), ("f16", 260, 260)])
def test_runs_on_one_handle_are_the_runs_on_fresh_ones(storage, nx, ny):
    """Porosity field A, then B (another Ergun diameter, so other constants),
    then A again, each long enough to replay a graph from either buffer
    parity, on one handle and on a fresh handle each: the same bits."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = dict(W.random_params(501, nx, ny), ergun=True)
    phis = [W.porosity_field(nx, ny, 0.4, hi, seed=502).reshape(-1) for hi in (0.9, 0.6)]
    one = cavity_for(cfg, storage=storage, phi=phis[0])
    for phi in (phis[0], phis[1], phis[0]):
        fresh = cavity_for(cfg, storage=storage, phi=phi)
        for c in (one, fresh):
            c.set_fields(porosity=phi).step(70).step(1).step(69)
        a, b = one.fields(), fresh.fields()
        for k in a:
            assert np.array_equal(a[k], b[k]), k
        assert one.get_state()[64:] == fresh.get_state()[64:]
        fresh.close()

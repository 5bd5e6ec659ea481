"""The lone last node of odd rows in the two-step walk, whose rows are spread
over the lanes of its strip's warp: a last segment of one row, of two and of
all but one, all rows in one segment, and a lattice whose last wall row is the
first of another segment.  The bits of single steps."""
import pytest

from paper_1608_04118_gb300 import workloads as W
from tests.test_gpu_march import _run, _same

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage,nx,ny,steps,field", [
    *[("f32", 131, 32_040 + k, 4, True) for k in range(0, 24, 1)],
    ("f32", 167_773, 25, 4, True), ("f32", 174_763, 24, 5, False), ("f32", 182_363, 23, 4, True),
    ("f32", 599_187, 7, 4, True), ("f32", 1_048_577, 4, 3, True),
    ("f16", 671_089, 25, 4, True), ("bf16", 2_396_747, 7, 3, False)])
def test_odd_columns_give_the_bits_of_single_steps(storage, nx, ny, steps, field):
    """131 x 32,040 and the 23 heights above it leave every remainder of a
    segment of up to 24 rows."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = dict(W.random_params(321, nx, ny), ergun=bool(field))
    phi = W.porosity_field(nx, ny, 0.4, 0.9, seed=323).reshape(-1) if field else None
    fields = W.random_fields(nx, ny, 322)
    _same(_run(cfg, storage, phi, fields, [steps]), _run(cfg, storage, phi, fields, [1] * steps),
          steps)

"""Narrow FP32 lattices under the default schedule: one step per launch where
the two-step walk would fill its strips poorly, two elsewhere; a schedule that
was set takes the walk at any width, with the same bits."""
import numpy as np
import pytest

from paper_1608_04118_gb300 import workloads as W
from tests.helpers import cavity_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,per", [
    (62, 17_000, 2), (63, 16_800, 1), (64, 16_500, 1), (96, 11_100, 1), (213, 5_000, 1),
    (213, 9_850, 2), (255, 4_200, 1), (256, 4_097, 2), (1024, 1024, 2), (1024, 1023, 1),
    (66, 63_750, 1), (124, 34_025, 2), (128, 32_968, 1), (129, 32_713, 2), (256, 16_584, 1), (306, 13_906, 2),
    (2048, 2048, 2)])
def test_steps_per_launch_by_width(nx, ny, per):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = dict(W.random_params(331, nx, ny), ergun=True)
    phi = W.porosity_field(nx, ny, 0.4, 0.9, seed=333).reshape(-1)
    a, b = (cavity_for(cfg, storage="f32", phi=phi) for _ in range(2))
    b.set_schedule(*b.schedule)
    fields = W.random_fields(nx, ny, 332)
    for c in (a, b):
        c.set_fields(porosity=phi, **fields).step(38)  # a captured graph and six more
    assert a.launches == b.launches == 38 and a.kernel_launches == 38 // per
    assert b.kernel_launches == (19 if nx * ny >= 1 << 20 else 38)
    fa, fb = a.fields(), b.fields()
    for k in fa:
        assert np.array_equal(fa[k], fb[k]), k
    a.close()
    b.close()

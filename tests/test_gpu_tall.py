"""Lattices with more rows of blocks than a grid holds: ltne_step refuses every
number of steps alike and leaves the handle as it was, also where kernels of
several steps have grids that fit; another schedule then steps them."""
import numpy as np
import pytest

from paper_1608_04118_gb300 import ltne as lt
from paper_1608_04118_gb300 import workloads as W
from tests.helpers import cavity_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,schedule,fits", [
    (64, 65_600, None, (32, 4, 2)),         # default: two nodes per thread, 128 x 1
    (64, 65_536, None, (32, 4, 2)),         # one row more than a grid holds
    (17, 65_600, (256, 1, 1), (64, 2, 1))])  # the one-node walk
def test_a_grid_that_does_not_fit_is_refused_before_any_step(nx, ny, schedule, fits):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cavity_for(W.random_params(701, nx, ny), storage="f32")
    if schedule:
        c.set_schedule(*schedule)
    c.set_fields(**W.random_fields(nx, ny, 702))
    before = c.fields()
    for n in (2, 1, 3, 35, 64):
        with pytest.raises(lt.LtneError) as err:
            c.step(n)
        assert err.value.code == lt.LTNE_ERR_CUDA
        assert c.launches == c.kernel_launches == 0
    after = c.fields()
    for k in before:
        assert np.array_equal(before[k], after[k]), k
    assert c.observables()["step"] == 0
    c.set_schedule(*fits).step(3)
    assert c.observables()["step"] == 3 and c.launches == 3
    c.close()


def test_the_tallest_lattice_of_the_default_schedule_steps():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cavity_for(W.random_params(703, 65, 65_535), storage="f32").set_fields().step(3)
    assert c.schedule == (128, 1, 2) and c.observables()["step"] == 3
    c.close()

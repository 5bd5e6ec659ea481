"""ltne_get_fields with some of its five pointers null, into pageable arrays:
every subset gives the values of the whole read and nothing else is written,
in the one-copy form of small lattices (padded rows among them) and in the
block-wise form above it."""
import ctypes as C

import numpy as np
import pytest

from paper_1608_04118_gb300 import ltne as lt
from paper_1608_04118_gb300 import workloads as W
from tests.helpers import cavity_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage,nx,ny,subsets", [
    ("f32", 37, 29, range(32)), ("f64", 64, 41, range(32)), ("f16", 500, 301, (8, 17, 22, 31)),
    ("f32", 1301, 1290, (8, 17, 31))])
def test_any_subset_of_the_fields(storage, nx, ny, subsets):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cavity_for(W.random_params(801, nx, ny), storage=storage)
    c.set_fields(**W.random_fields(nx, ny, 802)).step(3)
    whole = [c.fields()[k] for k in lt.FIELD_KEYS]
    for mask in subsets:
        got = [np.full((ny, nx), -7.0) for _ in range(5)]
        ptr = [g.ctypes.data_as(C.POINTER(C.c_double)) if mask >> k & 1 else None
               for k, g in enumerate(got)]
        assert lt._lib().ltne_get_fields(c.h, *ptr) == lt.LTNE_OK
        for k in range(5):
            assert np.array_equal(got[k], whole[k]) if mask >> k & 1 else (got[k] == -7.0).all()
    c.close()

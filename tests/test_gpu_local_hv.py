"""The local h_v of Eq. 52 at speeds whose squares are below FP32's normal
range: |u| = 1e-21 gives h_v = 4e-15 of its scale, which is all that moves the
fluid temperature off its reference where only the solid is warm."""
import numpy as np
import pytest

from tests.helpers import cavity_for, rel_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,schedule,chunks", [
    (64, 64, (64, 2, 1), [4]), (64, 64, (64, 2, 1), [1] * 4),  # tiles, one step a launch
    (260, 210, (64, 2, 1), [4]), (65, 61, (32, 4, 2), [4])])
def test_speeds_below_the_normal_range_count(nx, ny, schedule, chunks):
    """FP32 against FP64 storage, away from the side walls (the oracle keeps
    absolute populations, beside which such momenta vanish).  Tolerance: the
    logarithm and exponential of the power cost about 2e-6 of h_v, each step a
    few 1e-7 more; 1e-4 covers five evaluations twenty times over."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = dict(nx=nx, ny=ny, Ra=1e4, Pr=1.0, Da=1e-2, porosity=0.6, gamma_sf=1.0, sigma=1.0,
               T_hot=1.0, T_cold=0.0, T_ref=0.0, hv_local=1, Dp_over_L=0.0135)
    n = nx * ny
    ux, ts = np.full(n, 1e-21), np.full(n, 0.5)
    r = cavity_for(cfg, storage="f64").set_fields(ux=ux, T_s=ts)
    c = cavity_for(cfg, storage="f32").set_schedule(*schedule).set_fields(ux=ux, T_s=ts)
    inner = (slice(8, -8), slice(8, -8))
    for k in [0] + chunks:
        c.step(k)
        r.step(k)
        got, ref = c.fields()["Tf"][inner], r.fields()["Tf"][inner]
        assert 0 < ref.max() < 1e-11
        assert rel_l2(got, ref) <= 1e-4, k
    c.close()
    r.close()

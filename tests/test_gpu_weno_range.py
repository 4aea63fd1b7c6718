"""The FP32 WENO-5 faces at the jumps that hot walls make at the fast velocities
of the order-16 sets: a population's value over its weight is about 1 in the
gas and 1e12 to 1e19 in the emitted ghosts (T_w = 2.5 to 4), with differences of
thousands beside the jump, so that the squared ratio of two smoothness
indicators times a difference leaves the FP32 range unless it is bounded.
The line, pair and persistent kernels against the oracle, at the FP32 parity
bar of test_gpu_parity; at T_w = 4, where the order-15 expansion of the wall's
Maxwellian has grown to values of 700 and FP32 sums no longer meet that bar,
the state has to stay finite."""
import numpy as np
import pytest

from paper_1708_03249_gb300 import workloads as W
from test_gpu_parity import _check_fp32, run_pair

pytestmark = pytest.mark.gpu

_PHYS = dict(precision=W.FP32, Kn=0.1, ax=-0.1)
CASES = {
    "1d_hot_right": (W.make(Qx=16, Qy=16, nx=30, T_left=1.0, T_right=3.0, **_PHYS), False),
    "1d_hot_left": (W.make(Qx=16, Qy=16, nx=30, T_left=2.5, T_right=1.0, **_PHYS), False),
    "1d_persistent": (W.make(Qx=16, Qy=16, nx=30, T_left=3.0, T_right=1.0, **_PHYS), True),
    "2d_hot_right": (W.make(Qx=16, Qy=16, nx=17, ny=6, Ly=0.6, T_left=1.0, T_right=2.5, **_PHYS), False),
    "2d_hot_left": (W.make(Qx=16, Qy=16, nx=17, ny=6, Ly=0.6, T_left=3.0, T_right=1.0, **_PHYS), False),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_hot_walls_match_oracle(name):
    cfg, persistent = CASES[name]
    got, mom, N, refs = run_pair(cfg, 2, init=(1.0, 0.05, 0.0, 1.5), persistent=persistent)
    _check_fp32(got, mom, refs)


@pytest.mark.parametrize("ny", [1, 6])
def test_hotter_walls_stay_finite(ny):
    cfg = W.make(Qx=16, Qy=16, nx=17, ny=ny, Ly=0.6, T_left=1.0, T_right=4.0, **_PHYS)
    got, mom, N, refs = run_pair(cfg, 2, init=(1.0, 0.05, 0.0, 1.5), persistent=False)
    assert np.isfinite(got).all()

"""FP64 groups in 2D around the size from which they march: the kernel that each
side takes, and both against the oracle (odd numbers of rows, both slabs, both
schemes, a collisionless group, a force field).  Tolerance of test_gpu_parity:
1e-10 of max |f| up to order 8."""
import math

import pytest

from paper_1708_03249_gb300 import workloads as W
from test_gpu_parity import _check_fp64, run_pair

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

_PHYS = dict(precision=W.FP64, T_left=0.8, T_right=1.4, ax=-0.3, ay=-0.2, Ly=0.6)
CASES = {
    "8x4_generic": (W.make(Qx=4, Qy=4, nx=64, ny=32, Kn=0.05, **_PHYS), False),
    "8x4_marches": (W.make(Qx=4, Qy=4, nx=67, ny=31, Kn=0.05, **_PHYS), True),
    "8x4_marches_upwind": (W.make(Qx=4, Qy=4, nx=43, ny=49, Kn=0.05, advection=W.UPWIND2, **_PHYS), True),
    "16x8_generic": (W.make(Qx=8, Qy=8, nx=32, ny=16, Kn=0.05, **_PHYS), False),
    "16x8_marches": (W.make(Qx=8, Qy=8, nx=27, ny=19, Kn=0.05, stretch_A=0.5, **_PHYS), True),
    "16x8_marches_upwind": (W.make(Qx=8, Qy=8, nx=75, ny=7, Kn=0.05, advection=W.UPWIND2, **_PHYS), True),
    "16x8_marches_collisionless": (W.make(Qx=8, Qy=8, nx=103, ny=5, Kn=math.inf, **_PHYS), True),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_fp64_2d_matches_oracle(name):
    from paper_1708_03249_gb300 import hlb
    cfg, marches = CASES[name]
    with hlb.Handle(cfg, stream=torch.cuda.current_stream().cuda_stream) as h:
        assert (h.step_form(0)["segment_cells"] > 0) == marches
    got, mom, N, refs = run_pair(cfg, 2)
    _check_fp64(got, refs, 1e-10)

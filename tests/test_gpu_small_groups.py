"""The forms that small FP32 groups step with: the one-launch node pass from 257
nodes in 2D, the per-stage launches from 513 nodes of several 1D instances; at
both lines, against the oracle."""
import pytest

from paper_1708_03249_gb300 import workloads as W
from test_gpu_parity import _check_fp32, run_pair

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

_PHYS = dict(precision=W.FP32, T_left=0.8, T_right=1.4, Kn=0.05, ax=-0.3, ay=-0.2)


def _launches(cfg):
    from paper_1708_03249_gb300 import hlb
    with hlb.Handle(cfg, stream=torch.cuda.current_stream().cuda_stream) as h:
        h.init_equilibrium()
        h.launch_count(reset=True)
        h.step(3)
        return h.launch_count() // 3, h.step_form(0)["persistent"]


@pytest.mark.parametrize("Q,nx,ny,launches", [(4, 32, 8, 12), (4, 37, 7, 6), (8, 37, 7, 6), (16, 43, 6, 6)])
def test_small_2d_groups(Q, nx, ny, launches):
    cfg = W.make(Qx=Q, Qy=Q, nx=nx, ny=ny, Ly=0.6, **_PHYS)
    assert _launches(cfg) == (launches, False)
    got, mom, N, refs = run_pair(cfg, 2)
    _check_fp32(got, mom, refs)


@pytest.mark.parametrize("Q", [4, 8, 16])
@pytest.mark.parametrize("last,form", [(312, (1, True)), (313, (6, False))])
def test_small_1d_groups_of_several_instances(Q, last, form):
    cfgs = [W.make(Qx=Q, Qy=Q, nx=nx, **_PHYS) for nx in (6, 194, last)]
    assert _launches(cfgs) == form
    got, mom, N, refs = run_pair(cfgs, 2)
    _check_fp32(got, mom, refs)

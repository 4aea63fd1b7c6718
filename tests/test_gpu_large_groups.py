"""The lines above which large FP32 groups of few velocities take the separate
node kernels: the launches per step on both sides, and a short instance that
shares the group with a long one, against the oracle."""
import numpy as np
import pytest

from paper_1708_03249_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

_PHYS = dict(precision=W.FP32, T_left=0.8, T_right=1.4, Kn=0.05, ax=-0.3)


@pytest.mark.parametrize("kw,nodes,launches", [
    (dict(Qx=16, Nx_eq=7), 1 << 17, 6), (dict(Qx=16, Nx_eq=7), (1 << 17) + 1, 12),
    (dict(Qx=16), (1 << 17) + 1, 6),
    (dict(Qx=4, Qy=4), 1 << 19, 6), (dict(Qx=4, Qy=4), (1 << 19) + 1, 12),
])
def test_node_pass_of_large_groups(kw, nodes, launches):
    from oracle.solver import Solver, config_from
    from paper_1708_03249_gb300 import hlb
    cfgs = [W.make(nx=nx, **_PHYS, **kw) for nx in (41, nodes - 41)]
    with hlb.Handle(cfgs, stream=torch.cuda.current_stream().cuda_stream) as h:
        h.init_equilibrium(1.0, 0.05, 0.0, 1.1)
        V = h.values // h.nodes
        f = h.get_state().astype(np.float64)
        f[:41 * V] *= W.perturbation((41 * V,), seed=3, amplitude=0.05)
        h.set_state(f)
        f0 = h.get_state()[:41 * V].astype(np.float64)
        h.launch_count(reset=True)
        h.step(2)
        assert h.launch_count() == 2 * launches
        got = h.get_state()[:41 * V].astype(np.float64)
        h.moments()                                  # raises where the long instance is not finite
    s = Solver(config_from(cfgs[0]))
    s.f = f0.reshape(s.f.shape).copy()
    s.step(2)
    ref = s.f.reshape(-1)
    assert np.abs(got - ref).max() < 2e-5 * np.abs(ref).max()

"""The moments kernel of FP32 groups with 2Q_x a power of two (32 nodes per CTA,
eight lanes per node) against NumPy's FP64 sums of the same FP32 state: ragged
last CTAs, every row length from 4 to 32, absent axes, several instances in the
caller's order.  Tolerance: the FP32 momenta and products are rounded once per
term (2^-24 of the terms' magnitude sum), far below 1e-6 of the moment scales."""
import numpy as np
import pytest

from paper_1708_03249_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = {
    "row4": [W.make(Qx=2, nx=33, precision=W.FP32)],
    "row8": [W.make(Qx=4, Qy=4, nx=31, precision=W.FP32)],
    "row16_z": [W.make(Qx=8, Qy=4, Qz=4, nx=13, ny=5, Ly=0.3, precision=W.FP32)],
    "row32": [W.make(Qx=16, Qy=16, nx=65, precision=W.FP32)],
    "row32_no_y": [W.make(Qx=16, nx=32, precision=W.FP32)],
    "instances": [W.make(Qx=Q, Qy=4, nx=nx, precision=W.FP32) for Q, nx in ((4, 7), (8, 34), (4, 40), (8, 6))],
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_moments_match_fp64_sums(name):
    from paper_1708_03249_gb300 import hlb
    cfgs = CASES[name]
    with hlb.Handle(cfgs, stream=torch.cuda.current_stream().cuda_stream) as h:
        h.init_equilibrium(1.1, 0.2, 0.1, 1.2)
        f = (h.get_state().astype(np.float64) * W.perturbation(h.values, seed=9)).astype(np.float32)
        h.set_state(f)
        n, u, T, q = h.moments()
        tabs = [h.tables(i) for i in range(len(cfgs))]
    off = at = 0
    for c, t in zip(cfgs, tabs):
        nodes = c["nx"] * c["ny"]
        px, py, pz = t["px"], t["py"], t["pz"]
        size = nodes * px.size * py.size * pz.size
        g = f[off:off + size].astype(np.float64).reshape(nodes, pz.size, py.size, px.size)
        off += size
        D = 1 + (c["Qy"] > 0) + (c["Qz"] > 0)
        rn = g.sum((1, 2, 3))
        ru = np.stack([(g * px).sum((1, 2, 3)), (g * py[:, None]).sum((1, 2, 3)), (g * pz[:, None, None]).sum((1, 2, 3))], 1) / rn[:, None]
        c2 = sum((p - ru[:, k].reshape(-1, 1, 1, 1)) ** 2 for k, p in
                 enumerate((px, py[:, None], pz[:, None, None])[:3]) if (k == 0 or (c["Qy"], c["Qz"])[k - 1]))
        rT = (c2 * g).sum((1, 2, 3)) / (D * rn)
        rq = 0.5 * ((px - ru[:, 0].reshape(-1, 1, 1, 1)) * c2 * g).sum((1, 2, 3))
        s = slice(at, at + nodes)
        at += nodes
        for got, ref in ((n[s], rn), (u[s], ru), (T[s], rT), (q[s], rq)):
            assert np.abs(got - ref).max() < 1e-6

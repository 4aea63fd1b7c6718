"""The FP64 node pass (moments, factor lines and walls in one launch) and the 2D
FP64 marching kernel against the oracle, where they end or switch: one node
per CTA and eight (more than two nodes per SM, with a ragged last CTA), odd
numbers of rows, odd and absent axes, a force along p_z (the per-node kernel
with the pass's lines), a field, a collisionless instance among others, and flows
fast enough to leave the polynomial range of exp and erf.  Tolerances of
test_gpu_parity: 1e-10 of max |f| up to order 8."""
import math

import numpy as np
import pytest

from paper_1708_03249_gb300 import workloads as W
from test_gpu_parity import _check_fp64, run_pair

pytestmark = pytest.mark.gpu

_PHYS = dict(precision=W.FP64, T_left=0.8, T_right=1.4, Kn=0.05, ax=-0.3)
CASES = {
    "1d_eight_per_cta": (W.make(Qx=4, Qy=4, nx=701, advection=W.UPWIND2, ay=-0.2, **_PHYS), 2),
    "2d_8x4_odd_rows": (W.make(Qx=4, Qy=4, nx=29, ny=25, Ly=0.6, ay=-0.2, stretch_A=0.5, **_PHYS), 2),
    "2d_16x8_odd_rows": (W.make(Qx=8, Qy=8, nx=13, ny=7, Ly=0.6, ay=-0.2, **_PHYS), 2),
    "2d_16x8_upwind": (W.make(Qx=8, Qy=8, nx=10, ny=5, Ly=0.6, ay=-0.2, advection=W.UPWIND2, **_PHYS), 2),
    "2d_three_axes": (W.make(Qx=3, Qy=2, Qz=4, nx=11, ny=6, Ly=0.6, az=0.2, **_PHYS), 2),
    "2d_8x4_with_z": (W.make(Qx=4, Qy=4, Qz=2, nx=30, ny=27, Ly=0.6, ay=-0.2, **_PHYS), 1),
    "1d_no_y_odd_order": (W.make(Qx=5, nx=33, **_PHYS), 3),
    "mixed_with_collisionless": ([W.make(Qx=4, Qy=4, nx=nx, precision=W.FP64, Kn=Kn, T_right=1.3, ax=-0.2)
                                  for nx, Kn in ((19, 0.1), (45, math.inf), (7, 1.0))], 3),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_fp64_pass_matches_oracle(name):
    cfg, steps = CASES[name]
    got, mom, N, refs = run_pair(cfg, steps)
    _check_fp64(got, refs, 1e-10)


def test_fp64_pass_fast_flow():
    ux = 1.1
    cfg = W.make(Qx=4, Qy=4, nx=36, ay=-0.2, **_PHYS)
    got, mom, N, refs = run_pair(cfg, 2, init=(1.0, ux, 0.1, 1.0))
    _check_fp64(got, refs, 1e-10)


def test_fp64_weno_scale_and_jumps():
    # jumps of 100 decades between neighbouring cells: finite, and equal to the
    # same run with the state scaled by 2^-300 (the weights do not change under
    # a common scale)
    from paper_1708_03249_gb300 import hlb
    import torch
    cfg = W.make(Qx=4, nx=40, precision=W.FP64, Kn=math.inf, ax=-0.1, T_right=1.2)
    outs = []
    for scale in (1.0, 2.0 ** -300):
        with hlb.Handle(cfg, stream=torch.cuda.current_stream().cuda_stream) as h:
            h.init_equilibrium()
            f = h.get_state().reshape(40, 8)
            f[11:23] *= 1e-100
            h.set_state((f * scale).reshape(-1))
            h.step(6)
            outs.append(h.get_state() / scale)
    assert np.isfinite(outs[0]).all()
    np.testing.assert_allclose(outs[1], outs[0], rtol=1e-12, atol=1e-14)


_WIDE = dict(precision=W.FP64, dt=1e-4, T_left=1.0, T_right=1.2, ax=-0.5)


@pytest.mark.parametrize("name,cfg", [
    ("odd_cells", W.make(Qx=200, Nx_eq=12, nx=7, Kn=0.3, **_WIDE)),
    ("fibres_and_y_force", W.make(Qx=64, Qy=2, Nx_eq=12, nx=6, Kn=0.3, ay=-0.2, **_WIDE)),
    ("z_force_upwind", W.make(Qx=40, Qz=2, Nx_eq=8, nx=5, Kn=0.3, az=0.3, advection=W.UPWIND2, **_WIDE)),
    ("instances", [W.make(Qx=50, Nx_eq=10, nx=nx, Kn=Kn, **_WIDE) for nx, Kn in ((9, 0.2), (6, math.inf), (11, 1.0))]),
])
def test_wide_stage_kernel(name, cfg):
    # stage_wide_kernel: odd numbers of cells (a pair of one), CTAs that straddle
    # fibres and nodes, several axes, instances of different length
    got, mom, N, refs = run_pair(cfg, 3)
    _check_fp64(got, refs, 1e-9)


def test_wide_stage_kernel_two_cells_per_thread():
    # more than 19456 (pair, velocity) items: odd cells, a CTA that straddles instances
    cfg = [W.make(Qx=200, Nx_eq=12, nx=nx, Kn=Kn, **_WIDE) for nx, Kn in ((49, 0.3), (51, math.inf))]
    got, mom, N, refs = run_pair(cfg, 2)
    _check_fp64(got, refs, 1e-9)


def test_wide_stage_kernel_field():
    from oracle.solver import Solver, config_from
    from paper_1708_03249_gb300 import hlb
    import torch
    cfg = W.make(Qx=40, Nx_eq=8, nx=9, Kn=0.3, **_WIDE)
    field = 0.4 * np.sin(np.arange(9.0))[None, :]
    with hlb.Handle(cfg, stream=torch.cuda.current_stream().cuda_stream) as h:
        h.set_force_field(0, field)
        h.init_equilibrium()
        f0 = h.get_state() * W.perturbation(h.values, seed=3)
        h.set_state(f0)
        h.step(3)
        got = h.get_state()
    c = config_from(cfg)
    c.ax_field = field
    s = Solver(c)
    s.f = f0.reshape(s.f.shape).copy()
    s.step(3)
    _check_fp64(got, [s], 1e-9)

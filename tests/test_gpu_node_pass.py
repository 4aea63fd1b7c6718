"""The one-launch node pass of FP32 groups (moment sums, factor lines and walls)
against the oracle, at the sizes where its batches of 8 or 32 nodes (8 for rows of 32 and at most 9728 nodes), its rows and
its orders end: ragged and single batches, each row length (2 Qx = 8, 16, 32),
absent axes, a collisionless instance among others, and flows fast enough to
leave the polynomial range of exp and erf (|u_x| / sqrt(2T) > 0.7).  The
tolerances are the FP32 parity bar of test_gpu_parity."""
import math

import pytest

from paper_1708_03249_gb300 import workloads as W
from test_gpu_parity import _check_fp32, run_pair

pytestmark = pytest.mark.gpu

_PHYS = dict(precision=W.FP32, T_left=0.8, T_right=1.4, Kn=0.05, ax=-0.3)
CASES = {
    "1d_q4_one_ragged_batch": (W.make(Qx=4, Qy=4, nx=6, ay=-0.2, **_PHYS), 4),
    "1d_q8_two_batches": (W.make(Qx=8, Qy=8, nx=33, ay=-0.2, **_PHYS), 3),
    "1d_q16_two_batches": (W.make(Qx=16, Qy=16, nx=37, ay=-0.2, **_PHYS), 2),
    "1d_q16_no_y": (W.make(Qx=16, nx=65, **_PHYS), 3),
    "1d_low_order": (W.make(Qx=8, Qy=8, Nx_eq=4, Ny_eq=3, nx=31, ay=-0.2, **_PHYS), 3),
    "1d_full_range": (W.make(Qx=16, Qy=8, nx=40, x_basis=W.X_FULL, ay=-0.2, **_PHYS), 3),
    "2d_q4_1025_nodes": (W.make(Qx=4, Qy=4, nx=41, ny=25, Ly=0.6, ay=-0.2, advection=W.UPWIND2, **_PHYS), 2),
    "2d_q4_z": (W.make(Qx=4, Qy=4, Qz=4, nx=40, ny=27, Ly=0.6, ay=-0.2, **_PHYS), 1),
    "2d_q4_5041_nodes": (W.make(Qx=4, Qy=4, nx=71, ny=71, Ly=0.6, ay=-0.2, **_PHYS), 1),
    "1d_q16_9789_nodes": ([W.make(Qx=16, Qy=4, nx=nx, **_PHYS) for nx in (4903, 7, 4879)], 1),
    "mixed_with_collisionless": ([W.make(Qx=4, Qy=4, nx=nx, precision=W.FP32, Kn=Kn, T_right=1.3, ax=-0.2)
                                  for nx, Kn in ((19, 0.1), (45, math.inf), (7, 1.0))], 4),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_node_pass_matches_oracle(name):
    cfg, steps = CASES[name]
    got, mom, N, refs = run_pair(cfg, steps, persistent=False)
    _check_fp32(got, mom, refs)


@pytest.mark.parametrize("Q,ux", [(4, 1.1), (8, -1.2), (16, 1.05)])
def test_node_pass_fast_flow(Q, ux):
    cfg = W.make(Qx=Q, Qy=4, nx=36, ay=-0.2, **_PHYS)
    got, mom, N, refs = run_pair(cfg, 2, init=(1.0, ux, 0.1, 1.0), persistent=False)
    _check_fp32(got, mom, refs)

"""The FP64 node pass in groups of more than 16 nodes per SM (16 nodes per CTA):
a last CTA of one node, of fifteen, full ones; rows that fill its lanes and
rows that do not, absent axes, the full-range and Gauss-Laguerre bases, a
collisionless instance among others, a 2D group.  Against the oracle, 1e-10 of
max |f| (test_gpu_parity)."""
import math

import pytest

from paper_1708_03249_gb300 import workloads as W
from test_gpu_parity import _check_fp64, run_pair

pytestmark = pytest.mark.gpu

_PHYS = dict(precision=W.FP64, T_left=0.8, T_right=1.4, Kn=0.05, ax=-0.3)
CASES = {
    "8x4_one_left": (W.make(Qx=4, Qy=4, nx=2449, ay=-0.2, **_PHYS), 2),
    "16x8_fifteen_left": (W.make(Qx=8, Qy=8, nx=2447, ay=-0.2, **_PHYS), 1),
    "8x1": (W.make(Qx=4, nx=2464, **_PHYS), 2),
    "10x1_odd_order": (W.make(Qx=5, nx=2441, **_PHYS), 2),
    "6x2x4_z": (W.make(Qx=3, Qy=2, Qz=4, nx=2443, az=0.2, **_PHYS), 1),
    "full_range": (W.make(Qx=8, Qy=4, nx=2450, x_basis=W.X_FULL, **_PHYS), 1),
    "laguerre": (W.make(Qx=4, Qy=4, nx=2450, x_basis=W.X_LAGUERRE, **_PHYS), 1),
    "mixed_with_collisionless": ([W.make(Qx=4, Qy=4, nx=nx, precision=W.FP64, Kn=Kn, T_right=1.3, ax=-0.2)
                                  for nx, Kn in ((2401, 0.1), (45, math.inf), (7, 1.0))], 2),
    "2d_8x4": (W.make(Qx=4, Qy=4, nx=61, ny=41, Ly=0.6, ay=-0.2, **_PHYS), 1),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_sixteen_nodes_per_cta_match_oracle(name):
    cfg, steps = CASES[name]
    got, mom, N, refs = run_pair(cfg, steps)
    _check_fp64(got, refs, 1e-10)


def test_sixteen_nodes_per_cta_fast_flow():
    cfg = W.make(Qx=4, Qy=4, nx=2455, ay=-0.2, **_PHYS)
    got, mom, N, refs = run_pair(cfg, 1, init=(1.0, 1.1, 0.1, 1.0))
    _check_fp64(got, refs, 1e-10)

"""A channel and its mirror image (walls exchanged, cells and p_x reversed) give
the same bits: without collisions and force every term of a step has a mirror
image of the same rounding, so the ghosts of the two walls, the fluxes that fix
the emitted densities and those that the stage kernels apply must be rounded
alike, whichever kernel and segment forms them."""
import numpy as np
import pytest

from paper_1708_03249_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = {
    "line_16x8": (dict(Qx=8, Qy=8, nx=32), False),
    "line_32x16": (dict(Qx=16, Qy=16, nx=64), False),
    "pair_16x8": (dict(Qx=8, Qy=8, nx=32, ny=6), False),
    "persistent_16x8": (dict(Qx=8, Qy=8, nx=32), True),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_mirrored_channel_gives_the_same_bits(name):
    from paper_1708_03249_gb300 import hlb
    cfg, persistent = CASES[name]
    Q, nx, ny = cfg["Qx"], cfg["nx"], cfg.get("ny", 1)
    outs = []
    for mirror in (False, True):
        T = (1.4, 0.8) if mirror else (0.8, 1.4)
        with hlb.Handle(W.make(T_left=T[0], T_right=T[1], precision=W.FP32, **cfg),
                        stream=torch.cuda.current_stream().cuda_stream) as h:
            h.set_persistent(persistent)
            assert len(set(h.tables()["dx"])) == 1
            flip = lambda f: np.concatenate([f[:, ::-1, :, Q:], f[:, ::-1, :, :Q]], axis=-1)
            h.init_equilibrium(1.0, 0.0, 0.0, 1.0)
            f = h.get_state().reshape(ny, nx, -1, 2 * Q).astype(np.float64)
            f = (f * W.perturbation(f.shape, seed=11, amplitude=0.1)).astype(np.float32)
            h.set_state(flip(f) if mirror else f)
            h.step(4)
            g = h.get_state().reshape(f.shape)
            outs.append(flip(g) if mirror else g)
    np.testing.assert_array_equal(outs[0], outs[1])

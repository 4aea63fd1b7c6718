"""hlb_autotune on groups whose built-in segments are shorter than a multiple of 6
from 12 cells on: it times the built-in length too and keeps it where it is
the fastest (by 1.2 to 1.6 times on these handles), and the steps after it
give the same bits.  A form that it could not time is not switched on."""
import numpy as np
import pytest

from paper_1708_03249_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _stream():
    return torch.cuda.current_stream().cuda_stream


SHORT = {
    "fp64_2d": W.make(Qx=8, Qy=8, nx=95, ny=61, Ly=0.6, Kn=0.1, precision=W.FP64),
    "fp32_2d": W.make(Qx=8, Qy=8, nx=60, ny=40, Ly=0.6, Kn=0.1, precision=W.FP32),
    "fp32_1d": W.channel_1d_stretched(0.1),
}


@pytest.mark.parametrize("name", sorted(SHORT))
def test_autotune_keeps_the_short_built_in_segments(name):
    from paper_1708_03249_gb300 import hlb
    outs = []
    for tune in (False, True):
        with hlb.Handle(SHORT[name], stream=_stream()) as h:
            h.set_persistent(False)
            built_in = h.step_form(0)["segment_cells"]
            assert 0 < built_in < 12
            h.init_equilibrium(1.0, 0.05, 0.0, 1.1)
            if tune:
                seg = h.autotune()
                assert len(seg) == 1 and seg[0] >= 12 and seg[0] % 6 == 0
                assert h.step_form(0)["segment_cells"] == built_in
            h.step(3)
            outs.append(h.get_state())
    np.testing.assert_array_equal(outs[0], outs[1])


@pytest.mark.parametrize("what", ["per_launch_timing", "force_field"])
def test_autotune_switches_no_untimed_form_on(what):
    # with per-launch timing or a force field on, hlb_autotune can time the
    # per-stage launches alone: once that is off again the group steps as before
    from paper_1708_03249_gb300 import hlb
    cfg = W.make(Qx=8, Qy=8, nx=300, Kn=0.1, precision=W.FP32, ax=-0.2)
    with hlb.Handle(cfg, stream=_stream()) as h:
        assert not h.step_form(0)["persistent"]
        h.init_equilibrium()
        if what == "force_field":
            h.set_force_field(0, ax=np.full(300, 0.1))
        else:
            h.set_options(use_graphs=True, time_kernels=True)
        h.autotune()
        if what == "force_field":
            h.set_force_field(0)
        else:
            h.set_options(use_graphs=True, time_kernels=False)
        form = h.step_form(0)
        assert not form["persistent"] and form["tuned_ms"] == (0.0, 0.0)


def test_persistent_items_have_their_own_length():
    # the persistent kernel's segment items do not follow the per-stage
    # launches' segments: longer in a large group (an item reads its tables
    # anew), and untouched where the tuner lengthens or shortens the latter
    from paper_1708_03249_gb300 import hlb
    with hlb.Handle(W.make(Qx=8, Qy=8, nx=100000, Kn=0.1, precision=W.FP32), stream=_stream()) as h:
        per_stage = h.step_form(0)["segment_cells"]
        h.set_persistent(True)
        items = h.step_form(0)["segment_cells"]
        assert items > per_stage
        h.set_persistent(False)
        h.init_equilibrium()
        h.autotune()
        h.set_persistent(True)
        form = h.step_form(0)
        assert form["persistent"] and form["segment_cells"] == items


@pytest.mark.parametrize("nx", [6, 7, 9, 53])
def test_persistent_short_items_give_the_same_bits(nx):
    # items of 4 cells (one iteration each), ragged last ones among them,
    # against the lengths that the tuner may pick
    from paper_1708_03249_gb300 import hlb
    cfgs = [W.make(Qx=8, Qy=8, nx=n, Kn=0.1, precision=W.FP32, T_right=1.3, ax=-0.2) for n in (nx, 150)]
    outs = []
    for tune in (False, True):
        with hlb.Handle(cfgs, stream=_stream()) as h:
            h.set_persistent(True)
            h.init_equilibrium(1.0, 0.05, 0.0, 1.1)
            if tune:
                h.autotune()
            else:
                assert h.step_form(0)["segment_cells"] == 4
            persistent = h.step_form(0)["persistent"]
            h.step(5)
            outs.append(h.get_state())
    if persistent:
        np.testing.assert_array_equal(outs[0], outs[1])
    else:
        np.testing.assert_allclose(outs[0], outs[1], rtol=0, atol=2e-6 * np.abs(outs[1]).max())

"""The persistent kernel at length: the stored oracle runs of the seeded batched
instances (see test_gpu_long_runs) with every group switched to it, since its
default leaves groups of their size to the per-stage launches."""
import json

import numpy as np
import pytest

from paper_1708_03249_gb300 import workloads as W
from test_gpu_long_runs import _errors, _load, _stream

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")


@pytest.mark.parametrize("stochastic", [False, True], ids=["nearest", "stochastic"])
def test_persistent_batched_instances_at_length(stochastic):
    # the bars of the per-stage runs: 1e-5; with rounding to nearest 1e-4 for
    # the instances whose residual ends below what FP32 resolves per step
    from make_long_runs import BATCH_COUNT, initial_state
    from paper_1708_03249_gb300 import hlb
    insts = W.batched_instances(BATCH_COUNT)
    refs = [_load(f"batched_{i:02d}") for i in range(BATCH_COUNT)]
    by_len = {}
    for i, ref in enumerate(refs):
        assert json.loads(str(ref["config"])) == insts[i]
        by_len.setdefault(int(ref["steps"]), []).append(i)
    for steps, ids in by_len.items():
        with hlb.Handle([insts[i] for i in ids], stream=_stream()) as h:
            h.set_persistent(True)
            assert all(h.step_form(k)["persistent"] for k in range(len(ids)))
            h.set_rounding(stochastic)
            h.set_state(np.concatenate([initial_state(insts[i], int(refs[i]["seed"])).reshape(-1) for i in ids])
                        .astype(np.float32))
            h.step(steps)
            mom = h.moments()
            N, _ = h.diag()
        off = 0
        for k, i in enumerate(ids):
            nodes = insts[i]["nx"] * insts[i]["ny"]
            errs = _errors(mom, refs[i], slice(off, off + nodes))
            off += nodes
            stuck = not stochastic and float(refs[i]["residual"]) < 2.0 ** -24 / float(refs[i]["dt"])
            assert max(errs.values()) < (1e-4 if stuck else 1e-5), (i, errs)
            if not stuck:
                assert abs(N[k] / float(refs[i]["N"]) - 1.0) < 1e-5, i

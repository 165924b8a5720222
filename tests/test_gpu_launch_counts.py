"""Per-kernel timing sees every launch of a step: over the kernel kinds the counts
add up to launches_per_step, and the step timed launch by launch gives the bits
of the replayed one."""
import os

import numpy as np
import pytest

from paper_2409_10729_gb300 import inputs as I

pytestmark = pytest.mark.gpu
WEIGHTS = os.path.join(os.path.dirname(I.__file__), "gate_weights.npy")


@pytest.mark.parametrize("n", [(33,), (20, 17), (18, 11, 9)], ids=str)
@pytest.mark.parametrize("form", ["fp64", "fp64_fast", "mixed", "gated"])
def test_counts_add_up(form, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_10729_gb300 import mfc
    p, w = I.random_periodic(len(n), list(n), seed=6)
    states = []
    for timed in (False, True):
        s = mfc.Solver(p, form)
        if form == "gated":
            s.set_mlp_weights(np.load(WEIGHTS))
        s.set_state_prim(w)
        s.set_timing(timed)
        s.step_rk3(0.4, 2)
        states.append(s.get_state())
        counts = {k: v[1] for k, v in s.kernel_times().items()}
        assert sum(counts.values()) == (2 * s.launches_per_step() if timed else 0)
        if timed:
            assert counts["sweep_" + "xyz"[len(n) - 1]] == 6
            assert counts["stage_update"] == (6 if form == "gated" and len(n) == 3 else 0)
        s.close()
    assert np.array_equal(*states)

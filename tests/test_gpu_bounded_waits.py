"""GPU: a bounded wait that runs out inside the iteration kernels is reported as such by the calls that
check at intervals (to a tolerance, early stopping), not as iterations that did not converge."""
import numpy as np
import pytest

import gabp_synth
from gpu_common import ensure_built, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["tolerance", "early stop"])
def test_bounded_wait_in_a_checked_run(call):
    ensure_built()
    from paper_2404_12968_gb300 import GABP_KERNEL_TMA, GabpError
    p = gabp_synth.config_small(0)
    with solver(p, "fp32", kernel=GABP_KERNEL_TMA, debug_flags=1, check_every=1, max_iters=3) as s:
        before = s.get_messages()
        with pytest.raises(GabpError, match="bounded wait"):
            s.iterate(-1, 0.5) if call == "tolerance" else s.iterate_early_stop(10, 0.5)
        assert np.array_equal(s.get_messages(), before)
        assert s.stats()["iterations"] == 0
        assert np.isfinite(s.residual())   # the flag was cleared
    with solver(p, "fp32", kernel=GABP_KERNEL_TMA, check_every=1, max_iters=3) as s:   # the same call without the stall
        with pytest.raises(GabpError, match="max_iters"):
            s.iterate(-1, 0.5)


def test_bounded_wait_in_a_checked_batch():
    ensure_built()
    from paper_2404_12968_gb300 import GABP_KERNEL_TMA, Batch, GabpError
    probs = gabp_synth.config_batch(seed=7, count=3, lo=40, hi=90)
    with Batch(probs, kernel=GABP_KERNEL_TMA, tile_y=30, debug_flags=1, check_every=2) as b:
        with pytest.raises(GabpError, match="bounded wait"):
            b.iterate(-1, 0.3)
        b.residuals()   # the flag was cleared (the messages are unspecified)

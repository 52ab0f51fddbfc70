"""The pass time of the register-resident Frank-Wolfe is its launch alone: the view,
buffers and clears of a handle's first call are not in it."""
import numpy as np
import pytest

from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,kernel", [("exact", "fw_resident_kernel"), ("fp64", "fw_resident64_kernel")])
def test_first_call_times_the_launch_only(precision, kernel):
    from paper_2504_10937_gb300 import lds
    n, u, v, _ = synth.gnp_planted(300, 0.03, (12, 9), (0.9, 0.8), seed=7)
    try:
        lds.set_pass_profiling(True)
        with lds.Graph(n, u, v) as g:
            g.fw(1, precision=precision, want=())            # the library's own first use
        share = []
        for _ in range(5):
            with lds.Graph(n, u, v) as g:
                g.fw(1, precision=precision, want=())
                t = g.fw_timing()
                assert t["pass_kernel"] == kernel and t["pass_launches"] == 1 and t["pass_us"] > 0
                share.append(t["pass_us"] / (1000.0 * t["fw_ms"]))
    finally:
        lds.set_pass_profiling(False)
    # one iteration of a small graph is a few us; building its view and clears take more
    assert np.median(share) < 0.6

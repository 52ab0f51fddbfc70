"""The edge pass over quads with part of its vertices staged: sizes around the fewest
staged ids (4,096) and above them, few and many entries a block, against the symmetric
pass."""
import numpy as np
import pytest

from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


def _ring(n):
    return n, np.r_[0:n - 1, 0].astype(np.int32), np.r_[1:n, n - 1].astype(np.int32)


def _power_law(n, m):
    n, u, v, _ = synth.chung_lu(n, m, 2.2, seed=n, n_blocks=2, block_size_range=(20, 60))
    return n, u.astype(np.int32), v.astype(np.int32)


GRAPHS = {
    "ring_4094": lambda: _ring(4094),          # every id staged, the last counter's half unused
    "ring_4095": lambda: _ring(4095),
    "ring_4096": lambda: _ring(4096),          # one id past the staged ones
    "ring_5001": lambda: _ring(5001),
    "power_law_9k": lambda: _power_law(9001, 30000),
    "power_law_60k": lambda: _power_law(60001, 150000),
    "power_law_60k_dense": lambda: _power_law(60013, 700000),
}


@pytest.mark.parametrize("precision", ["exact", "fp32"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_partly_staged_quads_match_symmetric_pass(name, precision):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    with lds.Graph(n, u, v) as g:
        for N in (1, 2, 40):
            try:
                lds.set_fw_variant(1)
                want = g.fw(N, precision=precision)
                lds.set_fw_variant(5)
                got = g.fw(N, precision=precision)
                assert g.fw_timing()["pass_kernel"] == "fw_quad_kernel"
            finally:
                lds.set_fw_variant(0)
            for k in ("r", "R", "W", "last"):
                assert np.array_equal(got[k], want[k]), (N, k)

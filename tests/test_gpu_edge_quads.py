"""The edge pass over quads against the symmetric pass and the oracle's iterates where
the layout can go wrong: rows of 1 to 9 targets, one chunk, more vertices than the
shared memory holds, several folds, the last choices."""
import numpy as np
import pytest

from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


def _stars(n):
    """Hubs 0..8 and leaves joined to 1..9 of them: rows of those lengths."""
    u, v = [], []
    for x in range(9, n):
        k = (x - 9) % 9 + 1
        u += list(range(k))
        v += [x] * k
    return n, np.array(u, np.int32), np.array(v, np.int32)


GRAPHS = {
    "edge": lambda: (4, np.array([1], np.int32), np.array([3], np.int32)),
    "rows": lambda: _stars(700),
    "past_hot": lambda: synth.chung_lu(90001, 250000, 2.3, seed=7, n_blocks=2, block_size_range=(50, 120))[:3],
    "ring": lambda: (60000, np.r_[0:59999, 0].astype(np.int32), np.r_[1:60000, 59999].astype(np.int32)),
}


@pytest.mark.parametrize("precision", ["exact", "fp32"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_quads_match_symmetric_pass(name, precision):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    order = np.lexsort((v, u))
    with lds.Graph(n, u[order], v[order]) as g:
        for N in (0, 1, 2, 33, 70):
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

"""The vertex-node maximum flow's per-block counts against the pattern-node form: either
side of the sizes where they start (2,048 patterns; patterns per vertex) and end (8,192
vertices), ragged ranges, loops, pairs and triangles sorted by their first member, and
hubs.  The flow and the cut's side are whole numbers and match exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _network(nv, count, seed):
    rng = np.random.default_rng(seed)
    width = rng.choice([1, 2, 3], count, p=[0.1, 0.3, 0.6])
    members = (nv * rng.random((count, 3)) ** 3).astype(np.int64) % nv      # most on low ids
    pats = [tuple(dict.fromkeys(int(x) for x in r[:w])) for r, w in zip(members, width)]
    return sorted(pats)


@pytest.mark.parametrize("nv,count", [(1, 2048), (3, 2047), (3, 2048), (3, 2049), (40, 9001), (1024, 2048), (1025, 2050),
                                      (4096, 8191), (4096, 8192), (8191, 17001), (8192, 17001), (8193, 17001)])
@pytest.mark.parametrize("ratio", [0.7, 1.0, 1.6])
def test_forms_agree(nv, count, ratio):
    from paper_2504_10937_gb300 import lds
    pats = _network(nv, count, nv + count)
    q = 89
    p = max(1, int(ratio * q * len(pats) / nv))
    try:
        lds.set_flow_variant(1)
        want, side1 = lds.pattern_max_flow(nv, pats, p, q)
        lds.set_flow_variant(2)
        got, side2 = lds.pattern_max_flow(nv, pats, p, q)
    finally:
        lds.set_flow_variant(0)
    assert got == want and np.array_equal(side1, side2)


def test_wide_pattern_is_refused():
    from paper_2504_10937_gb300 import lds
    pats = _network(50, 3000, 7) + [(1, 2, 3, 4)]
    try:
        lds.set_flow_variant(2)
        with pytest.raises(lds.LdsError) as e:
            lds.pattern_max_flow(50, pats, 60, 1)
        assert e.value.status == lds.EINVAL
    finally:
        lds.set_flow_variant(0)

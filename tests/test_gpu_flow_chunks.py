"""The vertex-node maximum flow against the pattern-node form where its chunks can
go wrong: a hub of many 32-incidence chunks, degrees around a chunk's size, many
vertices of low degree, two- and three-member patterns and loops mixed."""
import numpy as np
import pytest

from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


def _network(kind):
    rng = synth.SplitMix64(11)
    if kind == "hub":                       # vertex 0 in 3,000 pairs; a ring; loops
        nv = 3001
        pats = [(0, i) for i in range(1, nv)] + [(i, i % 3000 + 1) for i in range(1, nv)]
        pats += [(int(x),) for x in rng.integers(0, nv, 500)]
    elif kind == "chunk_edges":             # cliques whose degrees are 31, 32 and 33
        pats, nv = [], 0
        for s in (32, 33, 34):
            iu, iv = np.triu_indices(s, 1)
            pats += [(int(a) + nv, int(b) + nv) for a, b in zip(iu, iv)]
            nv += s
        pats += [(0, 32), (33, 65)]
    elif kind == "sparse":                  # many vertices, few incidences each
        nv = 20000
        a, b = rng.integers(0, nv, 30000), rng.integers(0, nv, 30000)
        pats = [(int(x), int(y)) for x, y in zip(a, b) if x != y]
    else:                                   # triangles around a dense core, pairs and loops
        nv = 400
        t = rng.integers(0, nv, 3 * 6000).reshape(-1, 3) % np.array([nv, 60, 60])
        pats = [tuple(int(x) for x in r) for r in t if len(set(r.tolist())) == 3]
        pats += [tuple(r[:2]) for r in pats[:500]] + [(int(x),) for x in rng.integers(0, nv, 100)]
    return nv, pats


@pytest.mark.parametrize("kind", ["hub", "chunk_edges", "sparse", "triangles"])
@pytest.mark.parametrize("ratio", [0.6, 1.0, 1.7])        # rho against the mean ratio np / nv
def test_forms_agree(kind, ratio):
    from paper_2504_10937_gb300 import lds
    nv, pats = _network(kind)
    q = 97
    p = max(1, int(ratio * q * len(pats) / nv))
    try:
        lds.set_flow_variant(1)
        want, side1 = lds.pattern_max_flow(nv, pats, p, q)
        lds.set_flow_variant(2)
        got, side2 = lds.pattern_max_flow(nv, pats, p, q)
    finally:
        lds.set_flow_variant(0)
    assert got == want and np.array_equal(side1, side2)

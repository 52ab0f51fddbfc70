"""Triangle queries whose networks are gathered triangle by triangle (a set whose members'
lists are longer than T) and member by member (a small part of T): cliques joined by
bridges, with |T| around the 32-bit words of the gathered marks.  The answer is known in
closed form where nothing joins the cliques (every clique, densest first) and the oracle's
where bridges do; both are exact."""
from fractions import Fraction
from itertools import combinations

import numpy as np
import pytest

from oracle import graph as ograph
from oracle.decomp import ltds_exact

pytestmark = pytest.mark.gpu


def _bridged(sizes, bridged):
    ids = np.random.default_rng(sum(sizes)).permutation(sum(sizes) + 40)      # 40 isolated or bridge ends
    at, e, cliques = 0, [], []
    for s in sizes:
        mem = ids[at:at + s]
        cliques.append(tuple(sorted(int(x) for x in mem)))
        e += list(combinations(cliques[-1], 2))
        if bridged and at:
            e.append((int(ids[at - 1]), int(ids[at])))
        at += s
    u, v = np.array(sorted(tuple(sorted(p)) for p in e), np.int32).T
    return len(ids), u, v, sorted(cliques, key=lambda c: -len(c))


# |T| 1; 31 twice; 69; one clique with most of T; several alike
@pytest.mark.parametrize("sizes", [(3,), (6, 5, 3), (6, 4, 5), (7, 6, 5, 4), (40, 9, 8, 7), (20, 19, 18, 17, 16, 15)])
@pytest.mark.parametrize("bridged", [False, True])
@pytest.mark.parametrize("verify", ["bounds", "core", "whole"])
def test_cliques_are_the_answer(sizes, bridged, verify):
    from paper_2504_10937_gb300 import lds
    n, u, v, cliques = _bridged(sizes, bridged)
    with lds.Graph(n, u, v) as g:
        got = g.topk(len(sizes), "triangle", iters=60, precision="exact", verify=verify)
    if bridged:
        want = [(d, tuple(sorted(int(x) for x in m)))
                for d, m in ltds_exact(n, u, v, ograph.triangles(n, u, v))][:len(sizes)]
    else:
        want = [(Fraction((len(c) - 1) * (len(c) - 2), 6), c) for c in cliques]
    assert [(d, tuple(int(x) for x in m)) for d, m in got] == want


@pytest.mark.parametrize("sizes", [(6, 5, 3), (40, 9, 8, 7)])
def test_compact_numbers(sizes):
    from paper_2504_10937_gb300 import lds
    n, u, v, cliques = _bridged(sizes, True)
    want = np.zeros(n)
    for c in cliques:
        want[list(c)] = (len(c) - 1) * (len(c) - 2) / 6
    with lds.Graph(n, u, v) as g:
        num, den = g.compact_numbers("triangle")
    assert np.array_equal(np.asarray(num) * 6, np.asarray(den) * np.round(want * 6).astype(np.int64))

"""Core and tr-core peels against the oracle where the form changes: whole graphs in
one block (at most 8,192 vertices), the grid-wide form with the one-block tail,
masked subgraphs (through pruning), hubs of many chunks."""
from fractions import Fraction

import numpy as np
import pytest

from oracle import graph as ograph
from oracle import prune as oprune
from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


def _star_cliques(n):
    """A hub joined to everything, and cliques of falling size among the rest."""
    us, vs, off = [np.zeros(n - 1, np.int64)], [np.arange(1, n)], 1
    for s in range(40, 2, -1):
        iu, iv = np.triu_indices(s, 1)
        us.append(iu + off)
        vs.append(iv + off)
        off += s
    key = np.unique(np.concatenate(us) * n + np.concatenate(vs))
    return n, (key // n).astype(np.int32), (key % n).astype(np.int32)


GRAPHS = {
    "solo_small": lambda: synth.gnp_planted(400, 0.05, (20, 12), (0.9, 0.7), seed=3)[:3],
    "solo_limit": lambda: _star_cliques(8192),
    "past_limit": lambda: _star_cliques(8193),
    "grid_tail": lambda: synth.chung_lu(20011, 90000, 2.1, seed=4, n_blocks=3, block_size_range=(30, 200))[:3],
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_core_numbers_match_oracle(name):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    with lds.Graph(n, u, v) as g:
        assert np.array_equal(g.core_numbers("edge"), ograph.core_numbers(n, u, v))


@pytest.mark.parametrize("name", ["solo_small", "solo_limit", "past_limit"])
def test_tr_core_numbers_match_oracle(name):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    tris = ograph.triangles(n, u, v)
    with lds.Graph(n, u, v) as g:
        assert np.array_equal(g.core_numbers("triangle"), ograph.tr_core_numbers(n, tris))


@pytest.mark.parametrize("triangle", [False, True])
@pytest.mark.parametrize("share", [0.3, 0.9])       # of the vertices leave in the first round
@pytest.mark.parametrize("name", ["solo_small", "past_limit"])
def test_masked_peels_match_oracle(name, share, triangle):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    tris = ograph.triangles(n, u, v) if triangle else None
    full = ograph.tr_core_numbers(n, tris) if triangle else ograph.core_numbers(n, u, v)
    out = synth.SplitMix64(9).uniform(n) < share
    # the marked vertices fail rule 2 at once; the others only once the mask lowers
    # their core number below two thirds
    ub = [Fraction(10 ** 6)] * n
    lb = [Fraction(int(c) + 1) if o else Fraction(2 * int(c), 3) for c, o in zip(full, out)]
    _, _, rule1, rule2 = oprune.prune(n, u, v, range(n), [], ub, lb, tris=tris)
    want = np.zeros(n, np.uint8)
    want[sorted(rule1)] = 1
    want[sorted(rule2)] = 2
    with lds.Graph(n, u, v) as g:
        got = g.prune(ub, lb, "triangle" if triangle else "edge")
    assert np.array_equal(got, want)

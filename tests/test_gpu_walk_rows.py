"""The ExtractSG walk where positions have no row of their own (isolated vertices,
vertices in no triangle) and where its table has between 4 and 32 columns (few edges
a vertex): against the oracle and against windows of one candidate."""
import time
from fractions import Fraction

import numpy as np
import pytest

from oracle import extract_sg as osg
from oracle import fw as ofw
from oracle import graph as ograph
from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


def _spread(n, k, u, v, seed):
    """The graph (k, u, v) on k of n vertices, the others isolated."""
    ids = np.sort(np.random.default_rng(seed).permutation(n)[:k])
    return n, ids[np.asarray(u)].astype(np.int64), ids[np.asarray(v)].astype(np.int64)


MOSTLY_ISOLATED = {
    "gnp": lambda: _spread(3000, 300, *synth.gnp_planted(300, 0.02, (15, 10, 8), (0.9, 0.7, 0.95), seed=22)[1:3], 1),
    "ba": lambda: _spread(2500, 400, *synth.barabasi_albert(400, 3, seed=5)[1:], 2),
    "rmat": lambda: _spread(4000, 512, *synth.rmat(9, 6, 0.57, 0.19, 0.19, seed=24, n_cliques=2,
                                                   clique_size_range=(10, 25))[1:3], 3),
    "one_edge": lambda: (70, np.array([3], np.int64), np.array([40], np.int64)),
}


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("triangle", [False, True])
@pytest.mark.parametrize("name", sorted(MOSTLY_ISOLATED))
def test_isolated_vertices_match_oracle(name, triangle, variant):
    from paper_2504_10937_gb300 import lds
    n, u, v = MOSTLY_ISOLATED[name]()
    order = np.lexsort((v, u))
    u, v = u[order], v[order]
    tris = ograph.triangles(n, u, v)
    none = {x: Fraction(0) for x in range(n)}
    for N in (1, 2, 40):
        if triangle:
            R, W, Dn, _ = ofw.fw_tri_exact(n, tris, N)
            want = osg.extract_sg_tri(range(n), tris, W, Dn, none, none)
        else:
            R, W, Dn, _ = ofw.fw_edge_exact(n, u, v, N)
            want = osg.extract_sg_edge(range(n), u, v, W, Dn, none, none)
        with lds.Graph(n, u.astype(np.int32), v.astype(np.int32)) as g:
            g.fw(N, density="triangle" if triangle else "edge", precision="exact", want=())
            try:
                lds.set_extract_variant(variant)
                got = g.extract_sg()
            finally:
                lds.set_extract_variant(0)
        assert got["order"].tolist() == want["order"] and got["cuts"] == want["cuts"]
        assert [sorted(x.tolist()) for x in got["groups"]] == [sorted(x) for x in want["groups"]]
        assert [(Fraction(lo, Dn), Fraction(hi, Dn)) for lo, hi in got["intervals"]] == want["intervals"]


def _cycle(n, chords, seed):
    a = np.arange(n)
    r = np.random.default_rng(seed)
    return n, np.r_[a, r.integers(0, n, chords)].astype(np.int32), np.r_[(a + 1) % n, r.integers(0, n, chords)].astype(np.int32)


def _sparse(n, m, seed):
    r = np.random.default_rng(seed)
    return n, r.integers(0, n, m).astype(np.int32), r.integers(0, n, m).astype(np.int32)


NARROW = {
    "matching": lambda: (60000, np.arange(0, 60000, 2, dtype=np.int32), np.arange(1, 60000, 2, dtype=np.int32)),
    "cycle_chords": lambda: _cycle(50000, 5000, 1),
    "sparse": lambda: _sparse(70000, 50000, 2),
    "two_a_vertex": lambda: _sparse(60000, 110000, 3),
}


@pytest.mark.parametrize("precision", ["exact", "fp64"])
@pytest.mark.parametrize("name", sorted(NARROW))
def test_narrow_windows_match_single_candidates(name, precision):
    from paper_2504_10937_gb300 import lds
    n, u, v = NARROW[name]()
    with lds.Graph(n, u, v) as g:
        nact = n - g.info()["isolated"]
        assert 4 < (64 * (g.m + n) + (1 << 20)) // 8 // nact < 32
        for N in (1, 6, 50):
            g.fw(N, precision=precision, want=())
            many = g.extract_sg()
            try:
                lds.set_extract_variant(1)
                one = g.extract_sg()
            finally:
                lds.set_extract_variant(0)
            assert np.array_equal(one["order"], many["order"]) and one["cuts"] == many["cuts"]
            assert one["intervals"] == many["intervals"]
            assert [len(a) for a in one["groups"]] == [len(a) for a in many["groups"]]
            assert np.array_equal(one["remainder"], many["remainder"])


def test_a_long_chain_of_isolated_vertices_is_quick():
    # every isolated vertex is a candidate, and after binary64 iterations one chain runs
    # over all of them: 8.3 s with a row for each of 2^22 vertices
    from paper_2504_10937_gb300 import lds
    r = np.random.default_rng(3)
    u, v = r.integers(0, 50000, 150000).astype(np.int32), r.integers(0, 50000, 150000).astype(np.int32)
    groups = []
    for n in (1 << 16, 1 << 22):
        with lds.Graph(n, u, v) as g:
            g.fw(100, precision="fp64", want=())
            t = time.perf_counter()
            got = g.extract_sg()
            assert time.perf_counter() - t < 4.0
            # the chain ends at the last vertex, so the last group takes all isolated ones in
            assert sum(len(a) for a in got["groups"]) == n
            groups.append([a.tolist() for a in got["groups"][:-1]])
    assert len(groups[0]) > 1 and groups[0] == groups[1]

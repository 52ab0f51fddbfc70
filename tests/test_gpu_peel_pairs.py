"""tr-core numbers past the one-block sizes, where the whole list is peeled by pairs of
members and round stamps: members taken in one round (cliques, books around a common
edge), in rounds one apart, and skewed graphs.  Integers match the oracle exactly."""
import numpy as np
import pytest

from oracle import graph as ograph
from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu

N = 8300


def _join(parts, n=N):
    u = np.concatenate([p[0] for p in parts])
    v = np.concatenate([p[1] for p in parts])
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key = np.unique(lo.astype(np.int64) * n + hi)
    ring = np.arange(n - 1, dtype=np.int64)                     # no vertex isolated
    key = np.unique(np.concatenate([key, ring * n + ring + 1]))
    return n, (key // n).astype(np.int32), (key % n).astype(np.int32)


def _books():
    """Edges of 1 to 90 common neighbours, every other spine among higher ids."""
    parts, at = [], 0
    for k in range(1, 91):
        pages = np.arange(at + 2, at + 2 + k) if k % 2 else np.arange(at, at + k)
        a, b = (at, at + 1) if k % 2 else (at + k, at + k + 1)
        parts += [(np.r_[np.full(k, a), np.full(k, b), a], np.r_[pages, pages, b])]
        at += k + 2
    return _join(parts)


def _strips():
    """Squared paths (triangles i, i+1, i+2 in a row): taken from both ends, a round each."""
    i = np.arange(0, 6000)
    keep = i % 61 < 59
    return _join([(i[keep], i[keep] + 1), (i[keep], i[keep] + 2)])


def _cliques():
    parts, at = [], 0
    for s in [3, 4, 5, 31, 32, 33, 34, 64, 65, 66, 67, 3, 3, 12] * 4:
        iu, iv = np.triu_indices(s, 1)
        parts += [(iu + at, iv + at)]
        at += s - 1                                             # neighbours share a vertex
    return _join(parts)


GRAPHS = {
    "books": _books,
    "strips": _strips,
    "cliques": _cliques,
    "chung_lu": lambda: synth.chung_lu(20011, 90000, 2.2, seed=6, n_blocks=3, block_size_range=(20, 60))[:3],
    "rmat": lambda: synth.rmat(15, 6, 0.57, 0.19, 0.19, seed=8, n_cliques=3, clique_size_range=(10, 50))[:3],
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_tr_cores_match_oracle(name):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    tris = ograph.triangles(n, u, v)
    assert len(np.unique(np.concatenate([u, v]))) > 8192
    with lds.Graph(n, u, v) as g:
        assert np.array_equal(g.core_numbers("triangle"), ograph.tr_core_numbers(n, tris))

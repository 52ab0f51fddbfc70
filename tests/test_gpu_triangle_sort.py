"""GPU parity of the triangle list and its per-vertex index at the edges of their sorts:
around one block's and one tile's keys, and either side of the width where a triangle
still fits one 64-bit key.  Disjoint cliques give the expected lists in closed form;
whole numbers match exactly."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lds():
    from paper_2504_10937_gb300 import lds as _l
    _l.load()
    return _l


def _cliques(n, sizes, seed, pair_rest):
    """Disjoint cliques on scattered ids; pair_rest joins the other ids two by two."""
    rng = np.random.default_rng(seed)
    ids = rng.permutation(n)
    u, v, tri = [], [], []
    core = np.zeros(n, np.int64)
    at = 0
    for k in sizes:
        mem = np.sort(ids[at:at + k])
        at += k
        e = np.array(list(itertools.combinations(mem, 2)), np.int64)
        u.append(e[:, 0])
        v.append(e[:, 1])
        if k > 2:
            tri.append(np.array(list(itertools.combinations(mem, 3)), np.int64))
        core[mem] = (k - 1) * (k - 2) // 2
    if pair_rest:
        rest = ids[at:]
        rest = rest[: len(rest) // 2 * 2]
        u.append(rest[0::2])
        v.append(rest[1::2])
    t = np.concatenate(tri)
    t = t[np.lexsort((t[:, 2], t[:, 1], t[:, 0]))]
    return np.concatenate(u).astype(np.int32), np.concatenate(v).astype(np.int32), t, core


# |T| 1, 4, 2731 (3|T| just over 8,192), 8,195 and 16,215 (either side of two tiles), 100k
@pytest.mark.parametrize("sizes", [(3,), (4,), (26, 10, 5, 3), (37, 14, 9), (46, 15, 15, 10), (60, 55, 40, 3, 3)])
@pytest.mark.parametrize("n", [257, 1 << 12])
def test_lists_and_cores(lds, sizes, n):
    u, v, t, core = _cliques(n, sizes, sum(sizes) + n, False)
    with lds.Graph(n, u, v) as g:
        assert np.array_equal(g.triangles(), t)
        assert np.array_equal(g.core_numbers("triangle"), core)


@pytest.mark.parametrize("n", [1 << 21, (1 << 21) + 2])
def test_key_width(lds, n):
    sizes = (45, 40, 30, 3)
    u, v, t, core = _cliques(n, sizes, n & 1023, True)
    with lds.Graph(n, u, v) as g:
        assert np.array_equal(g.triangles(), t)
        assert np.array_equal(g.core_numbers("triangle"), core)

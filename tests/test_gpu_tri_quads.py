"""Triangle Frank-Wolfe over quads of c where the layout can go wrong: groups of 1 to
9 triangles (partial quads), one triangle in all, more vertices than the shared
memory holds, several folds, the last choices, both arithmetics."""
import numpy as np
import pytest

from oracle import fw as ofw
from oracle import graph as ograph
from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


def _books():
    """Pairs (a, b) with 1 to 9 common neighbours above both: groups of those sizes."""
    us, vs, off = [], [], 0
    for k in range(1, 10):
        us += [off] + [off] * k + [off + 1] * k
        vs += [off + 1] + list(range(off + 2, off + 2 + k)) * 2
        off += k + 2
    key = np.unique(np.array(us) * off + np.array(vs))
    return off, (key // off).astype(np.int32), (key % off).astype(np.int32)


def _many_triangles(n):
    """n vertices in n / 3 triangles joined by nothing: past the hot set."""
    b = np.arange(0, n, 3)
    u = np.concatenate([b, b, b + 1])
    v = np.concatenate([b + 1, b + 2, b + 2])
    key = np.unique(u * n + v)
    return n, (key // n).astype(np.int32), (key % n).astype(np.int32)


GRAPHS = {
    "one": lambda: (4, np.array([0, 0, 1], np.int32), np.array([1, 3, 3], np.int32)),
    "books": _books,
    "clique_40": lambda: synth.gnp_planted(60, 0.05, (40,), (1.0,), seed=1)[:3],
    "rmat_9": lambda: synth.rmat(9, 8, 0.57, 0.19, 0.19, seed=2, n_cliques=2, clique_size_range=(15, 25))[:3],
    "past_hot": lambda: _many_triangles(60000),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_tri_fw_matches_oracle(name):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    tris = ograph.triangles(n, u, v)
    with lds.Graph(n, u, v) as g:
        for N in (0, 1, 2, 33, 70):
            R, W, Dn, ch = ofw.fw_tri_exact(n, tris, N, record=True)
            got = g.fw(N, density="triangle", precision="exact")
            assert got["D"] == Dn and np.array_equal(got["R"], R) and np.array_equal(got["W"], W)
            if N:
                assert np.array_equal(got["last"], ch[-1].astype(np.uint8))
            r32, W32, _ = ofw.fw_tri_fp32(n, tris, N)
            got = g.fw(N, density="triangle", precision="fp32")
            assert np.array_equal(got["r"], r32.astype(np.float64)) and np.array_equal(got["W"], W32)
            assert np.array_equal(got["R"], np.bincount(tris.reshape(-1), W32.reshape(-1).astype(np.float64),
                                                        minlength=n).astype(np.int64))

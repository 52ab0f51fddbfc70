"""Triangle Frank-Wolfe with part of its vertices staged: sizes around the fewest staged
ids (4,096), triangles that mix staged and other vertices, more vertices than threads,
against the oracle's iterates."""
import numpy as np
import pytest

from oracle import fw as ofw
from oracle import graph as ograph
from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


def _strip(n):
    """0, 1, 2, ...: each vertex joined to the next two, n - 2 triangles."""
    a = np.arange(n - 1)
    u, v = np.r_[a, a[:-1]], np.r_[a + 1, a[:-1] + 2]
    key = np.unique(u * n + v)
    return n, (key // n).astype(np.int32), (key % n).astype(np.int32)


def _power_law(n, m):
    n, u, v, _ = synth.chung_lu(n, m, 2.2, seed=n, n_blocks=3, block_size_range=(20, 60))
    return n, u, v


GRAPHS = {
    "strip_4095": lambda: _strip(4095),        # every id staged
    "strip_4096": lambda: _strip(4096),        # one id past the staged ones
    "strip_4097": lambda: _strip(4097),
    "strip_70000": lambda: _strip(70000),
    "power_law_7k": lambda: _power_law(7001, 21000),
    "power_law_30k": lambda: _power_law(30011, 120000),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_partly_staged_triangles_match_oracle(name):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    u, v = np.asarray(u, np.int64), np.asarray(v, np.int64)
    tris = ograph.triangles(n, u, v)
    with lds.Graph(n, u.astype(np.int32), v.astype(np.int32)) as g:
        assert np.array_equal(g.triangles(), tris)
        for N in (1, 2, 30):
            R, W, Dn, ch = ofw.fw_tri_exact(n, tris, N, record=True)
            got = g.fw(N, density="triangle", precision="exact")
            assert got["D"] == Dn and np.array_equal(got["R"], R) and np.array_equal(got["W"], W)
            assert np.array_equal(got["last"], ch[-1].astype(np.uint8))
            r32, W32, _ = ofw.fw_tri_fp32(n, tris, N)
            got = g.fw(N, density="triangle", precision="fp32")
            assert np.array_equal(got["r"], r32.astype(np.float64)) and np.array_equal(got["W"], W32)
            assert np.array_equal(got["R"], np.bincount(tris.reshape(-1), W32.reshape(-1).astype(np.float64),
                                                        minlength=n).astype(np.int64))

"""GPU parity of ingest at the edges of its sorts and scans: one-block and tiled sizes,
ids at powers of two (the mark of a dropped pair is the largest key), long gaps of
isolated vertices.  Whole-number outputs match the oracle exactly."""
import numpy as np
import pytest

from oracle import fw as ofw
from oracle import graph as ograph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lds():
    from paper_2504_10937_gb300 import lds as _l
    _l.load()
    return _l


def _check(lds, n, a, b, fw=False):
    a, b = np.asarray(a, np.int32), np.asarray(b, np.int32)
    cu, cv = ograph.canonical_edges(n, a, b)
    deg = ograph.degrees(n, cu, cv)
    with lds.Graph(n, a, b) as g:
        gu, gv = g.edges()
        assert np.array_equal(gu, cu) and np.array_equal(gv, cv)
        info = g.info()
        loops = int(np.sum(a == b))
        assert (info["m"], info["self_loops"]) == (len(cu), loops)
        assert info["duplicates"] == len(a) - loops - len(cu)
        assert info["max_degree"] == int(deg.max(initial=0))
        assert info["isolated"] == int(np.sum(deg == 0))
        if fw:
            for variant in (0, 1):
                lds.set_fw_variant(variant)
                try:
                    got = g.fw(2)
                finally:
                    lds.set_fw_variant(0)
                R, W, D, _ = ofw.fw_edge_exact(n, cu, cv, 2)
                assert got["D"] == D and np.array_equal(got["R"], R) and np.array_equal(got["W"], W)


@pytest.mark.parametrize("pairs", [1, 15, 16, 17, 511, 512, 513, 4095, 4096, 4097, 20001])
@pytest.mark.parametrize("n", [2, 255, 256, 257, 65536, 65537])
def test_sort_sizes(lds, n, pairs):
    rng = np.random.default_rng(n * 31 + pairs)
    a, b = rng.integers(0, n, pairs), rng.integers(0, n, pairs)
    a[-1], b[-1] = n - 1, n - 1                      # the top key itself
    if pairs > 1:
        a[0], b[0] = n - 1, n - 2
    _check(lds, n, a, b, fw=pairs <= 513)


@pytest.mark.parametrize("n", [1, 8191, 8192, 8193, 16383, 16384, 16385, 3_000_001])
def test_scan_sizes_and_gaps(lds, n):
    rng = np.random.default_rng(n)
    ids = np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, 9)]))
    a, b = rng.choice(ids, 40), rng.choice(ids, 40)
    _check(lds, n, a, b, fw=n < 10_000)


def test_flag_word_scan_sizes(lds):
    # 32 flags a word: 16,384 words and one more
    for pairs in (262_143, 262_144, 262_145):
        rng = np.random.default_rng(pairs)
        _check(lds, 100_000, rng.integers(0, 100_000, pairs), rng.integers(0, 100_000, pairs))


@pytest.mark.parametrize("bad", [-1, 64, 2**31 - 1, -2**31])
def test_bad_ids_are_refused(lds, bad):
    for pairs in (1, 5000):
        a = np.arange(pairs, dtype=np.int32) % 64
        b = np.full(pairs, 1, np.int32)
        for arr in (a, b):
            keep = arr[-1]
            arr[-1] = bad
            with pytest.raises(lds.LdsError) as e:
                lds.Graph(64, a, b)
            assert e.value.status == lds.EINVAL
            arr[-1] = keep

"""The register-resident Frank-Wolfe against the cooperative pass, bit for bit, at the
edges of its launch shapes: one CTA, a cluster, the grid; rows longer than a CTA's
share; the last graph that fits the shared memory and the first that does not."""
import numpy as np
import pytest

from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


def _ring(n, extra=0):
    """A cycle of n vertices plus `extra` chords: exactly n + extra edges."""
    u = np.arange(n)
    v = (u + 1) % n
    cu = np.arange(extra) % (n - 3)
    cv = cu + 2 + np.arange(extra) // (n - 3)
    a, b = np.concatenate([u, cu]), np.concatenate([v, cv])
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    key = np.unique(lo * n + hi)
    return n, (key // n).astype(np.int32), (key % n).astype(np.int32)


def _hub(n):
    """A star inside a cycle: one row of n - 1 slots."""
    u = np.concatenate([np.zeros(n - 1, np.int64), np.arange(1, n - 1)])
    v = np.concatenate([np.arange(1, n), np.arange(2, n)])
    key = np.unique(u * n + v)
    return n, (key // n).astype(np.int32), (key % n).astype(np.int32)


GRAPHS = {
    "edge": lambda: (5, np.array([1], np.int32), np.array([3], np.int32)),
    "block_limit": lambda: _ring(1000, 1048),            # 4,096 slots
    "past_block": lambda: _ring(1000, 1049),
    "cluster_limit": lambda: _ring(4000, 6240),          # 20,480 slots
    "past_cluster": lambda: _ring(4000, 6241),
    "hub_row": lambda: _hub(9001),                       # a CTA of 9,000 slots and more
    "hub_too_long": lambda: _hub(17001),                 # past 16,384: not resident
    "smem_limit": lambda: _ring(54001),                  # words and row counts of a CTA just fit
    "past_smem": lambda: _ring(57500),
    "power_law": lambda: synth.chung_lu(20003, 150000, 2.2, seed=3, n_blocks=2, block_size_range=(100, 300))[:3],
}


@pytest.mark.parametrize("precision", ["exact", "fp32"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_resident_matches_the_pass(name, precision):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    with lds.Graph(n, u, v) as g:
        for N in (1, 2, 37):
            try:
                lds.set_fw_variant(5)
                want = g.fw(N, precision=precision)
            finally:
                lds.set_fw_variant(0)
            got = g.fw(N, precision=precision)
            kernel = g.fw_timing()["pass_kernel"]
            assert (kernel == "fw_resident_kernel") == (name not in ("hub_too_long", "past_smem"))
            assert got["D"] == want["D"]
            for k in ("r", "R", "W", "last"):
                assert np.array_equal(got[k], want[k]), (N, k)


@pytest.mark.parametrize("name", ["edge", "block_limit", "past_block", "past_cluster", "hub_row", "power_law"])
def test_resident_binary64_matches_the_launches(name):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    with lds.Graph(n, u, v) as g:
        for N in (1, 2, 37):
            try:
                lds.set_fw_variant(5)
                want = g.fw(N, precision="fp64")
                assert g.fw_timing()["pass_kernel"] == "fw64_slot_kernel"
            finally:
                lds.set_fw_variant(0)
            got = g.fw(N, precision="fp64")
            kernel = g.fw_timing()["pass_kernel"]
            assert (kernel == "fw_resident64_kernel") == (name != "hub_row")
            for k in ("r", "R", "W", "last"):
                assert np.array_equal(got[k], want[k]), (N, k)

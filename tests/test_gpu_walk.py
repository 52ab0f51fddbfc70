"""The windowed ExtractSG walk against itself one candidate at a time, at sizes
where a window can go wrong: more candidates than a window's 32 columns, chains
over several windows, runs of accepted single candidates, one block and many."""
import numpy as np
import pytest

from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu

GRAPHS = {
    "one_edge": lambda: (3, np.array([0], np.int32), np.array([2], np.int32)),
    "gnp_33": lambda: synth.gnp_planted(33, 0.15, (6,), (0.9,), seed=5)[:3],
    "gnp_2000": lambda: synth.workload_planted_gnp(seed=1)[:3],
    "power_law_5000": lambda: synth.chung_lu(5003, 20000, 2.2, seed=6, n_blocks=3, block_size_range=(10, 60))[:3],
    "ba_9000": lambda: synth.barabasi_albert(9001, 4, seed=7),
    "rmat_11": lambda: synth.rmat(11, 8, 0.57, 0.19, 0.19, seed=8, n_cliques=2, clique_size_range=(15, 30))[:3],
    # disjoint cliques of falling size: every candidate accepted on its own
    "cliques": lambda: _cliques(range(3, 60)),
}


def _cliques(sizes):
    us, vs, off = [], [], 0
    for s in sizes:
        iu, iv = np.triu_indices(s, 1)
        us.append(iu + off)
        vs.append(iv + off)
        off += s
    return off, np.concatenate(us).astype(np.int32), np.concatenate(vs).astype(np.int32)


@pytest.mark.parametrize("density", ["edge", "triangle"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_windows_match_single_candidates(name, density):
    from paper_2504_10937_gb300 import lds
    n, u, v = GRAPHS[name]()
    with lds.Graph(n, u, v) as g:
        for N in (1, 6, 80):
            g.fw(N, density=density, want=())
            try:
                lds.set_extract_variant(1)
                one = g.extract_sg()
                lds.set_extract_variant(0)
                many = g.extract_sg()
            finally:
                lds.set_extract_variant(0)
            assert np.array_equal(one["order"], many["order"]) and one["cuts"] == many["cuts"]
            assert one["intervals"] == many["intervals"] and one["D"] == many["D"]
            assert [len(a) for a in one["groups"]] == [len(a) for a in many["groups"]]
            assert np.array_equal(one["remainder"], many["remainder"])

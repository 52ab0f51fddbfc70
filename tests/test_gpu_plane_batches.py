"""Frank-Wolfe over quads in several launches: the iterates go on where a launch ended
(load words, exact loads), the fold adds onto weights that are not zero, and the last
choices come from a later batch of planes."""
import numpy as np
import pytest

from oracle import fw as ofw
from oracle import graph as ograph
from paper_2504_10937_gb300 import synth

pytestmark = pytest.mark.gpu


def _power_law():
    n, u, v, _ = synth.chung_lu(900, 4000, 2.2, seed=31, n_blocks=2, block_size_range=(12, 40))
    return n, np.asarray(u, np.int64), np.asarray(v, np.int64)


@pytest.mark.parametrize("N", [512, 513, 1100, 1200])
def test_edge_quads_over_several_launches_match_oracle(N):
    from paper_2504_10937_gb300 import lds
    n, u, v = _power_law()
    with lds.Graph(n, u.astype(np.int32), v.astype(np.int32)) as g:
        try:
            lds.set_fw_variant(5)
            exact, fp32 = g.fw(N, precision="exact"), g.fw(N, precision="fp32")
            assert g.fw_timing()["pass_kernel"] == "fw_quad_kernel"
            launches = lds.launch_count()
            g.fw(N, precision="exact", want=())
            assert lds.launch_count() - launches >= 2 * -(-N // 512)          # passes and folds
        finally:
            lds.set_fw_variant(0)
    R, W, Dn, ch = ofw.fw_edge_exact(n, u, v, N, record=True)
    assert exact["D"] == Dn and np.array_equal(exact["R"], R) and np.array_equal(exact["W"], W)
    assert np.array_equal(exact["r"], R / Dn) and np.array_equal(exact["last"].astype(bool), ch[-1])
    r32, W32, _ = ofw.fw_edge_fp32(n, u, v, N)
    assert np.array_equal(fp32["r"], r32.astype(np.float64)) and np.array_equal(fp32["W"], W32)
    assert np.array_equal(fp32["R"], ofw.edge_loads_from_W(n, u, v, W32, Dn))


@pytest.mark.parametrize("N", [512, 513, 1100])
def test_triangle_quads_over_several_launches_match_oracle(N):
    from paper_2504_10937_gb300 import lds
    n, u, v = _power_law()
    tris = ograph.triangles(n, u, v)
    with lds.Graph(n, u.astype(np.int32), v.astype(np.int32)) as g:
        exact = g.fw(N, density="triangle", precision="exact")
        fp32 = g.fw(N, density="triangle", precision="fp32")
    R, W, Dn, ch = ofw.fw_tri_exact(n, tris, N, record=True)
    assert exact["D"] == Dn and np.array_equal(exact["R"], R) and np.array_equal(exact["W"], W)
    assert np.array_equal(exact["last"], ch[-1].astype(np.uint8))
    r32, W32, _ = ofw.fw_tri_fp32(n, tris, N)
    assert np.array_equal(fp32["r"], r32.astype(np.float64)) and np.array_equal(fp32["W"], W32)
    assert np.array_equal(fp32["R"], np.bincount(tris.reshape(-1), W32.reshape(-1).astype(np.float64),
                                                 minlength=n).astype(np.int64))


@pytest.mark.parametrize("density", ["edge", "triangle"])
def test_padded_quads_in_batches_of_few_planes_match_one_after_the_other(density):
    # sizes at which the planes' bytes, not 512, bound a batch: the same state from N
    # iterations in one call as the oracle's on one component
    from paper_2504_10937_gb300 import lds
    k, N = 120_000, 601
    b = np.arange(0, 3 * k, 3, dtype=np.int32)
    u, v = (b, b + 1) if density == "edge" else (np.r_[b, b, b + 1], np.r_[b + 1, b + 2, b + 2])
    with lds.Graph(3 * k, u, v) as g:
        got = g.fw(N, density=density, precision="exact")
        assert g.fw_timing()["pass_kernel"] == ("fw_quad_kernel" if density == "edge" else "fw_tri_quad_kernel")
    if density == "edge":
        R, W, Dn, ch = ofw.fw_edge_exact(2, np.array([0]), np.array([1]), N, record=True)
        assert np.array_equal(got["R"].reshape(k, 3), np.tile(np.r_[R, 0], (k, 1)))
        assert np.array_equal(got["W"], np.full(k, W[0])) and (got["last"] == int(ch[-1][0])).all()
    else:
        R, W, Dn, ch = ofw.fw_tri_exact(3, np.array([[0, 1, 2]]), N, record=True)
        assert np.array_equal(got["R"].reshape(k, 3), np.tile(R, (k, 1)))
        assert np.array_equal(got["W"].reshape(k, 3), np.tile(W[0], (k, 1))) and (got["last"] == int(ch[-1][0])).all()
    assert got["D"] == Dn

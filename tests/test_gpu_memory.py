"""Device memory that the library keeps between calls: how much is held and used, that it
is given back, that a reset device starts anew, and that the walk of ExtractSG and the
choice planes of Frank-Wolfe keep to their bounds."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lds():
    from paper_2504_10937_gb300 import lds as _l
    _l.load()
    return _l


def _random(n, m, seed):
    r = np.random.default_rng(seed)
    return n, r.integers(0, n, m).astype(np.int32), r.integers(0, n, m).astype(np.int32)


def test_kept_memory_is_given_back(lds):
    import torch
    torch.cuda.init()
    g = lds.Graph(*_random(200_000, 4_000_000, 1))
    g.fw(20, want=())
    info = lds.memory_info()
    assert info["held"] >= info["peak"] >= info["in_use"] > 8 * g.m
    g.close()
    lds.release_memory()
    free0 = torch.cuda.mem_get_info()[0]
    g = lds.Graph(*_random(200_000, 4_000_000, 1))
    g.core_numbers()
    used = lds.memory_info()
    assert torch.cuda.mem_get_info()[0] <= free0 - used["in_use"]
    g.close()
    info = lds.memory_info()
    assert info["in_use"] <= used["in_use"] and info["held"] <= torch.cuda.mem_get_info()[1] // 32
    lds.release_memory()
    info = lds.memory_info()
    assert info["held"] - info["in_use"] < (64 << 20)
    assert torch.cuda.mem_get_info()[0] >= free0 - (64 << 20)


def test_frees_on_a_stream_of_its_own_are_done_when_the_handle_goes(lds):
    import torch
    before = lds.memory_info()["in_use"]
    s = torch.cuda.Stream()
    g = lds.Graph(*_random(100_000, 1_000_000, 2), stream=s.cuda_stream)
    g.topk(2, "edge", 20)
    assert lds.memory_info()["in_use"] > before
    g.close()
    assert lds.memory_info()["in_use"] == before


def test_release_while_a_handle_is_alive(lds):
    with lds.Graph(*_random(50_000, 300_000, 3)) as g:
        want = g.topk(3, "edge", 50)
        lds.release_memory()
        got = g.topk(3, "edge", 50)
        assert [(d, c.tolist()) for d, c in got] == [(d, c.tolist()) for d, c in want]


RESET = r"""
import ctypes, numpy as np
from paper_2504_10937_gb300 import lds
rt = ctypes.CDLL("libcudart.so")
r = np.random.default_rng(1)
u, v = r.integers(0, 3000, 20000).astype(np.int32), r.integers(0, 3000, 20000).astype(np.int32)
def go():
    with lds.Graph(3000, u, v) as g:
        a = int(g.fw(20)["R"].sum()), [(d, c.tolist()) for d, c in g.topk(2, "edge", 30)]
    assert lds.memory_info()["held"] > 0
    return a
want = go()
for _ in range(3):
    assert rt.cudaDeviceReset() == 0
    assert go() == want
lds.release_memory()
assert lds.memory_info()["held"] == 0
print("reset ok")
"""


def test_a_reset_device_starts_anew():
    env = dict(os.environ, PYTHONPATH=ROOT)
    env["LD_LIBRARY_PATH"] = "/usr/local/cuda/lib64:" + env.get("LD_LIBRARY_PATH", "")
    out = subprocess.run([sys.executable, "-c", RESET], env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and "reset ok" in out.stdout, out.stdout + out.stderr


@pytest.mark.parametrize("n,m", [(1 << 20, 200_000), (1 << 22, 100_000), (300_000, 150_000)])
def test_the_walk_keeps_to_its_bound(lds, n, m):
    # the table 64 B per edge and vertex and 1 MB, its other arrays 64 B per vertex and 32 per
    # active one, 8 more for the edges' numbers that stay on the handle; 256 B more a buffer
    with lds.Graph(*_random(n, m, 4)) as g:
        g.fw(30, want=())
        nact = n - g.info()["isolated"]
        before = lds.memory_info()["in_use"]
        lds.memory_info()
        g.extract_sg()
        grown = lds.memory_info()["peak"] - before
        assert grown <= 64 * (g.m + n) + (1 << 20) + 64 * n + 40 * nact + 32 * 256


def test_planes_of_padded_quads_keep_to_their_bound(lds):
    # one target a row, one triangle a group: every quad holds one entry.  Planes, weights
    # per entry (16 B a quad and plane set), loads and counts of the vertices, and the
    # results themselves, of which the last are replaced
    n = 1 << 20
    with lds.Graph(n, np.arange(0, n, 2, dtype=np.int32), np.arange(1, n, 2, dtype=np.int32)) as g:
        g.fw(1, want=())
        before = lds.memory_info()["in_use"]
        lds.memory_info()
        g.fw(600, want=())
        assert g.fw_timing()["pass_kernel"] == "fw_quad_kernel"
        assert lds.memory_info()["peak"] - before <= (96 + 16) * g.m + 16 * n + (1 << 20)
    t = 300_000
    b = np.arange(0, 3 * t, 3, dtype=np.int32)
    with lds.Graph(3 * t, np.r_[b, b, b + 1], np.r_[b + 1, b + 2, b + 2]) as g:
        g.fw(1, density="triangle", want=())
        before = lds.memory_info()["in_use"]
        lds.memory_info()
        g.fw(600, density="triangle", want=())
        assert lds.memory_info()["peak"] - before <= (192 + 32) * t + 16 * 3 * t + (1 << 20)

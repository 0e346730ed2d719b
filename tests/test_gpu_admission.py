"""The device memory a server reserves for a request covers its handle: sparse
and skewed graphs, cliques on both sides of every form of the lists of
higher-priority neighbours, a star, and nodes without edges."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402
from paper_2010_14058_gb300 import serve  # noqa: E402


def _dense(n, density, L):
    iu, ju = np.triu_indices(n, 1)
    keep = np.random.default_rng(n).random(len(iu)) < density
    return graphgen.csr_from_edges(n, iu[keep].astype(np.int32), ju[keep].astype(np.int32),
                                   (np.arange(n) % L).astype(np.uint8), L, "dense")


def _star(leaves, n, L):
    return graphgen.csr_from_edges(n, np.zeros(leaves, np.int32), np.arange(1, leaves + 1, dtype=np.int32),
                                   (np.arange(n) % L).astype(np.uint8), L, "star")


def _core(n, sparse, degree, L):
    """A clique whose nodes have neighbours of low degree too."""
    iu, ju = np.triu_indices(n, 1)
    rng = np.random.default_rng(n)
    eu = np.concatenate([iu, rng.integers(0, n, sparse * degree)]).astype(np.int64)
    ev = np.concatenate([ju, n + rng.integers(0, sparse, sparse * degree)]).astype(np.int64)
    key = np.unique(eu * (n + sparse) + ev)
    return graphgen.csr_from_edges(n + sparse, (key // (n + sparse)).astype(np.int32), (key % (n + sparse)).astype(np.int32),
                                   (np.arange(n + sparse) % L).astype(np.uint8), L, "core")


GRAPHS = {
    "cl_1k": lambda L: graphgen.chung_lu(200, 1000, 2.2, 40.0, L, 5),
    "cl_100k": lambda L: graphgen.chung_lu(20_000, 100_000, 2.2, 1200.0, L, 5),
    "cl_1m": lambda L: graphgen.chung_lu(200_000, 1_000_000, 2.1, 8000.0, L, 5),
    "er": lambda L: graphgen.erdos_renyi(5000, 40_000, L, 7),
    **{f"clique_{n}": (lambda n: lambda L: _dense(n, 1.0, L))(n) for n in (34, 100, 130, 300, 705, 707, 1500)},
    "dense_1500": lambda L: _dense(1500, 0.6, L),
    "core": lambda L: _core(300, 2500, 5, L),
    "star": lambda L: _star(70_000, 70_001, L),
    "alone": lambda L: _star(10, 300_000, L),
}


@pytest.mark.parametrize("L", [1, 5, 8])
@pytest.mark.parametrize("name", GRAPHS)
def test_reservation_covers_the_handle(name, L):
    g = GRAPHS[name](L)
    rp, col, ty = tg.to_device(g)
    h = tg.tg_build(rp, col, ty, L)
    tg.tg_count(h, 4, None, torch.empty(tg.tg_layout(L, 4)["global_slots"], dtype=torch.int64, device="cuda"))
    assert tg.tg_query_status(h) == 0
    request = serve.Request(0, L, g["row_ptr"], g["col"], g["types"])
    used = h.device_bytes
    h.free()
    assert used <= request.bytes_needed()
    # and the bound itself is one, without the bytes that the sizes alone reserve
    assert used <= serve.handle_bytes(np.diff(g["row_ptr"]), g["m"], L) + (1 << 20)

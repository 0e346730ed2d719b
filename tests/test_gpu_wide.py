"""Graphs with a degree of 2^16 and more: sampled 4-node rows against the
oracle, and the device memory of a count per edge and node (sums over the
triangle nodes of an edge are bounded by the adjacency entries, so they take
32 bits whatever the degrees)."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402


def book(pages, L):
    """Two adjacent hubs and `pages` common neighbours, joined in chains of eight: triangles and 4-cliques at the hubs' edge."""
    p = np.arange(2, pages + 2)
    chain = p[:-1][(p[:-1] - 2) % 8 < 7]
    eu = np.concatenate([[0], np.zeros(pages), np.ones(pages), chain]).astype(np.int32)
    ev = np.concatenate([[1], p, p, chain + 1]).astype(np.int32)
    return graphgen.csr_from_edges(pages + 2, eu, ev, (np.arange(pages + 2) % L).astype(np.uint8), L, "book")


@pytest.mark.parametrize("pages,L", [(65534, 8), (65535, 8), (70000, 3), (70000, 8), (70000, 1)])
def test_rows_and_memory(pages, L):
    g = book(pages, L)
    rp, col, ty = tg.to_device(g)
    lay = tg.tg_layout(L, 4)
    h = tg.tg_build(rp, col, ty, L)
    rows = torch.full((h.m, lay["per_edge_slots"]), -1, dtype=torch.int32, device="cuda")
    tg.tg_count(h, 4, rows, None)
    assert tg.tg_query_status(h) == 0
    tables = 3 * 2 * g["n"] * 4 * L                          # three buffers of the two hubs' counters
    assert h.device_bytes <= (40 * L * L + 96) * g["m"] + (16 * L * L + 192) * g["n"] + tables + (1 << 20)
    ids = np.unique(np.concatenate([[0, 1, pages, pages + 1, g["m"] - 1], np.random.default_rng(3).integers(0, g["m"], 40)]))
    want, _ = oracle.paper_edges(g, ids)
    got = rows[torch.as_tensor(ids, device="cuda")].cpu().numpy().view(np.uint32).astype(np.int64)
    np.testing.assert_array_equal(got, np.minimum(want, 2**32 - 1))
    h.free()

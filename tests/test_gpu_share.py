"""Triangles of nodes of short lists: one, two or eight warps per node by the
number of nodes (at the sizes where the rule changes) give the same rows."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402

N, L = 300, 4


@pytest.fixture(scope="module")
def graph():
    g = graphgen.chung_lu(N, 4200, 2.3, 90.0, L, 77)          # lists of 1 to more than 32 nodes
    return g, oracle.paper(g)


@pytest.mark.parametrize("warps,more", [(8, 0), (8, 1), (2, 0), (2, 1)])
def test_same_rows_at_the_lines(graph, warps, more):
    g, (rows, totals) = graph
    n = torch.cuda.get_device_properties(0).multi_processor_count * 64 // warps + more
    big = dict(g, row_ptr=np.concatenate([g["row_ptr"], np.full(n - N, g["row_ptr"][-1])]),
               types=np.concatenate([g["types"], np.zeros(n - N, dtype=np.uint8)]))   # nodes without edges
    rp, col, ty = tg.to_device(big)
    h = tg.tg_build(rp, col, ty, L)
    for k in (3, 4):
        lay = tg.tg_layout(L, k)
        per = torch.zeros((h.m, lay["per_edge_slots"]), dtype=torch.int32, device="cuda")
        tot = torch.zeros(lay["global_slots"], dtype=torch.int64, device="cuda")
        tg.tg_count(h, k, per, tot)
        got = per.cpu().numpy().view(np.uint32).astype(np.int64)
        np.testing.assert_array_equal(got, rows if k == 4 else rows[:, :2 * L])
        np.testing.assert_array_equal(tot.cpu().numpy(), totals[:lay["global_slots"]])
    assert tg.tg_query_status(h) == 0
    h.free()

"""Directed and edge-typed counts whose triangle cells exceed their budget:
the edges are counted in windows, with the rows and totals of one window, and
the handle takes no more memory than the budget for the cells."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402

BUDGET = 4 << 20                                             # of cycle_budget_mb = 1


def _directed(g, L, options):
    src = np.repeat(np.arange(g["n"]), np.diff(g["row_ptr"]))
    keep = (src < g["col"]) == ((src + g["col"]) % 3 > 0)    # one arc per edge
    tail, head = src[keep], g["col"][keep]
    rp = np.concatenate([[0], np.cumsum(np.bincount(tail, minlength=g["n"]))]).astype(np.int64)
    h = tg.tg_build_directed(torch.as_tensor(rp, device="cuda"), torch.as_tensor(head, device="cuda"),
                             torch.as_tensor(g["types"], device="cuda"), L, options=options)
    return h, tg.tg_directed_layout(L), tg.tg_count_directed3


def _edge_typed(g, L, options):
    rp, col, ty = tg.to_device(g)
    xi = torch.as_tensor(graphgen.edge_types(g, 4, 5), device="cuda")
    return tg.tg_build_edge_typed(rp, col, ty, xi, L, 4, options=options), tg.tg_edge_typed_layout(L, 4), tg.tg_count_edge_typed3


def _count(make, g, L, options, with_rows):
    h, lay, count = make(g, L, options)
    rows = torch.full((h.m, lay["per_edge_slots"]), -1, dtype=torch.int32, device="cuda") if with_rows else None
    totals = torch.full((lay["global_slots"],), -1, dtype=torch.int64, device="cuda")
    before = h.device_bytes
    for _ in range(2):
        count(h, rows, totals)
    assert tg.tg_query_status(h) == 0
    grown = h.device_bytes - before
    h.free()
    return None if rows is None else rows.cpu().numpy(), totals.cpu().numpy(), grown


# edges of a window: 32,768 (L = 8), 52,428 (L = 5), 262,144 (L = 1); edge-typed 13,107, 20,971 and 104,857
@pytest.mark.parametrize("m", [20_000, 104_857, 104_858, 130_000])
@pytest.mark.parametrize("make,L", [(_directed, 8), (_directed, 5), (_directed, 1), (_edge_typed, 8), (_edge_typed, 5),
                                    (_edge_typed, 1)])
def test_windows_give_the_same_counts(make, L, m):
    g = graphgen.chung_lu(m // 8, m, 2.2, 400.0, L, 17)
    rows, totals, _ = _count(make, g, L, None, True)
    for with_rows in (True, False):
        r, t, grown = _count(make, g, L, {"cycle_budget_mb": 1}, with_rows)
        assert grown <= BUDGET
        np.testing.assert_array_equal(t, totals)
        if with_rows:
            np.testing.assert_array_equal(r, rows)

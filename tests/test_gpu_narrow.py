"""4-node rows in 32-bit arithmetic (graphs whose typed degrees stay below
2^15) against 64-bit arithmetic: the same graph counted by itself and beside
a star that takes the handle over the line, and the largest products on both
sides of the line."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402

LINE = 1 << 15


def _csr(n, edges, types, L):
    src = np.concatenate([edges[:, 0], edges[:, 1]])
    dst = np.concatenate([edges[:, 1], edges[:, 0]])
    o = np.lexsort((dst, src))
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(src, minlength=n), out=rp[1:])
    return {"row_ptr": rp, "col": dst[o].astype(np.int32), "types": np.asarray(types, dtype=np.uint8), "L": L}


def _edges(g):
    src = np.repeat(np.arange(len(g["types"])), np.diff(g["row_ptr"]))
    keep = src < g["col"]
    return np.stack([src[keep], g["col"][keep]], axis=1).astype(np.int64)


def _count(g, pa):
    rp, col, ty = tg.to_device(g)
    h = tg.tg_build(rp, col, ty, g["L"])
    lay = tg.tg_pa_layout(g["L"]) if pa else tg.tg_layout(g["L"], 4)
    rows = torch.zeros((h.m, lay["per_edge_slots"]), dtype=torch.int32, device="cuda")
    totals = torch.zeros(lay["global_slots"], dtype=torch.int64, device="cuda")
    if pa:
        tg.tg_count_position_aware(h, rows, totals)
    else:
        tg.tg_count(h, 4, rows, totals)
    assert tg.tg_query_status(h) == 0
    out = rows.cpu().numpy().view(np.uint32).astype(np.int64), totals.cpu().numpy()
    h.free()
    return out


@pytest.mark.parametrize("pa", [False, True])
@pytest.mark.parametrize("L", range(1, 9))
def test_same_rows_in_both_widths(L, pa):
    g = graphgen.chung_lu(400, 5000, 2.2, 150.0, L, 700 + L)
    n, e = len(g["types"]), _edges(g)
    alone, totals = _count(g, pa)
    for leaves in (LINE - 1, LINE):                          # the last narrow and the first wide handle
        star = np.stack([np.full(leaves, n), np.arange(n + 1, n + 1 + leaves)], axis=1)
        types = np.concatenate([g["types"], np.zeros(1 + leaves, dtype=np.uint8)])
        rows, total = _count(_csr(n + 1 + leaves, np.concatenate([e, star]), types, L), pa)
        np.testing.assert_array_equal(rows[:len(e)], alone)
        if pa:
            continue
        # a star adds one edge, one 3-path and one 4-star class, of the one type
        extra = np.sort((total - totals)[total != totals])
        np.testing.assert_array_equal(extra, [leaves, leaves * (leaves - 1) // 2,
                                              leaves * (leaves - 1) * (leaves - 2) // 6])


@pytest.mark.parametrize("over", [0, 1])
def test_largest_products(over):
    """Two adjacent hubs of type 0, each with leaves of both types up to the line, or one leaf past it."""
    a = [LINE - 2 + over, LINE - 1]                          # (the other hub is a neighbour of type 0 too)
    b = [LINE - 2, LINE - 1]
    edges, types = [[0, 1]], [0, 0]
    for hub, leaves in ((0, a), (1, b)):
        for t in (0, 1):
            edges += [[hub, len(types) + k] for k in range(leaves[t])]
            types += [t] * leaves[t]
    g = _csr(len(types), np.array(edges, dtype=np.int64), types, 2)
    rows, _ = _count(g, False)
    row = rows[0]                                            # edge (0, 1) comes first
    P = 3                                                    # pairs (0,0), (0,1), (1,1)
    np.testing.assert_array_equal(row[:4], [a[0] + b[0], a[1] + b[1], 0, 0])
    np.testing.assert_array_equal(row[4 + P:4 + 2 * P],      # 4-paths centred at the edge
                                  [a[0] * b[0], a[0] * b[1] + a[1] * b[0], a[1] * b[1]])
    np.testing.assert_array_equal(row[4 + 2 * P:4 + 3 * P],  # 4-stars centred at either end
                                  [(a[0] * (a[0] - 1) + b[0] * (b[0] - 1)) // 2, a[0] * a[1] + b[0] * b[1],
                                   (a[1] * (a[1] - 1) + b[1] * (b[1] - 1)) // 2])
    assert row[4 + 3 * P:].sum() == 0

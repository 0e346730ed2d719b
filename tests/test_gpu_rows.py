"""Rows and totals of every number of types (the per-edge kernels are
instantiated per L and take one unordered type pair per thread): typed and
position-aware rows against the oracle, and ranges that start and end inside
a tile."""
import numpy as np
import pytest

import graphgen
import oracle
from gpu_helpers import gpu_count

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402


@pytest.mark.parametrize("L", range(1, 9))
def test_rows_of_every_type_count(L):
    g = graphgen.chung_lu(150, 1100, 2.2, 60.0, L, 300 + L)
    rows, totals = oracle.paper(g)
    pe, gl, st = gpu_count(g)
    assert st == 0, tg.STATUS[st]
    np.testing.assert_array_equal(pe, rows)
    np.testing.assert_array_equal(gl, totals)
    pe3, gl3, st = gpu_count(g, k=3)
    assert st == 0, tg.STATUS[st]
    np.testing.assert_array_equal(pe3, rows[:, :2 * L])
    np.testing.assert_array_equal(gl3, totals[:len(gl3)])
    rp, col, ty = tg.to_device(g)
    h = tg.tg_build(rp, col, ty, L)
    pa = tg.tg_pa_layout(L)
    per = torch.zeros((h.m, pa["per_edge_slots"]), dtype=torch.int32, device="cuda")
    tot = torch.zeros(pa["global_slots"], dtype=torch.int64, device="cuda")
    tg.tg_count_position_aware(h, per, tot)
    rows_pa, totals_pa = oracle.position_aware(g)
    np.testing.assert_array_equal(per.cpu().numpy().view(np.uint32).astype(np.int64), rows_pa)
    np.testing.assert_array_equal(tot.cpu().numpy(), totals_pa)
    lay = tg.tg_layout(L, 4)
    for b, e in ((0, 1), (3, 70), (63, 65), (1, h.m)):
        part = torch.zeros((e - b, lay["per_edge_slots"]), dtype=torch.int32, device="cuda")
        tg.tg_count_range(h, 4, b, e, part)
        np.testing.assert_array_equal(part.cpu().numpy().view(np.uint32).astype(np.int64), rows[b:e])
    assert tg.tg_query_status(h) == 0
    h.free()

"""Structures that only 4-node counts need are made before the first of them:
every order of 3-node, 4-node, range and position-aware counts on one handle
gives the oracle's rows, also on another stream than the build's."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402


@pytest.mark.parametrize("order", ["343", "r34", "43p", "p3r", "3p4"])
@pytest.mark.parametrize("hub_min_wedges", [1 << 14, 300])
def test_counts_in_any_order(order, hub_min_wedges):
    L = 3
    g = graphgen.chung_lu(200, 1500, 2.2, 80.0, L, 41)
    rows, totals = oracle.paper(g)
    rows_pa, totals_pa = oracle.position_aware(g)
    rp, col, ty = tg.to_device(g)
    h = tg.tg_build(rp, col, ty, L, options={"hub_min_wedges": hub_min_wedges})
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    for what in order:
        with torch.cuda.stream(s):
            k = 3 if what == "3" else 4
            lay = tg.tg_pa_layout(L) if what == "p" else tg.tg_layout(L, k)
            per = torch.zeros((h.m, lay["per_edge_slots"]), dtype=torch.int32, device="cuda")
            tot = torch.zeros(lay["global_slots"], dtype=torch.int64, device="cuda")
            if what == "p":
                tg.tg_count_position_aware(h, per, tot, stream=s)
            elif what == "r":
                tg.tg_count_range(h, 4, 0, h.m, per, stream=s)
            else:
                tg.tg_count(h, k, per, tot, stream=s)
            got = per.cpu().numpy().view(np.uint32).astype(np.int64)
            want = rows_pa if what == "p" else rows[:, :2 * L] if k == 3 else rows
            np.testing.assert_array_equal(got, want)
            if what != "r":
                wt = totals_pa if what == "p" else totals[:lay["global_slots"]]
                np.testing.assert_array_equal(tot.cpu().numpy(), wt)
        assert tg.tg_query_status(h) == 0
    h.free()

"""A call that fails on the host leaves a handle and a runtime that count on:
what the failed call had not launched is launched by the next one.  The
failures are the runtime's own: capturing the legacy stream, and synchronising
a stream that is being captured, both of which it refuses; no kernel of the
failed calls runs."""
import numpy as np
import pytest

import graphgen
import oracle
from capture import captured

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402

LEGACY = 1                                                   # cudaStreamLegacy


def failing_range(h, out, totals, s):
    """A range whose tiles are copied and synchronised while `s` is captured."""
    with captured(s), pytest.raises(tg.TGError):
        tg.tg_count_range(h, 4, 1, h.m - 1, out, totals, stream=s)


@pytest.fixture(scope="module")
def graph():
    g = graphgen.chung_lu(300, 3000, 2.2, 100.0, 3, 8)
    return g, oracle.paper(g)[0]


def test_a_count_after_a_failed_range(graph):
    g, rows = graph
    rp, col, ty = tg.to_device(g)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    lay = tg.tg_layout(g["L"], 4)
    with torch.cuda.stream(s):
        out = torch.full((g["m"], lay["per_edge_slots"]), -1, dtype=torch.int32, device="cuda")
        totals = torch.zeros(lay["global_slots"], dtype=torch.int64, device="cuda")
        h = tg.tg_build(rp, col, ty, g["L"], stream=s)
        tg.tg_count(h, 4, None, totals, stream=s)
        s.synchronize()
        failing_range(h, out, totals, s)
        tg.tg_count(h, 4, out, totals, stream=s)
        s.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32).astype(np.int64), rows)
        assert tg.tg_query_status(h) == 0
        h.free()


@pytest.mark.parametrize("before", [None, 3])
def test_a_range_after_a_failed_range(graph, before):
    g, rows = graph
    rp, col, ty = tg.to_device(g)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    lay = tg.tg_layout(g["L"], 4)
    with torch.cuda.stream(s):
        out = torch.full((g["m"], lay["per_edge_slots"]), -1, dtype=torch.int32, device="cuda")
        totals = torch.zeros(lay["global_slots"], dtype=torch.int64, device="cuda")
        h = tg.tg_build(rp, col, ty, g["L"], stream=s)
        if before:                                           # triangle counts without their sums per node
            tg.tg_count(h, before, None, totals, stream=s)
        s.synchronize()
        with pytest.raises(tg.TGError):                      # every working array is there, and nothing is counted
            tg.tg_count_batch(h, 4, out, totals, stream=LEGACY)
        failing_range(h, out, totals, s)
        tg.tg_count_range(h, 4, 0, h.m, out, stream=s)
        s.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32).astype(np.int64), rows)
        assert tg.tg_query_status(h) == 0
        h.free()

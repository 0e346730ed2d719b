"""Counts captured into a CUDA graph by the caller, as a handle's first: the
handle's working arrays are made meanwhile, are memory of their own (not the
graph's), and serve the replays and the calls after them alike.  Calls that a
capture refuses leave a handle that counts."""
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

L, X = 3, 2


def _graph(clique):
    if not clique:
        return graphgen.chung_lu(300, 3000, 2.2, 100.0, L, 8)
    iu, ju = np.triu_indices(710, 1)                         # lists that only arrays in global memory hold
    return graphgen.csr_from_edges(710, iu.astype(np.int32), ju.astype(np.int32), (np.arange(710) % L).astype(np.uint8),
                                   L, "clique")


def _directed(g, s):
    src = np.repeat(np.arange(g["n"]), np.diff(g["row_ptr"]))
    keep = (src < g["col"]) == ((src + g["col"]) % 3 > 0)    # one arc per edge
    tail, head = src[keep], g["col"][keep]
    rp = np.concatenate([[0], np.cumsum(np.bincount(tail, minlength=g["n"]))]).astype(np.int64)
    ty = torch.as_tensor(g["types"], device="cuda")
    h = tg.tg_build_directed(torch.as_tensor(rp, device="cuda"), torch.as_tensor(head, device="cuda"), ty, L, stream=s)
    return h, tg.tg_directed_layout(L), tg.tg_count_directed3


def _edge_typed(g, s):
    rp, col, ty = tg.to_device(g)
    xi = torch.as_tensor(graphgen.edge_types(g, X, 5), device="cuda")
    return tg.tg_build_edge_typed(rp, col, ty, xi, L, X, stream=s), tg.tg_edge_typed_layout(L, X), tg.tg_count_edge_typed3


@pytest.mark.parametrize("clique", [False, True])
@pytest.mark.parametrize("with_rows", [True, False])
@pytest.mark.parametrize("make", [_directed, _edge_typed])
def test_first_three_node_count_in_a_graph(make, with_rows, clique):
    g = _graph(clique)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        def outputs(h, lay):
            return (torch.full((h.m, lay["per_edge_slots"]), -1, dtype=torch.int32, device="cuda") if with_rows else None,
                    torch.full((lay["global_slots"],), -1, dtype=torch.int64, device="cuda"))

        def values(out):
            s.synchronize()
            return [x.cpu().numpy() for x in out if x is not None]

        h, lay, count = make(g, s)
        want_out = outputs(h, lay)
        count(h, *want_out, stream=s)
        want = values(want_out)
        h.free()
        h, _, _ = make(g, s)
        out = outputs(h, lay)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            count(h, *out, stream=s)
        for _ in range(3):
            [x.fill_(-1) for x in out if x is not None]
            graph.replay()
            for a, b in zip(values(out), want):
                np.testing.assert_array_equal(a, b)
        again = outputs(h, lay)                              # and without the graph
        count(h, *again, stream=s)
        for a, b in zip(values(again), want):
            np.testing.assert_array_equal(a, b)
        [x.fill_(-1) for x in out if x is not None]
        graph.replay()
        for a, b in zip(values(out), want):
            np.testing.assert_array_equal(a, b)
        assert tg.tg_query_status(h) == 0
        s.synchronize()
        del graph
        h.free()


@pytest.mark.parametrize("call", ["3", "4", "pa", "range", "handles"])
def test_counts_after_a_refused_capture(call):
    """A handle's first undirected count synchronises, which a capture refuses; the next one counts."""
    g = _graph(False)
    rows, totals = oracle.paper(g)
    rp, col, ty = tg.to_device(g)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    lay = tg.tg_pa_layout(L) if call == "pa" else tg.tg_layout(L, 3 if call == "3" else 4)
    with torch.cuda.stream(s):
        out = torch.full((g["m"], lay["per_edge_slots"]), -1, dtype=torch.int32, device="cuda")
        gl = torch.zeros(lay["global_slots"], dtype=torch.int64, device="cuda")
        h = tg.tg_build(rp, col, ty, L, stream=s)

        def count():
            if call == "pa":
                tg.tg_count_position_aware(h, out, gl, stream=s)
            elif call == "range":
                tg.tg_count_range(h, 4, 0, h.m, out, stream=s)
            elif call == "handles":
                tg.tg_count_handles([h], 4, gl, stream=s)
            else:
                tg.tg_count(h, int(call), out, gl, stream=s)

        s.synchronize()
        with captured(s), pytest.raises(tg.TGError):
            count()
        count()
        s.synchronize()
        if call == "pa":
            rows, totals = oracle.position_aware(g)
        if call != "handles":
            np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32).astype(np.int64), rows[:, :out.shape[1]])
        if call != "range":
            np.testing.assert_array_equal(gl.cpu().numpy(), totals[:len(gl)])
        assert tg.tg_query_status(h) == 0
        h.free()

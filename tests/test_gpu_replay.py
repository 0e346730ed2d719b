"""A captured batch is replayed after other counts on the same handle: the
working arrays that the graph points to are still the handle's.  A clique of
710 nodes has lists of higher-priority neighbours that only the arrays in
global memory hold.  Between capture and replay other handles take memory
from the library; their rows, and the batch's, stay the same."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402

N, L = 710, 3


def _clique():
    iu, ju = np.triu_indices(N, 1)
    types = (np.arange(N) % L).astype(np.uint8)
    return graphgen.csr_from_edges(N, iu.astype(np.int32), ju.astype(np.int32), types, L, "clique")


def _buffers(h, k, lay=None):
    lay = lay or tg.tg_layout(L, k)
    return (torch.full((h.m, lay["per_edge_slots"]), -1, dtype=torch.int32, device="cuda"),
            torch.full((lay["global_slots"],), -1, dtype=torch.int64, device="cuda"))


def _triangles(rows):
    """Every edge of the clique is in N - 2 triangles and no 3-path."""
    r = rows.cpu().numpy()
    assert (r[:, :L] == 0).all() and (r[:, L:2 * L].sum(1) == N - 2).all()
    return r


@pytest.mark.parametrize("between", [(4,), (3, 4), ("range",), ("sparse",), ("pa",), (4, "pa", "range")])
def test_three_node_batch_replayed_after_other_counts(between):
    rp, col, ty = tg.to_device(_clique())
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        h = tg.tg_build(rp, col, ty, L, stream=s)
        rows, totals = _buffers(h, 3)
        tg.tg_count_batch(h, 3, rows, totals, stream=s)
        s.synchronize()
        want, want_totals = _triangles(rows), totals.cpu().numpy()
        for what in between:
            if what == "range":
                tg.tg_count_range(h, 4, 5, 900, torch.empty((895, _buffers(h, 4)[0].shape[1]), dtype=torch.int32, device="cuda"),
                                  stream=s)
            elif what == "sparse":
                tg.tg_count_sparse(h, 4, torch.empty(h.m + 1, dtype=torch.int64, device="cuda"), stream=s)
            elif what == "pa":
                tg.tg_count_position_aware(h, *_buffers(h, 4, tg.tg_pa_layout(L)), stream=s)
            else:
                tg.tg_count(h, what, *_buffers(h, what), stream=s)
        others = []                                          # what the library has freed is theirs now
        for _ in range(3):
            o = tg.tg_build(rp, col, ty, L, stream=s)
            b = _buffers(o, 4)
            tg.tg_count(o, 4, *b, stream=s)
            others.append((o, b, b[0].cpu().numpy()))
        for _ in range(2):
            rows.fill_(-1), totals.fill_(-1)
            tg.tg_count_batch(h, 3, rows, totals, stream=s)
            s.synchronize()
            np.testing.assert_array_equal(_triangles(rows), want)
            np.testing.assert_array_equal(totals.cpu().numpy(), want_totals)
        for o, b, was in others:                             # rows of a range come from the arrays kept by the handle
            part = torch.full((o.m, was.shape[1]), -1, dtype=torch.int32, device="cuda")
            tg.tg_count_range(o, 4, 0, o.m, part, stream=s)
            s.synchronize()
            np.testing.assert_array_equal(part.cpu().numpy(), was)
            assert tg.tg_query_status(o) == 0
            o.free()
        assert tg.tg_query_status(h) == 0
        h.free()

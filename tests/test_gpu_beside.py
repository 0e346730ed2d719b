"""Kernels of one pass that run beside each other on side streams: the rows
and totals are those of the kernels run one after another (per-kernel timing
on, and a captured batch), also when several threads count on streams of
their own at once, so that sets of side streams are taken, given back and
taken again."""
import threading

import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_14058_gb300 as tg  # noqa: E402

GRAPHS = [(60, 90, 10.0, 2), (400, 6000, 150.0, 3), (3000, 40000, 900.0, 5)]


def _handle(shape, stream=None):
    n, m, wmax, L = shape
    rp, col, ty = tg.to_device(graphgen.chung_lu(n, m, 2.2, wmax, L, 900 + n))
    torch.cuda.synchronize()
    h = tg.tg_build(rp, col, ty, L, stream=stream)
    lay = tg.tg_layout(L, 4)
    return (h, torch.zeros((h.m, lay["per_edge_slots"]), dtype=torch.int32, device="cuda"),
            torch.zeros(lay["global_slots"], dtype=torch.int64, device="cuda"), (rp, col, ty))


def _serial(shape):
    h, rows, totals, _ = _handle(shape)
    tg.tg_set_timing(h, True)
    tg.tg_count(h, 4, rows, totals)
    assert tg.tg_query_status(h) == 0
    out = rows.cpu().numpy(), totals.cpu().numpy()
    h.free()
    return out


@pytest.mark.parametrize("shape", GRAPHS)
def test_beside_equals_one_after_another(shape):
    want = _serial(shape)
    h, rows, totals, keep = _handle(shape)
    for _ in range(3):
        rows.fill_(-1), totals.fill_(-1)
        tg.tg_count(h, 4, rows, totals)
        assert tg.tg_query_status(h) == 0
        np.testing.assert_array_equal(rows.cpu().numpy(), want[0])
        np.testing.assert_array_equal(totals.cpu().numpy(), want[1])
    h.free()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    h = tg.tg_build_batch(np.array([0, shape[0]], dtype=np.int64), *keep, shape[3], stream=s)
    for _ in range(2):                                               # captured, then replayed
        rows.fill_(-1), totals.fill_(-1)
        s.wait_stream(torch.cuda.current_stream())
        tg.tg_count_batch(h, 4, rows, totals, stream=s)
        s.synchronize()
        assert tg.tg_query_status(h) == 0
        np.testing.assert_array_equal(rows.cpu().numpy(), want[0])
        np.testing.assert_array_equal(totals.cpu().numpy(), want[1])
    h.free()


def test_several_threads_at_once():
    want = [_serial(g) for g in GRAPHS]
    failures = []

    def work(k):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                h, rows, totals, _ = _handle(GRAPHS[k % 3], stream)
                for _ in range(6):
                    rows.fill_(-1), totals.fill_(-1)
                    tg.tg_count(h, 4, rows, totals, stream=stream)
                    assert tg.tg_query_status(h) == 0
                    np.testing.assert_array_equal(rows.cpu().numpy(), want[k % 3][0])
                    np.testing.assert_array_equal(totals.cpu().numpy(), want[k % 3][1])
                h.free()
        except BaseException as e:                                   # noqa: BLE001 (reported by the test)
            failures.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(12)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures[0]

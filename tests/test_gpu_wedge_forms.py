"""Wedge anchors by form: an anchor's counters take one, two or four words per
wedge end by the number of its lower neighbours of one type, and its table and
group of threads follow its number of wedges.  One anchor joined to `mid`
middles, each joined to `per` ends of a pool, so that the counters reach the
top of their fields (every middle joined to end 0); full rows against the
oracle, with no anchor a hub."""
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


def fan(mid, per, pool, L, one_type, seed):
    """Anchor 0; middles 1..mid; ends after them.  End 0 meets every middle but the last (it stays below the anchor)."""
    rng = np.random.default_rng(seed)
    e0 = mid + 1
    edges = [np.stack([np.zeros(mid, np.int64), np.arange(1, mid + 1)], 1)]
    for v in range(1, mid + 1):
        ends = rng.choice(np.arange(1, pool), per - 1, replace=False)
        if v < mid:
            ends = np.concatenate([[0], ends])
        edges.append(np.stack([np.full(len(ends), v), e0 + ends], 1))
    extra = e0 + pool                                         # leaves that keep the anchor's degree the largest
    edges.append(np.stack([np.zeros(8, np.int64), extra + np.arange(8)], 1))
    E = np.concatenate(edges)
    n = extra + 8
    types = rng.integers(0, L, n).astype(np.uint8)
    if one_type:
        types[1:mid + 1] = L - 1
    return graphgen.csr_from_edges(n, E[:, 0].astype(np.int32), E[:, 1].astype(np.int32), types, L, "fan")


# fields: L = 3: 10 bits in one word; L = 5: 6, 10, 16 bits; L = 8: 4, 8, 16 bits
CASES = [(3, 1023, 3), (3, 1024, 3), (5, 63, 2), (5, 64, 2), (5, 1023, 4), (5, 1024, 6), (8, 15, 4), (8, 16, 4),
         (8, 255, 3), (8, 256, 7), (6, 31, 30), (6, 400, 28), (4, 255, 55), (2, 700, 20), (1, 40, 3)]


@pytest.mark.parametrize("one_type", [True, False])
@pytest.mark.parametrize("L,mid,per", CASES)
def test_anchor_forms_match_oracle(L, mid, per, one_type):
    g = fan(mid, per, max(4 * per, 200), L, one_type, seed=mid + per)
    rows, totals = oracle.paper(g)
    for options in ({"hub_min_wedges": 1 << 30}, {"hub_min_wedges": 1 << 30, "light_anchor_max_wedges": 2048},
                    {"light_anchor_max_wedges": 1, "hub_min_wedges": 1}):
        pe, gl, st = gpu_count(g, options=options)
        assert st == 0, tg.STATUS[st]
        np.testing.assert_array_equal(pe, rows)
        np.testing.assert_array_equal(gl, totals)

"""Star-like anchors: any number of lower neighbours of one type and few
wedges.  A hub of leaves of one type, some of them joined in disjoint pairs:
two wedges per pair, each with an end of its own, so the anchor's table gets
as many ends as it has wedges.  Rows against the oracle's, one edge of every
kind (a leaf, a paired leaf, a pair), and all edges of a kind alike."""
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

# light tables of 64 and 48 wedges, the line where four words per end began (65,536 neighbours, or 1,024), and the
# forms of a CTA
CASES = [(3, 70000, 32, 64), (3, 70000, 30, 64), (4, 65600, 32, 64), (3, 65535, 32, 64), (5, 1100, 24, 48),
         (5, 70000, 24, 48), (8, 70000, 32, 64), (3, 70000, 33, 64), (3, 70000, 400, 64), (4, 70000, 5000, 64)]


@pytest.mark.parametrize("L,leaves,pairs,light", CASES)
def test_star_with_pairs(L, leaves, pairs, light):
    ends = np.arange(1, 2 * pairs + 1).reshape(pairs, 2)
    eu = np.concatenate([np.zeros(leaves, np.int32), ends[:, 0]]).astype(np.int32)
    ev = np.concatenate([np.arange(1, leaves + 1), ends[:, 1]]).astype(np.int32)
    types = np.full(leaves + 1, L - 1, dtype=np.uint8)
    types[0] = 0
    g = graphgen.csr_from_edges(leaves + 1, eu, ev, types, L, "star")
    kind = np.zeros(g["m"], dtype=np.int64)                  # caller order: the hub's edges, then the pairs
    kind[:2 * pairs] = 1
    kind[leaves:] = 2
    first = [int(np.argmax(kind == k)) for k in range(3)]
    want, _ = oracle.paper_edges(g, np.array(first))
    pe, gl, st = gpu_count(g, options={"light_anchor_max_wedges": light})
    assert st == 0, tg.STATUS[st]
    for k in range(3):
        np.testing.assert_array_equal(pe[kind == k], np.broadcast_to(want[k], ((kind == k).sum(), want.shape[1])))
    lay = tg.tg_layout(L, 4)
    per = [int(gl[o:o + s].sum()) for o, s in zip(lay["global_block_offset"], lay["global_block_size"])]
    m, d, rest = leaves + pairs, leaves, leaves - 2
    assert per[0] == m and per[2] == pairs and per[6] == pairs * rest        # edges, triangles, tailed triangles
    assert per[1] == d * (d - 1) // 2 - pairs                                # 3-paths: around the hub, but not closed
    assert per[3] == per[5] == per[7] == per[8] == 0                         # 4-paths, -cycles, chordal cycles, cliques

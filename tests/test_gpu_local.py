"""Counts from the local graphs of the lists N+(u): one graph per form of the
enumeration (warp per node, small and large CTA, lists beyond shared memory),
with list lengths on both sides of every boundary (32 | 33, 128 | 129,
704 | 705), against dense integer products."""
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


def dense_graph(n, density, L, seed):
    """Random graph of n nodes; ids by degree give lists N+ of up to about density * n entries."""
    rng = np.random.default_rng(seed)
    iu, ju = np.triu_indices(n, 1)
    keep = rng.random(len(iu)) < density
    eu, ev = iu[keep].astype(np.int32), ju[keep].astype(np.int32)
    types = rng.integers(0, L, n).astype(np.uint8)
    return graphgen.csr_from_edges(n, eu, ev, types, L, f"dense n={n} p={density}")


def plus_lengths(g):
    deg = np.diff(g["row_ptr"])
    rank = np.empty(g["n"], dtype=np.int64)
    rank[np.lexsort((np.arange(g["n"]), deg))] = np.arange(g["n"])
    src = np.repeat(np.arange(g["n"]), deg)
    return np.bincount(src[rank[g["col"]] > rank[src]], minlength=g["n"])


CASES = [(34, 1.0, 1), (34, 1.0, 8), (40, 0.8, 3), (131, 1.0, 5), (300, 0.5, 6), (707, 1.0, 2), (1500, 0.6, 7)]


def test_cases_reach_every_form():
    top = {c[0]: int(plus_lengths(dense_graph(*c, seed=11)).max()) for c in CASES}
    assert top[34] == 33 and top[131] == 130 and top[707] == 706 and top[1500] > 800


@pytest.mark.parametrize("n,density,L", CASES)
def test_typed_triangles_match_dense_products(n, density, L):
    g = dense_graph(n, density, L, seed=11)
    pe, _, st = gpu_count(g, k=3)
    assert st == 0, tg.STATUS[st]
    src = np.repeat(np.arange(n), np.diff(g["row_ptr"]))
    A = np.zeros((n, n), dtype=np.float64)
    A[src, g["col"]] = 1
    i, j = np.nonzero(np.triu(A))
    for t in range(L):
        c = ((A * (g["types"] == t)) @ A)[i, j]               # below 2^53: exact
        np.testing.assert_array_equal(pe[:, L + t], c)


@pytest.mark.parametrize("n,density,L", CASES)
def test_four_node_rows_match_oracle(n, density, L):
    """Sums over triangle nodes and 4-cliques: sampled rows against Alg. 1-3; the 4-clique slots add up to six times
    the total, which is C(n, 4) on a complete graph."""
    g = dense_graph(n, density, L, seed=12)
    pe, gl, st = gpu_count(g)
    assert st == 0, tg.STATUS[st]
    rng = np.random.default_rng(5)
    ids = np.unique(rng.integers(0, g["m"], 40))
    rows, _ = oracle.paper_edges(g, ids)
    np.testing.assert_array_equal(pe[ids], rows)
    lay = tg.tg_layout(L, 4)
    off, size = lay["global_block_offset"][8], lay["global_block_size"][8]
    k4 = pe[:, lay["orbit_offset"][12]:lay["orbit_offset"][12] + lay["pairs"]]
    assert int(k4.sum()) == 6 * int(gl[off:off + size].sum())
    if density == 1.0:
        assert int(gl[off:off + size].sum()) == n * (n - 1) * (n - 2) * (n - 3) // 24

"""The closing step of the cluster search (LOOP mode, 4 <= K <= 11): the sets of size
K - 2 are built and closed by their parent, never stored.  Orders from the
last that does not take the step (3) to the last that does (11), on lattices and on dense
multigraphs (parallel bonds, degree 6, candidate lists longer than a warp),
against the depth-first search of the same context family (an arena of one
node: lists and their order bit for bit) and the oracle's lists."""
import numpy as np
import pytest

from paper_2512_10910_gb300 import inputs as I
from oracle import enumerate as E

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_10910_gb300 import pne  # noqa: E402


def _multigraph(n, m, seed):
    rng = np.random.default_rng(seed)
    deg, edges = [0] * n, []
    while len(edges) < m:
        a, b = (int(x) for x in rng.integers(0, n, size=2))
        if a != b and deg[a] < 6 and deg[b] < 6:
            edges.append((min(a, b), max(a, b)))
            deg[a] += 1
            deg[b] += 1
    return I.grid_graph(n, sorted(edges), [2] * m)


GRAPHS = {"square6x5": (lambda: I.square_lattice(6, 5, 2), (4, 5, 9, 10, 11)),
          "cubic3x3x3": (lambda: I.cubic_lattice(3, 3, 3, 2), (3, 4, 5, 8, 9)),
          "multigraph": (lambda: _multigraph(12, 30, 3), (3, 4, 5, 6, 7)),
          "multigraph_ring": (lambda: _multigraph(20, 40, 4), (4, 6, 7, 8))}


@pytest.mark.parametrize("name,K", [(g, K) for g, (_, Ks) in GRAPHS.items() for K in Ks])
def test_closing_step_lists(monkeypatch, name, K):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    net = GRAPHS[name][0]()
    net = I.random_tensors(net, 7)
    lists = []
    for limit in (None, "1"):
        if limit:
            monkeypatch.setenv("PNE_SEARCH_ARENA_MAX", limit)
        ctx = pne.Context(0)
        monkeypatch.delenv("PNE_SEARCH_ARENA_MAX", raising=False)
        try:
            (res,), (edges, _) = ctx.expand(net, K, pne.PNE_MODE_LOOP, pne.PNE_F64, export=True, use_cache=False)
        finally:
            ctx.close()
        lists.append((res["n_terms"], edges))
    assert lists[0][0] == lists[1][0]
    assert np.array_equal(lists[0][1], lists[1][1])
    got = sorted(tuple(int(x) for x in row if x >= 0) for row in lists[0][1])
    assert got == sorted(tuple(int(x) for x in c) for c in E.enumerate_clusters(net, K, E.LOOP))

"""K = 3 in LOOP mode closes sizes 2 and 3 from the single bonds (csrc/enumerate.cu):
one level and no children; the clusters are the oracle's, in the order in which a
search of higher order lists the same sizes, on graphs with parallel bonds, triangles
and several bonds between one pair of sites."""
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


NETS = {"square": lambda: I.square_lattice(5, 4, 3), "dense": lambda: _multigraph(10, 26, 1),
        "triples": lambda: _multigraph(4, 11, 2), "sparse": lambda: _multigraph(40, 60, 3),
        "pair": lambda: I.grid_graph(2, [(0, 1)] * 5, [2] * 5)}


@pytest.mark.parametrize("name", NETS)
def test_lists_and_levels(monkeypatch, name):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    net = I.random_tensors(NETS[name](), 7)
    lists = []
    for K in (3, 6):
        ctx = pne.Context(0)
        try:
            pne.pne_ctx_profile(ctx.h, True)
            _, (edges, _) = ctx.expand(net, K, pne.PNE_MODE_LOOP, pne.PNE_F64, export=True, use_cache=False)
            prof = pne.pne_ctx_profile_read(ctx.h)
        finally:
            ctx.close()
        if K == 3:
            assert "enum_children" not in prof and "enum_close_count" in prof
        lists.append([tuple(int(x) for x in row if x >= 0) for row in np.asarray(edges)])
    assert lists[0] == [c for c in lists[1] if len(c) <= 3]
    assert sorted(lists[0]) == sorted(tuple(int(x) for x in c) for c in E.enumerate_clusters(net, 3, E.LOOP))

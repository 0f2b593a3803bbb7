"""A search with the closing step (csrc/enumerate.cu) whose levels outgrow the
largest arena goes depth-first below the deepest level that fits, from the levels
that it has: one breadth-first search, not two, in a first search and in a later
one, with the lists of the unlimited search bit for bit."""
import numpy as np
import pytest

from paper_2512_10910_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_10910_gb300 import pne  # noqa: E402


@pytest.mark.parametrize("shape,K,limits", [((6, 6), 8, (1, 200, 900)), ((4, 3), 5, (1,)), ((3, 3, 3), 7, (100, 1500)),
                                            ((6, 5), 11, (1, 500, 4000))])
def test_one_breadth_first_search(monkeypatch, shape, K, limits):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    net = I.random_tensors(I.square_lattice(*shape, 2) if len(shape) == 2 else I.cubic_lattice(*shape, 2), 9)
    lists = []
    for limit in (None,) + limits:
        if limit:
            monkeypatch.setenv("PNE_SEARCH_ARENA_MAX", str(limit))
        ctx = pne.Context(0)
        monkeypatch.delenv("PNE_SEARCH_ARENA_MAX", raising=False)
        try:
            for _ in range(2):
                pne.pne_ctx_profile(ctx.h, True)
                (res,), (edges, _) = ctx.expand(net, K, pne.PNE_MODE_LOOP, pne.PNE_F64, export=True, use_cache=False)
                prof = pne.pne_ctx_profile_read(ctx.h)
                pne.pne_ctx_profile(ctx.h, False)
                assert prof["enum_roots"][0] == 1
                assert limit != limits[0] or "enum_dfs" in prof       # the smallest arena cannot hold the levels
                lists.append((res["n_terms"], res["log_abs"], edges))
        finally:
            ctx.close()
    for n, v, e in lists[1:]:
        assert n == lists[0][0] and v == lists[0][1]
        assert np.array_equal(e, lists[0][2])

"""Weight passing at the edges of its work split (csrc/rank.cu): rows of a
matricised tensor below, at and above one panel of 512 (one block, several
blocks, several panels of one block), odd bond dimensions (a column left out of
every Jacobi round), the largest dimension, mixed dimensions, and batches large
enough that a set gets one block.

Weights within 1e-9 of the oracle's and equal sweep counts, as the existing
weight-passing tests ask; a set of a batch against the same set alone within
1e-11 (its rows are split differently)."""
import numpy as np
import pytest

from paper_2512_10910_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_10910_gb300 import pne  # noqa: E402
from oracle import weights as OW  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    c = pne.Context(0)
    yield c
    c.close()


def _mixed():
    g = I.square_lattice(3, 3, 4)
    g.bond_dim[:] = [3, 3, 7, 4, 7, 9, 5, 8, 11, 6, 5, 6]
    return g


NETS = {"D2": lambda: I.square_lattice(3, 3, 2), "D5": lambda: I.square_lattice(3, 3, 5),
        "D8_one_panel": lambda: I.square_lattice(3, 3, 8), "D9_split": lambda: I.square_lattice(3, 3, 9),
        "D13_split": lambda: I.square_lattice(3, 3, 13), "mixed": _mixed, "pair_D16": lambda: I.square_lattice(2, 2, 16),
        "cubic_D3": lambda: I.cubic_lattice(3, 2, 2, 3)}


def _run(ctx, net, data=None, n=1):
    ns, keep = pne.network_struct(net, data=data, n_batch=n)
    w = pne.pne_weight_passing(ctx.h, ns, 0.8, 1e-11, 5000)
    try:
        return pne.pne_weights_read(ctx.h, w, n, net.n_bonds)
    finally:
        pne.pne_weights_destroy(w)
        del keep


@pytest.mark.parametrize("name", NETS)
def test_weights_match_the_oracle(ctx, name):
    net = I.random_tensors(NETS[name](), 17)
    _, S, ls, sweeps, _ = OW.weight_passing(net, 0.8, 1e-11, 5000)
    wts, sw, gls = _run(ctx, net)
    assert sw[0] == sweeps
    assert abs(gls[0] - ls) <= 1e-9 * max(1.0, abs(ls))
    for b in range(net.n_bonds):
        np.testing.assert_allclose(wts[0, b, :len(S[b])], S[b], rtol=0, atol=1e-9)


@pytest.mark.parametrize("D,n", [(9, 80), (9, 40), (4, 160), (3, 7)])
def test_a_set_of_a_batch_is_the_set_alone(ctx, D, n):
    g = I.square_lattice(3, 3, D)
    nets = [I.random_tensors(g, 60 + i) for i in range(n)]
    wts, sw, ls = _run(ctx, nets[0], np.concatenate([x.flat_data()[0] for x in nets]), n)
    for i in (0, n // 2, n - 1):
        w1, s1, l1 = _run(ctx, nets[i])
        assert sw[i] == s1[0]
        np.testing.assert_allclose(wts[i], w1[0], rtol=0, atol=1e-11)
        assert abs(ls[i] - l1[0]) <= 1e-11 * max(1.0, abs(l1[0]))

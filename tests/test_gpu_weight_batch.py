"""A tensor set of a batch gets the weights, the sweeps and the scale that it gets
alone, bit for bit: how the rows of a matricised tensor are split (csrc/rank.cu,
weight_passing_kernel) follows from the tensor, not from the blocks that a set of
the batch is given.  Tensors above one panel of rows with eight, four, two and one
block per set, and below it with two and one."""
import numpy as np
import pytest

from paper_2512_10910_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_10910_gb300 import pne  # noqa: E402


def _run(ctx, net, data=None, n=1):
    ns, keep = pne.network_struct(net, data=data, n_batch=n)
    w = pne.pne_weight_passing(ctx.h, ns, 0.8, 1e-11, 5000)
    try:
        return pne.pne_weights_read(ctx.h, w, n, net.n_bonds)
    finally:
        pne.pne_weights_destroy(w)
        del keep


@pytest.mark.parametrize("D,n", [(9, 12), (9, 30), (9, 60), (9, 100), (8, 60), (8, 100)])
def test_a_set_of_a_batch_is_the_set_alone_bit_for_bit(D, n):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    nets = [I.random_tensors(I.square_lattice(3, 3, D), 300 + i) for i in range(n)]
    ctx = pne.Context(0)
    try:
        wts, sw, ls = _run(ctx, nets[0], np.concatenate([x.flat_data()[0] for x in nets]), n)
        for i in (0, n // 3, n - 1):
            w1, s1, l1 = _run(ctx, nets[i])
            assert sw[i] == s1[0] and ls[i] == l1[0]
            assert np.array_equal(wts[i], w1[0])
    finally:
        ctx.close()

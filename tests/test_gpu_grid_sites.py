"""The site matrices of a grid contraction (csrc/dense.cu, grid_sites_kernel) with one
block per tensor and with a cluster of two, four and eight: a set contracted in a
large batch has the value it has alone bit for bit (alone it takes the most blocks),
and in FP64 the einsum's within the stated bound.  Many small tensors take one block:
a cluster of eight each cost a launch five times its time."""
import math

import numpy as np
import pytest

from paper_2512_10910_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import exact as Ex  # noqa: E402
from paper_2512_10910_gb300 import pne  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    c = pne.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("lx,ly,chi,sizes", [(3, 3, 2, (1, 700)), (2, 3, 5, (1, 5, 40)), (3, 3, 9, (2, 20, 300)),
                                             (3, 2, 16, (3, 30, 200))])
def test_values_do_not_depend_on_the_blocks(ctx, lx, ly, chi, sizes):
    nets = [I.random_tensors(I.square_lattice(lx, ly, chi), 40 + i) for i in range(3)]
    for dtype in (pne.PNE_F64, pne.PNE_TF32, pne.PNE_BF16):
        alone = [pne.pne_grid_contract(ctx.h, n, lx, ly, dtype, data=n.flat_data()[0])[0] for n in nets]
        if dtype == pne.PNE_F64:
            for n, r in zip(nets, alone):
                assert abs(r["log_abs"] - math.log(float(Ex.contract_einsum(n)))) <= 1e-12
        for size in sizes:
            data = np.concatenate([nets[i % 3].flat_data()[0] for i in range(size)])
            for i, r in enumerate(pne.pne_grid_contract(ctx.h, nets[0], lx, ly, dtype, data=data, n_batch=size)):
                assert r["log_abs"] == alone[i % 3]["log_abs"] and r["sign"] == alone[i % 3]["sign"]


def test_many_small_tensors_are_not_slowed_by_clusters(ctx):
    """Launch time per tensor of 9,000 tensors of up to 16 entries: 4 to 7 ns with one
    block each, 40 with eight; 20 lies a factor of two to three from both."""
    nets = [I.random_tensors(I.square_lattice(3, 3, 2), 40 + i) for i in range(4)]
    data = torch.from_numpy(np.concatenate([nets[i % 4].flat_data()[0] for i in range(1000)])).cuda()
    best = float("inf")
    for _ in range(6):
        pne.pne_ctx_profile(ctx.h, True)
        pne.pne_grid_contract(ctx.h, nets[0], 3, 3, pne.PNE_TF32, data=data, n_batch=1000)
        best = min(best, pne.pne_ctx_profile_read(ctx.h)["grid_sites"][1])
        pne.pne_ctx_profile(ctx.h, False)
    assert best * 1e6 / 9000 <= 20.0

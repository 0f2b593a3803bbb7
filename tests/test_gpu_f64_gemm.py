"""The FP64 products (csrc/dense.cu, f64_gemm_kernel) at the edges of their
units, runs and slabs: row, column and K remainders, several column blocks, one
column, padded rows, more runs than SMs, each register form.  Operands are
whole numbers, |A|, |B| <= 1000 and K <= 2000, so every partial sum is below
2^53 and the products are exact.  Grids: whole-number networks small enough for
the contraction to be exact, with power-of-two factors far apart (2^-900), a
rational oracle on the CPU, equality up to the logarithm's own rounding."""
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_2512_10910_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_10910_gb300 import pne  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    c = pne.Context(0)
    yield c
    c.close()


# batch, M, N, K, lda - K, ldc - N
PRODUCTS = [(1, 1, 1, 1, 0, 0), (1, 8, 4, 16, 0, 0), (1, 9, 5, 17, 0, 1), (2, 121, 121, 121, 0, 0),
            (1, 256, 256, 256, 0, 0), (1, 1331, 121, 33, 3, 2), (1, 7, 129, 2000, 1, 0), (3, 5000, 3, 31, 0, 0),
            (1, 20001, 1, 15, 0, 0), (1, 14641, 121, 48, 0, 0), (700, 12, 10, 20, 0, 0), (1, 333, 1031, 65, 0, 5),
            (160, 130, 127, 16, 0, 0)]


@pytest.mark.parametrize("batch,M,N,K,pa,pc", PRODUCTS)
def test_products(ctx, batch, M, N, K, pa, pc):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randint(-1000, 1001, (batch, M, K + pa), generator=g, device="cuda").double()[:, :, :K]
    B = torch.randint(-1000, 1001, (batch, N, K), generator=g, device="cuda").double()
    C = torch.full((batch, M, N + pc), 7.0, dtype=torch.float64, device="cuda")
    pne.pne_dense_gemm(ctx.h, pne.PNE_F64, A, B, C[:, :, :N])
    assert torch.equal(C[:, :, :N].cpu(), A.cpu() @ B.cpu().transpose(1, 2))
    assert bool((C[:, :, N:] == 7.0).all())              # nothing is written beyond the rows


def _exact_log(g, lx, ly, tensors, exps):
    """log of the contraction of whole-number tensors times 2^exps, all legs
    in site order, bond by bond with Python integers."""
    state, legs = np.array(1, dtype=object), []
    for v in range(lx * ly):
        bonds = [int(b) for b in g.legs(v)]
        shared = [b for b in bonds if b in legs]
        state = np.tensordot(state, tensors[v].astype(object),
                             axes=([legs.index(b) for b in shared], [bonds.index(b) for b in shared]))
        legs = [b for b in legs if b not in shared] + [b for b in bonds if b not in shared]
    f = Fraction(int(state)) * Fraction(2) ** sum(exps)
    return math.log(f.numerator) - math.log(f.denominator)


# lx, ly, dims of the horizontal and of the vertical bonds
GRIDS = [(2, 2, 2, 3), (3, 3, 2, 3), (4, 2, 5, 2), (2, 4, 1, 4), (3, 2, 11, 5)]


@pytest.mark.parametrize("lx,ly,dh,dv", GRIDS)
def test_grids(ctx, lx, ly, dh, dv):
    g = I.square_lattice(lx, ly, 2)
    for b, (s0, s1) in enumerate(g.bond_site):
        g.bond_dim[b] = dh if s1 == s0 + 1 else dv
    rng = np.random.default_rng(lx + ly + dh + dv)
    flats, want = [], []
    for i in range(3):
        ts = [rng.integers(0, 4, g.leg_dims(v)) for v in range(lx * ly)]
        ex = [int(x) for x in rng.integers(-900, 400, lx * ly)] if i else [0] * (lx * ly)
        flats.append(np.concatenate([np.ldexp(t.astype(np.float64), x).ravel() for t, x in zip(ts, ex)]))
        want.append(_exact_log(g, lx, ly, ts, ex))
    got = pne.pne_grid_contract(ctx.h, g, lx, ly, pne.PNE_F64, data=np.concatenate(flats), n_batch=3)
    for a, w in zip(got, want):
        assert abs(a["log_abs"] - w) <= 4 * 2.0 ** -52 * max(1.0, abs(w), 1300 * lx * ly)

"""Weight passing on strongly graded bonds (csrc/rank.cu, jacobi_columns): the
blocked Ising network far below T_c, whose weights fall by 25 decades over a
bond.  The leg transforms divide by them, so the small entries of the rotations
have to be right to their own size, or the value of the network moves: a gauge
change keeps it, and so does an expansion that keeps all but one index of each
bond.  Twelve bonds, about ten sweeps, sixteen terms to a product at 2^-53 each
are 2e-13 of the value; 2e-11 leaves a factor of a hundred."""
import math

import pytest

from paper_2512_10910_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import exact as Ex  # noqa: E402
from paper_2512_10910_gb300 import pne  # noqa: E402


@pytest.mark.parametrize("frac", [0.5, 0.53, 0.56, 0.6])
def test_cold_blocked_ising_keeps_its_value(frac):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    net = I.ising_blocked(3, 3, 4, math.log(1 + math.sqrt(2)) / 2 / frac)
    z0 = math.log(float(Ex.contract_einsum(net)))
    ctx = pne.Context(0)
    try:
        (r,), _, _, _ = ctx.rank_r(net, I.square3x3_pinwheel(), 15, 0, alpha=0.8, tol=1e-11, grid=(3, 3),
                                   dtype=pne.PNE_F64)
    finally:
        ctx.close()
    assert abs(math.expm1(r["log_abs"] - z0)) <= 2e-11

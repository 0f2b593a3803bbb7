"""The float-float row products (csrc/strip.cu, strip_apply_kernel) over every
bond dimension, even and odd (a row of the matrix is read two entries at a
time), against the FP64 ones.  A dot product of chi^2 terms is off by at most
3 chi^2 2^-48 of the sum of magnitudes, which for non-negative tensors is the
sum itself; a w x h patch takes w h of them, an eigenvalue w.  The power
iteration stops at 1e-14 in either arithmetic: 1e-13 on top."""
import numpy as np
import pytest

from paper_2512_10910_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_10910_gb300 import pne  # noqa: E402


@pytest.mark.parametrize("chi,L", [(2, 9), (3, 6), (4, 5), (5, 4), (6, 4), (7, 4), (8, 4)])
def test_float_float_products_against_fp64(chi, L):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    A = np.stack([I.uniform_random(chi, 70 + i) for i in range(3)])
    ctx = pne.Context(0)
    try:
        r64 = pne.pne_strip_expansion(ctx.h, A, L, arithmetic=0)
        rff = pne.pne_strip_expansion(ctx.h, A, L, arithmetic=1)
    finally:
        ctx.close()
    unit = 3 * chi * chi * 2.0 ** -48
    for a, b in zip(r64, rff):
        for w in range(1, L + 1):
            assert abs(a["log_lam"][w] - b["log_lam"][w]) <= 1e-13 + w * unit
            assert abs(a["log_gam"][w] - b["log_gam"][w]) <= 1e-13 + w * unit
            for h in range(1, L + 1):
                assert abs(a["log_z"][w][h] - b["log_z"][w][h]) <= 1e-13 + w * h * unit

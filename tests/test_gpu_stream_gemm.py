"""The persistent tensor-core GEMM (csrc/dense.cu, tc_stream_kernel) at the
edges of its tiles: row, column and K remainders, one and several column tiles
(also narrowed to reach more SMs), padded rows, unaligned results, more tiles
than SMs, and on grids every box width of the running tensor (16 to 128
contiguous bytes) and the gathered sites (an odd range, a left boundary).

Products: FP32 accumulation of the rounded inputs, |error| <= (K + 2) 2^-24
sum |a b| (the bound of the small-product kernel's test).  Grids: the stated
err_bound against FP64, non-negative networks."""
import math

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


def _rounded(x, dtype):
    b = x.contiguous().view(torch.int32)
    if dtype == pne.PNE_TF32:
        b = (b + 0x1000) & ~0x1FFF                       # nearest, ties away
    else:
        b = (b + 0x7FFF + ((b >> 16) & 1)) & ~0xFFFF     # nearest, ties to even
    return b.view(torch.float32).double()


# batch, M, N, K, lda - K, ldc - N
PRODUCTS = [(1, 128, 256, 256, 0, 0), (2, 129, 255, 260, 0, 0), (1, 1000, 257, 132, 4, 0), (3, 257, 304, 200, 0, 4),
            (1, 64, 2048, 520, 0, 0), (1, 127, 17, 1028, 8, 3), (5, 4133, 16, 64, 0, 0), (16, 2500, 48, 36, 0, 1)]


@pytest.mark.parametrize("dtype", [pne.PNE_TF32, pne.PNE_BF16], ids=["tf32", "bf16"])
@pytest.mark.parametrize("batch,M,N,K,pa,pc", PRODUCTS)
def test_products(ctx, dtype, batch, M, N, K, pa, pc):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(batch, M, K + pa, generator=g, device="cuda")[:, :, :K]
    B = torch.randn(batch, N, K, generator=g, device="cuda")
    C = torch.full((batch, M, N + pc), 7.0, device="cuda")
    pne.pne_dense_gemm(ctx.h, dtype, A, B, C[:, :, :N])
    ra, rb = _rounded(A, dtype), _rounded(B, dtype)
    ref, mag = ra @ rb.transpose(1, 2), ra.abs() @ rb.abs().transpose(1, 2)
    worst = float(((C[:, :, :N].double() - ref).abs() / mag).max())
    assert worst <= (K + 2) * 2.0 ** -24
    assert bool((C[:, :, N:] == 7.0).all())              # nothing is written beyond the rows


# dims of the vertical bonds and of the horizontal ones: Kh is the horizontal one
GRIDS = [(2, 2), (4, 4), (3, 8), (5, 16), (3, 32), (2, 64), (7, 7), (17, 3), (16, 12)]


@pytest.mark.parametrize("dv,dh", GRIDS)
def test_grids(ctx, dv, dh):
    g = I.square_lattice(3, 3, 2)
    for b, (s0, s1) in enumerate(g.bond_site):
        g.bond_dim[b] = dh if s1 == s0 + 1 else dv
    nets = [I.random_tensors(g, 40 + i) for i in range(3)]
    flat = np.concatenate([n.flat_data()[0] for n in nets])
    ref = pne.pne_grid_contract(ctx.h, g, 3, 3, pne.PNE_F64, data=flat, n_batch=3)
    for dt in (pne.PNE_TF32, pne.PNE_BF16):
        for a, b in zip(pne.pne_grid_contract(ctx.h, g, 3, 3, dt, data=flat, n_batch=3), ref):
            assert abs(math.expm1(a["log_abs"] - b["log_abs"])) <= a["err_bound"]

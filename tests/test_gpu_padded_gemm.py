"""Products whose rows of A are off the 16-byte boundaries (csrc/dense.cu,
launch_padded_stream: A copied to padded rows a piece at a time before the
persistent kernel) and results whose rows are (stored a line of one row at a
time): odd K, an odd pitch, a shifted start, few and many columns, several sets
to a piece, one set over several pieces.

FP32 accumulation of the rounded inputs, |error| <= (K + 2) 2^-24 sum |a b|
(the bound of the small-product kernel's test)."""
import pytest

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


# batch, M, N, K, first column of A, lda - K, ldc - N
PRODUCTS = [(1, 129, 255, 257, 0, 0, 0), (2, 1000, 995, 125, 0, 0, 0), (3, 257, 304, 200, 1, 0, 1),
            (1, 4133, 17, 65, 0, 3, 2), (40, 500, 33, 19, 2, 1, 0), (3, 70001, 16, 127, 0, 0, 0),
            (1, 300001, 16, 129, 0, 0, 1), (1, 64, 2047, 520, 3, 1, 0)]


@pytest.mark.parametrize("dtype", [pne.PNE_TF32, pne.PNE_BF16], ids=["tf32", "bf16"])
@pytest.mark.parametrize("batch,M,N,K,skip,pa,pc", PRODUCTS)
def test_products(ctx, dtype, batch, M, N, K, skip, pa, pc):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(batch, M, skip + K + pa, generator=g, device="cuda")[:, :, skip:skip + K]
    B = torch.randn(batch, N, K, generator=g, device="cuda")
    C = torch.full((batch, M, N + pc), 7.0, device="cuda")
    pne.pne_dense_gemm(ctx.h, dtype, A, B, C[:, :, :N])
    ra, rb = _rounded(A, dtype), _rounded(B, dtype)
    ref, mag = ra @ rb.transpose(1, 2), ra.abs() @ rb.abs().transpose(1, 2)
    assert float(((C[:, :, :N].double() - ref).abs() / mag).max()) <= (K + 2) * 2.0 ** -24
    assert bool((C[:, :, N:] == 7.0).all())              # nothing is written beyond the rows

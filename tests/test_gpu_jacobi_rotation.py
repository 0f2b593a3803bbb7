"""The rotation of weight passing's one-sided Jacobi (csrc/jacobi.h) against 60
decimal digits: cosine and sine each to its own size over inner products and
norm differences that are alike, graded up to FP32's range and beyond it, of
either sign, and equal norms.  A small entry of the accumulated rotations is a
few sines, so a sine off by more than FP64's roundings stays in it.  Sine and
cosine come from t (a few roundings: the difference of the norms, the residual
and the sum of the last step), s = t c, the correction and the products with it:
under eight roundings of 2^-53 each, 9e-16; 1e-15 is asked."""
import ctypes
import subprocess
from decimal import Decimal, localcontext

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_10910_gb300 import build  # noqa: E402

SOURCE = r"""
#include "jacobi.h"
__global__ void rotations(const double *a, const double *b, const double *g, double *cs, double *sn, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) pne::jacobi_rotation(a[i], b[i], g[i], cs[i], sn[i]);
}
extern "C" int run(const double *a, const double *b, const double *g, double *cs, double *sn, int n)
{
    rotations<<<(n + 127) / 128, 128>>>(a, b, g, cs, sn, n);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? (int)e : (int)cudaDeviceSynchronize();
}
"""


def _cases():
    rng = np.random.default_rng(11)
    n = 500
    a = 1.0 + rng.random(n)
    sign = lambda: rng.choice([-1.0, 1.0], n)  # noqa: E731
    out = []
    for h_dec, g_dec in ((0, 0), (0, 6), (6, 0), (0, 15), (0, 30)):
        h = sign() * 10.0 ** -(h_dec * rng.random(n)) * 0.9
        out.append((a, a + h, sign() * 10.0 ** -(g_dec * rng.random(n)) * (0.1 + rng.random(n))))
    out.append((a, a, sign() * rng.random(n)))                              # equal norms: 45 degrees
    out.append((a * 1e-40, a * 1e-40 * (1.5 + rng.random(n)), a * 1e-41))   # far from one
    out.append((a * 1e-18, a, sign() * 1e-10 * (0.1 + rng.random(n))))      # graded columns, nearly parallel
    return [np.concatenate(x) for x in zip(*out)]


def test_rotations_are_right_to_their_own_size(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    src, so = tmp_path / "rotations.cu", tmp_path / "rotations.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(so), str(src)], check=True)
    a, b, g = _cases()
    dev = [torch.from_numpy(x).cuda() for x in (a, b, g)] + [torch.zeros(len(a), dtype=torch.float64, device="cuda")
                                                            for _ in range(2)]
    torch.cuda.synchronize()
    lib = ctypes.CDLL(str(so))
    assert lib.run(*[ctypes.c_void_p(t.data_ptr()) for t in dev], ctypes.c_int(len(a))) == 0
    cs, sn = dev[3].cpu().numpy(), dev[4].cpu().numpy()
    worst = 0.0
    with localcontext() as lc:
        lc.prec = 60
        for i in range(len(a)):
            h, gi = Decimal(float(b[i])) - Decimal(float(a[i])), Decimal(float(g[i]))
            z = h / (2 * gi)
            t = (1 if z >= 0 else -1) / (abs(z) + (1 + z * z).sqrt())
            c = 1 / (1 + t * t).sqrt()
            if h == 0 and sn[i] < 0:
                t = -t                                                      # either way round is right
            for got, ref in ((cs[i], c), (sn[i], c * t)):
                worst = max(worst, abs(float((Decimal(float(got)) - ref) / ref)))
    print(f"largest relative error of a sine or cosine {worst:.2e}")
    assert worst <= 1e-15

"""Float-float dot products (csrc/float_float.h, ff_dot) against the compensated
dot product whose every step is error-free before it joins the FP32
compensation (the product split by an FMA of its own, the sum by Knuth's
two-sum), restated in numpy: sums of fewer than 16 terms are that product bit for
bit; longer ones, which round once more where a term is about as large as the sum,
have its rms error within 0.2% (0.07% in numpy, sampling error of 40,000 sums that
mostly agree below 0.1%)."""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_10910_gb300 import build  # noqa: E402

SIZES = (2, 3, 4, 9, 16, 25, 64)
SOURCE = r"""
#include "float_float.h"
template <int N>
__global__ void dots(const double *a, const double *x, float *out, int n)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    pne::ff_dot<N> d;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const pne::ffp u = pne::split_double(a[q * N + i]), v = pne::split_double(x[q * N + i]);
        d.term(i, u.h, u.l, v.h, v.l);
    }
    const pne::ffp r = d.value();
    out[2 * q] = r.h;
    out[2 * q + 1] = r.l;
}
#define CASE(N) case N: dots<N><<<(n + 127) / 128, 128>>>(a, x, out, n); break;
extern "C" int run(int N, const double *a, const double *x, float *out, int n)
{
    switch (N) { CASE(2) CASE(3) CASE(4) CASE(9) CASE(16) CASE(25) CASE(64) default: return -1; }
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? (int)e : (int)cudaDeviceSynchronize();
}
"""
F = np.float32


def _fma(a, b, c):
    """FP32 FMA: the product is exact in FP64, the sum rounded twice once in 2^29 times."""
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def _split(x):
    h = x.astype(F)
    return h, (x - h.astype(np.float64)).astype(F)


def _error_free(a, x):
    (ah, al), (xh, xl) = _split(a), _split(x)
    sh = np.zeros(len(a), F)
    c = np.zeros(len(a), F)
    for i in range(a.shape[1]):
        pr = ah[:, i] * xh[:, i]
        pe = _fma(ah[:, i], xh[:, i], -pr)
        t = sh + pr
        bb = t - sh
        c = c + (((sh - (t - bb)) + (pr - bb)) + pe)
        sh = t
        c = _fma(al[:, i], xh[:, i], _fma(ah[:, i], xl[:, i], c))
    h = sh + c
    return np.stack([h, c - (h - sh)], axis=1)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    d = tmp_path_factory.mktemp("ff")
    (d / "dots.cu").write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(d / "dots.so"), str(d / "dots.cu")],
                   check=True)
    return ctypes.CDLL(str(d / "dots.so"))


@pytest.mark.parametrize("signs", [False, True])
@pytest.mark.parametrize("N", SIZES)
def test_against_the_error_free_form(lib, N, signs):
    n = 40000
    rng = np.random.default_rng(100 * N + signs)
    a, x = (rng.standard_normal((2, n, N)) if signs else rng.random((2, n, N)) + 0.1)
    da, dx = torch.from_numpy(a.copy()).cuda(), torch.from_numpy(x.copy()).cuda()
    out = torch.zeros(n, 2, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    assert lib.run(N, *[ctypes.c_void_p(t.data_ptr()) for t in (da, dx, out)], n) == 0
    got, ref = out.cpu().numpy(), _error_free(a, x)
    if N < 16:
        assert np.count_nonzero(got != ref) == 0
        return
    exact = (a.astype(np.longdouble) * x.astype(np.longdouble)).sum(axis=1)
    size = np.abs(a * x).sum(axis=1)

    def rms(v):
        return float(np.sqrt(np.mean(((v.astype(np.longdouble).sum(axis=1) - exact) / size) ** 2)))
    print(f"N {N}: rms {rms(got):.4e}, error-free {rms(ref):.4e}")
    assert rms(got) <= 1.002 * rms(ref)

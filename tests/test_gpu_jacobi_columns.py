"""The one-sided Jacobi of weight passing (csrc/jacobi.h, jacobi_columns) by itself:
singular values, orthogonal columns and W = A V for even and odd sizes and graded
columns; and columns of NaN or of overflowing squares, where every place of the
singular values has to be written (a place left from the matrix before reads as a
good value, and a zero-or-NaN test of it passes).

Orthogonal columns: the rotations stop at |g| <= 1e-15 |x||y|, dots of up to 16
terms add 16 roundings: 1e-14.  Singular values and A V against the product with
FP64 numpy: about ten sweeps of 15 rotations a column, 2^-53 or two each: 1e-13 of
each column's own norm."""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_10910_gb300 import build  # noqa: E402

SOURCE = r"""
#include "jacobi.h"
using namespace pne;
__global__ void svd(const double *a, double *w, double *v, double *s, int n)
{
    __shared__ double W[kJacobiDim * kJacobiLd], V[kJacobiDim * kJacobiLd], sig[kJacobiDim];
    for (int e = threadIdx.x; e < n * n; e += kJacobiThreads) {
        W[e % n * kJacobiLd + e / n] = a[e];
        V[e % n * kJacobiLd + e / n] = e / n == e % n ? 1.0 : 0.0;
    }
    if (threadIdx.x < kJacobiDim) sig[threadIdx.x] = 7.0;
    __syncthreads();
    jacobi_columns(W, V, sig, n);
    __syncthreads();
    for (int e = threadIdx.x; e < n * n; e += kJacobiThreads) {
        w[e] = W[e % n * kJacobiLd + e / n];
        v[e] = V[e % n * kJacobiLd + e / n];
    }
    if (threadIdx.x < n) s[threadIdx.x] = sig[threadIdx.x];
}
extern "C" int run(const double *a, double *w, double *v, double *s, int n)
{
    svd<<<1, kJacobiThreads>>>(a, w, v, s, n);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? (int)e : (int)cudaDeviceSynchronize();
}
"""
SIZES = (1, 2, 3, 8, 15, 16)


@pytest.fixture(scope="module")
def svd(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    d = tmp_path_factory.mktemp("jacobi")
    (d / "svd.cu").write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(d / "svd.so"), str(d / "svd.cu")],
                   check=True)
    lib = ctypes.CDLL(str(d / "svd.so"))

    def call(a):
        n = len(a)
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()]
        dev += [torch.zeros(n * n, dtype=torch.float64, device="cuda") for _ in range(2)]
        dev += [torch.zeros(n, dtype=torch.float64, device="cuda")]
        torch.cuda.synchronize()
        assert lib.run(*[ctypes.c_void_p(t.data_ptr()) for t in dev], n) == 0
        w, v, s = (t.cpu().numpy() for t in dev[1:])
        return w.reshape(n, n), v.reshape(n, n), s
    return call


@pytest.mark.parametrize("decades", [0, 9])
@pytest.mark.parametrize("n", SIZES)
def test_columns_values_and_rotations(svd, n, decades):
    a = np.random.default_rng(n).standard_normal((n, n)) * 10.0 ** (-decades * np.arange(n) / max(n - 1, 1))
    w, v, s = svd(a)
    norms = np.linalg.norm(w, axis=0)
    assert np.all(s[:-1] >= s[1:])
    np.testing.assert_allclose(s, norms, rtol=1e-14)
    np.testing.assert_allclose(v.T @ v, np.eye(n), rtol=0, atol=1e-13)
    assert np.all(np.abs((w / norms).T @ (w / norms) - np.eye(n)) <= 1e-14)
    assert np.all(np.abs(w - a @ v) <= 1e-13 * (np.abs(a) @ np.abs(v)))
    if decades == 0:
        np.testing.assert_allclose(s, np.linalg.svd(a, compute_uv=False), rtol=1e-12)


@pytest.mark.parametrize("n", SIZES)
def test_every_singular_value_is_written(svd, n):
    a = np.random.default_rng(n).standard_normal((n, n))
    one = a.copy()
    one[0, n // 2] = np.nan
    for bad in (np.full((n, n), np.nan), one):
        s = svd(bad)[2]
        assert np.all(np.isnan(s))                    # one NaN reaches every column
    s = svd(a * 1e200)[2]                             # squares overflow: infinite norms
    assert np.all(~np.isfinite(s))

"""pne_dense_gemm from many threads on one context (csrc/dense.cu): products on
several streams at once are those of one thread, bit for bit, and threads that come
and go leave no host memory behind (the word in which a kernel tells that a wait
gave up is the call's, from the context's pool).  3 KB a thread were left before;
800 threads may leave 512 KB, a sixth of that."""
import threading

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


def test_threads_on_their_own_streams(ctx):
    dtypes = (pne.PNE_TF32, pne.PNE_BF16, pne.PNE_F64)
    shapes = ((1, 32, 16, 16), (2, 300, 64, 77), (1, 1024, 256, 128))      # copying and persistent kernels
    torch.manual_seed(3)
    work = []
    for dt in dtypes:
        for b, m, n, k in shapes:
            ft = torch.float64 if dt == pne.PNE_F64 else torch.float32
            A, B = torch.randn(b, m, k, device="cuda", dtype=ft), torch.randn(b, n, k, device="cuda", dtype=ft)
            C = torch.empty(b, m, n, device="cuda", dtype=ft)
            pne.pne_dense_gemm(ctx.h, dt, A, B, C)
            work.append((dt, A, B, C))
    torch.cuda.synchronize()
    wrong = []

    def job(i):
        try:
            s = torch.cuda.Stream()
            for dt, A, B, C in work[i % 3:] + work[:i % 3]:
                with torch.cuda.stream(s):
                    out = torch.zeros_like(C)
                pne.pne_dense_gemm(ctx.h, dt, A, B, out, stream=s.cuda_stream)
                if not torch.equal(out, C):
                    wrong.append((i, dt, tuple(A.shape)))
        except Exception as e:  # noqa: BLE001
            wrong.append((i, repr(e)))

    threads = [threading.Thread(target=job, args=(i,)) for i in range(12)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_threads_that_end_leave_nothing(ctx):
    A, B = torch.randn(1, 32, 16, device="cuda"), torch.randn(1, 16, 16, device="cuda")
    C = torch.empty(1, 32, 16, device="cuda")
    torch.cuda.synchronize()

    def data_kb():
        with open("/proc/self/status") as f:
            return int(next(ln for ln in f if ln.startswith("VmData")).split()[1])

    def threads(n):
        for _ in range(n):
            t = threading.Thread(target=pne.pne_dense_gemm, args=(ctx.h, pne.PNE_TF32, A, B, C))
            t.start()
            t.join()

    threads(200)
    before = data_kb()
    threads(800)
    assert data_kb() - before <= 512

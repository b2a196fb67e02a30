"""Stage calls of a program with two CUDA contexts on one device: each keeps its own
scratch, nothing is lost when calls alternate, and neither a stage call nor destroying a
sketch changes the calling thread's current context."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROWS, K = 100000, 64


@pytest.fixture(scope="module")
def sfd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1602_00412_gb300 import sfd
    return sfd


class Driver:
    def __init__(self):
        torch.zeros(1, device="cuda")
        self.d = ctypes.CDLL("libcuda.so.1")
        self.first, self.second = self.current(), ctypes.c_void_p()
        self.ok(self.d.cuCtxCreate_v2(ctypes.byref(self.second), 0, 0))
        self.second = self.second.value
        self.use(self.first)

    def ok(self, rc):
        assert rc == 0, rc

    def current(self):
        c = ctypes.c_void_p()
        self.ok(self.d.cuCtxGetCurrent(ctypes.byref(c)))
        return c.value

    def use(self, ctx):
        self.ok(self.d.cuCtxSetCurrent(ctypes.c_void_p(ctx)))

    def free(self):
        a, b = ctypes.c_size_t(), ctypes.c_size_t()
        self.ok(self.d.cuMemGetInfo_v2(ctypes.byref(a), ctypes.byref(b)))
        return a.value

    def array(self, a):
        p = ctypes.c_uint64()
        self.ok(self.d.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(a.nbytes)))
        self.ok(self.d.cuMemcpyHtoD_v2(p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes)))
        return p

    def get(self, p, a):
        out = np.empty_like(a)
        self.ok(self.d.cuMemcpyDtoH_v2(out.ctypes.data_as(ctypes.c_void_p), p, ctypes.c_size_t(out.nbytes)))
        return out

    def close(self):
        self.use(self.second)
        self.ok(self.d.cuCtxDestroy_v2(ctypes.c_void_p(self.second)))
        self.use(self.first)


@pytest.fixture()
def driver(sfd):
    d = Driver()
    yield d
    d.close()


def test_alternating_contexts(sfd, driver):
    L = sfd.load()
    X = np.random.default_rng(0).integers(-3, 4, (ROWS, K)).astype(np.float32)
    want = X.astype(np.float64).T @ X
    ctxs = (driver.first, driver.second)
    arrays = {}

    def call(ctx):
        driver.use(ctx)
        x, g = arrays[ctx]
        # 25 MB of scratch for the block and as much for the dense stages
        assert L.sfd_orthonormalize(ROWS, K, ctypes.c_void_p(x.value), K) == 0
        assert driver.current() == ctx
        driver.ok(driver.d.cuMemcpyHtoD_v2(x, X.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(X.nbytes)))
        assert L.sfd_gram(ROWS, K, ctypes.c_void_p(x.value), K, ctypes.c_void_p(g.value), 0) == 0
        assert np.array_equal(driver.get(g, np.empty((K, K), np.float32)).astype(np.float64), want)

    def trim():
        for ctx in ctxs:
            driver.use(ctx)
            sfd.sfd_destroy(sfd.sfd_create(50, 5, 1))
            assert driver.current() == ctx
        return driver.free()

    for ctx in ctxs:
        driver.use(ctx)
        arrays[ctx] = driver.array(X), driver.array(np.zeros((K, K), np.float32))
    for ctx in ctxs:
        call(ctx)
    before = trim()
    for _ in range(4):
        for ctx in ctxs:
            call(ctx)
    held = driver.free()
    assert before - held <= 2 * (64 << 20)  # one scratch of each context
    assert trim() == before


def test_idle_scratch_of_an_ended_context(sfd):
    # a context that ends with scratch idle in it: calls in another one go on as before
    L = sfd.load()
    X = np.random.default_rng(1).integers(-3, 4, (500, K)).astype(np.float32)
    want = X.astype(np.float64).T @ X
    for _ in range(6):
        d = Driver()
        for ctx in (d.second, d.first):
            d.use(ctx)
            x, g = d.array(X), d.array(np.zeros((K, K), np.float32))
            assert L.sfd_gram(500, K, ctypes.c_void_p(x.value), K, ctypes.c_void_p(g.value), 0) == 0
            assert np.array_equal(d.get(g, np.empty((K, K), np.float32)).astype(np.float64), want)
            for p in (x, g):
                d.ok(d.d.cuMemFree_v2(p))
        d.close()
    sfd.sfd_destroy(sfd.sfd_create(50, 5, 1))

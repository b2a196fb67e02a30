"""Stage calls while a stream of the caller is being captured. They are synchronous, so
in the global and thread-local modes CUDA refuses them: the call returns SFD_ECUDA, and
what earlier calls left is still there. In the relaxed mode, which forbids only what
touches the capturing stream, the dense stages run as ever and the capture goes on.
(The sparse stages wait for the whole device, which no mode allows.)"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
GLOBAL, THREAD_LOCAL, RELAXED = 0, 1, 2
SFD_ECUDA = 3


@pytest.fixture(scope="module")
def sfd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1602_00412_gb300 import sfd
    return sfd


class Capture:
    """a capture of an empty stream through the driver; `ended` is the status of its end"""

    def __init__(self, mode):
        self.d = ctypes.CDLL("libcuda.so.1")
        self.mode, self.stream, self.ended = mode, ctypes.c_void_p(), None

    def __enter__(self):
        assert self.d.cuStreamCreate(ctypes.byref(self.stream), 1) == 0
        assert self.d.cuStreamBeginCapture_v2(self.stream, self.mode) == 0
        return self

    def __exit__(self, *exc):
        graph = ctypes.c_void_p()
        self.ended = self.d.cuStreamEndCapture(self.stream, ctypes.byref(graph))
        if graph.value:
            self.d.cuGraphDestroy(graph)
        self.d.cuStreamDestroy_v2(self.stream)


def stages(sfd):
    """dense stage calls: name -> (call, its output, what it overwrites of its input)"""
    L = sfd.load()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    rng = np.random.default_rng(7)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    X, T, M = (dev(rng.standard_normal(s)) for s in ((3000, 40), (40, 40), (66, 500)))
    S = dev((lambda a: a @ a.T)(rng.standard_normal((70, 200))))
    G, Y, Q, B = (torch.empty(s, device="cuda") for s in ((40, 40), (3000, 40), (3000, 40), (33, 500)))
    w, V = torch.empty(35, device="cuda"), torch.empty((70, 35), device="cuda")
    return {
        "gram": (lambda: L.sfd_gram(3000, 40, p(X), 40, p(G), 0), [G], None),
        "gram_tf32": (lambda: L.sfd_gram(3000, 40, p(X), 40, p(G), 1), [G], None),
        "gemm": (lambda: L.sfd_gemm_ts(3000, 40, p(X), 40, p(T), 40, p(Y), 40, 0), [Y], None),
        "orthonormalize": (lambda: L.sfd_orthonormalize(3000, 40, p(Q), 40), [Q], (Q, X)),
        "symeig": (lambda: L.sfd_symeig(70, p(S), 35, p(w), p(V)), [w, V], None),
        "dense_shrink": (lambda: L.sfd_dense_shrink(66, 500, 33, p(M), p(B)), [B], None),
    }


NAMES = ["gram", "gram_tf32", "gemm", "orthonormalize", "symeig", "dense_shrink"]


def prepare(outs, restore):
    for o in outs:
        o.fill_(float("nan"))
    if restore:
        restore[0].copy_(restore[1])
    torch.cuda.synchronize()


@pytest.mark.parametrize("name", NAMES)
def test_relaxed_capture_goes_on(sfd, name):
    call, outs, restore = stages(sfd)[name]
    prepare(outs, restore)
    assert call() == 0
    want = [o.clone() for o in outs]
    prepare(outs, restore)
    with Capture(RELAXED) as c:
        rc = call()
    assert rc == 0 and c.ended == 0
    assert all(torch.equal(o, v) for o, v in zip(outs, want))


@pytest.mark.parametrize("name", NAMES)
@pytest.mark.parametrize("mode", [GLOBAL, THREAD_LOCAL])
def test_refused_call_loses_nothing(sfd, name, mode):
    call, outs, restore = stages(sfd)[name]

    def free_without_scratch():
        sfd.sfd_destroy(sfd.sfd_create(50, 5, 1))
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    prepare(outs, restore)
    assert call() == 0
    want = [o.clone() for o in outs]
    before = free_without_scratch()
    prepare(outs, restore)
    assert call() == 0  # leaves its scratch idle
    prepare(outs, restore)
    with Capture(mode) as c:
        rc = call()
    assert rc == SFD_ECUDA and c.ended != 0
    sfd.load().cudaGetLastError()  # the CUDA runtime (linked) keeps a refused call's error
    assert call() == 0
    assert all(torch.equal(o, v) for o, v in zip(outs, want))
    assert free_without_scratch() == before

"""Calls of one stage share the scratch that earlier calls left: results must not
depend on what ran before in it, on refused calls in between, or on other
threads' calls at the same time. The sparse products use whole numbers small
enough that every sum is exact in fp32, so they equal the dense fp64 product."""
import ctypes
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SFD_EINVAL = 1


@pytest.fixture(scope="module")
def sfd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1602_00412_gb300 import sfd
    return sfd


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


class Product:
    """rows of `lens` entries at random columns below d, and a dense factor for A X or A^T X"""

    def __init__(self, lens, d, k, transposed, seed):
        rng = np.random.default_rng(seed)
        m = len(lens)
        cols = [np.sort(rng.choice(d, n, replace=False)) for n in lens]
        self.A = np.zeros((m, d))
        for i, c in enumerate(cols):
            self.A[i, c] = rng.integers(1, 4, len(c))
        self.X = rng.integers(-3, 4, (m if transposed else d, k)).astype(np.float32)
        ld = (k + 3) // 4 * 4
        rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        idx = np.concatenate(cols).astype(np.int32) if rp[-1] else np.zeros(0, np.int32)
        val = np.concatenate([self.A[i, c] for i, c in enumerate(cols)]).astype(np.float32)
        Xp = np.zeros((self.X.shape[0], ld), np.float32)
        Xp[:, :k] = self.X
        self.m, self.d, self.k, self.ld, self.t = m, d, k, ld, transposed
        self.dev = [torch.from_numpy(a).cuda() for a in (rp, idx, val, Xp)]
        self.Y = torch.empty((d if transposed else m, ld), device="cuda")
        self.want = (self.A.T if transposed else self.A) @ self.X.astype(np.float64)

    def call(self, L, rp=None, idx=None):
        r, i, v, X = self.dev
        return L.sfd_csr_spmm(self.m, self.d, ptr(r if rp is None else rp),
                              ptr(i if idx is None else idx), ptr(v), self.k, ptr(X), self.ld,
                              ptr(self.Y), self.ld, int(self.t))

    def check(self, L):
        self.Y.fill_(float("nan"))
        torch.cuda.synchronize()
        assert self.call(L) == 0
        assert np.array_equal(self.Y[:, :self.k].cpu().numpy().astype(np.float64), self.want)


def products():
    rng = np.random.default_rng(5)
    out = []
    for t in (False, True):
        out += [Product([0, 3, 0], 7, 1, t, 1), Product([1], 1, 5, t, 2),
                Product([0, 0], 3, 4, t, 3),
                Product(list(rng.integers(0, 40, 1000)), 300, 100, t, 4),
                Product([900, 0, 2100, 5, 1], 2500, 33, t, 5),
                Product(list(rng.integers(0, 9, 5000)), 11, 200, t, 6)]
    return out


def test_products_in_used_scratch(sfd):
    L = sfd.load()
    P = products()
    for p in P + P[::-1] + P[::2]:
        p.check(L)


def test_refused_calls_leave_the_scratch_usable(sfd):
    L = sfd.load()
    for p in products():
        r, i = p.dev[0], p.dev[1]
        p.Y.fill_(-7.0)
        first = r.clone()
        first[0] = 1
        assert p.call(L, rp=first) == SFD_EINVAL
        if p.m > 1:
            falls = r.clone()
            falls[p.m - 1] = r[p.m] + 1
            assert p.call(L, rp=falls) == SFD_EINVAL
        if i.numel():
            for bad in (-1, p.d):
                ib = i.clone()
                ib[-1] = bad
                assert p.call(L, idx=ib) == SFD_EINVAL
        assert bool((p.Y == -7.0).all())
        p.check(L)


def test_threads_have_scratch_of_their_own(sfd):
    L = sfd.load()
    errors = []

    def work(seed):
        try:
            rng = np.random.default_rng(seed)
            P = products()
            rows, k = 3000 + 100 * seed, 20 + seed
            X = torch.from_numpy(rng.integers(-3, 4, (rows, k)).astype(np.float32)).cuda()
            G = torch.empty((k, k), device="cuda")
            torch.cuda.synchronize()
            want = (X.double().T @ X.double()).cpu()
            for rep in range(3):
                for p in P:
                    p.check(L)
                assert L.sfd_gram(rows, k, ptr(X), k, ptr(G), 0) == 0
                assert torch.equal(G.cpu().double(), want)
        except BaseException as e:  # noqa: BLE001 - reported by the main thread
            errors.append(e)

    T = [threading.Thread(target=work, args=(s,)) for s in range(6)]
    for t in T:
        t.start()
    for t in T:
        t.join()
    assert not errors, errors[0]


def test_stages_repeat_their_bits(sfd):
    # each stage's bits with fresh scratch (after a context is destroyed) and with scratch
    # that the other stages have written
    rng = np.random.default_rng(3)
    m = d = 300
    ell = 20
    M = torch.from_numpy(rng.standard_normal((2 * ell, d)).astype(np.float32)).cuda()
    X0 = torch.from_numpy(rng.standard_normal((2000, 33)).astype(np.float32)).cuda()
    A = Product(list(rng.integers(0, 30, m)), d, 4, False, 9)

    def run():
        B = torch.zeros((ell, d), device="cuda")
        Bp = torch.zeros((ell, d), device="cuda")
        Q = X0.clone()
        ev = torch.zeros(2 * ell, device="cuda")
        V = torch.zeros((2 * ell, 2 * ell), device="cuda")
        S = M[:, :2 * ell].contiguous()
        S = (S + S.T).contiguous()
        torch.cuda.synchronize()
        sfd.sfd_dense_shrink(2 * ell, d, ell, M, B)
        sfd.sfd_orthonormalize(2000, 33, Q, 33)
        sfd.sfd_symeig(2 * ell, S, 2 * ell, ev, V)
        info = sfd.sfd_bssh_buffer(m, d, ell, A.dev[0], A.dev[1], A.dev[2], 1, 0, Bp)
        A.check(sfd.load())
        return [t.cpu() for t in (B, Q, ev, V, Bp)] + [torch.tensor(info["delta_shrink"])]

    ctx = sfd.sfd_create(50, 5, 1)
    sfd.sfd_destroy(ctx)
    first = run()
    for p in products():
        p.check(sfd.load())
    for again in (run(), run()):
        assert all(torch.equal(a, b) for a, b in zip(first, again))


def test_scratch_given_back_without_a_sketch(sfd):
    # a program of stage calls alone: sfd_destroy(NULL) frees what they left
    L = sfd.load()
    rows, k = 400000, 64
    X = torch.ones((rows, k), device="cuda")
    G = torch.empty((k, k), device="cuda")

    def call():
        assert L.sfd_orthonormalize(rows, k, ptr(X), k) == 0  # 100 MB of scratch
        assert L.sfd_gram(rows, k, ptr(X), k, ptr(G), 0) == 0
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    call()
    L.sfd_destroy(None)
    free = torch.cuda.mem_get_info()[0]
    assert free - call() >= 100 << 20
    L.sfd_destroy(None)
    assert torch.cuda.mem_get_info()[0] == free
    L.sfd_destroy(None)
    call()


@pytest.mark.parametrize("bad", [-(2 ** 31), -70000, -7, 2500, 70000, 2 ** 31 - 1])
def test_far_column_indices_are_refused(sfd, bad):
    # the columns are sorted before the host has read the check's result: every index out
    # of range must be harmless there, near or far, one or many
    L = sfd.load()
    for p in products():
        i = p.dev[1]
        for where in (slice(-1, None), slice(None)):
            if not i.numel() or (bad >= 0 and bad < p.d):
                continue
            p.Y.fill_(-7.0)
            ib = i.clone()
            ib[where] = bad
            assert p.call(L, idx=ib) == SFD_EINVAL
            assert bool((p.Y == -7.0).all()) and bool((ib[where] == bad).all())
        p.check(L)
    m = d = 300
    A = Product(list(np.random.default_rng(2).integers(1, 30, m)), d, 4, False, 9)
    ib = A.dev[1].clone()
    ib[::3] = bad
    Bp = torch.full((20, d), -7.0, device="cuda")
    with pytest.raises(sfd.SfdError) as e:
        sfd.sfd_bssh_buffer(m, d, 20, A.dev[0], ib, A.dev[2], 1, 0, Bp)
    assert e.value.code == SFD_EINVAL and bool((Bp == -7.0).all())
    A.check(L)

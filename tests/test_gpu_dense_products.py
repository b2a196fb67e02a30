"""The FP32 Gram and small-matrix product at the edges of their tiles, of their
copies' widths (rows of any alignment) and of the rule that keeps the small
matrix in shared memory. Entries are whole numbers small enough that every sum
in any order is exact in fp32, so the results equal the fp64 reference."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1602_00412_gb300 import sfd
    return sfd.load()


def block(rows, n, ld, offset, seed):
    """rows x ld floats whose first element lies `offset` floats past a 256-byte boundary;
    NaN outside the n columns"""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    flat = torch.full((rows * ld + offset,), float("nan"), device="cuda")
    X = flat[offset:].view(rows, ld)
    X[:, :n] = torch.randint(-3, 4, (rows, n), device="cuda", generator=gen).float()
    return X


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("n,pad,offset", [(1, 0, 0), (7, 0, 1), (8, 0, 0), (9, 1, 2), (50, 6, 0),
                                          (100, 0, 2), (100, 4, 0), (127, 0, 0), (128, 0, 0),
                                          (129, 3, 0), (200, 0, 0), (200, 1, 3), (249, 7, 0),
                                          (255, 1, 1), (256, 0, 0)])
@pytest.mark.parametrize("rows", [1, 15, 17, 4865, 20011])
def test_gram_is_exact_on_whole_numbers(L, n, pad, offset, rows):
    X = block(rows, n, n + pad, offset, n + rows)
    G = torch.full((n, n), float("nan"), device="cuda")
    assert L.sfd_gram(rows, n, ptr(X), n + pad, ptr(G), 0) == 0
    Xd = X[:, :n].double()
    assert torch.equal(G.double(), Xd.T @ Xd)


# rows on both sides of where the forms change: 4864 for 200 columns, 19456 for 100 and
# fewer; 256 x 256 is too large to stay in shared memory
@pytest.mark.parametrize("n,kout,padx,pady,offset", [
    (1, 1, 0, 0, 0), (7, 9, 1, 0, 1), (16, 33, 0, 3, 0), (50, 50, 6, 6, 0), (50, 50, 0, 0, 2),
    (100, 100, 4, 4, 0), (100, 97, 0, 1, 3), (129, 65, 3, 7, 0), (200, 200, 0, 0, 0),
    (200, 130, 2, 2, 2), (255, 161, 1, 3, 0), (256, 256, 0, 0, 0)])
@pytest.mark.parametrize("rows", [1, 63, 4863, 4864, 4865, 9731, 19456, 19457, 40001])
def test_product_is_exact_on_whole_numbers(L, n, kout, padx, pady, offset, rows):
    X = block(rows, n, n + padx, offset, n + rows)
    T = block(n, kout, kout, offset, kout)
    flat = torch.full((rows * (kout + pady) + offset,), -7.0, device="cuda")
    Y = flat[offset:].view(rows, kout + pady)
    assert L.sfd_gemm_ts(rows, n, ptr(X), n + padx, ptr(T), kout, ptr(Y), kout + pady, 0) == 0
    assert torch.equal(Y[:, :kout].double(), X[:, :n].double() @ T.double())
    assert torch.all(Y[:, kout:] == -7.0)


@pytest.mark.parametrize("rows,ell", [(3, 2), (9, 5), (15, 8), (100, 50), (257, 129), (400, 200)])
def test_dense_shrink_of_two_blocks(L, rows, ell):
    # the Gram of a stack whose two blocks lie apart, its widths even and odd
    d = 997
    M = torch.from_numpy(np.random.default_rng(rows).standard_normal((rows, d))
                         .astype(np.float32)).cuda()
    B = torch.full((ell, d), float("nan"), device="cuda")
    assert L.sfd_dense_shrink(rows, d, ell, ptr(M), ptr(B)) == 0
    s = np.linalg.svd(M.cpu().numpy().astype(np.float64), compute_uv=False)
    want = np.sqrt(np.maximum(s[:ell] ** 2 - s[ell - 1] ** 2, 0))
    got = np.linalg.svd(B.cpu().numpy().astype(np.float64), compute_uv=False)
    # a shrunk value w moves by (error of s^2) / w, and by its square root near 0:
    # compare the squares, at the 2e-5 n^1/2 / 4 ||M||^2 the eigensolver is held to
    tol = 2e-5 * max(1, np.sqrt(rows) / 4) * s[0] ** 2
    assert np.all(np.abs(got ** 2 - want ** 2) <= tol)


# narrow outputs, whose CTAs take as many rows of warps as their rows need, and wide ones
# on both sides of where 64 rows a CTA leave half of the SMs empty (4,800 rows)
@pytest.mark.parametrize("n,kout,pad", [(50, 3, 0), (100, 20, 4), (200, 3, 1), (200, 20, 0),
                                        (250, 33, 2), (255, 193, 1), (256, 224, 0), (193, 255, 0)])
@pytest.mark.parametrize("rows", [2, 4799, 4801, 4863, 4865, 10000, 20011])
def test_narrow_and_wide_products_are_exact_on_whole_numbers(L, n, kout, pad, rows):
    X = block(rows, n, n + pad, 0, n + rows)
    T = block(n, kout, kout, 0, kout)
    Y = torch.full((rows + 1, kout), -7.0, device="cuda")
    assert L.sfd_gemm_ts(rows, n, ptr(X), n + pad, ptr(T), kout, ptr(Y), kout, 0) == 0
    assert torch.equal(Y[:rows].double(), X[:, :n].double() @ T.double())
    assert torch.all(Y[rows:] == -7.0)

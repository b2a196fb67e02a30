"""The accurate Cholesky factor (pairs of floats) of sfd_orthonormalize and of the
accurate passes of mixed precision, at the sizes where its kernels change form: the
inverse factor against one in float64, and through the public call what it gives for
blocks whose Gram's trace is beyond the largest float, and which subspace the result
spans."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [1, 3, 64, 65, 112, 113, 128, 129, 208, 209, 256]
# sfd::chol_inv(const float* G, int k, float* Rinv, float* work, int* flags,
# cudaStream_t, bool accurate)
CHOL_INV = "_ZN3sfd8chol_invEPKfiPfS2_PiP11CUstream_stb"


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


@pytest.mark.parametrize("k", SIZES)
@pytest.mark.parametrize("power", [0, -110, 126])
def test_inverse_factor_against_float64(sfd, k, power):
    # condition number 1e6, largest diagonal entry 1, times 2^power (at 126 the trace
    # overflows from k = 64 on). Rounding the result to fp32 is worth 2^-24 = 6e-8 at most,
    # 48 bits at this condition about 1e6 2^-46 = 1.4e-8; an fp32 factor is off by 1e-3.
    f = getattr(sfd.load(), CHOL_INV)
    rng = np.random.default_rng(k)
    Q, _ = np.linalg.qr(rng.standard_normal((k, k)))
    G = (Q * np.logspace(0, -6, k)) @ Q.T
    G = (G / G.diagonal().max()).astype(np.float32)
    G = np.tril(G) + np.tril(G, -1).T
    Gd = G.astype(np.float64)
    Gd += np.eye(k) * (np.trace(Gd) / k * 2.0 ** -20)
    want = np.linalg.inv(np.linalg.cholesky(Gd)).T
    Gt = torch.from_numpy(G * np.float32(2.0 ** power)).cuda()
    R = torch.full((k, k), np.nan, device="cuda")
    work = torch.zeros(k * (k | 1) + 64, device="cuda")
    flags = torch.zeros(16, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    f(ptr(Gt), k, ptr(R), ptr(work), ptr(flags), None, ctypes.c_bool(True))
    torch.cuda.synchronize()
    got = R.cpu().numpy().astype(np.float64) * 2.0 ** (power // 2)
    assert np.linalg.norm(got - want) <= 1e-7 * np.linalg.norm(want)
    assert int(flags[1]) == 0  # no pivot clamped


def block(rows, k, cond, seed):
    rng = np.random.default_rng(seed)
    U, _ = np.linalg.qr(rng.standard_normal((rows, k)))
    W, _ = np.linalg.qr(rng.standard_normal((k, k)))
    return (U * np.logspace(0, -np.log10(cond), k)) @ W.T


@pytest.mark.parametrize("k", [50, 100, 128, 200, 256])
def test_orthonormalize_where_the_trace_overflows(sfd, k):
    # every entry of the Gram is below 1e37, its trace above the largest float
    rows = 4 * k
    X = np.random.default_rng(k).standard_normal((rows, k))
    X = (X * np.sqrt(9e36 / (X ** 2).sum(0).max())).astype(np.float32)
    assert (X.astype(np.float64) ** 2).sum() > 3.5e38 or k == 50
    T = torch.from_numpy(X).cuda()
    sfd.sfd_orthonormalize(rows, k, T, k)
    Q = T.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(Q.T @ Q - np.eye(k)) < 5e-5 * k
    Xd = X.astype(np.float64)
    assert np.linalg.norm(Xd - Q @ (Q.T @ Xd)) < 1e-5 * np.linalg.norm(Xd)


@pytest.mark.parametrize("k", [3, 5, 63, 64, 65, 111, 112, 113, 129, 208, 209, 255])
@pytest.mark.parametrize("scale", [1.0, 1e-12])
def test_orthonormalize_spans_its_input(sfd, k, scale):
    # X = Q (Q^T X) with Q^T X upper triangular and positive on the diagonal, as the
    # Gram-Schmidt step leaves it: three products with rounded inverse factors, each off
    # by a few 2^-24 k^1/2 relative to the block it is applied to (a wrong subspace or
    # order of columns is off by 1). The smallest diagonal entry is at least 1e-4.
    rows = 4 * k + 3
    X = (block(rows, k, 1e4, k) * scale).astype(np.float32)
    ld = (k + 7) // 8 * 8
    T = torch.zeros((rows, ld), device="cuda")
    T[:, :k] = torch.from_numpy(X).cuda()
    sfd.sfd_orthonormalize(rows, k, T, ld)
    Q = T.cpu().numpy()[:, :k].astype(np.float64)
    Xd = X.astype(np.float64) / scale  # largest singular value 1
    R = Q.T @ Xd
    tol = 32 * np.sqrt(k) * 2.0 ** -24
    assert np.linalg.norm(Xd - Q @ R, 2) < tol
    assert np.linalg.norm(np.tril(R, -1), 2) < tol
    assert np.diag(R).min() > 0.9e-4

"""The small dense factorisations at the sizes where their kernels change form:
the eigensolver where the tridiagonalisation moves from one CTA to a cluster
(n = 128, 256), where reflectors are joined in incomplete groups of four, and
where the Cholesky factor of its CholeskyQR passes changes its tiling; and the
accurate Cholesky of sfd_orthonormalize at its own limits. Bounds are those of
the stage tests: a backward-stable fp32 eigensolver leaves errors of a few
n^1/2 units of 2^-24 relative to the largest eigenvalue."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1602_00412_gb300 import sfd
    return sfd


@pytest.mark.parametrize("n,nwant", [(4, 4), (5, 5), (6, 3), (7, 7), (8, 1), (63, 33), (64, 64),
                                     (65, 65), (112, 112), (113, 113), (127, 64), (128, 128),
                                     (129, 129), (130, 1), (160, 160), (161, 161), (223, 40),
                                     (225, 113), (255, 255), (256, 128), (257, 200), (511, 256)])
def test_symeig_at_the_edges_of_its_forms(lib, n, nwant):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n))
    Sf = ((A + A.T) / 2).astype(np.float32)
    ev = torch.full((nwant,), np.nan, device="cuda")
    V = torch.full((n, nwant), np.nan, device="cuda")
    lib.sfd_symeig(n, torch.from_numpy(Sf).cuda(), nwant, ev, V)
    w_ref = np.linalg.eigvalsh(Sf.astype(np.float64))[::-1]
    nrm = np.abs(w_ref).max()
    w = ev.cpu().numpy().astype(np.float64)
    tol = max(1, np.sqrt(n) / 4)
    assert np.all(np.abs(w - w_ref[:nwant]) <= 2e-5 * nrm * tol)
    Vh = V.cpu().numpy().astype(np.float64)
    R = Sf.astype(np.float64) @ Vh - Vh * w
    assert np.linalg.norm(R, axis=0).max() <= 1e-4 * nrm * tol
    assert np.linalg.norm(Vh.T @ Vh - np.eye(nwant)) <= 1e-3 * max(1, nwant / 16)


def test_symeig_more_than_256_vectors(lib):
    # the Cholesky factor of a block wider than 256 columns
    n = 300
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n))
    Sf = ((A + A.T) / 2).astype(np.float32)
    ev = torch.zeros(n, device="cuda")
    V = torch.zeros((n, n), device="cuda")
    lib.sfd_symeig(n, torch.from_numpy(Sf).cuda(), n, ev, V)
    Vh = V.cpu().numpy().astype(np.float64)
    R = Sf.astype(np.float64) @ Vh - Vh * ev.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(R, axis=0).max() <= 1e-4 * np.linalg.norm(Sf, 2) * np.sqrt(n) / 4
    assert np.linalg.norm(Vh.T @ Vh - np.eye(n)) <= 1e-3 * n / 16


@pytest.mark.parametrize("k", [3, 5, 63, 64, 65, 111, 112, 113, 129, 208, 209, 255])
@pytest.mark.parametrize("scale", [1.0, 1e-12])
def test_orthonormalize_at_the_edges_of_the_accurate_factor(lib, k, scale):
    rows, cond = 4 * k + 3, 1e4
    rng = np.random.default_rng(k)
    U, _ = np.linalg.qr(rng.standard_normal((rows, k)))
    W, _ = np.linalg.qr(rng.standard_normal((k, k)))
    X = ((U * np.logspace(0, -np.log10(cond), k)) @ W.T * scale).astype(np.float32)
    ld = (k + 7) // 8 * 8
    T = torch.zeros((rows, ld), device="cuda")
    T[:, :k] = torch.from_numpy(X).cuda()
    lib.sfd_orthonormalize(rows, k, T, ld)
    Q = T.cpu().numpy()[:, :k].astype(np.float64)
    assert np.linalg.norm(Q.T @ Q - np.eye(k)) < 5e-5 * k
    Qr, _ = np.linalg.qr(X.astype(np.float64))
    assert np.linalg.norm(Q @ (Q.T @ Qr) - Qr) < 1e-4 * cond * np.sqrt(k)

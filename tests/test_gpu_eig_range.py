"""The eigensolver over the range of scales of its fp32 input: eigenvalues are squared
singular values of a sketch, so they grow with the rows of a stream and with the square
of their units. An fp32 eigensolver leaves errors of a few n^1/2 units of 2^-24 of the
largest eigenvalue whatever the scale; below about 1e-12 the columns under the square
root of 64 times the smallest normal number, 8.7e-19, which are taken as zero, add to
that (n of them, each in two places)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SCALES = [1e-14, 1e-12, 1e-9, 1e13, 1e14, 1e16]


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1602_00412_gb300 import sfd
    return sfd


def dropped(n, largest):
    return np.sqrt(2.0 * n) * 8.7e-19 / largest


@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("n", [65, 128, 200, 400])
def test_symeig_scales(lib, n, scale):
    rng = np.random.default_rng(n)
    M = rng.standard_normal((n, 3 * n)) * (0.97 ** np.arange(n))[:, None]
    G = M @ M.T
    Sf = (G * (scale / np.linalg.eigvalsh(G)[-1])).astype(np.float32)
    w_ref = np.linalg.eigvalsh(Sf.astype(np.float64))[::-1]
    nwant = n // 2
    S = torch.from_numpy(Sf).cuda()
    for call in [lib.sfd_symeig] + ([lib.sfd_symeig_noalloc] if n <= 256 else []):
        ev = torch.full((nwant,), np.nan, device="cuda")
        V = torch.full((n, nwant), np.nan, device="cuda")
        call(n, S, nwant, ev, V)
        w = ev.cpu().numpy().astype(np.float64)
        Vh = V.cpu().numpy().astype(np.float64)
        off = dropped(n, scale)
        assert np.all(np.abs(w - w_ref[:nwant]) <= (4 * np.sqrt(n) * 2.0 ** -24 + off) * scale)
        R = Sf.astype(np.float64) @ Vh - Vh * w
        # vectors of eigenvalues tied at fp32 resolution are shifted apart: the residual
        # bound of the stage tests
        assert np.linalg.norm(R, axis=0).max() <= (1e-4 * np.sqrt(n) / 4 + off) * scale
        assert np.linalg.norm(Vh.T @ Vh - np.eye(nwant)) <= 1e-3 * max(1, nwant / 16)


@pytest.mark.parametrize("power", [-27, 0, 23])
@pytest.mark.parametrize("ell", [50, 100])
def test_dense_shrink_scales(lib, ell, power):
    # rows scaled by 2^power (an exact factor): largest eigenvalues about 1e-13, 1e3, 1e17
    from oracle import sfd as O
    from oracle.metrics import bbt_rel_diff
    rows, d = 2 * ell, 600
    rng = np.random.default_rng(ell)
    M = (rng.standard_normal((rows, d)) * (0.97 ** np.arange(rows))[:, None]).astype(np.float32)
    B = torch.zeros((ell, d), device="cuda")
    lib.sfd_dense_shrink(rows, d, ell, torch.from_numpy(M * np.float32(2.0 ** power)).cuda(), B)
    got = B.cpu().numpy().astype(np.float64) * 2.0 ** -power
    largest = np.linalg.norm(M.astype(np.float64), 2) ** 2 * 4.0 ** power
    tol = max(1e-5, 2 * rows * 2.0 ** -24) + dropped(rows, largest)
    assert bbt_rel_diff(got, O.dense_shrink(M.astype(np.float64), ell)) < tol


# root mean square over the seeds of ||S V - V diag(w)||_F / ||S|| where the reduction to
# tridiagonal form rounds each entry once per step, on these matrices
ONE_ROUNDING = {(65, 33): 7.59e-7, (128, 64): 8.86e-7, (200, 100): 1.008e-6}


def test_symeig_residuals_of_one_rounding_per_step(lib):
    # Rounding an entry twice per step of the reduction leaves 1.11 times these residuals
    # on average over the three sizes (the mean's own spread is 1 %).
    ratio = []
    for (n, nwant), want in ONE_ROUNDING.items():
        ms = 0.0
        for seed in range(64):
            rng = np.random.default_rng([n, seed])
            M = rng.standard_normal((n, 3 * n)) * (0.97 ** np.arange(n))[:, None]
            S = torch.from_numpy((M @ M.T).astype(np.float32)).cuda()
            ev = torch.zeros(nwant, device="cuda")
            V = torch.zeros((n, nwant), device="cuda")
            lib.sfd_symeig(n, S, nwant, ev, V)
            Sd, Vd, w = S.double(), V.double(), ev.double()
            ms += float((Sd @ Vd - Vd * w).norm() / torch.linalg.matrix_norm(Sd, 2)) ** 2 / 64
        ratio.append(np.sqrt(ms) / want)
    assert np.mean(ratio) < 1.07, ratio

"""GPU checks of the small dense kernels at the edges of their blocks: the
blocked Cholesky factor and inverse of the B-orthonormalisation (32-row
blocks), the 8 x 8-tiled FP64 products and the final ordering of the
eigensolver, through the C ABI."""
import numpy as np
import pytest
import scipy.linalg as la

from workloads import pencil_1d, pencil_2d_q1, start_block

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_21618_gb300 import api as a
    return a


@pytest.mark.parametrize("m", [1, 2, 31, 32, 33, 63, 64, 65, 97, 150])
def test_rayleigh_ritz_at_block_edges(api, m):
    # theta and the B-orthonormality of X against dense FP64, from a block
    # whose columns span six orders of magnitude (the column scaling's job)
    p = pencil_2d_q1(27, seed=12)
    A, B = p.A().toarray(), p.B().toarray()
    U = start_block(p.n, m, m) * np.geomspace(1.0, 1e-6, m)[None, :]
    h = api.Handle(p)
    theta, X, _ = h.rayleigh_ritz(torch.from_numpy(U).cuda())
    X = X.cpu().numpy()
    Q, _ = np.linalg.qr(U / np.linalg.norm(U, axis=0))
    ref = la.eigh(Q.T @ A @ Q, Q.T @ B @ Q, eigvals_only=True)
    np.testing.assert_allclose(theta.cpu().numpy(), ref, rtol=1e-11)
    assert np.abs(X.T @ (B @ X) - np.eye(m)).max() <= 1e-13 * max(m, 10)


@pytest.mark.parametrize("m", [2, 7, 8, 9, 31, 64, 65, 127, 129])
def test_syev_at_tile_edges(api, m):
    # bounds as for the other sizes: eigenvalues 1e-13 |S| max(1, m / 10),
    # orthogonality 1e-13 m, residual 1e-12 |S|
    rng = np.random.default_rng(m)
    S = np.diag(np.arange(1.0, m + 1)) + 1e-2 * rng.standard_normal((m, m))
    S = S + S.T
    h = api.Handle(pencil_1d(200))
    lam, Q = (t.cpu().numpy() for t in h.syev(torch.from_numpy(S).cuda()))
    nrm = np.linalg.norm(S, 2)
    assert np.abs(lam - la.eigvalsh(S)).max() <= 1e-13 * nrm * max(1, m / 10)
    assert np.abs(Q.T @ Q - np.eye(m)).max() <= 1e-13 * m
    assert np.abs(S @ Q - Q * lam[None, :]).max() <= 1e-12 * nrm

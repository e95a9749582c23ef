"""GPU checks of the multigrid level that is solved by its dense shifted
inverses (FP32): the blocked symmetric sweep at its block edges, through one
application of the preconditioner against the same cycle with FP64 inverses."""
import numpy as np
import pytest
import scipy.linalg as la

from workloads import pencil_1d

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_21618_gb300 import api as a
    return a


# level sizes of the 1D hierarchy: n / 3, rounded; 64-row blocks: one block
# exactly, one and a ragged second, several, the largest allowed
@pytest.mark.parametrize("n", [191, 192, 193, 385, 1000, 2500, 4600])
@pytest.mark.parametrize("N", [1, 3])
def test_exact_level_inverse_matches_fp64(api, n, N):
    p = pencil_1d(n)
    o = api.default_opts(precond=api.PRECOND_MG, mg_coarse=16, mg_shift_limit=1e30)
    levels = api.mg_describe(p, o)["levels"]
    assert len(levels) >= 3 and levels[1] <= 1536
    (ptr, col, val, nr, nc), rho = api.mg_transfer(p, 0, o)
    P = np.zeros((nr, nc))
    for i in range(nr):
        P[i, col[ptr[i]:ptr[i + 1]]] = val[ptr[i]:ptr[i + 1]]
    A, B = p.A().toarray(), p.B().toarray()
    rng = np.random.default_rng(n)
    # shifts at a few per cent of the level's spectrum (its condition ~1e3)
    sig = 0.02 * n * n * (rng.uniform(0.1, 1.0, N) + 1j * rng.uniform(0.2, 1.0, N))
    m = 5
    ldp = 6
    R = np.zeros((n, N, ldp), dtype=np.complex64)
    R[:, :, :m] = rng.standard_normal((n, N, m)) + 1j * rng.standard_normal((n, N, m))
    h = api.Handle(p, o)
    Z, used = h.precond_apply(api.Filter(sig, np.ones(N)),
                              torch.from_numpy(R.reshape(n, -1).view(np.float32).copy()).cuda(), m, ldp)
    assert used == 2
    Z = Z.cpu().numpy().view(np.complex64).reshape(n, N, ldp)
    w = (4.0 / 3.0) / rho
    for j in range(N):
        M = A - sig[j] * B
        D = w / np.diag(M)
        r = R[:, j, :m].astype(complex)
        x = D[:, None] * r
        z = x + P @ la.solve(P.T @ M @ P, P.T @ (r - M @ x))
        z = z + D[:, None] * (r - M @ z)
        # the bound of the other FP32 cycle checks with an inverse level
        assert np.linalg.norm(Z[:, j, :m] - z) <= 5e-4 * np.linalg.norm(z)

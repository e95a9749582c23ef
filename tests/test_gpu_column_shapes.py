"""GPU checks of the FP64 kernels' block shapes, which follow the column count
(warps may span several rows): the shifted block product entry by entry, and a
filter application (updates, directions, multigrid cycle) against exact LU."""
import numpy as np
import pytest
import scipy.linalg as la

from oracle import filter as ofilt
from oracle import poles
from workloads import pencil_1d, pencil_2d_q1, pencil_3d_elasticity, start_block

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

PENCILS = {"1d": lambda: pencil_1d(203), "2d": lambda: pencil_2d_q1(14, seed=2), "3d": lambda: pencil_3d_elasticity(5, seed=5)}


@pytest.fixture(scope="module")
def api(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_21618_gb300 import api as a
    return a


@pytest.mark.parametrize("mesh", list(PENCILS))
@pytest.mark.parametrize("N,m,ldp", [(1, 1, 2), (1, 3, 4), (3, 1, 2), (1, 35, 36), (4, 31, 32), (4, 36, 36), (2, 33, 34),
                                     (5, 13, 14), (16, 3, 4)])
def test_fp64_shifted_product_at_every_block_shape(api, mesh, N, m, ldp):
    # a row of at most 81 pairs, combined with the pole by four more operations: 2 (81 + 4) rounding units of
    # (|A| + |s| |B|) |P| per entry (twice for the complex parts)
    p = PENCILS[mesh]()
    s, w = poles.slrf_poles(N, 1.0, 0.01, 300.0)
    rng = np.random.default_rng(N * m)
    P = rng.standard_normal((p.n, N * ldp)) + 1j * rng.standard_normal((p.n, N * ldp))
    P.reshape(p.n, N, ldp)[:, :, m:] = 0
    h = api.Handle(p, api.default_opts(precond=api.PRECOND_JACOBI))
    mu = torch.zeros(N * m, dtype=torch.complex128, device="cuda")
    Q = h.shifted_spmm(api.Filter(s, w), torch.from_numpy(P).cuda(), m, ldp, prec=api.PREC_FP64, mu=mu).cpu().numpy()
    mu = mu.cpu().numpy()
    A, B = p.A(), p.B()
    for j, sig in enumerate(s):
        X = P[:, j * ldp:j * ldp + m]
        ref = A @ X - sig * (B @ X)
        size = abs(A) @ np.abs(X) + abs(sig) * (abs(B) @ np.abs(X))
        out = Q[:, j * ldp:j * ldp + m]
        assert (np.abs(out - ref) <= 2 * 2 * 85 * 2.0**-53 * size).all()
        # p^T q: the products' bound, n further terms summed
        bound = 2 * (2 * 85 + p.n) * 2.0**-53 * (np.abs(X) * size).sum(axis=0)
        assert (np.abs(mu[j * m:(j + 1) * m] - (X * ref).sum(axis=0)) <= bound).all()


@pytest.mark.parametrize("m", [1, 9, 36, 47])
@pytest.mark.parametrize("precond", [1, 2])
def test_fp64_filter_at_ragged_widths(api, m, precond):
    p = pencil_2d_q1(24, seed=3)
    lam = la.eigvalsh(p.A().toarray(), p.B().toarray())
    s, w = poles.slrf_poles(4, 1.0, 0.01, 0.5 * (lam[14] + lam[15]))
    V = start_block(p.n, m, 3)
    h = api.Handle(p, api.default_opts(precision=api.PREC_FP64, inner_tol=1e-13, inner_maxit=4000, precond=precond))
    U = h.filter_apply(api.Filter(s, w), torch.from_numpy(V).cuda())[0].cpu().numpy()
    ref = ofilt.filter_apply(p.A(), p.B(), s, w, V)
    assert np.linalg.norm(U - ref) <= 1e-10 * np.linalg.norm(ref)   # the bound of the filter at this inner tolerance

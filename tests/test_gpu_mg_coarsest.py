"""GPU checks of the FP64 coarsest-level solve (two real x complex products
with the level's eigenvectors) through slrf_precond_apply on one-level
hierarchies, where it is the exact shifted solve: level sizes and column counts
around the tile edges of its two forms, converged and padding columns apart."""
import numpy as np
import pytest

from oracle import poles
from workloads import pencil_1d

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_21618_gb300 import api as a
    return a


@pytest.mark.parametrize("n,N,m,ldp", [
    (1, 1, 1, 2), (3, 2, 1, 2), (4, 1, 8, 8), (5, 4, 3, 4), (31, 2, 5, 6), (33, 4, 9, 10), (200, 2, 30, 30),
    (255, 4, 7, 8), (256, 1, 300, 300),     # the last: the 32 x 16 tiles
    (250, 8, 75, 76),
])
def test_single_level_solve_matches_a_dense_solve(api, n, N, m, ldp):
    p = pencil_1d(n)
    s, w = poles.slrf_poles(N, 1.0, 0.01, 400.0)
    h = api.Handle(p, api.default_opts(precision=api.PREC_FP64, precond=api.PRECOND_MG))
    rng = np.random.default_rng(n + m)
    R = rng.standard_normal((n, N * ldp)) + 1j * rng.standard_normal((n, N * ldp))
    Z, lv = h.precond_apply(api.Filter(s, w), torch.from_numpy(R).cuda(), m, ldp, prec=api.PREC_FP64)
    assert lv == 1
    Z = Z.cpu().numpy()
    A, B = p.A().toarray(), p.B().toarray()
    # the bound of the other exact shifted solves at these sizes (rounding of the eigendecomposition times the
    # ratio of the largest eigenvalue, 12 n^2, to the poles' distance from the spectrum, ~100: 7e3 eps at n = 256)
    for j, sig in enumerate(s):
        ref = np.linalg.solve(A - sig * B, R[:, j * ldp:j * ldp + m])
        err = np.linalg.norm(Z[:, j * ldp:j * ldp + m] - ref, axis=0) / np.linalg.norm(ref, axis=0)
        assert err.max() <= 1e-12

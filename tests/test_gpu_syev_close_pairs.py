"""GPU check of the eigensolver of projected matrices beyond 160 columns on wide
spectra with close eigenvalues at their low end, where the refinement cannot
separate the pairs and the last Jacobi has to: per column no further from
S q = lam q than the FP64 Jacobi (eig_refine = 0)."""
import numpy as np
import pytest

from workloads import pencil_1d

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_21618_gb300 import api as a
    return a


def _residuals(api, S, **opts):
    h = api.Handle(pencil_1d(600), api.default_opts(**opts))
    lam, Q = (t.cpu().numpy() for t in h.syev(torch.from_numpy(S).cuda()))
    assert np.abs(Q.T @ Q - np.eye(S.shape[0])).max() <= 1e-13 * S.shape[0]
    return np.linalg.norm(S @ Q - Q * lam[None, :], axis=0)


@pytest.mark.parametrize("m", [161, 210, 300, 448])
@pytest.mark.parametrize("top", [1e4, 1e6])
@pytest.mark.parametrize("gap", [1e-9, 1e-7, 1e-6])
def test_close_pairs_at_the_low_end(api, m, top, gap):
    rng = np.random.default_rng(m)
    lam = np.geomspace(1.0, top, m)
    lam[1] = lam[0] + gap
    lam[2] = lam[1] + 3 * gap
    Qr, _ = np.linalg.qr(rng.standard_normal((m, m)))
    S = (Qr * lam[None, :]) @ Qr.T
    S = np.ascontiguousarray(0.5 * (S + S.T))
    r2, r0 = _residuals(api, S), _residuals(api, S, eig_refine=0)
    # a column holds at most a few entries of 1/2 eps ||S||_F that are left
    # alone, and rounding of the products: 4 eps ||S||_F in all
    assert np.all(r2 <= 10 * r0 + 4 * np.finfo(float).eps * np.linalg.norm(S))

"""GPU checks of the eigensolver of projected matrices up to 160 columns: the
one-block FP32 Jacobi with logged rotations, the vectors formed from the log,
and the FP64 refinement, through the C ABI, at the sizes where the position
layout changes (odd orders have a phantom row; 64, 128: lanes per position)."""
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


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 31, 45, 63, 64, 65, 66, 127, 128, 129, 130, 159, 160])
@pytest.mark.parametrize("kind", ["projected", "dense", "diagonal"])
@pytest.mark.parametrize("mode", [1, 2])
def test_syev_up_to_160(api, m, kind, mode):
    rng = np.random.default_rng(m)
    lam = 20.0 + 12.0 * rng.permutation(m)
    if kind == "dense":
        S = rng.standard_normal((m, m))
    elif kind == "diagonal":        # no rotation at all, columns in another order
        S = np.diag(lam) / 2
    else:
        S = np.diag(lam) / 2 + 5e-3 / np.sqrt(m) * rng.standard_normal((m, m)) * np.sqrt(np.outer(lam, lam))
    S = S + S.T
    h = api.Handle(pencil_1d(600), api.default_opts(eig_refine=mode))
    lam, Q = [t.cpu().numpy() for t in h.syev(torch.from_numpy(np.ascontiguousarray(S)).cuda())]
    nrm = np.linalg.norm(S, 2)
    assert np.abs(lam - la.eigvalsh(S)).max() <= 1e-13 * nrm * max(1, m / 10)
    assert np.abs(Q.T @ Q - np.eye(m)).max() <= 1e-13 * m
    assert np.abs(S @ Q - Q * lam[None, :]).max() <= 1e-12 * nrm

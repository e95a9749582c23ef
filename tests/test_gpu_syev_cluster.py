"""GPU checks of the eigensolver of projected matrices beyond 160 columns: the
double-float Jacobi on a thread-block cluster, its refinement and the
cooperative Jacobi behind it, through the C ABI, against LAPACK and against the
FP64 Jacobi (eig_refine = 0)."""
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


def _check(S, lam, Q):
    m = S.shape[0]
    nrm = np.linalg.norm(S, 2)
    assert np.abs(lam - la.eigvalsh(S)).max() <= 1e-13 * nrm * max(1, m / 10)
    assert np.abs(Q.T @ Q - np.eye(m)).max() <= 1e-13 * m
    assert np.abs(S @ Q - Q * lam[None, :]).max() <= 1e-12 * nrm


def _syev(api, S, **opts):
    h = api.Handle(pencil_1d(600), api.default_opts(**opts))
    return [t.cpu().numpy() for t in h.syev(torch.from_numpy(np.ascontiguousarray(S)).cuda())]


# 161: the first size of the path; odd sizes have a phantom row; 447 and 448
# fill the shared memory of the cluster; 449 is the cooperative Jacobi's
@pytest.mark.parametrize("m", [161, 162, 175, 255, 300, 301, 447, 448, 449])
@pytest.mark.parametrize("kind", ["projected", "dense"])
def test_syev_beyond_160(api, m, kind):
    rng = np.random.default_rng(m)
    if kind == "dense":
        S = rng.standard_normal((m, m))
    else:
        lam = 20.0 + 12.0 * np.arange(m)
        S = np.diag(lam) + 5e-3 / np.sqrt(m) * rng.standard_normal((m, m)) * np.sqrt(np.outer(lam, lam))
    S = S + S.T
    _check(S, *_syev(api, S))


@pytest.mark.parametrize("case", ["clusters", "wide", "zero", "scaled"])
def test_syev_beyond_160_spectra(api, case):
    m = 210
    rng = np.random.default_rng(3)
    Qr, _ = np.linalg.qr(rng.standard_normal((m, m)))
    if case == "clusters":      # exact multiplicity 5 and near-multiplicities
        lam = np.repeat(np.linspace(1, 50, 42), 5)
        lam[::7] += 1e-9 * lam[::7]
    elif case == "wide":        # six decades: the low end is left to the last stage
        lam = np.geomspace(1.0, 1e6, m)
    elif case == "zero":
        lam = np.zeros(m)
    else:                       # entries far outside FP32's range
        lam = np.linspace(1.0, 9.0, m) * 1e60
    S = (Qr * lam[None, :]) @ Qr.T
    S = 0.5 * (S + S.T)
    if case == "zero":
        S[:] = 0.0
        l, Q = _syev(api, S)
        assert np.all(l == 0.0) and np.abs(Q.T @ Q - np.eye(m)).max() <= 1e-13 * m
    else:
        _check(S, *_syev(api, S))


def test_signs_follow_the_fp64_jacobi(api):
    # near-degenerate triples mixed by ~45 degrees, as the modes of a cube are:
    # the double-float path takes the FP64 path's turns, so the vectors come
    # out with the same signs
    m = 189
    rng = np.random.default_rng(8)
    lam = np.repeat(20.0 + 30.0 * np.arange(m // 3), 3) * (1.0 + 1e-2 * rng.standard_normal(m))
    E = rng.standard_normal((m, m)) * 1e-2
    S = np.diag(lam) + 0.5 * (E + E.T) * np.sqrt(np.outer(lam, lam)) / np.sqrt(m)
    for k in range(0, m, 3):
        S[k:k + 3, k:k + 3] += 1e-2 * lam[k] * 0.5 * (E[k:k + 3, k:k + 3] + E[k:k + 3, k:k + 3].T) * 100
    l0, Q0 = _syev(api, S, eig_refine=0)
    l2, Q2 = _syev(api, S)
    np.testing.assert_allclose(l2, l0, rtol=0, atol=1e-12 * l0[-1])
    assert np.abs(Q2 - Q0).max() <= 1e-9

"""GPU check of the exact multigrid level's inverses on pencils whose entries lie
near the ends of FP32's range, where the square of a pivot under- or overflows:
scaling A and B by a power of two scales the preconditioner by its inverse."""
import dataclasses

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


def _cycle(api, p, sig, R, m, ldp):
    n, N = R.shape[:2]
    h = api.Handle(p, api.default_opts(precond=api.PRECOND_MG, mg_coarse=16, mg_shift_limit=1e30))
    Z, used = h.precond_apply(api.Filter(sig, np.ones(N)),
                              torch.from_numpy(R.reshape(n, -1).view(np.float32).copy()).cuda(), m, ldp)
    assert used == 2
    return Z.cpu().numpy().view(np.complex64).reshape(n, N, ldp)[:, :, :m].astype(complex)


@pytest.mark.parametrize("e", [-76, -73, -50, 50, 56, 60])
def test_scaled_pencil_scales_the_preconditioner(api, e):
    n, N, m, ldp = 600, 2, 5, 6
    p = pencil_1d(n)
    rng = np.random.default_rng(1)
    sig = 0.02 * n * n * (rng.uniform(0.1, 1.0, N) + 1j * rng.uniform(0.2, 1.0, N))
    R = np.zeros((n, N, ldp), dtype=np.complex64)
    R[:, :, :m] = rng.standard_normal((n, N, m)) + 1j * rng.standard_normal((n, N, m))
    z0 = _cycle(api, p, sig, R, m, ldp)
    z = _cycle(api, dataclasses.replace(p, a_val=p.a_val * 2.0 ** e, b_val=p.b_val * 2.0 ** e), sig, R, m, ldp)
    # each within 5e-4 of the FP64 cycle, the bound of the other FP32 cycle checks
    assert np.linalg.norm(z * 2.0 ** e - z0) <= 1e-3 * np.linalg.norm(z0)

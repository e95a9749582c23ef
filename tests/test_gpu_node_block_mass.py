"""GPU checks of the FP64 products A X, B X on node-block pencils, whose mass
part takes every third entry of a row, through the C ABI."""
import numpy as np
import pytest

from workloads import pencil_2d_q1, pencil_3d_elasticity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_21618_gb300 import api as a
    return a


@pytest.mark.parametrize("pencil,m", [("3d", 1), ("3d", 31), ("3d", 32), ("3d", 33), ("3d_rows2", 7), ("2d", 33)])
@pytest.mark.parametrize("want", [(True, True), (True, False), (False, True)])
def test_each_output_of_the_fp64_product(api, pencil, m, want):
    # a sum of at most 81 products: within 81 * 2^-53 of |M| |X| per entry;
    # graded columns, so that an entry taken from another dof shows
    p = pencil_2d_q1(21, seed=3) if pencil == "2d" else pencil_3d_elasticity(6, seed=5)
    h = api.Handle(p, api.default_opts(spmm_rows=2) if pencil == "3d_rows2" else None)
    X = np.random.default_rng(m).standard_normal((p.n, m)) * np.geomspace(1.0, 1e6, p.n)[:, None]
    Y, Z = h.spmm_ab(torch.from_numpy(X).cuda(), want_a=want[0], want_b=want[1])
    for out, M, w in ((Y, p.A(), want[0]), (Z, p.B(), want[1])):
        if w:
            assert (np.abs(out.cpu().numpy() - M @ X) <= 2 * 81 * 2.0**-53 * (abs(M) @ np.abs(X))).all()

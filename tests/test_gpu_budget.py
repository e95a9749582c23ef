"""GPU checks that calls keep to the memory budget (slrf_opts.mem_budget) they have
always sufficed with: the budgets below are the smallest ones that these calls
took on a GB300 (152 SMs: some workspaces are per SM) before their workspace was
rearranged."""
import numpy as np
import pytest

from workloads import pencil_1d

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("budgets of a 152-SM device")
    from paper_2503_21618_gb300 import api as a
    return a


@pytest.mark.parametrize("m,mode,budget", [(3, 2, 198500), (45, 2, 346004), (160, 2, 2044708),
                                           (161, 2, 2073012), (300, 2, 6684868), (448, 2, 14659108), (449, 2, 14738100),
                                           (160, 1, 2044708)])
def test_syev(api, m, mode, budget):
    rng = np.random.default_rng(m)
    S = rng.standard_normal((m, m))
    S = np.ascontiguousarray(S + S.T)
    h = api.Handle(pencil_1d(600), api.default_opts(mem_budget=budget, eig_refine=mode))
    lam = h.syev(torch.from_numpy(S).cuda())[0].cpu().numpy()
    assert np.abs(lam - np.linalg.eigvalsh(S)).max() <= 1e-13 * np.linalg.norm(S, 2) * max(1, m / 10)

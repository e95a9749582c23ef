"""GPU checks that calls keep to the memory budget (slrf_opts.mem_budget) they have
always sufficed with: the budgets below are the smallest ones that these calls
took on a GB300 (152 SMs: some workspaces are per SM) before their workspace was
rearranged."""
import numpy as np
import pytest

from workloads import pencil_1d, pencil_2d_q1, start_block, weyl_gamma

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


# the level solved by its inverses: 200, 333, 833 and 1 533 unknowns
@pytest.mark.parametrize("n,N,tc,budget", [(600, 1, 0, 1094244), (600, 1, 1, 2551396), (600, 4, 0, 2980116), (600, 4, 1, 8807956),
                                              (1000, 1, 0, 2154580), (1000, 1, 1, 5541524), (1000, 4, 0, 6312644), (1000, 4, 1, 19859652),
                                              (2500, 1, 0, 8660872), (2500, 1, 1, 27627848), (2500, 4, 0, 28904920), (2500, 4, 1, 104772056),
                                              (4600, 1, 0, 24483780), (4600, 1, 1, 82434052), (4600, 4, 0, 87408372), (4600, 4, 1, 319208692)])
def test_exact_level(api, n, N, tc, budget):
    m, ldp = 5, 6
    sig = 0.02 * n * n * (np.linspace(0.1, 1, N) + 1j * np.linspace(0.2, 1, N))
    R = torch.randn(n, N * ldp * 2, generator=torch.Generator("cuda").manual_seed(n), device="cuda")
    z = []
    for b in (budget, 0):
        h = api.Handle(pencil_1d(n), api.default_opts(precond=api.PRECOND_MG, mg_coarse=16, mg_shift_limit=1e30,
                                                      mg_exact_tc=tc, mem_budget=b))
        Z, used = h.precond_apply(api.Filter(sig, np.ones(N)), R, m, ldp)
        assert used == 2
        z.append(Z.cpu().numpy())
    assert np.array_equal(z[0], z[1])


@pytest.mark.parametrize("n,m,budget", [(50021, 127, 208177866), (50021, 211, 412084890)])
def test_gram(api, n, m, budget):
    g = torch.Generator("cuda").manual_seed(m)
    X, Y = (torch.randn(n, m, generator=g, dtype=torch.float64, device="cuda") for _ in range(2))
    G = api.Handle(pencil_1d(n), api.default_opts(mem_budget=budget)).gram(X, Y)
    assert (G - X.T @ Y).abs().max() <= 1e-13 * X.abs().max() * Y.abs().max() * n


@pytest.mark.parametrize("n,m,budget", [(6400, 298, 32913188)])
def test_tall_product(api, n, m, budget):
    g = torch.Generator("cuda").manual_seed(m)
    A = torch.randn(n, m, generator=g, dtype=torch.float64, device="cuda")
    B = torch.randn(m, m, generator=g, dtype=torch.float64, device="cuda")
    C = api.Handle(pencil_1d(n), api.default_opts(mem_budget=budget)).tall_product(A, B)
    assert (C - A @ B).abs().max() <= 1e-13 * A.abs().max() * B.abs().max() * m


# Gram, tall products and their smaller forms within one call
@pytest.mark.parametrize("n,m,budget", [(50021, 127, 525128286)])
def test_rayleigh_ritz(api, n, m, budget):
    p = pencil_1d(n)
    U = torch.randn(n, m, generator=torch.Generator("cuda").manual_seed(m), dtype=torch.float64, device="cuda")
    theta, X, resid = api.Handle(p, api.default_opts(mem_budget=budget)).rayleigh_ritz(U)[:3]
    theta0, X0, resid0 = api.Handle(p).rayleigh_ritz(U)[:3]
    assert (theta - theta0).abs().max() <= 1e-12 * theta0.abs().max()
    assert (resid - resid0).abs().max() <= 1e-10


# the whole default solve: the Krylov blocks come after the projection's
@pytest.mark.parametrize("size,nev,cols,budget", [(150, 80, 120, 745270286)])
def test_solve(api, size, nev, cols, budget):
    p, gamma = pencil_2d_q1(size), weyl_gamma("2d", nev)
    V0 = torch.from_numpy(start_block(p.n, cols, 3)).cuda()
    h = api.Handle(p, api.default_opts(mem_budget=budget))
    status = h.subspace_iterate(api.design_poles("slrf", 4, gamma, 1.0, 0.01), gamma, V0, tol=1e-8, max_outer=1)[4]
    assert status in (api.OK, api.NOT_CONVERGED, api.SUBSPACE_TOO_SMALL)

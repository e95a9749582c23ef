"""GPU checks of the digit products on the tensor cores (Grams, tall products)
at the edges of their tiles, K steps and slices, and of the values the digit
split has to carry exactly."""
import numpy as np
import pytest
from workloads import pencil_1d, start_block

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_21618_gb300 import api as a
    return a


# rows: below, at and above a K step (32) and a slice (at most 480 rows)
# columns: 64-row panels, 128-row tiles with one panel in the last
@pytest.mark.parametrize("n", [31, 32, 33, 479, 480, 481, 961, 5000])
@pytest.mark.parametrize("m", [1, 16, 63, 64, 65, 128, 129, 193])
def test_gram_at_tile_edges(api, n, m):
    n = max(n, 8)
    X, Y = start_block(n, m, 1), start_block(n, m, 2)
    G = api.Handle(pencil_1d(n)).gram(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()).cpu().numpy()
    assert np.abs(G - X.T @ Y).max() <= 1e-13 * np.abs(X).max() * np.abs(Y).max() * n


@pytest.mark.parametrize("value", [1.9999999999999998, 1.0, -1.9999999999999998])
def test_gram_of_extreme_constant_columns(api, value):
    # every digit product at its largest: the sums of a slice reach their bound
    n, m = 4801, 66
    X = np.full((n, m), value)
    X[:, 1::2] *= -1.0
    G = api.Handle(pencil_1d(n)).gram(torch.from_numpy(X).cuda(), torch.from_numpy(X).cuda()).cpu().numpy()
    np.testing.assert_allclose(G, X.T @ X, rtol=2e-15)


def test_gram_of_whole_numbers_is_exact(api):
    n, m = 3000, 70
    rng = np.random.default_rng(0)
    X, Y = rng.integers(-1000, 1001, (n, m)).astype(float), rng.integers(-1000, 1001, (n, m)).astype(float)
    G = api.Handle(pencil_1d(n)).gram(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()).cpu().numpy()
    np.testing.assert_array_equal(G, X.T @ Y)


@pytest.mark.parametrize("n", [63, 64, 65, 127, 129, 1000])
@pytest.mark.parametrize("k,m", [(1, 1), (31, 64), (32, 65), (33, 16), (150, 129), (480, 40), (481, 17), (512, 3)])
def test_tall_product_at_tile_edges(api, n, k, m):
    rng = np.random.default_rng(k)
    A, B = rng.standard_normal((n, k)), rng.standard_normal((k, m))
    C = api.Handle(pencil_1d(n)).tall_product(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()).cpu().numpy()
    assert np.all(np.abs(C - A @ B) <= 1e-13 * (np.abs(A) @ np.abs(B)))


@pytest.mark.parametrize("k", [160, 480, 512])
def test_tall_product_of_extreme_rows(api, k):
    n, m = 200, 70
    A, B = np.full((n, k), 1.9999999999999998), np.full((k, m), 1.9999999999999998)
    A[::2] *= -1.0
    C = api.Handle(pencil_1d(n)).tall_product(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()).cpu().numpy()
    np.testing.assert_allclose(C, A @ B, rtol=2e-15)

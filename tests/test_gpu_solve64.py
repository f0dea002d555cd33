"""FP64 solves with the factors (cf_getrs, cf_potrs): block, cluster and
super-block edges against substitution's own error bound, and the row order of
any list of interchanges."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def cf():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2108_09337_gb300 import cf as _cf
    return _cf


def _dev(A, ld=None):
    n, m = A.shape
    big = torch.zeros((m, ld or n), dtype=torch.float64)
    big[:, :n] = torch.from_numpy(np.ascontiguousarray(A.T))
    return big.cuda().t()[:n, :]


def _triangles(n, rng):
    L = np.tril(rng.uniform(-1, 1, (n, n)), -1) / np.sqrt(n)
    Um = np.triu(rng.uniform(-1, 1, (n, n)), 1) / np.sqrt(n) + np.diag(rng.uniform(0.5, 3, n) * rng.choice([-1, 1], n))
    return L, Um


def _within(T, X, B):
    """|b - T x| <= 2 (n + 4) u |T| |x|: n + 4 for the substitution (Higham 2002,
    theorem 8.5), as much for the product formed here."""
    n = T.shape[0]
    return (np.abs(B - T @ X) <= 2 * (n + 4) * U * (np.abs(T) @ np.abs(X))).all()


@pytest.mark.parametrize("n,nrhs,ld,ldb", [(1, 1, None, None), (63, 2, 70, 64), (64, 1, None, None), (65, 3, None, None),
                                           (129, 17, 131, 133), (577, 1, None, None), (2047, 1, None, None),
                                           (2048, 4, None, None), (2049, 2, 2051, 2050), (4161, 5, None, None)])
def test_solves_within_substitution_bound(cf, n, nrhs, ld, ldb):
    rng = np.random.default_rng(n + nrhs)
    L, Um = _triangles(n, rng)
    B = rng.standard_normal((n, nrhs))
    B[:, 0] = 0.0
    B[n // 2, 0] = 1.0                       # zeros on the way to the first entry
    ident = torch.arange(1, n + 1, dtype=torch.int32, device="cuda")
    eye = np.eye(n)
    # L alone (U = I), U alone (L = I)
    X = cf.getrs(_dev(L + eye, ld), ident, _dev(B, ldb)).cpu().numpy()
    assert _within(L + eye, X, B)
    X = cf.getrs(_dev(Um, ld), ident, _dev(B, ldb)).cpu().numpy()
    assert _within(Um, X, B)
    # both Cholesky triangles: L y = b, L^T x = y
    Lc = np.tril(Um.T)
    X = cf.potrs(_dev(Lc, ld), _dev(B, ldb)).cpu().numpy()
    R = np.abs(B - Lc @ (Lc.T @ X))
    assert (R <= 6 * (n + 4) * U * (np.abs(Lc) @ (np.abs(Lc.T) @ np.abs(X)))).all()
    assert cf.device_status() == cf.CF_OK


@pytest.mark.parametrize("n", [1, 2, 95, 127, 128, 129, 300, 1000, 2500])
@pytest.mark.parametrize("kind", ["lapack", "any", "one", "reverse"])
def test_row_order_of_interchanges(cf, n, kind):
    """ipiv played one interchange at a time; U = I and L = I leave P b."""
    rng = np.random.default_rng(n)
    i = np.arange(n)
    ip = {"lapack": lambda: i + (rng.random(n) * (n - i)).astype(int), "any": lambda: rng.integers(0, n, n),
          "one": lambda: np.full(n, n - 1), "reverse": lambda: n - 1 - i}[kind]()
    perm = np.arange(n)
    for k in range(n):
        perm[[k, ip[k]]] = perm[[ip[k], k]]
    b = rng.standard_normal((n, 1))
    X = cf.getrs(_dev(np.eye(n)), torch.from_numpy((ip + 1).astype(np.int32)).cuda(), _dev(b)).cpu().numpy()
    np.testing.assert_array_equal(X, b[perm])


def test_singular_and_non_finite_values_pass_through(cf):
    """Zero pivots and non-finite right-hand sides give what the division gives."""
    n = 70
    T = np.eye(n)
    T[40, 40] = 0.0
    T[50, 50] = np.inf
    b = np.ones((n, 2))
    b[10, 1], b[40, 1] = np.nan, 0.0
    ident = torch.arange(1, n + 1, dtype=torch.int32, device="cuda")
    X = cf.getrs(_dev(T), ident, _dev(b)).cpu().numpy()
    # forward: 0 * NaN = NaN reaches every row below 10; backward: every row above, and 0 * inf those above 40
    assert np.isnan(X[:, 1]).all()
    assert np.isposinf(X[40, 0]) and np.isnan(X[:40, 0]).all()
    assert X[50, 0] == 0 and (X[51:, 0] == 1).all() and (X[41:50, 0] == 1).all()

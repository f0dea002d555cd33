"""cf_getrs rounds every operation in one fixed order, whatever the number of
right-hand sides: a solution of an ill-conditioned system is what it was, to
the last bit, not one of the many within the error bound."""
import ctypes
import ctypes.util

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


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


def _fma():
    f = ctypes.CDLL(ctypes.util.find_library("m")).fma
    f.restype, f.argtypes = ctypes.c_double, [ctypes.c_double] * 3
    g = np.frompyfunc(f, 3, 1)
    return lambda a, b, c: g(a, b, c).astype(np.float64)


def _solve(T, b, lower):
    """Blocks of 128 in the triangle's order; in a block a rounded multiply and a
    rounded subtract per column, a rounded division by U's diagonal; then the
    other rows less one FMA chain over the block's columns, ascending."""
    fma, n, x = _fma(), T.shape[0], b.copy()
    starts = list(range(0, n, 128))
    for k0 in starts if lower else starts[::-1]:
        k1 = min(n, k0 + 128)
        for k in range(k0, k1) if lower else range(k1 - 1, k0 - 1, -1):
            if not lower:
                x[k] /= T[k, k]
            rows = slice(k + 1, k1) if lower else slice(k0, k)
            x[rows] = x[rows] - T[rows, k] * x[k]
        rows = slice(k1, n) if lower else slice(0, k0)
        acc = np.zeros(rows.stop - rows.start)
        if acc.size:
            for k in range(k0, k1):
                acc = fma(T[rows, k], np.full(acc.size, x[k]), acc)
            x[rows] = x[rows] - acc
    return x


def _factors(n, rng, scale):
    """L U packed; with scale, U's rows (and the right-hand sides) over 2^+-500."""
    LU = rng.uniform(-1, 1, (n, n)) / np.sqrt(n)
    LU[np.arange(n), np.arange(n)] = rng.uniform(0.5, 3, n) * rng.choice([-1, 1], n)
    d = 2.0 ** rng.integers(-500, 501, n) if scale else np.ones(n)
    return np.tril(LU, -1), np.triu(LU) * d[:, None], d


@pytest.mark.parametrize("scale", [False, True])
@pytest.mark.parametrize("n", [1, 31, 33, 127, 128, 129, 160, 300, 577, 2200])
def test_operation_order(cf, n, scale):
    rng = np.random.default_rng(n)
    L, Um, d = _factors(n, rng, scale)
    ident = torch.arange(1, n + 1, dtype=torch.int32, device="cuda")
    b = rng.standard_normal(n) * d
    B = _dev(np.stack([b, b[::-1]], axis=1)) if n == 300 else _dev(b[:, None])
    X = cf.getrs(_dev(Um, n + 1), ident, B).cpu().numpy()           # L = I
    np.testing.assert_array_equal(X[:, 0], _solve(Um, b, False))
    b = rng.standard_normal(n)
    X = cf.getrs(_dev(L + np.eye(n)), ident, _dev(b[:, None], n + 3)).cpu().numpy()      # U = I
    np.testing.assert_array_equal(X[:, 0], _solve(L, b, True))
    assert cf.device_status() == cf.CF_OK


@pytest.mark.parametrize("n,nrhs", [(1, 129), (65, 129), (256, 200), (257, 257), (300, 300), (577, 1025), (2200, 260)])
def test_many_right_hand_sides(cf, n, nrhs):
    """Above a few hundred right-hand sides the solves go block by block over
    all of them: the same bits with LU factors, substitution's bound with Cholesky's."""
    u = 2.0 ** -53
    rng = np.random.default_rng(n)
    L, Um, _ = _factors(n, rng, False)
    B = rng.standard_normal((n, nrhs))
    ip = torch.from_numpy(np.arange(n, 0, -1).astype(np.int32)).cuda()        # any list is played
    LU = _dev(L + Um, n + 2)
    X = cf.getrs(LU, ip, _dev(B, n + 1)).cpu().numpy()
    for c in (0, nrhs // 2, nrhs - 1):
        np.testing.assert_array_equal(X[:, [c]], cf.getrs(LU, ip, _dev(B[:, [c]])).cpu().numpy())
    Lc = np.tril(Um.T)
    X = cf.potrs(_dev(Lc, n + 2), _dev(B, n + 1)).cpu().numpy()
    R = np.abs(B - Lc @ (Lc.T @ X))
    assert (R <= 6 * (n + 4) * u * (np.abs(Lc) @ (np.abs(Lc.T) @ np.abs(X)))).all()
    assert cf.device_status() == cf.CF_OK

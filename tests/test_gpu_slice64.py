"""The FP64 Schur update from digit slices on the tensor cores (cf_getrf and
cf_potrf with their optimal workspace) against the oracle's measures and the
FP64 loop (minimal workspace)."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2108_09337_gb300 import inputs

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


def _minimal(cf, n, **kw):
    return torch.empty(cf.workspace_size("getrf", n, **kw), dtype=torch.uint8, device="cuda")


def _componentwise(A, LU, ip):
    """max |P A - L U| / (|L| |U|), the measure in which the FP64 loop is
    backward stable to about n u whatever the rows' and columns' scales; the
    product is formed in FP64 here, which adds at most another n u."""
    n = A.shape[0]
    perm = oracle.perm_from_ipiv(ip, n)
    L, Uf = np.tril(LU, -1) + np.eye(n), np.triu(LU)
    den = np.abs(L) @ np.abs(Uf)
    return (np.abs(A[perm] - L @ Uf) / np.where(den > 0, den, 1)).max()


# tile edges (128 rows, 64 columns), widths of one and two K blocks, widths
# that are no multiple of anything, ld > n
@pytest.mark.parametrize("n,v,ld", [(129, 128, None), (256, 64, 259), (257, 128, None), (321, 17, None),
                                    (640, 100, 641), (450, 65, None), (1283, 128, None)])
@pytest.mark.parametrize("grading", ["none", "rows", "columns", "both"])
def test_lu_componentwise_error(cf, n, v, ld, grading):
    """Row and column scalings over 2^+-200 included: |P A - L U| <= 2 n u |L||U|
    (the FP64 loop's own bound and the check's) with every element's update taken from slices."""
    A = inputs.uniform_pm1(n, seed=n + v)
    rng = np.random.default_rng(n)
    if grading in ("rows", "both"):
        A *= 2.0 ** rng.integers(-200, 201, (n, 1))
    if grading in ("columns", "both"):
        A *= 2.0 ** rng.integers(-200, 201, (1, n))
    dA = _dev(A, ld)
    ipiv, info = cf.getrf(dA, v=v)
    assert int(info.item()) == 0
    assert _componentwise(A, dA.cpu().numpy(), ipiv.cpu().numpy()) <= 2 * n * U


@pytest.mark.parametrize("n,v", [(129, 128), (321, 17), (640, 100), (1283, 128)])
def test_cholesky_componentwise_error(cf, n, v):
    S = inputs.spd_gram(n, seed=n)
    d = 2.0 ** np.random.default_rng(n).integers(-100, 101, n)
    S = S * d[:, None] * d[None, :]
    dS = _dev(S)
    assert int(cf.potrf(dS, v=v).item()) == 0
    L = np.tril(dS.cpu().numpy())
    den = np.abs(L) @ np.abs(L).T
    res = np.abs(S - L @ L.T)
    assert (res / den).max() <= 2 * n * U


def test_exact_integers(cf):
    """Integer factors: every product and sum is exact, so the factors are."""
    n = 200
    rng = np.random.default_rng(3)
    L0 = np.tril(rng.integers(-2, 3, (n, n)).astype(float), -1) + 4 * np.eye(n)
    dS = _dev(np.asfortranarray(L0 @ L0.T))
    assert int(cf.potrf(dS, v=32).item()) == 0
    np.testing.assert_array_equal(np.tril(dS.cpu().numpy()), L0)


@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e300, 1e-300])
def test_non_finite_and_extreme_rows_take_the_fp64_loop(cf, bad):
    """Where a value is not finite the result is what the FP64 loop gives;
    elsewhere both agree to rounding."""
    n = 700
    A = inputs.uniform_pm1(n, seed=8, shift=4.0 * np.sqrt(n))      # pivots stay on the diagonal
    A[650, 40] = bad
    out = []
    for work in (None, _minimal(cf, n)):
        dA = _dev(A)
        cf.getrf(dA, work=work)
        out.append(dA.cpu().numpy())
    a, b = out
    np.testing.assert_array_equal(np.isnan(a), np.isnan(b))
    np.testing.assert_array_equal(np.isposinf(a), np.isposinf(b))
    np.testing.assert_array_equal(np.isneginf(a), np.isneginf(b))
    ok = np.isfinite(b)
    scale = np.abs(np.where(ok, b, 0)).max(axis=1, keepdims=True)
    assert (np.abs(np.where(ok, a, 0) - np.where(ok, b, 0)) <= 100 * n * U * scale).all()


def test_minimal_and_null_workspaces_stay_accepted(cf):
    n = 300
    L = cf.lib()
    o = ctypes.byref(cf.options())
    assert L.cf_potrf_workspace_size(n, o) == 0
    assert L.cf_getrf_optimal_workspace_size(n, o) > L.cf_getrf_workspace_size(n, o)
    assert L.cf_getrf_optimal_workspace_size(100, o) < 1 << 20
    A, S = inputs.uniform_pm1(n, seed=1), inputs.spd_gram(n, seed=2)
    dA = _dev(A)
    ipiv, info = cf.getrf(dA, work=_minimal(cf, n))
    assert _componentwise(A, dA.cpu().numpy(), ipiv.cpu().numpy()) <= 2 * n * U
    dS = _dev(S)
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = L.cf_potrf(n, ctypes.c_void_p(dS.data_ptr()), n, ctypes.c_void_p(info.data_ptr()), None, 0, o,
                    ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0 and int(info.item()) == 0
    assert oracle.chol_residual(S, np.tril(dS.cpu().numpy())) <= 20.0

"""cf_getrf on matrices whose elements differ by many orders of magnitude in a
way that no row or column scaling takes out: every element of P A - L U stays
within the FP64 update's own bound, whatever else the matrix holds, and the
factors do not depend on the workspace given (its size, its alignment) or on the
schedule."""
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


def _dev(A):
    return torch.from_numpy(np.ascontiguousarray(A.T)).cuda().t()


def _componentwise(A, LU, ip):
    """max |P A - L U| / (|L| |U|): n u for the elimination, as much for the product formed here."""
    n = A.shape[0]
    L, Uf = np.tril(LU, -1) + np.eye(n), np.triu(LU)
    den = np.abs(L) @ np.abs(Uf)
    return (np.abs(A[oracle.perm_from_ipiv(ip, n)] - L @ Uf) / np.where(den > 0, den, 1)).max()


def _matrix(kind, n, t):
    """U[-1, 1] entries and elements of 2^t: one right of the first panel in a row that is pivoted there, a column
    with a few, a row of them but for one element, blocks of two units."""
    A = inputs.uniform_pm1(n, seed=n)
    big = 2.0 ** t
    if kind == "one":
        A[5, 0] = 2.0                                # the first pivot row
        A[5, n - 40] = big
    elif kind == "column":
        A[[3, n // 2, n - 2], n - 40] = big
    elif kind == "row":
        A[7, :] *= big
        A[7, n - 3] /= big
    else:
        A[n // 2:, n // 2:] *= big
        A[:64, :64] *= big
    return A


@pytest.mark.parametrize("kind", ["one", "column", "row", "blocks"])
@pytest.mark.parametrize("t", [20, 50, 100, 300])
@pytest.mark.parametrize("n,v", [(400, 128), (330, 50)])
def test_elements_of_two_magnitudes(cf, kind, t, n, v):
    A = _matrix(kind, n, t)
    out = []
    for how in ("default", "minimal", "one stream", "noalloc"):
        dA = _dev(A)
        if how == "noalloc":
            ipiv, info = cf.getrf_noalloc(dA, v=v)
        else:
            work = torch.empty(cf.workspace_size("getrf", n, v=v), dtype=torch.uint8, device="cuda")
            ipiv, info = cf.getrf(dA, v=v, work=work if how == "minimal" else None,
                                  lookahead=0 if how == "one stream" else 1)
        assert int(info.item()) == 0
        out.append((dA.cpu().numpy(), ipiv.cpu().numpy()))
    assert _componentwise(A, *out[0]) <= 2 * n * U
    for LU, ip in out[1:]:
        np.testing.assert_array_equal(LU, out[0][0])
        np.testing.assert_array_equal(ip, out[0][1])


@pytest.mark.parametrize("offset", [4, 8, 12, 16, 500])
@pytest.mark.parametrize("lookahead", [0, 1])
def test_work_of_any_int_alignment(cf, offset, lookahead):
    n = 300
    A = inputs.uniform_pm1(n, seed=2)
    ref = _dev(A)
    ipiv_ref, _ = cf.getrf(ref)
    size = cf.lib().cf_getrf_optimal_workspace_size(n, ctypes.byref(cf.options()))
    work = torch.empty(size + offset + 4, dtype=torch.uint8, device="cuda")
    work[offset + size:] = 77                        # nothing is written past the size asked for
    dA = _dev(A)
    ipiv, info = cf.getrf(dA, work=work[offset:offset + size], lookahead=lookahead)
    assert int(info.item()) == 0 and bool((work[offset + size:] == 77).all())
    np.testing.assert_array_equal(dA.cpu().numpy(), ref.cpu().numpy())
    np.testing.assert_array_equal(ipiv.cpu().numpy(), ipiv_ref.cpu().numpy())

"""The FP32 factorizations of a panel's leading block (LU on a 4 x 4 grid of 16 x
16 threads, Cholesky with a column per warp) at the edges of their thread grids,
through the refined solves: A x = b to the refinement's bar for every width, with
entries of one size and of sizes over many binades, and the failing pivot's
index."""
import numpy as np
import pytest
import torch

import oracle
from paper_2108_09337_gb300 import inputs

pytestmark = pytest.mark.gpu
WIDTHS = [1, 15, 16, 17, 33, 63, 64, 65, 127, 128, 131]


@pytest.fixture(scope="module")
def cf():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2108_09337_gb300 import cf as _cf
    return _cf


def _dev(A):
    return torch.from_numpy(np.ascontiguousarray(A.T)).cuda().t()


# Off-diagonal entries span 2^-2*spread .. 1; a strictly dominant diagonal keeps the
# refinement's contraction whatever the spread.
@pytest.mark.parametrize("spread", [0, 60])
@pytest.mark.parametrize("solver", ["gesv", "posv"])
@pytest.mark.parametrize("n", WIDTHS)
def test_leading_block_widths(cf, solver, n, spread):
    rng = np.random.default_rng(100 * n + spread)
    A = rng.uniform(-1, 1, (n, n)) * 2.0 ** -rng.integers(0, 2 * spread + 1, (n, n))
    if solver == "posv":
        A = np.tril(A, -1)
        A = A + A.T
    A[np.arange(n), np.arange(n)] = np.abs(A).sum(axis=1) + 1.0
    B = inputs.rhs_normal(n, 2, seed=3)
    f = cf.gesv_mixed if solver == "gesv" else cf.posv_mixed
    X, info, stats, st = f(_dev(A), _dev(B), prec="bf16")
    assert st == cf.CF_OK and int(info.item()) == 0 and stats.converged == 1
    assert oracle.backward_error(A, X.cpu().numpy(), B).max() <= 1e-14


@pytest.mark.parametrize("n,k", [(1, 0), (17, 15), (64, 16), (64, 63), (128, 0), (128, 127), (200, 130)])
def test_failing_pivot_index(cf, n, k):
    """Row and column k are zero but for the diagonal, which is negative
    (Cholesky) or zero (LU): the k-th pivot is the first to fail, info = k + 1."""
    A = np.eye(n) * 4.0 + 1.0 / n
    A[k, :] = A[:, k] = 0.0
    B = inputs.rhs_normal(n, 1, seed=3)
    for f, d in ((cf.posv_mixed, -1.0), (cf.gesv_mixed, 0.0)):
        A[k, k] = d
        info = f(_dev(A), _dev(B), prec="bf16")[1]
        assert int(info.item()) == k + 1


# LU-3 and the slab's LU-4 in one launch: fixed widths, other ones, ragged last
# panels (with 99, a panel of 64 columns at an odd column: a launch for each), and
# slabs with and without columns right of the panel.
@pytest.mark.parametrize("prec", ["f16", "bf16x3"])
@pytest.mark.parametrize("n,v", [(300, 7), (300, 48), (321, 64), (361, 99), (163, 99), (300, 128), (129, 64)])
def test_panel_solves_any_width(cf, n, v, prec):
    A = inputs.uniform_pm1(n, seed=n + v, shift=2 * np.sqrt(n))
    B = inputs.rhs_normal(n, 3, seed=3)
    X, info, stats, st = cf.gesv_mixed(_dev(A), _dev(B), prec=prec, v=v)
    assert st == cf.CF_OK and int(info.item()) == 0 and stats.converged == 1
    assert oracle.backward_error(A, X.cpu().numpy(), B).max() <= 1e-14

"""Failure detection of the FP64 kernels' bounded waits.  The failure is made
by a thread that does not send what others wait for: every wait for it gives up
after its limit, the kernel ends with every index in range, cf_device_status
reports CF_ERR_TIMEOUT once and is clear after, and the next call is right.
Nothing here faults, traps or hangs the GPU."""
import time

import numpy as np
import pytest
import torch

from paper_2108_09337_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cf():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2108_09337_gb300 import cf as _cf
    return _cf


def _dev(A):
    return torch.from_numpy(np.ascontiguousarray(A.T)).cuda().t()


def _times_out_once(cf, call):
    assert cf.device_status() == cf.CF_OK
    t0 = time.time()
    out = call()
    assert cf.device_status() == cf.CF_ERR_TIMEOUT        # synchronises
    dt = time.time() - t0
    assert dt < 5.0
    assert cf.device_status() == cf.CF_OK                 # reported once, then cleared
    return out


@pytest.mark.parametrize("m,w,leaf_h,arity", [(1, 1, 128, 2), (40, 7, 128, 2), (64, 20, 32, 2), (300, 128, 128, 8),
                                              (700, 100, 64, 3), (2048, 128, 128, 8), (129, 128, 1, 8)])
@pytest.mark.parametrize("spin", [1 << 10, 0])
def test_tournament_wait_runs_out(cf, m, w, leaf_h, arity, spin):
    P = _dev(inputs.uniform_pm1(max(m, w), seed=m)[:m, :w])
    ref = cf.tourn_select(P, leaf_h, arity).cpu().numpy()
    win = _times_out_once(cf, lambda: cf.tourn_select_withheld(P, leaf_h, arity, spin)).cpu().numpy()
    assert win.min() >= 0 and win.max() < m and len(set(win.tolist())) == min(m, w)
    np.testing.assert_array_equal(cf.tourn_select(P, leaf_h, arity).cpu().numpy(), ref)
    assert cf.device_status() == cf.CF_OK


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("n,nrhs,spin", [(130, 1, 1 << 10), (300, 3, 1 << 10), (2048, 1, 1 << 10), (2048, 2, 0),
                                         (2500, 1, 1 << 10)])
def test_solve_wait_runs_out(cf, mode, n, nrhs, spin):
    rng = np.random.default_rng(n)
    T = rng.uniform(-1, 1, (n, n)) / n + 2 * np.eye(n)
    X = _dev(rng.standard_normal((n, nrhs)))
    _times_out_once(cf, lambda: cf.tri_solve64_withheld(_dev(T), X, mode, spin))
    # the next solve is right
    b = rng.standard_normal((n, nrhs))
    if mode < 2:
        ident = torch.arange(1, n + 1, dtype=torch.int32, device="cuda")
        x = cf.getrs(_dev(T), ident, _dev(b)).cpu().numpy()
        r = (np.tril(T, -1) + np.eye(n)) @ (np.triu(T) @ x) - b
    else:
        x = cf.potrs(_dev(T), _dev(b)).cpu().numpy()
        r = np.tril(T) @ (np.tril(T).T @ x) - b
    assert cf.device_status() == cf.CF_OK
    assert np.abs(r).max() <= 6 * (n + 4) * 2.0 ** -53 * 16 * np.abs(b).max()

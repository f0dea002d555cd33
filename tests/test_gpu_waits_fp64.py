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

"""The refinement's solve with FP32 factors in FP64 arithmetic: every number of
right-hand sides that its kernels are made for, in one chain and in groups.

Tolerance: substitution through inverses of the 64 x 64 diagonal blocks, whose
condition is below 5 here as the triangles' is: n + 64 products per row, each
step's error at most 25 u of it, max |x| for every |x|."""
import numpy as np
import pytest
import torch

from tests import test_gpu_waits as waits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("n,nrhs", [(1, 1), (64, 4), (65, 5), (200, 8), (1000, 9), (1027, 16)])
@pytest.mark.parametrize("chains", [0, 1, 2])
def test_chains(mode, n, nrhs, chains):
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2108_09337_gb300 import cf
    T = waits._tri(n, mode, seed=n + mode)
    B = np.random.default_rng(n).standard_normal((n, nrhs))
    X = torch.from_numpy(np.ascontiguousarray(B.T)).cuda().t()
    cf.trsv_f32_f64x(waits._dev32(T), X, mode, chains)
    assert cf.device_status() == cf.CF_OK
    ref = waits._reference(T, np.asfortranarray(B), mode)
    assert np.abs(X.cpu().numpy() - ref).max() <= 25 * (n + 64) * 2.0 ** -53 * np.abs(ref).max()

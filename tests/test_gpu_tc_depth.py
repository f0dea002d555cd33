"""The tensor-core update on both sides of the depth where its epilogue
changes, ragged and narrow outputs included: small integers, so that every sum
is exact and the results are equal."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [64, 1600, 1664, 2048])
@pytest.mark.parametrize("m,n,lower", [(1, 1, False), (129, 257, False), (300, 640, False), (700, 700, True), (257, 100, False),
                                       (130, 300, True)])
@pytest.mark.parametrize("ksplit", [1, 2])
def test_integer_sums(k, m, n, lower, ksplit):
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2108_09337_gb300 import cf
    g = torch.Generator(device="cuda").manual_seed(k + m)
    A = torch.randint(-1, 2, (m, k), generator=g, device="cuda").half()
    B = torch.randint(-1, 2, (n, k), generator=g, device="cuda").half()
    C0 = torch.randint(-9, 10, (n, m + 3), generator=g, device="cuda").float()
    big = C0.clone()
    C = big.t()[:m, :]
    if ksplit == 1:
        cf.schur_update_lp(A, B, C, lower)
    else:
        cf.schur_update_lp_splitk(A, B, C, ksplit, lower)
    assert cf.device_status() == cf.CF_OK
    want = C0.clone()
    prod = (A.double() @ B.double().t()).float()
    want.t()[:m, :].sub_(prod.tril() if lower else prod)
    assert torch.equal(big, want)                     # the rows past m, too

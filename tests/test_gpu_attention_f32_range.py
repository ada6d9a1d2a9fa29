"""fp32 attention over values near the top of the fp32 range.  The scores jump by 5.5
(7.93 in log2 units, less than moves a row's softmax reference) between runs of 128
keys, in every split of the keys, so the probabilities against the reference reach
2^7.93.  sum p v with p <= 1 stays below 4096 * 5e34 = 2.1e38, so the outputs are
finite.  Tolerance: an fp32 sum of 4096 positive terms is off by at most 4096 * 2^-24
of its value in any order, 2.5e-4, and by its square root, 4e-6, for independent
roundings; 2e-5 leaves a factor of five."""
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def hsa():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_06892_gb300 as m
    m.lib()
    torch.cuda.set_device(0)
    assert m.hsa_get_device_error() == 0
    return m


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("H,n", [(1, 33), (40, 1200)])     # keys split over a cluster, and not
def test_large_values(hsa, H, n, D):
    N = 4096
    g = torch.Generator().manual_seed(D + n)
    q = torch.zeros((n, H, D))
    q[:, :, 0] = 1.0
    k = torch.randn((N, H, D), generator=g)
    k[:, :, 0] = 5.5 * (torch.arange(N) // 128 % 2).float()[:, None]
    v = (0.5 + 0.5 * torch.rand((N, H, D), generator=g)) * 5e34
    out = torch.empty((n, H, D), device=DEV)
    hsa.hsa_active_attention(q.to(DEV), None, n, k.to(DEV), v.to(DEV), out, scale=1.0)
    assert hsa.hsa_get_device_error() == 0
    ref = oracle.attention(q[:1].contiguous(), k, v, scale=1.0)     # every row is alike
    rel = (out.cpu().double() - ref).abs() / ref.abs()
    assert bool(torch.isfinite(out).all())
    assert rel.max().item() <= 2e-5

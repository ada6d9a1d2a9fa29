"""The boundary select where a range that holds too many keys holds one value only,
beside ranges that must be split further in the same pass: a statistic of few values,
one whose values are rounded to 8 bits of mantissa, and one value among neighbouring
floats.  Sizes at the ends of the select's range.  Equal to a stable sort."""
import pytest
import torch

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


def _stat(kind, N, gen):
    if kind == "few":
        return torch.randint(0, 8, (N,), generator=gen).float()
    if kind == "rounded":
        return torch.randn(N, generator=gen).exp().bfloat16().float()
    if kind == "two":                   # the range is one step of the last bit
        return torch.randint(0, 2, (N,), generator=gen).float() * 2.0 ** -23 + 1.0
    z = torch.randint(0, 4096, (N,), generator=gen).float() * 2.0 ** -23 + 1.0
    z[torch.rand(N, generator=gen) < 0.4] = 5.0
    z[torch.rand(N, generator=gen) < 0.1] = -2.0
    z[3], z[N - 5] = -3e38, 3e38
    return z


@pytest.mark.parametrize("kind", ["few", "rounded", "two", "beside"])
@pytest.mark.parametrize("N,K", [(4865, 4), (6145, 32), (98304, 4), (98305, 31), (360448, 3)])
def test_matches_stable_sort(hsa, kind, N, K):
    gen = torch.Generator().manual_seed(N + K)
    stat = _stat(kind, N, gen)
    cuts = sorted(torch.randint(0, N + 1, (K - 1,), generator=gen).tolist())
    counts = [b - a for a, b in zip([0] + cuts, cuts + [N])]
    g = torch.full((N,), -7, dtype=torch.int32, device=DEV)
    ws = torch.empty(hsa.hsa_partition_workspace_bytes(N), dtype=torch.uint8, device=DEV)
    hsa.hsa_partition(stat.to(DEV), 32, (32,) * K, counts, g, ws)
    assert hsa.hsa_get_device_error() == 0
    ref = torch.empty(N, dtype=torch.int32)
    order, lo = torch.sort(stat, stable=True).indices, 0
    for k in range(K - 1, -1, -1):
        ref[order[lo:lo + counts[k]]] = k
        lo += counts[k]
    assert torch.equal(g.cpu(), ref)

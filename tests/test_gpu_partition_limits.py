"""Partition on both sides of every limit between its paths: ranking up to 4864
tokens, the boundary select with 2048 bins up to 98304 and 4096 up to 360448, and the
radix sort beyond, whose scan takes more than one step per CTA above 524288 tokens.
Ties that straddle group boundaries, signed zeros, 1 to 32 groups, empty groups, and
statistics at any 4-byte alignment.  Equal to a stable sort of the statistic."""
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


def _check(hsa, stat, counts, shift):
    N, K = stat.numel(), len(counts)
    sd = torch.empty(N + shift, device=DEV)[shift:]
    sd.copy_(stat)
    g = torch.full((N,), -7, dtype=torch.int32, device=DEV)
    ws = torch.empty(hsa.hsa_partition_workspace_bytes(N), dtype=torch.uint8, device=DEV)
    hsa.hsa_partition(sd, 32, (32,) * K, counts, g, ws)
    ref = torch.empty(N, dtype=torch.int32)
    order, lo = torch.sort(stat + 0.0, stable=True).indices, 0
    for k in range(K - 1, -1, -1):
        ref[order[lo:lo + counts[k]]] = k
        lo += counts[k]
    assert torch.equal(g.cpu(), ref), (N, K, shift)


@pytest.mark.parametrize("N", [33, 4095, 4861, 4863, 4864, 4865, 98304, 98305, 360449, 524289,
                               1000003, 2097153])
def test_both_sides_of_the_limits(hsa, N):
    gen = torch.Generator().manual_seed(N)
    stat = torch.randn(N, generator=gen).exp()
    stat[N // 3: N // 3 + N // 5] = stat[7]            # ties across blocks and CTAs
    stat[5], stat[6] = -0.0, 0.0
    at = int((stat < stat[7]).sum())                   # first rank of the ties
    for K, shift in ((1, 0), (2, 1), (5, 2), (32, 0), (32, 3)):
        cuts = sorted(torch.randint(0, N + 1, (K - 1,), generator=gen).tolist())
        _check(hsa, stat, [b - a for a, b in zip([0] + cuts, cuts + [N])], shift)
    cut = N - at - N // 10                             # inside the run of ties
    for counts in ((cut, N - cut), (0, cut, N - cut), (cut, N - cut, 0), (0, N, 0)):
        _check(hsa, stat, counts, 1)
    assert hsa.hsa_get_device_error() == 0

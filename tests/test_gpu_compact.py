"""Active set and token reordering at the sizes where their launch changes: one
CTA, one cluster with one token per thread, clusters with four, several rounds;
group ids at any 4-byte alignment.  Whole numbers: equal to the definition."""
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


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("N", [1, 33, 1024, 1025, 8191, 8192, 8193, 32768, 32769, 393216, 393217,
                               786433])
def test_compaction(hsa, N, shift):
    gen = torch.Generator().manual_seed(N + shift)
    g = torch.randint(0, 3, (N + shift,), generator=gen, dtype=torch.int32)[shift:]
    gd = torch.empty(N + shift, dtype=torch.int32, device=DEV)[shift:]
    gd.copy_(g)
    idx = torch.full((N,), -7, dtype=torch.int32, device=DEV)
    pos = torch.full((N + shift,), -7, dtype=torch.int32, device=DEV)[shift:]
    hsa.hsa_partition_active(gd, 8, (8, 4, 2), 2, idx, pos)      # groups 0 and 1
    on = g < 2
    n = int(on.sum())
    rank = torch.cumsum(on.int(), 0).int() - 1
    assert torch.equal(idx[:n].cpu(), torch.nonzero(on).reshape(-1).int())
    assert bool((idx[n:] == -7).all())
    assert torch.equal(pos.cpu(), torch.where(on, rank, torch.full_like(rank, -1)))
    order, where, new = (torch.full((N,), -7, dtype=torch.int32, device=DEV) for _ in range(3))
    hsa.hsa_reorder_tokens(gd, int((g == 0).sum()), order, where, new)
    ref = torch.cat((torch.nonzero(g != 0).reshape(-1), torch.nonzero(g == 0).reshape(-1)))
    assert torch.equal(order.cpu(), ref.int())
    assert torch.equal(where.cpu()[ref], torch.arange(N, dtype=torch.int32))
    assert torch.equal(new.cpu(), g[ref])
    assert hsa.hsa_get_device_error() == 0


@pytest.mark.parametrize("N", [5, 9000, 400000])
def test_bad_group_is_skipped_and_reported(hsa, N):
    g = torch.zeros(N, dtype=torch.int32, device=DEV)
    g[N - 1] = 7
    g[N // 2] = -1
    idx = torch.full((N,), -7, dtype=torch.int32, device=DEV)
    pos = torch.empty(N, dtype=torch.int32, device=DEV)
    hsa.hsa_partition_active(g, 8, (8, 4), 1, idx, pos)
    assert hsa.hsa_get_device_error() == -6
    keep = torch.ones(N, dtype=torch.bool)
    keep[N - 1] = keep[N // 2] = False
    assert torch.equal(idx[:N - 2].cpu(), torch.nonzero(keep).reshape(-1).int())
    assert int(pos[N - 1]) == int(pos[N // 2]) == -1

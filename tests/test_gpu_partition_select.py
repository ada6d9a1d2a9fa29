"""The boundary select over the statistics that take its different turns: bins
that hold few keys, ranges split once or more (outliers that stretch the range
over a dense middle), values that more tokens share than a list holds, 32
groups, empty groups, statistics at any 4-byte alignment.  Equal to a stable
sort of the statistic."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"
FLT_MAX = torch.finfo(torch.float32).max


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
    z = torch.randn(N, generator=gen)
    if kind == "lognormal":
        return z.exp()
    if kind == "outliers":              # the whole fp32 range around a dense middle
        z = 1 + z * 1e-4
        z[torch.randperm(N, generator=gen)[:9]] = torch.tensor(
            [FLT_MAX, -FLT_MAX, 0.0, -0.0, 1e-40, -1e-40, 3.0, -3.0, 1e30])
        return z
    if kind == "shared":                # a few values, each shared by thousands
        return torch.tensor([-1.0, 0.0, -0.0, 2.5, 7.0])[torch.randint(0, 5, (N,), generator=gen)]
    if kind == "mixed":                 # one shared value inside a spread
        z = z.exp()
        z[torch.rand(N, generator=gen) < 0.4] = 1.25
        return z
    if kind == "narrow":                # neighbouring floats
        return torch.randint(0, 900, (N,), generator=gen).float() * 2.0 ** -23 + 1.0
    return torch.full((N,), -4.0)


def _reference(stat, counts):
    order = torch.sort(stat.double() + 0.0, stable=True).indices
    g = torch.empty(stat.numel(), dtype=torch.int32)
    lo = 0
    for k in range(len(counts) - 1, -1, -1):
        g[order[lo:lo + counts[k]]] = k
        lo += counts[k]
    return g


@pytest.mark.parametrize("kind", ["lognormal", "outliers", "shared", "mixed", "narrow", "equal"])
@pytest.mark.parametrize("N,K,shift", [(5000, 4, 0), (12033, 4, 1), (40000, 32, 0), (75603, 3, 2),
                                       (360448, 5, 0)])
def test_matches_stable_sort(hsa, kind, N, K, shift):
    gen = torch.Generator().manual_seed(N + K)
    stat = _stat(kind, N, gen)
    cuts = sorted(torch.randint(0, N + 1, (K - 1,), generator=gen).tolist())
    if K == 5:
        cuts = [0, cuts[1], cuts[1], N]                # empty groups, at both ends too
    counts = [b - a for a, b in zip([0] + cuts, cuts + [N])]
    sd = torch.empty(N + shift, device=DEV)[shift:]
    sd.copy_(stat)
    g = torch.full((N,), -7, dtype=torch.int32, device=DEV)
    ws = torch.empty(hsa.hsa_partition_workspace_bytes(N), dtype=torch.uint8, device=DEV)
    hsa.hsa_partition(sd, 32, (32,) * K, counts, g, ws)
    assert hsa.hsa_get_device_error() == 0
    assert torch.equal(g.cpu(), _reference(stat, counts))


def test_nan_is_reported(hsa):
    N = 20000
    stat = torch.randn(N)
    stat[::3] = float("nan")
    stat[1::3] = torch.tensor([-1], dtype=torch.int32).view(torch.float32)   # NaN, sign set
    g = torch.empty(N, dtype=torch.int32, device=DEV)
    ws = torch.empty(hsa.hsa_partition_workspace_bytes(N), dtype=torch.uint8, device=DEV)
    hsa.hsa_partition(stat.to(DEV), 8, (8, 4), (N // 2, N // 2), g, ws)
    assert hsa.hsa_get_device_error() == -5

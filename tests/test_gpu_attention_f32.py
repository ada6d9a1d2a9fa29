"""fp32 active attention over the shapes that change its launch plan: a CTA of
128 rows or of 32 with its warps on different keys, clusters of 1 to 8 CTAs
that split the keys, ragged tiles, empty shares of the keys, two key sources.

Bound: an fp32 sum of n terms of either order is off by about sqrt(n) 2^-24 of
the terms' norm; with N(0,1) inputs and up to 6000 keys that is 5e-6 of an
output of order 1, and the exponent's argument (|x| <= 64 in log2 units, one
rounding) adds 64 * 2^-24 * ln 2 = 3e-6.  1e-4 leaves a factor of ten for the
largest of a million outputs and for the larger scores of the scaled case."""
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"
ATOL = 1e-4


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
@pytest.mark.parametrize("M,B,H,n", [
    (1, 0, 1, 1), (31, 0, 3, 31), (33, 0, 2, 32), (129, 0, 1, 33),
    (1000, 0, 4, 257), (0, 700, 2, 129), (255, 514, 5, 128), (6000, 77, 2, 640),
    (1500, 36, 40, 1536),
])
def test_matches_oracle(hsa, M, B, H, n, D):
    N = M + B
    q = synth.normal((N, H, D), 1)
    k, v = synth.normal((N, H, D), 2), synth.normal((N, H, D), 3)
    idx = synth.uniform_subset(N, n, 4)
    rows = list(range(0, n, max(1, n // 40))) + [n - 1]       # the oracle's rows
    ref = oracle.attention(q, k, v, q_idx=idx[rows].contiguous())
    out = torch.full((n, H, D), 7.0, device=DEV)
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    if B == 0:
        hsa.hsa_active_attention(qd, idx.to(DEV), n, kd, vd, out)
    else:
        hsa.hsa_active_attention_prefix(qd, idx.to(DEV), n, kd[:M].contiguous(),
                                        vd[:M].contiguous(), kd[M:].contiguous(),
                                        vd[M:].contiguous(), out)
    assert hsa.hsa_get_device_error() == 0
    assert (out.cpu().double()[rows] - ref).abs().max().item() <= ATOL


@pytest.mark.parametrize("D", [64, 128])
def test_growing_and_masked_scores(hsa, D):
    """Scores that grow along the keys move every row's reference many times;
    keys at -inf (an infinite component against a negative one) weigh nothing,
    also where they fill whole tiles; a bad index gives a zero query (the mean
    of V) and is reported."""
    N, H, n = 1000, 2, 200
    q = synth.normal((n, H, D), 5).abs()
    k, v = synth.normal((N, H, D), 6), synth.normal((N, H, D), 7)
    k *= torch.linspace(0.1, 8.0, N)[:, None, None]
    ref = oracle.attention(q, k, v)
    out = torch.empty((n, H, D), device=DEV)
    hsa.hsa_active_attention(q.to(DEV), None, n, k.to(DEV), v.to(DEV), out)
    assert (out.cpu().double() - ref).abs().max().item() <= ATOL
    keep = torch.ones(N, dtype=torch.bool)
    keep[64:320] = False
    keep[::7] = False
    kd = k.clone()
    kd[~keep, :, 0] = -float("inf")
    ref = oracle.attention(q, k[keep].contiguous(), v[keep].contiguous())
    hsa.hsa_active_attention(q.to(DEV), None, n, kd.to(DEV), v.to(DEV), out)
    assert (out.cpu().double() - ref).abs().max().item() <= ATOL
    assert hsa.hsa_get_device_error() == 0
    idx = torch.arange(n, dtype=torch.int32)
    idx[3] = N
    qn = synth.normal((N, H, D), 8)
    hsa.hsa_active_attention(qn.to(DEV), idx.to(DEV), n, k.to(DEV), v.to(DEV), out)
    assert hsa.hsa_get_device_error() == -6
    assert (out[3].cpu().double() - v.double().mean(0)).abs().max().item() <= ATOL

"""Rotation of rows whose vectors fall in every way on the lanes of a warp: heads
that divide a lane group and heads that do not, rows shorter than a warp, longer
than one pass, and with a remainder.  bf16 results equal the definition's (fp32
fused multiply-adds, rounded once), so they match the oracle bit for bit."""
import pytest
import torch

import oracle
import synth

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


@pytest.mark.parametrize("H,D", [(1, 8), (3, 8), (1, 16), (2, 24), (1, 64), (5, 72), (9, 96),
                                 (7, 64), (12, 128), (13, 128), (3, 256), (1, 512)])
def test_rows_and_scatter(hsa, H, D):
    N, n = 300, 131
    g = torch.Generator().manual_seed(H * D)
    ang = torch.rand((N, D // 2), generator=g, dtype=torch.float64) * 6.3
    table = torch.stack((torch.cos(ang), torch.sin(ang)), dim=-1).float()
    idx = synth.uniform_subset(N, n, 3)
    x = synth.normal((n, H, D), 4, "bf16")
    kc, vc = synth.normal((N, H, D), 5, "bf16"), synth.normal((N, H, D), 6, "bf16")
    vf = synth.normal((n, H, D), 7, "bf16")
    ref = oracle.rope_rows(x.clone(), idx, table)
    xd, td, idxd = x.to(DEV), table.to(DEV), idx.to(DEV)
    hsa.hsa_rope_rows(xd, idxd, n, td)
    assert torch.equal(xd.cpu(), ref)
    kd, vd = kc.to(DEV), vc.to(DEV)
    hsa.hsa_kv_sync_scatter_rope(kd, vd, x.to(DEV), vf.to(DEV), idxd, n, td)
    kc[idx.long()], vc[idx.long()] = ref, vf
    assert torch.equal(kd.cpu(), kc) and torch.equal(vd.cpu(), vc)
    assert hsa.hsa_get_device_error() == 0

"""The attention kernel's bounded wait running out, in the forms that differ after it:
both head dimensions (two and three S buffers), one key tile and many, whole units and
units whose keys are split (their pieces and the merge), two key sources.  No fault: the
test hook withholds the first value tile.  The call reports HSA_ERR_TIMEOUT, and the
same context then runs the same call correctly."""
import time

import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


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
@pytest.mark.parametrize("M,B,H,n,split", [(100, 0, 1, 70, False), (700, 0, 2, 300, False),
                                           (2000, 0, 2, 300, True), (900, 520, 1, 256, True)])
def test_timeout_is_reported_and_context_survives(hsa, M, B, H, n, split, D):
    N = M + B
    q = synth.normal((n, H, D), 1, "bf16")
    k, v = synth.normal((N, H, D), 2, "bf16"), synth.normal((N, H, D), 3, "bf16")
    dev = [t.cuda() for t in (q, k[:M].contiguous(), v[:M].contiguous(), k[M:].contiguous(),
                              v[M:].contiguous())]
    out = torch.empty((n, H, D), dtype=torch.bfloat16, device="cuda")
    ws = None
    if split:
        ws = torch.zeros(hsa.hsa_active_attention_workspace_bytes(n, N, H, D), dtype=torch.uint8,
                         device="cuda")

    def call():
        c0 = hsa.hsa_launch_count()
        if B:
            hsa.hsa_active_attention_prefix(dev[0], None, n, *dev[1:], out, workspace=ws)
        else:
            hsa.hsa_active_attention(*dev[:1], None, n, *dev[1:3], out, workspace=ws)
        assert hsa.hsa_launch_count() - c0 == (2 if split else 1)

    assert hsa.hsa_test_inject_attention_stall(1) == 0
    try:
        t0 = time.time()
        call()
        status = hsa.hsa_get_device_error()          # synchronises
        elapsed = time.time() - t0
    finally:
        hsa.hsa_test_inject_attention_stall(0)
    assert status == -7                               # HSA_ERR_TIMEOUT
    assert elapsed < 30.0
    call()
    assert hsa.hsa_get_device_error() == 0
    ref = oracle.attention(q, k, v)
    err = out.cpu().double() - ref
    assert err.abs().max() <= 2e-2 and err.norm() / ref.norm() <= 1e-2

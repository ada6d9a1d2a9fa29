"""The grid-stride kernels past their first pass: more rows than the grid has lane
groups (the index of the next row is loaded one row ahead), more vectors than it has
threads, one and two vectors per thread, a bad index or position in a later pass.
Rotations, the cached Euler step and the velocity cache equal the oracle bit for bit;
the statistic, fp32 sums of C absolute values, a division and a fused multiply-add,
within 5e-5 of it."""
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


@pytest.mark.parametrize("H,D", [(5, 64), (12, 64), (3, 72)])
def test_rotations(hsa, H, D):
    N, n = 120000, 90000
    gen = torch.Generator().manual_seed(H * D)
    ang = torch.rand((N, D // 2), generator=gen) * 6.3
    table = torch.stack((torch.cos(ang), torch.sin(ang)), dim=-1)
    idx = synth.uniform_subset(N, n, 3)
    x, vf = synth.normal((n, H, D), 4, "bf16"), synth.normal((n, H, D), 7, "bf16")
    ref = oracle.rope_rows(x.clone(), idx, table)
    bad = 85003                                        # a row of a later pass
    idx_bad = idx.clone()
    idx_bad[bad] = N
    for ix in (idx, idx_bad):
        want = ref.clone()
        keep = torch.ones(n, dtype=torch.bool)
        if ix is idx_bad:
            want[bad] = x[bad]
            keep[bad] = False
        xd, td, id_ = x.to(DEV), table.to(DEV), ix.to(DEV)
        hsa.hsa_rope_rows(xd, id_, n, td)
        assert hsa.hsa_get_device_error() == (0 if ix is idx else -6)
        assert torch.equal(xd.cpu(), want)
        kd, vd = (torch.full((N, H, D), 9.0, dtype=torch.bfloat16, device=DEV) for _ in range(2))
        hsa.hsa_kv_sync_scatter_rope(kd, vd, x.to(DEV), vf.to(DEV), id_, n, td)
        assert hsa.hsa_get_device_error() == (0 if ix is idx else -6)
        kr, vr = (torch.full((N, H, D), 9.0, dtype=torch.bfloat16) for _ in range(2))
        kr[ix[keep].long()], vr[ix[keep].long()] = ref[keep], vf[keep]
        assert torch.equal(kd.cpu(), kr) and torch.equal(vd.cpu(), vr)


@pytest.mark.parametrize("bad", [False, True])
@pytest.mark.parametrize("N,C", [(200003, 16), (30001, 48), (50001, 64), (25000, 128), (30000, 256)])
def test_euler_and_statistic(hsa, N, C, bad):
    x, vh = synth.normal((N, C), 1), synth.normal((N, C), 2)
    idx = synth.uniform_subset(N, N // 2, 3)
    vfr = synth.normal((idx.numel(), C), 10)
    pos = torch.full((N,), -1, dtype=torch.int32)
    pos[idx.long()] = torch.arange(idx.numel(), dtype=torch.int32)
    given = pos.clone()
    if bad:
        pos[N - 2] = -1                                # a bad entry counts as none
        given[N - 2] = idx.numel()
    stat_ref = torch.full((N,), 0.25, dtype=torch.float64)
    want_x, want_v = x.clone(), vh.clone()
    oracle.l1rel_accumulate(vh.clone(), vfr, pos, 0.5, stat_ref)
    oracle.cached_euler_f32(want_x, want_v, vfr, pos, -0.025)
    fresh, at = vfr.to(DEV), given.to(DEV)
    for fused in (False, True):
        xd, vd = x.to(DEV), vh.to(DEV)
        if fused:
            stat = torch.full((N,), 0.25, device=DEV)
            hsa.hsa_cached_euler_l1rel(xd, vd, fresh, at, -0.025, stat, 0.5)
            assert torch.all((stat.cpu().double() - stat_ref).abs() <= 5e-5 * stat_ref.abs())
            assert bool((stat.cpu()[pos < 0] == 0.25).all())
        else:
            hsa.hsa_cached_euler(xd, vd, fresh, at, -0.025)
        assert hsa.hsa_get_device_error() == (-6 if bad else 0)
        assert torch.equal(xd.cpu(), want_x) and torch.equal(vd.cpu(), want_v)

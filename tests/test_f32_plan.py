"""The launch plan of fp32 attention, with no GPU: its clusters are never larger
than the device can hold resident (on a slice of a GPU a larger one would not
launch), and on a whole GPU the small layers split their keys."""
import pytest


@pytest.fixture(scope="module")
def hsa():
    from paper_2605_06892_gb300 import build as b
    b.build()
    import paper_2605_06892_gb300 as m
    m.lib()
    return m


SHAPES = [(n, N, H) for n in (1, 31, 256, 640, 3072, 40000)
          for N in (1, 127, 129, 1024, 6144, 40000) for H in (1, 4, 32)]


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("sms", [4, 19, 152])
@pytest.mark.parametrize("most", [1, 2, 4, 8])
def test_clusters_fit_the_device(hsa, D, sms, most):
    for n, N, H in SHAPES:
        for wide, deep in ((most, most), (1, most), (most, 1)):
            p = hsa.hsa_test_f32_cluster(n, N, H, D, sms, wide, deep)
            splits = p % 256
            assert splits in (1, 2, 4, 8)
            assert splits <= (deep if p >= 256 else wide), (n, N, H, wide, deep)
            assert splits == 1 or splits <= (N + 31) // 32     # no CTA without keys


def test_small_layers_split_their_keys(hsa):
    """256 queries x 4 heads leave 152 SMs idle without a split."""
    for D in (64, 128):
        assert hsa.hsa_test_f32_cluster(256, 1024, 4, D, 152, 8, 8) % 256 > 1
        assert hsa.hsa_test_f32_cluster(256, 1024, 4, D, 152, 1, 1) % 256 == 1


def test_refused_sizes(hsa):
    with pytest.raises(hsa.HsaError):
        hsa.hsa_test_f32_cluster(1, 1, 1, 96, 152, 8, 8)

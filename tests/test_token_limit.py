"""Token counts up to the int32 limit of the interface, with no GPU: the partition's
workspace holds the two key and two token buffers of 4N bytes and a counter per
digit and tile of 4096 tokens, and grows with N, right up to 2^31 - 1."""
import pytest


@pytest.fixture(scope="module")
def hsa():
    from paper_2605_06892_gb300 import build as b
    b.build()
    import paper_2605_06892_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("back", [0, 1, 255, 4095, 4096, 400000])
def test_workspace_up_to_the_int32_limit(hsa, back):
    N = 2 ** 31 - 1 - back
    tiles = -(-N // 4096)
    need = 4 * ((4 * N + 255) // 256 * 256) + 256 * tiles * 4
    assert hsa.hsa_partition_workspace_bytes(N) == need

"""Gather and KV-sync scatter over the row lengths where the copy changes form.

A lane moves 1 to 12 vectors of 16 bytes per row, whole and ragged; few rows, and
more rows than lane groups in the grid, so that a group walks several rows.  Copies
are exact: every byte is compared, also of the rows that must stay as they were.
"""
import pytest
import torch

import paper_2605_06892_gb300 as hsa

pytestmark = pytest.mark.gpu

VECS = (1, 3, 16, 32, 33, 64, 65, 96, 97, 128, 129, 160, 161, 192, 193, 224, 225, 256, 257, 384)


@pytest.mark.parametrize("rows", (7, 3000, 90000))
@pytest.mark.parametrize("vecs", VECS)
def test_row_copies_move_every_byte(vecs, rows):
    if rows * vecs > 90000 * 160:
        rows = 90000 * 160 // vecs
    g = torch.Generator(device="cuda").manual_seed(vecs * 7 + rows)
    n = rows - rows // 3

    def ints(count):
        return torch.randint(-2 ** 31, 2 ** 31, (count, 4 * vecs), dtype=torch.int32,
                             device="cuda", generator=g)

    idx = torch.randperm(rows, device="cuda", generator=g)[:n].sort().values
    idx32 = idx.int()
    src, dst = ints(rows), ints(n)
    hsa.hsa_gather_active(src, idx32, n, dst)
    assert torch.equal(dst, src[idx])

    def rows_of(t):
        return t.view(torch.float32).view(t.shape[0], 1, 4 * vecs)

    k, v, kf, vf = ints(rows), ints(rows), ints(n), ints(n)
    want_k, want_v = k.clone(), v.clone()
    want_k[idx], want_v[idx] = kf, vf
    hsa.hsa_kv_sync_scatter(rows_of(k), rows_of(v), rows_of(kf), rows_of(vf), idx32, n)
    assert torch.equal(k, want_k) and torch.equal(v, want_v)
    assert hsa.hsa_get_device_error() == 0

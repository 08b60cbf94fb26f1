"""Squint at insert over factors, row widths, alignments and ring positions: integer results, equal to a plain torch mean."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _ref(frames, f):
    n, c, h, w = frames.shape
    s = frames.to(torch.int64).reshape(n, c, h // f, f, w // f, f).sum((3, 5))
    return ((s + f * f // 2) // (f * f)).to(torch.uint8)


# n, c, h, w, f: whole and ragged 16-byte rows, one output a row, odd factors, few rows and many, rows of 12 KB
# and rows that do not fit in shared memory (the last two)
@pytest.mark.parametrize("n,c,h,w,f", [(1, 1, 1, 1, 1), (5, 3, 128, 128, 4), (3, 3, 84, 84, 4), (2, 3, 36, 108, 4),
                                       (4, 3, 34, 46, 2), (7, 1, 17, 19, 1), (2, 2, 9, 15, 3), (3, 3, 10, 10, 5),
                                       (1, 1, 8, 8, 8), (400, 3, 16, 20, 4), (33, 3, 64, 64, 2), (1, 1, 8, 3072, 4),
                                       (2, 1, 8, 16000, 4), (1, 2, 2, 50001, 1)])
@pytest.mark.parametrize("off_src,off_ring", [(0, 0), (1, 2), (4, 1), (6, 3)])
def test_squint_store_bit_exact(n, c, h, w, f, off_src, off_ring):
    from paper_2602_21203_gb300 import ops
    g = torch.Generator().manual_seed(n + 3 * h + w + f)
    size = n * c * h * w
    buf = torch.randint(0, 256, (size + off_src,), dtype=torch.uint8, generator=g).cuda()
    frames = buf[off_src:].view(n, c, h, w)
    slots = n + 2
    per = c * (h // f) * (w // f)
    rbuf = torch.full((slots * per + off_ring + 5,), 99, dtype=torch.uint8, device="cuda")
    for slot0 in (0, slots - 1, slots + 3):
        rbuf.fill_(99)
        ring = rbuf[off_ring:off_ring + slots * per].view(slots, c, h // f, w // f)
        ops.squint_store(frames, ring, slot0, f)
        want = torch.full_like(ring, 99)
        want[(torch.arange(n, device="cuda") + slot0) % slots] = _ref(frames, f)
        assert torch.equal(ring, want)
        assert bool((rbuf[:off_ring] == 99).all()) and bool((rbuf[off_ring + slots * per:] == 99).all())


# rows just too short and just long enough for the staged kernel
@pytest.mark.parametrize("w,f", [(12, 2), (14, 2), (24, 4), (28, 4), (36, 6), (2, 2), (4, 4)])
def test_squint_store_short_rows(w, f):
    test_squint_store_bit_exact(37, 3, 5 * f, w, f, 3, 1)
    test_squint_store_bit_exact(37, 3, 5 * f, w, f, 0, 0)


# other factors on both sides of the share of a warp that a row has to fill
@pytest.mark.parametrize("ws,f", [(15, 3), (16, 3), (31, 3), (33, 3), (19, 5), (20, 6), (39, 7), (40, 7), (22, 8), (30, 10), (31, 10)])
def test_squint_store_share_of_a_warp(ws, f):
    test_squint_store_bit_exact(11, 3, 4 * f, ws * f, f, 5, 2)
    test_squint_store_bit_exact(11, 3, 4 * f, ws * f, f, 0, 0)

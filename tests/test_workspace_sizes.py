"""Workspace sizes of blocks: a workspace of the size answered for a full block takes
every shorter one (the last block of an acquisition), so the answer never falls as
the frame count grows."""

import random

import pytest

import paper_2407_20692_gb300 as cpi


def _regions(bits, ha, wa, hb, wb):
    stride = max(ha, hb) * (wa + wb)
    stride = stride if bits == 8 else (stride + 31) // 32 * 4
    return (cpi.cpi_frames(0x1000, bits, ha, wa, 0, 0, wa + wb, stride, 0),
            cpi.cpi_frames(0x1000, bits, hb, wb, wa, 0, wa + wb, stride, 0))


@pytest.mark.parametrize("bits,ha,wa,hb,wb,block,short", [
    (8, 39, 30, 25, 21, 8020, 7872), (1, 64, 64, 12, 23, 3277, 2841), (1, 44, 44, 16, 30, 6538, 5960),
    (1, 32, 32, 16, 16, 10240, 9216), (1, 51, 42, 14, 22, 6179, 5929)])
def test_a_full_blocks_workspace_takes_this_shorter_block(bits, ha, wa, hb, wb, block, short):
    a, b = _regions(bits, ha, wa, hb, wb)
    assert cpi.cpi_correlate_workspace_size(a, b, short) <= cpi.cpi_correlate_workspace_size(a, b, block)
    assert cpi.cpi_acq_workspace_size(a, b, short) <= cpi.cpi_acq_workspace_size(a, b, block)


def test_sizes_grow_with_the_frame_count():
    rng = random.Random(7)
    for _ in range(400):
        bits = rng.choice([1, 8])
        a, b = _regions(bits, *(int(2 ** rng.uniform(2, 7)) for _ in range(4)))
        ns = sorted({int(2 ** rng.uniform(4, 17)) for _ in range(60)})
        sizes = [cpi.cpi_correlate_workspace_size(a, b, n) for n in ns]
        assert sizes == sorted(sizes), (bits, a.height, a.width, b.height, b.width)

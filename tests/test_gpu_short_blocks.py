"""Blocks shorter than the one a workspace was sized for: an acquisition's last block
and an accumulating call, at sizes where the shorter block is planned in more frame
chunks than the full one.  Sums against exact integer products."""

import numpy as np
import pytest
import torch

import paper_2407_20692_gb300 as cpi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


@pytest.mark.parametrize("bits,ha,wa,hb,wb,block,short", [
    (8, 39, 30, 25, 21, 8020, 7872), (1, 64, 64, 12, 23, 3277, 2841), (1, 44, 44, 16, 30, 6538, 5960),
    (1, 32, 32, 16, 16, 10240, 9216)])
def test_last_block_in_the_full_blocks_workspace(bits, ha, wa, hb, wb, block, short):
    rng = np.random.default_rng(block)
    n, rows, cols = block + short, max(ha, hb), wa + wb
    img = rng.integers(0, 2 if bits == 1 else 7, (n, rows, cols), dtype=np.uint8)
    data = img.reshape(n, -1)
    if bits == 1:
        data = np.packbits(np.pad(data, ((0, 0), (0, -data.shape[1] % 32))), axis=1, bitorder="little")
    stride = data.shape[1]
    host = torch.from_numpy(data).pin_memory()
    frames = host.cuda()
    regions = lambda t: (cpi.frames(t, bits, ha, wa, 0, 0, cols, stride), cpi.frames(t, bits, hb, wb, wa, 0, cols, stride))
    va, vb = (torch.from_numpy(v.reshape(n, -1)).cuda().double() for v in (img[:, :ha, :wa], img[:, :hb, wa:]))
    want = (va.T @ vb).long(), va.sum(0).long(), vb.sum(0).long()
    sums = lambda: [torch.zeros(s, dtype=torch.int64, device="cuda") for s in ((ha * wa, hb * wb), ha * wa, hb * wb)]
    a, b = regions(frames)

    got = sums()
    h = cpi.cpi_acq_begin(a, b, block, *got, torch.empty(cpi.cpi_acq_workspace_size(a, b, block), dtype=torch.uint8,
                                                        device="cuda"))
    cpi.cpi_acq_push(h, host[:block], block)
    cpi.cpi_acq_push(h, host[block:], short)
    cpi.cpi_acq_end(h)
    assert cpi.cpi_device_status() == 0
    assert all(torch.equal(x, y) for x, y in zip(got, want))

    got = sums()
    ws = torch.empty(cpi.cpi_correlate_workspace_size(a, b, block), dtype=torch.uint8, device="cuda")
    for t, k in ((frames[:block], block), (frames[block:], short)):
        cpi.cpi_correlate_accumulate(*regions(t), k, *got, ws)
    torch.cuda.synchronize()
    assert cpi.cpi_device_status() == 0
    assert all(torch.equal(x, y) for x, y in zip(got, want))

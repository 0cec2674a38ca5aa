"""Raw moments on the tile shapes a single correlation's plan chooses between: 256
columns, or 128 where they fill the last wave better; ragged tiles, K blocks and
frame chunks of both operand kinds.  Sums against exact products (float32 sums of
binary products below 2^24, float64 for counts)."""

import numpy as np
import pytest
import torch

import paper_2407_20692_gb300 as cpi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


@pytest.mark.parametrize("bits,ha,wa,hb,wb,n", [
    (8, 100, 100, 16, 17, 300),      # 158 wide tiles or 237 narrow ones on 152 SMs: narrow
    (1, 100, 100, 16, 17, 700),
    (1, 33, 64, 30, 40, 2500),       # 17 tile rows, 10 K blocks
    (1, 64, 64, 32, 32, 5000),       # whole tiles, 20 K blocks
    (1, 3, 43, 64, 300, 2400),       # 2 tile rows, the second with one pixel, many columns
    (1, 1, 100, 160, 160, 2400),     # a single tile row
    (1, 64, 64, 40, 40, 70000),      # two frame chunks
])
def test_sums_on_every_tile_shape(bits, ha, wa, hb, wb, n):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(ha * 1000 + wb)
    rows, cols = max(ha, hb), (wa + wb + 31) // 32 * 32
    img = torch.zeros((n, rows, cols), dtype=torch.uint8, device="cuda")
    va = torch.randint(0, 2 if bits == 1 else 7, (n, ha * wa), generator=gen, device="cuda", dtype=torch.uint8)
    vb = torch.randint(0, 2 if bits == 1 else 7, (n, hb * wb), generator=gen, device="cuda", dtype=torch.uint8)
    img[:, :ha, :wa] = va.view(n, ha, wa)
    img[:, :hb, wa:wa + wb] = vb.view(n, hb, wb)
    stride = rows * cols
    if bits == 1:
        stride //= 8
        w = torch.tensor([1, 2, 4, 8, 16, 32, 64, 128], dtype=torch.uint8, device="cuda")
        img = torch.cat([(img[i:i + 512].view(-1, stride, 8) * w).sum(-1, dtype=torch.uint8) for i in range(0, n, 512)])
    lay = dict(row_stride=cols, frame_stride_bytes=stride)
    a, b = cpi.frames(img, bits, ha, wa, x0=0, **lay), cpi.frames(img, bits, hb, wb, x0=wa, **lay)
    ma, mb = ha * wa, hb * wb
    ws = torch.full((cpi.cpi_correlate_workspace_size(a, b, n),), 255, dtype=torch.uint8, device="cuda")
    s_ab = torch.empty((ma, mb), dtype=torch.int64, device="cuda")
    s_a, s_b = (torch.empty(m, dtype=torch.int64, device="cuda") for m in (ma, mb))
    cpi.cpi_correlate(a, b, n, s_ab, s_a, s_b, torch.empty((ma, mb), dtype=torch.float64, device="cuda"), None, ws)
    torch.cuda.synchronize()
    assert cpi.cpi_device_status() == 0
    dt = torch.float32 if bits == 1 else torch.float64
    want = torch.zeros((ma, mb), dtype=torch.float64, device="cuda")
    for i in range(0, n, 16384):
        want += (va[i:i + 16384].to(dt).T @ vb[i:i + 16384].to(dt)).double()
    assert torch.equal(s_ab.double(), want)
    assert np.array_equal(s_a.cpu().numpy(), va.sum(0, dtype=torch.int64).cpu().numpy())
    assert np.array_equal(s_b.cpu().numpy(), vb.sum(0, dtype=torch.int64).cpu().numpy())

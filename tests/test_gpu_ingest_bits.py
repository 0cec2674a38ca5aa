"""Binary frames whose regions start at any bit and whose rows are no whole number
of words: the word path writes the partial 32-pixel tile at a row's end.  Sums and
marginals against exact integer products of the same values."""

import numpy as np
import pytest
import torch

import paper_2407_20692_gb300 as cpi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


def _check(data, bits, a, b, va, vb, n):
    ra, rb = cpi.frames(data, bits, **a), cpi.frames(data, bits, **b)
    ma, mb = va.shape[1], vb.shape[1]
    ws = torch.full((cpi.cpi_correlate_workspace_size(ra, rb, n),), 255, dtype=torch.uint8, device="cuda")
    s_ab = torch.empty((ma, mb), dtype=torch.int64, device="cuda")
    s_a, s_b = (torch.empty(m, dtype=torch.int64, device="cuda") for m in (ma, mb))
    cpi.cpi_correlate(ra, rb, n, s_ab, s_a, s_b, torch.empty((ma, mb), dtype=torch.float64, device="cuda"), None, ws)
    torch.cuda.synchronize()
    assert cpi.cpi_device_status() == 0
    assert np.array_equal(s_ab.cpu().numpy(), va.T.astype(np.int64) @ vb.astype(np.int64))
    assert np.array_equal(s_a.cpu().numpy(), va.sum(0, dtype=np.int64))
    assert np.array_equal(s_b.cpu().numpy(), vb.sum(0, dtype=np.int64))


@pytest.mark.parametrize("ha,wa,hb,wb,x0,n,order", [
    (6, 8, 5, 33, 0, 300, 0), (9, 37, 4, 31, 5, 257, 1), (2, 100, 13, 9, 7, 129, 0), (70, 65, 3, 32, 0, 513, 1),
    (5, 7, 5, 40, 0, 200, 0)])        # the last: rows under 8 pixels take the bit-wise path
def test_binary_regions_at_any_bit(ha, wa, hb, wb, x0, n, order):
    rng = np.random.default_rng(wa * 100 + wb)
    rows, cols = max(ha, hb), x0 + wa + wb + 3
    stride = (rows * cols + 31) // 32 * 4
    img = rng.integers(0, 2, (n, rows, cols), dtype=np.uint8)
    flat = np.zeros((n, stride * 8), dtype=np.uint8)
    flat[:, :rows * cols] = img.reshape(n, -1)
    packed = np.packbits(flat, axis=1, bitorder="little" if order == 0 else "big")
    data = torch.from_numpy(packed).cuda()
    lay = dict(row_stride=cols, frame_stride_bytes=stride, bit_order=order)
    _check(data, 1, dict(height=ha, width=wa, x0=x0, **lay), dict(height=hb, width=wb, x0=x0 + wa, **lay),
           img[:, :ha, x0:x0 + wa].reshape(n, -1), img[:, :hb, x0 + wa:x0 + wa + wb].reshape(n, -1), n)

"""Binary regions in wide frames, the last frame stored without what follows its last
pixel: sums and marginals equal exact integer products."""

import numpy as np
import pytest
import torch

import paper_2407_20692_gb300 as cpi
from test_gpu_ingest_bits import _check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


@pytest.mark.parametrize("ha,wa,hb,wb,x0,gap,tail,n,order", [
    (5, 8, 5, 9, 3, 200, 0, 300, 0),         # rows 7 words apart
    (4, 33, 3, 31, 40, 900, 50, 129, 1),     # padding behind the region
    (7, 40, 6, 64, 0, 0, 9, 260, 0),
    (3, 30, 9, 61, 1, 450, 3, 128, 1),
    (3, 30, 9, 61, 1, 5000, 3, 128, 1)])     # rows so far apart that the bit-wise path takes them
def test_region_at_the_end_of_the_buffer(ha, wa, hb, wb, x0, gap, tail, n, order):
    rng = np.random.default_rng(wa * 100 + wb)
    rows, cols = max(ha, hb), x0 + wa + gap + wb
    last = (max((ha - 1) * cols + x0 + wa, (hb - 1) * cols + cols) - 1) // 8      # byte of the last pixel
    stride = (last + 1 + tail + 3) // 4 * 4
    img = rng.integers(0, 2, (n, rows, cols), dtype=np.uint8)
    flat = rng.integers(0, 2, (n, max(stride * 8, rows * cols)), dtype=np.uint8)
    flat[:, :rows * cols] = img.reshape(n, -1)
    packed = np.packbits(flat[:, :stride * 8], axis=1, bitorder="little" if order == 0 else "big")
    data = torch.from_numpy(packed.reshape(-1)[:(n - 1) * stride + last + 1].copy()).cuda()
    lay = dict(row_stride=cols, frame_stride_bytes=stride, bit_order=order)
    _check(data, 1, dict(height=ha, width=wa, x0=x0, **lay), dict(height=hb, width=wb, x0=x0 + wa + gap, **lay),
           img[:, :ha, x0:x0 + wa].reshape(n, -1), img[:, :hb, x0 + wa + gap:].reshape(n, -1), n)

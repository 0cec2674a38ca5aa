"""The denoiser's output may lie on its input, wholly or in part: the results are those
of separate buffers, bit for bit.  Widths of the tensor-core layers, of the FP32 ones
and of the direct convolutions."""

import numpy as np
import pytest
import torch

import paper_2407_20692_gb300 as cpi
from test_gpu_denoise import _dev, _gamma, _model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


@pytest.mark.parametrize("hb,wb,ha,wa", [(9, 7, 40, 64), (6, 8, 33, 41), (2, 2, 2, 2)])
@pytest.mark.parametrize("shift", [0, 1, -1, 37])
def test_output_on_the_input(hb, wb, ha, wa, shift):
    n = hb * wb * ha * wa
    model = _dev(_model(71))
    g = _dev(_gamma(72, hb, wb, ha, wa)).view(-1)
    ws = torch.empty(cpi.cpi_denoise_workspace_size(ha, wa, hb, wb), dtype=torch.uint8, device="cuda")
    want = torch.empty_like(g)
    cpi.cpi_denoise(model, g, want, ha, wa, hb, wb, ws)
    buf = torch.zeros(n + 128, dtype=torch.float32, device="cuda")
    src, dst = buf[64:64 + n], buf[64 + shift:64 + shift + n]
    src.copy_(g)
    cpi.cpi_denoise(model, src, dst, ha, wa, hb, wb, ws)
    torch.cuda.synchronize()
    assert cpi.cpi_device_status() == 0
    assert np.array_equal(dst.cpu().numpy().view(np.uint32), want.cpu().numpy().view(np.uint32))

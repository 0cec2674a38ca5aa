"""The denoiser on images of any width: one padded line of pixels in units of 128
to 1024 (csrc/denoise_line.cu).  Shapes at its edges: odd widths, rows longer
than a unit (three separate bands are staged), a line that ends inside a unit,
one angular pixel, and images too small for the line's buffers (direct
convolutions).  The comparisons and their tolerances are test_gpu_denoise.py's."""

import numpy as np
import pytest
import torch

import paper_2407_20692_gb300 as cpi
from oracle import denoiser as dn
from test_gpu_denoise import _dev, _gamma, _model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


@pytest.mark.parametrize("hb,wb,ha,wa", [(4, 4, 17, 83), (3, 3, 9, 250), (2, 2, 5, 700), (6, 5, 24, 41), (1, 1, 63, 127),
                                         (2, 2, 2, 2), (5, 7, 31, 16), (8, 8, 40, 129), (2, 1, 3, 1100)])
def test_denoise_any_width_matches_oracle(hb, wb, ha, wa):
    blob = _model(31)
    g = _gamma(32 + wa, hb, wb, ha, wa)
    ws = torch.full((cpi.cpi_denoise_workspace_size(ha, wa, hb, wb),), 255, dtype=torch.uint8, device="cuda")
    out = torch.empty_like(_dev(g))
    cpi.cpi_denoise(_dev(blob), _dev(g), out, ha, wa, hb, wb, ws)
    torch.cuda.synchronize()
    assert cpi.cpi_device_status() == 0
    want = dn.denoise(blob, g.reshape(-1, ha, wa), hb, wb).reshape(hb * wb, -1)
    s = dn.scale_of(g)
    d = np.abs(out.cpu().numpy() - want) * s
    ymax = np.abs(want).max() * s
    assert d.max() <= 2e-3 * ymax, d.max() / ymax
    assert d.mean() <= 2e-5 * ymax, d.mean() / ymax


def _grad(blob, g, t, hb, wb, ha, wa):
    """Loss and gradient from a workspace full of NaN: nothing may be read that the call has not written."""
    ws = torch.full((cpi.cpi_denoise_workspace_size(ha, wa, hb, wb, training=True),), 255, dtype=torch.uint8,
                    device="cuda")
    grad = torch.empty(cpi.DENOISER_PARAMS, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    cpi.cpi_denoise_grad(_dev(blob), _dev(g), _dev(t), ha, wa, hb, wb, grad, loss, ws)
    torch.cuda.synchronize()
    assert cpi.cpi_device_status() == 0
    return grad.cpu().numpy(), float(loss.item())


@pytest.mark.parametrize("hb,wb,ha,wa", [(4, 4, 17, 83), (2, 2, 6, 300), (3, 5, 31, 40), (2, 3, 70, 64), (3, 2, 33, 128),
                                         (2, 2, 2, 2), (2, 2, 8, 40), (16, 16, 40, 37), (1, 2, 5, 700)])
def test_denoise_gradient_any_width_matches_oracle(hb, wb, ha, wa):
    blob = _model(41)
    g = _gamma(42 + wa, hb, wb, ha, wa)
    t = _gamma(43 + wa, hb, wb, ha, wa) * 0.5 + g * 0.5
    got, loss = _grad(blob, g, t, hb, wb, ha, wa)
    want_loss, want = dn.loss_and_grad(blob, g.reshape(-1, ha, wa), t.reshape(-1, ha, wa), hb, wb)
    assert abs(loss - want_loss) <= 1e-4 * want_loss
    o = 0
    for ci, co in dn.LAYERS:
        n = co * ci * 9 + co
        gl, wl = got[o:o + n], want[o:o + n]
        assert np.abs(gl - wl).max() <= 2e-3 * np.abs(wl).max(), (ci, co, np.abs(gl - wl).max() / np.abs(wl).max())
        o += n
    again, loss2 = _grad(blob, g, t, hb, wb, ha, wa)
    assert np.array_equal(got.view(np.uint32), again.view(np.uint32)) and loss2 == loss

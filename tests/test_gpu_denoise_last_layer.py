"""Weight gradients of the denoiser's last layer against 64 bits, where truncated
tensor-core sums would show: hidden activations that are exact (the network passes
relu(x) and relu(-x) on), output gradients of one sign, so that
    dW[c][tap] = sum over pixels of dy(pixel) a3[c](neighbour)
has terms of one sign, known from the inputs.

Tolerance 2e-7: what remains are about 30 rounded FP32 additions of the runs' sums per
CTA and as many over the CTAs, an rms of 6e-8, times three.  (Runs of 256 pixels
instead of 64: 3.1e-7 at 32x32 vs 16x16; FP32 throughout: 4.8e-7.)"""

import numpy as np
import pytest
import torch

import paper_2407_20692_gb300 as cpi
from oracle import denoiser as dn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


def _relative_errors(hb, wb, ha, wa):
    rng = np.random.default_rng(ha * 100 + wa)
    g = (0.01 * rng.standard_normal((hb * wb, ha * wa))).astype(np.float32)
    t = (-0.05 - 0.01 * rng.random(g.shape)).astype(np.float32)
    blob = np.zeros(cpi.DENOISER_PARAMS, dtype=np.float32)
    at = [sum(co * ci * 9 + co for ci, co in dn.LAYERS[:k]) for k in range(5)]
    blob[at[0]:at[0] + 32 * 81].reshape(32, 9, 3, 3)[:, 4, 1, 1] = np.where(np.arange(32) % 2 == 0, 1.0, -1.0)
    for k in (1, 2):
        blob[at[k]:at[k] + 32 * 288].reshape(32, 32, 3, 3)[np.arange(32), np.arange(32), 1, 1] = 1.0
    dev = lambda a: torch.tensor(a, device="cuda")
    ws = torch.empty(cpi.cpi_denoise_workspace_size(ha, wa, hb, wb, training=True), dtype=torch.uint8, device="cuda")
    grad = torch.empty(cpi.DENOISER_PARAMS, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    cpi.cpi_denoise_grad(dev(blob), dev(g), dev(t), ha, wa, hb, wb, grad, loss, ws)
    torch.cuda.synchronize()
    assert cpi.cpi_device_status() == 0
    s = dn.scale_of(g)
    x = (dev(g) * torch.tensor(s, dtype=torch.float32, device="cuda")).to(torch.bfloat16).double().view(hb * wb, ha, wa)
    dy = (x - dev(t).double().view_as(x) * s) * 2.0 / g.size           # the last layer's weights are 0: y = x
    want = torch.empty((2, 3, 3), dtype=torch.float64)
    for i, a3 in enumerate((x.clamp(min=0), (-x).clamp(min=0))):
        p = torch.nn.functional.pad(a3, (1, 1, 1, 1))
        for ky in range(3):
            for kx in range(3):
                want[i, ky, kx] = (dy * p[:, ky:ky + ha, kx:kx + wa]).sum()
    want = want.repeat(16, 1, 1)
    got = grad[at[3]:at[3] + 288].view(32, 3, 3).cpu().double()
    return (got - want) / want


@pytest.mark.parametrize("hb,wb,ha,wa", [(16, 16, 32, 32), (12, 11, 30, 128), (13, 16, 29, 41), (16, 16, 60, 33)])
def test_sums_of_one_sign_are_not_biased(hb, wb, ha, wa):
    assert _relative_errors(hb, wb, ha, wa).abs().max().item() <= 2e-7


def test_bias_at_64_wide_is_no_larger_than_that_of_the_images_own_pixels():
    """Images 64 wide sum a CTA's pixels in tensor-core accumulators to the end: 8.09e-6
    low at this size in one accumulator over the pixels of the images, 8.20e-6 with the
    zero column of the padded line summed too."""
    assert _relative_errors(12, 16, 60, 64).mean().abs().item() <= 8.1e-6

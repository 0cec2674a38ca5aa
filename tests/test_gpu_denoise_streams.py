"""Denoiser calls on several streams at once, each with its own workspace: lines short
enough that kernels of different streams share SMs and their tensor memory.  Every
call's result is the one it has alone, bit for bit."""

import numpy as np
import pytest
import torch

import paper_2407_20692_gb300 as cpi
from test_gpu_denoise import _dev, _gamma, _model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


def test_calls_on_three_streams_equal_calls_alone():
    shapes = [(32, 32, 8, 9), (24, 64, 6, 8), (42, 64, 12, 9)]
    calls = []
    for k, (ha, wa, hb, wb) in enumerate(shapes):
        g = _gamma(50 + k, hb, wb, ha, wa)
        c = dict(shape=(ha, wa, hb, wb), model=_dev(_model(60 + k)), g=_dev(g), t=_dev(0.5 * g))
        for name, train in (("ws", False), ("wst", True)):
            c[name] = torch.empty(cpi.cpi_denoise_workspace_size(ha, wa, hb, wb, training=train), dtype=torch.uint8,
                                  device="cuda")
        calls.append(c)

    def run(c, stream):
        out = torch.empty_like(c["g"])
        grad = torch.empty(cpi.DENOISER_PARAMS, dtype=torch.float32, device="cuda")
        loss = torch.empty(1, dtype=torch.float32, device="cuda")
        stream.wait_stream(torch.cuda.default_stream())
        cpi.cpi_denoise(c["model"], c["g"], out, *c["shape"], c["ws"], stream)
        cpi.cpi_denoise_grad(c["model"], c["g"], c["t"], *c["shape"], grad, loss, c["wst"], stream)
        return out, grad, loss

    streams = [torch.cuda.Stream() for _ in calls]
    alone = []
    for c in calls:
        alone.append(run(c, streams[0]))
        torch.cuda.synchronize()
    for _ in range(10):
        got = [run(c, s) for c, s in zip(calls, streams)]
        torch.cuda.synchronize()
        assert cpi.cpi_device_status() == 0
        for x, y in zip(got, alone):
            for u, v in zip(x, y):
                assert np.array_equal(u.cpu().numpy().view(np.uint32), v.cpu().numpy().view(np.uint32))

"""The x stage on interleaved rows (calls of enough planes for a copy of Gamma in
their workspace) against the row-major one (fewer planes): the same planes must
come out bit for bit.  Shapes at the edges of its plan: rows short of a group of
four, one to many row sets, CTAs of one to sixteen warps, several CTAs per SM, a
ragged last band, an odd number of angular columns, stacks of several launches."""

import numpy as np
import pytest
import torch

from gpu_util import refocus_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


@pytest.mark.parametrize("ha,wa,hb,wb,n", [
    (64, 64, 3, 24, 64), (33, 36, 2, 9, 40), (7, 8, 3, 12, 33), (61, 32, 2, 25, 150), (130, 128, 2, 16, 48),
    (45, 100, 1, 11, 129), (9, 260, 2, 20, 61), (18, 512, 1, 17, 40), (1, 4, 2, 9, 60), (96, 96, 2, 31, 300)])
def test_interleaved_rows_equal_row_major(ha, wa, hb, wb, n):
    rng = np.random.default_rng(ha * 1000 + wa)
    g32 = torch.tensor(rng.standard_normal((hb * wb, ha * wa)).astype(np.float32), device="cuda")
    alpha = np.concatenate([rng.uniform(0.4, 1.6, n - 2), [40.0, -1.0]])     # taps far outside and mirrored too
    beta = np.concatenate([rng.uniform(-0.6, 0.6, n - 2), [-30.0, 2.0]])
    full = refocus_gpu(g32, ha, wa, hb, wb, alpha, beta)
    for p in {0, 1, 3, n // 2, n - 3, n - 2, n - 1}:
        one = refocus_gpu(g32, ha, wa, hb, wb, alpha[p:p + 1], beta[p:p + 1])   # 1 plane: no room for the copy
        assert np.array_equal(full[p], one[0]), p

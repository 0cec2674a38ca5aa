"""The x stage on interleaved rows against the row-major one: a stack large enough for
it, and the same planes one by one, which take the row-major form, must come out bit
for bit.  Which form ran is read from the workspace, where the interleaved one leaves
its copy of Gamma ([slice][4 rows][column, 2 zero columns on either side][row]).
Shapes at the edges of its plan: rows short of a group of four, one to several row
sets, CTAs of one to sixteen warps, a ragged last band, one and odd numbers of angular
columns, stacks of several launches, planes short of a block of four."""

import numpy as np
import pytest
import torch

import paper_2407_20692_gb300 as cpi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _ready(cuda_ready):
    yield


def _interleaved(g, ha, wa):
    s, groups = g.shape[0], (ha + 3) // 4
    x = torch.zeros((s, groups * 4, wa + 4), dtype=torch.float32, device="cuda")
    x[:, :ha, 2:wa + 2] = g.view(s, ha, wa)
    return x.view(s, groups, 4, wa + 4).transpose(2, 3).contiguous().view(-1)


def _run(g, copy, ha, wa, hb, wb, alpha, beta):
    """The stack, and whether the interleaved form ran."""
    ws = torch.full((cpi.cpi_refocus_workspace_size(ha, wa, hb, wb, len(alpha)),), 255, dtype=torch.uint8, device="cuda")
    out = torch.empty((len(alpha), ha, wa), dtype=torch.float32, device="cuda")
    cpi.cpi_refocus(g, ha, wa, hb, wb, cpi.plane_array(alpha, beta), out, ws)
    torch.cuda.synchronize()
    assert cpi.cpi_device_status() == 0
    left = ws[:ws.numel() // 4 * 4].view(torch.float32)
    for chunk in range(1, 129):      # planes per launch, whose images come first
        at = (chunk * hb * ha * wa + 63) // 64 * 64
        if at + copy.numel() <= left.numel() and torch.equal(left[at:at + copy.numel()], copy):
            return out, True
    return out, False


@pytest.mark.parametrize("ha,wa,hb,wb,n", [
    (83, 83, 37, 37, 128), (61, 32, 40, 25, 150), (130, 128, 12, 16, 128), (45, 100, 24, 11, 129), (9, 260, 20, 60, 119),
    (202, 512, 10, 2, 61), (96, 96, 20, 31, 300), (13, 7, 200, 5, 300), (37, 250, 30, 9, 95), (70, 50, 30, 29, 127),
    (3, 31, 400, 3, 103), (40, 40, 160, 1, 128)])
def test_interleaved_form_equals_row_major(ha, wa, hb, wb, n):
    rng = np.random.default_rng(ha * 1000 + wa)
    g = torch.tensor(rng.standard_normal((hb * wb, ha * wa)).astype(np.float32), device="cuda")
    copy = _interleaved(g, ha, wa)
    alpha = np.concatenate([rng.uniform(0.4, 1.6, n - 2), [40.0, -1.0]])     # taps far outside and mirrored too
    beta = np.concatenate([rng.uniform(-0.6, 0.6, n - 2), [-30.0, 2.0]])
    full, form = _run(g, copy, ha, wa, hb, wb, alpha, beta)
    assert form
    for p in {0, 1, 3, n // 2, n - 4, n - 3, n - 2, n - 1}:
        one, form = _run(g, copy, ha, wa, hb, wb, alpha[p:p + 1], beta[p:p + 1])
        assert not form
        assert torch.equal(full[p].view(torch.int32), one[0].view(torch.int32)), p


@pytest.mark.parametrize("ha,wa,hb,wb,n", [(26, 411, 40, 2, 24), (13, 442, 43, 24, 34), (57, 60, 63, 18, 42)])
def test_stacks_that_the_copy_splits_for_nothing(ha, wa, hb, wb, n):
    """The copy would split these stacks, and their y stages do not fill the GPU or the
    last waves of units weigh more."""
    g = torch.zeros((hb * wb, ha * wa), dtype=torch.float32, device="cuda")
    alpha = np.linspace(0.5, 1.5, n)
    assert not _run(g + 1.0, _interleaved(g + 1.0, ha, wa), ha, wa, hb, wb, alpha, 1.0 - alpha)[1]

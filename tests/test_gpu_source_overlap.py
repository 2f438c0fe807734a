"""The 5D source of a 4D source that lies in the output's own memory."""

import numpy as np
import pytest
import torch

from _util import make_pair, to_gpu, to_np
from paper_2602_14454_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_2602_14454_gb300 import build
    build.build()


# a slice that the source writes (first, last) or clears (1), and a field that starts inside one and ends in the next
@pytest.mark.parametrize("c", [0.0, 0.5])
@pytest.mark.parametrize("at", [0.0, 0.5, 1.0, 4.0])
def test_source_in_place(at, c):
    dims, Ls = (4, 4, 2, 6), 5
    op, _ = make_pair(dims, Ls, 1.8, 0.03, 1.0, c, "standard", 1.0, seed=3)
    b4 = to_gpu(inputs.gaussian_4d(dims, 6))
    want = to_np(op.source_5d(b4))
    b5 = torch.zeros(op.shape5(), dtype=torch.complex128, device="cuda")
    part = b5.view(-1)[int(at * b4.numel()):][:b4.numel()].view(b4.shape)
    part.copy_(b4)
    assert np.array_equal(to_np(op.source_5d(part, out=b5)), want)
    after = torch.zeros(2 * b5.numel(), dtype=torch.complex128, device="cuda")   # adjacent, not overlapping
    after[b5.numel():b5.numel() + b4.numel()] = b4.view(-1)
    out = op.source_5d(after[b5.numel():b5.numel() + b4.numel()].view(b4.shape), out=after[:b5.numel()].view(b5.shape))
    assert np.array_equal(to_np(out), want)

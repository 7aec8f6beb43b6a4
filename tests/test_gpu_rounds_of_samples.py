"""Samples of a query in rounds of 32: windows of one whole round, of one sample more, of two; against the CPU oracle."""
import pytest
import torch

import parity_util as pu
from test_gpu_parity import small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("window", [(1, 1, 17), (2, 4, 4), (1, 3, 11), (4, 4, 4)])     # 17, 32, 33, 64 samples
def test_rounds_of_samples(d, window):
    q, k, v, off, dout = small_problem(3, 7, 9, 2, d, window, torch.bfloat16, 1.3, 960 + d)
    off.view(-1)[5::101] = float("nan")          # dead samples
    off.view(-1)[7::89] = 1e9
    pu.full_parity(q, k, v, off, dout, window)

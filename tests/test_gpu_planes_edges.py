"""The plane-by-plane forwards on grids whose last tiles lie partly outside them (an instance of its own for 128 channels) and on grids of
whole tiles, with more tiles than the GPU has SMs; against the CPU oracle."""
import pytest
import torch

import oracle
import parity_util as pu
from paper_2607_22696_b200 import binding
from test_gpu_parity import small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("grid,heads", [((8, 12, 40), 6), ((5, 9, 41), 8), ((6, 11, 33), 8), ((1, 2, 9), 80), ((4, 13, 40), 8)])
@pytest.mark.parametrize("window", [(3, 3, 3), (3, 5, 5), (3, 7, 7)])
def test_tiles_at_the_edges(grid, heads, window, d):
    T, H, W = grid
    assert ((T + 3) // 4) * ((H + 3) // 4) * ((W + 7) // 8) * heads > 148
    bounded = window == (3, 3, 3)
    q, k, v, off, _ = small_problem(*grid, heads, d, window, torch.bfloat16, 0.4, 990 + d + T)
    off = off.clamp_(-0.999, 0.999) if bounded else torch.zeros_like(off)
    ref_out, ref_lse = oracle.forward(q, k, v, off, T, H, W, heads, d, window)
    out = torch.full(q.shape, float("nan"), dtype=q.dtype, device="cuda")
    lse = torch.full((T, H, W, heads), float("nan"), device="cuda")
    dev = [z.cuda() for z in (q, k, v, off)]
    if bounded:
        binding.dsa3d_forward_bounded_offsets(*dev, T, H, W, heads, d, window, out, lse)
    else:
        binding.dsa3d_forward_fixed_window(*dev[:3], T, H, W, heads, d, window, out, lse)
    torch.cuda.synchronize()
    assert binding.dsa3d_device_timeout_flag() == 0
    pu.assert_close("out", out, ref_out.view(q.shape), torch.bfloat16)
    pu.assert_close("lse", lse, ref_lse.view(T, H, W, heads), torch.bfloat16)

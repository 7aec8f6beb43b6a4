"""Keys whose logits overflow to minus infinity in fp32 (rows that a caller masks so): their weight is 0 wherever they lie in a window."""
import pytest
import torch

import oracle
import parity_util as pu
from paper_2607_22696_b200 import binding
from test_gpu_parity import small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("window", [(2, 2, 2), (3, 3, 3), (3, 5, 5), (3, 7, 7)])
def test_fixed_window_with_masked_keys(window, d):
    """One row of keys in three along t and along y stays (in two for the smallest window), so that every query has a key, or a dead sample
    with logit 0, and in the larger windows whole runs of kernel rows, as the threads of a query share them, are masked."""
    T, H, W, heads = 5, 11, 19, 2
    q, k, v, off, _ = small_problem(T, H, W, heads, d, window, torch.bfloat16, 1.0, 980 + d)
    every = min(3, window[0])
    masked = torch.ones(T, H, W, dtype=torch.bool)
    masked[1::every, 1::every] = False
    q[..., 0] = 8.0
    k[..., 0] = torch.where(masked[..., None], torch.tensor(-3e38), k[..., 0].float()).to(k.dtype)      # 8 * -3e38 is below fp32's range
    ref_out, ref_lse = oracle.forward(q.view(-1, heads, d), k, v, torch.zeros_like(off).view(T * H * W, heads, -1, 3), T, H, W, heads, d, window)
    out = torch.full(q.shape, float("nan"), dtype=q.dtype, device="cuda")
    lse = torch.full((T, H, W, heads), float("nan"), device="cuda")
    binding.dsa3d_forward_fixed_window(q.cuda(), k.cuda(), v.cuda(), T, H, W, heads, d, window, out, lse)
    torch.cuda.synchronize()
    assert bool(torch.isfinite(ref_lse).all())
    pu.assert_close("out", out, ref_out.view(q.shape), torch.bfloat16)
    pu.assert_close("lse", lse, ref_lse.view(T, H, W, heads), torch.bfloat16)

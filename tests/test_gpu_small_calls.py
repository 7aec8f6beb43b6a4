"""fp32 calls too small to fill the chip run with a CTA per item whose groups of lanes (8, 16 or 32) take the samples in turn: windows
with fewer samples than groups, as many, a few more, and many rounds; against the CPU oracle (tolerances of parity_util)."""
import pytest
import torch

import parity_util as pu
from test_gpu_parity import small_problem

pytestmark = pytest.mark.gpu
F32 = torch.float32


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("shape,window,kind", [
    ((1, 1, 1, 1), (1, 1, 2), "normal"),         # one item
    ((3, 4, 5, 2), (1, 2, 2), "normal"),         # 4 samples: one each for 128 channels, idle groups for the others
    ((2, 3, 5, 3), (1, 4, 4), "normal"),         # 16: one each for 32 channels
    ((3, 4, 6, 2), (3, 3, 3), "normal"),
    ((3, 4, 6, 2), (3, 3, 3), "int"),            # one corner has a weight, three more a derivative
    ((2, 4, 7, 1), (3, 7, 7), "normal"),
])
def test_fp32_items_split_over_a_cta(d, shape, window, kind):
    q, k, v, off, dout = small_problem(*shape, d, window, F32, 1.2, 900 + d + shape[2])
    if kind == "int":
        off = off.round()
    off.view(-1)[5::101] = float("nan")          # dead samples
    pu.full_parity(q, k, v, off, dout, window)


@pytest.mark.parametrize("heads", [1, 3])
@pytest.mark.parametrize("d", [32, 64, 128])
def test_fp32_items_on_both_sides_of_the_line(d, heads):
    """The last size that is split (148 * 16 lanes per head), and a column more, which is not: the same sums in other orders (1e-5 and
    1e-4 as against the oracle)."""
    window, W = (2, 2, 2), 37
    H = 148 * 16 * 4 // (d * W)
    assert H * W * (d // 4) == 148 * 16
    q, k, v, off, dout = (z.cuda() for z in small_problem(1, H, W + 1, heads, d, window, F32, 1.0, 920 + d))
    res = []
    for cut in ([z[:, :, :W].contiguous() for z in (q, k, v, off, dout)], (q, k, v, off, dout)):
        dims = tuple(cut[0].shape)
        out = pu.gpu_forward(*cut[:4], dims, window)
        res.append(tuple(out) + tuple(pu.gpu_backward(*cut[:4], out[1], cut[4], dims, window)))
    inner = W - 12                               # columns that no sample of which reaches the cut (offsets N(0, 1))
    for name, a, b, bound in zip(("out", "lse", "dq", "dk", "dv", "doffsets"), *res, (1e-5, 1e-5, 1e-4, 1e-4, 1e-4, 1e-4)):
        assert float((a[:, :, :inner] - b[:, :, :inner]).abs().max()) <= bound, name

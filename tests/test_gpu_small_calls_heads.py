"""fp32 calls of few tokens take other kernels the more heads they have: the bits of a head stay the same, and are right."""
import pytest
import torch

import parity_util as pu
from paper_2607_22696_b200 import binding
from test_gpu_parity import small_problem

pytestmark = pytest.mark.gpu
F32 = torch.float32


@pytest.mark.parametrize("d,grid", [(32, (4, 8, 8)), (64, (2, 8, 9)), (128, (2, 6, 6))])      # just below the line of the forward
@pytest.mark.parametrize("window", [(1, 1, 2), (2, 2, 2), (1, 3, 5), (1, 4, 4), (1, 1, 17), (3, 3, 3), (3, 7, 7)])
@pytest.mark.parametrize("kind", ["normal", "int", "mixed"])
def test_heads_of_a_small_call_keep_their_bits(d, grid, window, kind):
    heads = 25                                   # (the backward sorts a million samples and more, in sums of another order)
    q, k, v, off, dout = (z.cuda() for z in small_problem(*grid, heads, d, window, F32, 1.3, 1000 + d))
    if kind == "int":
        off = off.round()
    elif kind == "mixed":                        # items and single samples on the grid among others
        off[:, :, ::2] = off[:, :, ::2].round()
        off.view(-1, 3)[::3].round_()
    off.view(-1)[5::101] = float("nan")          # dead samples

    def run(lo, hi):
        dims = (*grid, hi - lo, d)
        cut = [z[:, :, :, lo:hi].contiguous() for z in (q, k, v, off, dout)]
        out, lse = pu.gpu_forward(*cut[:4], dims, window)
        return (out, lse, *pu.gpu_backward(*cut[:4], lse, cut[4], dims, window))

    whole = run(0, heads)
    for lo, hi in ((0, 1), (5, 9), (9, 23)):
        part = run(lo, hi)
        for name, a, b in zip(("out", "lse", "dq", "dk", "dv", "doffsets"), whole, part):
            a = a[:, :, :, lo:hi]
            if name in ("dk", "dv"):             # sums of atomics in any order
                assert float((a - b).abs().max()) <= pu.F32_BWD_ATOL, (name, lo, hi)
            else:
                assert torch.equal(a, b), (name, lo, hi)


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("window,kind", [((2, 2, 2), "normal"), ((1, 3, 5), "int"), ((3, 3, 3), "normal"), ((3, 3, 3), "int"), ((3, 7, 7), "normal")])
def test_small_calls_of_many_heads_against_the_oracle(d, window, kind):
    q, k, v, off, dout = small_problem(2, 4, 7, 48, d, window, F32, 1.2, 1010 + d)
    if kind == "int":
        off = off.round()
    off.view(-1)[5::101] = float("nan")
    pu.full_parity(q, k, v, off, dout, window)


@pytest.mark.parametrize("d,grid", [(32, (4, 8, 8)), (64, (2, 8, 9)), (128, (2, 6, 6))])
@pytest.mark.parametrize("heads", [1, 25])
def test_residual_of_small_calls(d, grid, heads):
    window, dims = (3, 3, 3), (*grid, heads, d)
    q, k, v, off, add = (z.cuda() for z in small_problem(*dims, window, F32, 1.3, 1020 + d))
    out, lse = pu.gpu_forward(q, k, v, off, dims, window)
    both, lse2 = torch.empty_like(out), torch.empty_like(lse)
    binding.dsa3d_forward_residual(q, k, v, off, add, *dims, window, both, lse2)
    assert torch.equal(both, out + add) and torch.equal(lse, lse2)      # one fp32 addition


@pytest.mark.parametrize("d,grid", [(32, (4, 8, 8)), (64, (2, 8, 9)), (128, (2, 6, 6))])
@pytest.mark.parametrize("heads", [1, 25])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_dead_samples_of_a_query_that_is_not_finite(d, grid, heads, bad):
    """A sample without a corner inside the grid has the logit 0 whatever q holds: a query with no others has out = 0, lse = ln P, also
    beside queries whose samples all lie on the grid."""
    window, dims = (3, 3, 3), (*grid, heads, d)
    q, k, v, off, _ = small_problem(*dims, window, F32, 1.3, 1030 + d)
    off = off.round()
    rows = torch.zeros(dims[:4], dtype=torch.bool)
    rows.view(-1)[::3] = True
    q[rows], off[rows] = bad, 1e6
    out, lse = pu.gpu_forward(*(z.cuda() for z in (q, k, v, off)), dims, window)
    out, lse = out.cpu(), lse.cpu()
    assert float(out[rows].abs().max()) == 0.0 and float((lse[rows] - torch.tensor(27.0).log()).abs().max()) <= 1e-6
    assert bool(torch.isfinite(out).all() and torch.isfinite(lse).all())

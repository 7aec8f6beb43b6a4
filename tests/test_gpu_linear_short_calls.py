"""Backward of the offsets' linear layer: short calls, whose dbias is the same from call to call, and more outputs than a grid has
blocks along y for."""
import pytest
import torch

from paper_2607_22696_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("O", [1296, 81, 5, 2052])          # whole vectors, odd rows, less than a strip, several strips and padding
@pytest.mark.parametrize("tokens", [1, 31, 65, 512, 1024, 1025, 2048])
def test_dbias_of_short_calls_is_repeatable(tokens, O):
    C = 64
    g = torch.Generator(device="cuda").manual_seed(tokens + O)
    u = torch.randn(tokens, C, generator=g, device="cuda").bfloat16()
    w = (torch.randn(O, C, generator=g, device="cuda") / 8).bfloat16()
    doff = torch.randn(tokens, O, generator=g, device="cuda")
    n = binding.dsa3d_offsets_linear_backward_workspace_bytes(tokens, C, O, torch.bfloat16)
    ws = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")
    ref_db, ref_du, ref_dw = doff.double().sum(0), doff.bfloat16().double() @ w.double(), doff.bfloat16().double().T @ u.double()
    first = None
    for _ in range(30):
        du, dw, db = torch.full_like(u, float("nan")), torch.full((O, C), float("nan"), device="cuda"), torch.full((O,), float("nan"), device="cuda")
        binding.dsa3d_offsets_linear_backward(u, w, doff, tokens, C, O, du, dw, db, ws)
        first = db if first is None else first
        assert torch.equal(db, first)
    # fp32 sums of `tokens` and O terms of products that are exact in fp32: a few rounding errors of their magnitudes
    assert float((db - ref_db).abs().max()) <= 1e-6 * tokens ** 0.5 * float(doff.abs().max()) + 1e-6
    assert float((dw - ref_dw).norm()) <= 1e-5 * float(ref_dw.norm())
    assert float((du.double() - ref_du).norm()) <= 2.0 ** -8 * float(ref_du.norm())


def test_du_of_more_outputs_than_blocks_of_64_fit_a_grid():
    tokens, C, O = 2, 8, 64 * 65535 + 8
    g = torch.Generator(device="cuda").manual_seed(7)
    w = torch.randn(O, C, generator=g, device="cuda").bfloat16()
    doff = torch.randn(tokens, O, generator=g, device="cuda")
    n = binding.dsa3d_offsets_linear_backward_workspace_bytes(tokens, C, O, torch.bfloat16)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    du = torch.full((tokens, C), float("nan"), dtype=torch.bfloat16, device="cuda")
    u = torch.zeros(tokens, C, dtype=torch.bfloat16, device="cuda")
    binding.dsa3d_offsets_linear_backward(u, w, doff, tokens, C, O, du, None, None, ws)
    torch.cuda.synchronize()
    assert binding.dsa3d_device_timeout_flag() == 0
    ref = doff.bfloat16().double() @ w.double()
    # one chain of 4.2 million fp32 additions beside the rounding to bf16
    assert float((du.double() - ref).norm()) <= 1e-2 * float(ref.norm())

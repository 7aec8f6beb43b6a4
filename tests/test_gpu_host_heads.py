"""dsa3d_step_host by groups of heads: group sizes, a last group that is smaller, the fall back to slabs of frames."""
import pytest
import torch

import parity_util as pu
from paper_2607_22696_b200 import binding
from test_gpu_parity import small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,dims", [
    (torch.bfloat16, (3, 45, 80, 5, 128)),       # four heads of 256 bytes make a group: too few, slabs of frames
    (torch.bfloat16, (3, 45, 80, 7, 128)),       # groups of two, the last of one
    (torch.bfloat16, (3, 30, 52, 16, 64)),       # groups of four
    (torch.bfloat16, (2, 30, 52, 17, 128)),      # five groups, the last of one
    (torch.float32, (2, 30, 52, 11, 64)),        # 0.93 million samples: by rows, as its groups
    (torch.float32, (3, 30, 52, 9, 64)),         # 1.1 million: the whole by sorted samples, its groups by rows
])
def test_host_step_by_groups_of_heads(dtype, dims):
    """dsa3d_step_host copies groups of heads out of and into host tensors (from 8 MB a tensor on); the device entry points on the whole."""
    window = (3, 3, 3)
    T, H, W, heads, d = dims
    host = [z.pin_memory() for z in small_problem(*dims, window, dtype, 1.0, 940 + heads)]
    assert host[0].numel() * host[0].element_size() >= 8 << 20
    q, off = host[0], host[3]
    res = [torch.empty_like(q, pin_memory=True), torch.empty(dims[:4], pin_memory=True), *(torch.empty_like(q, pin_memory=True) for _ in range(3)),
           torch.empty_like(off, pin_memory=True)]
    nbytes = binding.dsa3d_step_host_arena_bytes(*dims, window, dtype)
    arena = torch.full((nbytes + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    for _ in range(2):                           # the second call over what the first one left
        for z in res:
            z.fill_(float("nan"))
        binding.dsa3d_step_host(*host, *dims, window, *res, arena[:nbytes])
        torch.cuda.synchronize()
    assert bool((arena[nbytes:] == 0xA5).all())
    dev = [z.cuda() for z in host]
    want = pu.gpu_forward(*dev[:4], dims, window)
    want += tuple(pu.gpu_backward(*dev[:4], want[1], dev[4], dims, window))
    for i, (name, a, b) in enumerate(zip(("out", "lse", "dq", "dk", "dv", "doffsets"), res, want)):
        if i < 2 or (i in (2, 5) and (dtype == torch.bfloat16 or T * H * W * heads * 27 < 10 ** 6)):
            assert torch.equal(a, b.cpu()), name         # the same sums in the same order
        else:
            pu.assert_close(name, a, b.cpu(), dtype, backward=True)

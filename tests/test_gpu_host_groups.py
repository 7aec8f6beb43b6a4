"""dsa3d_step_host by groups of heads beside pipelined steps on the same arena, from memory that is not all page-locked, and with offsets
too narrow for strided uploads; against the device entry points."""
import pytest
import torch

import parity_util as pu
from paper_2607_22696_b200 import binding
from test_gpu_parity import small_problem

pytestmark = pytest.mark.gpu
BF16, F32 = torch.bfloat16, torch.float32
NAMES = ("out", "lse", "dq", "dk", "dv", "doffsets")


def _results(host, pin=True):
    q, off = host[0], host[3]
    lse = torch.empty(q.shape[:4], pin_memory=pin)
    return [z.fill_(float("nan")) for z in (torch.empty_like(q, pin_memory=pin), lse, *(torch.empty_like(q, pin_memory=pin) for _ in range(3)),
                                            torch.empty_like(off, pin_memory=pin))]


def _check(host, res, dims, window, what, bits=True):
    dev = [z.cuda() for z in host]
    want = pu.gpu_forward(*dev[:4], dims, window)
    want += tuple(pu.gpu_backward(*dev[:4], want[1], dev[4], dims, window))
    for name, a, b in zip(NAMES, res, want):
        if name in ("dk", "dv") or not bits:     # sums of atomics in any order
            pu.assert_close(f"{what} {name}", a, b.cpu(), host[0].dtype, backward=True)
        else:
            assert torch.equal(a, b.cpu()), (what, name)


def _arena(dims, window, dtype):
    n = binding.dsa3d_step_host_arena_bytes(*dims, window, dtype)
    return torch.full((n,), 0xA5, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("dtype,dims", [(BF16, (3, 45, 80, 7, 128)), (BF16, (4, 30, 52, 16, 64)), (F32, (2, 30, 52, 11, 64))])
def test_pipelined_steps_before_and_after_steps_by_groups(dtype, dims):
    """No flush and no synchronisation in between: the buffers of one lie across those of the other in the arena."""
    window = (3, 3, 3)
    assert binding.dsa3d_test_step_group_heads(*dims, window, dtype) > 0
    arena = _arena(dims, window, dtype)
    order = "PGPPGGP"                            # pipelined, by groups
    hosts = [[z.pin_memory() for z in small_problem(*dims, window, dtype, 1.0, 960 + i)] for i in range(len(order))]
    results = [_results(h) for h in hosts]
    torch.cuda.synchronize()
    for kind, h, r in zip(order, hosts, results):
        (binding.dsa3d_step_host_pipelined if kind == "P" else binding.dsa3d_step_host)(*h, *dims, window, *r, arena)
    binding.dsa3d_step_host_flush()
    torch.cuda.synchronize()
    for i, (h, r) in enumerate(zip(hosts, results)):
        _check(h, r, dims, window, f"step {i} ({order[i]})")


@pytest.mark.parametrize("pageable", [0, 3, 6, 8, "all"])   # q, offsets, lse, dk, every tensor
def test_memory_that_is_not_page_locked(pageable):
    dims, window = (3, 45, 80, 7, 128), (3, 3, 3)
    host = [z.pin_memory() for z in small_problem(*dims, window, BF16, 1.0, 970)]
    res = _results(host)
    if pageable == "all":
        host, res = [z.clone() for z in host], _results(host, pin=False)
    elif pageable < 5:
        host[pageable] = host[pageable].clone()
        assert not host[pageable].is_pinned()
    else:
        res[pageable - 5] = res[pageable - 5].clone()
        assert not res[pageable - 5].is_pinned()
    binding.dsa3d_step_host(*host, *dims, window, *res, _arena(dims, window, BF16))
    torch.cuda.synchronize()
    _check(host, res, dims, window, f"pageable {pageable}")


@pytest.mark.parametrize("dtype,dims", [(BF16, (3, 45, 80, 7, 128)), (F32, (2, 45, 80, 5, 128)), (F32, (2, 45, 80, 19, 32))])
@pytest.mark.parametrize("window", [(1, 1, 1), (1, 1, 2), (1, 1, 3), (1, 2, 3)])
def test_narrow_offsets(dtype, dims, window):
    """12 bytes per sample and head: on both sides of 64 per token and group, the last group narrower than the others."""
    assert binding.dsa3d_test_step_group_heads(*dims, window, dtype) > 0
    host = [z.pin_memory() for z in small_problem(*dims, window, dtype, 1.0, 975)]
    res = _results(host)
    n = binding.dsa3d_step_host_arena_bytes(*dims, window, dtype)
    arena = torch.full((n + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        binding.dsa3d_step_host(*host, *dims, window, *res, arena[:n])
    torch.cuda.synchronize()
    assert bool((arena[n:] == 0xA5).all())
    _check(host, res, dims, window, f"window {window}")

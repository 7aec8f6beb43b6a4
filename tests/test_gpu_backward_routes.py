"""The routes of the bf16 backward: samples sorted by key cell (the default), the gather kernel with the tile pre-reduction of
dK/dV (DSA3D_TILE, and where the workspace is too small for a pass of the sort) and the gather kernel with every
contribution an atomic add (DSA3D_TILE=0).  Every gradient of each is compared with the CPU oracle element by
element at the bf16 tolerance, and the routes with one another."""
import pytest
import torch

import oracle
import parity_util as pu
from paper_2607_22696_b200 import binding, inputs
from test_gpu_parity import small_problem

pytestmark = pytest.mark.gpu
BF16, F32 = torch.bfloat16, torch.float32


ROUTES = {"cells": None, "tiles": "4,8,8,6", "rows": "0"}


@pytest.fixture(params=sorted(ROUTES))
def route(request, monkeypatch):
    if ROUTES[request.param] is None:
        monkeypatch.delenv("DSA3D_TILE", raising=False)
    else:
        monkeypatch.setenv("DSA3D_TILE", ROUTES[request.param])
    yield request.param
    assert binding.dsa3d_device_timeout_flag() == 0


@pytest.mark.parametrize("shape,window,sigma", [
    ((5, 7, 9, 3, 64), (3, 3, 3), 1.0),          # ragged everywhere
    ((9, 17, 19, 2, 128), (3, 3, 3), 2.0),       # several tiles per axis, offsets that reach the halo's edge
    ((13, 9, 26, 1, 128), (3, 3, 3), 4.0),       # many corners beyond the halo: the gather kernel's own scatter
    ((4, 8, 8, 2, 64), (2, 2, 2), 0.7),          # exactly one tile of the pre-reduction, even window
    ((6, 10, 12, 2, 128), (1, 1, 1), 1.5),
    ((1, 1, 1, 1, 128), (3, 3, 3), 0.5),
    ((1, 9, 40, 2, 64), (3, 3, 3), 1.0),
    ((12, 1, 11, 2, 128), (3, 3, 3), 1.0),
])
def test_route_matches_the_oracle(shape, window, sigma, route):
    pu.full_parity(*small_problem(*shape, window, BF16, sigma, 900 + shape[0] + shape[2]), window)


@pytest.mark.parametrize("window", [(3, 5, 5), (3, 7, 7), (4, 8, 8)])
def test_windows_of_more_than_32_samples(window, route):
    pu.full_parity(*small_problem(6, 11, 13, 2, 128, window, BF16, 1.5, 910), window)
    pu.full_parity(*small_problem(5, 9, 10, 2, 64, window, BF16, 0.3, 911), window)


def test_zero_integer_and_dead_offsets(route):
    """Zero offsets put a window's samples into one cell each; integer offsets leave corner weights of exactly 0
    and 1; NaN, infinite and huge offsets give dead samples, which must reach no kernel's sums."""
    q, k, v, off, dout = small_problem(8, 12, 17, 2, 128, (3, 3, 3), BF16, 1.0, 920)
    pu.full_parity(q, k, v, torch.zeros_like(off), dout, (3, 3, 3))
    ioff = inputs.uniform_int(off.shape, 921, 3, -3, 3, F32)
    pu.full_parity(q, k, v, ioff, dout, (3, 3, 3))
    bad = off.clone()
    flat = bad.view(-1)
    flat[5::97] = float("nan")
    flat[11::89] = float("inf")
    flat[17::83] = -3.0e38
    pu.full_parity(q, k, v, bad, dout, (3, 3, 3))


@pytest.mark.parametrize("dims", [(10, 14, 18, 3, 128), (7, 9, 22, 2, 64), (5, 12, 13, 3, 32)])
def test_routes_agree(dims, monkeypatch):
    """The routes sum the same fp32 terms in other orders; rounded to bf16 two results are at most one step apart, 2^-7 of a value or, near zero, of the tensor's size.  doffsets stays fp32: 54 dot
    products of 128 terms at 2^-24 each, far below 1e-4."""
    window = (3, 3, 3)
    q, k, v, off, dout = small_problem(*dims, window, BF16, 2.0, 930)
    dev = [z.cuda() for z in (q, k, v, off, dout)]
    out, lse = pu.gpu_forward(*dev[:4], dims, window)
    got = {}
    for name, tile in ROUTES.items():
        monkeypatch.delenv("DSA3D_TILE", raising=False) if tile is None else monkeypatch.setenv("DSA3D_TILE", tile)
        got[name] = pu.gpu_backward(*dev[:4], lse, dev[4], dims, window)
    for other in ("tiles", "rows"):
        for a, b in zip(got["cells"][:3], got[other][:3]):                   # dq, dk, dv
            a, b = a.float(), b.float()
            step = (b.abs() * 2.0 ** -7).clamp_min(float(b.pow(2).mean().sqrt()) * 2.0 ** -7)
            assert bool(((a - b).abs() <= step).all())
        a, b = got["cells"][3], got[other][3]
        assert float((a - b).abs().max()) <= 1e-4 * max(1.0, float(b.abs().max()))
    assert torch.equal(got["tiles"][0], got["rows"][0]) and torch.equal(got["tiles"][3], got["rows"][3])      # the same gather kernel


@pytest.mark.parametrize("d", [32, 64, 128])
def test_weights_of_dv_keep_their_32_bits(d, route):
    """Pairs of queries sample almost the same position with opposite dO: a key's dV is the difference of two weights in
    (0, 1) that agree in 15 to 18 bits.  Grid positions below 8 leave fractions of 2^-21, so the weights are exact in fp32
    (lse 0, one sample: alpha is 1) and only their products and the sum round: 2^-23 of |dO| <= 2 each, twice, beside
    the rounding of the result, 2^-9 of it."""
    T, H, W, heads = 3, 6, 8, 2
    g = torch.Generator().manual_seed(951)
    q = torch.zeros(T, H, W, heads, d, dtype=BF16)
    k, v = (torch.randn(q.shape, generator=g).to(BF16) for _ in range(2))
    dout = torch.randn(T, H, W // 2, 1, heads, d, generator=g).clamp_(-2, 2).to(BF16)
    dout = torch.cat([dout, -dout], dim=3).view(q.shape).contiguous()
    f = torch.randint(100000, 2000000, (T, H, W // 2, heads), generator=g)
    near = f + torch.randint(8, 64, f.shape, generator=g)
    frac = torch.stack([f, near], dim=3).view(T, H, W, heads).double() * 2.0 ** -21
    x = torch.arange(W).view(1, 1, W, 1)
    off = torch.zeros(T, H, W, heads, 1, 3)
    off[..., 0, 2] = ((x // 2 * 2).double() + frac - x).float()
    assert torch.equal(x.float() + off[..., 0, 2], ((x // 2 * 2).double() + frac).float())
    dims = (T, H, W, heads, d)
    dev = [z.cuda() for z in (q, k, v, off, dout)]
    out, lse = pu.gpu_forward(*dev[:4], dims, (1, 1, 1))
    dv = pu.gpu_backward(*dev[:4], lse, dev[4], dims, (1, 1, 1))[2].cpu().double()
    ref = oracle.backward(q, k, v, off, dout, T, H, W, heads, d, (1, 1, 1))[2].view(q.shape)
    assert float(ref.abs().max()) > 2.0 ** -17
    assert bool(((dv - ref).abs() <= ref.abs() * 2.0 ** -8 + 2.0 ** -21).all())


@pytest.mark.parametrize("shape", [(19, 9, 10, 2, 128), (6, 10, 12, 3, 64)])
def test_host_step_in_slabs_of_frames(shape, route):
    """dsa3d_step_host walks the video in slabs of frames: each slab's launches add the contributions of that
    slab's queries only, to every key its frames can reach."""
    window = (3, 3, 3)
    q, k, v, off, dout = small_problem(*shape, window, BF16, 1.3, 940)
    dims = tuple(q.shape)
    pin = lambda z: z.clone().pin_memory()
    hin = [pin(z) for z in (q, k, v, off, dout)]
    hout = {n: torch.full_like(q, float("nan")).pin_memory() for n in ("out", "dq", "dk", "dv")}
    hout["lse"] = torch.full(dims[:4], float("nan")).pin_memory()
    hout["doff"] = torch.full_like(off, float("nan")).pin_memory()
    arena = torch.empty(binding.dsa3d_step_host_arena_bytes(*dims, window, BF16), dtype=torch.uint8, device="cuda")
    binding.dsa3d_step_host(*hin, *dims, window, hout["out"], hout["lse"], hout["dq"], hout["dk"], hout["dv"],
                            hout["doff"], arena)
    torch.cuda.synchronize()
    T, H, W, heads, d = dims
    refs = oracle.backward(q, k, v, off, dout, T, H, W, heads, d, window)
    for name, got, ref in zip(("dq", "dk", "dv", "doffsets"), (hout["dq"], hout["dk"], hout["dv"], hout["doff"]), refs):
        pu.assert_close(name, got, ref, BF16, backward=True)

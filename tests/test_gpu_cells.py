"""The kernels behind dsa3d_forward / dsa3d_backward that list or sort samples, at the sizes where they can go wrong: query
tiles are 4 x 4 x 6 (t, y, x), cell blocks 4 x 4 x 3, samples more than 12 positions off their tile leave the bins, a warp takes
four, two or one query (windows of at most 8, 16, more samples) and 32 samples at a time.  Compared with the CPU oracle
element by element (tolerances of parity_util), the fp32 route also with the row kernels it replaces."""
import pytest
import torch

import parity_util as pu
from paper_2607_22696_b200 import autograd as ops, binding, inputs
from test_gpu_parity import small_problem

pytestmark = pytest.mark.gpu
BF16, F32 = torch.bfloat16, torch.float32


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("shape,window,sigma", [
    ((4, 4, 6, 2), (3, 3, 3), 1.0),              # one tile exactly
    ((5, 5, 7, 1), (3, 3, 3), 1.5),              # one position beyond it on every axis
    ((3, 3, 5, 2), (2, 2, 2), 0.7),              # one short; four queries per warp
    ((4, 8, 13, 1), (2, 2, 3), 1.0),             # 12 samples: two queries per warp, 13 odd
    ((2, 9, 12, 1), (1, 4, 4), 1.0),             # 16 samples exactly
    ((2, 5, 9, 1), (1, 1, 1), 1.0),
    ((5, 7, 8, 1), (2, 4, 4), 1.0),              # 32 samples exactly
    ((4, 6, 9, 1), (3, 3, 4), 2.0),              # 36: a second round of four
    ((3, 40, 60, 1), (1, 3, 3), 9.0),            # samples beyond the bins of their tile
])
def test_tile_edges_and_windows(shape, window, sigma, d):
    pu.full_parity(*small_problem(*shape, d, window, BF16, sigma, 700 + shape[2] + d), window)


def test_rows_that_are_not_32_byte_aligned():
    window = (3, 3, 3)
    q, k, v, off, dout = small_problem(5, 6, 8, 1, 64, window, BF16, 1.0, 720)
    dims = tuple(q.shape)

    def shifted(z):
        buf = torch.empty(z.numel() + 8, dtype=z.dtype, device="cuda")
        out = buf[8:].view(z.shape)
        out.copy_(z)
        assert out.data_ptr() % 32 == 16
        return out

    dev = [z.cuda() for z in (q, k, v, off, dout)]
    out, lse = pu.gpu_forward(*dev[:4], dims, window)
    want = pu.gpu_backward(*dev[:4], lse, dev[4], dims, window)
    got = pu.gpu_backward(shifted(q), dev[1], dev[2], dev[3], lse, shifted(dout), dims, window)
    for a, b in ((got[0], want[0]), (got[3], want[3])):
        assert torch.equal(a, b)                 # the same sums in the same order
    for a, b in ((got[1], want[1]), (got[2], want[2])):
        pu.assert_close("dk, dv", a, b.cpu(), BF16, backward=True)


@pytest.mark.parametrize("d,window,shape,sigma,kind", [
    (32, (3, 3, 3), (9, 32, 43, 3), 1.0, "normal"),
    (64, (3, 3, 3), (7, 33, 55, 3), 9.0, "normal"),      # many samples beyond the bins
    (128, (3, 3, 3), (8, 33, 48, 3), 1.5, "normal"),
    (64, (3, 7, 7), (3, 37, 62, 1), 2.0, "normal"),
    (64, (3, 3, 3), (9, 32, 44, 3), 0.0, "int"),         # the check leaves these to the row kernel
    (64, (4, 4, 1), (8, 33, 80, 3), 1.0, "normal"),      # the smallest window
])
def test_fp32_storage_from_a_million_samples_on(d, window, shape, sigma, kind, monkeypatch):
    """Both routes sum the same terms in other orders.  A gradient element adds up to 8 P + 8 * (samples of a cell) products of
    numbers of order 1; at 2^-24 each, and their signs random, the two differ by far less than 1e-4."""
    T, H, W, heads = shape
    P = window[0] * window[1] * window[2]
    q, k, v, off, dout = (z.cuda() for z in small_problem(T, H, W, heads, d, window, F32, max(sigma, 0.1), 730 + d))
    if kind == "int":
        off = inputs.uniform_int((T, H, W, heads, P, 3), 731, 3, -3, 3, F32).cuda()
    off.view(-1)[7::9973] = float("nan")                 # dead samples
    dims = (T, H, W, heads, d)
    assert T * H * W * heads * P >= 1000000
    nbytes = binding.dsa3d_backward_workspace_bytes(*dims, window, F32)
    assert nbytes > 0
    out, lse = pu.gpu_forward(q, k, v, off, dims, window)

    def backward(workspace):
        g = [torch.full_like(z, float("nan")) for z in (q, q, q, off)]
        binding.dsa3d_backward(q, k, v, off, lse, dout, *dims, window, *g, workspace)
        return g

    whole = backward(torch.full((nbytes,), 0xFF, dtype=torch.uint8, device="cuda"))
    parts = backward(torch.full((nbytes * 2 // 5,), 0xFF, dtype=torch.uint8, device="cuda"))     # several passes
    rows = backward(None)
    monkeypatch.setenv("DSA3D_TILE", "0")
    again = backward(torch.empty(nbytes, dtype=torch.uint8, device="cuda"))
    for name, a, b, c, e in zip(("dq", "dk", "dv", "doffsets"), whole, parts, rows, again):
        assert bool(torch.isfinite(c).all())
        scale = max(1.0, float(c.abs().max()))
        for other in (a, b, e):
            assert float((other - c).abs().max()) <= pu.F32_BWD_ATOL * scale, name


@pytest.mark.parametrize("dtype,dims,window,scratch", [
    (F32, (26, 40, 48, 1, 64), (3, 3, 3), 36 << 20),     # four passes, the last of two frames
    (F32, (30, 24, 90, 1, 32), (4, 2, 2), 12 << 20),     # eight of four frames
    (BF16, (64, 68, 120, 1, 32), (1, 1, 2), None),       # the workspace the library asks for
])
def test_passes_over_frames_stay_inside_the_workspace(dtype, dims, window, scratch):
    """Passes in the middle of the video use the most scratch.  Bytes behind the workspace keep their pattern, and the gradients
    are those of the row kernels (tolerances as in the tests around this one)."""
    T, H, W, heads, d = dims
    front = 8 * T * H * W * heads * d if dtype == BF16 else 256          # accumulators, or gate words
    nbytes = scratch or binding.dsa3d_backward_workspace_bytes(*dims, window, dtype)
    passes, largest = binding.dsa3d_test_backward_passes(*dims, window, dtype, nbytes - front)
    assert passes >= 3 and largest <= nbytes - front
    q, k, v, off, dout = (z.cuda() for z in small_problem(*dims, window, dtype, 1.5, 740 + T))
    _, lse = pu.gpu_forward(q, k, v, off, dims, window)
    guard = 4 << 20

    def backward():
        buf = torch.full((nbytes + guard,), 0xA5, dtype=torch.uint8, device="cuda")
        g = [torch.full_like(z, float("nan")) for z in (q, q, q, off)]
        binding.dsa3d_backward(q, k, v, off, lse, dout, *dims, window, *g, buf[:nbytes])
        assert bool((buf[nbytes:] == 0xA5).all())
        return g

    got = backward()
    with pytest.MonkeyPatch.context() as mp:
        mp.setenv("DSA3D_TILE", "0")
        want = backward()
    for name, a, b in zip(("dq", "dk", "dv", "doffsets"), got, want):
        pu.assert_close(name, a, b.cpu(), dtype, backward=True)


def test_a_captured_fp32_call_shares_nothing_with_calls_on_other_streams():
    """The fp32 route is chosen on the device by the offsets.  A graph of a call with real-valued offsets, replayed on one stream
    while more than 512 calls with integer ones run on another, gives what the call gives alone."""
    window, dims = (3, 3, 3), (6, 32, 40, 5, 32)
    q, k, v, off, dout = (z.cuda() for z in small_problem(*dims, window, F32, 1.5, 761))
    grid = inputs.uniform_int(tuple(off.shape), 762, 3, -2, 2, F32).cuda()
    nbytes = binding.dsa3d_backward_workspace_bytes(*dims, window, F32)
    assert nbytes > 0
    lse = {id(o): pu.gpu_forward(q, k, v, o, dims, window)[1] for o in (off, grid)}

    class Call:
        def __init__(self, offsets):
            self.offsets, self.g = offsets, [torch.full_like(z, float("nan")) for z in (q, q, q, off)]
            self.ws = torch.full((nbytes,), 0xFF, dtype=torch.uint8, device="cuda")

        def __call__(self):
            binding.dsa3d_backward(q, k, v, self.offsets, lse[id(self.offsets)], dout, *dims, window, *self.g, self.ws)

        def check(self, want):
            for name, a, b in zip(("dq", "dk", "dv", "doffsets"), self.g, want):
                assert float((a - b).abs().max()) <= pu.F32_BWD_ATOL * max(1.0, float(b.abs().max())), name

    alone = {}
    for o in (off, grid):
        c = Call(o)
        c()
        alone[id(o)] = c.g
    captured, eager = Call(off), Call(grid)
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph):
        captured()
    with torch.cuda.stream(side):
        for _ in range(600):
            eager()
    for _ in range(300):
        graph.replay()
        captured.check(alone[id(off)])
    torch.cuda.synchronize()
    eager.check(alone[id(grid)])


@pytest.mark.parametrize("frames", [6, 34])             # slabs of one frame, and of five with enough samples to be sorted
@pytest.mark.parametrize("old_arena", [False, True])
def test_fp32_host_step_with_and_without_room_for_the_sort(frames, old_arena):
    """The sort's workspace comes last in the arena and fp32 does without it: an arena that ends before it is taken too."""
    window, dims = (3, 3, 3), (frames, 30, 52, 5, 32)
    host = small_problem(*dims, window, F32, 1.5, 763)
    q, k, v, off, dout = host
    nbytes = binding.dsa3d_step_host_arena_bytes(*dims, window, F32)
    buffers = sum((z.numel() * 4 + 255) // 256 * 256 * n for z, n in ((q, 10), (off, 2), (q[..., 0], 1)))
    assert (nbytes > buffers) == (frames == 34) and nbytes >= buffers
    if old_arena:
        nbytes = buffers
    hin = [z.clone().pin_memory() for z in host]
    hout = [torch.full(z.shape, float("nan")).pin_memory() for z in (q, q[..., 0], q, k, v, off)]     # out, lse, dq, dk, dv, doffsets
    buf = torch.full((nbytes + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    binding.dsa3d_step_host(*hin, *dims, window, *hout, buf[:nbytes])
    torch.cuda.synchronize()
    assert bool((buf[nbytes:] == 0xA5).all())
    dev = [z.cuda() for z in host]
    out, lse = pu.gpu_forward(*dev[:4], dims, window)
    want = (out, lse) + tuple(pu.gpu_backward(*dev[:4], lse, dev[4], dims, window))
    for name, a, b in zip(("out", "lse", "dq", "dk", "dv", "doffsets"), hout, want):
        assert float((a - b.cpu()).abs().max()) <= pu.F32_BWD_ATOL * max(1.0, float(b.abs().max())), name


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("window,shape", [((2, 2, 2), (3, 5, 7, 2)), ((3, 3, 3), (1, 4, 8, 3)), ((3, 5, 5), (3, 7, 11, 1)),
                                          ((3, 7, 7), (4, 9, 17, 2))])
def test_fixed_window_gradients_do_not_depend_on_asking_for_doffsets(d, window, shape):
    """Without dOffsets the tables hold the window alone and a thread per token forms the coefficients: tokens that are and
    are not a multiple of 32, every window with a table."""
    T, H, W, heads = shape
    P = window[0] * window[1] * window[2]
    dims = (T, H, W, heads, d)
    q, k, v, _, dout = (z.cuda() for z in small_problem(*dims, window, BF16, 0.5, 750 + P))
    out, lse = torch.empty_like(q), torch.empty(dims[:4], dtype=F32, device="cuda")
    binding.dsa3d_forward_fixed_window(q, k, v, *dims, window, out, lse)
    results = []
    for doff in (torch.empty((T, H, W, heads, P, 3), dtype=F32, device="cuda"), None):
        ws = torch.full((binding.dsa3d_backward_fixed_window_workspace_bytes(*dims, window, BF16),), 0xFF, dtype=torch.uint8, device="cuda")
        g = [torch.full_like(q, float("nan")) for _ in range(3)]
        binding.dsa3d_backward_fixed_window(q, k, v, lse, dout, *dims, window, *g, doff, ws)
        results.append(g)
    torch.cuda.synchronize()
    for a, b in zip(*results):
        assert bool(torch.isfinite(b.float()).all()) and torch.equal(a, b)


def test_autograd_takes_what_has_to_be_converted_and_raises_what_the_library_refuses():
    window = (3, 3, 3)
    q, k, v, off, dout = (z.cuda() for z in small_problem(3, 4, 5, 2, 64, window, BF16, 1.0, 770))
    leaves = [z.requires_grad_() for z in (q, k, v, off)]
    want = torch.autograd.grad(ops.dsa3d(*leaves, window), leaves, dout)
    other = [z.detach().transpose(1, 2).contiguous().transpose(1, 2).requires_grad_() for z in leaves]     # not contiguous
    got = torch.autograd.grad(ops.dsa3d(*other, window), other, dout)
    for i in (0, 3):
        assert torch.equal(got[i], want[i])
    with pytest.raises(ValueError):
        ops.dsa3d(q.detach().cpu(), k, v, off, window)
    with pytest.raises(binding.Dsa3dError):              # 48 channels
        ops.dsa3d(*(z.detach()[..., :48].contiguous() for z in (q, k, v)), off, window)
    out = ops.dsa3d(*leaves, window)
    buf = torch.zeros(dout.numel() + 1, dtype=BF16, device="cuda")
    with pytest.raises(binding.Dsa3dError):              # a gradient off its 16-byte alignment, refused in the backward
        torch.autograd.grad(out, leaves, buf[1:].view(dout.shape))


@pytest.mark.parametrize("contiguous", [True, False])    # the compiled function, and the one that converts
def test_fp32_backward_on_a_card_too_full_for_the_sort(contiguous):
    """The room to sort in is several times the tensors; where it does not fit, the row kernels run."""
    window, dims = (3, 3, 3), (8, 30, 52, 8, 32)
    q, k, v, off, dout = (z.cuda() for z in small_problem(*dims, window, F32, 1.5, 780))
    if not contiguous:
        q = q.transpose(1, 2).contiguous().transpose(1, 2)
    leaves = [z.requires_grad_() for z in (q, k, v, off)]
    want = torch.autograd.grad(ops.dsa3d(*leaves, window), leaves, dout)
    nbytes = binding.dsa3d_backward_workspace_bytes(*dims, window, F32)
    out = ops.dsa3d(*leaves, window)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    room = torch.cuda.memory_reserved() + 3 * q.numel() * 4 + off.numel() * 4 + (64 << 20)
    assert nbytes > 128 << 20
    torch.cuda.set_per_process_memory_fraction(room / total)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        got = torch.autograd.grad(out, leaves, dout)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    for name, a, b in zip(("dq", "dk", "dv", "doffsets"), got, want):
        assert float((a - b).abs().max()) <= pu.F32_BWD_ATOL * max(1.0, float(b.abs().max())), name

"""How the cell-sorted backward divides a problem when its scratch is short: by heads, then by frames.  A pass in the middle of
the video reaches more key blocks than the first one (samples fall into blocks before its own frames too), and none may use
more than the scratch it was given.  Host arithmetic; the same on the GPU in test_gpu_cells.py."""
import random

import pytest
import torch

from paper_2607_22696_b200 import binding, build

BF16, F32 = torch.bfloat16, torch.float32


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


def scratch_of(dims, window, dtype):
    """What a call with the workspace the library asks for has for the passes."""
    T, H, W, heads, d = dims
    nbytes = binding.dsa3d_backward_workspace_bytes(*dims, window, dtype)
    return nbytes - (8 * T * H * W * heads * d if dtype == BF16 else 256)


@pytest.mark.parametrize("dims,window,dtype,scratch", [
    ((32, 68, 120, 2, 64), (3, 7, 7), F32, None),            # the library's own workspace
    ((128, 68, 120, 2, 64), (3, 3, 3), F32, None),
    ((64, 68, 120, 1, 32), (1, 1, 1), BF16, None),
    # dsa3d_backward_noalloc's array: four frames at the start would fit, four in the middle do not
    ((62, 45, 80, 1, 32), (2, 2, 2), BF16, 2 * 8 * 1024 * 1024 * 4 - 8 * 62 * 45 * 80 * 32),
])
def test_every_pass_fits_its_scratch(dims, window, dtype, scratch):
    scratch = scratch_of(dims, window, dtype) if scratch is None else scratch
    passes, largest = binding.dsa3d_test_backward_passes(*dims, window, dtype, scratch)
    assert passes > dims[3] or passes == 0                   # divided by frames, or left to the row kernels
    assert largest <= scratch


def test_every_pass_fits_whatever_scratch_it_is_given():
    rng = random.Random(5)
    divided = 0
    for _ in range(3000):
        dims = (rng.randint(1, 90), rng.randint(1, 40), rng.randint(1, 60), rng.randint(1, 5), rng.choice([32, 64, 128]))
        window = (rng.randint(1, 3), rng.randint(1, 7), rng.randint(1, 7))
        whole = binding.dsa3d_test_backward_passes(*dims, window, BF16, 1 << 60)
        assert whole[0] == 1
        scratch = int(whole[1] * rng.uniform(0.02, 1.1))
        passes, largest = binding.dsa3d_test_backward_passes(*dims, window, BF16, scratch)
        assert largest <= scratch
        divided += passes > dims[3]
    assert divided > 300


def test_fp32_host_step_asks_for_what_its_slabs_can_use():
    """The host step runs by slabs of an eighth of the video.  Slabs too small to be sorted ask for no room to sort in."""
    def extra(dims, window=(3, 3, 3)):
        T, H, W, heads, d = dims
        items, up = T * H * W * heads, lambda x: (x + 255) // 256 * 256
        buffers = 10 * up(items * d * 4) + 2 * up(items * 27 * 12) + up(items * 4)
        return binding.dsa3d_step_host_arena_bytes(*dims, window, F32) - buffers

    assert extra((8, 30, 52, 8, 64)) == 0                    # slabs of one frame
    assert extra((64, 12, 10, 8, 64)) == 0                   # of eight, 207,360 samples
    whole = binding.dsa3d_backward_workspace_bytes(64, 30, 52, 8, 64, (3, 3, 3), F32)
    assert 0 < extra((64, 30, 52, 8, 64)) < whole            # of eight, 2.7 million

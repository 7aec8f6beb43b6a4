"""Which host steps go by groups of heads, and how many heads a group has.  Host arithmetic; the steps themselves in
test_gpu_host_groups.py and test_gpu_host_heads.py."""
import pytest
import torch

from paper_2607_22696_b200 import binding, build

BF16, F32 = torch.bfloat16, torch.float32


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


@pytest.mark.parametrize("dtype,dims,group", [
    (BF16, (8, 45, 80, 16, 128), 4),             # rows of 1 KB, four groups
    (BF16, (8, 45, 80, 12, 128), 2),             # ... would be three: 512 bytes
    (BF16, (3, 45, 80, 7, 128), 2),
    (BF16, (3, 45, 80, 6, 128), 0),              # three groups of 512 bytes: too few
    (BF16, (3, 45, 80, 5, 128), 0),
    (BF16, (4, 30, 52, 16, 64), 4),              # 512 bytes: rows of 1 KB make two groups
    (BF16, (2, 30, 52, 17, 128), 4),
    (BF16, (2, 4, 64, 256, 64), 32),             # eight groups at most, whatever their width
    (BF16, (3, 30, 52, 16, 64), 4),
    (F32, (2, 30, 52, 11, 64), 2),
    (F32, (3, 30, 52, 9, 64), 2),
    (F32, (8, 45, 80, 8, 64), 2),
    (F32, (8, 45, 80, 4, 128), 1),
    (F32, (8, 45, 80, 3, 128), 0),
    (BF16, (1, 1, 1024, 32, 128), 4),            # tensors of 8 MB go by groups, of a token less they do not
    (BF16, (1, 1, 1023, 32, 128), 0),
])
def test_heads_of_a_group(dtype, dims, group):
    assert binding.dsa3d_test_step_group_heads(*dims, (3, 3, 3), dtype) == group


def test_a_group_covers_all_heads_in_eight_and_refused_shapes_are_refused():
    for heads in range(1, 300):
        group = binding.dsa3d_test_step_group_heads(4, 64, 64, heads, 64, (1, 1, 2), BF16)
        assert group == 0 or 4 <= -(-heads // group) <= 8
    with pytest.raises(binding.Dsa3dError):
        binding.dsa3d_test_step_group_heads(4, 8, 8, 2, 48, (3, 3, 3), BF16)

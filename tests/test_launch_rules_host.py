"""Launch rules of the kernels as host functions of sizes, without a GPU."""
import pytest

from launch_rules import rules


@pytest.mark.parametrize("cap", [0, -1, 1, 152, 1 << 22, 1 << 23, 1 << 30])
@pytest.mark.parametrize("items", [0, 1, 8, 9, 1 << 20, (1 << 25) + 1, 1 << 28, 1 << 40])
def test_copy_grid_strides_in_int(items, cap):
    """A copy kernel's thread steps from its index to the next by the grid's threads (block
    ids) or warps (items, fewer than 2^28: one is 8 rows of a pool of under 2^31), in int:
    no step from inside the range may leave an int."""
    r = rules()
    ctas, threads = r.grid_ctas(items, cap), r.copy_threads()
    assert 1 <= ctas <= max(1, -(-items * 32 // threads))
    assert cap <= 0 or ctas <= max(1, cap)
    most = 2 ** 31 - 1
    assert r.inline_blocks() - 1 + ctas * threads <= most
    assert min(items, 1 << 28) - 1 + ctas * threads // 32 <= most

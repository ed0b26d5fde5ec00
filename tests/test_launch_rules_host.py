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


@pytest.mark.parametrize("sms", [132, 152])
def test_migrations_beside_decode_stride(sms):
    """A move that decode may run beside is a few CTAs an SM, which keep their slots; one by
    itself has no bound; the caller's limit holds in both."""
    ctas = rules().migration_ctas
    assert ctas(0, 0, sms) == 0 and ctas(0, 1, sms) == 16 * sms
    for limit in (1, 8, sms, 16 * sms - 1):
        assert ctas(limit, 0, sms) == ctas(limit, 1, sms) == limit
    assert ctas(1 << 20, 0, sms) == 1 << 20 and ctas(1 << 20, 1, sms) == 16 * sms

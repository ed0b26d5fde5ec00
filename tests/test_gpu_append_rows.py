"""Appends whose new block ids ride in the launch: the blocks' bytes and the
session's device table row, at the edges of a block and of the launch's room."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def device_row(pool, sid):
    """The session's row and length as the device has them."""
    n = len(pool.session_block_table(sid))
    row = torch.empty(n, dtype=torch.int32, device="cuda")
    length = torch.empty(1, dtype=torch.int32, device="cuda")
    pool.batch_tables([sid], row, n, length)
    return row.cpu().tolist(), int(length.item())


@pytest.mark.parametrize("bt", [16, 64])
@pytest.mark.parametrize("lru", [False, True])
@pytest.mark.parametrize("hkv", [1, 2, 3, 8])
# 2 048 blocks of 16 tokens fill the launch; one more goes through a table write
@pytest.mark.parametrize("parts", [[1], [16], [17, 47, 1], [5, 32768], [7, 32769 + 16], [64, 1, 63]])
def test_append_rows(cuda_dev, bt, lru, hkv, parts):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2609_25782_gb300 import Pool
    L, d = 2, 128
    total = sum(parts)
    nb = -(-total // bt) + 3
    cap = total * L * 2 * hkv * d * 2 + 256
    pool = Pool(num_layers=L, num_hot_blocks=nb, cold_bytes=cap, num_q_heads=hkv, num_kv_heads=hkv,
                block_tokens=bt, max_sessions=2, max_batch=1, max_context=total, alloc_seed=3,
                lru_residency=lru)
    pool.hot.zero_()
    sid = pool.session_create(total)
    g = torch.Generator(device="cuda").manual_seed(1)
    want = torch.zeros(L, 2, hkv, nb * bt, d, dtype=torch.bfloat16, device="cuda")
    at = 0
    for n in parts:
        k, v = (torch.randn(L, n, hkv, d, device="cuda", generator=g).bfloat16() for _ in range(2))
        pool.session_append(sid, k, v)
        want[:, 0, :, at:at + n] = k.transpose(1, 2)
        want[:, 1, :, at:at + n] = v.transpose(1, 2)
        at += n
        row, length = device_row(pool, sid)
        assert length == at and row == pool.session_block_table(sid)
    blocks = torch.as_tensor(np.asarray(pool.session_block_table(sid), dtype=np.int64), device="cuda")
    got = pool.hot_view()[blocks].permute(1, 2, 3, 0, 4, 5).reshape(L, 2, hkv, -1, d)
    assert torch.equal(got, want[:, :, :, :got.shape[3]])   # rows past the tokens stay zero
    assert pool.check_device() == 0

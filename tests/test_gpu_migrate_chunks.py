"""Moves that begin or end beside a migration chunk's edge (8 tokens), against
the tokens that were appended, bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bt", [16, 64])
@pytest.mark.parametrize("lru", [False, True])
@pytest.mark.parametrize("t1,t2", [(7, 8), (8, 9), (9, 24), (23, 25), (57, 71), (64, 120)])
def test_pack_and_unpack_at_chunk_edges(cuda_dev, bt, lru, t1, t2):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2609_25782_gb300 import Pool
    L, hkv, d = 2, 2, 128
    nb = -(-t2 // bt)
    pool = Pool(num_layers=L, num_hot_blocks=nb, cold_bytes=1 << 22, num_q_heads=hkv, num_kv_heads=hkv,
                block_tokens=bt, max_sessions=2, max_batch=1, max_context=256, alloc_seed=5,
                lru_residency=lru)
    g = torch.Generator(device="cuda").manual_seed(2)
    kv = torch.randn(2, L, t2, hkv, d, device="cuda", generator=g).bfloat16()
    sid, other = pool.session_create(t2), pool.session_create(t2)
    want = kv.permute(1, 0, 3, 2, 4)                     # [L][K|V][Hkv][T][D]
    for a, b in ((0, t1), (t1, t2)):
        pool.session_append(sid, kv[0, :, a:b].contiguous(), kv[1, :, a:b].contiguous())
        pool.session_pause(sid)
        # Another session takes every block, so the image alone holds the tokens.
        pool.session_append(other, torch.zeros_like(kv[0]), torch.zeros_like(kv[1]))
        assert torch.equal(pool.image(sid)[:, :, :, :b], want[:, :, :, :b])
        pool.session_destroy(other)
        pool.shuffle_free(b)
        pool.session_resume(sid)
        row = torch.as_tensor(pool.session_block_table(sid), device="cuda", dtype=torch.int64)
        got = pool.hot_view()[row].permute(1, 2, 3, 0, 4, 5).reshape(L, 2, hkv, -1, d)
        assert torch.equal(got[:, :, :, :b], want[:, :, :, :b])
        other = pool.session_create(t2)
    assert pool.check_device() == 0


@pytest.mark.parametrize("lru", [False, True])
def test_moves_on_another_stream_than_decode(cuda_dev, lru):
    """After a decode call, moves on another stream take the grid whose CTAs stride over the
    chunks: 64 runs of 901 chunks are more than the 8 warps of 16 CTAs on each SM, and so
    are 8 layers of 3 601 groups of two tokens."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2609_25782_gb300 import Pool
    L, hkv, d, t, bt = 8, 4, 128, 7201, 16
    nb = -(-t // bt)
    pool = Pool(num_layers=L, num_hot_blocks=nb, cold_bytes=2 * nb * bt * L * 2 * hkv * d * 2,
                num_q_heads=hkv, num_kv_heads=hkv, max_sessions=2, max_batch=1, max_context=t,
                alloc_seed=5, lru_residency=lru)
    g = torch.Generator(device="cuda").manual_seed(2)
    kv = torch.randn(2, L, t, hkv, d, device="cuda", generator=g).bfloat16()
    want = kv.permute(1, 0, 3, 2, 4)                     # [L][K|V][Hkv][T][D]
    sid, other = pool.session_create(t), pool.session_create(t)
    pool.session_append(sid, kv[0], kv[1])
    tables = torch.zeros(1, nb, dtype=torch.int32, device="cuda")
    lens = torch.zeros(1, dtype=torch.int32, device="cuda")
    pool.batch_tables([sid], tables, nb, lens)
    q = torch.zeros(1, hkv, d, dtype=torch.bfloat16, device="cuda")
    out = torch.empty(1, hkv, d, device="cuda")
    pool.decode_attention(0, q, tables, lens, 1, nb, 1.0, out)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        pool.session_pause(sid, side)
        # appended there too
        pool.session_append(other, kv[1], kv[0], side)
        assert torch.equal(pool.image(sid), want)
        row = torch.as_tensor(pool.session_block_table(other), device="cuda", dtype=torch.int64)
        got = pool.hot_view()[row].permute(1, 2, 3, 0, 4, 5).reshape(L, 2, hkv, -1, d)
        assert torch.equal(got[:, :, :, :t], want.flip(1))
        pool.session_destroy(other)
        pool.shuffle_free(3)
        pool.session_resume(sid, side)
        row = torch.as_tensor(pool.session_block_table(sid), device="cuda", dtype=torch.int64)
        got = pool.hot_view()[row].permute(1, 2, 3, 0, 4, 5).reshape(L, 2, hkv, -1, d)
        assert torch.equal(got[:, :, :, :t], want)
    side.synchronize()
    assert pool.check_device() == 0

"""The end of a decode call is the end of all its kernels, whatever the lengths.

Tables wider than every session launch a combine kernel that finds nothing to
merge: sessions of one split, or of few splits in a grid long enough for the
split kernel to merge them itself. The next overlapped call, or a graph's next
node, comes after the combine alone, so the combine must not end before the
split kernel: outputs are the same bits as from tables of the sessions' own
width, also with a consumer right behind each call.
"""
import math

import numpy as np
import pytest
import torch

from test_gpu_parity import direct_case, gpu_decode, pkg  # noqa: F401

pytestmark = pytest.mark.gpu

L = 4


# (lengths, table width in tokens): CTAs unshared, at 4 kv-heads
WIDE = [
    # 8 splits x 4 x 40 = 1 280: sessions of 1..4 splits merged by the split kernel, register combine
    ([1025 + 61 * i for i in range(39)] + [5], 8192),
    # 4 x 4 x 40 = 640 of one split each, register combine
    ([30 + 25 * i for i in range(40)], 4096),
    # 20 x 4 x 16 = 1 280 of 1..4 splits, four-warp combine
    ([1025 + 200 * i for i in range(15)] + [900], 40000),
    # 20 x 4 x 12 = 960 of one split each, four-warp combine
    ([11 + 90 * i for i in range(12)], 40000),
    # shared splits: every row waits, one-split sessions among them
    ([700, 3], 4096), ([1000] * 4 + [20] * 4, 4096),
]


@pytest.mark.parametrize("lens,tokens", WIDE)
@pytest.mark.parametrize("bt", [16, 64])
def test_wide_tables(pkg, lens, tokens, bt):  # noqa: F811
    n = len(lens)
    pool, _, tables, q = direct_case(pkg, lens, L=L, bt=bt, seed=41, max_batch=20 * n)
    want = torch.from_numpy(np.concatenate([gpu_decode(pool, l, q, tables, lens) for l in range(L)]))
    width = -(-tokens // bt)
    t = torch.as_tensor(np.pad(tables, ((0, 0), (0, width - tables.shape[1])), constant_values=-1),
                        device="cuda")
    s = torch.as_tensor(np.asarray(lens, dtype=np.int32), device="cuda")
    q = q.contiguous()
    outs = torch.empty(3, L, n, 32, 128, device="cuda")   # overlapped, behind a consumer, from a graph
    step = torch.empty(n, 32, 128, device="cuda")
    copies = torch.empty(L, n, 32, 128, device="cuda")

    def calls(out, consumer):
        st = torch.cuda.current_stream()
        for l in range(L):
            pool.decode_attention(l, q[l], t, s, n, width, 1 / math.sqrt(128),
                                  step if consumer else out[l], st, overlap_previous=l > 0 and not consumer)
            if consumer:
                out[l].copy_(step)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        g = torch.cuda.CUDAGraph()
        g.capture_begin()
        calls(outs[2], False)
        calls(copies, True)
        g.capture_end()
    for _ in range(5):
        outs.fill_(float("nan"))
        copies.fill_(float("nan"))
        calls(outs[0], False)
        calls(outs[1], True)
        g.replay()
        torch.cuda.synchronize()
        for got in (*outs, copies):
            assert torch.equal(got.double().cpu(), want)
    assert pool.check_device() == 0


@pytest.mark.parametrize("n,tokens", [(1, 3000), (8, 4096), (24, 3000), (40, 700)])
def test_call_of_bad_lengths_between_two_others(pkg, n, tokens):  # noqa: F811
    """Rows of a bad length do no work, but a call of nothing else still ends after
    the call before it: the next overlapped call waits for both."""
    lens = [tokens - 7 * i for i in range(n)]
    pool, _, tables, q = direct_case(pkg, lens, L=2, seed=43, max_batch=2 * n)
    want = torch.from_numpy(np.concatenate([gpu_decode(pool, l, q, tables, lens) for l in range(2)]))
    t = torch.as_tensor(tables, device="cuda")
    s = torch.as_tensor(np.asarray(lens, dtype=np.int32), device="cuda")
    bad = torch.zeros_like(s)
    width, scale = t.shape[1], 1 / math.sqrt(128)
    out, none = torch.empty(2, n, 32, 128, device="cuda"), torch.full((n, 32, 128), 7.0, device="cuda")
    for _ in range(5):
        out.fill_(float("nan"))
        st = torch.cuda.current_stream()
        pool.decode_attention(0, q[0], t, s, n, width, scale, out[0], st)
        for _ in range(3):
            pool.decode_attention(0, q[0], t, bad, n, width, scale, none, st, overlap_previous=True)
        pool.decode_attention(1, q[1], t, s, n, width, scale, out[1], st, overlap_previous=True)
        torch.cuda.synchronize()
        assert torch.equal(out.double().cpu(), want)
        assert torch.equal(none, torch.full_like(none, 7.0))
        assert pool.check_device() == pkg.kvtier.KV_DEVICE_BAD_LENGTH
    assert pool.check_device() == 0

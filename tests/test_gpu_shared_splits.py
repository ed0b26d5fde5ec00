"""Splits shared by several CTAs, the launch shape of small decode grids.

A grid that would leave SMs idle gives each split to 2 or 8 CTAs, whose
accumulator states the combine joins. Which CTA takes which tiles follows from
the split plan, so an output is the same bits as from an unshared split (the
same sessions inside a batch too large to share), and within the parity bound
of the oracle. The lengths sit at the edges: one token, one tile, fewer tiles
than accumulators, a split's end, a partial last tile and a full last ring.
"""
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from launch_rules import decode_shape, pool_part_rows
from test_gpu_parity import TOL, direct_case, gpu_decode, host_hot, pkg, scaled_err  # noqa: F401

pytestmark = pytest.mark.gpu


# (lengths of one call, table width in tokens, KV heads, CTAs that share a split
# on a GPU of 152 SMs)
CASES = [
    ([1024], 1024, 4, 1), ([900] * 8, 1024, 4, 1),
    ([1], 1040, 4, 8), ([16], 2048, 4, 8), ([17], 2048, 4, 8), ([127], 2048, 4, 8),
    ([129], 2048, 4, 8), ([1024], 2048, 4, 8), ([1025], 2048, 4, 8), ([2047], 2048, 4, 8),
    ([4096], 4096, 4, 8), ([4097], 5120, 4, 8), ([8193], 8704, 4, 8),
    ([9300], 9728, 4, 2), ([16384], 16384, 4, 2), ([16391], 16448, 4, 2), ([19000], 19008, 4, 2),
    ([2048, 1, 1025, 700], 2048, 4, 8), ([33, 1023, 15, 1040], 1088, 4, 8),
    ([3000, 2049] * 2, 3072, 4, 2),
    # two and three CTAs per SM
    ([2500, 4096, 15, 1024] * 2, 4096, 4, 2), ([4096, 1, 3000, 17, 2048] * 2, 4096, 4, 2),
    # tables of more than 16 splits; a chain of more splits than one batch of loads (35 splits)
    ([40000], 40000, 4, 2), ([70001], 70016, 4, 2), ([33000, 500], 33024, 4, 2),
    ([37000], 37120, 1, 2), ([40000, 36000], 40000, 1, 2),
]


@pytest.mark.parametrize("lens,tokens,hkv,shared", CASES)
@pytest.mark.parametrize("bt,scale", [(16, 1 / math.sqrt(128)), (64, 0.5)])
def test_shared_splits(pkg, lens, tokens, hkv, shared, bt, scale):  # noqa: F811
    n = len(lens)
    many = lens + [100] * (520 // (n * hkv))    # a batch too large to share
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        room = pool_part_rows(len(many), max(many), 8 * hkv, hkv, 152)
        kw = dict(bt=bt, hq=8 * hkv, hkv=hkv, part_rows=room)
        assert decode_shape(tokens, n, **kw).sub == shared
        assert decode_shape(max(many), len(many), **kw).sub == 1
    pool, sess, tables, q = direct_case(pkg, many, L=1, Hq=8 * hkv, Hkv=hkv, bt=bt, seed=17,
                                        max_batch=len(many))
    pool._scale = scale                         # 0.5: logits of std 5.7, so the maximum moves late
    width = -(-tokens // bt)
    wide = np.pad(tables, ((0, 0), (0, max(0, width - tables.shape[1]))), constant_values=-1)
    got = gpu_decode(pool, 0, q[:, :n], wide[:n, :width].copy(), lens)[0]
    whole = gpu_decode(pool, 0, q, tables, many)[0]
    assert np.array_equal(got.view(np.int64), whole[:n].view(np.int64))
    hot = host_hot(pool, 17, sess, many, tables)
    ref = oracle.paged_decode(hot, q[:, :n].cpu().view(torch.int16).numpy().view(np.uint16),
                              tables[:n], lens, scale, 8 * hkv)
    assert scaled_err(got, ref[0]) <= TOL
    assert pool.check_device() == 0


# Grids of several waves whose splits differ in length start with the longest
# sessions (up to 32 of them): each row once, whatever its rank, ties included.
LONGEST_FIRST = [17003, 20, 17003, 1, 16400, 5000, 64, 17003, 1] + [700 + 37 * (i % 5) for i in range(24)]


@pytest.mark.parametrize("n", [9, 31, 32, 33])
@pytest.mark.parametrize("bt", [16, 64])
def test_longest_first(pkg, n, bt):  # noqa: F811
    lens = LONGEST_FIRST[:n]
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert decode_shape(max(lens), n, bt=bt).by_length == (n <= 32)
    pool, sess, tables, q = direct_case(pkg, lens, L=1, bt=bt, seed=23, max_batch=n)
    got = gpu_decode(pool, 0, q, tables, lens)[0]
    for i in range(n):
        one = gpu_decode(pool, 0, q[:, i:i + 1], tables[i:i + 1], lens[i:i + 1])[0, 0]
        assert np.array_equal(one.view(np.int64), got[i].view(np.int64))
    ref = oracle.paged_decode(host_hot(pool, 23, sess, lens, tables),
                              q.cpu().view(torch.int16).numpy().view(np.uint16), tables, lens,
                              1 / math.sqrt(128), 32)
    assert scaled_err(got, ref[0]) <= TOL
    assert pool.check_device() == 0


# Tables of one split run kernels of their own, at 1, 2 and 3 CTAs per SM: the bits are those of
# the same sessions in tables of two splits.
@pytest.mark.parametrize("n", [9, 45, 99])
@pytest.mark.parametrize("bt,hkv", [(16, 4), (64, 4), (16, 1)])
def test_tables_of_one_split(pkg, n, bt, hkv):  # noqa: F811
    lens = ([1, 15, 16, 17, 127, 128, 129, 1023, 1024] * 11)[:n]
    pool, sess, tables, q = direct_case(pkg, lens, L=2, Hq=8 * hkv, Hkv=hkv, bt=bt, seed=19,
                                        max_batch=4 * n)
    pool._scale = 0.5
    wide = np.pad(tables, ((0, 0), (0, tables.shape[1])), constant_values=-1)
    got = gpu_decode(pool, -1, q, tables, lens)
    assert np.array_equal(got.view(np.int64), gpu_decode(pool, -1, q, wide, lens).view(np.int64))
    ref = oracle.paged_decode(host_hot(pool, 19, sess, lens, tables),
                              q.cpu().view(torch.int16).numpy().view(np.uint16), tables, lens, 0.5,
                              8 * hkv)
    assert scaled_err(got, ref) <= TOL
    t = torch.as_tensor(tables, device="cuda")
    s = torch.as_tensor(np.asarray(lens, dtype=np.int32), device="cuda")
    out = torch.empty(2, n, 8 * hkv, 128, device="cuda")
    for l in range(2):
        pool.decode_attention(l, q[l].contiguous(), t, s, n, t.shape[1], 0.5, out[l], overlap_previous=l > 0)
    torch.cuda.synchronize()
    assert np.array_equal(out.double().cpu().numpy().view(np.int64), got.view(np.int64))
    assert pool.check_device() == 0


@pytest.mark.parametrize("n", [9, 32])
@pytest.mark.parametrize("bt", [16, 64])
@pytest.mark.parametrize("bf16", [False, True])
def test_longest_first_fused_layers(pkg, n, bt, bf16):  # noqa: F811
    """The same with each row's newest token from k_new and v_new, in overlapped calls layer by
    layer: rows of k_new, v_new and out are the batch's, whatever their rank in the grid."""
    L, lens = 3, LONGEST_FIRST[:n]
    pool, _, tables, q = direct_case(pkg, lens, L=L, bt=bt, seed=29, max_batch=n)
    want = torch.from_numpy(np.concatenate([gpu_decode(pool, l, q, tables, lens) for l in range(L)]))
    hot = pool.hot_view()
    at = torch.as_tensor([int(tables[b, (t - 1) // bt]) for b, t in enumerate(lens)], device="cuda")
    slot = torch.as_tensor([(t - 1) % bt for t in lens], device="cuda")
    new = hot[at, :, :, :, slot].clone()                   # [B][L][K|V][Hkv][D]
    k_new, v_new = (new[:, :, i].transpose(0, 1).contiguous() for i in (0, 1))
    before = pool.hot.clone()
    hot[at, :, :, :, slot] = float("nan")
    t = torch.as_tensor(tables, device="cuda")
    s = torch.as_tensor(np.asarray(lens, dtype=np.int32), device="cuda")
    out = torch.empty(L, n, 32, 128, dtype=torch.bfloat16 if bf16 else torch.float32, device="cuda")
    for l in range(L):
        pool.decode_append_attention(l, q[l], k_new[l], v_new[l], t, s, n, t.shape[1],
                                     1 / math.sqrt(128), out[l], overlap_previous=l > 0)
    torch.cuda.synchronize()
    assert torch.equal(out.cpu(), want.float().to(out.dtype))
    assert torch.equal(pool.hot.view(torch.int16), before.view(torch.int16))
    assert pool.check_device() == 0

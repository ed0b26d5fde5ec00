"""Splits shared by several CTAs, the launch shape of small decode grids.

A grid that would leave SMs idle gives each split to 2, 4 or 8 CTAs, whose
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
from test_gpu_parity import TOL, direct_case, gpu_decode, host_hot, pkg, scaled_err  # noqa: F401

pytestmark = pytest.mark.gpu


def ctas(lens, bt=16, Hkv=4):
    """CTAs of the unshared grid: splits for the table width x kv-heads x rows."""
    from paper_2609_25782_gb300 import kvtier
    return kvtier.kv_decode_splits(-(-max(lens) // bt) * bt) * Hkv * len(lens)


# (lengths of one call, CTAs that share a split on a GPU of 128 to 159 SMs)
@pytest.mark.parametrize("lens,shared", [
    ([1], 8), ([16], 8), ([17], 8), ([127], 8), ([129], 8), ([1024], 8), ([1025], 8),
    ([4096], 8), ([4097], 4), ([8192], 4), ([8193], 4), ([9300], 2), ([16384], 2), ([16391], 2), ([19000], 2),
    ([1024] * 8, 4), ([2048, 1, 1025, 700], 4), ([33, 1023, 15, 1040], 4), ([3000, 2049] * 2, 2),
])
@pytest.mark.parametrize("bt,scale", [(16, 1 / math.sqrt(128)), (64, 0.5)])
def test_shared_splits(pkg, lens, shared, bt, scale):  # noqa: F811
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if 128 <= sms < 160:
        assert shared * ctas(lens, bt) <= sms and (shared == 8 or 2 * shared * ctas(lens, bt) > sms)
    n = len(lens)
    many = lens + [100] * (160 // n)            # a batch with at least 160 CTAs shares nothing
    pool, sess, tables, q = direct_case(pkg, many, L=1, bt=bt, seed=17, max_batch=len(many))
    pool._scale = scale                         # 0.5: logits of std 5.7, so the maximum moves late
    width = -(-max(lens) // bt)
    got = gpu_decode(pool, 0, q[:, :n], tables[:n, :width].copy(), lens)[0]
    whole = gpu_decode(pool, 0, q, tables, many)[0]
    assert np.array_equal(got.view(np.int64), whole[:n].view(np.int64))
    hot = host_hot(pool, 17, sess, many, tables)
    ref = oracle.paged_decode(hot, q[:, :n].cpu().view(torch.int16).numpy().view(np.uint16),
                              tables[:n], lens, scale, 32)
    assert scaled_err(got, ref[0]) <= TOL
    assert pool.check_device() == 0

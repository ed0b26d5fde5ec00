"""Launch rules of the kernels as host functions of sizes, without a GPU."""
import random

import pytest

from launch_rules import decode_shape, pool_part_rows, rules, splits_of


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


# (tokens, batch, further sizes) -> CTAs that share a split, CTAs per SM, tiles in flight before
# the previous call ends (overlapped), merge in the split kernel, one split, longest first,
# combine; at 152 SMs. Each side of every line that the rule draws.
SHAPES = [
    # tables of one split: 8 warps per CTA up to one CTA per SM, then 2 or 3 per SM by the last wave
    ((1024, 1, {}), (1, 1, 0, 0, 1, 0, 0)), ((1024, 38, {}), (1, 1, 0, 0, 1, 0, 0)),
    ((1024, 39, {}), (1, 2, 0, 0, 1, 0, 0)), ((1024, 76, {}), (1, 2, 0, 0, 1, 0, 0)),
    ((1024, 77, {}), (1, 3, 0, 0, 1, 0, 0)), ((1024, 116, {}), (1, 2, 0, 0, 1, 0, 0)),
    ((1024, 400, {}), (1, 3, 0, 4, 1, 0, 0)),
    # 8 CTAs share a split up to two per SM, one per kv-head, split and session
    ((1040, 1, {}), (8, 2, 0, 0, 0, 0, 1)), ((9728, 1, {}), (2, 1, 2, 0, 0, 0, 1)),
    ((9216, 1, {}), (8, 2, 0, 0, 0, 0, 1)), ((2048, 4, {}), (8, 2, 0, 0, 0, 0, 1)),
    ((2048, 5, {}), (2, 1, 2, 0, 0, 0, 1)),
    # 2 CTAs: up to one, two and three per SM
    ((2048, 9, {}), (2, 1, 2, 0, 0, 0, 1)), ((2048, 10, {}), (2, 2, 1, 0, 0, 0, 1)),
    ((2048, 19, {}), (2, 2, 1, 0, 0, 0, 1)), ((2048, 20, {}), (2, 3, 1, 0, 0, 0, 1)),
    ((2048, 28, {}), (2, 3, 1, 0, 0, 0, 1)), ((2048, 29, {}), (1, 2, 1, 0, 0, 0, 1)),
    ((2048, 38, {}), (1, 2, 1, 0, 0, 0, 1)), ((2048, 39, {}), (1, 3, 0, 0, 0, 0, 1)),
    # more than 16 splits: shared up to two per SM, never paced unshared
    ((40000, 1, {}), (2, 2, 1, 0, 0, 0, 1)), ((77824, 1, {}), (2, 2, 1, 0, 0, 0, 1)),
    ((79872, 1, {}), (1, 2, 0, 0, 0, 0, 1)),
    # at least 8 CTAs per SM: up to four splits merge in the split kernel, and no wider table
    # means no combine
    ((4096, 75, {}), (1, 2, 0, 0, 0, 0, 1)), ((4096, 76, {}), (1, 2, 0, 4, 0, 0, 0)),
    ((5120, 76, {}), (1, 2, 0, 4, 0, 0, 1)),
    # the longest sessions first: 2 to 32 of them, one layer, splits of unequal length
    ((17408, 9, {}), (1, 2, 0, 0, 0, 1, 1)), ((32768, 32, {}), (1, 3, 0, 4, 0, 1, 1)),
    ((32768, 33, {}), (1, 3, 0, 4, 0, 0, 1)), ((16384, 16, {}), (1, 3, 0, 0, 0, 0, 1)),
    ((32768, 16, dict(layers=2)), (1, 3, 0, 4, 0, 0, 1)),
]


@pytest.mark.parametrize("case,want", SHAPES)
def test_decode_shape(case, want):
    tokens, batch, kw = case
    sub, per_sm, pace, merge, one, first, combine = want
    for overlap in (False, True):
        d = decode_shape(tokens, batch, overlap=overlap, **kw)
        assert (d.sub, d.per_sm, d.merge_max, d.one_split, d.by_length, d.combine) == \
            (sub, per_sm, merge, one, first, combine)
        assert d.pace == (pace if overlap else 0)
        # the kernels that carry the pacing
        assert not d.pace or d.sub == 2 or ((d.sub, d.per_sm) == (1, 2) and not d.one_split and not d.by_length)
        assert d.wide == (splits_of(tokens) > 16)


def drawn_call(rng):
    hkv, group = rng.choice([1, 2, 4, 8]), rng.choice([1, 2, 4, 8])
    return dict(tokens=int(2 ** rng.uniform(4, 17)), batch=int(2 ** rng.uniform(0, 6)),
                bt=rng.choice([16, 64]), hq=hkv * group, hkv=hkv, layers=rng.choice([1, 1, 2, 48]),
                sms=rng.choice([132, 148, 152]), overlap=rng.random() < 0.5)


def rows_of(c):
    return c["layers"] * c["batch"] * c["hq"] * splits_of(-(-c["tokens"] // c["bt"]) * c["bt"])


def test_decode_shape_keeps_to_the_workspace():
    """Whatever room there is beyond the unshared rows, a shared call's rows fit it, and with none
    no split is shared."""
    rng = random.Random(5)
    shared = set()
    for _ in range(4000):
        c = drawn_call(rng)
        tokens, batch = c.pop("tokens"), c.pop("batch")
        rows = rows_of(dict(c, tokens=tokens, batch=batch))
        for room in (rows, 2 * rows - 1, 2 * rows, 8 * rows - 1, 8 * rows):
            d = decode_shape(tokens, batch, part_rows=room, **c)
            assert d.sub * rows <= room          # 2 or 8 rows of a shared split
            assert not d.pace or d.sub == 2 or ((d.sub, d.per_sm) == (1, 2) and not d.one_split
                                                and not d.by_length)
            shared.add((room // rows, d.sub))
    assert shared == {(1, 1), (2, 1), (2, 2), (7, 1), (7, 2), (8, 1), (8, 2), (8, 8)}


def test_pool_has_room_for_every_shared_call():
    """A call that a pool accepts shares its splits as with unlimited room."""
    rng = random.Random(6)
    for _ in range(4000):
        c = drawn_call(rng)
        tokens, batch = c.pop("tokens"), c.pop("batch")
        table = -(-tokens // c["bt"]) * c["bt"]
        context = int(table * 2 ** rng.uniform(0, 4))
        least = -(-rows_of(dict(c, tokens=tokens, batch=batch)) // (c["hq"] * splits_of(context)))
        have = pool_part_rows(least + rng.choice([0, 0, 3]), context, c["hq"], c["hkv"], c["sms"])
        assert decode_shape(tokens, batch, part_rows=have, **c) == decode_shape(tokens, batch, **c)

"""Timed cases of the hot/cold KV path, through the package's public entry points.

Each case is one thing a serving program has the library do, at one size:

decode     one decode step over sessions at scattered physical blocks: one layer's call by
           itself, the layers' calls in turn (direct, or replayed from a CUDA graph as a serving
           engine replays its decode steps), the same with the step's new token written by the
           decode kernel, or every layer in one call
resume     paused sessions brought back into the hot pool while others leave it (a tool call
           returns, another session waits): cold image -> hot blocks and the batch's tables
turn       a session's context is written, then the session is paused: append and pack
residency  the block-residency pool: a new session's context pushes another session's blocks out,
           the batch of that session then fetches them back (and evicts, writing the new image)

Shapes are the repository's: head_dim 128, 32 query and 4 KV heads, 48 layers (96 KiB of bf16
K and V per token), 16- or 64-token blocks, contexts from a few hundred to 128K tokens.
"""
import math

import numpy as np
import torch

from paper_2609_25782_gb300 import Pool

D = 128


def _case(name, kind, **kw):
    c = {"name": name, "kind": kind, "layers": 48, "hq": 32, "hkv": 4, "bt": 16}
    c.update(kw)
    return c


def listed():
    return [
        # one layer's attention for four short chats: the smallest call, latency and host count
        _case("layer_4x512-2k", "decode", mode="layer", layers=1, batch=4, tmin=512, tmax=2048,
              q_std=1.0, lens_seed=1),
        # a single agent's decode step early in its task; peaked scores, as trained heads have
        _case("step_1x3k", "decode", mode="graph", batch=1, tmin=3001, tmax=3001, q_std=4.0,
              lens_seed=2),
        # a single agent at the paper's mean context
        _case("step_1x16k", "decode", mode="graph", batch=1, tmin=16391, tmax=16391, q_std=1.0,
              lens_seed=3),
        # a single agent with a very long context, 64-token blocks
        _case("step_1x100k_bt64", "decode", mode="graph", bt=64, batch=1, tmin=100003,
              tmax=100003, q_std=1.0, lens_seed=4),
        # a small batch whose new tokens are written by the decode kernel itself
        _case("fused_8x2k-6k", "decode", mode="fused", layers=16, batch=8, tmin=2048, tmax=6144,
              q_std=2.0, lens_seed=5),
        # the agentic trace's batch: 16 decoding sessions of very unequal lengths, bf16 outputs
        _case("step_16x2k-30k", "decode", mode="calls", batch=16, tmin=2048, tmax=30000,
              q_std=1.0, out="bf16", lens_seed=6),
        # the headline decode step: 32 sessions of 8K-32K tokens, all 48 layers
        _case("step_32x8k-32k", "decode", mode="calls", batch=32, tmin=8192, tmax=32768,
              q_std=1.0, lens_seed=7),
        # many short sessions, every layer in one call, 8 KV heads in groups of 4
        _case("all_96x200-3k_bt64", "decode", mode="all", layers=12, hkv=8, bt=64, batch=96,
              tmin=200, tmax=3000, q_std=1.0, lens_seed=8),
        # one short session leaves for a tool call, another comes back
        _case("resume_1x2k", "resume", batch=1, tmin=2100, tmax=2100, lens_seed=9),
        # several long sessions come back at once
        _case("resume_3x12k-32k", "resume", batch=3, tmin=12000, tmax=32768, lens_seed=10),
        # one turn's context (a tool result or a user message) is appended, then the pause packs it
        _case("turn_1x1536", "turn", batch=1, tmin=1536, tmax=1536, lens_seed=11),
        # block residency under pressure: one arriving session against four of the running batch
        _case("residency_4x2k-6k", "residency", batch=4, tmin=2048, tmax=6144, new=5000,
              lens_seed=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: at most 24 GB of KV, so never above the largest."""
    kind = rng.choice(["decode"] * 6 + ["resume", "resume", "turn", "turn", "residency"])
    hkv, hq = rng.choice([(4, 32), (4, 32), (4, 32), (8, 32), (4, 16), (8, 64), (2, 16)])
    c = {"kind": kind, "hq": hq, "hkv": hkv, "bt": rng.choice([16, 16, 64]),
         "layers": rng.choice([4, 16, 28, 48]), "lens_seed": rng.randrange(1 << 20)}
    if kind == "decode":
        c["mode"] = rng.choice(["layer", "graph", "graph", "fused", "calls", "all"])
        if c["mode"] == "layer":
            c["layers"] = 1
        c["out"] = rng.choice(["fp32", "fp32", "bf16"])
        c["q_std"] = rng.choice([1.0, 2.0, 4.0])
        limit, tmax, bmax = (4e9 if c["mode"] == "fused" else 24e9), 131072, 128
    else:
        limit, tmax, bmax = (6e9 if kind == "resume" else 2e9), 32768, 8
    c["tmax"] = _log_int(rng, 200, tmax)
    c["tmin"] = min(c["tmax"], _log_int(rng, 200, c["tmax"])) if rng.random() < 0.7 else c["tmax"]
    token = _token_bytes(c)
    most = max(1, min(bmax, int(limit / (c["tmax"] * token))))
    c["batch"] = _log_int(rng, 1, most)
    if c["tmax"] * token > limit:       # one long session of a wide model: fewer layers
        c["layers"] = max(1, int(c["layers"] * limit / (c["tmax"] * token)))
    if kind == "residency":
        c["new"] = rng.randint(max(1, c["tmin"] // 2), sum(_lengths(c)))
    return c


# ---- sizes ---------------------------------------------------------------------------------

def _token_bytes(c):
    return c["layers"] * 2 * c["hkv"] * D * 2


def _lengths(c):
    """The sessions' lengths: uniform in [tmin, tmax], the same for every seed of the values."""
    r = np.random.RandomState(c["lens_seed"])
    return [int(x) for x in r.randint(c["tmin"], c["tmax"] + 1, c["batch"])]


def _blocks(t, bt):
    return -(-t // bt)


def work(c):
    lens, tok = _lengths(c), _token_bytes(c)
    n = sum(lens)
    if c["kind"] == "decode":
        rows = c["layers"] * c["batch"] * c["hq"] * D
        b = n * tok + rows * 2 + rows * (2 if c.get("out") == "bf16" else 4)
        if c["mode"] == "fused":        # the new tokens: read once, written once to the pool
            b += c["batch"] * tok
        return {"bytes": b, "flops": 4 * n * c["layers"] * c["hq"] * D}
    if c["kind"] == "resume":           # both groups: image read, blocks written
        return {"bytes": 2 * 2 * n * tok}
    if c["kind"] == "turn":             # k and v read, blocks written; blocks read, image written
        return {"bytes": 4 * n * tok}
    back = min(c["new"] + c["bt"] - 1, n)     # residency: about as many tokens leave and return
    return {"bytes": (4 * c["new"] + 2 * back) * tok}


# ---- inputs --------------------------------------------------------------------------------

def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)


def _fill(t, seed, salt, std=1.0):
    """N(0, std) values in place, from the seed alone; large buffers in pieces."""
    g, flat, piece = _gen(seed, salt), t.view(-1), 1 << 30
    for i in range(0, flat.numel(), piece):
        flat[i:i + piece].normal_(0.0, std, generator=g)
    return t


def _normal(shape, seed, salt, std=1.0):
    return _fill(torch.empty(shape, dtype=torch.bfloat16, device="cuda"), seed, salt, std)


def _placement(c, seed):
    """Decode: each session's blocks at random places of the hot arena."""
    lens, bt = _lengths(c), c["bt"]
    width = max(_blocks(t, bt) for t in lens)
    perm = np.random.RandomState(seed & 0x7FFFFFFF).permutation(sum(_blocks(t, bt) for t in lens))
    tab = np.full((len(lens), width), -1, dtype=np.int32)
    at = 0
    for i, t in enumerate(lens):
        tab[i, :_blocks(t, bt)] = perm[at:at + _blocks(t, bt)]
        at += _blocks(t, bt)
    return lens, tab


def _query_shape(c):
    return (c["layers"], c["batch"], c["hq"], D)


def _prepare_decode(c, seed):
    lens, tab = _placement(c, seed)
    calls = c["layers"] if c["mode"] == "all" else 1
    pool = Pool(num_layers=c["layers"], num_hot_blocks=int((tab >= 0).sum()), cold_bytes=256,
                num_q_heads=c["hq"], num_kv_heads=c["hkv"], block_tokens=c["bt"], max_sessions=1,
                max_batch=calls * c["batch"], max_context=max(lens))
    _fill(pool.hot, seed, 1)
    dtype = torch.bfloat16 if c.get("out") == "bf16" else torch.float32
    s = {"case": c, "pool": pool, "tables": torch.from_numpy(tab).cuda(),
         "lens": torch.tensor(lens, dtype=torch.int32, device="cuda"), "width": tab.shape[1],
         "q": _normal(_query_shape(c), seed, 2, c["q_std"]),
         "out": torch.zeros(_query_shape(c), dtype=dtype, device="cuda")}
    if c["mode"] == "fused":
        shape = (c["layers"], c["batch"], c["hkv"], D)
        s["k_new"], s["v_new"] = _normal(shape, seed, 3), _normal(shape, seed, 4)
    if c["mode"] in ("graph", "fused"):
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _layer_calls(s)             # the step once, then recorded
            g = torch.cuda.CUDAGraph()
            g.capture_begin()
            _layer_calls(s)
            g.capture_end()
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = g
    return s


def _layer_calls(s):
    """The decode step of a model: each layer's attention in turn, layer l > 0 allowed to start
    its reads while layer l - 1's call drains."""
    c, pool, st = s["case"], s["pool"], torch.cuda.current_stream()
    for l in range(c["layers"]):
        if c["mode"] == "fused":
            pool.decode_append_attention(l, s["q"][l], s["k_new"][l], s["v_new"][l], s["tables"],
                                         s["lens"], c["batch"], s["width"], 1 / math.sqrt(D),
                                         s["out"][l], st, overlap_previous=l > 0)
        else:
            pool.decode_attention(l, s["q"][l], s["tables"], s["lens"], c["batch"], s["width"],
                                  1 / math.sqrt(D), s["out"][l], st, overlap_previous=l > 0)


def _run_decode(s):
    c = s["case"]
    if c["mode"] in ("graph", "fused"):
        s["graph"].replay()
    elif c["mode"] == "calls":
        _layer_calls(s)
    else:                               # one call: the only layer, or all of them
        layer = 0 if c["mode"] == "layer" else -1
        s["pool"].decode_attention(layer, s["q"], s["tables"], s["lens"], c["batch"], s["width"],
                                   1 / math.sqrt(D), s["out"], torch.cuda.current_stream())
    # the fused step also writes the tokens into the hot arena
    return [s["out"], s["pool"].hot] if c["mode"] == "fused" else [s["out"]]


def _session_pool(c, seed, hot_blocks, images, lru=False):
    cap = sum(-(-t * _token_bytes(c) // 256) * 256 for t in images)
    pool = Pool(num_layers=c["layers"], num_hot_blocks=hot_blocks, cold_bytes=cap,
                num_q_heads=c["hq"], num_kv_heads=c["hkv"], block_tokens=c["bt"],
                max_sessions=len(images), max_batch=c["batch"], max_context=max(images),
                alloc_seed=int(seed), lru_residency=lru)
    pool.hot.zero_()
    return pool


def _batch_state(c, pool, sids, lens):
    width = max(_blocks(t, c["bt"]) for t in lens)
    return {"case": c, "pool": pool, "sids": sids, "width": width,
            "tables": torch.zeros(len(lens), width, dtype=torch.int32, device="cuda"),
            "lens": torch.zeros(len(lens), dtype=torch.int32, device="cuda")}


def _prepare_resume(c, seed):
    """Two groups of sessions of the same lengths, the hot pool as large as one of them."""
    lens = _lengths(c)
    pool = _session_pool(c, seed, sum(_blocks(t, c["bt"]) for t in lens), lens + lens)
    _fill(pool.cold, seed, 5)
    away = [pool.session_create_paused(t, t) for t in lens]
    sids = [pool.session_create_paused(t, t) for t in lens]
    st = torch.cuda.current_stream()
    for sid in sids:
        pool.session_resume(sid, st)
    s = _batch_state(c, pool, sids, lens)
    s["away"] = away
    return s


def _run_resume(s):
    pool, st = s["pool"], torch.cuda.current_stream()
    for out, back in ((s["sids"], s["away"]), (s["away"], s["sids"])):
        for sid in reversed(out):       # nothing new since the resume: the pause writes nothing
            pool.session_pause(sid, st)
        for sid in back:
            pool.session_resume(sid, st)
    pool.batch_tables(s["sids"], s["tables"], s["width"], s["lens"], st)
    return [pool.hot, s["tables"], s["lens"]]


def _new_kv(c, n, seed, salt):
    return (_normal((c["layers"], n, c["hkv"], D), seed, salt),
            _normal((c["layers"], n, c["hkv"], D), seed, salt + 1))


def _prepare_turn(c, seed):
    lens = _lengths(c)
    pool = _session_pool(c, seed, sum(_blocks(t, c["bt"]) for t in lens), lens)
    pool.cold.zero_()
    return {"case": c, "pool": pool, "lens": lens,
            "sids": [pool.session_create(t) for t in lens],
            "kv": [_new_kv(c, t, seed, 10 + 2 * i) for i, t in enumerate(lens)]}


def _run_turn(s):
    pool, st = s["pool"], torch.cuda.current_stream()
    for sid in s["sids"]:               # the sessions of the pass before have ended
        pool.session_destroy(sid)
    s["sids"] = [pool.session_create(t) for t in s["lens"]]
    for sid, (k, v) in zip(s["sids"], s["kv"]):
        pool.session_append(sid, k, v, st)
    for sid in s["sids"]:
        pool.session_pause(sid, st)
    return [pool.image(sid) for sid in s["sids"]]


def _prepare_residency(c, seed):
    """A running batch that fills the hot pool, and the context of a session about to arrive."""
    lens = _lengths(c)
    pool = _session_pool(c, seed, sum(_blocks(t, c["bt"]) for t in lens), [c["new"]] + lens, True)
    _fill(pool.cold, seed, 5)
    new = pool.session_create(c["new"])
    sids = [pool.session_create_paused(t, t) for t in lens]
    st = torch.cuda.current_stream()
    for sid in sids:
        pool.session_resume(sid, st)
    s = _batch_state(c, pool, sids, lens)
    s["new"], s["kv"] = new, _new_kv(c, c["new"], seed, 10)
    pool.batch_tables(sids, s["tables"], s["width"], s["lens"], st)
    return s


def _run_residency(s):
    pool, st = s["pool"], torch.cuda.current_stream()
    pool.session_destroy(s["new"])
    s["new"] = pool.session_create(s["case"]["new"])
    pool.session_append(s["new"], s["kv"][0], s["kv"][1], st)
    pool.batch_tables(s["sids"], s["tables"], s["width"], s["lens"], st)
    return [pool.image(s["new"]), pool.hot, s["tables"], s["lens"]]


_PREPARE = {"decode": _prepare_decode, "resume": _prepare_resume, "turn": _prepare_turn,
            "residency": _prepare_residency}
_RUN = {"decode": _run_decode, "resume": _run_resume, "turn": _run_turn,
        "residency": _run_residency}


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def run(state):
    return _RUN[state["case"]["kind"]](state)


# ---- what another correct implementation gives ----------------------------------------------

def tolerance(c):
    """Migrations move bytes. A decode output keeps K, V, the scores and the sums as they are and
    has its softmax weights in bf16 for the product with V: against 64 bits it was off by 1.6e-3 of
    its norm (less with peaked scores) at every length, and by 2.3e-3 with outputs in bf16.
    Stated is four times that."""
    if c["kind"] != "decode":
        return "exact"
    return {"rel": 9.2e-3 if c.get("out") == "bf16" else 6.4e-3}


def _pops(n, seed):
    """The order in which blocks leave a new pool's free list: 0..n-1 shuffled from the top by
    splitmix64 draws, taken from its end."""
    mask, st, v = (1 << 64) - 1, int(seed) & ((1 << 64) - 1), list(range(n))
    for i in range(n - 1, 0, -1):
        st = (st + 0x9E3779B97F4A7C15) & mask
        z = st
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        z ^= z >> 31
        j = (z * (i + 1)) >> 64
        v[i], v[j] = v[j], v[i]
    return v[::-1]


def _exact_tables(c, seed):
    """Where the batch's blocks are: popped session by session from the new pool's free list."""
    lens, bt = _lengths(c), c["bt"]
    pops = _pops(sum(_blocks(t, bt) for t in lens), seed)
    tab = np.full((len(lens), max(_blocks(t, bt) for t in lens)), -1, dtype=np.int32)
    at = 0
    for i, t in enumerate(lens):
        tab[i, :_blocks(t, bt)] = pops[at:at + _blocks(t, bt)]
        at += _blocks(t, bt)
    return lens, tab, pops


def _place(hot, c, image, blocks, t):
    """An image [L][2][Hkv][t][D] into its blocks of hot [NB][L][2][Hkv][bt][D]."""
    bt = c["bt"]
    full = t // bt
    idx = torch.as_tensor(np.asarray(blocks[:_blocks(t, bt)], dtype=np.int64), device="cuda")
    if full:
        hot[idx[:full]] = image[:, :, :, :full * bt].unflatten(3, (full, bt)) \
            .permute(3, 0, 1, 2, 4, 5)
    if t > full * bt:
        hot[idx[full], :, :, :, :t - full * bt] = image[:, :, :, full * bt:]


def _images(c, seed, sizes):
    """The cold arena filled as `prepare` fills it, as one image per size."""
    per = c["layers"] * 2 * c["hkv"] * D
    cap = [-(-t * per * 2 // 256) * 128 for t in sizes]
    cold = _fill(torch.empty(max(sum(cap), 128), dtype=torch.bfloat16, device="cuda"), seed, 5)
    at = np.concatenate([[0], np.cumsum(cap)])
    return [cold[at[i]:at[i] + per * t].view(c["layers"], 2, c["hkv"], t, D)
            for i, t in enumerate(sizes)]


def _exact_decode(c, seed):
    lens, tab = _placement(c, seed)
    nb, L, hkv, bt, hq = int((tab >= 0).sum()), c["layers"], c["hkv"], c["bt"], c["hq"]
    hot = _fill(torch.empty(nb * L * 2 * hkv * bt * D, dtype=torch.bfloat16, device="cuda"),
                seed, 1).view(nb, L, 2, hkv, bt, D)
    q = _normal(_query_shape(c), seed, 2, c["q_std"]).view(L, c["batch"], hkv, hq // hkv, D)
    out = torch.empty(L, c["batch"], hkv, hq // hkv, D, dtype=torch.float64, device="cuda")
    for b, t in enumerate(lens):
        idx = torch.as_tensor(tab[b, :_blocks(t, bt)].astype(np.int64), device="cuda")
        if c["mode"] == "fused":
            shape = (L, c["batch"], hkv, D)
            at = hot[int(tab[b, _blocks(t, bt) - 1]), :, :, :, (t - 1) % bt]
            at[:, 0] = _normal(shape, seed, 3)[:, b]
            at[:, 1] = _normal(shape, seed, 4)[:, b]
        for l in range(L):
            k, v = (hot[idx, l, i].transpose(0, 1).reshape(hkv, -1, D)[:, :t].double()
                    for i in (0, 1))
            p = torch.softmax(q[l, b].double() @ k.transpose(1, 2) / math.sqrt(D), dim=-1)
            out[l, b] = p @ v
    out = out.view(_query_shape(c))
    return [out, hot.view(-1)] if c["mode"] == "fused" else [out]


def exact(c, seed):
    if c["kind"] == "decode":
        return _exact_decode(c, seed)
    bt, L, hkv = c["bt"], c["layers"], c["hkv"]
    if c["kind"] == "turn":
        return [torch.stack(_new_kv(c, t, seed, 10 + 2 * i), 1).transpose(2, 3).contiguous()
                for i, t in enumerate(_lengths(c))]
    lens, tab, pops = _exact_tables(c, seed)
    hot = torch.zeros(len(pops), L, 2, hkv, bt, D, dtype=torch.bfloat16, device="cuda")
    tables = [torch.from_numpy(tab).cuda(), torch.tensor(lens, dtype=torch.int32, device="cuda")]
    if c["kind"] == "resume":   # the other group's session had the same blocks, last one first
        images, first = _images(c, seed, lens + lens), []
        for i, t in enumerate(lens):
            _place(hot, c, images[i], tab[i, :_blocks(t, bt)][::-1], t)
        images = images[len(lens):]
    else:       # the arriving session takes the batch's first blocks, last one first; they go back
        images = _images(c, seed, [c["new"]] + lens)[1:]
        k, v = _new_kv(c, c["new"], seed, 10)
        new = torch.stack((k, v), 1).transpose(2, 3).contiguous()
        n = _blocks(c["new"], bt)
        _place(hot, c, new, pops[:n][::-1], c["new"])
        first = [new]
    for i, t in enumerate(lens):
        _place(hot, c, images[i], tab[i], t)
    return first + [hot.view(-1)] + tables

"""The measured cases of the ValueDiff eviction library: what they are, how
their inputs are made, how one pass runs and what its outputs must be.

A pass is one call (or, in the two-call form, the append and the eviction) of
the Python binding on a cache that is held at its budget, as a serving loop
makes it: a block boundary of block prompt processing, a decode step, or a
score / dispersion read-out.  A state holds several caches (sequences served
in turn) and a pool of new blocks or tokens, so that repeated passes keep
seeing rows that a cache has not seen before; pass i takes cache i mod G.

Fields of a case: ``op`` (block, decode, score), the shape of the cache,
``N`` / ``B`` budget and appended rows, ``spare`` slots beyond N + B,
``variant``, ``mu`` (running or recompute), ``fused`` (append inside the
eviction call, or vd_append before it), ``holefill`` layout, ``ragged``
(per-sequence budgets through N_dev), ``keys`` / ``attn`` / ``sigma`` /
``scores`` (the scoring options and optional outputs) and ``gen`` (the value
distribution).
"""
from __future__ import annotations

import math

import torch

import paper_2609_23314_gb300 as vd

VARIANT = {"l2": vd.VD_SCORE_L2, "dir": vd.VD_SCORE_DIR, "norm": vd.VD_SCORE_NORM}
BASE = dict(op="block", n_seq=1, n_layer=1, n_kv_head=8, head_dim=128, N=2048, B=128, spare=0,
            variant="l2", mu="running", fused=True, holefill=False, ragged=False, keys=False,
            attn=False, sigma=False, scores=False, gen="gauss_outlier")


def _case(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # the smallest block-processing step: two heads, budget 128, blocks of 32 (launch latency)
        _case("block_tiny", n_kv_head=2, head_dim=64, N=128, B=32),
        # an engine that evicts layer by layer: the 8 KV heads of one layer, budget 2048
        _case("block_layer"),
        # block prompt processing of an 8B-class GQA model, all 36 layers in one call
        _case("block_gqa", n_layer=36),
        # the same model with the mean recomputed at every event and the append as a call of its own
        _case("block_gqa_recompute", n_layer=36, mu="recompute", fused=False),
        # block prompt processing of a wide-head model, budget 4096, heavy-tailed value norms
        _case("block_wide", n_layer=42, head_dim=256, N=4096, B=256, gen="student_t"),
        # the same step in the layout that only refills the evicted slots
        _case("holefill_block_wide", n_layer=42, head_dim=256, N=4096, B=256, gen="student_t",
              holefill=True),
        # one user's decode step: one token in, one out, in each of 32 x 8 heads
        _case("decode_one", op="decode", n_layer=32, N=4096, B=1, gen="drift"),
        # batched decode of 64 sequences (the largest case: 34 GB of cache)
        _case("decode_batched", op="decode", n_seq=64, n_layer=32, N=4096, B=1, gen="drift"),
        # long generations of different lengths, each with a budget of its own, hole-fill layout
        _case("holefill_decode_ragged", op="decode", n_seq=16, n_layer=28, n_kv_head=4, N=4224,
              B=1, holefill=True, ragged=True, gen="two_cluster"),
        # the direction-only rule at a block boundary
        _case("block_dir", n_layer=36, variant="dir"),
        # several ragged prompts, a head dim that is no power of two, attention weights and sigma
        _case("block_options_odd", n_seq=3, n_layer=24, n_kv_head=6, head_dim=96, N=1000, B=100,
              spare=37, ragged=True, attn=True, sigma=True, mu="recompute"),
        # scores and their dispersion of a whole cache, mean from scratch (analysis of a prompt)
        _case("score_wide", op="score", n_layer=42, head_dim=256, N=4096, B=1, mu="recompute",
              fused=False, sigma=True, scores=True, gen="student_t"),
    ]


def _cache_bytes(c):
    return 4 * c["n_seq"] * c["n_layer"] * c["n_kv_head"] * _capacity(c) * c["head_dim"]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    c = dict(BASE)
    c["op"] = rng.choice(["block", "block", "block", "decode", "decode", "score"])
    c["head_dim"] = rng.choice([64, 80, 96, 128, 128, 128, 192, 256])
    c["N"] = log_int(64, 8192)
    c["B"] = min(c["N"], log_int(8, 512)) if c["op"] == "block" else 1
    c["spare"] = rng.choice([0, 0, 0, log_int(1, 300)])
    c["n_seq"], c["n_layer"], c["n_kv_head"] = log_int(1, 64), log_int(1, 48), log_int(1, 16)
    while _cache_bytes(c) > 4 << 30:  # keep a case well below the largest listed one
        k = max(("n_seq", "n_layer", "n_kv_head"), key=lambda f: c[f])
        c[k] = max(1, c[k] // 2)
    c["variant"] = rng.choice(["l2"] * 7 + ["dir"] * 2 + ["norm"])
    c["mu"] = rng.choice(["running", "running", "recompute"])
    c["gen"] = rng.choice(["gauss_outlier", "student_t", "drift", "two_cluster"])
    if c["op"] == "score":
        c["fused"] = False
        c["keys"] = rng.random() < 0.3
        c["sigma"] = c["variant"] == "l2" and rng.random() < 0.6
        c["scores"] = True
        return c
    c["ragged"] = c["n_seq"] > 1 and rng.random() < 0.5
    c["fused"] = rng.random() < 0.75
    extra = c["op"] == "block" and rng.random() < 0.25
    if extra:
        c["keys"] = rng.random() < 0.4
        c["attn"] = rng.random() < 0.5
        c["sigma"] = c["variant"] == "l2" and rng.random() < 0.5
    c["holefill"] = not extra and rng.random() < 0.3
    c["scores"] = rng.random() < 0.15
    return c


# ---------------------------------------------------------------------------
# sizes
# ---------------------------------------------------------------------------
def _capacity(c):
    return c["N"] + (0 if c["op"] == "score" else c["B"]) + c["spare"]


def _units(c):
    return c["n_seq"] * c["n_layer"] * c["n_kv_head"]


def _budgets(c):
    """Budget (and cached rows) per sequence: N, or 60-100 % of it where ragged."""
    if not c["ragged"]:
        return [c["N"]] * c["n_seq"]
    return [max(1, c["N"] - (s * 7919 % 97) * c["N"] * 4 // 970) for s in range(c["n_seq"])]


def _slots_and_blocks(c):
    """How many caches a state holds, and how many new blocks: 12 GB of caches
    at most, and two budgets and 8192 rows of new tokens where 3 GB hold them."""
    cache = _cache_bytes(c)
    g = max(1, min(128 if cache < 32 << 20 else 16, (12 << 30) // cache))
    if c["op"] == "score":
        return g, 0
    block = 4 * _units(c) * c["B"] * c["head_dim"]
    p = max(8, min(256, max(2 * c["N"], 8192) // c["B"] + 1, (3 << 30) // block))
    return g, p


# ---------------------------------------------------------------------------
# inputs: per unit a random mean, per-token scales or clusters, K with less
# spread than V (the shapes of the value distributions the method is for)
# ---------------------------------------------------------------------------
def _means(c, g, dev):
    U, d = _units(c), c["head_dim"]
    m = torch.randn(U, 1, d, generator=g, device=dev)
    m *= torch.rand(U, 1, 1, generator=g, device=dev) * 1.5 + 0.5
    mk = torch.randn(U, 1, d, generator=g, device=dev)
    ak = math.sqrt(2.0 * d) * 1.4 / (torch.rand(U, 1, 1, generator=g, device=dev) * 2.5 + 1.5)
    return m, mk, ak / math.sqrt(d)


def _fill(c, means, dst_k, dst_v, g, new):
    """Random rows into dst_k, dst_v [U, rows, d] (bf16), some units at a time."""
    m, mk, ak = means
    U, rows, d = dst_v.shape
    dev = dst_v.device
    step = max(1, (64 << 20) // (rows * d))
    kind = c["gen"]
    if kind == "drift" and not new:
        kind = "gauss_outlier"
    for u0 in range(0, U, step):
        sl = slice(u0, min(U, u0 + step))
        n = sl.stop - sl.start
        z = torch.randn(n, rows, d, generator=g, device=dev)
        if kind == "gauss_outlier":
            r = torch.exp(0.5 * torch.randn(n, rows, 1, generator=g, device=dev))
            r = torch.where(torch.rand(n, rows, 1, generator=g, device=dev) < 0.02, r * 8.0, r)
            z *= r
            z += m[sl]
        elif kind == "student_t":
            t = torch.randn(n, rows, 4, generator=g, device=dev)
            chi = t[..., 1:].square().mean(-1, keepdim=True).sqrt()
            z *= (t[..., :1] / chi).abs()
            z += m[sl]
        elif kind == "two_cluster":
            far = torch.rand(n, rows, 1, generator=g, device=dev) < 0.2
            z *= 0.5
            z += torch.where(far, -2.0 * m[sl], 2.0 * m[sl])
        else:  # drift: a mean that has walked some way from the cached rows'
            z += m[sl] + 0.3
        dst_v[sl] = z
        z.normal_(generator=g)
        z *= ak[sl]
        z += mk[sl]
        dst_k[sl] = z


def _inputs(c, seed):
    """The buffers of a state: caches [G, ...], new blocks [P, ...], weights."""
    dev = "cuda"
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    G, P = _slots_and_blocks(c)
    us, d, cap = (c["n_seq"], c["n_layer"], c["n_kv_head"]), c["head_dim"], _capacity(c)
    U = _units(c)
    means = _means(c, g, dev)
    kk = torch.zeros((G,) + us + (cap, d), dtype=torch.bfloat16, device=dev)
    vv = torch.zeros_like(kk)
    for i in range(G):
        _fill(c, means, kk[i].view(U, cap, d), vv[i].view(U, cap, d), g, False)
    kn = torch.empty((P,) + us + (c["B"], d), dtype=torch.bfloat16, device=dev)
    vn = torch.empty_like(kn)
    for i in range(P):
        _fill(c, means, kn[i].view(U, c["B"], d), vn[i].view(U, c["B"], d), g, True)
    attn = None
    if c["attn"]:  # softmax-like weights: positive, below one, summing to about one
        attn = torch.empty(us + (cap,), dtype=torch.float32, device=dev)
        attn.exponential_(generator=g)
        attn /= 4.0 * cap
    return dict(k=kk, v=vv, kn=kn, vn=vn, attn=attn)


# ---------------------------------------------------------------------------
# one state, one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c = case
    x = _inputs(c, seed)
    dev = x["k"].device
    us, d, cap = (c["n_seq"], c["n_layer"], c["n_kv_head"]), c["head_dim"], _capacity(c)
    budgets = _budgets(c)
    n_dev = torch.tensor(budgets, dtype=torch.int32, device=dev) if c["ragged"] else None
    lens = torch.tensor(budgets, dtype=torch.int32, device=dev)
    running = c["mu"] == "running"
    same = len(set(budgets)) == 1

    def rows(t):
        """The cached rows as integers: one view, or one for each sequence where they differ."""
        t = t.view(torch.int16)
        if same:
            return t[:, :, :, :budgets[0]]
        return [t[s, :, :, :b] for s, b in enumerate(budgets)]

    slots = []
    for i in range(x["k"].shape[0]):
        cache = vd.Cache(x["k"][i], x["v"][i], lens.clone())
        s = dict(cache=cache, rs=None, kept=None, evicted=None, scores=None, sigma=None, pos=None)
        if running:
            s["rs"] = torch.zeros(us + (d,), dtype=torch.float64, device=dev)
            vd.vd_running_sum_init_ex(cache, c["keys"], s["rs"])
        if c["op"] == "block":
            s["kept"] = torch.zeros(us + (c["N"],), dtype=torch.int32, device=dev)
        elif c["op"] == "decode":
            s["evicted"] = torch.zeros(us, dtype=torch.int32, device=dev)
        if c["scores"]:
            s["scores"] = torch.zeros(us + (cap,), dtype=torch.float32, device=dev)
        if c["sigma"]:
            s["sigma"] = torch.zeros(us, dtype=torch.float32, device=dev)
        if c["holefill"]:
            pos = torch.arange(cap, dtype=torch.int32, device=dev)
            s["pos"] = pos.expand(us + (cap,)).contiguous()
        out = {f: s[f] for f in ("scores", "sigma") if s[f] is not None}
        if c["op"] != "score":
            out.update(len=cache.len, k=rows(cache.k), v=rows(cache.v),
                       **{f: s[f] for f in ("kept", "evicted") if s[f] is not None})
            if running:
                out["running_sum"] = s["rs"]
            if c["holefill"]:
                out["pos"] = s["pos"][..., :min(budgets)]
        s["out"] = out
        slots.append(s)
    first_new = []
    if c["holefill"]:  # position of the first new row, one row per event of a cache
        start = torch.arange(4096, dtype=torch.int32, device=dev)[:, None] * c["B"]
        first_new = list((start + lens[None, :]).contiguous().unbind(0))
    return dict(case=c, slots=slots, n_dev=n_dev, kn=x["kn"].unbind(0), vn=x["vn"].unbind(0),
                attn=x["attn"], first_new=first_new, step=0, variant=VARIANT[c["variant"]],
                mu=vd.VD_MU_RUNNING if running else vd.VD_MU_RECOMPUTE)


def run(state):
    c, i = state["case"], state["step"]
    state["step"] = i + 1
    s = state["slots"][i % len(state["slots"])]
    cache, var, mu, rs = s["cache"], state["variant"], state["mu"], s["rs"]
    if c["op"] == "score":
        vd.vd_score_ex(cache, var, c["keys"], s["scores"], s["sigma"], mu=mu, running_sum=rs)
        return s["out"]
    event = i // len(state["slots"])
    b = (i + event) % len(state["kn"])
    kn, vn = state["kn"][b], state["vn"][b]
    N, B, n_dev = c["N"], c["B"], state["n_dev"]
    hole = {}
    if c["holefill"]:
        hole = dict(pos=s["pos"], pos_first_new=state["first_new"][event % 4096])
    if not c["fused"]:
        vd.vd_append(cache, kn, vn, B)
    if c["op"] == "decode":
        if c["fused"]:
            vd.vd_append_evict_decode(cache, kn, vn, N, n_dev, var, mu, rs, s["evicted"], None,
                                      s["scores"], **hole)
        elif c["holefill"]:
            vd.vd_evict_decode_holefill(cache, N, hole["pos"], hole["pos_first_new"], n_dev, var,
                                        mu, rs, s["evicted"], None, s["scores"])
        else:
            vd.vd_evict_decode(cache, N, n_dev, var, mu, rs, s["evicted"], None, s["scores"])
    elif c["keys"] or c["attn"] or c["sigma"]:
        if c["fused"]:
            vd.vd_append_evict_block_ex(cache, kn, vn, B, N, n_dev, var, mu, rs, c["keys"],
                                        state["attn"], s["kept"], s["scores"], s["sigma"])
        else:
            vd.vd_evict_block_ex(cache, N, n_dev, B, var, mu, rs, c["keys"], state["attn"],
                                 s["kept"], s["scores"], s["sigma"])
    elif c["fused"]:
        vd.vd_append_evict_block(cache, kn, vn, B, N, n_dev, var, mu, rs, s["kept"], s["scores"],
                                 **hole)
    elif c["holefill"]:
        vd.vd_evict_block_holefill(cache, N, hole["pos"], hole["pos_first_new"], n_dev, B, var,
                                   mu, rs, s["kept"], s["scores"])
    else:
        vd.vd_evict_block(cache, N, n_dev, B, var, mu, rs, s["kept"], s["scores"])
    return s["out"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Scored rows read once; where rows move, the other tensor's moved rows
    read and both tensors' moved rows written once.  Moved rows: a block event
    evicts B + new of N + B rows, so in slot order nearly all of N move; one
    evicted row of a decode step leaves half of them in place on average; the
    hole-fill layout moves about half of the new rows."""
    c = case
    heads, d = c["n_layer"] * c["n_kv_head"], c["head_dim"]
    total = flops = 0
    for n0 in _budgets(c):
        n = n0 + (0 if c["op"] == "score" else c["B"])
        b = n * d * 2
        if c["op"] != "score":
            moved = c["B"] // 2 + 1 if c["holefill"] else n0 if c["op"] == "block" else n0 // 2
            b += 3 * moved * d * 2
            b += 4 * c["N"] if c["op"] == "block" else 4
        if c["mu"] == "running":
            b += d * 8 * (1 if c["op"] == "score" else 2)
        b += 4 * n * (int(c["scores"]) + int(c["attn"])) + 4 * int(c["sigma"])
        total += heads * b
        flops += heads * 4 * n * d
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """Scores, sigma: fp32 arithmetic on exact inputs.  Kept rows and bytes
    are whole numbers and equal, except where two scores at the budget's edge
    lie within rounding of each other: then one unit keeps the other row,
    which shifts its rows between the two slots and changes its running sum
    by the rows' difference."""
    if case["op"] == "score":
        return {"rel": 1e-6}
    return {"rel": 5e-5, "max": 0.05, "differ": 0.005}


# ---------------------------------------------------------------------------
# the first pass of a state in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _scores64(c, x, mean):
    if c["variant"] == "norm":
        return x.square().sum(-1).sqrt()
    if c["variant"] == "l2":
        return (x - mean).square().sum(-1).sqrt()
    nv, nm = x.square().sum(-1).sqrt(), mean.square().sum(-1).sqrt()
    cos = (x * mean).sum(-1) / (nv * nm)
    return 1.0 - torch.where((nv > 0) & (nm > 0), cos, torch.zeros_like(cos))


def exact(case, seed):
    c = case
    if not (c["scores"] or c["sigma"] or (c["mu"] == "running" and c["op"] != "score")):
        return None
    x = _inputs(c, seed)
    us, d, cap = (c["n_seq"], c["n_layer"], c["n_kv_head"]), c["head_dim"], _capacity(c)
    src, new = ("k", "kn") if c["keys"] else ("v", "vn")
    dev = x["k"].device
    scores = torch.zeros(us + (cap,), dtype=torch.float64, device=dev) if c["scores"] else None
    sigma = torch.zeros(us, dtype=torch.float64, device=dev) if c["sigma"] else None
    sums = torch.zeros(us + (d,), dtype=torch.float64, device=dev)
    evicts = c["op"] != "score"
    for s, n0 in enumerate(_budgets(c)):
        for layer in range(c["n_layer"]):
            rows = x[src][0][s, layer, :, :n0].double()
            if evicts:
                rows = torch.cat([rows, x[new][0][s, layer].double()], 1)
            n = rows.shape[1]
            mean = rows.mean(1, keepdim=True)
            sc = _scores64(c, rows, mean)
            if sigma is not None:
                sigma[s, layer] = sc.std(1, correction=0)
            if x["attn"] is not None:
                a = x["attn"][s, layer, :, :n].double()
                sc = a / (1.0 - a) * sc
            if scores is not None:
                scores[s, layer, :, :n] = sc
            if evicts:  # stable: equal scores keep the earlier row
                kept = torch.sort(sc, dim=1, descending=True, stable=True)[1][:, :n0]
                sums[s, layer] = torch.gather(rows, 1, kept[..., None].expand(-1, -1, d)).sum(1)
    out = {f: t for f, t in (("scores", scores), ("sigma", sigma)) if t is not None}
    if evicts:
        out.update(len=None, k=None, v=None)
        out["kept" if c["op"] == "block" else "evicted"] = None
        if c["mu"] == "running":
            out["running_sum"] = sums
        if c["holefill"]:
            out["pos"] = None
    return out

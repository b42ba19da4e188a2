"""The resident kernel (a unit's scored rows in the shared memory of its
cluster) against the streaming kernel on the same inputs, over the forms it
accepts: both layouts, rules, mean modes, fused and two-call, block and decode,
scoring options, ragged lengths and budgets, cluster sizes that divide nothing, slices
that end mid-row-group or are empty, heavy ties and non-finite rows.
VD_RESIDENT=0 forces the streaming kernel, VD_RESIDENT=c the resident one on
clusters of c CTAs (100 + c: both tensors resident).  Needs a GB300.

The two compute every score with the same operations in the same order; only
the order of the mean's double-float sums differs, which moves the two-part
mean by at most 1e-12 of the data's scale.  So scores are compared at 1e-6
relative (16 fp32 roundings), everything else exactly, running sums at 1e-12
of the summed magnitudes."""
from __future__ import annotations

import itertools

import pytest
import torch

import oracle
import paper_2609_23314_gb300 as vd
from paper_2609_23314_gb300 import build, workloads as wl
from test_gpu_parity import evict_and_check, filled_cache
from vd_gpu import evictions, units_view

pytestmark = pytest.mark.gpu

L2, DIR, NORM = vd.VD_SCORE_L2, vd.VD_SCORE_DIR, vd.VD_SCORE_NORM
REC, RUN = vd.VD_MU_RECOMPUTE, vd.VD_MU_RUNNING


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    vd.load_library()
    torch.cuda.set_device(0)


def make(n_seq, L, H, cap, d, seed, edit=None):
    st = wl.TokenStream("gauss_outlier", n_seq * L * H, d, seed=seed)
    k, v = st.next(cap)
    shape = (n_seq, L, H, cap, d)
    k, v = k.view(shape).contiguous(), v.view(shape).contiguous()
    if edit is not None:
        edit(k, v)
    return k, v


def step(force, k, v, lens, N, B, var, mu, decode, fused, budgets, options, monkeypatch):
    # (options["pos"]: hole-fill layout, positions of the cached rows)
    """One event of the cache k, v (lens rows each, the last B of them new)
    under VD_RESIDENT=force; every output, the cache and the status."""
    monkeypatch.setenv("VD_RESIDENT", str(force))
    monkeypatch.setenv("VD_SMALL_PATH", "0")
    n_seq, L, H, cap, d = k.shape
    us = (n_seq, L, H)
    cache = vd.Cache(k.clone(), v.clone(), torch.tensor([n - B for n in lens], dtype=torch.int32,
                                                        device="cuda"))
    keys = bool(options.get("keys"))
    rs = None
    if mu == RUN:
        rs = torch.zeros(us + (d,), dtype=torch.float64, device="cuda")
        vd.vd_running_sum_init_ex(cache, keys, rs)
    new = []
    for t in (k, v):
        rows = torch.stack([t[s, :, :, n - B:n] for s, n in enumerate(lens)]).contiguous()
        new.append(rows)
    if fused:  # the staged rows are not in the cache
        for s, n in enumerate(lens):
            cache.k[s, :, :, n - B:] = 0
            cache.v[s, :, :, n - B:] = 0
    else:
        vd.vd_append(cache, new[0], new[1], B)
    n_dev = torch.tensor(budgets, dtype=torch.int32, device="cuda") if budgets else None
    kept = torch.full(us + (N,), -7, dtype=torch.int32, device="cuda")
    ev = torch.full(us, -7, dtype=torch.int32, device="cuda")
    sc = torch.full(us + (cap,), -3.0, device="cuda")
    sg = torch.full(us, -3.0, device="cuda") if options.get("sigma") else None
    attn = None
    if options.get("attn"):
        g = torch.Generator(device="cuda").manual_seed(3)
        attn = torch.rand(us + (cap,), generator=g, device="cuda") * 0.02
    pos = options["pos"].clone() if "pos" in options else None
    out = dict(kept_idx_out=kept, scores_out=sc)
    how = dict(N_dev=n_dev, variant=var, mu=mu, running_sum=rs)
    if pos is not None:
        first = torch.tensor([10 ** 6 + 1000 * s for s in range(n_seq)], dtype=torch.int32,
                             device="cuda")
        how.update(pos=pos, pos_first_new=first)

    def event():
        if decode and fused:
            vd.vd_append_evict_decode(cache, *new, N, evicted_out=ev, **how, **out)
        elif decode and pos is not None:
            vd.vd_evict_decode_holefill(cache, N, evicted_out=ev, **how, **out)
        elif decode:
            vd.vd_evict_decode(cache, N, evicted_out=ev, **how, **out)
        elif pos is not None and not fused:
            vd.vd_evict_block_holefill(cache, N, B=B, **how, **out)
        elif options and pos is None:
            call = vd.vd_append_evict_block_ex if fused else vd.vd_evict_block_ex
            call(cache, *((*new, B) if fused else ()), N, **({} if fused else dict(B=B)),
                 score_keys=keys, attn=attn, dispersion_out=sg, **how, **out)
        elif fused:
            vd.vd_append_evict_block(cache, *new, B, N, **how, **out)
        else:
            vd.vd_evict_block(cache, N, B=B, **how, **out)

    took = evictions(event)  # a forced size that does not fit would run the streaming kernel
    units = n_seq * L * H
    if force == 0:
        assert {k for k, _ in took} == {"evict_kernel"}
    else:
        assert took == [("resident_evict_kernel", units * (force % 100))], (force, took)
    event()
    if pos is not None:
        for s, m in enumerate(cache.len.tolist()):
            pos[s, ..., m:] = 0  # unspecified there
        sg = pos.float()
    status = vd.vd_get_device_status()
    return cache, rs, kept, ev, sc, sg, status


def compare(forces, k, v, lens, N, B, var, mu, decode, fused, monkeypatch, budgets=None,
            options=None, score_rtol=1e-6):
    args = (k, v, lens, N, B, var, mu, decode, fused, budgets, options or {}, monkeypatch)
    want = step(0, *args)
    for force in forces:
        got = step(force, *args)
        assert got[6] == want[6]
        assert torch.equal(got[0].len, want[0].len)
        assert torch.equal(got[2], want[2]), force
        assert torch.equal(got[3], want[3]), force
        assert torch.equal(got[4] == -3.0, want[4] == -3.0)
        torch.testing.assert_close(got[4], want[4], rtol=score_rtol, atol=0, equal_nan=True)
        if options and "pos" in options:
            assert torch.equal(got[5], want[5]), force
        elif got[5] is not None:
            torch.testing.assert_close(got[5], want[5], rtol=1e-6, atol=0, equal_nan=True)
        for s, n in enumerate(want[0].len.tolist()):
            for a, b in ((got[0].k, want[0].k), (got[0].v, want[0].v)):
                assert torch.equal(a[s, :, :, :n].view(torch.int16),
                                   b[s, :, :, :n].view(torch.int16)), force
        if want[1] is not None and bool(torch.isfinite(want[1]).all()):
            scale = max(1.0, units_view(v).float().abs().nan_to_num(0, 0, 0).sum(dim=1).max().item())
            assert torch.max(torch.abs(got[1] - want[1])).item() <= 1e-12 * scale


FORMS = list(itertools.product([L2, DIR, NORM], [REC, RUN], [False, True], [False, True]))


@pytest.mark.parametrize("var,mu,decode,fused", FORMS)
def test_forms(var, mu, decode, fused, monkeypatch):
    """Every form; ragged lengths, one sequence that does not evict; C from
    one CTA to more CTAs than there are 4-row groups."""
    B = 1 if decode else 37
    for d, cap, forces in ((128, 333, (1, 3, 8, 102)), (96, 300, (2, 7, 105)), (8, 50, (1, 16, 104)),
                           (256, 131, (4, 11))):
        N = cap - B
        lens = [cap, N + 1, N] if not decode else [cap, N, cap - 2]
        lens = [max(n, B) for n in lens]
        budgets = [N, N, N] if not decode else [N, N, N - 1]
        k, v = make(3, 1, 2, cap, d, seed=d + B)
        compare(forces, k, v, lens, N, B, var, mu, decode, fused, monkeypatch, budgets)


@pytest.mark.parametrize("var,mu", [(L2, REC), (L2, RUN), (DIR, RUN), (NORM, RUN)])
@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("options", [dict(keys=True), dict(attn=True), dict(sigma=True),
                                     dict(keys=True, attn=True, sigma=True)],
                         ids=["keys", "attn", "sigma", "all"])
def test_options(var, mu, fused, options, monkeypatch):
    if options.get("sigma") and var != L2:
        options = dict(options, sigma=False)
    for d, cap, forces in ((64, 700, (1, 5, 106)), (200, 210, (3,))):
        N, B = cap * 3 // 4, cap // 5
        k, v = make(2, 2, 1, cap, d, seed=d)
        compare(forces, k, v, [cap - 3, N + 2], N, B, var, mu, False, fused, monkeypatch,
                [N, N - 5], options)


@pytest.mark.parametrize("kind", ["all_equal", "many_equal", "two_values", "nan", "inf", "huge"])
@pytest.mark.parametrize("decode", [False, True])
def test_ties_and_nonfinite(kind, decode, monkeypatch):
    """Threshold buckets with more than 256 keys, exact ties across slices,
    keys at both ends of their range."""
    def edit(k, v):
        n = v.shape[3]
        if kind == "all_equal":
            v[:] = 1.5
        elif kind == "many_equal":
            v[:, :, :, n // 4:] = v[:, :, :, :1]
        elif kind == "two_values":
            v[:] = 1.0
            v[:, :, :, ::3] = -1.0
        elif kind == "nan":
            v[:, :, :, 5, 3] = float("nan")
        elif kind == "inf":
            v[:, :, :, n - 1, 0] = float("inf")
        elif kind == "huge":
            v[:, :, :, 7] = 1e18
            v[:, :, :, 8:40] = 0.0
    cap = 1300
    B = 1 if decode else 300
    k, v = make(1, 1, 2, cap, 64, seed=9, edit=edit)
    for var, mu in ((NORM, REC), (L2, REC)):
        compare((1, 2, 9, 104), k, v, [cap], cap - B, B, var, mu, decode, False, monkeypatch)


def shuffled_positions(n_seq, L, H, cap, seed):
    """Distinct positions in no slot order, as after many hole-fill events."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    p = torch.rand(n_seq, L, H, cap, generator=g, device="cuda").argsort(-1)
    return (3 * p).to(torch.int32)


@pytest.mark.parametrize("var,mu,decode,fused", FORMS)
def test_holefill_forms(var, mu, decode, fused, monkeypatch):
    """Hole-fill layout: budgets above the cached rows (new rows kept in
    place), below them (movers from the cache too), and equal; positions that
    do not follow the slots; duplicates, so that positions decide ties."""
    def edit(k, v):
        v[:, :, :, 1::7] = v[:, :, :, :1]
    B = 1 if decode else 37
    for d, cap, forces in ((128, 333, (1, 3, 8)), (96, 300, (2, 7)), (8, 50, (1, 16)),
                           (256, 131, (4, 11))):
        N = cap - B
        lens = [cap, N + 1, N] if not decode else [cap, N, cap - 2]
        lens = [max(n, B) for n in lens]
        budgets = [N, max(1, N - 9), N] if not decode else [N, N, N - 2]
        k, v = make(3, 1, 2, cap, d, seed=d + B, edit=edit)
        compare(forces, k, v, lens, N, B, var, mu, decode, fused, monkeypatch, budgets,
                dict(pos=shuffled_positions(3, 1, 2, cap, d)))


@pytest.mark.parametrize("kind", ["all_equal", "many_equal", "nan"])
@pytest.mark.parametrize("decode", [False, True])
def test_holefill_ties(kind, decode, monkeypatch):
    def edit(k, v):
        n = v.shape[3]
        if kind == "all_equal":
            v[:] = 1.5
        elif kind == "many_equal":
            v[:, :, :, n // 4:] = v[:, :, :, :1]
        else:
            v[:, :, :, 5, 3] = float("nan")
    cap = 1300
    B = 1 if decode else 300
    k, v = make(1, 1, 2, cap, 64, seed=9, edit=edit)
    for var, N in ((NORM, cap - B), (L2, cap - B)) + (() if decode else ((NORM, 900),)):
        compare((1, 2, 9), k, v, [cap], N, B, var, REC, decode, False, monkeypatch,
                options=dict(pos=shuffled_positions(1, 1, 2, cap, 4)))


@pytest.mark.parametrize("N", [1, 2, 255, 1023])
def test_budget_edges(N, monkeypatch):
    cap = 1024
    k, v = make(1, 1, 3, cap, 64, seed=N)
    compare((1, 6, 16, 103), k, v, [cap], N, cap - N, L2, RUN, False, True, monkeypatch)


def test_rejected_lengths_leave_the_unit_alone(monkeypatch):
    """The same status codes as the streaming kernel, and nothing written."""
    for force in (0, 3):
        monkeypatch.setenv("VD_RESIDENT", str(force))
        monkeypatch.setenv("VD_SMALL_PATH", "0")
        for ln, n_dev, code in ((90, None, 7), (-1, None, 7), (80, 0, 8), (80, 61, 8)):
            k, v = make(1, 1, 2, 80, 64, seed=1)
            cache = vd.Cache(k.clone(), v.clone(), torch.tensor([ln], dtype=torch.int32,
                                                                device="cuda"))
            nd = None if n_dev is None else torch.tensor([n_dev], dtype=torch.int32, device="cuda")
            vd.vd_evict_block(cache, 60, nd, 20, L2)
            assert vd.vd_get_device_status() == code
            assert int(cache.len[0]) == ln
            assert torch.equal(cache.v, v) and torch.equal(cache.k, k)


# sequences, layers, KV heads, capacity, head dim -> CTAs per unit of the resident
# kernel that the library picks by itself, or None for the streaming kernel
AUTOMATIC = {
    "long-rows": ((1, 1, 2, 1500, 128), 12),          # few units: the most CTAs per unit
    "half-sms": ((1, 4, 19, 700, 128), 4),            # 76 units, 304 CTAs: two per SM
    "two-per-sm": ((2, 4, 38, 200, 128), 1),          # 304 units: the last with one wave
    "over-two-per-sm": ((2, 1, 153, 200, 128), 1),    # 306: three share an SM
    "many-waves": ((3, 5, 80, 230, 96), 1),           # 1200 units
    "too-large": ((2, 1, 153, 700, 128), None),       # one CTA per SM: the streaming kernel
}


@pytest.mark.parametrize("decode", [False, True], ids=["block", "decode"])
@pytest.mark.parametrize("case", list(AUTOMATIC))
def test_automatic_dispatch_matches_oracle(orc, case, decode, monkeypatch):
    """The plans the library makes by itself, on both sides of the rule's lines
    (for 152 SMs), against the fp64 oracle on a sample of the units."""
    for name in ("VD_RESIDENT", "VD_SMALL_PATH", "VD_CLUSTER_SIZE"):
        monkeypatch.delenv(name, raising=False)
    (n_seq, L, H, cap, d), ctas = AUTOMATIC[case]
    B = 1 if decode else 30
    N = cap - B
    cache = filled_cache(n_seq, L, H, cap, d, [cap] * n_seq, seed=cap)
    units = cache.units
    rs = torch.zeros(cache.unit_shape() + (d,), dtype=torch.float64, device="cuda")
    cache.len.fill_(N)
    vd.vd_running_sum_init(cache, rs)
    cache.len.fill_(cap)

    def event():
        if decode:
            vd.vd_evict_decode(cache, N, None, oracle.L2, RUN, rs)
        else:
            vd.vd_evict_block(cache, N, None, B, oracle.L2, RUN, rs)

    took = evictions(event)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        if ctas is None:
            assert {k for k, _ in took} == {"evict_kernel"}
        elif decode and ctas > 1:  # decode: three CTAs per SM
            assert took[0][0] == "resident_evict_kernel" and took[0][1] >= units * ctas
        else:
            assert took == [("resident_evict_kernel", units * ctas)], took
    evict_and_check(orc, cache, N, B, oracle.L2, RUN, rs, units=range(0, units, max(1, units // 40)),
                    decode=decode)
    ref = torch.zeros_like(rs)
    vd.vd_running_sum_init(cache, ref)
    scale = units_view(cache.v).float().abs().sum(dim=1).max().item()
    assert torch.max(torch.abs(ref - rs)).item() <= 1e-12 * scale

"""A wait for bulk copies that gives up (VD_WAIT_LIMIT lowers its limit to no
poll at all, so that it always does): the call records VD_ERR_TIMEOUT, the
unit's rows, positions and running sum and the sequence's length stay as they
were, and the same call without the limit then gives what it gives on a fresh
cache.  Only the wait for the other tensor that follows the first one's
compaction (one buffer for both) cannot leave the unit as it was; it leaves
that tensor and the length.  Needs a GB300."""
from __future__ import annotations

import pytest
import torch

import paper_2609_23314_gb300 as vd
from paper_2609_23314_gb300 import build, workloads as wl
from vd_gpu import new_cache, units_view

pytestmark = pytest.mark.gpu

TIMEOUT = 5
SCORED, OTHER = "0", "4194304:0"  # which wait gives up


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    vd.load_library()
    torch.cuda.set_device(0)
    yield
    assert vd.vd_get_device_status() == 0


def make(n_seq, L, H, cap, d, lens, B):
    cache = new_cache(n_seq, L, H, cap, d)
    st = wl.TokenStream("gauss_outlier", cache.units, d, device="cuda", seed=cap + d)
    wl.fill_rows(st, units_view(cache.k), units_view(cache.v), cap)
    us = cache.unit_shape()
    k, v = (t.view(us + (B, d)).contiguous() for t in st.next(B))
    cache.len.copy_(torch.tensor(lens, dtype=torch.int32))
    rs = torch.zeros(us + (d,), dtype=torch.float64, device="cuda")
    vd.vd_running_sum_init(cache, rs)
    pos = (3 * torch.rand(us + (cap,), device="cuda").argsort(-1)).to(torch.int32)
    first = torch.full((n_seq,), 10 ** 6, dtype=torch.int32, device="cuda")
    return dict(k=cache.k, v=cache.v, len=cache.len, rs=rs, pos=pos, first=first, kn=k, vn=v)


def clone(s):
    return {k: t.clone() for k, t in s.items()}


def evict(s, N, B, decode, holefill):
    """The fused call on the state s; the kept slots."""
    cache = vd.Cache(s["k"], s["v"], s["len"])
    kept = torch.full(cache.unit_shape() + (N,), -7, dtype=torch.int32, device="cuda")
    hole = dict(pos=s["pos"], pos_first_new=s["first"]) if holefill else {}
    if decode:
        vd.vd_append_evict_decode(cache, s["kn"], s["vn"], N, None, vd.VD_SCORE_L2,
                                  vd.VD_MU_RUNNING, s["rs"], None, kept, **hole)
    else:
        vd.vd_append_evict_block(cache, s["kn"], s["vn"], B, N, None, vd.VD_SCORE_L2,
                                 vd.VD_MU_RUNNING, s["rs"], kept, **hole)
    return kept


def same(a, b, names):
    for n in names:
        x, y = a[n], b[n]
        if x.dtype == torch.bfloat16:
            x, y = x.view(torch.int16), y.view(torch.int16)
        assert torch.equal(x, y), n


# route: (VD_RESIDENT, n_seq, L, H, capacity, head dim); None: the short-cache
# kernel, with and without the cluster that sets the lengths
ROUTES = {"short-cluster": (None, 2, 1, 3, 160, 64), "short-single": (None, 3, 1, 1, 96, 128),
          "short-many": (None, 3, 5, 4, 60, 64), "resident-1": (1, 3, 1, 2, 300, 96),
          "resident-3": (3, 2, 2, 1, 300, 128), "resident-both": (105, 2, 1, 2, 333, 64)}


@pytest.mark.parametrize("which", [SCORED, OTHER], ids=["scored", "other"])
@pytest.mark.parametrize("decode", [False, True], ids=["block", "decode"])
@pytest.mark.parametrize("holefill", [False, True], ids=["ordered", "holefill"])
@pytest.mark.parametrize("route", list(ROUTES))
def test_evictions(route, holefill, decode, which, monkeypatch):
    force, n_seq, L, H, cap, d = ROUTES[route]
    if holefill and (force is None or force >= 100 or which == OTHER):
        pytest.skip("no such form")
    monkeypatch.setenv("VD_SMALL_PATH", "1" if force is None else "0")
    if force is not None:
        monkeypatch.setenv("VD_RESIDENT", str(force))
    B = 1 if decode else 20
    N = cap - B
    lens = [N] * n_seq
    if force is None:  # the short-cache kernel also waits before it only appends
        lens[0] = N - B
    base = make(n_seq, L, H, cap, d, lens, B)
    want = clone(base)
    want["kept"] = evict(want, N, B, decode, holefill)
    assert vd.vd_get_device_status() == 0
    got = clone(base)
    monkeypatch.setenv("VD_WAIT_LIMIT", which)
    kept = evict(got, N, B, decode, holefill)
    assert vd.vd_get_device_status() == TIMEOUT
    if which == OTHER and force is not None and force < 100:
        same(got, base, ["k", "len"])  # V is compacted: the unit is unspecified
        return
    assert bool((kept == -7).all())
    same(got, base, list(base))
    monkeypatch.delenv("VD_WAIT_LIMIT")
    got["kept"] = evict(got, N, B, decode, holefill)
    assert vd.vd_get_device_status() == 0
    names = ["kept", "len", "rs"] + (["pos"] if holefill else [])
    same(got, want, names)
    for s, n in enumerate(want["len"].tolist()):
        same({x: got[x][s, ..., :n, :] for x in "kv"}, {x: want[x][s, ..., :n, :] for x in "kv"},
             "kv")


@pytest.mark.parametrize("mu", [vd.VD_MU_RECOMPUTE, vd.VD_MU_RUNNING], ids=["recompute", "running"])
@pytest.mark.parametrize("d", [64, 256])
def test_score_only(d, mu, monkeypatch):
    s = make(2, 1, 3, 1500, d, [1500, 1400], 1)
    cache = vd.Cache(s["k"], s["v"], s["len"])
    out = []
    for limit in (None, "0", None):
        if limit is None:
            monkeypatch.delenv("VD_WAIT_LIMIT", raising=False)
        else:
            monkeypatch.setenv("VD_WAIT_LIMIT", limit)
        sc = torch.full(cache.unit_shape() + (1500,), -1.0, device="cuda")
        vd.vd_score_ex(cache, vd.VD_SCORE_L2, scores_out=sc, mu=mu,
                       running_sum=s["rs"] if mu == vd.VD_MU_RUNNING else None)
        assert vd.vd_get_device_status() == (0 if limit is None else TIMEOUT)
        out.append(sc)
    assert torch.equal(out[0], out[2])

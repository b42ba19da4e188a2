"""Calls of every kind back to back on one stream, on the same caches: short-cache,
resident, streaming and split evictions, split score passes, appends and
length updates, all of them programmatic dependents of what runs before them
(the second part of a split launch does not even wait before it reads), with
copies and a memset in between.  Without a synchronisation, and replayed from
a CUDA graph, they give the bytes that they give with one after every call.
Needs a GB300."""
from __future__ import annotations

import pytest
import torch

import paper_2609_23314_gb300 as vd
from paper_2609_23314_gb300 import build, workloads as wl
from vd_gpu import launched_kernels, new_cache

pytestmark = pytest.mark.gpu

UNITS = 168    # above the SM count: hole-fill block and score calls split
ROUNDS = 6
N, B, D = 256, 64, 128
SHORT_N, SHORT_D = 90, 64


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    vd.load_library()
    torch.cuda.set_device(0)
    yield
    assert vd.vd_get_device_status() == 0


class State:
    """An ordered cache x, a hole-fill cache z and a short cache y, empty, with
    their running sums, the blocks of every round, and staging for one."""

    def __init__(self):
        self.x, self.z = (new_cache(1, 21, 8, N + B, D) for _ in range(2))
        self.y = new_cache(1, 21, 8, SHORT_N + B, SHORT_D)
        us = self.x.unit_shape()
        f64 = dict(dtype=torch.float64, device="cuda")
        self.rx, self.rz = torch.zeros(us + (D,), **f64), torch.zeros(us + (D,), **f64)
        self.ry = torch.zeros(us + (SHORT_D,), **f64)
        self.pos = torch.zeros(us + (N + B,), dtype=torch.int32, device="cuda")
        self.first = torch.zeros(1, dtype=torch.int32, device="cuda")
        blocks = wl.TokenStream("gauss_outlier", UNITS, D, device="cuda", seed=3)
        short = wl.TokenStream("gauss_outlier", UNITS, SHORT_D, device="cuda", seed=4)
        self.blocks = [[t.view(us + (B, -1)).contiguous() for t in st.next(B)]
                       for st in (blocks, short) for _ in range(ROUNDS)]
        self.new = [torch.zeros_like(t) for t in self.blocks[0]]
        self.short = [torch.zeros_like(t) for t in self.blocks[ROUNDS]]
        self.scores = torch.zeros(us + (N + B,), device="cuda")
        self.sigma = torch.zeros((ROUNDS,) + us, device="cuda")
        self.kept = torch.full((ROUNDS,) + us + (N,), -7, dtype=torch.int32, device="cuda")

    def outputs(self):
        out = {"lens": torch.cat([c.len for c in (self.x, self.y, self.z)])}
        for name in ("rx", "ry", "rz", "pos", "scores", "sigma", "kept"):
            out[name] = getattr(self, name)
        for name, c, n in (("x", self.x, N), ("y", self.y, SHORT_N), ("z", self.z, N)):
            out["k" + name], out["v" + name] = c.k[..., :n, :], c.v[..., :n, :]
        out["pos"] = self.pos[..., :N]
        return {k: t.contiguous().view(torch.uint8).clone() for k, t in out.items()}


def calls(s, monkeypatch):
    """One closure per call or copy, in order."""
    RUN = vd.VD_MU_RUNNING

    def route(resident):
        if resident:
            monkeypatch.delenv("VD_RESIDENT", raising=False)
        else:
            monkeypatch.setenv("VD_RESIDENT", "0")

    def copy(dst, src):
        for a, b in zip(dst, src):
            a.copy_(b)

    def block(c, new, n, rs, resident, **kw):
        route(resident)
        vd.vd_append_evict_block(c, *new, B, n, None, vd.VD_SCORE_L2, RUN, rs, **kw)

    def two_calls(c, new, n, rs, resident):
        route(resident)
        vd.vd_append(c, *new, B)
        vd.vd_evict_block(c, n, None, B, vd.VD_SCORE_L2, RUN, rs)

    def score(r):
        vd.vd_score_ex(s.x, vd.VD_SCORE_L2, scores_out=s.scores, dispersion_out=s.sigma[r],
                       mu=RUN, running_sum=s.rx)

    for r in range(ROUNDS):
        resident = r % 2 == 0
        yield lambda: copy(s.new, s.blocks[r])
        if r % 3 == 2:
            yield lambda: two_calls(s.x, s.new, N, s.rx, resident)
        else:
            yield lambda: block(s.x, s.new, N, s.rx, resident, kept_idx_out=s.kept[r])
        yield lambda: score(r)
        yield lambda: block(s.z, s.new, N, s.rz, resident, pos=s.pos, pos_first_new=s.first)
        yield lambda: s.first.add_(B)
        yield lambda: copy(s.short, s.blocks[ROUNDS + r])
        yield lambda: block(s.y, s.short, SHORT_N, s.ry, True)
        yield lambda: two_calls(s.y, s.short, SHORT_N, s.ry, True)
        yield lambda: s.scores[..., :1].zero_()
        yield lambda: score(r)


def test_mixed_calls(monkeypatch):
    want = State()
    for call in calls(want, monkeypatch):
        call()
        torch.cuda.synchronize()
    assert vd.vd_get_device_status() == 0
    expected = want.outputs()

    free = State()
    torch.cuda.synchronize()
    for call in calls(free, monkeypatch):
        call()
    torch.cuda.synchronize()
    got = free.outputs()
    assert all(torch.equal(expected[k], got[k]) for k in expected), "without synchronisation"

    static = State()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        for call in calls(static, monkeypatch):
            call()
    graph.replay()
    torch.cuda.synchronize()
    got = static.outputs()
    assert all(torch.equal(expected[k], got[k]) for k in expected), "replayed"

    # every kernel takes part
    kernels = [k for c in calls(static, monkeypatch) for k, _ in launched_kernels(c)]
    assert {"small_evict_kernel", "resident_evict_kernel", "evict_kernel", "vd_append_kernel",
            "vd_len_add_kernel", "vd_len_clamp_kernel"} <= set(kernels)

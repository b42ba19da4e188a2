"""The score pass for head dims off the batched path, and for the Dir rule at
every head dim, at the edges of its batches: row counts around the rows a CTA
takes per stage and per batch, idle lanes (d / 8 no power of two), one or two
lanes per row.  Scores against the fp64 oracle at the bound of
``vd_gpu.score_tolerance``; evictions through every kernel that holds the pass
(block and decode, both layouts) on clusters of 1 and 2 CTAs.  Needs a GB300."""
from __future__ import annotations

import pytest
import torch

import oracle
import paper_2609_23314_gb300 as vd
from paper_2609_23314_gb300 import build
from test_gpu_parity import evict_and_check, filled_cache
from vd_gpu import bits, check_scores

pytestmark = pytest.mark.gpu

CASES = [(d, v) for d in (8, 16, 24, 72, 80, 96, 112, 192, 248)
         for v in (oracle.L2, oracle.DIR, oracle.NORM)]
CASES += [(d, oracle.DIR) for d in (64, 128, 256)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    vd.load_library()
    torch.cuda.set_device(0)
    yield
    assert vd.vd_get_device_status() == 0


@pytest.mark.parametrize("d,var", CASES)
def test_scores_at_batch_edges(orc, d, var):
    lens = [1, 2, 3, 7, 8, 9, 31, 33, 63, 65, 127, 130]
    cache = filled_cache(len(lens), 1, 2, max(lens), d, lens, seed=d)
    sc = torch.full(cache.unit_shape() + (max(lens),), -1.0, device="cuda")
    vd.vd_score(cache, var, sc)
    for s, n in enumerate(lens):
        for h in range(2):
            got = sc[s, 0, h].cpu().numpy()
            check_scores(orc, var, bits(cache.v[s, 0, h, :n]), got[:n])
            assert (got[n:] == -1.0).all()


@pytest.mark.parametrize("d,var", [c for c in CASES if c[0] in (16, 80, 192, 128)])
@pytest.mark.parametrize("cluster", ["1", "2"])
def test_every_kernel_with_the_pass(orc, d, var, cluster, monkeypatch):
    monkeypatch.setenv("VD_CLUSTER_SIZE", cluster)
    if d < 64 and cluster == "2":
        pytest.skip("segments of 64 bytes")
    for decode in (False, True):
        B = 1 if decode else 23
        N = 131
        cache = filled_cache(2, 1, 2, N + B, d, [N + B, N + 1], seed=d + B)
        evict_and_check(orc, cache, N, B, var, vd.VD_MU_RECOMPUTE, None, decode=decode)
        # the hole-fill layout keeps the same tokens
        a = filled_cache(1, 1, 2, N + B, d, [N + B], seed=d)
        b = vd.Cache(a.k.clone(), a.v.clone(), a.len.clone())
        pos = torch.arange(N + B, dtype=torch.int32, device="cuda").expand(1, 1, 2, -1).contiguous()
        first = torch.tensor([N], dtype=torch.int32, device="cuda")
        if decode:
            vd.vd_evict_decode(a, N, variant=var)
            vd.vd_evict_decode_holefill(b, N, pos, first, variant=var)
        else:
            vd.vd_evict_block(a, N, B=B, variant=var)
            vd.vd_evict_block_holefill(b, N, pos, first, B=B, variant=var)
        order = torch.argsort(pos[..., :N], dim=-1)[..., None].expand(-1, -1, -1, -1, d)
        for x, y in ((a.k, b.k), (a.v, b.v)):
            y = torch.gather(y[..., :N, :].view(torch.int16), 3, order)
            assert torch.equal(x[..., :N, :].view(torch.int16), y)

"""The 8-head indexer and the 16-head attention (needs a B200): warp-per-query kernels at the edges of their ranges, against
the oracle."""
import pytest
import torch

from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload, PrefillWorkload

import parity_util as pu

pytestmark = pytest.mark.gpu

SMALL = CONFIGS["cfg1"]


@pytest.mark.parametrize("change", [
    dict(L=1), dict(L=15), dict(L=133),                              # less than a tile, no candidates yet
    dict(L=700, M=16, Ksp=512, W=64),                                # the largest budget the warp form takes (1024 slots)
    dict(L=1500, M=4, P=128, B=8, Ksp=300, W=16),                    # 16 sub-blocks a page, a ragged last page
    dict(L=2100, M=2, P=256, B=8, Ksp=128, W=200),                   # 32 sub-blocks a page
    dict(L=900, M=17, Ksp=256),                                      # one page more than that: the block form
    dict(L=1000, hi_enable=False, M=8, Ksp=400),                     # every page, the warp form
    dict(L=1100, hi_enable=False, M=8, Ksp=400),                     # every page, too many slots for it
    dict(L=17000, M=8, R=1),                                         # more than 256 pages; a query per attention warp
])
def test_small_prefill(cuda_device, change):
    cfg = SMALL.replace(**{"name": "small", "seed": 7, **change})
    wl = PrefillWorkload(cfg, cuda_device)
    wl.prepare()
    pages = torch.empty((cfg.L, cfg.M), dtype=torch.int32, device=cuda_device)
    wl.index(pages_out=pages)
    want_idx = wl.sparse_idx.clone()
    wl.step()
    assert wl.ctx.status() == 0 and torch.equal(want_idx, wl.sparse_idx)
    queries = pu.boundary_queries(cfg, 0, cfg.L, 60, seed=3)
    m = pu.check_prefill(wl, queries, pages=pages if cfg.hi_enable else None)
    print(change, m.summary())
    m.assert_ok(pu.TOL_BF16)


@pytest.mark.parametrize("change", [dict(L=6000), dict(L=6000, M=16, Ksp=700), dict(L=20000, P=128, M=8), dict(L=9000, P=256, M=4, B=8),
                                    dict(L=1000, hi_enable=False, Ksp=400), dict(L=40, W=4)])
def test_chunks_give_the_lists_of_the_whole_run(cuda_device, change):
    """The indexer's lists do not depend on how many queries a call has (one, four or sixteen warps per query)."""
    cfg = SMALL.replace(**{"name": "chunks", "seed": 8, "R": 1, **change})

    def lists(n_query):
        wl = PrefillWorkload(cfg, cuda_device, q_pos0=cfg.L - n_query, n_query=n_query)
        wl.prepare()
        pages = torch.empty((n_query, cfg.M), dtype=torch.int32, device=cuda_device)
        wl.index(pages_out=pages)
        assert wl.ctx.status() == 0
        return wl.sparse_idx, wl.n_sparse, pages

    whole = lists(cfg.L)
    for n_query in (1, 17, 140, 149, 500, 600, 1300):
        if n_query < cfg.L:
            assert all(torch.equal(a, b[-n_query:]) for a, b in zip(lists(n_query), whole)), n_query


@pytest.mark.parametrize("batch,split", [(1, 0), (3, 2), (5, 3), (130, 1)])
def test_small_paged_decode(cuda_device, batch, split):
    cfg = SMALL.replace(name="small_dec", mode="decode", batch=batch, ctx_lo=1, ctx_hi=3000, kv_page=64, R=1, seed=batch)
    wl = DecodeWorkload(cfg, cuda_device)
    wl.prepare()
    wl.ctx.tune(2, split)          # LSA_TUNE_ATTN_SPLIT
    wl.step()
    assert wl.ctx.status() == 0
    m = pu.check_decode(wl, range(min(batch, 12)))
    print(batch, split, m.summary())
    m.assert_ok(pu.TOL_BF16)


@pytest.mark.parametrize("W,Ksp,M", [(64, 64, 4), (1024, 512, 16)])
@pytest.mark.parametrize("n_query", [1, 148, 149, 592, 593, 889])
def test_attention_of_few_queries(cuda_device, n_query, W, Ksp, M):
    """One, four and eight warps per query, at the counts where they change hands on 148 SMs (592 and 888 with few and many rows)."""
    cfg = SMALL.replace(name="few", L=3000, W=W, Ksp=Ksp, M=M, seed=n_query)
    wl = PrefillWorkload(cfg, cuda_device, q_pos0=cfg.L - n_query, n_query=n_query)
    wl.prepare()
    wl.step()
    assert wl.ctx.status() == 0
    m = pu.check_prefill(wl, range(wl.q_pos0, cfg.L, max(1, n_query // 10)))
    print(n_query, W, m.summary())
    m.assert_ok(pu.TOL_BF16)

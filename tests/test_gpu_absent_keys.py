"""Attention reads nothing but the listed cache rows into its results (needs a B200): every other row is NaN, and the row counts are
no multiples of a tile.  And what is not finite in the listed rows or the queries shows in the results."""
import numpy as np
import pytest
import torch

from oracle import reference_run as ref
from paper_2608_01662_b200 import binding
from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,batch,split,gather", [("cfg1", 1, 0, 0), ("cfg1", 9, 0, 0), ("cfg1", 9, 1, 0), ("cfg1", 200, 0, 0), ("cfg4", 1, 0, 0),
                                                     ("cfg4", 9, 0, 0), ("cfg4", 160, 0, 0), ("cfg4", 9, 0, 1), ("cfg4", 160, 0, 1)])
def test_rows_of_nobody_in_a_pool(cuda_device, base, batch, split, gather):
    cfg = CONFIGS[base].replace(name="nobody", mode="decode", batch=batch, ctx_lo=1, ctx_hi=700, kv_page=64, R=1, M=4, Ksp=64, W=100, seed=batch)
    wl = DecodeWorkload(cfg, cuda_device)
    wl.prepare()
    wl.ctx.tune(2, split)          # LSA_TUNE_ATTN_SPLIT
    wl.ctx.tune(4, gather)         # LSA_TUNE_ATTN_GATHER
    # a page of nobody in front of the pool: no sequence has row 0
    front = lambda t, rows: torch.cat([torch.zeros_like(t[:rows]), t])  # noqa: E731
    wl.page_table = torch.where(wl.page_table >= 0, wl.page_table + 1, -1)
    wl.keys = {n: front(t, 64) for n, t in wl.keys.items()}
    wl.kmean = front(wl.kmean, 64 // cfg.B)
    owned = torch.zeros((wl.n_pg + 1) * 64, dtype=torch.bool, device=cuda_device)
    for b in range(batch):
        s = torch.arange(int(wl.ctx_len[b]), device=cuda_device)
        owned[wl.page_table[b][s // 64].long() * 64 + s % 64] = True
    own_v = wl.v[0].data_ptr() != wl.k[0].data_ptr()
    wl.k[0] = torch.where(owned[:, None], front(wl.k[0], 64), float("nan"))
    wl.v[0] = torch.where(owned[:, None], front(wl.v[0], 64), float("nan")) if own_v else wl.k[0][:, :cfg.d_v]
    wl.step()
    assert wl.ctx.status() == 0
    m = pu.check_decode(wl, range(min(batch, 20)))
    m.assert_ok(pu.TOL_BF16)
    assert all(torch.isfinite(o).all() for o in wl.out)


@pytest.mark.parametrize("base,n_query", [("cfg1", 50), ("cfg1", 1300), ("cfg3", 50), ("cfg3", 300)])
def test_rows_that_no_query_attends(cuda_device, base, n_query):
    """No sink: row 0 and everything between the listed rows and the window is nobody's."""
    n_key, W, K = 3000, 37, 12
    cfg = CONFIGS[base].replace(L=n_key, S=0, W=W, Ksp=K, R=1)
    params = binding.make_params(cfg)
    ctx = binding.Context(params, n_query, n_key, 1, device=cuda_device)
    g = torch.Generator(device=cuda_device).manual_seed(n_query)
    draw = lambda *shape: torch.randn(shape, generator=g, device=cuda_device).to(torch.bfloat16)  # noqa: E731
    q, k = draw(n_query, cfg.H, cfg.d_qk), draw(n_key, cfg.d_qk)
    v = k[:, :cfg.d_v] if cfg.mla else draw(n_key, cfg.d_v)
    q_pos0 = n_key - n_query
    idx = torch.full((n_query, K), -1, dtype=torch.int32, device=cuda_device)
    n_sparse = torch.arange(n_query, dtype=torch.int32, device=cuda_device) % K
    listed = 100 + torch.arange(K, dtype=torch.int32, device=cuda_device)
    idx[:] = torch.where(torch.arange(K, device=cuda_device)[None] < n_sparse[:, None], listed[None], -1)
    k[:100] = float("nan")
    k[100 + K:q_pos0 - W + 1] = float("nan")
    if not cfg.mla:
        v[:100] = float("nan")
        v[100 + K:q_pos0 - W + 1] = float("nan")
    out = torch.empty((n_query, cfg.H, cfg.d_v), dtype=torch.bfloat16, device=cuda_device)
    lse = torch.empty((n_query, cfg.H), dtype=torch.float32, device=cuda_device)
    ctx.sparse_attn(q, k, v, idx, n_sparse, q_pos0, n_query, n_key, out, lse)
    assert ctx.status() == 0 and torch.isfinite(out).all() and torch.isfinite(lse).all()
    caches = ref.HostCaches(np.zeros((n_key, 1)), None, [pu.to_np(k)], [pu.to_np(v)], cfg.B, n_key=n_key)
    m = pu.Metrics()
    for i in range(0, n_query, 7):
        want, want_lse = ref.attend_query(q_pos0 + i, [pu.to_np(q[i])], caches, pu.to_np(idx[i])[:int(n_sparse[i])], S=0, W=W,
                                          sm_scale=cfg.sm_scale, d_v=cfg.d_v)
        m.add_out(pu.to_np(out[i]), want[0], pu.to_np(lse[i]), want_lse[0])
    m.assert_ok(pu.TOL_BF16)


@pytest.mark.parametrize("base,n_query", [("cfg1", 40), ("cfg1", 1300), ("cfg3", 40)])
def test_what_is_not_finite_shows(cuda_device, base, n_query):
    """A NaN in one head of a query: that head's output is NaN and no other changes.  A NaN in a cache row: every head of the queries
    that attend it."""
    n_key, W, K = 2000, 50, 4
    cfg = CONFIGS[base].replace(L=n_key, S=0, W=W, Ksp=K, R=1)
    ctx = binding.Context(binding.make_params(cfg), n_query, n_key, 1, device=cuda_device)
    g = torch.Generator(device=cuda_device).manual_seed(n_query)
    draw = lambda *shape: torch.randn(shape, generator=g, device=cuda_device).to(torch.bfloat16)  # noqa: E731
    q, k = draw(n_query, cfg.H, cfg.d_qk), draw(n_key, cfg.d_qk)
    v = k[:, :cfg.d_v] if cfg.mla else draw(n_key, cfg.d_v)
    idx = torch.full((n_query, K), -1, dtype=torch.int32, device=cuda_device)
    n_sparse = torch.zeros(n_query, dtype=torch.int32, device=cuda_device)
    q_pos0 = n_key - n_query

    def run():
        out = torch.empty((n_query, cfg.H, cfg.d_v), dtype=torch.bfloat16, device=cuda_device)
        ctx.sparse_attn(q, k, v, idx, n_sparse, q_pos0, n_query, n_key, out)
        assert ctx.status() == 0
        return out

    plain = run()
    assert torch.isfinite(plain).all()
    q[7, 3, 5] = float("nan")
    got = run()
    assert torch.isnan(got[7, 3]).all()
    got[7, 3] = plain[7, 3]
    assert torch.equal(got, plain)
    q[7, 3, 5] = 0.5
    row = q_pos0 + 20
    k[row, 0] = float("nan")
    got = run()
    attends = (torch.arange(n_query, device=cuda_device) >= 20) & (torch.arange(n_query, device=cuda_device) < 20 + W)
    assert torch.isnan(got[attends]).all() and torch.isfinite(got[~attends]).all()

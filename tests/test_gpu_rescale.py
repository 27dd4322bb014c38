"""64-head attention where a row's maximum grows by more than the kernel lets stand (needs a B200): O, the row sums and the tile's
weights are rescaled in either half of a tile; and every number of rows around a tile's and an MMA step's edges."""
import numpy as np
import pytest
import torch

from oracle import reference_run as ref
from paper_2608_01662_b200 import binding
from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("listed", [False, True])
@pytest.mark.parametrize("gain", [0.0, 0.125, 1.0])
def test_growing_rows(cuda_device, listed, gain):
    """Query i attends i + 1 rows, in the window (whole tiles by TMA) or from its list; the scores' spread grows along them."""
    n = 200
    cfg = CONFIGS["cfg3"].replace(L=n + 256, S=0, W=1 if listed else 256, Ksp=256, R=1)
    ctx = binding.Context(binding.make_params(cfg), n, n + 256, 1, device=cuda_device)
    g = torch.Generator(device=cuda_device).manual_seed(int(gain * 8) + listed)
    draw = lambda *shape: torch.randn(shape, generator=g, device=cuda_device)  # noqa: E731
    q_pos0 = 256 if listed else 0
    q, k = draw(n, cfg.H, cfg.d_qk).to(torch.bfloat16), draw(n + 256, cfg.d_qk)
    k = (k * (1.0 + gain * torch.arange(n + 256, device=cuda_device)[:, None].remainder(256))).to(torch.bfloat16)
    idx = torch.full((n, cfg.Ksp), -1, dtype=torch.int32, device=cuda_device)
    n_sparse = torch.zeros(n, dtype=torch.int32, device=cuda_device)
    if listed:
        n_sparse = torch.arange(n, dtype=torch.int32, device=cuda_device)
        places = torch.arange(cfg.Ksp, dtype=torch.int32, device=cuda_device)
        idx = torch.where(places[None] < n_sparse[:, None], places[None], -1)
    out = torch.empty((n, cfg.H, cfg.d_v), dtype=torch.bfloat16, device=cuda_device)
    lse = torch.empty((n, cfg.H), dtype=torch.float32, device=cuda_device)
    ctx.sparse_attn(q, k, k[:, :cfg.d_v], idx, n_sparse, q_pos0, n, n + 256, out, lse)
    assert ctx.status() == 0
    caches = ref.HostCaches(np.zeros((n + 256, 1)), None, [pu.to_np(k)], [pu.to_np(k[:, :cfg.d_v])], cfg.B, n_key=n + 256)
    for i in [0, 14, 15, 16, 17, 30, 31, 32, 33, 47, 48, 62, 63, 64, 65, 80, 95, 96, 126, 127, 128, 129, 144, 160, 191, 192, 193, n - 1]:
        want, want_lse = ref.attend_query(q_pos0 + i, [pu.to_np(q[i])], caches, pu.to_np(idx[i])[:int(n_sparse[i])], S=0, W=cfg.W,
                                          sm_scale=cfg.sm_scale, d_v=cfg.d_v)
        # bf16 weights and results: 2^-9 of the values' norm each, a few of those
        got = pu.to_np(out[i])
        assert np.linalg.norm(got - want[0]) <= 1e-2 * np.linalg.norm(want[0]), i
        assert np.abs(pu.to_np(lse[i]) - want_lse[0]).max() <= 1e-4 * max(1.0, np.abs(want_lse[0]).max()), i


# one kernel for each number of row splits; several tiles a split
@pytest.mark.parametrize("batch,split", [(2, 1), (150, 1), (2, 2), (2, 4), (2, 8), (2, 16),
                                         (16, 0), (34, 0),         # as many splits as the batch gets: four and two
                                         (1, 0), (2, 0)])          # 16, the value dims in four and in two parts
@pytest.mark.parametrize("gain", [0.01, 0.125])
def test_growing_rows_of_a_row_list(cuda_device, batch, split, gain):
    """Paged caches: a sequence attends all of its rows in order, and the scores' spread grows along them."""
    cfg = CONFIGS["cfg4"].replace(batch=batch, ctx_lo=2050, ctx_hi=2300, R=2, seed=batch + split)
    wl = DecodeWorkload(cfg, cuda_device)
    assert cfg.ctx_hi <= cfg.S + cfg.Ksp + cfg.W
    grow = torch.ones(wl.k[0].shape[0], device=cuda_device)
    for row in wl.page_table.long():
        pages = row[row >= 0]
        place = torch.arange(pages.numel() * cfg.kv_page, device=cuda_device)
        grow[pages[place // cfg.kv_page] * cfg.kv_page + place % cfg.kv_page] = 1.0 + gain * place
    for k in wl.k:
        k.mul_(grow[:, None])
    wl.prepare()
    wl.ctx.tune(2, split)          # LSA_TUNE_ATTN_SPLIT
    wl.step()
    assert wl.ctx.status() == 0
    pools = (pu.to_np(wl.ctx_len), pu.to_np(wl.page_table), pu.to_np(wl.keys["k"]), pu.to_np(wl.keys["scale"]))
    for b in sorted({0, 1, batch // 2, batch - 1} & set(range(batch))):
        caches, t = pu.decode_caches(wl, b, pools)
        chosen = pu.to_np(wl.sparse_idx[b])[:int(wl.n_sparse[b])]
        assert len(chosen) == t + 1 - cfg.S - cfg.W
        want, want_lse = ref.attend_query(t, [pu.to_np(q[b]) for q in wl.q], caches, chosen, S=cfg.S, W=cfg.W, sm_scale=cfg.sm_scale, d_v=cfg.d_v)
        for r in range(cfg.R):      # the bounds of the test above
            got = pu.to_np(wl.out[r][b])
            assert np.linalg.norm(got - want[r]) <= 1e-2 * np.linalg.norm(want[r]), (b, r)
            assert np.abs(pu.to_np(wl.lse[r][b]) - want_lse[r]).max() <= 1e-4 * max(1.0, np.abs(want_lse[r]).max()), (b, r)

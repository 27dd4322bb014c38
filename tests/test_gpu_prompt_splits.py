"""Prompt chunks at the end of a long cache (needs a B200): a query block's tiles of mean keys dealt to several blocks, and large
budgets whose pages are tiles of their own or halves of one.  Inputs of small whole numbers, so that pages and tokens must be
the oracle's."""
import pytest
import torch

from oracle import reference_run as ref
from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import PrefillWorkload

import parity_util as pu

pytestmark = pytest.mark.gpu


# 1024 keys are a tile of 128 sub-blocks: 31 tiles (one block), 32 and a ragged 33rd (two), 67 (four), 128 (eight)
@pytest.mark.parametrize("n_key,n_query,P,M,Ksp", [(31 * 1024, 9, 128, 32, 2048), (32 * 1024 + 200, 9, 128, 32, 2048), (67 * 1024 + 1, 17, 64, 64, 512),
                                                   (128 * 1024, 5, 256, 16, 1024), (20000, 7, 128, 96, 2048), (20000, 7, 64, 130, 3000),
                                                   (20000, 7, 256, 40, 2048)])
def test_chunk_at_the_end(cuda_device, n_key, n_query, P, M, Ksp):
    cfg = CONFIGS["cfg3"].replace(L=n_key, P=P, M=M, Ksp=Ksp, W=64, key_dtype="bf16", R=1, seed=n_key)
    wl = PrefillWorkload(cfg, cuda_device, q_pos0=n_key - n_query, n_query=n_query)
    g = torch.Generator().manual_seed(M)
    for t, hi in ((wl.q_idx, 1), (wl.keys["k"], 1), (wl.w, 3)):
        t.copy_(torch.randint(-hi, hi + 1, t.shape, generator=g).to(t.dtype))
    wl.prepare()
    pages = torch.empty((n_query, M), dtype=torch.int32, device=cuda_device)
    wl.index(pages_out=pages)
    assert wl.ctx.status() == 0
    caches = ref.HostCaches(pu.to_np(wl.keys["k"]), None, [], [], cfg.B, n_key=n_key)
    for i in (0, n_query // 2, n_query - 1):
        t = n_key - n_query + i
        want, want_pages = ref.select_query(t, pu.to_np(wl.q_idx[i]), pu.to_np(wl.w[i]), caches, P=P, B=cfg.B, M=M, Ksp=Ksp, S=cfg.S, W=cfg.W)
        got, n, gp = pu.to_np(wl.sparse_idx[i]), int(wl.n_sparse[i]), pu.to_np(pages[i])
        assert list(gp[gp >= 0]) == list(want_pages), t
        assert n == len(want) and list(got[:n]) == list(want) and (got[n:] == -1).all(), t

"""Indexer scores at the ends of fp32 (needs a B200): heads whose dot products leave its range, or come near its end (a head below it
counts as 0, the oracle's ReLU, whatever the form of the head sum), and heads that cancel but for its last bits."""
import pytest
import torch

from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload, PrefillWorkload

import parity_util as pu

pytestmark = pytest.mark.gpu

BELOW, NEAR = (1, 2, 4, 7, 11, 14, 30, 45, 63), (5, 6, 12, 37)   # heads: even, odd, in either half of each eight


def _far_heads(wl):
    """Keys of positive numbers, the first dim 1, 1.25 or 1.5; heads BELOW have dot products of some -1e39 (-inf in fp32), heads NEAR
    some 2.5e38, whose double is infinite, with weights that make them count as much as any other."""
    g = torch.Generator().manual_seed(3)
    k = wl.keys["k"]
    kf = torch.rand((k.shape[0], k.shape[1]), generator=g) * 0.25 + 0.01
    kf[:, 0] = 1.0 + 0.25 * torch.randint(0, 3, (k.shape[0],), generator=g)
    if "scale" in wl.keys:
        k.copy_(kf.to(torch.float8_e4m3fn).view(torch.uint8))
        wl.keys["scale"].fill_(1.0)
    else:
        k.copy_(kf.to(torch.bfloat16))
    for h in BELOW:
        wl.q_idx[:, h] = -torch.rand(wl.q_idx[:, h].shape, generator=g).to(wl.q_idx) * 1.0e38 - 2.0e38
    for h in NEAR:
        wl.q_idx[:, h] = 0.0
        wl.q_idx[:, h, 0] = 1.9e38
        wl.w[:, h] = wl.w[:, h] * 1.0e-38


# prompt; the same with many queries; flat; large budget
@pytest.mark.parametrize("base,change,n_query", [("cfg2", dict(L=9000, M=16), 40), ("cfg3", dict(L=9000, M=16), 40), ("cfg2", dict(L=3000, M=8), 3000),
                                                 ("cfg2", dict(L=6000, hi_enable=False), 20), ("cfg3", dict(L=20000, hi_enable=False), 20),
                                                 ("cfg2", dict(L=20000, M=80), 20), ("cfg3", dict(L=20000, M=80), 20)])
def test_prompt(cuda_device, base, change, n_query):
    cfg = CONFIGS[base].replace(**{"R": 1, "Ksp": 256, "W": 130, "seed": 9, **change})
    wl = PrefillWorkload(cfg, cuda_device, q_pos0=cfg.L - n_query, n_query=n_query)
    _far_heads(wl)
    wl.prepare()
    pages = torch.empty((n_query, cfg.M), dtype=torch.int32, device=cuda_device)
    wl.index(pages_out=pages)
    assert wl.ctx.status() == 0
    m = pu.check_prefill(wl, range(wl.q_pos0, wl.q_pos0 + n_query, max(1, n_query // 12)), check_attention=False, pages=pages if cfg.hi_enable else None)
    print(base, change, m.summary())
    m.assert_ok(pu.TOL_BF16)


@pytest.mark.parametrize("key_dtype", ["e4m3", "bf16"])
@pytest.mark.parametrize("change", [dict(), dict(P=128, kv_page=128, M=8), dict(hi_enable=False)])
def test_decode(cuda_device, key_dtype, change):
    cfg = CONFIGS["cfg4"].replace(**{"batch": 6, "ctx_lo": 3000, "ctx_hi": 9000, "M": 16, "Ksp": 256, "R": 1, "W": 130, "seed": 9, "key_dtype": key_dtype, **change})
    wl = DecodeWorkload(cfg, cuda_device)
    _far_heads(wl)
    wl.prepare()
    wl.index()
    assert wl.ctx.status() == 0
    m = pu.check_decode(wl, range(cfg.batch), check_attention=False)
    print(key_dtype, change, m.summary())
    m.assert_ok(pu.TOL_BF16)


@pytest.mark.parametrize("groups", [1, 2])
@pytest.mark.parametrize("base,B", [("cfg2", 4), ("cfg2", 8), ("cfg2", 16), ("cfg3", 8)])   # 32, 16 and 8 mean keys a page
def test_pages_of_cancelling_heads(cuda_device, base, B, groups):
    """Head dot products of 2^22 + e and 2^22 with weights 1 and -1: a mean key counts e, exact as long as its heads are added up before
    it meets the page's other mean keys (a page's sum of one head, up to 2^27, is not).  Page scores are integers one apart."""
    L, n_query = 9000, 3000
    cfg = CONFIGS[base].replace(R=1, Ksp=256, W=130, seed=9, L=L, P=128, M=16, B=B)
    wl = PrefillWorkload(cfg, cuda_device, q_pos0=L - n_query, n_query=n_query)
    wl.ctx.tune(0, groups)             # LSA_TUNE_COARSE_GROUPS
    n_pages, spp = -(-L // cfg.P), cfg.P // B
    g = torch.Generator().manual_seed(B)
    total = torch.randperm(n_pages, generator=g) + 2 * spp      # of a page: dealt to its mean keys, the last one takes the rest
    e = torch.randint(0, 3, (n_pages, spp), generator=g)
    e[:, -1] = total - e[:, :-1].sum(1)
    code = torch.zeros((n_pages * spp, cfg.d_I))
    code[:, 0] = 256.0                                          # e4m3 codes with a scale of 8, or their products: 2048, e
    code[:, 1:17] = (e.reshape(-1, 1) - 16 * torch.arange(16)).clamp(0, 16)    # in parts of at most 16: exact in e4m3
    code = code.repeat_interleave(B, 0)[:L]
    if "scale" in wl.keys:
        wl.keys["k"].copy_(code.to(torch.float8_e4m3fn).view(torch.uint8))
        wl.keys["scale"].fill_(8.0)
    else:
        wl.keys["k"].copy_((8.0 * code).to(torch.bfloat16))
    wl.q_idx.zero_()
    wl.w.zero_()
    for plus, minus in ((0, 1), (12, 45)):
        wl.q_idx[:, [plus, minus], 0] = 2048.0
        wl.q_idx[:, plus, 1:17] = 0.125
        wl.w[:, plus], wl.w[:, minus] = 1.0, -1.0
    wl.prepare()
    pages = torch.empty((n_query, cfg.M), dtype=torch.int32, device=cuda_device)
    wl.index(pages_out=pages)
    assert wl.ctx.status() == 0
    m = pu.check_prefill(wl, range(wl.q_pos0, wl.q_pos0 + n_query, 157), check_attention=False, pages=pages)
    s = m.summary()
    assert s["page_sets_differ"] == 0 and s["min_overlap"] == 1.0, s

"""Indexer heads whose dot products leave the range of fp32, or come near its end (needs a B200): a head below it counts as 0 (the
oracle's ReLU), whatever the form of the head sum."""
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

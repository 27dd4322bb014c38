"""Selection of at most 4096 keys by one block (needs a B200): inputs of small whole numbers, whose scores are exact in fp32 in
any order of summation, so that pages and tokens must be the oracle's, ties by position included."""
import pytest
import torch

from oracle import reference_run as ref
from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload, PrefillWorkload

import parity_util as pu

pytestmark = pytest.mark.gpu

# equal: nothing but ties.  few: a handful of values.  outlier: a few keys 64 x as large (several passes).  tiny: scores of
# some 2^-135, whose range has no finite reciprocal (bit by bit).  plain: hundreds of values.
KINDS = ("equal", "few", "outlier", "tiny", "plain")


def _whole_numbers(wl, kind, seed):
    g = torch.Generator().manual_seed(seed)

    def draw(t, hi):
        return t.copy_(torch.randint(-hi, hi + 1, t.shape, generator=g).to(t.dtype))

    draw(wl.q_idx, 1)
    draw(wl.keys["k"], 1)
    if kind == "outlier":
        wl.keys["k"][torch.randperm(len(wl.keys["k"]), generator=g)[:max(1, len(wl.keys["k"]) // 400)].to(wl.keys["k"].device)] *= 64
    draw(wl.w, 3 if kind == "plain" else 1)
    if kind in ("few", "equal"):
        wl.w[:, 1:] = 0
    if kind == "equal":
        wl.w.zero_()
    if kind == "tiny":
        wl.w *= 2.0 ** -140


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("M,Ksp,hi", [(64, 2048, 9000), (3, 100, 700), (16, 4, 2500), (1, 64, 6000)])
def test_paged(cuda_device, kind, M, Ksp, hi):
    cfg = CONFIGS["cfg4"].replace(batch=9, ctx_lo=5, ctx_hi=hi, key_dtype="bf16", R=1, M=M, Ksp=Ksp, seed=M + Ksp)
    wl = DecodeWorkload(cfg, cuda_device)
    _whole_numbers(wl, kind, M)
    wl.prepare()
    wl.index()
    assert wl.ctx.status() == 0
    for b in range(cfg.batch):
        caches, t = pu.decode_caches(wl, b)
        want, _ = ref.select_query(t, pu.to_np(wl.q_idx[b]), pu.to_np(wl.w[b]), caches, P=cfg.P, B=cfg.B, M=M, Ksp=Ksp, S=cfg.S, W=cfg.W)
        got = pu.to_np(wl.sparse_idx[b])
        n = int(wl.n_sparse[b])
        assert n == len(want) and list(got[:n]) == list(want) and (got[n:] == -1).all(), (b, t)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("L,P,M,Ksp", [(5400, 128, 32, 2048), (1500, 64, 3, 200), (9000, 64, 64, 4096)])
def test_prompt(cuda_device, kind, L, P, M, Ksp):
    cfg = CONFIGS["cfg3"].replace(L=L, P=P, M=M, Ksp=Ksp, W=64, key_dtype="bf16", R=1, seed=L)
    wl = PrefillWorkload(cfg, cuda_device)
    _whole_numbers(wl, kind, L)
    wl.prepare()
    pages = torch.empty((L, M), dtype=torch.int32, device=cuda_device)
    wl.index(pages_out=pages)
    assert wl.ctx.status() == 0
    caches = ref.HostCaches(pu.to_np(wl.keys["k"]), None, [], [], cfg.B, n_key=L)
    for t in pu.boundary_queries(cfg, 0, L, 12, seed=1):
        want, want_pages = ref.select_query(t, pu.to_np(wl.q_idx[t]), pu.to_np(wl.w[t]), caches, P=P, B=cfg.B, M=M, Ksp=Ksp, S=cfg.S, W=cfg.W)
        got, n, gp = pu.to_np(wl.sparse_idx[t]), int(wl.n_sparse[t]), pu.to_np(pages[t])
        assert list(gp[gp >= 0]) == list(want_pages), t
        assert n == len(want) and list(got[:n]) == list(want) and (got[n:] == -1).all(), t


@pytest.mark.parametrize("kind", ["few", "plain"])
@pytest.mark.parametrize("pages", [1023, 1024, 1025, 1100])
def test_pages_of_long_contexts(cuda_device, kind, pages):
    """Pages of 128 tokens on either side of the count where their selection changes hands (page 0 holds the sink, the last one the window)."""
    cfg = CONFIGS["cfg4"].replace(batch=2, ctx_lo=pages * 128 + 130, ctx_hi=pages * 128 + 130, key_dtype="bf16", R=1, M=8, P=128, kv_page=128, W=130,
                                  Ksp=256, seed=pages, H=16, d_qk=128, d_v=128, mla=False)
    wl = DecodeWorkload(cfg, cuda_device)
    _whole_numbers(wl, kind, pages)
    wl.prepare()
    listed = torch.empty((cfg.batch, cfg.M), dtype=torch.int32, device=cuda_device)
    for knob in (0, 2):
        wl.ctx.tune(5, knob)       # LSA_TUNE_FINE_PAGED_TC
        wl.index(pages_out=listed)
        assert wl.ctx.status() == 0
        caches, t = pu.decode_caches(wl, 1)
        want, want_pages = ref.select_query(t, pu.to_np(wl.q_idx[1]), pu.to_np(wl.w[1]), caches, P=cfg.P, B=cfg.B, M=cfg.M, Ksp=cfg.Ksp, S=cfg.S, W=cfg.W)
        assert list(pu.to_np(listed[1])) == list(want_pages)
        assert list(pu.to_np(wl.sparse_idx[1]))[:len(want)] == list(want)


@pytest.mark.parametrize("kind", ["few", "plain"])
@pytest.mark.parametrize("M,Ksp", [(3, 100), (9, 4), (64, 612)])
def test_contexts_about_the_window(cuda_device, kind, M, Ksp):
    """Sequences inside their window, which select nothing, beside some that do."""
    cfg = CONFIGS["cfg4"].replace(batch=33, ctx_lo=255, ctx_hi=900, key_dtype="bf16", R=1, M=M, Ksp=Ksp, seed=M + Ksp)
    wl = DecodeWorkload(cfg, cuda_device)
    edge = [1, 255, 256, 259, 260, 261, 262, 323, 324]
    wl.ctx_len[:len(edge)] = torch.minimum(torch.tensor(edge, dtype=torch.int32, device=cuda_device), (wl.page_table[:len(edge)] >= 0).sum(1).int() * 64)
    _whole_numbers(wl, kind, M)
    wl.prepare()
    pages = torch.empty((cfg.batch, M), dtype=torch.int32, device=cuda_device)
    wl.index(pages_out=pages)
    assert wl.ctx.status() == 0
    for b in range(cfg.batch):
        caches, t = pu.decode_caches(wl, b)
        want, want_pages = ref.select_query(t, pu.to_np(wl.q_idx[b]), pu.to_np(wl.w[b]), caches, P=cfg.P, B=cfg.B, M=M, Ksp=Ksp, S=cfg.S, W=cfg.W)
        got, gp, n = pu.to_np(wl.sparse_idx[b]), pu.to_np(pages[b]), int(wl.n_sparse[b])
        assert list(gp[gp >= 0]) == list(want_pages), (b, t)
        assert n == len(want) and list(got[:n]) == list(want) and (got[n:] == -1).all(), (b, t)

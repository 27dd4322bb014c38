"""What the indexer writes stays inside the caller's lists (needs a B200): guard words around them."""
import pytest
import torch

from oracle import reference_run as ref
from paper_2608_01662_b200 import binding
from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload, PrefillWorkload

import parity_util as pu

pytestmark = pytest.mark.gpu

GUARD = -77
PAD = 4096      # guard words on either side


def guarded(shape, device):
    """(view of int32 [shape], the tensor it lies in)."""
    n = 1
    for d in shape:
        n *= d
    whole = torch.full((n + 2 * PAD,), GUARD, dtype=torch.int32, device=device)
    return whole[PAD:PAD + n].view(shape), whole


def assert_guards(whole):
    assert (whole[:PAD] == GUARD).all() and (whole[-PAD:] == GUARD).all()


# Without the hierarchy a query has every eligible page: 14, 14, 1 and 3 at the end of these caches.
@pytest.mark.parametrize("base,L,M,P", [("cfg1", 1000, 8, 64), ("cfg1", 1000, 1, 64), ("cfg1", 300, 4, 256), ("cfg3", 1500, 2, 128)])
def test_pages_without_the_hierarchy(cuda_device, base, L, M, P):
    """At most M pages are listed, the first eligible ones."""
    cfg = CONFIGS[base].replace(L=L, M=M, P=P, B=8, Ksp=64, R=1, hi_enable=False, seed=L)
    wl = PrefillWorkload(cfg, cuda_device)
    wl.prepare()
    pages, whole = guarded((L, M), cuda_device)
    wl.index(pages_out=pages)
    assert wl.ctx.status() == 0
    assert_guards(whole)
    got = pu.to_np(pages)
    for t in range(L):
        n = (t - cfg.W) // P - cfg.S // P + 1 if t - cfg.W >= cfg.S else 0
        want = [cfg.S // P + i for i in range(min(n, M))]
        assert list(got[t]) == want + [-1] * (M - len(want)), t


class EmptyLists:
    """In place of a workload's lists of no entries per query: an address with guard words on either side."""

    def __init__(self, wl, n):
        self.whole = torch.full((2 * PAD,), GUARD, dtype=torch.int32, device=wl.device)
        self.counts, self.counts_whole = guarded((n,), wl.device)
        wl.sparse_idx, wl.n_sparse = self.whole.data_ptr() + 4 * PAD, self.counts

    def check(self):
        assert (self.whole == GUARD).all() and (self.counts == 0).all()
        assert_guards(self.counts_whole)


# Every way a selection is made: rows of the flat indexer (few: clusters; many), the fine stages, the warp-per-query indexer
# and the block form beside it, large budgets with short and long rows.
@pytest.mark.parametrize("base,change,n_query", [
    ("cfg3", dict(L=20000, hi_enable=False), 6), ("cfg2", dict(L=17000, hi_enable=False), 300), ("cfg2", dict(L=6000, hi_enable=False), 40),
    ("cfg2", dict(L=9000, M=16), 200), ("cfg3", dict(L=9000), 200), ("cfg1", dict(L=3000), 200), ("cfg1", dict(L=3000, M=32), 200),
    ("cfg3", dict(L=30000, M=48), 20), ("cfg3", dict(L=30000, M=160), 20), ("cfg2", dict(L=4000, pooling="minmax", M=8), 50),
])
def test_no_sparse_keys_prompt(cuda_device, base, change, n_query):
    """k_sparse = 0: sink and window only, nothing written."""
    cfg = CONFIGS[base].replace(**{"Ksp": 0, "R": 1, "W": 130, "seed": 5, **change})
    wl = PrefillWorkload(cfg, cuda_device, q_pos0=cfg.L - n_query, n_query=n_query)
    wl.prepare()
    lists = EmptyLists(wl, n_query)
    wl.step()
    assert wl.ctx.status() == 0
    lists.check()
    _check_band(cfg, wl, range(0, n_query, 7))


def _check_band(cfg, wl, queries):
    caches = ref.HostCaches(pu.to_np(wl.keys["k"]), pu.to_np(wl.keys["scale"]) if "scale" in wl.keys else None,
                            [pu.to_np(k) for k in wl.k], [pu.to_np(v) for v in wl.v], cfg.B, n_key=wl.n_key)
    m = pu.Metrics()
    for i in queries:
        want, want_lse = ref.attend_query(wl.q_pos0 + i, [pu.to_np(q[i]) for q in wl.q], caches, [], S=cfg.S, W=cfg.W,
                                          sm_scale=cfg.sm_scale, d_v=cfg.d_v)
        m.add_out(pu.to_np(wl.out[0][i]), want[0], pu.to_np(wl.lse[0][i]) if wl.lse[0] is not None else None, want_lse[0])
    m.assert_ok(pu.TOL_BF16)


@pytest.mark.parametrize("change", [
    dict(), dict(key_dtype="bf16", batch=40), dict(P=128, kv_page=128, M=16), dict(batch=1), dict(hi_enable=False),
    dict(hi_enable=False, ctx_hi=20000), dict(hi_enable=False, ctx_hi=20000, batch=90),
    dict(H_I=8, d_I=64, key_dtype="bf16"),
])
@pytest.mark.parametrize("knob", [0, 1, 2])
def test_no_sparse_keys_decode(cuda_device, change, knob):
    cfg = CONFIGS["cfg4"].replace(**{"batch": 5, "ctx_lo": 1, "ctx_hi": 3000, "M": 8, "Ksp": 0, "R": 1, "W": 130, "seed": 6, **change})
    wl = DecodeWorkload(cfg, cuda_device)
    wl.prepare()
    wl.ctx.tune(5, knob)           # LSA_TUNE_FINE_PAGED_TC
    lists = EmptyLists(wl, cfg.batch)
    wl.step()
    assert wl.ctx.status() == 0
    lists.check()
    m = pu.Metrics()
    for b in range(min(5, cfg.batch)):
        caches, t = pu.decode_caches(wl, b)
        want, want_lse = ref.attend_query(t, [pu.to_np(q[b]) for q in wl.q], caches, [], S=cfg.S, W=cfg.W, sm_scale=cfg.sm_scale, d_v=cfg.d_v)
        m.add_out(pu.to_np(wl.out[0][b]), want[0], pu.to_np(wl.lse[0][b]), want_lse[0])
    m.assert_ok(pu.TOL_BF16)


@pytest.mark.parametrize("change", [dict(L=3000), dict(L=17000, hi_enable=False)])
def test_no_sparse_keys_from_host_buffers(cuda_device, change):
    """The list takes no room in the staging area: its address is that of the counts."""
    n_query = 100
    cfg = CONFIGS["cfg3"].replace(**{"Ksp": 0, "R": 1, "W": 130, "M": 8, **change})
    wl = PrefillWorkload(cfg, cuda_device, with_lse=False, q_pos0=cfg.L - n_query, n_query=n_query)
    wl.prepare()
    nbytes = binding.host_stage_bytes(wl.params, 32)
    whole = [torch.full((nbytes + 8 * PAD,), 77, dtype=torch.uint8, device=cuda_device) for _ in range(2)]
    out = [torch.zeros(o.shape, dtype=o.dtype).pin_memory() for o in wl.out]
    wl.ctx.layer_group_host(wl.q_idx.cpu().pin_memory(), wl.w.cpu().pin_memory(), wl.keys["k"], wl.keys["scale"], wl.kmean, wl.q_pos0, n_query,
                            wl.n_key, [q.cpu().pin_memory() for q in wl.q], wl.k, wl.v, out, 32, [t[4 * PAD:4 * PAD + nbytes] for t in whole])
    assert wl.ctx.status() == 0
    torch.cuda.synchronize()
    assert all((t[:4 * PAD] == 77).all() and (t[-4 * PAD:] == 77).all() for t in whole)
    wl.out = out
    _check_band(cfg, wl, range(0, n_query, 7))

"""Selection of long rows (needs a B200), one block per row and a cluster per row: bit-exact against the oracle, also where
the sample of the row misleads (then the radix select takes over) and where the ties at the threshold have to be cut."""
import numpy as np
import pytest
import torch

from oracle import lsa_oracle as orc
from paper_2608_01662_b200 import binding
from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload

import parity_util as pu

pytestmark = pytest.mark.gpu


def _sampled(n):
    """The items that the kernels may sample: quads at every n / (m / 4)-th place, for each sample size m."""
    return np.unique(np.concatenate([((np.arange(m // 4, dtype=np.int64) * n // (m // 4)) & ~3)[:, None] + np.arange(4)
                                     for m in (4096, 8192, 16384)]).ravel())


def _row(kind, n, rng):
    if kind == "normal":
        return rng.standard_normal(n)
    if kind == "ties":            # a handful of values: thousands of items at the threshold
        return np.round(rng.standard_normal(n) * 2) / 2
    if kind == "equal":
        return np.full(n, -1.25)
    if kind == "sampled_high":    # every sampled item is large, few others are: fewer than k are collected
        x = rng.standard_normal(n)
        x[_sampled(n)] += 100.0
        return x
    if kind == "sampled_low":     # the other way round: more than there is room for
        x = rng.standard_normal(n) + 100.0
        x[_sampled(n)] -= 100.0
        return x
    x = rng.standard_normal(n)    # "piece": all of the selection in one corner of the row
    x[n // 2:n // 2 + 5000] += 50.0
    return x


KINDS = ("normal", "ties", "equal", "sampled_high", "sampled_low", "piece")


@pytest.mark.parametrize("n_cand,k,n_query", [(16384, 1, 300), (16640, 700, 9), (16385, 2048, 257), (65537, 2048, 260), (40000, 4100, 258), (140001, 300, 257),
                                              (16384, 2048, 6), (49153, 8192, 6), (131073, 2048, 12), (600001, 2048, 6),
                                              # a block per row although few; the radix select by clusters, and by blocks
                                              (20001, 2048, 40), (70000, 8192, 20), (16385, 8192, 9), (16384, 8192, 258)])
def test_select_long_rows(cuda_device, n_cand, k, n_query):
    rng = np.random.default_rng(n_cand + k)
    rows = np.stack([_row(kind, n_cand, rng) for kind in KINDS]).astype(np.float32)
    params = binding.make_params(CONFIGS["cfg1"].replace(S=5, W=77))
    ctx = binding.Context(params, n_query, n_cand, device=cuda_device)
    scores = torch.from_numpy(rows).to(cuda_device)[torch.arange(n_query, device=cuda_device) % len(KINDS)]
    idx = torch.empty((n_query, k), dtype=torch.int32, device=cuda_device)
    cnt = torch.empty((n_query,), dtype=torch.int32, device=cuda_device)
    for in_range in (False, True):
        q_pos0 = n_cand - n_query
        ctx.select(scores, None, q_pos0, k, in_range, idx, cnt)
        assert ctx.status() == 0
        for i in (*range(len(KINDS)), n_query - 1):
            want = orc.select_fp32(rows[i % len(KINDS)], None, q_pos0 + i, k, apply_range=in_range, S=5, W=77)
            got = idx[i].cpu().numpy()
            assert int(cnt[i]) == len(want) and np.array_equal(got[:len(want)], want) and (got[len(want):] == -1).all(), (i, in_range)


# the last columns of the scoring range at the query's position, and positions past 2^31
@pytest.mark.parametrize("n_cand,n_query", [(1000, 5), (20000, 5), (20000, 300)])
@pytest.mark.parametrize("q_pos0", [(1 << 31) - 1 - 80, (1 << 31) + 70, 1 << 40])
def test_queries_at_far_positions(cuda_device, n_cand, n_query, q_pos0):
    """apply_range with positions that do not fit 32 bits: every candidate from the sink on is in range."""
    rng = np.random.default_rng(n_cand)
    rows = rng.standard_normal((n_query, n_cand)).astype(np.float32)
    k = 500
    ctx = binding.Context(binding.make_params(CONFIGS["cfg1"].replace(S=5, W=77)), n_query, n_cand, device=cuda_device)
    idx = torch.empty((n_query, k), dtype=torch.int32, device=cuda_device)
    cnt = torch.empty((n_query,), dtype=torch.int32, device=cuda_device)
    ctx.select(torch.from_numpy(rows).to(cuda_device), None, q_pos0, k, True, idx, cnt)
    assert ctx.status() == 0
    for i in (0, n_query - 1):
        want = orc.select_fp32(rows[i], None, q_pos0 + i, k, apply_range=True, S=5, W=77)
        assert int(cnt[i]) == len(want) == k and np.array_equal(idx[i].cpu().numpy(), want)


@pytest.mark.parametrize("batch", [2, 40, 257])
def test_flat_decode_lists_its_rows(cuda_device, batch):
    """The selection of long rows by clusters writes the cache rows as well; for more rows than get a cluster a kernel of its own does."""
    cfg = CONFIGS["cfg4"].replace(batch=batch, ctx_lo=300, ctx_hi=20000, hi_enable=False, R=1, Ksp=1024, seed=batch)
    wl = DecodeWorkload(cfg, cuda_device)
    wl.prepare()
    wl.step()
    assert wl.ctx.status() == 0
    m = pu.check_decode(wl, range(0, batch, max(1, batch // 12)))
    print(batch, m.summary())
    m.assert_ok(pu.TOL_FP8)

"""Decode batches larger than the chip (needs a B200): blocks of the attention kernel go on to further sequences, whose first
tiles are requested ahead of their queries.  Repeated steps give the same bits and no wait runs out."""
import pytest
import torch

from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,lo,hi,layers", [(200, 1, 700, 3), (320, 700, 1600, 2), (449, 1, 130, 2)])
def test_blocks_that_go_on(cuda_device, batch, lo, hi, layers):
    wl = DecodeWorkload(CONFIGS["cfg4"].replace(batch=batch, ctx_lo=lo, ctx_hi=hi, R=layers, Ksp=256, M=16, seed=batch))
    wl.prepare()
    wl.step()
    first = [o.clone() for o in wl.out]
    differ = torch.zeros((), dtype=torch.int64, device=cuda_device)
    for _ in range(150):
        for o in wl.out:
            o.fill_(7.0)
        wl.step()
        for a, b in zip(first, wl.out):
            differ += (a.view(torch.int16) != b.view(torch.int16)).sum()
    assert wl.ctx.status() == 0 and int(differ) == 0


@pytest.mark.parametrize("batch,lo,hi", [(1, 20000, 20000), (3, 1, 400), (7, 900, 3000)])
def test_sixteen_splits(cuda_device, batch, lo, hi):
    """Sixteen row splits of a sequence, also where most of them have no rows."""
    cfg = CONFIGS["cfg4"].replace(batch=batch, ctx_lo=lo, ctx_hi=hi, R=2, seed=batch)
    wl = DecodeWorkload(cfg, cuda_device)
    wl.prepare()
    wl.ctx.tune(2, 16)             # LSA_TUNE_ATTN_SPLIT
    wl.step()
    assert wl.ctx.status() == 0
    m = pu.check_decode(wl, range(batch))
    m.assert_ok(pu.TOL_BF16)


@pytest.mark.parametrize("batch,lo,hi", [(1, 20000, 20000), (1, 300, 300), (2, 700, 30000), (3, 1, 5000)])
def test_parts_of_the_value_dims(cuda_device, batch, lo, hi):
    """Few sequences: the value dims of a split in parts, each by a cluster of its own, give the bits of the undivided ones."""
    cfg = CONFIGS["cfg4"].replace(batch=batch, ctx_lo=lo, ctx_hi=hi, R=2, seed=batch)
    wl = DecodeWorkload(cfg, cuda_device)
    wl.prepare()
    wl.step()
    parts = [t.clone() for t in wl.out + wl.lse]
    m = pu.check_decode(wl, range(batch))
    m.assert_ok(pu.TOL_BF16)
    wl.ctx.tune(2, 16)             # LSA_TUNE_ATTN_SPLIT
    wl.step()
    assert wl.ctx.status() == 0
    assert all(torch.equal(a, b) for a, b in zip(parts, wl.out + wl.lse))


@pytest.mark.parametrize("batch,lo,hi", [(16, 700, 6000), (22, 1, 400), (34, 900, 3000), (45, 1, 2500)])
def test_splits_that_do_not_divide_the_rows(cuda_device, batch, lo, hi):
    """Batches between the numbers of clusters that run at once, which three or six splits would serve; some splits have no rows."""
    cfg = CONFIGS["cfg4"].replace(batch=batch, ctx_lo=lo, ctx_hi=hi, R=2, seed=batch)
    wl = DecodeWorkload(cfg, cuda_device)
    wl.prepare()
    wl.step()
    assert wl.ctx.status() == 0
    m = pu.check_decode(wl, range(0, batch, 3))
    m.assert_ok(pu.TOL_BF16)


@pytest.mark.parametrize("batch,lo,hi,split", [(16, 700, 6000, 4), (22, 1, 400, 4), (34, 900, 3000, 2), (45, 1, 2500, 2)])
def test_splits_are_powers_of_two(cuda_device, batch, lo, hi, split):
    """The bits of a call that asks for the number of splits (other numbers made short contexts and some batches slower)."""
    wl = DecodeWorkload(CONFIGS["cfg4"].replace(batch=batch, ctx_lo=lo, ctx_hi=hi, R=2, seed=batch), cuda_device)
    wl.prepare()
    wl.step()
    chosen = [t.clone() for t in wl.out + wl.lse]
    wl.ctx.tune(2, split)          # LSA_TUNE_ATTN_SPLIT
    wl.step()
    assert wl.ctx.status() == 0
    assert all(torch.equal(a, b) for a, b in zip(chosen, wl.out + wl.lse))

"""Decode batches larger than the chip (needs a B200): blocks of the attention kernel go on to further sequences, whose first
tiles are requested ahead of their queries.  Repeated steps give the same bits and no wait runs out."""
import pytest
import torch

from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import DecodeWorkload

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

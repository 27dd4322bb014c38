"""What the indexer writes stays inside the caller's lists (needs a B200): guard words around them."""
import pytest
import torch

from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import PrefillWorkload

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

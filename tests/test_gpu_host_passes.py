"""lsa_layer_group_host in one pass, two and many (needs a B200): the bytes of the device-resident run."""
import pytest
import torch

from paper_2608_01662_b200 import binding
from paper_2608_01662_b200.configs import CONFIGS
from paper_2608_01662_b200.workload import PrefillWorkload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_query,stage_queries,layers", [(1, 64, 1), (300, 300, 3), (301, 300, 2), (1000, 128, 4)])
def test_host_passes_equal_the_device_run(cuda_device, n_query, stage_queries, layers):
    cfg = CONFIGS["cfg3"].replace(name="host_passes", L=3000, M=8, Ksp=512, W=384, R=layers, seed=n_query)
    wl = PrefillWorkload(cfg, cuda_device, with_lse=False, q_pos0=cfg.L - n_query, n_query=n_query)
    wl.prepare()
    wl.step()
    torch.cuda.synchronize()
    stage = [torch.empty(binding.host_stage_bytes(wl.params, stage_queries), dtype=torch.uint8, device=cuda_device) for _ in range(2)]
    q_idx, w, q = wl.q_idx.cpu().pin_memory(), wl.w.cpu().pin_memory(), [x.cpu().pin_memory() for x in wl.q]
    for _ in range(3):   # back to back on the same buffers: a call's copies follow the one before
        out = [torch.zeros(o.shape, dtype=o.dtype).pin_memory() for o in wl.out]
        wl.ctx.layer_group_host(q_idx, w, wl.keys["k"], wl.keys["scale"], wl.kmean, wl.q_pos0, n_query, wl.n_key, q, wl.k, wl.v, out,
                                stage_queries, stage)
    torch.cuda.current_stream(cuda_device).synchronize()   # the stream the context was made on waits for every copy
    assert wl.ctx.status() == 0
    for a, b in zip(out, wl.out):
        assert torch.equal(a, b.cpu())


def test_no_queries_and_a_graph(cuda_device):
    """A call without queries does nothing, also under capture; a call with some replays from a graph."""
    cfg = CONFIGS["cfg3"].replace(name="host_graph", L=2000, M=8, Ksp=256, W=130, R=2, seed=2)
    n_query, sq = 100, 32
    side = torch.cuda.Stream(device=cuda_device)
    with torch.cuda.stream(side):
        wl = PrefillWorkload(cfg, cuda_device, with_lse=False, q_pos0=cfg.L - n_query, n_query=n_query)
        wl.prepare()
        stage = [torch.empty(binding.host_stage_bytes(wl.params, sq), dtype=torch.uint8, device=cuda_device) for _ in range(2)]
        q_idx, w, q = wl.q_idx.cpu().pin_memory(), wl.w.cpu().pin_memory(), [x.cpu().pin_memory() for x in wl.q]
        out = [torch.zeros(o.shape, dtype=o.dtype).pin_memory() for o in wl.out]

        def call(n):
            wl.ctx.layer_group_host(q_idx, w, wl.keys["k"], wl.keys["scale"], wl.kmean, wl.q_pos0, n, wl.n_key, q, wl.k, wl.v, out, sq, stage)

        call(0)
        call(n_query)
        side.synchronize()
        want = [o.clone() for o in out]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            call(0)
            call(n_query)
        for o in out:
            o.zero_()
        graph.replay()
        side.synchronize()
    assert wl.ctx.status() == 0
    for a, b in zip(want, out):
        assert torch.equal(a, b)

